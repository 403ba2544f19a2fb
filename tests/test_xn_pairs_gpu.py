"""Eq. e:xn2 in pairs of floats: the result is the rounding of the exact solution, over the whole
range of the fast form and beyond it, and for every length and alignment of the arrays."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def art():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art as A
    return A


def _exact(x0, g, n, alpha, dt):
    """Eq. e:xn2 in extended precision, written without cancellation."""
    q = np.longdouble
    x0, g, n, alpha, dt = (np.asarray(v).astype(q) for v in (x0, g, n, np.float32(alpha), np.float32(dt)))
    a = alpha * n
    r = np.sqrt(g * (g + 4 * a))
    h = g + 2 * a + r
    B = np.where(x0 > 0.5, (g + r) / h - (1 - x0), x0 - 2 * a / h)
    K, E = np.exp(-r * dt), -np.expm1(-r * dt)
    with np.errstate(invalid="ignore", divide="ignore"):  # the branch not taken
        return _select(x0, g, a, r, h, B, K, E, dt)


def _select(x0, g, a, r, h, B, K, E, dt):
    up = 2 * a / h + r * B * K / ((g + r) / 2 + a * (1 - x0) + a * B * K)
    down = (x0 * r + h / 2 * -B * E) / (r + a * -B * E)
    ad = a * dt
    dark = (x0 + (1 - x0) * ad) / (1 + (1 - x0) * ad)
    return np.where(g > 0, np.where(B > 0, up, down), dark)


def _inputs(n, seed, decades):
    rng = np.random.default_rng(seed)
    nH = (10.0 ** rng.uniform(-decades / 2, decades / 2, n)).astype(np.float32)
    gam = (10.0 ** rng.uniform(-decades, decades, n)).astype(np.float32)
    gam[rng.random(n) < 0.1] = 0.0
    x = np.where(rng.random(n) < 0.5, 10.0 ** rng.uniform(-8, 0, n), rng.random(n)).astype(np.float32)
    x[:: 97] = 0.0
    x[1:: 97] = 1.0
    x[2:: 97] = np.float32(1) - np.float32(2.0) ** -24
    return nH, gam, x


@pytest.mark.parametrize("decades,alpha,dt", [
    (2, 2e-4, 5.0), (3, 0.02, 3.0), (4, 1.0, 1e-3), (4, 1.0, 1e3), (8, 3e-13, 1e12), (12, 1e-5, 7.0),
])
def test_quadratic_update_rounds_the_exact_solution(art, decades, alpha, dt):
    nH, gam, x = _inputs(200_000, decades, decades)
    t = [torch.from_numpy(v.copy()).cuda() for v in (gam, nH, x)]
    art.xn_update(*t, alpha, dt, method="a")
    got = t[2].cpu().numpy()
    want = _exact(x, gam, nH, alpha, dt)
    # half an ulp of the result, and 2^-34 relative for the arithmetic in two floats; cells
    # outside its range go through FP64, whose cancelling form is good to 2^-53 of 1
    ulp = np.spacing(np.abs(want.astype(np.float32))).astype(np.longdouble)
    err = np.abs(got.astype(np.longdouble) - want)
    bar = 0.5 * ulp + 2.0 ** -34 * np.abs(want) + 2.0 ** -52
    assert (err <= bar).all(), float((err / bar).max())


@pytest.mark.parametrize("n,shift", [(1, 0), (3, 0), (4, 0), (1021, 0), (1024, 1), (4099, 3), (300_000, 2)])
@pytest.mark.parametrize("method", ["a", "b"])
def test_lengths_and_alignments_agree(art, n, shift, method):
    nH, gam, x = _inputs(n + 4, n + shift, 2)

    def run(off):
        t = [torch.zeros(n + 8, device="cuda")[off:off + n] for _ in range(4)]
        for d, v in zip(t, (gam, nH, x)):
            d.copy_(torch.from_numpy(v[:n].copy()))
        art.xn_update(t[0], t[1], t[2], 2e-4, 5.0, nH0_out=t[3], method=method)
        return t[2].cpu(), t[3].cpu()

    (a, b), (c, d) = run(0), run(shift)
    assert torch.equal(a, c) and torch.equal(b, d)
    assert torch.equal(b, a * torch.from_numpy(nH[:n].copy()))
