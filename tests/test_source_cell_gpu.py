"""The rate (and force) in the cells of a single source, which the substep size follows: the same
bits in every run, schedule, block size and number of rays per lane."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1711_06277_gb300 import synth

pytestmark = pytest.mark.gpu

N = 24


# the middle of a cell, a place without symmetry, an edge (4 cells) and a corner (8 cells)
@pytest.mark.parametrize("u", [(10.5, 12.5, 11.5), (9.3, 14.71, 10.06), (12.0, 9.5, 12.0), (12.0, 12.0, 12.0)])
@pytest.mark.parametrize("level0", [2, 3, 4, 6])   # 6, 24, 96 and 1536 sums per cell
@pytest.mark.parametrize("force,bins", [(False, 1), (True, 1), (True, 2)])
def test_source_cells_repeat_bit_for_bit(u, level0, force, bins):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art
    rho = torch.from_numpy(synth.lognormal_field(N, 1.0, seed=3).astype(np.float32)).cuda()
    g = art.Grid(rho, 1.0 / N, nH=rho)
    g.add_sources([[x / N for x in u]], [1.0])
    if bins == 2:
        g.set_nonionizing([3.0])
    lo = [int(np.ceil(x)) - 1 for x in u]
    cells = tuple(slice(a, int(x) + 1) for a, x in zip(lo[::-1], u[::-1]))

    def run(**kw):
        o = g.trace(art.Params(level0=level0, sigma_H=6.0, sigma_d=2.0, tau_max=30.0, **kw), force=force)
        both = [o["gamma"][cells]] + ([o["force"][(slice(None),) + cells]] if force else [])
        return torch.cat([t.reshape(-1) for t in both]).cpu().numpy().tobytes()

    want = run()
    for kw in [{}] * 5 + [dict(schedule="plain"), dict(block_threads=64), dict(queue_capacity=4096)]:
        assert run(**kw) == want, kw
    g.close()


def test_substep_size_repeats():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art
    x = torch.full((N, N, N), 1e-4, device="cuda")
    nH = torch.ones_like(x)
    g = art.Grid(x, 1.0 / N)
    g.add_sources([[10.5 / N, 12.5 / N, 11.5 / N]], [1.0])
    p = art.Params(level0=4, sigma_H=100.0 * N)
    got = {float(art.dt_substep(g.trace(p, force=False, stats=False)["gamma"], nH, x, 1.0).cpu()) for _ in range(12)}
    assert len(got) == 1
    g.close()


@pytest.mark.parametrize("level0", [2, 3, 4])
@pytest.mark.parametrize("force", [False, True])
def test_overflowing_rate_is_infinite(level0, force):
    """The rate of the source's cell beyond the largest float: plus infinity, and no NaN."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art
    rho = torch.full((N, N, N), 1e-6, device="cuda")
    g = art.Grid(rho, 1.0)
    g.add_sources([[10.5, 12.5, 11.5]], [2e38 * 12 * 4 ** level0])   # every base ray is a float
    gamma = g.trace(art.Params(level0=level0, sigma_H=1.0), force=force)["gamma"]
    assert float(gamma[11, 12, 10]) == float("inf")
    assert not bool(torch.isnan(gamma).any())
    g.close()
