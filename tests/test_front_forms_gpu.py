"""Every form of the kernels at the edges of their fronts: with and without a force, one and two
bins, dust and a cutoff, at small capacities and block sizes and with a base front that is walked two
rays per lane (more base rays than the chip has threads)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1711_06277_gb300 import synth
from tests import parity as PA

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def art():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art as A
    return A


def _wide(level0):
    """Sources whose base rays outnumber the threads of a launch (640 per SM), so that the base
    front is walked two rays per lane."""
    threads = 640 * torch.cuda.get_device_properties(0).multi_processor_count
    n = threads // (12 * 4 ** level0) + 2
    assert n * 12 * 4 ** level0 > threads
    return n


def _case(art, shape, nsrc, level0, dust, d_max, bins, seed, **kw):
    nz, ny, nx = shape
    rng = np.random.default_rng(seed)
    rho = (0.2 + rng.random(shape)).astype(np.float32)
    nH = (1.3 * rho).astype(np.float32) if dust else None
    dx = 1.0 / max(shape)
    pos = np.array([nx, ny, nz]) * dx * rng.uniform(0.1, 0.9, (nsrc, 3))
    L = synth.power_law_luminosities(nsrc, seed=seed)
    sd = 1.5 if dust else 0.0
    p = art.Params(tau_max=30.0, sigma_H=3.0, sigma_d=sd, level0=level0, d_max=d_max, **kw)
    g = art.Grid(torch.from_numpy(rho).cuda(), dx, nH=None if nH is None else torch.from_numpy(nH).cuda())
    g.add_sources(pos, L)
    Ln = 2.0 * L[::-1].copy() if bins == 2 else None
    if bins == 2:
        g.set_nonionizing(Ln)
    prob = O.Problem(nH0=rho, pos=pos, L=L, dx=dx, nH=nH, sigma_H=3.0, sigma_d=sd, level0=level0,
                     tau_max=30.0, d_max=d_max, Ln=Ln)
    return g, p, prob, rng


@pytest.mark.parametrize("force", [False, True])
@pytest.mark.parametrize("bins,dust,d_max", [(1, False, 0.0), (1, True, 0.23), (2, True, 0.0), (2, True, 0.23)])
@pytest.mark.parametrize("shape,nsrc,level0,kw", [
    ((20, 24, 18), 3, 1, dict(queue_capacity=4)),
    ((20, 24, 18), 5, 3, dict(queue_capacity=520)),
    ((33, 31, 34), 7, 4, dict(block_threads=96)),
    ((20, 24, 18), 3, 2, dict(schedule="plain", block_threads=64)),
    ((40, 36, 44), None, 4, dict()),
])
def test_trace_forms_match_oracle(art, shape, nsrc, level0, kw, bins, dust, d_max, force):
    g, p, prob, _ = _case(art, shape, nsrc or _wide(level0), level0, dust, d_max, bins, 5, **kw)
    out = g.trace(p, force=force, energy=True)
    st = out["stats"]
    ref = O.trace(prob, nthreads=8, count_hits=True)
    # summation bounds of the cells' deposit counts, as in the other parity tests
    PA.compare_field(out["gamma"].cpu().numpy(), ref.gamma, what="gamma", hits=ref.hits)
    PA.compare_field(out["energy"].cpu().numpy(), ref.energy, what="energy", hits=ref.hits)
    if force and bins == 1:
        chi = prob.nH0.astype(np.float64) * 3.0 + (0.0 if prob.nH is None else prob.nH.astype(np.float64) * 1.5)
        PA.compare_force(out["force"].cpu().numpy(), ref.force, chi * ref.energy, hits=ref.hits)
    elif force:
        # against the largest force: the second bin's share of a cell's bound is not known here
        err = np.abs(out["force"].cpu().numpy() - ref.force).max() / np.abs(ref.force).max()
        assert err <= PA.REL
    assert st["rays_per_level"] == ref.rays_per_level.tolist()
    assert abs(st["crossings"] - ref.crossings) <= 4 * ref.near_tie_rays
    assert st["destroy"] == st["destroy_expected"]
    assert abs(st["L_escaped"] - ref.escaped) <= PA.CONS * ref.L_in
    if bins == 2:
        assert abs(st["Ln_escaped"] - ref.escaped_n) <= PA.CONS * ref.Ln_in
    g.close()


@pytest.mark.parametrize("force,dust,d_max", [(False, False, 0.0), (False, True, 0.0), (True, False, 0.0),
                                              (True, True, 0.23), (False, False, 0.23)])
@pytest.mark.parametrize("level0", [4, 5])
def test_sweep_of_a_wide_base_front_matches_oracle(art, level0, force, dust, d_max):
    shape = (40, 36, 44)
    g, p, prob, rng = _case(art, shape, _wide(level0), level0, dust, d_max, 1, 9)
    w = rng.random(shape).astype(np.float32)
    v = rng.uniform(-1, 1, (3,) + shape).astype(np.float32) if force else None
    grad, dL, st = g.trace_backward(p, torch.from_numpy(w).cuda(),
                                    v=None if v is None else torch.from_numpy(v).cuda())
    rg, rL, _ = O.trace_adjoint(prob, w.astype(np.float64), nthreads=8,
                                v=None if v is None else v.astype(np.float64))
    # as in the other tests of the sweep: relative to the largest gradient, and per source
    assert np.abs(grad.cpu().numpy() - rg).max() / np.abs(rg).max() <= 1e-5
    assert np.abs(dL.cpu().numpy() / rL - 1).max() <= 1e-6
    assert st["destroy"] == st["destroy_expected"]
    g.close()
