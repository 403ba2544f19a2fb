"""Matrices that are no rotations are accepted; whatever they make of the directions, every ray
ends."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1711_06277_gb300 import synth

pytestmark = pytest.mark.gpu

R = np.linalg.qr(np.random.default_rng(7).standard_normal((3, 3)))[0]


@pytest.mark.parametrize("rot", [np.zeros((3, 3)), 1e-9 * R, 0.1 * np.eye(3), 0.3 * R, 0.6 * np.eye(3), 3.0 * R,
                                 np.diag([1.0, 0.0, 0.0]), np.diag([0.2, 0.0, 0.0]), np.diag([1e9, 1.0, 1e-9])])
@pytest.mark.parametrize("sigma", [0.0, 4.0])
def test_every_ray_ends(rot, sigma):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art
    n = 16
    rho = torch.from_numpy(synth.lognormal_field(n, 1.0, seed=5).astype(np.float32)).cuda()
    g = art.Grid(rho, 1.0 / n)
    g.add_sources([[0.5, 0.5, 0.5], [0.3, 0.61, 0.47]], [1.0, 2.0])
    for schedule in ("persistent", "plain"):
        p = art.Params(level0=2, sigma_H=sigma, rot=rot, schedule=schedule, wait_limit_s=5.0)
        st = g.trace(p)["stats"]
        assert st["status"] == 0 and st["destroy"] == st["destroy_expected"]
    assert g.trace_backward(p, torch.ones_like(rho))[2]["status"] == 0
    assert np.isfinite(g.estimate_work(p)).all()
    g.close()
