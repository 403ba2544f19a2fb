"""A front beyond its capacity in the plain schedule: the next level traces the children that
fitted and nothing that an earlier trace left in the buffer."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level0,capacity", [(2, 64), (2, 4), (4, 100), (4, 6000)])
@pytest.mark.parametrize("bins", [1, 2])
def test_overflowing_front_holds_no_earlier_rays(level0, capacity, bins):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import _lib as C
    from paper_1711_06277_gb300 import art
    n = 64
    rho = torch.ones((n, n, n), device="cuda")
    g = art.Grid(rho, 1.0 / n, nH=rho)
    kw = dict(level0=level0, sigma_H=8.0, sigma_d=2.0, schedule="plain")

    def source(lum):
        g.clear_sources()
        g.add_sources([[0.5, 0.5, 0.5]], [lum])
        if bins == 2:
            g.set_nonionizing([lum])

    source(1e6)
    g.trace(art.Params(**kw))                      # fills the fronts with bright rays
    source(1.0)
    out = {"gamma": torch.empty_like(rho), "force": torch.empty((3, n, n, n), device="cuda")}
    with pytest.raises(C.ArtError) as e:
        g.trace(art.Params(queue_capacity=capacity, **kw), out=out)
    assert e.value.status == C.ART_EQUEUE_OVERFLOW
    # FP32 sums of at most the source's photons (hydrogen absorbs 8/10 of them)
    absorbed = float(out["gamma"].double().sum()) / n ** 3
    assert absorbed <= 0.8 * (1 + 1e-5)
    # the children that fitted were traced: rates beyond the split radius of the base level
    c = torch.arange(n, device="cuda") + 0.5 - n / 2
    r = torch.sqrt(c[:, None, None] ** 2 + c[None, :, None] ** 2 + c[None, None, :] ** 2)
    assert bool((out["gamma"][r > np.sqrt(3 / (4 * np.pi)) * 2 ** level0 + 1.8] > 0).any())
    assert g.trace(art.Params(**kw))["stats"]["status"] == 0
    g.close()
