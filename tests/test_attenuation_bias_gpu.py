"""The attenuation factor phi(x) = (1 - e^-x)/x of the forward trace has no bias between 1 and 2."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chi", [1.5, 2.25])
def test_absorbed_photons_equal_those_of_the_reverse_sweep(chi):
    """One cell, 786,432 rays from its middle with x = chi ds. The forward trace's absorbed
    photons (an FP64 ledger of the losses L x phi) against the reverse sweep's (an FP64 sum of
    chi L ds phi, phi chosen by x). A segment's terms carry a few FP32 roundings that differ
    between the two, of either sign: at most 5 units of 2^-24. With at least N / 48 distinct
    rays (the symmetries of the cube) their mean stays below 6 x 5 x 2^-24 / (N / 48)^(1/2)."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art
    level = 8
    n = 12 * 4 ** level
    rho = torch.ones((1, 1, 1), device="cuda")
    g = art.Grid(rho, 1.0)
    g.add_sources([[0.5, 0.5, 0.5]], [0.75])   # L / n and chi are powers of two and short numbers
    p = art.Params(level0=level, level_max=level, sigma_H=chi, tau_max=30.0)
    st = g.trace(p)["stats"]
    dL = float(g.trace_backward(p, torch.ones_like(rho))[1].cpu()[0])
    unit = float(np.float32(1.0 / n)) * n       # the sweep's rays carry 1 / n rounded to FP32
    swept = 0.75 * dL / unit
    assert abs(st["L_absorbed"] / swept - 1.0) < 6 * 5 * 2.0 ** -24 / (n / 48) ** 0.5
    g.close()
