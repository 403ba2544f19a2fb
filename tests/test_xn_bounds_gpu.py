"""The neutral-fraction update writes the cells it was given and no others, whatever the length and
alignment of the arrays."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["a", "b"])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 1021, 4096])
def test_neighbours_are_untouched(n, shift, method):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art
    lo = 4 + shift
    gam, nH, xn, out = (torch.full((n + 16,), v, device="cuda") for v in (2.0, 3.0, 0.5, -7.0))
    art.xn_update(gam[lo:lo + n], nH[lo:lo + n], xn[lo:lo + n], 0.1, 0.3, nH0_out=out[lo:lo + n], method=method)
    inside = torch.zeros(n + 16, dtype=torch.bool, device="cuda")
    inside[lo:lo + n] = True
    assert bool((xn[~inside] == 0.5).all()) and bool((out[~inside] == -7.0).all())
    assert bool((gam == 2.0).all()) and bool((nH == 3.0).all())
    assert len(torch.unique(xn[inside])) == 1 and float(xn[lo]) < 0.5   # ionization wins
    assert bool((out[inside] == 3.0 * xn[inside]).all())
