"""Eq. e:dtss over arrays of every length and alignment: the minimum does not depend on how the
cells are grouped."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,shift", [(1, 0), (3, 0), (1021, 0), (4096, 1), (300_003, 2), (1 << 21, 3)])
def test_dt_is_the_same_for_every_alignment(n, shift):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1711_06277_gb300 import art
    rng = np.random.default_rng(n)
    v = [(10.0 ** rng.uniform(-2, 2, n)).astype(np.float32), (10.0 ** rng.uniform(-1, 3, n)).astype(np.float32),
         rng.random(n).astype(np.float32)]

    def run(off):
        t = [torch.zeros(n + 8, device="cuda")[off:off + n] for _ in v]
        for d, s in zip(t, v):
            d.copy_(torch.from_numpy(s))
        return float(art.dt_substep(*t, 0.02, 0.1).cpu())

    assert run(0) == run(shift)
