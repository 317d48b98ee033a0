"""The soft threshold's vector form and its remainders: lengths about four, eight
and a block, arrays that start off a 16-byte boundary, in place."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4, 5, 7, 8, 9, 2047, 2048, 2049, 40001])
@pytest.mark.parametrize("off", [0, 1])
def test_lengths_and_alignments(n, off):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_12879_gb300 import lrstv as L
    x = torch.from_numpy(np.random.default_rng(n).standard_normal(n + off).astype(np.float32)).cuda()[off:]
    d = float(np.float32(0.4))
    want = torch.where(x > d, x - d, torch.where(x < -d, x + d, torch.zeros_like(x)))
    y = torch.full((n + off + 3,), 7.0, device="cuda")
    L.lrstv_soft_threshold(x, d, out=y[off:off + n])
    assert torch.equal(y[off:off + n], want) and bool((y[off + n:] == 7).all()) and bool((y[:off] == 7).all())
    L.lrstv_soft_threshold(x, d, out=x)
    assert torch.equal(x, want)
