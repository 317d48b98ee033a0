"""lrstv_zsolve on cubes far below one: the split products keep their digits down to where FP32 itself loses them.

The solve is homogeneous and the scales are powers of two, so only what falls below FP32's normal range can change the
relative error: operands' low halves below 2^-126 in tiles whose largest value is at least 2^-95 (2^-31 of it), and results
below 2^-126 (2^-24 of 2^-126 against values of about 2^-115): together under 2e-8 beside the error at scale one.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2204_12879_gb300 import lrstv
    return lrstv


def _error(L, x, shape, mu):
    import torch
    z = L.lrstv_zsolve(torch.from_numpy(x.reshape(-1)).cuda(), shape, mu).double().cpu().numpy().reshape(x.shape)
    P = sum((4 * np.sin(np.pi * np.arange(n) / n) ** 2).reshape([-1 if b == a else 1 for b in range(3)])
            for a, n in enumerate(x.shape))
    want = np.fft.ifftn(np.fft.fftn(x.astype(np.float64)) / (mu * (1 + P))).real
    return np.linalg.norm(z - want) / max(np.linalg.norm(want), 1e-300)


@pytest.mark.parametrize("shape", [(45, 40, 30), (130, 67, 9), (16, 16, 1)])
def test_small_cubes_keep_their_digits(L, shape):
    x = np.random.default_rng(3).standard_normal(shape[::-1]).astype(np.float32)
    mu = float(np.float32(0.7))
    base = _error(L, x, shape, mu)
    for k in (60, 94, 96, 102, 108, 112, 115):
        err = _error(L, np.ldexp(x, -k).astype(np.float32), shape, mu)
        print(shape, "2^-%d" % k, err, "at one", base)
        assert err <= base + 2e-8


def test_one_large_value_among_small_ones(L):
    """Tiles above and below the line in one cube, and tiles of zeros."""
    shape = (140, 70, 6)
    rng = np.random.default_rng(5)
    x = np.zeros(shape[::-1], np.float32)
    x[:3] = np.ldexp(rng.standard_normal((3, 70, 140)), -110)
    x[1, 3, 5] = 1.0
    assert _error(L, x, shape, 1.0) <= 2e-6
    assert _error(L, np.zeros_like(x), shape, 1.0) == 0.0
