"""The t-SVT near the ends of FP32's range.

Tolerance.  As in the edge tests of the blocked Jacobi: a pair left alone moves the SVT by at most t tol in its plane, so
a slice by at most t tol nc / sqrt(2), and rounding adds 2e-6 of the slice's norm.
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


@pytest.mark.parametrize("fro", [1.70e19, 1.74e19, 1.80e19, 1.84e19])
@pytest.mark.parametrize("shape", [(20, 18, 1), (64, 40, 1), (300, 24, 1)])
def test_slices_whose_squared_norm_just_fits(L, shape, fro):
    """||W||_F^2 between 2.9e38 and FP32's largest value, 3.40e38 = (1.845e19)^2."""
    import torch
    n1, n2, _ = shape
    rng = np.random.default_rng(n1)
    A = rng.standard_normal((n2, n1)) + 1.0
    A = np.asarray(A * (fro / np.linalg.norm(A)), np.float32)
    t = float(np.float32(0.3 * fro / np.sqrt(min(n1, n2))))
    U, s, Vh = np.linalg.svd(A.astype(np.float64), full_matrices=False)
    want = (U * np.maximum(s - t, 0.0)) @ Vh
    out, sw = L.lrstv_tsvt(torch.from_numpy(A).cuda(), shape, t, sweeps=True)
    got = out.cpu().numpy().astype(np.float64).reshape(want.shape)
    tol = 8 * np.sqrt(max(n1, n2)) * 2.0 ** -24 / 0.3
    bound = t * tol * min(n1, n2) / np.sqrt(2) + 2e-6 * fro
    print(shape, fro, "sweeps", sw, "error", np.linalg.norm(got - want), "bound", bound)
    assert 0 < sw < 60
    assert np.linalg.norm(got - want) <= bound
