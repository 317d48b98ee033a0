"""The blocked Jacobi of the t-SVT at the edges of its tiles, against an FP64 SVD of every Fourier slice.

Columns are taken in panels of 16 and rows in groups of 16 and tiles of 128, so the sides straddle these; odd and even
panel counts, a single panel, wide and tall slices.  Both schedules run (a workspace with the task queue's scratch, and
the call without any).

Tolerance.  A column pair is left alone at a relative inner product of tol = 8 sqrt(nr) 2^-24 max(1, rms / t), which
moves the SVT by at most t tol in the plane of the pair; over the nc^2 / 2 pairs of a slice that is at most
t tol nc / sqrt(2) in the Frobenius norm.  The rounding of the products (22-bit halves, some 10 sweeps) and of the DFTs
adds 2e-6 of the slice's own norm.  The inverse DFT carries the slices' norms over (Parseval, 1 / n3).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 3), (2, 1, 4), (2, 2, 3), (15, 15, 3), (16, 16, 3), (17, 16, 4), (17, 17, 3), (31, 33, 3), (32, 32, 3),
          (33, 32, 2), (47, 49, 3), (64, 48, 3), (65, 64, 2), (127, 20, 3), (128, 33, 2), (129, 40, 2), (145, 97, 2),
          (200, 208, 1), (255, 17, 2), (256, 64, 2), (257, 33, 2), (300, 40, 1), (512, 31, 2)]


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2204_12879_gb300 import lrstv
    return lrstv


def _slices(A, t):
    """The t-SVT of A (n3, n2, n1) in FP64 and the bound above on its error's 2-norm."""
    spec = np.fft.fft(A, axis=0)
    nr, nc = max(A.shape[1:]), min(A.shape[1:])
    out, bound2 = np.empty_like(spec), 0.0
    for k, M in enumerate(spec):
        U, s, Vh = np.linalg.svd(M, full_matrices=False)
        out[k] = (U * np.maximum(s - t, 0.0)) @ Vh
        fro = np.linalg.norm(M)
        tol = 8 * np.sqrt(nr) * 2.0 ** -24 * max(1.0, fro / np.sqrt(nc) / t)
        bound2 += (t * tol * nc / np.sqrt(2) + 2e-6 * fro) ** 2
    return np.fft.ifft(out, axis=0).real, np.sqrt(bound2 / A.shape[0])


def _data(shape, kind, seed):
    rng = np.random.default_rng(seed)
    n1, n2, n3 = shape
    A = rng.standard_normal((n3, n2, n1))
    if kind == "graded":  # column norms over five decades
        A *= np.logspace(0, -5, n1)[None, None, :]
    elif kind == "equal":  # equal columns: every pair of them is parallel
        A = np.repeat(A[:, :, :1], n1, axis=2)
    return np.asarray(A, np.float32)


@pytest.mark.parametrize("kind", ["dense", "graded", "equal"])
@pytest.mark.parametrize("shape", SHAPES)
def test_tsvt_edges(L, shape, kind):
    import torch
    A = _data(shape, kind, sum(shape))
    spec = np.abs(np.fft.fft(A.astype(np.float64), axis=0))
    t = float(np.float32(0.3 * np.sqrt((spec ** 2).sum() / (shape[2] * min(shape[0], shape[1])))))
    want, bound = _slices(A.astype(np.float64), t)
    x = torch.from_numpy(A).cuda()
    out, sw = L.lrstv_tsvt(x, shape, t, sweeps=True)
    alone = torch.empty_like(out)
    L.lrstv_tsvt_noalloc(x, shape, t, alone)
    assert 0 <= sw < 60
    for got in (out, alone):
        err = np.linalg.norm(got.cpu().numpy().astype(np.float64).reshape(want.shape) - want)
        print(shape, kind, "sweeps", sw, "error", err, "bound", bound)
        assert err <= bound


def test_slices_without_a_finite_norm_run_no_rotation(L):
    """Values whose squares overflow FP32: the slices end without a sweep's rotations and stay finite."""
    import torch
    shape = (20, 18, 1)
    A = np.full((1, 18, 20), 1e20, np.float32)
    out, sw = L.lrstv_tsvt(torch.from_numpy(A).cuda(), shape, 1.0, sweeps=True)
    assert sw == 1 and bool(torch.isfinite(out).all())
    bad = A.copy()
    bad[0, 3, 4] = np.nan
    out, sw = L.lrstv_tsvt(torch.from_numpy(bad).cuda(), shape, 1.0, sweeps=True)
    assert sw == 1 and bool(torch.isnan(out).any())


def test_schedule_flags_change_nothing(L):
    import torch
    shape = (70, 65, 9)
    y = torch.from_numpy(_data(shape, "dense", 5)).cuda()
    got = []
    for extra in (0, L.FLAG_JACOBI_PER_SLICE, L.FLAG_JACOBI_PANEL16):
        with L.Plan(*shape, L.Params.make(70, 65, max_iter=8, flags=L.FLAG_WARM_START | extra)) as p:
            got.append(p.run(y)[0])
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])
