"""Slices of few columns: one CTA of the FP32 kernels each, in calls, plans and batches alike, on both sides of the line
(48 columns + rows <= 816 up to 256 rows, 12 columns above).

Data and tolerance of the t-SVT are those of the blocked Jacobi's edge tests; a batch's cubes are those of plans of their
own, bit for bit.
"""
import numpy as np
import pytest

from .test_gpu_jacobi_blocked import _data, _slices
from .test_gpu_tsvt_routes import _threshold

pytestmark = pytest.mark.gpu

# (rows, columns) at the line, one column beyond it, and the smallest
SHAPES = [(1, 1, 5), (2, 1, 4), (7, 5, 3), (16, 16, 4), (17, 16, 3), (48, 16, 4), (17, 48, 3), (49, 16, 3), (144, 14, 3),
          (144, 15, 3), (240, 12, 2), (13, 240, 3), (256, 11, 3), (257, 12, 3), (13, 257, 2), (512, 1, 4), (5, 512, 3)]


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2204_12879_gb300 import lrstv
    return lrstv


@pytest.mark.parametrize("kind", ["dense", "graded", "equal"])
@pytest.mark.parametrize("shape", SHAPES)
def test_tsvt_of_few_columns(L, shape, kind):
    import torch
    A = _data(shape, kind, 11 + sum(shape))
    t = _threshold(A)
    want, bound = _slices(A.astype(np.float64), t)
    out, sw = L.lrstv_tsvt(torch.from_numpy(A).cuda(), shape, t, sweeps=True)
    err = np.linalg.norm(out.cpu().numpy().astype(np.float64).reshape(want.shape) - want)
    print(shape, kind, "sweeps", sw, "error", err, "bound", bound)
    assert 0 <= sw < 60 and err <= bound
    # every value cut: no sweep is run
    spec = np.abs(np.fft.fft(A.astype(np.float64), axis=0))
    top = float(np.float32(1.01 * np.sqrt((spec ** 2).sum((1, 2)).max())))
    out, sw = L.lrstv_tsvt(torch.from_numpy(A).cuda(), shape, top, sweeps=True)
    assert sw == 0 and not bool(out.any())


@pytest.mark.parametrize("shape,kernel", [((20, 8, 3), "k_jacobi_pk"), ((48, 16, 3), "k_jacobi_pk"),
                                          ((512, 4, 3), "k_jacobi("), ((80, 16, 3), "k_jacobi_tasks"),
                                          ((300, 13, 3), "k_jacobi_tasks")])
def test_kernel_of_few_columns(L, shape, kernel):
    """The blocked Jacobi's launches took up to 2.1 times as long on slices of few columns."""
    import torch
    A = _data(shape, "dense", 3)
    x, t = torch.from_numpy(A).cuda(), _threshold(A)
    names = []
    for _ in range(3):  # a process's first profile can come back without kernels
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
            L.lrstv_tsvt(x, shape, t)
            torch.cuda.synchronize()
        names = [e.key for e in prof.key_averages() if "jacobi" in e.key]
        if names:
            break
    if not names:
        pytest.skip("the profiler lists no kernels")
    assert all(kernel in n for n in names), names


@pytest.mark.parametrize("mode", ["cold", "warm", "graph"])
def test_batch_equals_plans(L, mode):
    """Groups of few columns (one launch for two cubes), tall ones of few columns and the common launch in one batch."""
    import torch
    shapes = [(20, 8, 5), (40, 33, 6), (20, 8, 5), (300, 9, 3), (300, 9, 3), (5, 7, 4), (270, 20, 3)]
    flags = {"cold": 0, "warm": L.FLAG_WARM_START, "graph": L.FLAG_WARM_START | L.FLAG_GRAPH}[mode]
    prms = [L.Params.make(s[0], s[1], max_iter=12, flags=flags) for s in shapes]
    ys = [torch.rand(int(np.prod(s)), generator=torch.Generator().manual_seed(i)).cuda() for i, s in enumerate(shapes)]
    with L.Batch(shapes, prms) as b:
        X, S = b.run(ys)
        again = b.run(ys, X, S)  # the recorded graph, where there is one
        assert again[0] is X
        torch.cuda.synchronize()
        assert all(b.plan(i).stats().jacobi_unconverged == 0 for i in range(len(shapes)))
    for s, prm, y, x, sp in zip(shapes, prms, ys, X, S):
        with L.Plan(*s, prm) as p:
            want = p.run(y)
        assert torch.equal(x, want[0]) and torch.equal(sp, want[1])
