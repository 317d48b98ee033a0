"""What the blocked Jacobi leaves as it is: a slice that needs no rotation keeps its FP32 values (its 22-bit halves would
end 2^-39 below the slice's norm), and the threshold is applied with the same sums whichever kernel applies it.
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


@pytest.mark.parametrize("shape", [(1, 1, 1), (16, 15, 1), (40, 33, 1), (225, 40, 1), (300, 31, 1)])
def test_orthogonal_columns_keep_their_digits(L, shape):
    """Diagonal slices with entries over fifteen decades: the t-SVT with t = 0 is the slice itself.  Two DFTs of one band and
    one product with the identity: a split to 22 bits each, 4 times 2^-21 of each entry together."""
    import torch
    n1, n2, _ = shape
    d = np.logspace(0, -15, min(n1, n2)).astype(np.float32)
    A = np.zeros((n2, n1), np.float32)
    A[np.arange(d.size), np.arange(d.size)] = d
    out, sw = L.lrstv_tsvt(torch.from_numpy(A).cuda(), shape, 0.0, sweeps=True)
    got = out.cpu().numpy().reshape(n2, n1)
    assert sw == 1
    assert np.all(np.abs(got - A) <= 4 * 2.0 ** -21 * np.abs(A))


@pytest.mark.parametrize("shape", [(40, 33, 6), (64, 65, 5), (241, 35, 3), (258, 20, 3)])
def test_threshold_in_the_jacobi_or_after_it(L, shape):
    """A cold E-step thresholds V where the sweeps end; a warm-startable plan's keeps V and scales it in a kernel of its own:
    the same bits."""
    import torch
    N = int(np.prod(shape))
    g = torch.Generator().manual_seed(N)
    y, F = torch.rand(N, generator=g).cuda(), torch.randn(3 * N, generator=g).cuda()
    got, sweeps = [], []
    for flags in (0, L.FLAG_WARM_START):
        # alpha / mu0 = 0.4 of the RMS column norm of a slice of unit noise
        alpha = 0.4 * float(np.sqrt(shape[2] * max(shape[:2]))) * 1e-2
        with L.Plan(*shape, L.Params.make(shape[0], shape[1], alpha=alpha, flags=flags)) as pl:
            pl.init(y)
            pl.set("F", F)
            pl.step_e()
            got.append(pl.get("E"))
            sweeps.append(pl.stats().jacobi_max_sweeps)
    assert sweeps[0] == sweeps[1] > 1
    assert float(got[0].norm()) > 0
    assert torch.equal(got[0], got[1])
