"""With full multilinear ranks the Tucker projection is the identity: the eigen-solver's
bases at sizes about its warps' pair lists (32 pairs a warp), odd, single and largest."""
import numpy as np
import pytest

from tests.gpu_util import dev, f32, host, maxabs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 2, 3), (3, 1, 2), (31, 33, 5), (63, 64, 4), (65, 66, 3), (128, 130, 2),
                                   (224, 20, 3)])
def test_full_ranks_change_nothing(shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_12879_gb300 import lrstv as L
    Y = f32(np.random.default_rng(sum(shape)).uniform(size=shape))
    got = []
    for ranks in (None, shape):
        with L.Plan(*shape, L.Params.make(shape[0], shape[1], max_iter=3)) as p:
            if ranks:
                p.set_tucker(ranks)
            got.append(host(p.run(dev(Y))[0], shape))
    # a projection multiplies by six n x n bases, each orthonormal to 2^-22 after its
    # Newton-Schulz step, its products rounded to 2^-24: 3 x 6 x (2^-22 + 2^-24) of
    # values near one, and the iteration's own response to them (a factor of two)
    assert maxabs(got[0], got[1]) <= 2 * 18 * (2.0 ** -22 + 2.0 ** -24)
