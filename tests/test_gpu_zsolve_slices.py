"""The Z-solve's spatial passes treat the spectrum's slices as one tall or one
wide matrix: tiles of 128 rows and 64 columns that begin and end inside slices,
single rows and columns, and few slices, against the oracle's solve."""
import numpy as np
import pytest

from tests.gpu_util import dev, f32, host, maxabs

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 2), (1, 70, 9), (127, 3, 5), (128, 64, 6), (129, 65, 7), (43, 64, 24), (64, 64, 31), (8, 200, 9),
          (200, 9, 2)]


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2204_12879_gb300 import lrstv
    return lrstv


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_tiles_across_slices(L, orc, shape, bf16):
    n1, n2, n3 = shape
    T = f32(np.random.default_rng(n1 + n2).standard_normal(shape))
    w = (1.0, 0.6, 1.4)
    with L.Plan(n1, n2, n3, L.Params.make(n1, n2, w=w, flags=L.FLAG_BF16X3 if bf16 else 0)) as p:
        p.init(dev(np.zeros(shape)))
        p.set("TZ", dev(T))
        p.step_z()
        mu, _ = p.mu
        got = host(p.get("Z"), shape)
        assert p.stats().gemm_errors == 0
    ref = orc.zsolve(T, mu, w)
    # 3xTF32 carries 2^-21 a term, 3xBF16 2^-17, through six unitary passes
    assert maxabs(got, ref) <= (2e-4 if bf16 else 1e-5) * np.abs(ref).max()


@pytest.mark.parametrize("shape", SHAPES + [(145, 145, 66)])
def test_single_operator_error(L, orc, shape):
    """lrstv_zsolve on the tensor cores, its small split products summed first."""
    T = f32(np.random.default_rng(sum(shape)).standard_normal(shape))
    w = (1.0, 0.6, 1.4)
    got = host(L.lrstv_zsolve(dev(T), shape, 0.7, w), shape)
    ref = orc.zsolve(T, 0.7, w)
    # a pass over K terms: the dropped lo*lo and two truncations of each chunk (3 x
    # 2^-23), the sum of K / 8 chunks, rounded tables and results (2^-24 each); two
    # passes a mode, of which each is unitary up to its scale
    u = 2.0 ** -24
    bound = sum(2 * (6 + np.ceil(k / 8) + 2) * u for k in shape)
    err = np.linalg.norm(np.asarray(got, np.float64) - ref) / np.linalg.norm(ref)
    print(shape, "error", err, "bound", bound)
    assert err <= bound
