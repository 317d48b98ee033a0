"""The plans' split products are as accurate as FP32 ones: a Z-solve on the tensor cores (3xTF32) is no further from FP64
than the same solve with FP32 FMAs.  (Sums that take the small split products after the large ones are truncated six
times a chunk instead of twice, and were further off on small cubes.)
"""
import numpy as np
import pytest

from synthetic import hsi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2204_12879_gb300 import lrstv
    return lrstv


@pytest.mark.parametrize("shape", [(45, 74, 20), (43, 97, 8), (101, 55, 38)])
def test_z_step_no_further_off_than_fp32(L, shape):
    import torch
    _, noisy = hsi.make_cube(hsi.Recipe(*shape, 6, 40, (0.1, 0.2), 0.2), 11)
    T = torch.from_numpy(hsi.flat(noisy)).cuda()
    x = T.double().cpu().numpy().reshape(shape[::-1])
    mu = 0.7
    P = sum((4 * np.sin(np.pi * np.arange(n) / n) ** 2).reshape([-1 if b == a else 1 for b in range(3)])
            for a, n in enumerate(x.shape))
    want = np.fft.ifftn(np.fft.fftn(x) / (mu * (1 + P))).real
    err = {}
    for name, flags in (("tf32", 0), ("fp32", L.FLAG_SIMT_GEMM)):
        with L.Plan(*shape, L.Params.make(shape[0], shape[1], flags=flags)) as pl:
            pl.set("TZ", T)
            pl.set_mu(mu, 0)
            pl.step_z()
            z = pl.get("Z").double().cpu().numpy().reshape(want.shape)
        err[name] = np.linalg.norm(z - want) / np.linalg.norm(want)
    print(shape, err)
    assert err["tf32"] <= err["fp32"]
