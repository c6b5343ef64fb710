"""The FP32 separable product on the tensor cores (csrc/sep32.cu) at the edges
of its tiles, K blocks, K slices and amplitude range, against the FP64 oracle.

Bound, per unit of sum|A_j|: each factor of a product carries the error of its
sine or cosine (8.3e-8), of the FP16 split (2^-23) and of the amplitude product
(2^-24), at most 2 sqrt 2 times that over a term; the dropped lo*lo 2^-23; the
four hi*hi steps of a K block drop at most 2^-23 of the block's sum each, times
sqrt 2; each block's FP32 addition rounds by 2^-24.  In all below 2e-6 plus
2^-24 per K block."""
import numpy as np
import pytest

from gpu_util import max_abs, sum_abs_A, to_dev
from workloads import make_cloud

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1002_0916_gb300 as cg
    return cg


@pytest.fixture(scope="module")
def h(cg):
    handle = cg.cgh_create(0)
    yield handle
    cg.cgh_destroy(handle)


def _check(cg, h, oracle_mod, c, scale=1.0):
    import torch
    pts, A, z = to_dev(c)
    I = cg.cgh_forward(pts, A, z, c.lam, c.p, c.Nx, c.Ny, method="sep_fp32", handle=h)
    torch.cuda.synchronize()
    assert cg.cgh_last_device_status(h) == cg.CGH_OK
    got = I.cpu().numpy().astype(np.float64) / scale
    c.A = (c.A.astype(np.float64) / scale)
    tol = (2e-6 + -(-c.N // 32) * 2.0 ** -24) * sum_abs_A(c)
    assert max_abs(got, oracle_mod.forward(c)) <= tol


# one-pixel and one-column tiles, one past each tile width and the 256-row
# tile, an odd width (scalar stores); N around the 32-point K block and, on a
# small frame, long enough for many K slices
@pytest.mark.parametrize("Nx,Ny,N", [
    (1, 1, 1), (16, 256, 31), (112, 257, 32), (113, 256, 33), (129, 300, 64), (161, 40, 65),
    (193, 128, 5), (257, 129, 1000), (515, 258, 300), (40, 30, 4000), (1030, 513, 100)])
def test_edges(cg, h, oracle_mod, Nx, Ny, N):
    c = make_cloud(9 + Nx + N, N, Nx, Ny, integer=bool(N & 1), zlo=0.05, zhi=0.6, lam=532e-9,
                   p=8e-6)
    _check(cg, h, oracle_mod, c)


@pytest.mark.parametrize("scale", [2.0 ** 100, 2.0 ** -90])
def test_amplitude_range(cg, h, oracle_mod, scale):
    """Amplitudes far outside FP16's range, with whole K blocks 2^-20 smaller,
    of zero or of negative amplitude."""
    c = make_cloud(31, 200, 150, 70, integer=False, zlo=0.2, zhi=0.9, lam=633e-9, p=6.4e-6)
    c.A[32:64] *= 2.0 ** -20
    c.A[64:96] = 0.0
    c.A[96:128] *= -1.0
    c.A = (c.A * np.float32(scale)).astype(np.float32)
    _check(cg, h, oracle_mod, c, scale)
