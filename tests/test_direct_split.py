"""The direct method's split plan (csrc/direct.cu) around whole numbers of
waves of resident CTAs, and its partial tiles where the scratch of
cgh_forward_noalloc has little or no room for them."""
import ctypes

import numpy as np
import pytest

from gpu_util import max_abs, sum_abs_A, to_dev
from workloads import make_cloud

pytestmark = pytest.mark.gpu
# the library's bound for the direct method, max |I - I_ref| / sum |A_j|
TOL = 1e-4


@pytest.fixture(scope="module")
def cg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1002_0916_gb300 as cg
    return cg


@pytest.mark.parametrize("dx", [-1, 0, 1])
@pytest.mark.parametrize("waves", [1, 2])
@pytest.mark.parametrize("shape", [(64, 32, 16, 4, 64, 0, 8, 8), (32, 32, 8, 4, 64, 0, 8, 8),
                                   (32, 32, 2, 2, 64, 0, 1, 0)])
def test_around_whole_waves(cg, oracle_mod, shape, waves, dx):
    """Tile counts of, one below and one above whole waves of two CTAs per SM:
    deterministic, and against the one-CTA-per-tile grid and the oracle."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = waves * 2 * sms + dx
    rows = next(r for r in range(2, tiles + 1) if tiles % r == 0 and tiles // r <= 400)
    Nx, Ny = tiles // rows * shape[0], rows * shape[1]
    c = make_cloud(7 + tiles, 320, Nx, Ny, integer=False, zlo=0.5, zhi=1.5, lam=633e-9, p=6e-6)
    pick = sorted({0, Ny // 2, Ny - 1})
    ref = oracle_mod.forward(c, rows=pick)
    pts, A, z = to_dev(c)
    h = cg.cgh_create(0)

    def fwd(schedule):
        cg.cgh_set_direct_schedule(h, schedule)
        return cg.cgh_forward(pts, A, z, c.lam, c.p, Nx, Ny, method="direct",
                              handle=h).cpu().numpy()
    try:
        cg.cgh_set_direct_tile(h, shape)
        s1, s2, g = fwd("split"), fwd("split"), fwd("grid")
        assert cg.cgh_last_device_status(h) == cg.CGH_OK
        assert np.array_equal(s1, s2)
        # the same terms in another order
        assert max_abs(s1, g) <= 1e-5 * sum_abs_A(c)
        assert max_abs(s1[pick], ref) <= TOL * sum_abs_A(c)
    finally:
        cg.cgh_destroy(h)


@pytest.mark.parametrize("N,Nx,Ny", [
    (512, 1920, 1000),   # 12 MB of rotation tables: little room for partial tiles
    (680, 1024, 1024),   # 11 MB
    (900, 1000, 1072),   # 15 MB: none
])
def test_noalloc_with_little_room(cg, N, Nx, Ny):
    import torch
    c = make_cloud(60 + N, N, Nx, Ny, integer=False, zlo=0.4, zhi=1.4, lam=532e-9, p=8e-6)
    pts, A, z = to_dev(c)
    ref = cg.cgh_forward(pts, A, z, c.lam, c.p, Nx, Ny, method="direct")
    for _ in range(2):
        out = torch.full((Ny, Nx), float("nan"), device="cuda")
        st = cg.lib.cgh_forward_noalloc(
            ctypes.c_void_p(pts.data_ptr()), ctypes.c_void_p(A.data_ptr()),
            ctypes.c_void_p(z.data_ptr()), N, ctypes.c_double(c.lam), ctypes.c_double(c.p), Nx, Ny,
            ctypes.c_void_p(out.data_ptr()),
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert st == cg.CGH_OK
        assert max_abs(out.cpu().numpy(), ref.cpu().numpy()) <= TOL * sum_abs_A(c)
