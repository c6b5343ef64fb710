"""Columns of the CTA-pair tiles (csrc/umma2.cu): the plan's width narrowed to
equal whole sixteens that fill the waves of SM pairs.  Widths at both ends (32
columns, the plan's), tiles whose last 16 columns follow whole 32-column pieces,
and frames one past a tile.  The one-CTA kernel adds the same products in the
same order, so the bits agree."""
import pytest

from gpu_util import to_dev
from workloads import make_cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["sep_fp16x3", "sep_bf16"])
@pytest.mark.parametrize("Nx,Ny,width", [
    (1, 257, 112), (33, 300, 144), (129, 256, 224), (1300, 1300, 160),  # 32, 32, 32, 112 columns
    (1900, 2300, 256), (1901, 2300, 256), (1793, 2050, 256),            # 240, 240, 240
    (1664, 1664, 224), (2816, 1024, 160),                               # 176, 160
])
def test_equal_one_cta_tiles(method, Nx, Ny, width):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1002_0916_gb300 as cg
    c = make_cloud(31 + Nx, 45, Nx, Ny, integer=False, zlo=0.2, zhi=0.8, lam=532e-9, p=8e-6)
    pts, A, z = to_dev(c)
    h = cg.cgh_create(0)
    try:
        out = {}
        for tiling, w in (("pairs", width), ("single", 128)):
            cg.cgh_set_gemm_plan(h, tiling, w)
            buf = torch.full((Ny * Nx + 8,), 7.0, device="cuda")
            cg.cgh_forward(pts, A, z, c.lam, c.p, Nx, Ny, method=method, handle=h,
                           out=buf[4:-4].view(Ny, Nx))
            torch.cuda.synchronize()
            assert cg.cgh_last_device_status(h) == cg.CGH_OK
            assert torch.all(buf[:4] == 7.0) and torch.all(buf[-4:] == 7.0)
            out[tiling] = buf[4:-4]
        assert torch.equal(out["pairs"], out["single"])
    finally:
        cg.cgh_destroy(h)
