"""Column tiles of the batch's CTA-pair items (csrc/umma2.cu, csrc/batch.cu):
frames around whole tiles of 128 columns and whole thirty-twos, 1 to 3 rounds
of items over the SM pairs.  One-CTA items add the same products in the same
order, so the bits agree."""
import pytest

from gpu_util import to_dev
from workloads import make_cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths", [
    (1, 31, 32, 33, 96, 127, 128, 129), (130, 160, 161, 255, 256, 257, 289, 300), (1000, 2047)])
def test_pair_items_equal_one_cta_items(widths):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1002_0916_gb300 as cg
    probs = []
    for i, Nx in enumerate(widths):
        c = make_cloud(70 + Nx, 20 + 37 * i, Nx, 1500 if Nx > 900 else 90 + 83 * i, integer=False,
                       zlo=0.3, zhi=0.9, lam=532e-9, p=8e-6)
        pts, A, z = to_dev(c)
        probs.append({"points": pts, "A": A, "z": z, "lam": c.lam, "p": c.p, "Nx": c.Nx,
                      "Ny": c.Ny, "buf": torch.full((c.Ny * c.Nx + 8,), 7.0, device="cuda")})
        probs[-1]["out"] = probs[-1]["buf"][4:-4].view(c.Ny, c.Nx)
    h = cg.cgh_create(0)
    try:
        got = {}
        for tiles in ("pairs", "single"):
            cg.cgh_set_gemm_tiles(h, tiles)
            for pr in probs:
                pr["buf"].fill_(7.0)
            cg.cgh_batch(probs, method="sep_fp16x3", handle=h)
            torch.cuda.synchronize()
            assert cg.cgh_last_device_status(h) == cg.CGH_OK
            assert all(torch.all(pr["buf"][:4] == 7.0) and torch.all(pr["buf"][-4:] == 7.0)
                       for pr in probs)
            got[tiles] = [pr["out"].clone() for pr in probs]
        for Nx, a, b in zip(widths, got["pairs"], got["single"]):
            assert torch.equal(a, b), Nx
    finally:
        cg.cgh_destroy(h)
