"""The kind of items that an untuned split-FP16 batch takes (csrc/batch.cu)."""
import pytest

from gpu_util import to_dev
from workloads import make_cloud

pytestmark = pytest.mark.gpu


# low frames in many items, in few, tall frames, one long problem beside many
# short ones (by the 76 SM pairs of the GPU)
@pytest.mark.parametrize("sizes,kind", [
    ([(1024, 100, 4000)] * 12, "single"), ([(1024, 100, 4000)] * 8, "pairs"),
    ([(1000, 1024, 500)] * 6, "pairs"), ([(1024, 300, 2000)] * 5, "single"),
    ([(1500, 1500, 3000)] + [(60, 60, 5)] * 300, "pairs"),
    ([(1536, 1280, 3000)] * 2 + [(640, 640, 1200)] * 3, "pairs")])
def test_default_items(sizes, kind):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1002_0916_gb300 as cg
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the counts are those of 152 SMs")
    probs = []
    for i, (Nx, Ny, N) in enumerate(sizes):
        c = make_cloud(7 + i, N, Nx, Ny, integer=False, zlo=0.3, zhi=0.9, lam=532e-9, p=8e-6)
        pts, A, z = to_dev(c)
        probs.append({"points": pts, "A": A, "z": z, "lam": c.lam, "p": c.p, "Nx": Nx, "Ny": Ny,
                      "out": torch.empty((Ny, Nx), device="cuda")})
    h = cg.cgh_create(0)
    try:
        got = {}
        for tiles in ("auto", "pairs", "single"):
            cg.cgh_set_gemm_tiles(h, tiles)
            if tiles == "auto":
                assert cg.cgh_batch_plan(h, probs, "sep_fp16x3")["gemm_tiling"] == kind
            for pr in probs:
                pr["out"].fill_(float("nan"))
            cg.cgh_batch(probs, method="sep_fp16x3", handle=h)
            torch.cuda.synchronize()
            assert cg.cgh_last_device_status(h) == cg.CGH_OK
            got[tiles] = [pr["out"].clone() for pr in probs]
        for a, b, c in zip(got["auto"], got["pairs"], got["single"]):
            assert torch.equal(a, b) and torch.equal(a, c)
    finally:
        cg.cgh_destroy(h)
