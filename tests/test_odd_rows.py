"""Epilogue stores of the tensor-core products by row alignment (csrc/umma_epi.cuh):
32-byte, 16-byte and single-float rows, at widths around the 16-column pieces
that odd rows go through, for every forward method on the tensor cores.  The
same pixels of a wider, aligned frame are the reference: each is the same sum
in the same order whatever the store, so the bits agree."""
import numpy as np
import pytest

from gpu_util import to_dev
from workloads import make_cloud

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1002_0916_gb300 as cg
    return cg


@pytest.mark.parametrize("method", ["sep_fp16x3", "sep_bf16", "sep_fp32"])
@pytest.mark.parametrize("Nx,Ny", [(257, 300), (271, 257), (259, 131), (260, 290), (264, 385)])
def test_row_alignments(cg, method, Nx, Ny):
    import torch
    c = make_cloud(50 + Nx, 40, Nx, Ny, integer=False, zlo=0.2, zhi=0.8, lam=532e-9, p=8e-6)
    pts, A, z = to_dev(c)
    h = cg.cgh_create(0)
    try:
        def fwd(nx, out=None):
            return cg.cgh_forward(pts, A, z, c.lam, c.p, nx, Ny, method=method, handle=h, out=out)
        if method != "sep_fp32":
            cg.cgh_set_gemm_plan(h, "pairs", 112)
        wide = fwd(336)[:, :Nx]
        buf = torch.full((Ny * Nx + 9,), 7.0, device="cuda")
        for shift in (0, 1, 4):  # 32-byte, 4-byte and 16-byte aligned outputs
            out = buf[shift:shift + Ny * Nx].view(Ny, Nx)
            got = fwd(Nx, out)
            torch.cuda.synchronize()
            assert torch.equal(got, wide)
            assert torch.all(buf[:shift] == 7.0) and torch.all(buf[shift + Ny * Nx:] == 7.0)
            buf.fill_(7.0)
    finally:
        cg.cgh_destroy(h)
