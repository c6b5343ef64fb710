"""The adjoint over the layouts of dL/dI, chunks of points and strip widths that
its kernels take differently: the same results."""
import numpy as np
import pytest

from gpu_util import to_dev
from test_adjoint_edges import EPS, _reference
from workloads import grad_field, make_cloud

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


def _backward(cg, h, c, Gd, method, n=slice(None)):
    import torch
    pts, A, z = (t[n].contiguous() for t in to_dev(c))
    gp, gA, gz = cg.cgh_backward(pts, A, z, c.lam, c.p, c.Nx, c.Ny, Gd, method=method, handle=h)
    torch.cuda.synchronize()
    assert cg.cgh_last_device_status(h) == cg.CGH_OK
    return [gp[:, 0].cpu().numpy(), gp[:, 1].cpu().numpy(), gA.cpu().numpy(), gz.cpu().numpy()]


# strips (60 x 50) and products (300 x 201), even and odd rows
@pytest.mark.parametrize("method", ["direct", "sep_fp32"])
@pytest.mark.parametrize("Nx,Ny", [(60, 50), (61, 50), (300, 201), (301, 201)])
def test_alignment_of_the_gradient_field(cg, h, method, Nx, Ny):
    """G at each 4-byte offset from a 16-byte boundary: the bits of an aligned
    copy."""
    import torch
    c = make_cloud(3, 200, Nx, Ny, integer=False, zlo=0.3, zhi=0.9, lam=532e-9, p=6.4e-6)
    G = torch.from_numpy(grad_field(4, Nx, Ny)).cuda()
    want = _backward(cg, h, c, G, method)
    for off in (1, 2, 3):
        buf = torch.full((Nx * Ny + 8,), float("nan"), device="cuda")
        Gd = buf[off:off + Nx * Ny].view(Ny, Nx)
        Gd.copy_(G)
        for a, b in zip(_backward(cg, h, c, Gd, method), want):
            assert np.array_equal(a, b)


def test_chunks_of_points(cg, h):
    """32768 columns: the tables of 3968 points fill a chunk.  The points of the
    first chunk have the bits of a call of their own, those of the second agree
    with one to rounding."""
    import torch
    n, N = 3968, 4300
    c = make_cloud(5, N, 32768, 33, integer=False, zlo=0.3, zhi=0.9, lam=532e-9, p=6.4e-6)
    G = torch.from_numpy(grad_field(6, c.Nx, c.Ny)).cuda()
    both = _backward(cg, h, c, G, "sep_fp32")
    for a, b in zip(both, _backward(cg, h, c, G, "sep_fp32", slice(0, n))):
        assert np.array_equal(a[:n], b)
    for a, b in zip(both, _backward(cg, h, c, G, "sep_fp32", slice(n, N))):
        assert np.linalg.norm(a[n:] - b) <= 2 * EPS * np.linalg.norm(b)


def test_strip_widths(cg, h):
    """The direct adjoint just below 2^25 updates (strips of 16 columns) and just
    above (32): the same points agree within both bounds."""
    import torch
    c = make_cloud(7, 1003, 183, 183, integer=False, zlo=0.3, zhi=0.9, lam=532e-9, p=6.4e-6)
    G = grad_field(8, c.Nx, c.Ny)
    Gd = torch.from_numpy(G).cuda()
    assert 183 * 183 * 1000 < 2 ** 25 < 183 * 183 * 1003
    wide, narrow = _backward(cg, h, c, Gd, "direct"), _backward(cg, h, c, Gd, "direct", slice(1000))
    for a, b, bound in zip(wide, narrow, _reference(c, G)[1]):
        assert np.all(np.abs(a[:1000] - b) <= 2 * EPS * bound[:1000])
