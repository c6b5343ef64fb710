"""The adjoint over the whole range of magnitudes of dL/dI and of point counts,
against FP64 sums in numpy; bounds as in test_adjoint_edges.py."""
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


def _backward(cg, c, G, method):
    import torch
    h = cg.cgh_create(0)
    try:
        gp, gA, gz = cg.cgh_backward(*to_dev(c), c.lam, c.p, c.Nx, c.Ny, torch.from_numpy(G).cuda(),
                                     method=method, handle=h)
        torch.cuda.synchronize()
        assert cg.cgh_last_device_status(h) == cg.CGH_OK
    finally:
        cg.cgh_destroy(h)
    gp = gp.cpu().numpy().astype(np.float64)
    return [gp[:, 0], gp[:, 1], gA.cpu().numpy(), gz.cpu().numpy()]


# both sides of 2^-100 and 2^-110, the smallest normal and a subnormal FP32
# number (the gradients round to multiples of 2^-149), and large fields
@pytest.mark.parametrize("method", ["sep_fp32", "sep_fp16x3", "direct"])
@pytest.mark.parametrize("scale", [1e-31, 2.0 ** -99, 2.0 ** -105, 2.0 ** -112, 1e-37, 2.0 ** -126,
                                   2.0 ** -135, 2.0 ** 100])
def test_size_of_the_gradient_field(cg, method, scale):
    c = make_cloud(21, 150, 130, 70, integer=False, zlo=0.2, zhi=0.9, lam=532e-9, p=6.4e-6)
    G = (grad_field(23, c.Nx, c.Ny) * scale).astype(np.float32)
    assert np.abs(G).max() > 0
    for v, ref, bound in zip(_backward(cg, c, G, method), *_reference(c, G)):
        assert np.all(np.abs(v - ref) <= EPS * bound + 2.0 ** -149)


# more points than 65535 groups of 128, in strips of 16 columns (1 x 3 pixels)
# and of 32 (5 x 1), and in the separable adjoint two chunks of points
@pytest.mark.parametrize("Nx,Ny", [(1, 3), (5, 1)])
@pytest.mark.parametrize("method", ["direct", "sep_fp32"])
def test_many_points(cg, method, Nx, Ny):
    N = 65535 * 128 + 1000
    c = make_cloud(5, N, Nx, Ny, integer=False, zlo=0.2, zhi=0.9, lam=532e-9, p=6.4e-6)
    G = grad_field(6, Nx, Ny)
    for v, ref, bound in zip(_backward(cg, c, G, method), *_reference(c, G)):
        assert np.all(np.abs(v - ref) <= EPS * bound)


def test_sums_past_the_range_of_fp32(cg):
    """A field with the sign of sin(phi) (x - x_j) of one point.  Partial sums
    that are FP32 numbers but not their total, which 2 P A brings back into range;
    and infinite partial sums: an infinite gradient, not NaN."""
    c = make_cloud(8, 1, 512, 64, integer=False, zlo=0.4, zhi=0.5, lam=532e-9, p=3.74e-6)
    c.A[:] = 0.5
    P = np.pi * c.p * c.p / (c.lam * float(c.z[0]))
    dx, dy = np.arange(512) - float(c.xy[0, 0]), np.arange(64) - float(c.xy[0, 1])
    w = np.sin(P * (dx[None, :] ** 2 + dy[:, None] ** 2)) * dx[None, :]
    top, strip = 2.0 ** 128, np.abs(w).reshape(64, 32, 16).sum((0, 2)).max()
    size = 1.2e33
    assert np.abs(w).sum() * size > 4 * top and strip * size < top
    G = (np.sign(w) * size).astype(np.float32)
    got = _backward(cg, c, G, "direct")
    ref, bound = _reference(c, G)
    for k in (0, 1):
        assert abs(ref[k][0]) < top and abs(got[k][0] - ref[k][0]) <= EPS * bound[k][0]
    # (no column's sum of G sin(phi) is past the range, its product with x - x_j is)
    size = 4e36
    assert 64 * size < top < strip * size
    assert _backward(cg, c, (np.sign(w) * size).astype(np.float32), "direct")[0][0] == np.inf
