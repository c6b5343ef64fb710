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
