"""The adjoint's kernels (csrc/adj32.cu and the direct strips of
csrc/backward.cu) at the edges of their tiles, against FP64 sums in numpy.

Bound: every sum's error is at most EPS times the sum of the absolute values
of its terms, with |x - x_j| enlarged by a tile's 128 columns (the weights are
taken relative to the tile and shifted).  Sines, cosines and the FP16 splits
cost below 1e-6; the FP32 additions 2^-24 for each of a lane's 64 columns and
each of the K blocks or rows of a run (at most 70 and 1100 here, the latter
with the random signs of G: about its root): 1e-5 in all."""
import numpy as np
import pytest

from gpu_util import to_dev
from workloads import grad_field, make_cloud

pytestmark = pytest.mark.gpu
EPS = 1e-5


@pytest.fixture(scope="module")
def cg():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1002_0916_gb300 as cg
    return cg


def _reference(c, G):
    """(gradient, bound on the absolute sum of its terms) per output."""
    xy, A, z = (v.astype(np.float64) for v in (c.xy, c.A, c.z))
    G = G.astype(np.float64)
    P = np.pi * c.p * c.p / (c.lam * z)
    dx = np.arange(c.Nx)[:, None] - xy[:, 0][None, :]
    dy = np.arange(c.Ny)[:, None] - xy[:, 1][None, :]
    ex, ey = (np.exp(1j * np.remainder(P * d * d, 2 * np.pi)) for d in (dx, dy))
    W, Wy = G.T @ ey, G @ ex                     # Nx x N, Ny x N
    phx, phy = ex * W, ey * Wy                   # real: cos, imag: sin of the full phase
    ax, ay = np.abs(G).sum(0)[:, None], np.abs(G).sum(1)[:, None]
    bx, by = np.abs(dx) + 128, np.abs(dy) + 128
    g = [2 * P * A * (phx.imag * dx).sum(0), 2 * P * A * (phy.imag * dy).sum(0),
         phx.real.sum(0), P * A / z * ((phx.imag * dx * dx).sum(0) + (phy.imag * dy * dy).sum(0))]
    b = [2 * P * np.abs(A) * (ax * bx).sum(0), 2 * P * np.abs(A) * (ay * by).sum(0),
         np.full(c.N, ax.sum()),
         P * np.abs(A) / z * ((ax * bx * bx).sum(0) + (ay * by * by).sum(0))]
    return g, b


# one pixel; a row and a column; one past the product's 256-row and column
# tiles, the strips' 16 columns, 32-row stages and 128-point groups; odd and
# unaligned widths; the longer axis either way; a wide frame of two point
# chunks
@pytest.mark.parametrize("method", ["sep_fp32", "direct"])
@pytest.mark.parametrize("Nx,Ny,N", [
    (1, 1, 1), (1, 300, 5), (300, 1, 129), (17, 33, 127), (257, 225, 128), (64, 1100, 130),
    (515, 66, 257), (449, 193, 33), (32768, 3, 4300),
    # strips of 32 columns of the direct adjoint (2^25 updates on)
    (31, 1111, 1000), (33, 1025, 1001), (96, 399, 900)])
def test_edges(cg, method, Nx, Ny, N):
    import torch
    c = make_cloud(3 + Nx + N, N, Nx, Ny, integer=bool(N & 1), zlo=0.2, zhi=0.9, lam=532e-9,
                   p=6.4e-6)
    G = grad_field(17 + N, Nx, Ny, scale=3e4)
    h = cg.cgh_create(0)
    try:
        pts, A, z = to_dev(c)
        gp, gA, gz = cg.cgh_backward(pts, A, z, c.lam, c.p, Nx, Ny, torch.from_numpy(G).cuda(),
                                     method=method, handle=h)
        torch.cuda.synchronize()
        assert cg.cgh_last_device_status(h) == cg.CGH_OK
    finally:
        cg.cgh_destroy(h)
    gp = gp.cpu().numpy().astype(np.float64)
    got = [gp[:, 0], gp[:, 1], gA.cpu().numpy(), gz.cpu().numpy()]
    for v, ref, bound in zip(got, *_reference(c, G)):
        assert np.all(np.abs(v - ref) <= EPS * bound)
