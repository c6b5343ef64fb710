"""The separable methods' adjoint on both sides of the lines that choose how it
runs, against FP64 sums in numpy; bounds as in test_adjoint_edges.py."""
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


def _check(cg, Nx, Ny, N):
    import torch
    c = make_cloud(40 + Nx + N, N, Nx, Ny, integer=bool(N & 1), zlo=0.2, zhi=0.9, lam=532e-9,
                   p=6.4e-6)
    G = grad_field(41 + N, Nx, Ny, scale=3.0)
    h = cg.cgh_create(0)
    out = []
    try:
        for method in ("sep_fp32", "sep_fp16x3"):
            gp, gA, gz = cg.cgh_backward(*to_dev(c), c.lam, c.p, Nx, Ny,
                                         torch.from_numpy(G).cuda(), method=method, handle=h)
            torch.cuda.synchronize()
            assert cg.cgh_last_device_status(h) == cg.CGH_OK
            gp = gp.cpu().numpy()
            out.append([gp[:, 0], gp[:, 1], gA.cpu().numpy(), gz.cpu().numpy()])
    finally:
        cg.cgh_destroy(h)
    for u, v in zip(*out):
        assert np.array_equal(u, v)
    for v, ref, bound in zip(out[0], *_reference(c, G)):
        assert np.all(np.abs(v - ref) <= EPS * bound)


# the K of the longer axis cut into slices, along either axis
@pytest.mark.parametrize("Nx,Ny,N", [(32768, 33, 129), (33, 32768, 200), (8192, 50, 1000)])
def test_slices_of_a_long_axis(cg, Nx, Ny, N):
    _check(cg, Nx, Ny, N)


# the strips of the direct adjoint (small and low frames) and the products, each
# side of every line between them, and the products at the edges of their tiles
@pytest.mark.parametrize("Nx,Ny,N", [
    (1, 1, 1), (91, 90, 5000), (128, 64, 5000), (129, 64, 3000), (129, 65, 3000), (256, 128, 366),
    (256, 128, 367), (257, 128, 64), (512, 64, 762), (512, 64, 763), (2000, 20, 256),
    (2000, 20, 255), (2000, 21, 256), (8192, 1, 7), (8193, 1, 255), (7, 1024, 64), (7, 1025, 64),
    (1, 1100, 1), (3, 1500, 127), (17, 1030, 128), (40, 1025, 257), (32768, 2, 100)])
def test_strips_and_products(cg, Nx, Ny, N):
    _check(cg, Nx, Ny, N)


def test_accuracy_of_a_small_frame(cg):
    """Phases of a small part of a turn, where sin(phi) is small and needs a
    relative error: every gradient within 1e-6 of FP64 (the strips with the
    hardware's sines are 2e-6 off here)."""
    import torch
    for seed in range(3):
        c = make_cloud(seed, 1000, 16, 16, integer=False, zlo=0.5, zhi=1.5, lam=532e-9, p=6.4e-6)
        G = grad_field(seed + 9, 16, 16)
        gp, gA, gz = cg.cgh_backward(*to_dev(c), c.lam, c.p, 16, 16, torch.from_numpy(G).cuda(),
                                     method="sep_fp32")
        got = [gp[:, 0], gp[:, 1], gA, gz]
        for v, ref in zip(got, _reference(c, G)[0]):
            v = v.cpu().numpy().astype(np.float64)
            assert np.linalg.norm(v - ref) <= 1e-6 * np.linalg.norm(ref)


def test_scratch_of_a_low_frame_and_many_points(cg):
    """The strips' partial sums would take 5 GiB here, the products work in chunks
    of 1 GiB; 40 points against FP64."""
    import torch
    c = make_cloud(77, 1000000, 8192, 1, integer=False, zlo=0.2, zhi=0.9, lam=532e-9, p=6.4e-6)
    G = grad_field(78, 8192, 1)
    h = cg.cgh_create(0)
    try:
        args = (*to_dev(c), c.lam, c.p, c.Nx, c.Ny, torch.from_numpy(G).cuda())
        outs = [torch.empty((c.N, 5), device="cuda")]  # (the outputs' memory, held before)
        del outs
        free = torch.cuda.mem_get_info()[0]
        gp, gA, gz = cg.cgh_backward(*args, method="sep_fp32", handle=h)
        torch.cuda.synchronize()
        assert cg.cgh_last_device_status(h) == cg.CGH_OK
        assert free - torch.cuda.mem_get_info()[0] < 2.5 * 2 ** 30
    finally:
        cg.cgh_destroy(h)
    some = np.linspace(0, c.N - 1, 40).astype(int)
    c.xy, c.A, c.z = c.xy[some], c.A[some], c.z[some]
    gp = gp.cpu().numpy()[some]
    got = [gp[:, 0], gp[:, 1], gA.cpu().numpy()[some], gz.cpu().numpy()[some]]
    for v, ref, bound in zip(got, *_reference(c, G)):
        assert np.all(np.abs(v - ref) <= EPS * bound)
