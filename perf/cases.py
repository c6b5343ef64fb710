"""The performance cases of the point-source Fresnel hologram library: the
calls its users make, over the sizes they make them at.

Each case is one pass through the public entry points of
``paper_1002_0916_gb300``: a hologram (``cgh_forward``), a hologram into host
memory (``cgh_forward_host``), a step of fitting a point cloud to a target
hologram (``CGHFunction`` forward, squared loss, adjoint), or many uneven
holograms in one call (``cgh_batch``).  The point clouds follow the recipe of
the repository's workloads: x, y uniform over the frame (integer or continuous
pixel coordinates), z and A uniform, visible wavelengths, micrometre pitches.
Nothing is tuned for a size beforehand: the calls take the library's defaults.

``exact`` is Eq. 1 (and its gradients) in FP64 with plain torch operations.
"""
import math

import numpy as np
import torch

import paper_1002_0916_gb300 as cg

METHOD_NAMES = ("direct", "sep_fp32", "sep_fp16x3", "sep_fp16", "sep_bf16")
WAVELENGTHS = (633e-9, 532e-9, 473e-9)
BATCH_SIDES = tuple(range(512, 2049, 128))
MOST_UPDATES = 3840 * 2160 * 16384  # point-pixel updates of the largest single hologram


def _forward(name, method, nx, ny, n, integer, zlo, zhi, lam, pitch):
    return {"name": name, "kind": "forward", "method": method, "nx": nx, "ny": ny, "n": n,
            "integer": integer, "zlo": zlo, "zhi": zhi, "lam": lam, "pitch": pitch}


def listed():
    cases = [
        # One small zone-plate frame, as in an interactive preview: launches and
        # latency are all of it.
        _forward("direct_256x256_n64", "direct", 256, 256, 64, True, 0.5, 1.0, 532e-9, 8e-6),
        # The paper's Table 1 frame with the default method: one video frame for a
        # spatial light modulator.
        _forward("direct_1920x1024_n1024", "direct", 1920, 1024, 1024, True, 0.5, 1.5,
                 633e-9, 6.4e-6),
        # A 4K frame of a dense object with the default method: the largest single
        # hologram.
        _forward("direct_3840x2160_n16384", "direct", 3840, 2160, 16384, False, 0.3, 2.0,
                 532e-9, 3.74e-6),
        # The last row of the paper's Table 1 by the FP32 separable method.
        _forward("sep_fp32_1920x1024_n3584", "sep_fp32", 1920, 1024, 3584, True, 0.5, 1.5,
                 633e-9, 6.4e-6),
        # The same video frame by the split tensor-core method (a display loop that
        # stays on the GPU).
        _forward("sep_fp16x3_1920x1024_n1024", "sep_fp16x3", 1920, 1024, 1024, True, 0.5, 1.5,
                 633e-9, 6.4e-6),
        # A 4K frame of a dense object at single-pass precision: previews of large
        # scenes.
        _forward("sep_bf16_3840x2160_n16384", "sep_bf16", 3840, 2160, 16384, False, 0.3, 2.0,
                 532e-9, 3.74e-6),
        # A hologram from pinned host buffers into pinned host memory at a panel
        # size that no tile divides (a host program without device code of its own).
        dict(_forward("host_sep_fp16x3_1366x768_n777", "sep_fp16x3", 1366, 768, 777, False,
                      0.5, 1.5, 532e-9, 6.4e-6), kind="host"),
    ]
    # Fitting a cloud to a target hologram: forward, squared loss and the
    # gradients with respect to every point's position, amplitude and depth, at
    # full HD with the default methods, ...
    cases.append(dict(_forward("fit_direct_1920x1080_n4096", "direct", 1920, 1080, 4096, False,
                               0.5, 1.5, 532e-9, 6.4e-6), kind="fit"))
    # ... a cropped, odd-sized region in FP32 separable form, ...
    cases.append(dict(_forward("fit_sep_fp32_1023x767_n1999", "sep_fp32", 1023, 767, 1999, False,
                               0.5, 1.5, 532e-9, 6.4e-6), kind="fit"))
    # ... and full HD on the tensor cores.
    cases.append(dict(_forward("fit_sep_fp16x3_1920x1080_n4096", "sep_fp16x3", 1920, 1080, 4096,
                               False, 0.5, 1.5, 532e-9, 6.4e-6), kind="fit"))
    # A queue of uneven holograms (sizes, point counts, colours) in one call: a
    # small queue in FP32, and a rendering server's on the tensor cores.
    cases.append({"name": "batch_direct_16", "kind": "batch", "method": "direct", "count": 16,
                  "sizes": 0, "zlo": 0.5, "zhi": 1.5, "pitch": 8e-6})
    cases.append({"name": "batch_sep_fp16x3_64", "kind": "batch", "method": "sep_fp16x3",
                  "count": 64, "sizes": 0, "zlo": 0.5, "zhi": 1.5, "pitch": 8e-6})
    return cases


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any of the calls, frames from 128 x 128 to
    3840 x 2160 (odd sides included), 16 to 16384 points."""
    kind = rng.choice(("forward", "forward", "forward", "host", "fit", "fit", "batch"))
    optics = {"zlo": rng.choice((0.3, 0.5)), "zhi": rng.choice((1.0, 1.5, 2.0)),
              "pitch": rng.choice((3.74e-6, 6.4e-6, 8e-6))}
    if kind == "batch":
        return {"kind": "batch", "method": rng.choice(("direct", "sep_fp16x3")),
                "count": rng.randint(2, 16), "sizes": rng.randint(1, 10 ** 6), **optics}
    nx, ny = _log_uniform(rng, 128, 3840), _log_uniform(rng, 128, 2160)
    if rng.random() < 0.5:  # a panel's sides: multiples of 8
        nx, ny = (nx + 7) // 8 * 8, (ny + 7) // 8 * 8
    most = MOST_UPDATES // (4 if kind == "fit" else 1)
    n = min(_log_uniform(rng, 16, 16384), most // (nx * ny))
    method = rng.choice(METHOD_NAMES[:3] if kind == "fit" else METHOD_NAMES)
    return {"kind": kind, "method": method, "nx": nx, "ny": ny, "n": n,
            "integer": rng.random() < 0.5, "lam": rng.choice(WAVELENGTHS), **optics}


# ------------------------------------------------------------------ inputs
def _cloud(rng, n, nx, ny, integer, zlo, zhi):
    """(points, A, z) of one cloud on the host, float32."""
    if integer:
        x, y = rng.integers(0, nx, n), rng.integers(0, ny, n)
    else:
        x, y = rng.uniform(0, nx, n), rng.uniform(0, ny, n)
    z, a = rng.uniform(zlo, zhi, n), rng.uniform(0.0, 1.0, n)
    xy = np.stack([x, y], axis=1).astype(np.float32)
    return tuple(torch.from_numpy(np.ascontiguousarray(v, dtype=np.float32)) for v in (xy, a, z))


def _sizes(case):
    """Nx, Ny, N and wavelength of every problem of a batch: part of the case."""
    rng = np.random.default_rng(case["sizes"])
    return [(int(rng.choice(BATCH_SIDES)), int(rng.choice(BATCH_SIDES)),
             int(rng.integers(100, 8193)), WAVELENGTHS[int(rng.integers(0, 3))])
            for _ in range(case["count"])]


def _problems(case, seed):
    rng = np.random.default_rng(seed)
    out = []
    for nx, ny, n, lam in _sizes(case):
        pts, a, z = (t.cuda() for t in _cloud(rng, n, nx, ny, True, case["zlo"], case["zhi"]))
        out.append({"points": pts, "A": a, "z": z, "lam": lam, "p": case["pitch"],
                    "Nx": nx, "Ny": ny})
    return out


def _single(case, seed):
    rng = np.random.default_rng(seed)
    return _cloud(rng, case["n"], case["nx"], case["ny"], case["integer"], case["zlo"],
                  case["zhi"])


def _target(case, seed):
    """The target hologram of a fit: that of an independent cloud."""
    rng = np.random.default_rng([seed, 1])
    pts, a, z = (t.cuda() for t in _cloud(rng, case["n"], case["nx"], case["ny"],
                                          case["integer"], case["zlo"], case["zhi"]))
    return _hologram64(pts, a, z, case["lam"], case["pitch"], case["nx"], case["ny"]).float()


def prepare(case, seed):
    if case["kind"] == "batch":
        problems = _problems(case, seed)
        for pr in problems:
            pr["out"] = torch.empty((pr["Ny"], pr["Nx"]), dtype=torch.float32, device="cuda")
        return case, problems
    cloud = _single(case, seed)
    if case["kind"] == "host":
        pinned = [t.pin_memory() for t in cloud]
        out = torch.empty((case["ny"], case["nx"]), dtype=torch.float32).pin_memory()
        return case, pinned + [out, cg.default_handle()]
    state = [t.cuda() for t in cloud]
    if case["kind"] == "fit":
        for t in state:
            t.requires_grad_(True)
        state.append(_target(case, seed))
    return case, state


def run(state):
    case, data = state
    if case["kind"] == "batch":
        cg.cgh_batch(data, method=case["method"])
        return [pr["out"] for pr in data]
    args = (case["lam"], case["pitch"], case["nx"], case["ny"])
    if case["kind"] == "host":
        points, a, z, out, handle = data
        return cg.cgh_forward_host(points, a, z, *args, out=out, method=case["method"],
                                   handle=handle)
    if case["kind"] == "fit":
        points, a, z, target = data
        image = cg.CGHFunction.apply(points, a, z, *args, case["method"], case["method"])
        loss = (image - target).square().sum()
        grads = torch.autograd.grad(loss, (points, a, z))
        return [image.detach(), loss.detach(), *grads]
    points, a, z = data
    return cg.cgh_forward(points, a, z, *args, method=case["method"])


# -------------------------------------------------------------------- work
def work(case):
    """Bytes: the cloud (16 per point), the hologram written, for a fit also the
    target read and the three gradients written.  Operations: per point-pixel
    update two multiply-adds of the separable sum of Eq. 1, and for a fit the two
    transforms of dL/dI (four multiply-adds)."""
    if case["kind"] == "batch":
        sizes = _sizes(case)
        return {"bytes": sum(16 * n + 4 * nx * ny for nx, ny, n, _ in sizes),
                "flops": sum(4 * n * nx * ny for nx, ny, n, _ in sizes)}
    n, px = case["n"], case["nx"] * case["ny"]
    if case["kind"] == "fit":
        return {"bytes": 32 * n + 8 * px, "flops": 12 * n * px}
    return {"bytes": 16 * n + 4 * px, "flops": 4 * n * px}


# ------------------------------------------------------------------- exact
def _tables64(points, z, lam, pitch, count, axis):
    """cos and sin of P_j (u - u_j)^2 for u = 0 .. count - 1: count x N, FP64."""
    u = torch.arange(count, dtype=torch.float64, device=points.device)[:, None]
    d = u - points[:, axis].double()[None, :]
    turns = (pitch * pitch / (2.0 * lam)) / z.double()[None, :] * d * d
    turns -= torch.round(turns)
    angle = turns.mul_(2.0 * math.pi)
    return torch.cos(angle), torch.sin(angle)


def _hologram64(points, a, z, lam, pitch, nx, ny):
    cx, sx = _tables64(points, z, lam, pitch, nx, 0)
    cy, sy = _tables64(points, z, lam, pitch, ny, 1)
    ad = a.double()
    return (cy * ad) @ cx.T - (sy * ad) @ sx.T


def _gradients64(points, a, z, lam, pitch, nx, ny, g):
    ad, zd = a.double(), z.double()
    p = math.pi * pitch * pitch / (lam * zd)
    tables = [_tables64(points, z, lam, pitch, n, axis) for axis, n in ((0, nx), (1, ny))]
    sums = []
    for axis, n, field in ((0, nx, g), (1, ny, g.T)):
        (c, s), (co, so) = tables[axis], tables[1 - axis]
        wc, ws = field.T @ co, field.T @ so  # n x N
        d = torch.arange(n, dtype=torch.float64, device=points.device)[:, None] \
            - points[:, axis].double()[None, :]
        sin_sum = s * wc + c * ws
        sums.append(((c * wc - s * ws).sum(0), (sin_sum * d).sum(0), (sin_sum * d * d).sum(0)))
    (gc, gx, gxx), (_, gy, gyy) = sums
    return [torch.stack([2 * p * ad * gx, 2 * p * ad * gy], dim=1), gc,
            p * ad / zd * (gxx + gyy)]


def exact(case, seed):
    if case["kind"] == "batch":
        return [_hologram64(pr["points"], pr["A"], pr["z"], pr["lam"], pr["p"], pr["Nx"],
                            pr["Ny"]) for pr in _problems(case, seed)]
    cloud = [t.cuda() for t in _single(case, seed)]
    args = (case["lam"], case["pitch"], case["nx"], case["ny"])
    image = _hologram64(*cloud, *args)
    if case["kind"] != "fit":
        return image.cpu() if case["kind"] == "host" else image
    diff = image - _target(case, seed).double()
    return [image, diff.square().sum(), *_gradients64(*cloud, *args, 2.0 * diff)]
