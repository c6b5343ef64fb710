"""The quarter-turn sine and cosine polynomials of the tables (cos_poly.h,
sincos_fixed in csrc/sep32.cuh) in FP32, as the kernels evaluate them, against
FP64."""
import os
import re

import numpy as np
import pytest

HDR = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_1002_0916_gb300", "csrc", "cos_poly.h")
# values of at most 1: the last multiply-add's rounding and the leading term's,
# half an FP32 unit in the last place of 1 each, with as much for the fit
TOL = 2.0 ** -23


@pytest.mark.parametrize("prefix,exact", [("QSIN_C", np.sin), ("QCOS_C", np.cos)])
def test_error_over_half_a_quarter_turn_each_way(prefix, exact):
    c = [float(np.float32(float(v))) for v in
         re.findall(r"constexpr float " + prefix + r"\d+ = ([-0-9.e+]+)f;", open(HDR).read())]
    assert len(c) == (4 if prefix == "QSIN_C" else 5)
    x = np.concatenate([np.linspace(-0.5, 0.5, 200001), [0.0, 2.0 ** -33, -2.0 ** -33]])
    x = x.astype(np.float32)
    z = (x * x).astype(np.float32)
    p = np.full_like(z, c[-1])
    for k in c[-2::-1]:  # a fused multiply-add: FP64 holds the product exactly
        p = (p.astype(np.float64) * z + k).astype(np.float32)
    if prefix == "QSIN_C":
        p = (p * x).astype(np.float32)
    ref = exact(np.pi / 2 * x.astype(np.float64))
    assert np.abs(p - ref).max() <= TOL
    if prefix == "QSIN_C":  # relative, down to the smallest phases
        nz = x != 0
        assert np.abs(p[nz] / ref[nz] - 1).max() <= 2 * TOL
