"""The GELU of the epilogues, x Phi(x) = max(x, 0) - |x| 2^q(|x|): its coefficients as the kernel source has them, evaluated in
float32 as the kernel does, against 64 bits."""
import math
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_15618_b200", "csrc", "fm_gemm_tc.cuh")


def _coefficients():
    text = open(SRC).read()
    body = text[text.index("inline float2 gelu2"):]
    first = float(re.search(r"uint64_t q = pack\((-?[\d.e+-]+)f", body).group(1))
    rest = [float(v.strip().rstrip("f")) for v in re.search(r"K\[10\] = \{(.*?)\}", body, re.S).group(1).split(",")]
    limit = float(re.search(r"fminf\(fabsf\(a\), ([\d.]+)f\)", body).group(1))
    return [first] + rest, limit


def _gelu(x):
    f = np.float32
    K, limit = _coefficients()
    c = np.minimum(np.abs(x), f(limit))
    q = np.full_like(x, f(K[0]))
    for k in K[1:]:
        q = (q.astype(np.float64) * c + np.float64(f(k))).astype(f)            # one rounding, as a fused multiply-add
    g = (c * np.exp2(q.astype(np.float64)).astype(f)).astype(f)
    return (0.5 * (x + np.abs(x)).astype(np.float64) - g).astype(f), q.astype(np.float64), g.astype(np.float64)


@pytest.mark.parametrize("lo,hi", [(-1e-3, 1e-3), (-1.0, 1.0), (-7.0, 7.0), (-9.0, 9.0), (6.99, 7.01), (-7.01, -6.99), (-1e4, 1e4)])
def test_error_stays_within_its_roundings(lo, hi):
    x = np.linspace(lo, hi, 40001).astype(np.float32)
    y, q, g = _gelu(x)
    ref = np.array([0.5 * v * math.erfc(-v / math.sqrt(2.0)) for v in x.astype(np.float64)])
    # half a unit of the result, the roundings of q (of the size of its last terms) and of 2^q and its product, the fit
    bound = 2.0 ** -24 * np.abs(ref) + g * (2.0 ** -22 + 2.0 ** -23 * (1.0 + np.abs(q))) + 1e-9
    assert (np.abs(y - ref) <= bound).all(), np.max(np.abs(y - ref) / bound)


def test_special_values():
    with np.errstate(invalid="ignore"):
        y, _, _ = _gelu(np.array([0.0, 1e30, -1e30, np.inf], dtype=np.float32))
    assert y[0] == 0 and y[1] == np.float32(1e30) and abs(y[2]) < 1e-10 and np.isinf(y[3])
