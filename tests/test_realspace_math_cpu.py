"""The pair kernel's polynomial for exp(x^2) erfc(x), read from the source, against a 64-bit erfcx."""
import os
import re

import numpy as np
import pytest

from helpers import ROOT

special = pytest.importorskip("scipy.special")


def coefficients():
    src = open(os.path.join(ROOT, "paper_2009_12617_gb300", "csrc", "realspace.cu")).read()
    body = src[src.index("F2 erfcx_pos(F2 x04)"):]
    body = body[body.index("F2 p ="):body.index("return")]
    return [np.float32(c) for c in re.findall(r"f2_all\((-?[0-9.e-]+)f\)", body)]


def test_erfcx_polynomial():
    """t Q(t), t = 1 / (1 + 2 x / 5) in (0, 1]: the FP32 coefficients in 64-bit arithmetic within 2.9e-8 of erfcx(x); in
    FP32 arithmetic within 2.5e-7 (Horner's rule with terms of both signs, and the last product)."""
    c = coefficients()
    assert len(c) == 11
    t = np.concatenate([np.linspace(1e-4, 1.0, 400001), np.geomspace(1e-8, 1e-4, 10001)]).astype(np.float32)
    t64 = t.astype(np.float64)
    ref = special.erfcx((1.0 / t64 - 1.0) * 2.5)
    p64, p32 = np.full_like(t64, c[0]), np.full_like(t, c[0])
    for k in c[1:]:
        p64, p32 = p64 * t64 + np.float64(k), p32 * t + k
    assert np.abs(p64 * t64 / ref - 1.0).max() < 2.9e-8
    assert np.abs((p32 * t).astype(np.float64) / ref - 1.0).max() < 2.5e-7
