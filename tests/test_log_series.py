"""The polynomial that gives -2 ln(1 - d) to the noise of the packed updates
below d = 2^-5, with the FP32 coefficients of the source, against the
logarithm in 64 bits.  No GPU is needed."""
import os
import re

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0803_2826_gb300", "csrc")


def _coefficients():
    """Highest first, down to the coefficient of d: the multiply-adds of box_muller2 in order."""
    src = open(os.path.join(CSRC, "f32x2.cuh")).read()
    body = src[src.index("void box_muller2("):]
    named = {k: float(v) for k, v in re.findall(r"\b(kLog\d) = ([0-9.]+)f", src)}
    value = lambda t: eval(t.replace("f", ""), {}, {}) if not t.startswith("k") else named[t]  # noqa: E731
    first = re.search(r"F2 t = fma2\(d1, f2s\(([^)]*)\), f2s\(([^)]*)\)\);", body)
    out = [value(first.group(1)), value(first.group(2))]
    end = body.index("const F2 ser = d1 * t;")
    out += [value(m) for m in re.findall(r"t = fma2\(d1, t, f2s\(([^)]*)\)\);", body[:end])]
    return [float(np.float32(v)) for v in out]


def test_remainder():
    d = np.linspace(0.0, 2.0 ** -5, 100001)[1:]
    p = np.zeros_like(d)
    for c in _coefficients():
        p = p * d + c
    # the one-node map's series, six Taylor terms, leaves below 2^-32
    assert np.abs(p * d / (-2.0 * np.log1p(-d)) - 1.0).max() < 2.0 ** -32
