"""The polynomial that stands for part of the exponentials in the tensor-core softmax: its coefficients, as written in the source,
against 2^f in float64 over the interval it is used on."""
import os
import re

import numpy as np

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_18484_b200", "csrc", "tc_common.cuh")


def test_relative_error():
    body = open(SRC).read().split("float2 ex2_poly2(float2 x)")[1].split("return y;")[0]
    c = [float(v) for v in re.findall(r"make_float2\(([0-9.]+)f, \1f\)", body)]
    assert len(c) == 4 and c[3] == 1.0                        # cubic, ..., constant: exactly one (results below 2^-127 are zero)
    f = np.linspace(-0.5, 0.5, 20001)
    err = ((c[0] * f + c[1]) * f + c[2]) * f + c[3]
    err = err / 2.0 ** f - 1.0
    # the best cubic with this constant is 1.0128e-4 off; one digit less in the last coefficient would add 1e-7
    assert np.abs(err).max() <= 1.02e-4 and abs(err.mean()) <= 5e-5
