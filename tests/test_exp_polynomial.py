"""The degree-5 polynomial of the pair forward kernel (ex2_poly2_deg5), evaluated in float32 on the CPU with the
coefficients of the source: its largest and its mean relative error over the reduced argument, and the scaling by 2^n."""
import os
import re

import numpy as np

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_05693_b200", "csrc", "tc_common.cuh")


def ex2_poly2_deg5(x):
    text = open(SRC).read()
    body = text[text.index("void ex2_poly2_deg5"):]
    body = body[:body.index("r0 = ")]
    c = [np.float64(np.float32(v)) for call in re.findall(r"fma2g\((.*?)\);", body)
         for v in dict.fromkeys(re.findall(r"(\d+\.\d+)f", call))]
    assert len(c) == 6
    x = np.maximum(x.astype(np.float32), np.float32(-126))
    t = x + np.float32(12582912.0)
    f = x - (t - np.float32(12582912.0))
    p = (f.astype(np.float64) * c[0] + c[1]).astype(np.float32)
    for v in c[2:]:
        p = (p.astype(np.float64) * f.astype(np.float64) + v).astype(np.float32)
    return (p.view(np.uint32) + (t.view(np.uint32) << np.uint32(23))).view(np.float32)


def test_error_of_the_degree_5_polynomial():
    x = np.linspace(-0.5, 0.5, 400001).astype(np.float32)
    err = ex2_poly2_deg5(x).astype(np.float64) / np.exp2(x.astype(np.float64)) - 1
    assert np.abs(err).max() < 1.8e-7      # 1.1e-7 of the fit and one rounding, 2^-24
    assert abs(err.mean()) < 3e-8          # the sums of a row's weights are as far off as the mean
    wide = np.linspace(-120, 8, 1000001).astype(np.float32)   # logits may exceed the row maximum in use by 2^8
    err = ex2_poly2_deg5(wide).astype(np.float64) / np.exp2(wide.astype(np.float64)) - 1
    assert np.abs(err).max() < 1.8e-7
