"""The cubic in s^2 that stands for atanh(s) / s in the noise radius (csrc/philox.cuh): its error on the
reduced range, as the comment beside it states it."""
import os
import re

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_cubic_against_atanh():
    text = open(os.path.join(ROOT, "paper_2602_16486_gb300", "csrc", "philox.cuh")).read()
    body = text[text.index("void box_muller("):]
    c3, c2, c1, c0 = [float(v or 1) for v in re.findall(r"float\(-4\.0 \*(?: ([0-9.]+) \*)? V\)", body)]
    stated = [float(v) for v in re.search(r"relative error ([0-9.e-]+),\s*// ([0-9.e-]+) with the coefficients", text).groups()]
    s = np.sqrt(np.linspace(1e-9, ((np.sqrt(2) - 1) / (np.sqrt(2) + 1)) ** 2, 200001, dtype=np.longdouble))
    exact = np.arctanh(s) / s
    for rounded, bound in zip((np.longdouble, np.float32), stated):
        k = [np.longdouble(rounded(v)) for v in (c0, c1, c2, c3)]
        err = np.abs((k[0] + s**2 * (k[1] + s**2 * (k[2] + s**2 * k[3]))) / exact - 1).max()
        assert 0.9 * bound < err < 1.05 * bound, (float(err), bound)  # the figure, to its two digits
    assert max(stated) < 2.0 ** -26  # below FP32 rounding
