"""The sliding phase search's 16QAM distance (csrc/common.cuh, qam_dist) in its own arithmetic:
|x| - l / sqrt10 per dimension as one fused product and sum, so that the outer level carries
three times the error of a rounded 1 / sqrt10 and no rounding of its own."""
import os
import re

import numpy as np

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_06311_gb300", "csrc", "common.cuh")


def _body():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    return text[text.index("float qam_dist("):text.index("unsigned qam_bits(")]


def test_the_level_is_not_rounded():
    body = _body()
    c = np.float32(float(re.search(r"const float c = ([0-9.]+)f;", body).group(1)))
    assert len(re.findall(r"__fmaf_rn\([^;]*\? -3\.f : -1\.f, c, fabsf\(z\.[xy]\)\)", body)) == 2
    rng = np.random.default_rng(5)
    x = np.abs(rng.normal(0, 0.7, 400_000)).astype(np.float32)
    outer = x * np.float32(np.sqrt(10.0)) > 2
    lv = np.where(outer, 3.0, 1.0)
    got = (x.astype(np.float64) - lv * float(c)).astype(np.float32)      # exact in FP64, then one rounding
    want = x.astype(np.float64) - lv / np.sqrt(10.0)
    # half an ulp of the result and three times the error of the rounded 1 / sqrt10
    err = np.abs(got - want) - 2.0 ** -24 * np.abs(want)
    bound = 3 * abs(float(c) - 1 / np.sqrt(10.0)) * (1 + 1e-6)
    assert err.max() <= bound < 7e-9
    # a rounded outer level is over five times further off
    rounded = abs(float(np.float32(3) * c) - 3 / np.sqrt(10.0))
    assert rounded > 5 * bound
