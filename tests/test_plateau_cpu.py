"""The FP32 plateau test of the on-chip iterations (csrc/dpf_plateau.h), compiled
for the host, against the FP64 decision it stands for."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2603_28203_gb300", "csrc")

SRC = """
#include "dpf_plateau.h"
extern "C" int side(float best, float sum, double threshold) {
  return dpf::plateau_side(sum, dpf::plateau_bar(best, (float)(1.0 - threshold)));
}
"""


@pytest.fixture(scope="module")
def side(tmp_path_factory):
    d = tmp_path_factory.mktemp("plateau")
    (d / "t.cpp").write_text(SRC)
    so = str(d / "t.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I" + CSRC, str(d / "t.cpp"),
                    "-o", so], check=True)
    f = C.CDLL(so).side
    f.argtypes = [C.c_float, C.c_float, C.c_double]
    return f


@pytest.mark.parametrize("threshold", [1e-4, 0.0, -0.5, 0.1, 0.9, 0.97, 0.99, 0.998, 0.9999, 1 - 1e-6, 1 - 2.0 ** -40, 1.0, 2.0])
def test_the_fp32_answer_is_the_fp64_answer(side, threshold):
    """Sums around the bar, by single FP32 steps and by relative distances; an
    answer of 0 leaves the decision to FP64 and is due near the bar only."""
    rng = np.random.default_rng(3)
    told = 0
    for best in np.concatenate([10.0 ** rng.uniform(-12, 12, 200), [1e-44, 1e-38, 3e38, 0.0]]).astype(np.float32):
        bar = np.float64(best) * (1.0 - threshold)
        with np.errstate(over="ignore"):
            near = [np.float32(bar)]
            for _ in range(15):  # one step further down and up each
                near = [np.nextafter(near[0], np.float32(-np.inf))] + near + [np.nextafter(near[-1], np.float32(np.inf))]
            near += list((bar * (1 + np.concatenate([d := 10.0 ** rng.uniform(-8, -1, 40), -d]))).astype(np.float32))
        for x in near:
            if not np.isfinite(x) or x < 0:
                continue
            s = side(best, x, threshold)
            below = np.float64(x) < np.float64(best) * (1.0 - threshold)
            assert s == 0 or (s > 0) == below, (best, x)
            if s == 0 and 1e-25 < bar < 1e36:
                assert abs(np.float64(x) - bar) <= 2e-6 * bar
            told += s != 0
    assert told > 0 or threshold >= 1.0
