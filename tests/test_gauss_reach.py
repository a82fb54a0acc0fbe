"""How far the FP32 edge kernels visit the radial basis (csrc/gauss_reach.h): for weights of one scale, of
scales that rise and fall over the centres, and with channels of zeros, what is left out of a filter value or of its
distance derivative is at most 2^-25 of the largest term kept, on a grid finer than the one it was worked out on;
weights that allow nothing to be left out get the whole reach."""
import os
import subprocess

import numpy as np
import pytest

import paper_2506_04055_gb300 as eng

SRC = os.path.join(os.path.dirname(os.path.abspath(eng.__file__)), "csrc")
PROGRAM = r"""
#include <cstdio>
#include "gauss_reach.h"
int main() {
  int rows, K;
  while (std::fread(&rows, 4, 1, stdin) == 1 && std::fread(&K, 4, 1, stdin) == 1) {
    std::vector<float> w((size_t)rows * K);
    if (std::fread(w.data(), 4, w.size(), stdin) != w.size()) return 1;
    std::printf("%.9g\n", ctd::gauss_reach(w.data(), rows, K, K));
  }
}
"""
LEAST, WHOLE = 6.3246, 14.5


@pytest.fixture(scope="module")
def reach(tmp_path_factory):
    d = tmp_path_factory.mktemp("reach")
    (d / "r.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-I", SRC, str(d / "r.cpp"), "-o", str(d / "r")], check=True)

    def go(w):
        w = np.ascontiguousarray(w, np.float32)
        data = np.array(w.shape, np.int32).tobytes() + w.tobytes()
        return float(subprocess.run([str(d / "r")], input=data, check=True, capture_output=True).stdout)

    return go


def _worst(w, X):
    """Largest ratio of what is left out to the largest term kept, over channels and distances."""
    K = w.shape[1]
    k = np.arange(K)
    worst = 0.0
    for x in np.arange(0.0, K - 1 + 1e-9, 0.01):
        first = max(0, int(np.ceil(x - X))) // 4 * 4
        if first == 0:
            continue
        t = np.abs(x - k)
        for term in (np.exp(-0.5 * t * t), t * np.exp(-0.5 * t * t)):
            term = np.abs(w.astype(np.float64)) * term
            lost, kept = term[:, :first].sum(1), term[:, first:].max(1)
            with np.errstate(divide="ignore", invalid="ignore"):
                worst = max(worst, float(np.nan_to_num(lost / kept, nan=0.0, posinf=np.inf).max()))
    return worst


@pytest.mark.parametrize("K", [2, 4, 7, 12, 16, 20, 27, 32])
@pytest.mark.parametrize("scale", ["one", "rising", "falling", "steep", "random", "zeros"])
def test_left_out_terms_are_below_the_rounding(reach, K, scale):
    rng = np.random.default_rng(K)
    w = rng.normal(size=(96, K))
    k = np.arange(K)
    w *= {"one": 1.0 + 0 * k, "rising": np.exp(0.4 * k), "falling": np.exp(-0.4 * k), "steep": np.exp(-1.5 * k),
          "random": np.exp(3.0 * rng.normal(size=(96, K))), "zeros": (rng.random((96, K)) < 0.5)}[scale]
    w = w.astype(np.float32)
    X = reach(w)
    assert LEAST - 1e-4 <= X <= WHOLE
    if X < WHOLE:
        assert _worst(w, X + 1e-6) <= 2.0 ** -25   # 1e-6: the kernel's own rounding of the distance
    if scale == "one":
        assert X < 8.0


def test_far_weights_alone_are_all_visited(reach):
    w = np.zeros((96, 20), np.float32)
    assert reach(w) == pytest.approx(LEAST)
    w[5, 3] = 1.0   # the last of its group: visited up to where FP32 has zero for it
    assert reach(w) == WHOLE
