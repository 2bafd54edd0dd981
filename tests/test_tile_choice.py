"""The tile tuner's choice among timed trials, with made-up timings (host
code, compiled from the library's own header): every shape is timed over the
same number of steps, whichever side of the half-millisecond line each one's
trial falls on."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2112_15071_gb300", "csrc")
SRC = r"""
#include "ews_tuner.cuh"
// Trials of shapes 1 .. n that take us[k] a step; the steps of each trial of
// the last choice go to steps[].
extern "C" int choose(const float* us, int n, int nt, int stop_at, int* steps) {
    std::vector<int> cand;
    for (int k = 0; k < n; ++k) cand.push_back(k + 1), steps[k] = 0;
    return ews::fastest_shape(cand, nt, [&](int shape, int T, float* ms) {
        if (shape == stop_at) return false;
        *ms = 1e-3f * us[shape - 1] * T;
        steps[shape - 1] = T;
        return true;
    });
}
"""


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    d = tmp_path_factory.mktemp("tuner")
    src, so = str(d / "choose.cc"), str(d / "choose.so")
    open(src, "w").write(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    lib = ctypes.CDLL(so)

    def f(us, nt=100, stop_at=0):
        steps = (ctypes.c_int * len(us))()
        best = lib.choose((ctypes.c_float * len(us))(*us), len(us), nt, stop_at, steps)
        return best, list(steps)
    return f


# microseconds a step of the shapes, the default first; six steps of the
# default take 0.54, 0.51 / 0.49, 0.06 and 6 ms
@pytest.mark.parametrize("us,best", [
    ([90, 82, 95, 85], 2),            # the faster shape's six steps take 0.49 ms
    ([85, 80, 74, 83], 3), ([81, 90, 76, 70], 4),
    ([85, 84, 84.5, 90], 1), ([81, 80, 85, 82], 1),      # within 2 % of the default
    ([10, 9.5, 9.0, 11], 3), ([1000, 900, 1100, 850], 4)])
def test_every_shape_runs_the_same_steps(choose, us, best):
    got, steps = choose(us)
    assert got == best
    assert len(set(steps)) == 1, steps
    assert steps[0] == 6 if us[0] * 6 >= 500 else 6 < steps[0] <= 64


def test_trials_end_with_the_run(choose):
    assert choose([10, 5], nt=4) == (2, [4, 4])
    assert choose([10, 5], nt=9) == (2, [9, 9])
    # a trial that fails ends the choice
    assert choose([10, 5, 1], stop_at=2)[0] == 1
