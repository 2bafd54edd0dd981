"""The tuner's host code, compiled from the library's own header.  The choice
of a tile shape among timed trials, with made-up timings: every shape is timed
over the same number of steps, whichever side of the half-millisecond line each
one's trial falls on.  And what a batch's choice is kept under: everything it
was timed with."""
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
extern "C" int same_key(const int* a, int na, const int* b, int nb) {
    // boundary, exec, steps, device, then 4 numbers a shot
    auto key = [](const int* p, int n) {
        std::vector<std::array<int, 4>> s;
        for (int k = 4; k + 3 < n; k += 4) s.push_back({p[k], p[k + 1], p[k + 2], p[k + 3]});
        return ews::batch_key(s, p[0], p[1], p[2], p[3]);
    };
    return key(a, na) == key(b, nb);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("tuner")
    src, so = str(d / "choose.cc"), str(d / "choose.so")
    open(src, "w").write(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.fixture
def choose(lib):
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


def test_a_batch_choice_is_kept_under_all_it_depends_on(lib):
    def same(a, b):
        return bool(lib.same_key((ctypes.c_int * len(a))(*a), len(a), (ctypes.c_int * len(b))(*b), len(b)))
    base = [1, 0, 6, 0, 96, 80, 64, 0, 48, 48, 48, 0]
    assert same(base, base)
    assert same(base, base[:4] + base[8:] + base[4:8])           # the shots in another order
    for k in range(len(base)):                                   # any number another
        assert not same(base, base[:k] + [base[k] + 1] + base[k + 1:]), k
    assert not same(base, base + base[4:8]) and not same(base, base[:8])
    # the shape asked for belongs to its grid
    assert not same(base[:7] + [4] + base[8:], base[:11] + [4])
