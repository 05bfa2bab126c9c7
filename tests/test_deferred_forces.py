"""The order in which a call launches its steps and the sums of their forces (csrc/deferred.h), with fakes of the
launches: whatever step or sum fails, every step that ran has its force summed once, in order, or is reported."""
import ctypes
import subprocess

import pytest

from paper_0904_4504_gb300 import builder as B

SOURCE = r"""
#include "deferred.h"
// log[k]: times step k's force was summed; fail_step / fail_sum: the launch of that number fails (-1: none)
extern "C" int run(long n, int most, long fail_step, int fail_sum, long* ran, int* lost, int* log) {
    int sums = 0;
    *ran = 0;
    return lbm::run_deferred(n, most,
        [&](long k, int held) {
            if (k != *ran || held >= most) return 77;      // steps in order, a place that exists
            if (k == fail_step) return 5;
            ++*ran;
            return 0;
        },
        [&](int held) {
            if (held < 1 || held > most) return 78;
            if (sums++ == fail_sum) return 6;
            for (long k = *ran - held; k < *ran; ++k) ++log[k];
            return 0;
        }, lost);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("deferred")
    (d / "run.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wall", "-Werror", f"-I{B.CSRC}", str(d / "run.cpp"),
                    "-o", str(d / "run.so")], check=True)
    f = ctypes.CDLL(str(d / "run.so")).run
    f.argtypes = [ctypes.c_long, ctypes.c_int, ctypes.c_long, ctypes.c_int, ctypes.POINTER(ctypes.c_long),
                  ctypes.POINTER(ctypes.c_int), ctypes.POINTER(ctypes.c_int)]

    def call(n, most, fail_step=-1, fail_sum=-1):
        ran, lost, log = ctypes.c_long(), ctypes.c_int(), (ctypes.c_int * max(n, 1))()
        rc = f(n, most, fail_step, fail_sum, ctypes.byref(ran), ctypes.byref(lost), log)
        return rc, ran.value, lost.value, list(log[:n])
    return call


@pytest.mark.parametrize("most", [1, 4, 64])
def test_every_step_that_ran_is_summed(run, most):
    for n in [0, 1, 2, 3, 4, 5, 8, 63, 64, 65, 130]:
        assert run(n, most) == (0, n, 0, [1] * n)
        for at in range(n):
            rc, ran, lost, log = run(n, most, fail_step=at)
            assert (rc, ran, lost) == (5, at, 0) and log == [1] * at + [0] * (n - at)


@pytest.mark.parametrize("most", [1, 4, 64])
def test_sums_that_fail_are_reported(run, most):
    for n in [1, 3, 4, 5, 65, 130]:
        for at in range(-(-n // most)):
            rc, ran, lost, log = run(n, most, fail_sum=at)
            assert rc == 6 and log == [1] * (at * most) + [0] * (n - at * most) and ran == at * most + lost and lost > 0
        for step in range(n):  # a step, then the sum of what ran before it
            rc, ran, lost, log = run(n, most, fail_step=step, fail_sum=step // most)
            assert (rc, ran) == (5, step) and sum(log) + lost == step and lost == step % most
