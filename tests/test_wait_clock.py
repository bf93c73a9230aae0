"""The clock of the bounded device waits (lbm_wait.h, compiled for the host):
steady polling gives up after a second; a context that is switched out for any
time in the middle of a wait does not end it; every wait ends."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1407_4524_gb300", "csrc")

# polls `step` ns apart, with a gap of `hole` ns before poll number `at`; prints
# the number of polls until the wait gives up (-1: not within `limit`)
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "lbm_wait.h"
int main(int argc, char **argv) {
    const unsigned long long step = strtoull(argv[1], 0, 10), hole = strtoull(argv[2], 0, 10);
    const long long at = atoll(argv[3]), limit = atoll(argv[4]);
    unsigned long long now = 1700000000000000000ull;
    lbm::WaitClock c{now, 0ull};
    for (long long k = 1; k <= limit; ++k) {
        now += k == at ? hole : step;
        if (lbm::wait_over(c, now)) {
            std::printf("%lld", k);
            return 0;
        }
    }
    std::printf("-1");
}
"""


@pytest.fixture(scope="module")
def polls(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("wait")
    src, exe = d / "wait.cpp", d / "wait"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return lambda *a: int(subprocess.run([str(exe)] + [str(v) for v in a], capture_output=True, text=True,
                                         check=True).stdout)


@pytest.mark.parametrize("step", [1000, 64000, 5000000])
def test_steady_polling_gives_up_after_a_second(polls, step):
    assert polls(step, step, 1, 10 ** 7) == 10 ** 9 // step + 1


@pytest.mark.parametrize("hole", [2 * 10 ** 8, 1100000000, 30 * 10 ** 9, 3600 * 10 ** 9])
@pytest.mark.parametrize("at", [1, 400, 800])
def test_a_switched_out_context_does_not_end_a_wait(polls, at, hole):
    # 1 ms polls: a tenth of a second and more of polling is left after the gap
    # (a gap, however long, counts an eighth of a second)
    assert polls(10 ** 6, hole, at, at + 70) == -1
    assert polls(10 ** 6, hole, at, 2000) == 877  # 125 counted for the gap, then over a second in all


def test_polls_that_are_always_late_still_end(polls):
    assert polls(10 ** 9, 10 ** 9, 1, 100) == 9
