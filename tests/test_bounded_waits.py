"""The bounded waits of the transform kernels (csrc/waits.h), driven on the host by a simulated
barrier: a wait for another role ends when a role has failed; the wait for products and copies
under way, before their memory is given up, ends only when they are done or its own limit is
reached, and a failed role does not shorten it."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1212_1397_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "waits.h"
// one wait: kind, poll after which the barrier completes, poll at which another role fails (-1: never), limit
int main(int, char** a) {
  const int kind = atoi(a[1]), complete = atoi(a[2]), failing = atoi(a[3]), limit = atoi(a[4]);
  volatile int fail = 0;
  int polls = 0;
  auto done = [&] {
    if (polls == failing) fail = 1;
    return ++polls > complete;
  };
  auto rest = [] {};
  const bool ok = kind ? helm6::wait_flight(done, rest, &fail, limit) : helm6::wait_role(done, rest, &fail, limit, 64);
  printf("%d %d %d\n", (int)ok, polls, (int)fail);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("waits")
    src = d / "waits.cpp"
    src.write_text(SOURCE)
    exe = str(d / "waits")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", exe], check=True)
    return exe


def run(program, kind, complete, failing, limit):
    out = subprocess.run([program, str(kind), str(complete), str(failing), str(limit)], check=True,
                         capture_output=True, text=True).stdout.split()
    return tuple(int(v) for v in out)  # ok, polls, fail flag


@pytest.mark.parametrize("complete", [0, 1, 63, 64, 65, 1000, 99999])
@pytest.mark.parametrize("failing", [-1, 0, 1, 64, 500])
def test_work_under_way_is_waited_for(program, complete, failing):
    ok, polls, fail = run(program, 1, complete, failing, 100000)
    assert ok == 1 and polls == complete + 1
    assert fail == (1 if 0 <= failing <= complete else 0)


def test_the_limit_holds_and_raises_the_flag(program):
    assert run(program, 1, 10 ** 9, -1, 1000) == (0, 1000, 1)
    assert run(program, 1, 10 ** 9, 3, 1000) == (0, 1000, 1)
    assert run(program, 0, 10 ** 9, -1, 1000) == (0, 1000, 1)


@pytest.mark.parametrize("failing", [0, 63, 64, 500])
def test_a_role_gives_up_when_another_has_failed(program, failing):
    ok, polls, fail = run(program, 0, 10 ** 9, failing, 100000)
    assert ok == 0 and fail == 1 and failing < polls <= failing + 64
    assert run(program, 0, 10, -1, 100000) == (1, 11, 0)
