"""Side streams of a call (csrc/branches.h, the fork and join of the size
kernels): whatever launch or stream call fails, every branch that was forked is
joined into the caller's stream before the call returns, and the first failure
is what it returns."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_15797_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "branches.h"
// argv: number of branches, what fails (fork, launch, join, -), at which branch
int main(int, char** v) {
  const int n = atoi(v[1]), at = atoi(v[3]);
  auto step = [&](const char* what) {
    return [=](int i) { printf("%s%d ", what, i); return !strcmp(v[2], what) && i == at ? 10 + i : 0; };
  };
  printf("-> %d\n", mog::run_branches(n, 0, step("fork"), step("launch"), step("join")));
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("branches")
    (d / "main.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")], check=True)
    return str(d / "main")


def _run(program, n, what, at):
    out = subprocess.run([program, str(n), what, str(at)], check=True, capture_output=True, text=True).stdout
    steps, status = out.strip().split("-> ")
    return steps.split(), int(status)


@pytest.mark.parametrize("n", [1, 2, 4])
def test_all_succeed(program, n):
    steps, status = _run(program, n, "-", 0)
    assert status == 0
    assert steps == [f"{w}{i}" for i in range(n) for w in ("fork", "launch")] + [f"join{i}" for i in range(n)]


@pytest.mark.parametrize("what", ["fork", "launch", "join"])
@pytest.mark.parametrize("at", range(4))
def test_a_failure_leaves_no_forked_branch_unjoined(program, what, at):
    steps, status = _run(program, 4, what, at)
    assert status == 10 + at
    forked = [s[4:] for s in steps if s.startswith("fork") and not (what == "fork" and s == f"fork{at}")]
    assert [s[4:] for s in steps if s.startswith("join")] == forked
    if what != "join":   # nothing more is launched after a failure
        assert not any(s.startswith("launch") and int(s[6:]) > at for s in steps)


def test_the_size_kernels_are_launched_through_it():
    with open(os.path.join(CSRC, "api.cu")) as f:
        text = f.read()
    body = text[text.index("mog_status launch_buckets("):]
    body = body[:body.index("\n}\n")]
    assert "return run_branches<mog_status>(n, MOG_OK, fork, run, join);" in body
