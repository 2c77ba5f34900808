"""The choice between the two kernels of 256 x 256 galaxies (csrc/routes.h) goes by
how many of them there are, not by the batch: for every bucket count that a batch
may have exactly one of the launched kernels takes the galaxies, and it is the one
on whose side of the line that count is (in batches of many thousands the kernel
of many, which then is never what the call waits for)."""

import os
import shutil
import subprocess

import pytest

FAR = 19456   # galaxies of a batch above which the kernel of many runs alone
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_15797_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "routes.h"
constexpr int FAR = 19456;
struct Params { int64_t max_galaxies = INT64_MAX; int bucket_min = 0, bucket_max = INT32_MAX; };
// argv: the batch's count, the line, what the launch of the kernel of few returns
int main(int, char** v) {
  Params p;
  p.max_galaxies = atoll(v[1]);
  const int fails = atoi(v[3]);
  const int e = mog::launch_by_count(
      p, atoi(v[2]), FAR, 0, [&] { printf("fork 0 0\n"); return 0; },
      [&](const Params& q, bool beside) {
        printf("%s %d %d\n", beside ? "few_beside" : "few", q.bucket_min, q.bucket_max);
        return fails;
      },
      [&](const Params& q) { printf("many %d %d\n", q.bucket_min, q.bucket_max); return 0; },
      [&] { printf("join 0 0\n"); return 0; });
  printf("status %d\n", e);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("routes")
    (d / "main.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")], check=True)
    return str(d / "main")


def _run(program, count, line, fails=0):
    out = subprocess.run([program, str(count), str(line), str(fails)], check=True, capture_output=True, text=True).stdout
    rows = [r.split() for r in out.splitlines()]
    return [r[0] for r in rows[:-1]], {r[0]: (int(r[1]), int(r[2])) for r in rows[:-1]}, int(rows[-1][1])


@pytest.mark.parametrize("line", [114, 228, 1216])
@pytest.mark.parametrize("count", [1, 113, 114, 115, 228, 229, 1215, 1216, 1217, 19_456, 19_457, 2**31 - 1, 2**63 - 1])
def test_one_kernel_takes_every_bucket_count(program, count, line):
    steps, ranges, status = _run(program, count, line)
    assert status == 0
    assert steps == (["few"] if count <= line else ["many"] if count > FAR else ["fork", "few_beside", "many", "join"])
    kernels = {k.split("_")[0]: r for k, r in ranges.items() if k not in ("fork", "join")}
    for here in {0, 1, line - 1, line, line + 1, min(count, 2**31 - 1)}:
        if here > count:
            continue
        takes = [k for k, (lo, hi) in kernels.items() if lo <= here <= hi]
        assert takes == ["few" if here <= line and count <= FAR else "many"], here


def test_a_failed_launch_is_returned_and_joined(program):
    steps, _, status = _run(program, 5000, 1216, fails=7)
    assert status == 7 and steps == ["fork", "few_beside", "join"]


def test_both_kernels_of_both_directions_follow_it():
    for name in ("render_fwd256", "render_fwd256c", "render_bwd256", "render_bwd256c"):
        with open(os.path.join(CSRC, name + ".cu")) as f:
            text = f.read()
        assert "if (count < p.bucket_min || count > p.bucket_max) return;" in text, name
        if not name.endswith("c"):
            assert "return launch_by_count(" in text, name
