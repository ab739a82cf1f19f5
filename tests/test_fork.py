"""Side streams are joined on every way out of a call (csrc/fork.cuh), shown on
the CPU: the class is compiled against stand-ins of the two runtime calls it
makes, which log what they are given and fail on request.  And every function
that launches on a plan's side streams does so inside a Fork.
"""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2406_14920_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

HARNESS = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include "fork.cuh"
static int calls = 0, fail_at = 0;  // call number that fails (0: none)
static cudaError_t step() { return ++calls == fail_at ? cudaErrorUnknown : cudaSuccess; }
extern "C" cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  std::printf("record %d on %d\n", (int)(intptr_t)e, (int)(intptr_t)s);
  return step();
}
extern "C" cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  std::printf("wait %d for %d\n", (int)(intptr_t)s, (int)(intptr_t)e);
  return step();
}
// a call over n side streams (10, 11, ..; events 20, 21, ..) that gives up at launch `stop` (0: does not)
static int call(int n, int stop) {
  cudaStream_t side[4];
  cudaEvent_t done[4];
  for (intptr_t b = 0; b < 4; ++b) side[b] = (cudaStream_t)(10 + b), done[b] = (cudaEvent_t)(20 + b);
  eri::Fork f((cudaStream_t)1, side, (cudaEvent_t)2, done);
  if (f.open(n) != cudaSuccess) return -1;
  for (int l = 1; l <= 6; ++l) {
    if (l == stop) return -2;
    std::printf("launch\n");
  }
  if (f.join() != cudaSuccess) return -3;
  std::printf("rest\n");
  return 0;
}
int main(int, char** v) {
  fail_at = std::atoi(v[3]);
  std::printf("rc %d\n", call(std::atoi(v[1]), std::atoi(v[2])));
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("fork")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", os.path.join(CUDA, "include"), str(src), "-o", str(exe)],
                   check=True)
    return lambda *a: subprocess.run([str(exe), *map(str, a)], check=True, capture_output=True,
                                     text=True).stdout.split("\n")[:-1]


def _joined(log, n):
    return all(f"record {20 + b} on {10 + b}" in log and f"wait 1 for {20 + b}" in log for b in range(n))


@pytest.mark.parametrize("n", [1, 3])
def test_joined_once_at_the_end(harness, n):
    log = harness(n, 0, 0)
    assert log[-1] == "rc 0" and log[-2] == "rest" and _joined(log, n)
    assert sum(x.startswith("wait 1 ") for x in log) == n


@pytest.mark.parametrize("stop", [1, 4])
def test_joined_after_a_failed_launch(harness, stop):
    log = harness(3, stop, 0)
    assert log[-1] == "rc -2" and _joined(log, 3)


def test_joined_streams_of_a_failed_fork(harness):
    log = harness(3, 0, 3)  # the second side stream cannot be forked
    assert log[-1] == "rc -1" and _joined(log, 1) and not _joined(log, 2)


@pytest.mark.parametrize("fail", [5, 6, 8])
def test_a_failed_join_is_reported_and_the_others_joined(harness, fail):
    log = harness(3, 0, fail)
    assert log[-1] == "rc -3" and "rest" not in log
    assert all(f"record {20 + b} on {10 + b}" in log for b in range(3))
    assert sum(x.startswith("wait 1 ") for x in log) >= 2


def test_no_streams_no_calls(harness):
    assert harness(0, 0, 0) == ["launch"] * 6 + ["rest", "rc 0"]


def test_every_use_of_a_side_stream_is_inside_a_fork():
    for name in ("plan.cu", "nuclear.cu", "xc.cu"):
        src = open(os.path.join(CSRC, name)).read()
        # functions at the left margin, from their opening to the closing brace at the margin
        for body in re.findall(r"^\S[^\n;]*\{\n(.*?)^\}", src, re.M | re.S):
            if re.search(r"P->branch\[", body):
                assert "Fork side(" in body and "side.join()" in body
        assert "->fork(" not in src and "->join(" not in src
