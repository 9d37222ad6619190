"""Fork and join of the layer step's side stream, compiled for the host against a recording stand-in of the CUDA runtime: work on the
side stream is joined on every way out, so that nothing writes the caller's workspace after a call that failed half-way."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNTIME = r"""
#pragma once
#include <string>
typedef int cudaStream_t; typedef int cudaEvent_t; typedef int cudaError_t;
enum { cudaSuccess = 0 };
extern std::string log_; extern int fail_at_, calls_;
inline cudaError_t step_(const std::string& s) { if (++calls_ == fail_at_) { log_ += "!"; return 1; } log_ += s + " "; return 0; }
inline cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return step_("record" + std::to_string(e) + "@" + std::to_string(s)); }
inline cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { return step_("wait" + std::to_string(e) + "@" + std::to_string(s)); }
"""

MAIN = r"""
#include <cuda_runtime.h>
#include <cstdio>
std::string log_; int fail_at_ = 0, calls_ = 0;
#include "side_branch.cuh"
static int body(int leave_early) {
  cafeq::SideBranch b;
  if (!b.fork(1, 2, 10, 20)) return 4;
  log_ += "work@2 ";
  if (leave_early) return 2;
  log_ += "work@1 ";
  if (!b.join()) return 4;
  log_ += "after ";
  return 0;
}
int main(int, char** a) {
  fail_at_ = a[2][0] - '0';
  int rc = body(a[1][0] == '1');
  std::printf("%d %s\n", rc, log_.c_str());
}
"""


def test_the_side_branch_is_joined_on_every_way_out(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "main.cc").write_text(MAIN)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-I", str(tmp_path), "-I", os.path.join(ROOT, "paper_2511_19705_b200", "csrc"), "-o", exe,
                    str(tmp_path / "main.cc")], check=True)

    def run(early, fail):
        return subprocess.run([exe, early, fail], check=True, capture_output=True, text=True).stdout.split()

    fork, join = ["record10@1", "wait10@2"], ["record20@2", "wait20@1"]
    assert run("0", "0") == ["0"] + fork + ["work@2", "work@1"] + join + ["after"]   # joined once
    assert run("1", "0") == ["2"] + fork + ["work@2"] + join                         # left in between: joined all the same
    assert run("0", "1") == ["4", "!"]                                               # never forked: nothing to join
    assert run("0", "2") == ["4", "record10@1", "!"]


def test_the_layer_step_uses_it():
    src = open(os.path.join(ROOT, "paper_2511_19705_b200", "csrc", "layer_step.cuh")).read()
    assert "SideBranch" in src and "cudaStreamWaitEvent" not in src
