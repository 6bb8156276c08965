"""The fork to a handle's side stream and its join (class Forked), with the CUDA
runtime replaced by functions that write down what was called: on every way out of
the scope the call's stream waits for the side stream."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2001_06111_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <string>
#include "bt_internal.cuh"
static int fail_at, calls;
static cudaError_t call(const char *what) {
    printf("%s ", what);
    return ++calls == fail_at ? cudaErrorUnknown : cudaSuccess;
}
static const cudaStream_t kMain = (cudaStream_t)1, kSide = (cudaStream_t)2;
static const cudaEvent_t kFork = (cudaEvent_t)3, kJoin = (cudaEvent_t)4;
extern "C" {
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    return call(e == kFork && s == kMain ? "fork" : e == kJoin && s == kSide ? "join" : "wrong-record");
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    return call(e == kFork && s == kSide ? "side-waits" : e == kJoin && s == kMain ? "main-waits" : "wrong-wait");
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return call(s == kSide ? "sync-side" : "sync-main"); }
}
static cudaError_t work(const std::string &how) {
    bt::Side s;
    s.stream = kSide;
    s.fork = kFork;
    s.join = kJoin;
    bt::Forked f(s, kMain);
    if (how == "unused") return f.join();
    BT_CUDA(f.fork());
    printf("work ");
    if (how == "error") return cudaErrorUnknown;
    return f.join();
}
int main(int argc, char **argv) {
    fail_at = argc > 2 ? atoi(argv[2]) : 0;
    const cudaError_t e = work(argv[1]);
    printf(e == cudaSuccess ? "ok" : "failed");
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("side")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", inc, str(d / "p.cpp"), "-o", str(d / "p"),
                    "-Wl,--unresolved-symbols=ignore-all"], check=True)
    return str(d / "p")


@pytest.mark.parametrize("args,want", [
    (["done"], "fork side-waits work join main-waits ok"),
    # an error between fork and join
    (["error"], "fork side-waits work join main-waits failed"),
    (["unused"], "ok"),
    # a call of the fork or the join fails itself (the n-th)
    (["done", "1"], "fork failed"),
    (["done", "2"], "fork side-waits failed"),
    (["done", "3"], "fork side-waits work join sync-side failed"),
    (["done", "4"], "fork side-waits work join main-waits sync-side failed"),
    (["error", "3"], "fork side-waits work join sync-side failed"),
])
def test_joined_on_every_way_out(program, args, want):
    assert subprocess.run([program, *args], capture_output=True, text=True, check=True).stdout == want
