"""The calls' device allocator when the host is out of memory, with the CUDA runtime and
operator new replaced: the allocation fails as one of the device would, gives back
what it took, and no exception leaves it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2001_06111_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <new>
static int allow = 1 << 30;  // calls of operator new that still succeed
void *operator new(size_t n) {
    if (allow-- <= 0) throw std::bad_alloc();
    return malloc(n);
}
void operator delete(void *p) noexcept { free(p); }
void operator delete(void *p, size_t) noexcept { free(p); }
#include "bt_internal.cuh"
static int held;
extern "C" {
cudaError_t cudaMallocFromPoolAsync(void **p, size_t, cudaMemPool_t, cudaStream_t) {
    ++held;
    *p = malloc(16);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) {
    --held;
    free(p);
    return cudaSuccess;
}
}
int main(int, char **argv) {
    bt::Alloc al{};
    allow = atoi(argv[1]);
    int got = 0;
    for (int i = 0; i < 100; ++i) got += al.get<int>(1) != nullptr;
    allow = 1 << 30;
    const bool told = al.err == cudaErrorMemoryAllocation;
    const int live = (int)al.live.size(), was = held;
    al.undo_to(0);
    printf("%d %d %d %d %d", got, told, live, was, held);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("alloc")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    (d / "p.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", inc, str(d / "p.cpp"), "-o", str(d / "p"),
                    "-Wl,--unresolved-symbols=ignore-all"], check=True)
    return str(d / "p")


@pytest.mark.parametrize("grows", [0, 1, 4, 1000])
def test_host_out_of_memory(program, grows):
    out = subprocess.run([program, str(grows)], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    got, told, live, was, left = map(int, out.stdout.split())
    assert got == live == was and left == 0
    assert (told, got) == (0, 100) if grows == 1000 else told == 1 and got < 100
