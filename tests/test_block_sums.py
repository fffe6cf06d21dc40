"""The block sums of block_sum.cuh, compiled for the host and run thread by
thread, for every block size of the kernels that call them (col_kernels.h,
row_kernels.h): a shuffle names and reads lanes that exist, and the sum is
that of all the block's threads."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1011_3582_gb300", "csrc")
# vector types and launch variables of a block, as far as the headers use them
CUDA_RUNTIME = r"""
#pragma once
#include <cmath>
#include <cstdlib>
#include <pthread.h>
#define __host__
#define __device__
#define __forceinline__ inline
#define __shared__ static
struct float2 { float x, y; };
struct double2 { double x, y; };
struct Dim { int x; };
inline thread_local Dim threadIdx;
inline Dim blockDim;
inline pthread_barrier_t block_barrier, warp_barrier[32];
inline double lane_value[1024];
inline bool bad;
inline void __syncthreads() { pthread_barrier_wait(&block_barrier); }
inline double __shfl_down_sync(unsigned mask, double v, int d) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n = blockDim.x - 32 * warp < 32 ? blockDim.x - 32 * warp : 32;
    if (n < 32 && mask >> n) bad = true;
    lane_value[threadIdx.x] = v;
    pthread_barrier_wait(&warp_barrier[warp]);
    const double o = lane + d < n ? lane_value[threadIdx.x + d] : lane + d < 32 ? NAN : v;
    pthread_barrier_wait(&warp_barrier[warp]);
    return o;
}
"""
PROGRAM = r"""
#include <cstdio>
#include <cuda_runtime.h>
#include "block_sum.cuh"
#include "col_kernels.h"
#include "row_kernels.h"
using namespace fftlb;
static double out;
template <int NT> void *thread(void *p) {
    threadIdx.x = (int)(size_t)p;
    block_sum_store<NT>(1.0 + threadIdx.x, &out);
    return nullptr;
}
template <int NT> void check(const char *kind, int size, int n) {
    pthread_t t[NT];
    blockDim.x = NT;
    bad = false;
    pthread_barrier_init(&block_barrier, nullptr, NT);
    for (int w = 0; w < (NT + 31) / 32; ++w) pthread_barrier_init(&warp_barrier[w], nullptr, NT - 32 * w < 32 ? NT - 32 * w : 32);
    for (int i = 0; i < NT; ++i) pthread_create(&t[i], nullptr, thread<NT>, (void *)(size_t)i);
    for (int i = 0; i < NT; ++i) pthread_join(t[i], nullptr);
    std::printf("%s %d %d %d %d %.0f\n", kind, size, n, NT, bad ? 1 : 0, out);
}
template <int SIZE, int... N> void cols() { (check<col_p(SIZE, N) * col_tw(SIZE, N)>("col", SIZE, N), ...); }
template <int SIZE, int... H> void rows() { (check<row_nt(SIZE, H)>("row", SIZE, H), ...); }
int main() {
    cols<4, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048>();
    cols<8, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024>();
    rows<4, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024>();
    rows<8, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512>();
    check<128>("line", 8, 4);
}
"""


def test_block_sums_use_lanes_that_exist(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    for name, text in (("cuda_runtime.h", CUDA_RUNTIME), ("vector_types.h", CUDA_RUNTIME), ("sums.cpp", PROGRAM)):
        (tmp_path / name).write_text(text)
    exe = tmp_path / "sums"
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "sums.cpp"), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout
    lines = [l.split() for l in out.split("\n") if l]
    assert len(lines) == 15 + 13 + 13 + 11 + 1
    for kind, *v in lines:
        size, n, nt, bad, total = map(float, v)
        assert not bad and total == nt * (nt + 1) / 2, (kind, v)
