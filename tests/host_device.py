"""Device code of csrc/*.cuh run on the host: the headers, with their inline
PTX blanked, compiled by g++ against stand-ins for what they use of CUDA; one
thread per lane, barriers for __syncwarp, __syncthreads and shuffles.  For
code that touches no global state and whose waits are the barriers alone."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1011_3582_gb300", "csrc")

RUNTIME = r"""
#pragma once
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <pthread.h>
#include <vector>
#define __host__
#define __device__
#define __global__
#define __forceinline__ inline
#define __shared__
#define __constant__
#define __grid_constant__
#define __align__(n)
#define __launch_bounds__(...)
struct float2 { float x, y; };
struct double2 { double x, y; };
struct float4 { float x, y, z, w; };
struct uint4 { unsigned x, y, z, w; };
inline float2 make_float2(float x, float y) { return {x, y}; }
inline double2 make_double2(double x, double y) { return {x, y}; }
inline float4 make_float4(float x, float y, float z, float w) { return {x, y, z, w}; }
struct Dim { unsigned x = 0, y = 0, z = 0; };
inline thread_local Dim threadIdx, blockIdx;
inline Dim blockDim, gridDim;
inline double lane_value[2048];
// a block of blockDim.x threads; threads of one warp that take part in a
// shuffle or a __syncwarp meet at the warp's barrier, so all of them have to
inline pthread_barrier_t block_barrier, warp_barrier[64];
inline void run_block(int nt, const std::function<void()> &body) {
    blockDim.x = nt;
    pthread_barrier_init(&block_barrier, nullptr, nt);
    for (int w = 0; 32 * w < nt; ++w) pthread_barrier_init(&warp_barrier[w], nullptr, nt - 32 * w < 32 ? nt - 32 * w : 32);
    struct Arg { int i; const std::function<void()> *f; };
    std::vector<pthread_t> t(nt);
    std::vector<Arg> a(nt);
    for (int i = 0; i < nt; ++i) {
        a[i] = {i, &body};
        pthread_create(&t[i], nullptr, [](void *p) -> void * {
            threadIdx.x = ((Arg *)p)->i;
            (*((Arg *)p)->f)();
            return nullptr;
        }, &a[i]);
    }
    for (auto &x : t) pthread_join(x, nullptr);
}
inline void warp_meet() { pthread_barrier_wait(&warp_barrier[threadIdx.x >> 5]); }
inline void __syncwarp(unsigned = ~0u) { warp_meet(); }
inline void __syncthreads() { pthread_barrier_wait(&block_barrier); }
inline int __syncthreads_or(int) { __syncthreads(); return 0; }
template <typename T> T shfl(T v, int src) {
    lane_value[threadIdx.x] = v;
    warp_meet();
    const T o = src >= 0 && src < (int)blockDim.x ? (T)lane_value[src] : (T)NAN;
    warp_meet();
    return o;
}
template <typename T> T __shfl_xor_sync(unsigned, T v, int m) { return shfl(v, (int)threadIdx.x ^ m); }
template <typename T> T __shfl_down_sync(unsigned, T v, int d) { return shfl(v, (int)threadIdx.x + d); }
template <typename T> T __ldg(const T *p) { return *p; }
template <typename T> T __ldcs(const T *p) { return *p; }
template <typename T> void __stcs(T *p, T v) { *p = v; }
inline float __fmul_rn(float a, float b) { volatile float r = a * b; return r; }
inline float __fadd_rn(float a, float b) { volatile float r = a + b; return r; }
inline float __fsub_rn(float a, float b) { volatile float r = a - b; return r; }
inline float2 __fadd2_rn(float2 a, float2 b) { return {a.x + b.x, a.y + b.y}; }
inline float __uint_as_float(unsigned u) { float v; std::memcpy(&v, &u, 4); return v; }
inline unsigned __float_as_uint(float v) { unsigned u; std::memcpy(&u, &v, 4); return u; }
inline long long __double_as_longlong(double v) { long long u; std::memcpy(&u, &v, 8); return u; }
inline size_t __cvta_generic_to_shared(const void *p) { return (size_t)p; }
inline int atomicOr(int *p, int v) { const int o = *p; *p |= v; return o; }
inline int min(int a, int b) { return a < b ? a : b; }
inline int max(int a, int b) { return a > b ? a : b; }
struct CUtensorMap { char b[128]; };
namespace cooperative_groups {
struct Cluster {
    unsigned block_rank() const { return 0; }
    template <typename T> T *map_shared_rank(T *p, int) const { return p; }
};
inline Cluster this_cluster() { return {}; }
}
"""


def blank_asm(text):
    """Every asm statement replaced by an empty one."""
    out, i = [], 0
    for m in re.finditer(r"\basm(\s+volatile)?\s*\(", text):
        if m.start() < i:
            continue
        out.append(text[i:m.start()] + "(void)0")
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0) if text[i] != '"' else 0
            if text[i] == '"':
                i = text.index('"', i + 1)
            i += 1
    return "".join(out) + text[i:]


def run(tmp_path, program, timeout=600):
    """The output lines of `program` (C++ source), split into words."""
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    for path in glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")):
        text = blank_asm(open(path).read()).replace("uint32_t ok;", "uint32_t ok = 1;")
        (tmp_path / os.path.basename(path)).write_text(text)
    (tmp_path / "runtime_stand_in.h").write_text(RUNTIME)
    for name in ("cuda.h", "cuda_runtime.h", "vector_types.h", "cooperative_groups.h"):
        (tmp_path / name).write_text('#include "runtime_stand_in.h"\n')
    (tmp_path / "program.cpp").write_text(program)
    exe = tmp_path / "program"
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-pthread", "-I", str(tmp_path), str(tmp_path / "program.cpp"), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=timeout).stdout
    return [l.split() for l in out.split("\n") if l]
