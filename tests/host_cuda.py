"""Device headers compiled for the host: a stand-in for the CUDA runtime header with
the keywords empty and the intrinsics that the headers use as their IEEE
definitions, so that device arithmetic can be tested without a GPU."""
import os
import subprocess


ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2303_14280_gb300", "csrc")

RUNTIME = r"""
#pragma once
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstring>
#define __device__
#define __host__
#define __global__
#define __shared__ static
#define __forceinline__ inline
struct float2 { float x, y; };
struct double2 { double x, y; };
struct float4 { float x, y, z, w; };
struct dim3_ { unsigned x, y, z; };
static dim3_ threadIdx{0, 0, 0}, blockDim{1, 1, 1};
typedef int cudaError_t;
typedef struct st_* cudaStream_t;
inline void __syncthreads() {}
inline float2 make_float2(float x, float y) { return {x, y}; }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
inline float __double2float_rn(double a) { return (float)a; }
inline long long __double_as_longlong(double a) { long long r; std::memcpy(&r, &a, 8); return r; }
inline double __longlong_as_double(long long a) { double r; std::memcpy(&r, &a, 8); return r; }
inline int __double2loint(double a) { return (int)(unsigned)(__double_as_longlong(a) & 0xffffffffll); }
inline int __double2hiint(double a) { return (int)(__double_as_longlong(a) >> 32); }
inline double __hiloint2double(int h, int l) {
  return __longlong_as_double((long long)(((unsigned long long)(unsigned)h << 32) | (unsigned)l));
}
inline float rsqrtf(float a) { return 1.0f / std::sqrt(a); }
using std::fma;
"""


def run(tmp_path, source):
    """Compile the source with the stand-in header and return what it prints."""
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    src, exe = tmp_path / "harness.cpp", tmp_path / "harness"
    src.write_text(source)
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", str(tmp_path), "-I", CSRC,
                        "-I", os.path.join(ROOT, "include"), str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
