"""Arithmetic of the CUDA sources on the CPU: named functions are taken from a .cu
file as they stand, compiled as plain C++ (round to nearest, nothing fused; the
device may fuse a product and a sum, which only rounds less) and called through
ctypes.  A test of a bound then tests the expressions that run, not a copy."""
import ctypes
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2210_03211_gb300", "csrc")

SHIM = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
using std::min; using std::max; using std::fma; using std::fmaf; using std::isfinite;
#define __device__
#define __forceinline__ inline
struct int4 { int x, y, z, w; };
struct float4 { float x, y, z, w; };
static inline float __uint2float_rn(uint32_t v) { return (float)v; }
static inline double __uint2double_rn(uint32_t v) { return (double)v; }
static inline double __int2double_rn(int32_t v) { return (double)v; }
static inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
template <typename T> static inline T __ldcg(const T *p) { T v; std::memcpy(&v, p, sizeof v); return v; }
struct CommRec { int32_t n; uint32_t m2, vol; int32_t gid; };   // sixteen bytes, read as an int4
struct RunArgs { const CommRec *comm; float *litF; const double *gcc; double cc; };
"""


def constant(text, name):
    return re.search(r"constexpr [^;=]*\b%s = [^;]*;" % name, text).group(0)


def function(text, name):
    m = re.search(r"__device__ __forceinline__ [\w ]*\b%s\(" % name, text)
    start = m.start()
    line = text[start:text.index("\n", start) + 1]
    if line.rstrip().endswith("}"):   # on one line
        return line
    return text[start:text.index("\n}\n", start) + 3]


def build(tmp, functions, constants, exports, files=("lf_internal.cuh", "lf_run.cu")):
    """A ctypes library of `functions` and `constants` of the sources plus `exports`."""
    text = "\n".join(open(os.path.join(CSRC, f)).read() for f in files)
    src = SHIM + "\n".join(constant(text, c) for c in constants) + "\n"
    src += "\n".join(function(text, f) for f in functions) + exports
    cpp, lib = os.path.join(str(tmp), "device_math.cpp"), os.path.join(str(tmp), "device_math.so")
    with open(cpp, "w") as f:
        f.write(src)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", "-shared", "-fPIC",
                           "-o", lib, cpp, "-lm"])
    return ctypes.CDLL(lib)
