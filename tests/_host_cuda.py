"""Device code of the library compiled for the host: a passage of a source file
under a small shim of the CUDA intrinsics it uses (plain binary32 operations,
no contraction), so that its arithmetic is tested as it stands, without a GPU."""
from __future__ import annotations

import ctypes
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_14306_gb300", "csrc")

SHIM = r"""
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstring>
using std::isfinite;
#define __device__
#define __forceinline__ inline
#define __noinline__ __attribute__((noinline))
struct float4 { float x, y, z, w; };
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fdiv_rn(float a, float b) { return a / b; }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static inline int __float_as_int(float x) { int i; memcpy(&i, &x, 4); return i; }
static inline float __int_as_float(int i) { float x; memcpy(&x, &i, 4); return x; }
// a quotient off by ULPS units in its last place (2 at most for the intrinsic)
#ifndef ULPS
#define ULPS 0
#endif
static inline float __fdividef(float a, float b) { return __int_as_float(__float_as_int(a / b) + ULPS); }
"""


def passage(name: str, first: str, behind: str) -> str:
    """The text of csrc/name from `first` up to `behind` (each found once)."""
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    assert text.count(first) == 1 and text.count(behind) == 1, (first, behind)
    return text[text.index(first):text.index(behind)]


def compile_host(directory, code: str, *flags: str) -> ctypes.CDLL:
    src, lib = os.path.join(directory, "host.cpp"), os.path.join(directory, "host.so")
    with open(src, "w") as f:
        f.write(SHIM + code)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fwrapv", "-fno-strict-aliasing", "-shared",
                    "-fPIC", *flags, src, "-o", lib], check=True, capture_output=True, text=True)
    return ctypes.CDLL(lib)
