"""Offsets of points beyond 2^31 floats (clouds of more than 715,827,882 points,
which a context may be created for): the grid kernel's read of the input
points, built for the host."""
import ctypes as C

import pytest

import _host_cuda as H

CODE = r"""
#include <vector>
#define __ldg host_ldg
struct { unsigned x; } threadIdx;
constexpr int kThreads = 512;
static int min(int a, int b) { return a < b ? a : b; }
static std::vector<unsigned long long> reads;
static float host_ldg(const float* p) { reads.push_back(reinterpret_cast<uintptr_t>(p)); return 0.0f; }
%s
// addresses read, from the points' own, for thread tid of a block with points [a, b)
extern "C" int reads_of(int tid, int a, int b, unsigned long long* out, int room) {
    const uintptr_t base = 1 << 20;
    threadIdx.x = static_cast<unsigned>(tid);
    reads.clear();
    for_points(reinterpret_cast<const float*>(base), a, b, [](int, const float*) {});
    int n = 0;
    for (unsigned long long r : reads)
        if (n < room) out[n++] = r - base;
    return n;
}
"""


@pytest.mark.parametrize("first", [0, 715827800, 2**30 - 5000])
def test_input_points(tmp_path, first):
    text = H.passage("hav_sampler.cu", "template <typename F>\n__device__ __forceinline__ void for_points(",
                     "// The boxes of this block's work items of the level")
    lib = H.compile_host(tmp_path, CODE % text)
    out = (C.c_ulonglong * 20000)()
    for tid in (0, 77, 511):
        n = lib.reads_of(tid, first, first + 3001, out, 20000)
        seen = set(out[:n])
        want = {4 * (3 * i + a) for i in range(first + tid, first + 3001, 512) for a in range(3)}
        last = {4 * (3 * (first + 3000) + a) for a in range(3)}  # (read in place of points behind the last)
        assert want <= seen <= want | last
