"""Addresses of large calls: points beyond 2^31 floats (clouds of more than 715,827,882 points,
which a context may be created for): the grid kernel's read of the input
points, built for the host, and the slots of its tables."""
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


TABLE = r"""
static unsigned long long touched;
static unsigned atomicAnd(unsigned* p, unsigned) { touched = reinterpret_cast<uintptr_t>(p); return ~0u; }
static unsigned long long atomicCAS(unsigned long long* p, unsigned long long e, unsigned long long) {
    touched = reinterpret_cast<uintptr_t>(p);
    return e;
}
constexpr unsigned long long kEmptyKey = ~0ull;
%s
extern "C" long long bit_of(int cap, unsigned cell, unsigned long long* at) {
    long long slot = -1;
    const bool fresh = set_bit(reinterpret_cast<unsigned long long*>(uintptr_t(1) << 20), cap, cell, &slot);
    *at = touched - (1 << 20);
    return fresh ? slot : -2;
}
extern "C" long long key_of(int cap, unsigned long long key, unsigned long long* at, unsigned long long* hash) {
    const long long r = insert_key(reinterpret_cast<unsigned long long*>(uintptr_t(1) << 20), cap, key);
    *at = touched - (1 << 20);
    *hash = slot_mix(key);
    return r & ~(1ll << 62);
}
"""


# tables of the smallest capacity to 2^32 slots (an eighth full with 2^29 points)
@pytest.mark.parametrize("cap", [6, 7, 17, 30, 31, 32])
def test_table_slots(tmp_path, cap):
    mix = H.passage("hav_device.cuh", "__device__ __forceinline__ unsigned long long slot_mix(",
                    "// Slot hash of the block-local sets")
    bit = H.passage("hav_sampler.cu", "__device__ __forceinline__ bool set_bit(", "// The units of a tile whose cells or keys")
    key = H.passage("hav_sampler.cu", "__device__ __noinline__ long long insert_key(",
                    "// A bisection pass over this block's work items")
    lib = H.compile_host(tmp_path, TABLE % (mix + bit + key))
    lib.bit_of.restype = lib.key_of.restype = C.c_longlong
    at, h = C.c_ulonglong(), C.c_ulonglong()
    top = min(64 << cap, 2**32 - 1)
    for cell in [0, 1, 63, 64, top - 1, top // 2, top // 3, (1 << min(cap, 31)) - 1]:
        slot = lib.bit_of(cap, C.c_uint(cell), C.byref(at))
        assert slot == cell % 2**cap
        assert at.value == 8 * slot + 4 * ((cell >> cap) // 32)
    for k in (0, 5, 12345678901234567, 2**63 - 1):
        slot = lib.key_of(cap, C.c_ulonglong(k), C.byref(at), C.byref(h))
        assert slot == h.value >> (64 - cap) and at.value == 8 * slot
