// Device helpers of the HAVSampler kernels: memory-order primitives, the
// Eq. 2 voxel key, the Section 3.2 centre distance, hashing, block scans and
// the bounded grid barrier.
#pragma once

#include <cuda_runtime.h>

#include "hav_internal.h"

namespace havk {

constexpr unsigned long long kSpinNs = 2000000000ull;  // 2 s per barrier wait
constexpr unsigned int kSpinIters = 1u << 26;

// ------------------------------------------------------------------ memory ops
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_strong64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int ld_volatile(const int* p) { return *(const volatile int*)p; }
__device__ __forceinline__ unsigned ld_volatile_u(const unsigned* p) { return *(const volatile unsigned*)p; }
__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Monotone map of binary32 onto uint32 (larger float -> larger code).
__device__ __forceinline__ uint32_t enc_f(float x) {
    uint32_t b = __float_as_uint(x);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float dec_f(uint32_t e) {
    return __uint_as_float((e & 0x80000000u) ? (e & 0x7fffffffu) : ~e);
}

// -------------------------------------------------------------------- hashing
// Slot hash: a 64-bit mixer (xor-shift / multiply rounds).  The global table
// indexes by its top bits, the block-local sets by its low bits.
__device__ __forceinline__ unsigned long long slot_mix(unsigned long long k) {
    k ^= k >> 32;
    k *= 0xd6e8feb86659fd93ull;
    k ^= k >> 32;
    k *= 0xd6e8feb86659fd93ull;
    k ^= k >> 32;
    return k;
}
// Slot hash of the block-local sets (any mixing works there): multiplicative
// hashing of the two 32-bit halves, top bits.
__device__ __forceinline__ unsigned smem_hash(unsigned long long k, int log2) {
    const unsigned h = static_cast<unsigned>(k) * 0x9E3779B1u + static_cast<unsigned>(k >> 32) * 0x85EBCA77u;
    return h >> (32 - log2);
}
// Cut-off priority: the SplitMix64 output finaliser (Steele, Lea, Flood 2014).
__device__ __forceinline__ unsigned long long priority(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// Draw `counter` of the SplitMix64 generator (Steele, Lea, Flood 2014)
// started at `seed`: the state advances by the golden-ratio step before each
// output, so draw c finalises seed + (c + 1) * step.
__device__ __forceinline__ unsigned long long random_draw(unsigned seed, unsigned long long counter) {
    return priority(static_cast<unsigned long long>(seed) + (counter + 1ull) * 0x9E3779B97F4A7C15ull);
}

// ------------------------------------------------------------ Eq. 2 voxel keys
// The cell indices are kept as integral binary32 values: floor(x / v) and
// floor(min / v) are exact floats, and their difference u is exact whenever
// the true u is below 2^21 (Sterbenz's lemma when both exceed 2^21 in size,
// small exact integers otherwise); a true u >= 2^21 rounds to a value >= 2^21,
// so the range test below is exact as well.
struct Grid {
    float v[3];
    float fmin[3];
    float r[3];  // RN(1 / v) where it is a normal number, else 0 (floor_div_r)
};

__device__ __forceinline__ bool floor_div(float x, float v, float* f) {
    const float q = __fdiv_rn(x, v);
    const float fl = floorf(q);
    if (!(fabsf(fl) < 4.6e18f)) return false;  // |floor| < 2^62 and finite, as the key range requires
    *f = fl;
    return true;
}

// floor(RN(x / v)), the Eq. 2 cell, through the reciprocal r = RN(1 / v) (a
// normal number): q = RN(x * r) equals x / v up to a relative 2^-23 (two
// roundings), and RN(x / v) is within a relative 2^-24 of x / v, so
// |RN(x / v) - q| < (|q| + 1) 2^-22.  If q lies farther than
// b = (|q| + 1) 2^-21 from both integers around it (b < d = q - floor(q) <
// RN(1 - b)), RN(x / v) lies strictly between them and both floors agree.
// Near an integer (or with |q| >= 2^21, where b exceeds 1, a quotient below
// the normal range, which leaves d within b of 0 or 1, r = 0, or x not
// finite) the quotient is taken correctly rounded and floored.  Either way
// the result is the floor of the correctly rounded quotient.
__device__ __forceinline__ bool floor_div_r(float x, const Grid& g, int a, float* f) {
    const float q = __fmul_rn(x, g.r[a]);
    const float n = floorf(q);
    const float d = __fsub_rn(q, n);
    const float b = __fmul_rn(__fadd_rn(fabsf(q), 1.0f), 4.76837158203125e-07f);  // (|q| + 1) 2^-21
    if (d > b && d < __fsub_rn(1.0f, b)) {
        *f = n;
        return true;
    }
    return floor_div(x, g.v[a], f);
}

// The grid of voxel size v = s * aspect; mn is the bounding box's minimum.
__device__ inline bool make_grid(float s, const float r[3], const float mn[3], Grid* g) {
    for (int a = 0; a < 3; ++a) {
        const float v = __fmul_rn(s, r[a]);
        if (!(v > 0.0f) || !isfinite(v)) return false;
        g->v[a] = v;
        const float rv = __fdiv_rn(1.0f, v);
        g->r[a] = (rv >= 1.17549435e-38f && rv <= 3.40282347e+38f) ? rv : 0.0f;
        if (!floor_div(mn[a], v, &g->fmin[a])) return false;
    }
    return true;
}

// Up to this many cells from the origin the loops below find a cell without a
// division: r = __fdividef(1, v) is within 2 units of its last place of 1 / v, a
// relative 2^-22, so that x * r, rounded to an integer, is within 0.82 of x / v
// (0.5 for the integer, 0.25 for r, 0.07 where the product is rounded first).
// From 2^21 on it is not within 1, and from 2^22 on kMagic below rounds to even
// integers.
constexpr float kFarCells = 1048576.0f;  // 2^20

// floor(RN(x / v)) without a division.  k is an integer within 1 of x / v (the
// nearest to x * r for any r close to 1 / v), |k| < kFarCells; rem = x - k v is then
// exact: a multiple of ulp(v) / 2 (or x itself, k = 0) of size below 2 v, and
// fma rounds once.  Away from the integer, |x / v - k| > |k| 2^-24 (half the
// spacing of binary32 below k at most), RN(x / v)
// lies on the side of k that rem's sign tells.  Near it, RN(x / v) >= k exactly
// when x / v is at least the midpoint of k and the binary32 number below it
// (a tie goes to k, whose last bit is 0), k - 2^(e - 24) with e the exponent of
// that number (k > 0) or of k (k < 0).  Range of v: floor_cells' caller.
__device__ __forceinline__ float floor_near(float x, float v, float k, float rem) {
    if (!(fabsf(k) < kFarCells) || (k == 0.0f && fabsf(x) <= __fmul_rn(v, 1e-30f) && x != 0.0f))
        return floorf(__fdiv_rn(x, v));  // (out of range, or a quotient that may underflow)
    const int kb = __float_as_int(k);
    const float p = __int_as_float((k > 0.0f ? kb - 1 : kb) & 0x7f800000);  // 2^e (0 for k = 0)
    const float t = __fmul_rn(v, __fmul_rn(p, 5.9604644775390625e-08f));    // v 2^(e - 24)
    return rem >= -t ? k : __fsub_rn(k, 1.0f);
}

// A grid over a level's bounding box [mn, mx], with what the counting loops
// need to turn a point of the box into its cell's relative indices without
// divisions or conversions: the cell of every such point lies between the
// cells of mn and mx (the floor of Eq. 2 is monotone), so with `fast` set
// (every axis spans fewer than 2^21 cells, 2^-100 < v < 2^100) no point needs a
// range check.
struct BoxGrid {
    Grid g;                    // (r = 0: cell_key divides)
    float ra[3];               // 1 / v, approximately
    int ci[3];                 // -(kMagicBits + floor(mn / v)) per axis (floor_bits; of no use in a far box)
    float amb;                 // kNear times the largest v: |rem| up to |k| amb (+ amb 2^-70) is near an integer
                               // (infinite where the box leaves kFarCells: every point is near)
    unsigned nx, nxy;          // cells along x, and in an x-y layer (where `cells` is below 2^32)
    unsigned c0;               // ci[0] + nx ci[1] + nxy ci[2] mod 2^32 (cell_number)
    int ok, fast;              // the grid is representable; every cell index is in range
    unsigned long long cells;  // grid cells the box spans
};
constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23: q + kMagic is kMagic + the integer nearest to q for |q| < 2^22
constexpr int kMagicBits = 0x4B400000;
constexpr float kNear = 0x1.01p-24f;  // 2^-24 and what the products of the test may lose

// The bits of kMagic + floor(RN(p / v)) per axis for a point of the box of a
// fast grid; false where an axis is near an integer (one point in 10^5 to 10^6
// of a scene) or the box is far from the origin (near_width: the division then
// decides; 2^22 cells away and more, k would be off by more than |k| amb tells).
// Without conversion or rounding instructions, which run at a fraction of the
// rate of additions: k = (q + kMagic) - kMagic, and the bits of q + kMagic are
// kMagicBits + k; six instructions an axis.
__device__ __forceinline__ bool floor_bits(const float p[3], const float r[3], const float v[3], float amb, int t[3]) {
    const float amb0 = __fmul_rn(amb, 8.4703294725430034e-22f);  // 2^-70 amb
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float s = __fmaf_rn(p[a], r[a], kMagic);
        const float k = __fsub_rn(s, kMagic);
        const float rem = __fmaf_rn(-k, v[a], p[a]);
        ok = ok && fabsf(rem) > __fmaf_rn(fabsf(k), amb, amb0);
        t[a] = __float_as_int(s) + (__float_as_int(rem) >> 31);
    }
    return ok;
}

// Relative cell indices u = floor(RN(p / v)) - floor(RN(mn / v)) near an integer.
static __device__ __noinline__ void floor_cells_near(const float p[3], const BoxGrid& B, int u[3]) {
#pragma unroll 1
    for (int a = 0; a < 3; ++a) {
        const float k = __fsub_rn(__fadd_rn(__fmul_rn(p[a], B.ra[a]), kMagic), kMagic);
        const float f = floor_near(p[a], B.g.v[a], k, __fmaf_rn(-k, B.g.v[a], p[a]));
        u[a] = static_cast<int>(__fsub_rn(f, B.g.fmin[a]));
    }
}

__device__ __forceinline__ void floor_cells(const float p[3], const BoxGrid& B, int u[3]) {
    if (floor_bits(p, B.ra, B.g.v, B.amb, u)) {
#pragma unroll
        for (int a = 0; a < 3; ++a) u[a] += B.ci[a];
    } else {
        floor_cells_near(p, B, u);
    }
}

// What a counting loop keeps of a fast grid of fewer than 2^32 - 1 cells in
// registers, for the number u_x + nx (u_y + ny u_z) of a point's cell.
constexpr unsigned kNoCell = 0xffffffffu;
struct CellMap {
    float r[3], v[3], amb;
    unsigned nx, nxy, c0;
    const BoxGrid* b;
    __device__ __forceinline__ explicit CellMap(const BoxGrid& B)
        : r{B.ra[0], B.ra[1], B.ra[2]}, v{B.g.v[0], B.g.v[1], B.g.v[2]}, amb(B.amb), nx(B.nx), nxy(B.nxy), c0(B.c0),
          b(&B) {}
    // false: near an integer (then near(), below)
    __device__ __forceinline__ bool fast(const float4& q, unsigned* c) const {
        const float p[3] = {q.x, q.y, q.z};
        int t[3];
        const bool ok = floor_bits(p, r, v, amb, t);
        *c = c0 + static_cast<unsigned>(t[0]) + nx * static_cast<unsigned>(t[1]) + nxy * static_cast<unsigned>(t[2]);
        return ok;
    }
    __device__ __forceinline__ unsigned near(const float4& q) const {
        const float p[3] = {q.x, q.y, q.z};
        int u[3];
        floor_cells_near(p, *b, u);
        return static_cast<unsigned>(u[0]) + nx * static_cast<unsigned>(u[1]) + nxy * static_cast<unsigned>(u[2]);
    }
};

// One axis of a BoxGrid of size s * r: v, 1 / v, the cell f0 of mn, and the
// cells the box [mn, mx] has along it (0: 2^21 and more, or not for the loops
// above).  False: not representable.
static __device__ __noinline__ bool box_axis(float s, float r, float mn, float mx, float* v_out, float* rv_out, float* f0,
                                         unsigned* span) {
    const float v = __fmul_rn(s, r);
    *v_out = v;
    *rv_out = 0.0f;
    *f0 = 0.0f;
    *span = 0u;
    if (!(v > 0.0f) || !isfinite(v)) return false;
    const float rv = __fdividef(1.0f, v);  // (approximate: it only has to find a neighbouring integer)
    const bool normal = v > 7.8886090522101181e-31f && v < 1.2676506002282294e30f;  // 2^-100, 2^100
    *rv_out = rv;
    float f[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float x = e ? mx : mn;
        const float k = __fsub_rn(__fadd_rn(__fmul_rn(x, rv), kMagic), kMagic);
        if (normal && fabsf(k) < kFarCells) {
            f[e] = floor_near(x, v, k, __fmaf_rn(-k, v, x));
        } else if (!floor_div(x, v, &f[e])) {
            return e == 1;  // (mx alone: the grid stands, without a span)
        }
        if (e == 0) *f0 = f[0];
    }
    const float u = __fsub_rn(f[1], f[0]);
    if (normal && u >= 0.0f && u < 2097152.0f) *span = static_cast<unsigned>(u) + 1u;
    return true;
}

// What an axis (box_axis) adds to BoxGrid::amb, the largest of the three times
// kNear: v, or infinity where a cell of the box lies `limit` from the origin
// (kFarCells at most).
__device__ __forceinline__ float near_width(float v, float f0, unsigned span, float limit = kFarCells) {
    return (fabsf(f0) < limit && fabsf(f0 + static_cast<float>(span)) < limit) ? v : INFINITY;
}

// key = u_x | u_y << 21 | u_z << 42 with u = floor(x / v) - floor(min / v).
__device__ __forceinline__ bool cell_key(const float p[3], const Grid& g, unsigned long long* key,
                                         float f[3]) {
    unsigned long long k = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (!floor_div_r(p[a], g, a, &f[a])) return false;
        const float u = __fsub_rn(f[a], g.fmin[a]);
        if (!(u >= 0.0f && u < 2097152.0f)) return false;
        k |= static_cast<unsigned long long>(static_cast<unsigned>(u)) << (21 * a);
    }
    *key = k;
    return true;
}

// At most this many voxels are occupied at size s: the grid cells the
// bounding box [mn, mx] spans, floor(mx / v) - floor(mn / v) + 1 per axis (the
// floor of Eq. 2 is monotone in the coordinate).  LLONG_MAX when the grid is
// not representable.
__device__ __forceinline__ long long cell_bound(float s, const float r[3], const float mn[3], const float mx[3]) {
    long long b = 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float v = __fmul_rn(s, r[a]);
        float f0, f1;
        if (!(v > 0.0f) || !isfinite(v) || !floor_div(mn[a], v, &f0) || !floor_div(mx[a], v, &f1)) return LLONG_MAX;
        const float u = __fsub_rn(f1, f0);
        if (!(u >= 0.0f && u < 1048576.0f)) return LLONG_MAX;
        b *= static_cast<long long>(u) + 1;
    }
    return b;
}

// Section 3.2: squared distance to the voxel centre v * (g + 0.5).
__device__ __forceinline__ float centre_d2(const float p[3], const Grid& g, const float f[3]) {
    float d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float c = __fmul_rn(g.v[a], __fadd_rn(f[a], 0.5f));
        d[a] = __fsub_rn(p[a], c);
    }
    const float xy = __fadd_rn(__fmul_rn(d[0], d[0]), __fmul_rn(d[1], d[1]));
    return __fadd_rn(xy, __fmul_rn(d[2], d[2]));
}

// Find or insert `key` in a global open-addressed table by linear probing;
// *fresh tells whether this call inserted it.  Returns the slot, or -1 after
// a full sweep (table full).
__device__ __forceinline__ long long find_or_insert(unsigned long long* T, int cap_log2,
                                                    unsigned long long key, bool* fresh) {
    const unsigned long long mask = (1ull << cap_log2) - 1;
    unsigned long long slot = slot_mix(key) >> (64 - cap_log2);
    *fresh = false;
    for (unsigned long long probe = 0; probe <= mask; ++probe) {
        const unsigned long long cur = ld_strong64(T + slot);
        if (cur == key) return static_cast<long long>(slot);
        if (cur == kEmptyKey) {
            const unsigned long long prev = atomicCAS(T + slot, kEmptyKey, key);
            if (prev == kEmptyKey) {
                *fresh = true;
                return static_cast<long long>(slot);
            }
            if (prev == key) return static_cast<long long>(slot);
        }
        slot = (slot + 1) & mask;
    }
    return -1;
}

// find_or_insert for U keys at once: the first probe of every key is issued
// before any result is used (memory-level parallelism); keys equal to
// kEmptyKey are skipped.  slot[u] = -1 after a full sweep (table full).
template <int U>
__device__ __forceinline__ void find_or_insert_batch(unsigned long long* const (&T)[U], int cap_log2,
                                                     const unsigned long long (&key)[U],
                                                     long long (&slot)[U], bool (&fresh)[U]) {
    const unsigned mask = static_cast<unsigned>((1ull << cap_log2) - 1);
    unsigned sl[U];
    unsigned long long cur[U];
    // every probe is a compare-and-swap (it returns the slot's key whether or
    // not it swaps: one round trip per probe), and the probes of all U keys
    // are in flight together
#pragma unroll
    for (int u = 0; u < U; ++u) {
        sl[u] = static_cast<unsigned>(slot_mix(key[u]) >> (64 - cap_log2));
        cur[u] = (key[u] != kEmptyKey) ? atomicCAS(T[u] + sl[u], kEmptyKey, key[u]) : kEmptyKey;
    }
    bool open[U];
    bool any = false;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        fresh[u] = false;
        slot[u] = -1;
        open[u] = false;
        if (key[u] == kEmptyKey) continue;
        if (cur[u] == kEmptyKey || cur[u] == key[u]) {
            slot[u] = sl[u];
            fresh[u] = (cur[u] == kEmptyKey);
        } else {
            open[u] = true;
            any = true;
        }
    }
    // collisions: linear probing from the next slot
    for (unsigned probe = 1; any && probe <= mask; ++probe) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (!open[u]) continue;
            sl[u] = (sl[u] + 1) & mask;
            cur[u] = atomicCAS(T[u] + sl[u], kEmptyKey, key[u]);
        }
        any = false;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (!open[u]) continue;
            if (cur[u] == kEmptyKey || cur[u] == key[u]) {
                slot[u] = sl[u];
                fresh[u] = (cur[u] == kEmptyKey);
                open[u] = false;
            } else {
                any = true;
            }
        }
    }
}

// Warp-aggregated append to a shared-memory list: every lane of the warp
// calls it (flag false for lanes with nothing to add); returns the lane's
// position, or -1.
template <typename T>
__device__ __forceinline__ int warp_append(bool flag, T* counter) {
    const unsigned m = __ballot_sync(0xffffffffu, flag);
    if (!m) return -1;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    T base = 0;
    if (lane == leader) base = atomicAdd(counter, static_cast<T>(__popc(m)));
    base = __shfl_sync(0xffffffffu, base, leader);
    return flag ? static_cast<int>(base) + __popc(m & ((1u << lane) - 1u)) : -1;
}

// As warp_append with one counter per key (key indexes counters): the lanes
// of each key share one atomic add.  Whole warp calls, converged.
template <typename T>
__device__ __forceinline__ int warp_append_keyed(bool flag, int key, T* counters) {
    const unsigned m = __ballot_sync(0xffffffffu, flag);
    if (!m) return -1;
    int pos = -1;
    if (flag) {
        const int lane = threadIdx.x & 31;
        const unsigned grp = __match_any_sync(m, key);
        const int leader = __ffs(grp) - 1;
        T base = 0;
        if (lane == leader) base = atomicAdd(counters + key, static_cast<T>(__popc(grp)));
        base = __shfl_sync(m, base, leader);
        pos = static_cast<int>(base) + __popc(grp & ((1u << lane) - 1u));
    }
    return pos;
}

// Block-local set in shared memory (a filter in front of the global table):
// returns the slot holding `key` and whether this call inserted it, or -1
// when the probe limit is reached (the caller then goes to the global table).
template <int kSlots>
__device__ __forceinline__ int smem_insert(unsigned long long* set, unsigned long long key, bool* fresh) {
    static_assert(kSlots > 1 && (kSlots & (kSlots - 1)) == 0, "power of two");
    unsigned slot = smem_hash(key, __builtin_ctz(kSlots));
    *fresh = false;
#pragma unroll 1
    for (int probe = 0; probe < 32; ++probe) {
        const unsigned long long cur = set[slot];
        if (cur == key) return static_cast<int>(slot);
        if (cur == kEmptyKey) {
            const unsigned long long prev = atomicCAS(set + slot, kEmptyKey, key);
            if (prev == kEmptyKey) {
                *fresh = true;
                return static_cast<int>(slot);
            }
            if (prev == key) return static_cast<int>(slot);
        }
        slot = (slot + 1) & (kSlots - 1);
    }
    return -1;
}

// ------------------------------------------------ Section 3.3 search steps
// The next size of a search with bracket (lo, hi): a pending first guess,
// 2 lo while doubling up (the guided start), else the bisection midpoint in
// binary32.
__device__ __forceinline__ float next_size(float lo, float hi, bool up, float first) {
    if (first > 0.0f) return first;
    const float d = __fmul_rn(lo, 2.0f);
    if (up && d < hi) return d;
    return __fmul_rn(__fadd_rn(lo, hi), 0.5f);
}

// Size at node c of the search subtree below the current state (heap order:
// child 2c + 1 follows a count below m_l, 2c + 2 a count above k_max): the
// path from the root follows the bits of c + 1 below its leading one (0: too
// few voxels, hi = s; 1: too many, lo = s), each step as next_size takes it.
__device__ __forceinline__ float cand_size(float lo, float hi, bool up, float first, int c) {
    const int x = c + 1;
    const int depth = 31 - __clz(x);
    float s = next_size(lo, hi, up, first);
#pragma unroll 1
    for (int b = depth - 1; b >= 0; --b) {
        if ((x >> b) & 1) {
            lo = s;
        } else {
            hi = s;
            up = false;
        }
        s = next_size(lo, hi, up, 0.0f);
    }
    return s;
}

// Eq. 3 budget of layer l (0-based).
__device__ __forceinline__ long long layer_budget(long long m, int layers, int ratio, int l) {
    long long S = 0, pw = 1;
#pragma unroll 1
    for (int i = 0; i < layers; ++i) {
        S += pw;
        pw *= ratio;
    }
    long long used = 0;
    pw = 1;
#pragma unroll 1
    for (int i = 0; i < layers - 1; ++i) {
        const long long mi = m * pw / S;
        if (i == l) return mi;
        used += mi;
        pw *= ratio;
    }
    return m - used;
}

// ------------------------------------------------------------ block helpers
template <typename T>
__device__ __forceinline__ T warp_incl_scan(T x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Exclusive scan over the block; *total receives the sum.  All threads call it.
template <typename T, int kBlock = kThreads>
__device__ T block_excl_scan(T v, T* total, T* scratch /* >= 32 */) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int kWarps = kBlock / 32;
    T x = warp_incl_scan(v);
    if (lane == 31) scratch[wid] = x;
    __syncthreads();
    if (wid == 0) {
        T w = (lane < kWarps) ? scratch[lane] : T(0);
        w = warp_incl_scan(w);
        scratch[lane] = w;
    }
    __syncthreads();
    const T before = wid ? scratch[wid - 1] : T(0);
    *total = scratch[kWarps - 1];
    __syncthreads();
    return before + x - v;
}

// Sum over the block (every thread receives it).
__device__ __forceinline__ unsigned block_sum(unsigned v, unsigned* scratch /* >= 32 */) {
    const unsigned w = __reduce_add_sync(0xffffffffu, v);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) scratch[wid] = w;
    __syncthreads();
    unsigned t = 0;
#pragma unroll
    for (int k = 0; k < kThreads / 32; ++k) t += scratch[k];
    __syncthreads();
    return t;
}

// Grid barrier with a bounded wait.  Arrival is a release reduction on a
// counter that only grows within a launch (zeroed by the host before it);
// barrier number e of the launch completes when the counter reaches
// e * nblocks, so no block has to act as the last arriver.  Returns false
// (for the whole block) when this or another block gave up; the caller then
// leaves the kernel.
__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Grid barrier that also sums one count over the blocks.  Each block adds
// 2^48 + add to `word`; the barrier is complete when the arrival field (bits
// 48..63, mod 2^16) reaches uses * nblocks.  Between two uses of the same
// word every block has passed a barrier on the other word, so no block adds
// to it again before all have read it: the change of the low 48 bits since
// this block's last reading is exactly this barrier's sum.  The caller keeps
// the low field below 2^48.  Bounded like grid_wait_impl.
//
// Both barriers come in two halves.  The arrival orders every write the block
// made before it; work between the arrival and the wait (writes that only the
// block's next arrival has to publish) overlaps the wait for the other blocks.
__device__ inline void fused_arrive_impl(unsigned long long* word, unsigned* uses, unsigned long long add) {
    __syncthreads();
    if (threadIdx.x == 0) {
        *uses += 1u;
        const unsigned long long inc = (1ull << 48) | add;
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(word), "l"(inc) : "memory");
    }
}

__device__ inline bool fused_wait_impl(unsigned long long* word, GlobalHdr* gh, unsigned nblocks,
                                       const unsigned* uses, unsigned long long* last,
                                       unsigned long long* delta, int* s_flag) {
    if (threadIdx.x == 0) {
        int fail = 0;
        const unsigned target = (*uses * nblocks) & 0xffffu;
        const unsigned long long t0 = globaltimer();
        unsigned long long v = 0;
        int ab = 0;
        for (unsigned it = 0;; ++it) {
            ab = ld_volatile(&gh->abort);  // in flight together with the poll
            v = ld_acquire64(word);
            if ((static_cast<unsigned>(v >> 48) & 0xffffu) == target) break;
            if ((it & 31) == 31) {
                if (ab || it > kSpinIters || globaltimer() - t0 > kSpinNs) {
                    fail = 1;
                    break;
                }
            }
            if (it > 64) __nanosleep(32);
        }
        if (fail) {
            atomicExch(&gh->abort, 1);
            atomicCAS(&gh->status, 0, static_cast<int>(HAV_ERR_TIMEOUT));
        }
        const unsigned long long c = v & ((1ull << 48) - 1ull);
        *delta = c - *last;
        *last = c;
        *s_flag = fail | ab;
    }
    __syncthreads();
    return *s_flag == 0;
}

__device__ inline void grid_arrive_impl(Barrier* bar, unsigned* epoch) {
    __syncthreads();
    if (threadIdx.x == 0) {
        *epoch += 1u;
        // The block barrier above orders every thread's writes before this
        // release; the acquire load in the wait orders them before every
        // thread's reads after its closing block barrier.  No further fence
        // is needed.
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&bar->count) : "memory");
    }
}

__device__ inline bool grid_wait_impl(Barrier* bar, GlobalHdr* gh, unsigned nblocks, const unsigned* epoch,
                                      int* s_flag) {
    if (threadIdx.x == 0) {
        int fail = 0;
        const unsigned target = *epoch * nblocks;
        const unsigned long long t0 = globaltimer();
        int ab = 0;
        for (unsigned it = 0;; ++it) {
            // the abort flag is read in the same round trip as the poll (a
            // relaxed load ahead of the acquire), not after the barrier
            ab = ld_volatile(&gh->abort);
            if (ld_acquire(&bar->count) >= target) break;
            if ((it & 31) == 31) {
                if (ab || it > kSpinIters || globaltimer() - t0 > kSpinNs) {
                    fail = 1;
                    break;
                }
            }
            if (it > 64) __nanosleep(32);
        }
        if (fail) {
            atomicExch(&gh->abort, 1);
            atomicCAS(&gh->status, 0, static_cast<int>(HAV_ERR_TIMEOUT));
        }
        *s_flag = fail | ab;
    }
    __syncthreads();
    return *s_flag == 0;
}

__device__ inline bool grid_sync_impl(Barrier* bar, GlobalHdr* gh, unsigned nblocks, unsigned* epoch,
                                      int* s_flag) {
    grid_arrive_impl(bar, epoch);
    return grid_wait_impl(bar, gh, nblocks, epoch, s_flag);
}

}  // namespace havk
