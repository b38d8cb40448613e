// Small levels on thread-block clusters, and on single CTAs.
//
// The same sampler as hav_chain_kernel (Sections 3.2-3.4 and Eq. 3, with the
// same readings), for levels of at most 32,768 points: one cluster of Q = 8
// or 16 CTAs per segment (16 where every segment's cluster runs at once; 16 is
// above the portable cluster size and is used where the device schedules it),
// or one CTA per segment (Q = 1).
//
// The search is spread over the cluster by candidate, not by point: every CTA
// sees all points of the level and counts the voxels of one size, a node of
// the subtree of the next log2(Q) steps below the search's state, in its own
// shared memory.  A pass then takes log2(Q) steps (4 on 16 CTAs), exchanges
// nothing but Q counts, and ends with one cluster barrier.  With the points
// spread over the CTAs instead, every point's key went to the CTA that owned
// its voxel, a compare-and-swap round trip of about 1 us per probe through
// distributed shared memory, and a pass of one step took 4.2-5.6 us (measured
// on GB300, 16 CTAs, 16,384-20,876 points).  On one CTA the count costs no
// atomics and nothing to empty, and a warp prepares the next grids meanwhile: a
// pass over 1,000 points 2.3 -> 1.5 us.  What bounds both is latency and the
// instructions of a point: of a pass of 1,000 points, 1.3 us are short serial
// sections of a few dozen instructions between barriers; of one of 20,876
// points on 16 CTAs, 13 us in the finest sizes of a LiDAR scan, 6 us are the
// points' cells (each CTA sees all of them: 36 instructions a point), 4 the
// look at the words (a third of it their random bank conflicts), 1.5 the
// undecided points and the rest such sections.  Measured on GB300, whole calls:
// 1,000-point room to 250 57.5 -> 43.7 us, 16,384 uniform points to 4,096 80.4
// -> 63.6 us, LiDAR chain 20,876 -> 16,384 -> 4,096 -> 1,024 -> 512 364 -> 289
// us, 64 clouds of 1,000-4,000 points, two levels, 144 -> 105 us.
//
// The selection at s* is spread by voxel: every CTA hands the points of its share
// to the CTAs that their voxels hash to, as records that those fetch, so that the
// table of a voxel's closest point is in a CTA's own shared memory too.  Only the
// records, the cut-off histograms, the boundary bin's candidates and the counts of kept points
// cross the cluster, and the taken marks through the staged points in global
// memory (a level of at most kPtsSmem points also has a copy in shared memory,
// re-marked at the start of a layer; Q = 1 works on that copy alone).

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "hav.h"
#include "hav_device.cuh"
#include "hav_internal.h"

namespace cg = cooperative_groups;

namespace havk {
namespace {

// Threads per CTA: half of what would fit, for 128 registers a thread (no
// spills) and half the warps to pass through a phase's fixed instructions; the
// kernel's phases are short, and instruction fetches and barriers bounded them
// at 1,024 threads.
constexpr int kST = 512;
constexpr int kWarps = kST / 32;
constexpr int kPtsSmem = 4096;   // levels of at most this many points have a copy in shared memory (64 KB)
constexpr int kSelMax = 8192;    // slots of a CTA's part of the selection table at most (128 KB)
constexpr int kMaxQ = 16;        // largest cluster
constexpr long long kWideMin = 8192;  // points from which a launch may take the kernels built for kWide
constexpr int kCutBits = 6;      // cut-off histogram over the top priority bits
constexpr int kCutBins = 1 << kCutBits;
constexpr int kOpenA = kSelMax / 8 * 7;  // undecided points of a pass that are listed (in later rounds, alternately the rest)
constexpr unsigned kManyOpen = 0xffffffffu;
constexpr int kMaxOpen = 32;     // undecided points of a pass that a warp compares with one another
constexpr int kCandAll = 1024;   // boundary-bin candidates of the cluster that every CTA receives
constexpr size_t kPtsBytes = static_cast<size_t>(kPtsSmem) * 16;
constexpr size_t kTabBytes = static_cast<size_t>(kSelMax) * 16;
static_assert(kSmallMax <= 8 * (kSelMax / 2), "an 8-CTA cluster's parts are at most half full on average");
static_assert(kSmallMax <= 32768, "a point index fits 16 bits, also as index + 1");
// every point of a level has its cell number and at least one 16-bit word, or a slot
static_assert((kPtsBytes + kTabBytes) / 4 >= kSmallMax + kSmallMax / 2 && kTabBytes / 4 > 2 * kPtsSmem, "pass table");
// the selection's tables and the records of a share, where n > kPtsSmem and where not
static_assert(16 * (2 * kSmallMax / 8) + 16 * (kSmallMax / 8) <= kPtsBytes + kTabBytes, "selection, large level");
static_assert(16 * (2 * kPtsSmem / 8) + 16 * (kPtsSmem / 8) <= kTabBytes, "selection, small level");

template <int Q>
__host__ __device__ constexpr int qlog2() {
    return Q == 16 ? 4 : (Q == 8 ? 3 : 0);
}

// How a pass counts distinct voxels among the cells the bounding box spans.
//   kDirect, kHash  Every point writes its cell number beside it and its index
//            into its cell's 16-bit word (kDirect: one word per cell; kHash: a
//            hashed word) and, behind a block barrier, reads the word back.
//            Its own index: it stands for the cell.  Another's: that point's
//            cell tells whether the two share it; if not (kHash), all points of
//            the cell go on to the next round, under another hash.  Each word's
//            cell ends with its round, so every round ends some.  No atomics,
//            and nothing to empty: no word is read that this round did not
//            write.  (A bitmap and a table of cell numbers, one shared-memory
//            atomic per point, took 1.7 to 2.5 times as long: neighbouring
//            points' atomics meet in one word.)
//   kWide    (2^32 cells and more, in the kernels built for it) kHash on the cell
//            numbers modulo 2^32.  A point that reads one of its own number compares the cells
//            themselves (wide_check), a look at the points that share a voxel.
//            Where the cells differ, all points of the one that the word does not
//            stand for do so (equal numbers read the same word): they are
//            collected with their keys, and their distinct keys added.  In a
//            scan hardly two cells share a number.  (16 CTAs, a LiDAR scan of
//            24,000 points to 97 of 100, one layer: 213 us by kIndex, 113 so; a
//            pass 30 us, 17 to 21 by kHash.)
//   kIndex   (a cell index that may be out of range, more points with a shared
//            number than are collected, or 2^32 cells elsewhere) open addressing
//            on (16 key bits, point index) with atomics, compared through the
//            indexed point's key
// kWide's code is in kernels of its own (template argument kW), taken for large
// budgets (launch_small): in one kernel with the other ways it cost registers that
// every pass then spilled (16,384 uniform points to 4,096, caches cold, 68.3 us
// without it, 72.0 with it).
enum : int { kSkip = 0, kDirect = 1, kHash = 2, kWide = 3, kIndex = 4 };

// A pass's size, its grid over the level's box, and how a pass counts it.
struct PassGrid {
    BoxGrid bg;
    float sv;
    int mode;
    unsigned nslots;  // 16-bit words of kDirect, kHash and kWide
    int far;          // the box leaves kFarLoop: far_cells
};

struct SmallSmem {
    // written by every CTA into every CTA's copy, at its rank
    unsigned long long pass[2][kMaxQ];  // count (low 32 bits) and errors of a pass (1: range), by pass parity
    uint32_t box[kMaxQ][6];             // bounding box codes of its share of the level's points
    int bad[kMaxQ];                     // a coordinate of its share is not finite
    int part_cnt[kMaxQ];                // its count, for prefixes (shortfall, compaction)
    int2 rec[kMaxQ];                    // its records for this CTA: first, count
    uint32_t hist[kMaxQ][kCutBins];     // its voxels per cut-off bin
    unsigned errs[kMaxQ];               // its selection errors (1: range, 2: table full)
    int ncand[kMaxQ];                   // its boundary-bin candidates
    // this CTA's
    float mn[3], mx[3], s_hi;
    int nonfinite;
    int ml[kMaxLayers], kmax[kMaxLayers];
    int pre[kMaxIters];       // counts at s_hi / 2^(k+1) of this level's earlier layers (-1: none)
    float st_s[kMaxIters];    // the sizes s_hi / 2^(k+1), and the cells the box spans at them
    long long st_b[kMaxIters];
    // the search of a layer (held by warp 0)
    float lo, hi, first, s_star;
    float node_s[kMaxQ];      // the sizes of a pass's nodes
    float tr_s[kMaxIters];    // its steps for the trace, written out once it has ended
    int tr_K[kMaxIters];
    int up, pre_on, t, skipped, accepted, err, go;
    // Q > 1: the grid of this CTA's node and the root's; Q = 1: the grids after
    // either outcome of a pass, by pass parity; [4] the selection's
    PassGrid pg[5];
    unsigned wcnt[2][kWarps];  // counts of the warps, by pass parity
    unsigned acc_err;
    uint32_t own_hist[kCutBins];
    int bin_cnt[kMaxQ];  // records of this CTA's share by owner: counts, then places
    unsigned nlist;           // slots the selection filled
    int nopen[2];             // undecided points of a kHash round, by its parity
    int ntwin;                // points of cells that share another's number (kWide)
    unsigned own_cand;        // this CTA's boundary-bin candidates, at the front of the slot list
    int cut_bin, cut_below, kstar;
    unsigned eb;
    int red_i[kWarps];
    uint32_t redu[6][kWarps];
};

// Shared memory: the points of a level of at most kPtsSmem (on larger levels
// more room for the tables), the tables, the received candidates, the list of
// selected slots, the rest.
constexpr size_t kListOff = kPtsBytes + kTabBytes + 8 * static_cast<size_t>(kCandAll);
constexpr size_t kSmOff = kListOff + 2 * static_cast<size_t>(kSelMax);
constexpr size_t kSmallDyn = kSmOff + sizeof(SmallSmem);
static_assert(kSmallDyn <= 227 * 1024, "shared memory of one CTA");
extern __shared__ __align__(16) unsigned char dyn[];
__device__ __forceinline__ SmallSmem& smem() { return *reinterpret_cast<SmallSmem*>(dyn + kSmOff); }

// The share of a level's points that CTA r of the cluster stages and compacts.
template <int Q>
__device__ __forceinline__ int part_start(int n, int r) {
    return n / Q * r + n % Q * r / Q;
}

// CTA r's copy of a shared-memory variable (this CTA's own when Q = 1).
template <int Q, typename T>
__device__ __forceinline__ T* at_rank(cg::cluster_group& cl, T* p, int r) {
    if constexpr (Q == 1) {
        (void)cl;
        (void)r;
        return p;
    } else {
        return cl.map_shared_rank(p, r);
    }
}

template <int Q>
__device__ __forceinline__ void csync(cg::cluster_group& cl) {
    if constexpr (Q == 1) {
        (void)cl;
        __syncthreads();
    } else {
        cl.sync();
    }
}

// The cluster barrier in parts: an arrival that orders the thread's earlier
// writes, one that orders nothing, and the wait.
__device__ __forceinline__ void cluster_arrive_release() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive_relaxed() {
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__device__ __forceinline__ void seg_fail(SegHdr* sh, GlobalHdr* gh, int seg, int code) {
    atomicCAS(&sh[seg].status, 0, code);
    atomicCAS(&gh->status, 0, code);
}

// Phase timer (HAV_FLAG_PHASE_TIMES): thread 0 of the first cluster's CTA 0
// appends (time, tag) records after the grid kernel's, tag = phase << 24 |
// level << 16 | layer << 8 | pass with the grid kernel's phase numbers.  The
// records of a call are a prefix of the zeroed buffer, so the first free one
// is found by bisection.
struct SmallTimer {
    unsigned long long* rec;
    int cap, n;
    __device__ __noinline__ void open(const Plan& P, bool on) {
        rec = on ? P.ptimes : nullptr;
        cap = P.ptimes_cap;
        n = 0;
        if (!rec) return;
        int lo = 0, hi = cap;  // rec[2k] != 0 exactly for k < n
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (rec[2 * mid] != 0ull) lo = mid + 1;
            else hi = mid;
        }
        n = lo;
        if (n == 0) mark(0u);  // no earlier kernel in this call: the start record
    }
    __device__ __noinline__ void mark(unsigned tag) {
        if (rec && n < cap) {
            rec[2 * n] = globaltimer();
            rec[2 * n + 1] = tag;
            ++n;
        }
    }
    __device__ __forceinline__ void mark(int phase, int level, int layer, int pass) {
        if (rec)
            mark((static_cast<unsigned>(phase) << 24) | (static_cast<unsigned>(level) << 16) |
                 (static_cast<unsigned>(layer) << 8) | static_cast<unsigned>(pass));
    }
};

// Exclusive prefix of v over the block, and its total.
__device__ __noinline__ int scan_int(int v, int* total) {
    SmallSmem& sm = smem();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int x = warp_incl_scan(v);
    if (lane == 31) sm.red_i[wid] = x;
    __syncthreads();
    const int w = lane < kWarps ? sm.red_i[lane] : 0;
    const int e = warp_incl_scan(w);
    *total = __shfl_sync(0xffffffffu, e, 31);
    const int before = __shfl_sync(0xffffffffu, e - w, wid);
    __syncthreads();
    return before + x - v;
}

// The box of this CTA's share of the points, and whether a coordinate is not
// finite, into every CTA's copy (ordered by the cluster barrier that follows).
template <int Q>
__device__ __noinline__ void box_out(const float* mnv, const float* mxv, int bad, int rank) {
    cg::cluster_group cl = cg::this_cluster();
    SmallSmem& sm = smem();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint32_t lo = __reduce_max_sync(0xffffffffu, isfinite(mnv[k]) ? ~enc_f(mnv[k]) : 0u);
        const uint32_t hi = __reduce_max_sync(0xffffffffu, isfinite(mxv[k]) ? enc_f(mxv[k]) : 0u);
        if (lane == 0) {
            sm.redu[k][wid] = lo;
            sm.redu[3 + k][wid] = hi;
        }
    }
    bad = __syncthreads_or(bad);
    if (wid < 6) {  // warp k reduces value k
        const uint32_t code = __reduce_max_sync(0xffffffffu, lane < kWarps ? sm.redu[wid][lane] : 0u);
        if (lane < Q) *at_rank<Q>(cl, &sm.box[rank][wid], lane) = code;
    } else if (wid == 6 && lane < Q) {
        *at_rank<Q>(cl, &sm.bad[rank], lane) = bad;
    }
}

// Points of a level as the loops read them: the copy at the front of shared
// memory, or the staged points in global memory (through L2: other CTAs mark
// them taken); the pass tables lie behind that copy, or at the front.
template <bool SM>
__device__ __forceinline__ float4 load_point(const float4* stg, int i) {
    if constexpr (SM) return reinterpret_cast<const float4*>(dyn)[i];
    else return __ldcg(stg + i);
}
template <bool SM>
__device__ __forceinline__ uint32_t* pass_area() {
    return reinterpret_cast<uint32_t*>(SM ? dyn + kPtsBytes : dyn);
}

// The counting functions are not inlined: their loops get the registers of a
// thread (128) that the kernel around them does not hold across the call.

// The points t0 + b T of a thread's set bits b to the list, of which the first
// `room` are kept (whole warps; one atomic a warp).
__device__ __noinline__ void append_open(unsigned long long bits, int t0, int T, unsigned short* list, int room) {
    SmallSmem& sm = smem();
    const int mine = __popcll(bits), upto = warp_incl_scan(mine);
    int pos = 0;
    if ((threadIdx.x & 31) == 31 && upto) pos = atomicAdd(&sm.nopen[0], upto);
    pos = __shfl_sync(0xffffffffu, pos, 31) + upto - mine;
    for (; bits; bits &= bits - 1ull, ++pos)
        if (pos < room) list[pos] = static_cast<unsigned short>(t0 + (__ffsll(static_cast<long long>(bits)) - 1) * T);
}

// The key of a point's cell (a fast grid).
__device__ __forceinline__ unsigned long long key_of(const float4& q, const BoxGrid& B) {
    const float p[3] = {q.x, q.y, q.z};
    int u[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) u[a] = static_cast<int>(__fsub_rn(floorf(__fdiv_rn(p[a], B.g.v[a])), B.g.fmin[a]));
    return static_cast<unsigned long long>(u[0]) | (static_cast<unsigned long long>(u[1]) << 21) |
           (static_cast<unsigned long long>(u[2]) << 42);
}

// kWide: the keys collected, in the room of the received candidates (which the
// cut-off fills, cluster barriers later).
__device__ __forceinline__ unsigned long long* twin_keys() {
    return reinterpret_cast<unsigned long long*>(dyn + kPtsBytes + kTabBytes);
}
__device__ __forceinline__ void add_twin(unsigned long long key) {
    const int pos = atomicAdd(&smem().ntwin, 1);
    if (pos < kCandAll) twin_keys()[pos] = key;
}

// kWide, behind a round's reads: of this thread's points that took another's word
// for their cell's (set bits: point t0 + b T, or the one listed there), those whose
// cells differ.
template <bool SM>
__device__ __noinline__ void wide_check(const float4* stg, const PassGrid* pg, const unsigned short* word, unsigned nslots,
                                        unsigned mult, unsigned long long bits, int t0, int T, const unsigned short* list) {
    const uint32_t* const area = pass_area<SM>();
#pragma unroll 1
    for (; bits; bits &= bits - 1ull) {
        int i = t0 + (__ffsll(static_cast<long long>(bits)) - 1) * T;
        if (list) i = list[i];
        const float4 a = load_point<SM>(stg, i), b = load_point<SM>(stg, word[__umulhi(area[i] * mult, nslots)]);
        const unsigned long long key = key_of(a, pg->bg);
        if (key != key_of(b, pg->bg)) add_twin(key);
    }
}

// The cells that this thread counts of those collected; kManyOpen where they are too many.
__device__ __noinline__ unsigned count_twins() {
    __syncthreads();
    const int twins = smem().ntwin;
    if (twins > kCandAll) return kManyOpen;
    const unsigned long long* const key = twin_keys();
    unsigned won = 0;
#pragma unroll 1
    for (int k = threadIdx.x; k < twins; k += kST) {
        bool seen = false;
#pragma unroll 1
        for (int e = 0; e < k && !seen; ++e) seen = key[e] == key[k];
        won += seen ? 0u : 1u;
    }
    return won;
}

// The cells of the c points listed in `list` that this thread's count: rounds
// among themselves with other hashes (what a round leaves goes to `other`, and
// to and fro), the last few by a warp.  In every thread kManyOpen where a round
// leaves too many.
template <bool SM, bool kW>
__device__ __noinline__ unsigned settle_open(const float4* stg, const PassGrid* pg, unsigned short* word, unsigned nslots,
                                             int c, unsigned short* list, int list_room, unsigned short* other,
                                             int other_room) {
    const uint32_t* const area = pass_area<SM>();
    const bool wide = kW && pg->mode == kWide;
    SmallSmem& sm = smem();
    unsigned mult = 0xB7A56463u, won = 0;
#pragma unroll 1
    for (int round = 1; c > kMaxOpen; ++round) {
        mult = mult * 0x85EBCA77u + 0xC2B2AE3Eu;  // (odd again)
        if (threadIdx.x == 0) sm.nopen[round & 1] = 0;
#pragma unroll 1
        for (int k = threadIdx.x; k < c; k += kST) {
            const unsigned i = list[k];
            word[__umulhi(area[i] * mult, nslots)] = static_cast<unsigned short>(i);
        }
        __syncthreads();
        unsigned long long same = 0;
        int b = 0;
#pragma unroll 1
        for (int k = threadIdx.x; k < c; k += kST) {
            const unsigned i = list[k], mine = area[i], w = word[__umulhi(mine * mult, nslots)];
            if (w == i) {
                ++won;
            } else if (area[w] != mine) {
                const int pos = atomicAdd(&sm.nopen[round & 1], 1);
                if (pos < other_room) other[pos] = static_cast<unsigned short>(i);
            } else if (kW) {
                same |= 1ull << b;
            }
            if (kW) ++b;
        }
        if (wide) wide_check<SM>(stg, pg, word, nslots, mult, same, threadIdx.x, kST, list);
        __syncthreads();
        c = sm.nopen[round & 1];
        if (c > other_room) return kManyOpen;
        unsigned short* const l = list;
        list = other;
        other = l;
        const int r = list_room;
        list_room = other_room;
        other_room = r;
    }
    if (threadIdx.x < 32) {  // the first of every cell counts
        const unsigned lane = threadIdx.x, mine = static_cast<int>(lane) < c ? area[list[lane]] : kNoCell;
        unsigned same = __match_any_sync(0xffffffffu, mine);
        if (wide)
            same = __match_any_sync(
                0xffffffffu, static_cast<int>(lane) < c ? key_of(load_point<SM>(stg, list[lane]), pg->bg) : ~0ull);
        won += (static_cast<int>(lane) < c && __ffs(same) - 1 == static_cast<int>(lane)) ? 1u : 0u;
    }
    return won;
}

// The first loop of count_cells over a box far from the origin, where a warp
// seldom has no point near an integer: the cells are divided for without a first
// look.  (16 CTAs, 20,000 points, voxels 2^18 / 2^22 cells from the origin: 143 / 126
// us a call, with the second look at every point 235 / 200, near the origin 94.  The
// loops cost the same at about 2^16 cells.)
constexpr float kFarLoop = 65536.0f;  // cells from the origin
template <bool SM, int T>
__device__ __noinline__ void far_cells(const float4* stg, int n, const PassGrid* pg, unsigned short* word, unsigned mult,
                                       int t0) {
    constexpr int kIn = 2;
    uint32_t* const area = pass_area<SM>();
    const bool hash = pg->mode != kDirect;
    const unsigned nslots = pg->nslots, nx = pg->bg.nx, nxy = pg->bg.nxy;
    const float v[3] = {pg->bg.g.v[0], pg->bg.g.v[1], pg->bg.g.v[2]};
    const float f0[3] = {pg->bg.g.fmin[0], pg->bg.g.fmin[1], pg->bg.g.fmin[2]};
#pragma unroll 1
    for (int i0 = t0; i0 < n; i0 += kIn * T) {
        float4 q[kIn];
#pragma unroll
        for (int k = 0; k < kIn; ++k) q[k] = load_point<SM>(stg, min(i0 + k * T, n - 1));
#pragma unroll
        for (int k = 0; k < kIn; ++k) {
            const int i = i0 + k * T;
            if (i >= n) break;
            const float p[3] = {q[k].x, q[k].y, q[k].z};
            unsigned u[3];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                u[a] = static_cast<unsigned>(static_cast<int>(__fsub_rn(floorf(__fdiv_rn(p[a], v[a])), f0[a])));
            const unsigned c = min(u[0] + nx * u[1] + nxy * u[2], kNoCell - 1u);  // (kWide: any number)
            const bool in = __float_as_int(q[k].w) >= 0;
            area[i] = in ? c : kNoCell;
            if (in) word[hash ? __umulhi(c * mult, nslots) : c] = static_cast<unsigned short>(i);
        }
    }
}

// kDirect, kHash and kWide: the cells this thread's points (t0, t0 + T, ...) stand for.  The
// area holds the points' cell numbers and nslots 16-bit words behind them.  kRare: of a far
// box, or (kW) kWide, in a function of its own: code beside the loops below costs every pass.
template <bool SM, int T, bool kRare, bool kW>
__device__ __noinline__ unsigned count_cells(const float4* stg, int n, const PassGrid* pg, int t0) {
    // Points of a group: more of them cost padding in the last group and code (16 / 8 /
    // 4 / 2 / 1 on 16 CTAs, LiDAR chain of 20,876 points: 343 / 291 / 275 / 288 / 320 us)
    constexpr int kIn = (SM && T != kST) ? 3 : 4;
    static_assert(kSmallMax <= 64 * kST, "one bit per point of a thread: n <= 64 T");
    uint32_t* const area = pass_area<SM>();
    unsigned short* const word = reinterpret_cast<unsigned short*>(area + n);
    const bool hash = pg->mode != kDirect;
    const unsigned nslots = pg->nslots;
    const unsigned mult = 0x9E3779B1u;
    SmallSmem& sm = smem();
    if (threadIdx.x == 0) {
        sm.nopen[0] = 0;
        if (kRare && kW) sm.ntwin = 0;
    }
    // group(i0, all): the points i0, i0 + T, ... of which `all`, or those below n, are there.
    // A thread's loops run over whole groups, free of range checks, and one more
    auto each = [&](auto&& group) {
        int i0 = t0;
        if constexpr (!SM) {
#pragma unroll 1
            for (; i0 + (kIn - 1) * T < n; i0 += kIn * T) group(i0, std::true_type{});
        }
#pragma unroll 1
        for (; i0 < n; i0 += kIn * T) group(i0, std::false_type{});
    };
    if (kRare && (!kW || pg->far)) {
        far_cells<SM, T>(stg, n, pg, word, mult, t0);
    } else {
        const CellMap cell(pg->bg);
        each([&](int i0, auto all) {
            float4 q[kIn];
            unsigned c[kIn];
#pragma unroll
            for (int k = 0; k < kIn; ++k)
                q[k] = load_point<SM>(stg, all.value ? i0 + k * T : min(i0 + k * T, n - 1));
            unsigned near = 0u;  // points near a cell's face: one branch for all of them
#pragma unroll
            for (int k = 0; k < kIn; ++k) near |= cell.fast(q[k], &c[k]) ? 0u : (1u << k);
            if (near) {
#pragma unroll
                for (int k = 0; k < kIn; ++k)
                    if ((near >> k) & 1u) c[k] = cell.near(q[k]);
            }
#pragma unroll
            for (int k = 0; k < kIn; ++k) {
                const int i = i0 + k * T;
                if (kRare && kW) c[k] = min(c[k], kNoCell - 1u);  // (kWide: any number)
                if (__float_as_int(q[k].w) < 0) c[k] = kNoCell;  // taken
                if (all.value || i < n) {
                    area[i] = c[k];
                    if (c[k] != kNoCell)
                        word[hash ? __umulhi(c[k] * mult, nslots) : c[k]] = static_cast<unsigned short>(i);
                }
            }
        });
    }
    __syncthreads();
    unsigned won = 0;
    if (!hash) {
        each([&](int i0, auto all) {
            unsigned c[kIn];
#pragma unroll
            for (int k = 0; k < kIn; ++k) c[k] = (all.value || i0 + k * T < n) ? area[i0 + k * T] : kNoCell;
#pragma unroll
            for (int k = 0; k < kIn; ++k)
                if (c[k] != kNoCell) won += (word[c[k]] == i0 + k * T) ? 1u : 0u;
        });
        return won;
    }
    // a slot's last writer stands for its cell; the points of the other cells that
    // share the slot are listed (a bit per point, then their indices)
    unsigned long long left = 0, same = 0;
    int k0 = 0;
    each([&](int i0, auto all) {
        unsigned c[kIn], w[kIn], bits = 0u, eq = 0u;
#pragma unroll
        for (int k = 0; k < kIn; ++k) c[k] = (all.value || i0 + k * T < n) ? area[i0 + k * T] : kNoCell;
#pragma unroll
        for (int k = 0; k < kIn; ++k) w[k] = (c[k] != kNoCell) ? word[__umulhi(c[k] * mult, nslots)] : 0u;
#pragma unroll
        for (int k = 0; k < kIn; ++k) {
            const unsigned other = area[w[k]];
            if (c[k] != kNoCell) {
                won += (w[k] == static_cast<unsigned>(i0 + k * T)) ? 1u : 0u;
                bits |= (other != c[k]) ? (1u << k) : 0u;
                if (kRare && kW) eq |= (other == c[k] && w[k] != static_cast<unsigned>(i0 + k * T)) ? (1u << k) : 0u;
            }
        }
        left |= static_cast<unsigned long long>(bits) << k0;
        if (kRare && kW) same |= static_cast<unsigned long long>(eq) << k0;
        k0 += kIn;
    });
    const bool wide = kRare && kW && pg->mode == kWide;
    if (wide) wide_check<SM>(stg, pg, word, nslots, mult, same, t0, T, nullptr);
    unsigned short* const list = reinterpret_cast<unsigned short*>(dyn + kListOff);
    append_open(left, t0, T, list, kOpenA);
    __syncthreads();
    int c = sm.nopen[0];
    unsigned more;
    if (c <= kOpenA) {
        more = settle_open<SM, kRare && kW>(stg, pg, word, nslots, c, list, kOpenA, list + kOpenA, kSelMax - kOpenA);
    } else {
        // too many for the list (levels near 32,768 points in about as many cells):
        // half of the words, which are done with, take it
        const int half = static_cast<int>(nslots / 2);
        __syncthreads();
        if (threadIdx.x == 0) sm.nopen[0] = 0;
        __syncthreads();
        append_open(left, t0, T, word + half, half);
        __syncthreads();
        c = sm.nopen[0];
        if (c > half) return kManyOpen;
        more = settle_open<SM, kRare && kW>(stg, pg, word, half, c, word + half, half, list, kSelMax);
    }
    if (more == kManyOpen) return kManyOpen;
    won += more;
    if (wide) {
        const unsigned own = count_twins();
        if (own == kManyOpen) return kManyOpen;
        won += own;
    }
    return won;
}

// kHash where many cells share slots: rounds with other hashes until few points
// are undecided (every round decides a cell at least).
template <bool SM, int T>
__device__ __noinline__ unsigned count_open(int n, const PassGrid* pg, int t0) {
    uint32_t* const area = pass_area<SM>();
    unsigned short* const word = reinterpret_cast<unsigned short*>(area + n);
    unsigned short* const list = reinterpret_cast<unsigned short*>(dyn + kListOff);
    SmallSmem& sm = smem();
    const unsigned nslots = pg->nslots;
    unsigned mult = 0x27D4EB2Fu, won = 0;
    unsigned long long open = ~0ull;  // bit k: point t0 + k T is undecided
#pragma unroll 1
    for (int round = 0; round < n; ++round) {
        __syncthreads();
        if (threadIdx.x == 0) sm.nopen[0] = 0;
#pragma unroll 1
        for (int k = 0, i = t0; i < n; ++k, i += T)
            if (((open >> k) & 1ull) && area[i] != kNoCell)
                word[__umulhi(area[i] * mult, nslots)] = static_cast<unsigned short>(i);
        __syncthreads();
        unsigned long long left = 0;
#pragma unroll 1
        for (int k = 0, i = t0; i < n; ++k, i += T)
            if (((open >> k) & 1ull) && area[i] != kNoCell) {
                const unsigned w = word[__umulhi(area[i] * mult, nslots)];
                if (w == static_cast<unsigned>(i)) ++won;
                else if (area[w] != area[i]) left |= 1ull << k;
            }
        open = left;
        for (; left; left &= left - 1ull) {
            const int pos = atomicAdd(&sm.nopen[0], 1);
            if (pos < kMaxOpen) list[pos] = static_cast<unsigned short>(t0 + (__ffsll(static_cast<long long>(left)) - 1) * T);
        }
        __syncthreads();
        const int c = sm.nopen[0];
        if (c <= kMaxOpen) {
            if (static_cast<int>(threadIdx.x) < c) {
                const unsigned mine = area[list[threadIdx.x]];
                bool seen = false;
                for (int k = 0; k < static_cast<int>(threadIdx.x) && !seen; ++k) seen = area[list[k]] == mine;
                won += seen ? 0u : 1u;
            }
            break;
        }
        mult = mult * 0x85EBCA77u + 0xC2B2AE3Eu;  // (odd again)
    }
    return won;
}

// kIndex: the number of points whose voxel was new; more words than points.
template <bool SM, int T>
__device__ __noinline__ unsigned count_index(const float4* src, int n, const PassGrid* pg, int t0) {
    uint32_t* const area = pass_area<SM>();
    const Grid& G = pg->bg.g;
    constexpr unsigned kArea = static_cast<unsigned>((SM ? kTabBytes : kPtsBytes + kTabBytes) / 4);
    const unsigned nslots = min(static_cast<unsigned>(2 * n + 64), kArea);
    const int tid = threadIdx.x;
    for (unsigned k = tid; k < nslots; k += kST) area[k] = 0u;
    __syncthreads();
    unsigned fresh = 0;
    for (int i = t0; i < n; i += T) {
        const float4 q = load_point<SM>(src, i);
        if (__float_as_int(q.w) < 0) continue;
        const float p[3] = {q.x, q.y, q.z};
        unsigned long long key;
        float f[3];
        if (!cell_key(p, G, &key, f)) {
            smem().acc_err = 1u;
            continue;
        }
        const unsigned h = static_cast<unsigned>(slot_mix(key) >> 32);
        const uint32_t entry = (h << 16) | static_cast<uint32_t>(i + 1);
        unsigned slot = __umulhi(h, nslots);
        for (unsigned probe = 0; probe < nslots; ++probe) {
            uint32_t cur = *reinterpret_cast<volatile uint32_t*>(area + slot);
            if (cur == 0u) {
                cur = atomicCAS(area + slot, 0u, entry);
                if (cur == 0u) {
                    ++fresh;
                    break;
                }
            }
            if ((cur >> 16) == (h & 0xffffu)) {
                const float4 q2 = load_point<SM>(src, static_cast<int>(cur & 0xffffu) - 1);
                const float p2[3] = {q2.x, q2.y, q2.z};
                unsigned long long key2;
                if (cell_key(p2, G, &key2, f) && key2 == key) break;
            }
            if (++slot == nslots) slot = 0u;
        }
    }
    return fresh;
}

// The voxels of a size that this thread's points (t0, t0 + T, ...) count.  (On one CTA
// far boxes take the general way: its few points hardly repay the code, 1,000 points
// 48.3 us with it, 47.2 without.)
template <bool SM, int T, bool kW>
__device__ __forceinline__ unsigned count_pass(const float4* stg, int n, const PassGrid* pg, int t0) {
    constexpr bool kCluster = T == kST;
    const int mode = pg->mode;
    if (mode == kDirect || mode == kHash || (kW && mode == kWide)) {
        const unsigned won = (kCluster && (pg->far || (kW && mode == kWide)))
                                 ? count_cells<SM, kST, true, kW>(stg, n, pg, t0)
                                 : count_cells<SM, T, false, kW>(stg, n, pg, t0);
        if (won != kManyOpen) return won;
        if (!kW || mode != kWide) return count_open<SM, T>(n, pg, t0);
        __syncthreads();  // (the count's area is filled anew)
        return count_index<SM, T>(stg, n, pg, t0);
    }
    if (mode == kIndex) return count_index<SM, T>(stg, n, pg, t0);
    return 0u;
}

// The grids of up to ten sizes over the level's box into sm.pg[first ...], how
// a pass counts them, by one warp: lanes [3 o, 3 o + 3) take size o (sv, alike
// in those lanes), a lane per axis.
template <bool kW>
__device__ __noinline__ void set_grids(int first, int sizes, float sv, const float* aspect, int n, unsigned area_words) {
    SmallSmem& sm = smem();
    const int lane = threadIdx.x & 31;
    const int o = lane / 3, ax = lane < 30 ? lane - 3 * o : 0, lead = lane < 30 ? 3 * o : 27;
    float v, rv, f0;
    unsigned span;
    const bool ok = box_axis(sv, aspect[ax], sm.mn[ax], sm.mx[ax], &v, &rv, &f0, &span);
    const unsigned okm = __ballot_sync(0xffffffffu, ok) >> lead;
    const unsigned nx = __shfl_sync(0xffffffffu, span, lead), ny = __shfl_sync(0xffffffffu, span, lead + 1),
                   nz = __shfl_sync(0xffffffffu, span, lead + 2);
    const int ci = (fabsf(f0) < 4194304.0f) ? -(kMagicBits + static_cast<int>(f0)) : 0;
    const unsigned part = static_cast<unsigned>(ci) * (ax == 0 ? 1u : (ax == 1 ? nx : nx * ny));
    const unsigned c0 = part + __shfl_sync(0xffffffffu, part, lead + 1) + __shfl_sync(0xffffffffu, part, lead + 2);
    const float vn = near_width(v, f0, span, kFarLoop);
    const float vmax = fmaxf(vn, fmaxf(__shfl_sync(0xffffffffu, vn, lead + 1), __shfl_sync(0xffffffffu, vn, lead + 2)));
    if (o < sizes && lane < 30) {
        PassGrid& g = sm.pg[first + o];
        g.bg.g.v[ax] = v;
        g.bg.g.r[ax] = 0.0f;
        g.bg.ra[ax] = rv;
        g.bg.g.fmin[ax] = f0;
        g.bg.ci[ax] = ci;
        if (ax == 0) {
            const bool all_ok = (okm & 7u) == 7u, fast = all_ok && nx && ny && nz;
            const unsigned long long cells = static_cast<unsigned long long>(nx) * ny * nz;
            // 16-bit words behind the cell numbers; for the load, 4 a point of kHash and kWide
            const unsigned words = 2u * (area_words - static_cast<unsigned>(n));
            const bool direct = fast && cells <= words;
            g.sv = sv;
            g.mode = !fast ? (all_ok ? kIndex : kSkip) : (direct ? kDirect : (cells < kNoCell ? kHash : (kW ? kWide : kIndex)));
            g.nslots = direct ? static_cast<unsigned>(cells) : min(words, 4u * static_cast<unsigned>(n));
            g.far = isinf(vmax) ? 1 : 0;
            g.bg.amb = __fmul_rn(vmax, kNear);
            g.bg.nx = nx;
            g.bg.nxy = nx * ny;
            g.bg.c0 = c0;
            g.bg.ok = all_ok ? 1 : 0;
            g.bg.fast = fast ? 1 : 0;
            g.bg.cells = cells;
        }
    }
    __syncwarp();
}

// The CTA whose part of the selection table holds a voxel.
template <int Q>
__device__ __forceinline__ int voxel_rank(unsigned long long key) {
    unsigned h = static_cast<unsigned>(key) * 0x9E3779B1u + static_cast<unsigned>(key >> 32) * 0x85EBCA77u;
    h = (h ^ (h >> 15)) * 0xC2B2AE35u;
    return (Q == 1) ? 0 : static_cast<int>(h >> (32 - qlog2<Q>()));
}

// A point's voxel key and (word, level index) for the selection at s*; false
// when it takes no part (taken) or its key is out of range.
__device__ __forceinline__ bool select_key(const Plan& P, const float4& q, int i, const BoxGrid& B,
                                           unsigned long long* key, unsigned long long* packed, unsigned* ebits) {
    if (__float_as_int(q.w) < 0) return false;
    const float p[3] = {q.x, q.y, q.z};
    float f[3];
    if (B.fast) {
        int u[3];
        floor_cells(p, B, u);
        *key = static_cast<unsigned long long>(u[0]) | (static_cast<unsigned long long>(u[1]) << 21) |
               (static_cast<unsigned long long>(u[2]) << 42);
#pragma unroll
        for (int a = 0; a < 3; ++a) f[a] = __fadd_rn(B.g.fmin[a], __int2float_rn(u[a]));  // (exact)
    } else if (!cell_key(p, B.g, key, f)) {
        *ebits |= 1u;
        return false;
    }
    const unsigned word = (P.select == HAV_SELECT_RANDOM)
                              ? static_cast<unsigned>(random_draw(P.seed, static_cast<unsigned long long>(i)) >> 32)
                              : __float_as_uint(centre_d2(p, B.g, f));
    *packed = (static_cast<unsigned long long>(word) << 32) | static_cast<unsigned>(i);
    return true;
}

// Section 3.2: a point into this CTA's part of the selection table: per voxel
// the smallest packed in vals; the first point of a voxel counts it in the
// cut-off histogram and lists its slot.  Whole warp calls.
__device__ __forceinline__ void select_insert(SmallSmem& sm, bool in, unsigned long long key, unsigned long long packed,
                                              unsigned long long* keys, unsigned long long* vals, unsigned mask,
                                              unsigned short* list, unsigned* ebits) {
    bool nw = false;
    unsigned slot = 0;
    if (in) {
        slot = static_cast<unsigned>(slot_mix(key) >> 32) & mask;
        unsigned probe = 0;
        for (; probe <= mask; ++probe) {
            unsigned long long cur = *reinterpret_cast<volatile unsigned long long*>(keys + slot);
            if (cur == kEmptyKey) {
                cur = atomicCAS(keys + slot, kEmptyKey, key);
                if (cur == kEmptyKey) {
                    nw = true;
                    break;
                }
            }
            if (cur == key) break;
            slot = (slot + 1) & mask;
        }
        if (probe > mask) *ebits |= 2u;
        else if (packed < *reinterpret_cast<volatile unsigned long long*>(vals + slot)) atomicMin(vals + slot, packed);
        if (nw) atomicAdd(sm.own_hist + static_cast<int>(priority(key) >> (64 - kCutBits)), 1u);
    }
    const int pos = warp_append(nw, &sm.nlist);
    if (pos >= 0) list[pos] = static_cast<unsigned short>(slot);
}

// Levels [first_level, P.L) of every segment; level first_level > 0 reads its
// input through orig[(first_level - 1) & 1].
template <int Q, bool kW>
__global__ void __cluster_dims__(Q, 1, 1) __launch_bounds__(kST, 1)
    hav_small_kernel(const __grid_constant__ Plan P, int first_level) {
    cg::cluster_group cl = cg::this_cluster();
    SmallSmem& sm = smem();
    float4* pts = reinterpret_cast<float4*>(dyn);  // x, y, z, original index (sign bit: taken)
    unsigned long long* ch = reinterpret_cast<unsigned long long*>(dyn + kPtsBytes + kTabBytes);  // [Q][kCandAll / Q]
    unsigned short* list = reinterpret_cast<unsigned short*>(dyn + kListOff);
    constexpr int kCandCap = kCandAll / Q;

    const int tid = threadIdx.x;
    const int lane = tid & 31, wid = tid >> 5;
    const int rank = static_cast<int>(cl.block_rank());
    const int cluster_id = blockIdx.x / Q;
    const int nclusters = gridDim.x / Q;
    unsigned char* ws = P.ws;
    SegHdr* sh = reinterpret_cast<SegHdr*>(ws + P.lay.seghdr);
    GlobalHdr* gh = reinterpret_cast<GlobalHdr*>(ws + P.lay.ghdr);
    hav_layer_trace* trace = reinterpret_cast<hav_layer_trace*>(ws + P.lay.trace);
    const int S = P.S;
    const bool write_tr = (rank == 0 && tid == 0);
    constexpr int kNodes = (Q == 1) ? 1 : Q - 1;  // sizes a pass evaluates: a full subtree
    SmallTimer tm;
    tm.open(P, write_tr && cluster_id == 0);

    for (int seg = cluster_id; seg < S; seg += nclusters) {
        // an error from earlier levels (another kernel) carries on: first m points
        int err = ld_volatile(&sh[seg].status);
        // the segment's last search of the call so far (guided start), from the
        // kernel that ran the earlier levels
        float gs = (first_level > 0) ? sh[seg].guide_s : 0.0f;
        int gm = (first_level > 0) ? sh[seg].guide_m : 0;
        csync<Q>(cl);  // every CTA runs, and is done with the previous segment
        for (int j = first_level; j < P.L; ++j) {
            const int n = static_cast<int>((j == 0) ? (P.off0[seg + 1] - P.off0[seg]) : P.m[j - 1][seg]);
            const int m = P.m[j][seg];
            const int a = part_start<Q>(n, rank), b = part_start<Q>(n, rank + 1);
            const int L = b - a;
            float4* stg = reinterpret_cast<float4*>(ws + P.lay.ord[j & 1]) + P.off0[seg];
            const bool in_smem = n <= kPtsSmem;
            uint32_t* area = reinterpret_cast<uint32_t*>(in_smem ? dyn + kPtsBytes : dyn);
            const unsigned area_words =
                static_cast<unsigned>(in_smem ? kTabBytes / 4 : (kPtsBytes + kTabBytes) / 4);

            // --------------------------------------------- points and bbox
            // (a later level was staged by the previous level's compaction)
            if (j == first_level) {
                long long ibase = 0;  // this segment's first input position in the level array
#pragma unroll 1
                for (int s2 = 0; s2 < seg && j > 0; ++s2) ibase += P.m[j - 1][s2];
                const int32_t* orig_in = reinterpret_cast<const int32_t*>(ws + P.lay.orig[(j + 1) & 1]) + ibase;
                float mnv[3] = {INFINITY, INFINITY, INFINITY}, mxv[3] = {-INFINITY, -INFINITY, -INFINITY};
                int bad = 0;
#pragma unroll 1
                for (int i = tid; i < L; i += kST) {
                    const int o = (j == 0) ? (a + i) : orig_in[a + i];
                    const float* p = P.points + 3 * (P.off0[seg] + o);
                    const float4 q = make_float4(p[0], p[1], p[2], __int_as_float(o));
                    if constexpr (Q == 1) pts[i] = q;
                    else __stcg(stg + a + i, q);
                    const float c3[3] = {q.x, q.y, q.z};
                    for (int k = 0; k < 3; ++k) {
                        if (!isfinite(c3[k])) bad = 1;
                        mnv[k] = fminf(mnv[k], c3[k]);
                        mxv[k] = fmaxf(mxv[k], c3[k]);
                    }
                }
                box_out<Q>(mnv, mxv, bad, rank);
                csync<Q>(cl);
            }
            tm.mark(1, j, 0, 0);
            // the bracket (0, s_hi] of Section 3.3 from the shares' boxes, in every
            // CTA (warp 0), and the layers' budgets (warp 1)
            if (wid == 0) {
                const int nf = __any_sync(0xffffffffu, lane < Q && sm.bad[lane < Q ? lane : 0] != 0);
                float lo = 0.0f, hi = 0.0f;  // lane k: axis k
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const uint32_t c0 = __reduce_max_sync(0xffffffffu, lane < Q ? sm.box[lane][k] : 0u);
                    const uint32_t c1 = __reduce_max_sync(0xffffffffu, lane < Q ? sm.box[lane][3 + k] : 0u);
                    if (j == 0 && rank == 0 && lane == 0) {
                        sh[seg].bbox[0][k] = c0;
                        sh[seg].bbox[0][3 + k] = c1;
                    }
                    if (lane == k) {
                        lo = dec_f(~c0);
                        hi = dec_f(c1);
                    }
                }
                if (n == 0 || nf || err) lo = hi = 0.0f;
                float s_hi = 0.0f;
                if (lane < 3) {
                    sm.mn[lane] = lo;
                    sm.mx[lane] = hi;
                    s_hi = fmaxf(0.0f, __fdiv_rn(__fsub_rn(hi, lo), P.aspect[lane]));
                }
                s_hi = fmaxf(fmaxf(s_hi, __shfl_sync(0xffffffffu, s_hi, 1)), __shfl_sync(0xffffffffu, s_hi, 2));
                if (lane == 0) {
                    if (s_hi == 0.0f) s_hi = 1.0f;
                    sm.s_hi = s_hi;
                    sm.nonfinite = nf;
                    sm.acc_err = 0u;
                }
                if (lane < kMaxIters) sm.pre[lane] = -1;
            } else if (wid == 1 && lane < P.layers) {
                const long long ml = layer_budget(m, P.layers, P.ratio, lane);
                sm.ml[lane] = static_cast<int>(ml);
                sm.kmax[lane] = static_cast<int>(ml + ml * P.sigma_num / P.sigma_den);
            }
            if (Q > 1 && in_smem)
#pragma unroll 1
                for (int i = tid; i < n; i += kST) pts[i] = __ldcg(stg + i);
            __syncthreads();
            if (!err && sm.nonfinite) {
                err = HAV_ERR_NONFINITE;
                if (write_tr) seg_fail(sh, gh, seg, err);
            }
            if (!err && !isfinite(sm.s_hi)) {
                err = HAV_ERR_RANGE;
                if (write_tr) seg_fail(sh, gh, seg, err);
            }
            // the sizes s_hi / 2^(k+1) of the plain bisection's leading steps and
            // the cells the box spans at them (cell_bound), a lane per quotient
            if (P.search == HAV_SEARCH_BISECT && tid < 8 * kMaxIters) {
                const int k = tid >> 3, g = tid & 7, ax = g < 6 ? g >> 1 : 0;
                float sv = sm.s_hi;
#pragma unroll 1
                for (int h = 0; h <= k; ++h) sv = __fmul_rn(__fadd_rn(0.0f, sv), 0.5f);
                const float v = __fmul_rn(sv, P.aspect[ax]);
                float fl = 0.0f;
                const bool ok = v > 0.0f && isfinite(v) && floor_div((g & 1) ? sm.mx[ax] : sm.mn[ax], v, &fl);
                const float f1 = __shfl_down_sync(0xffffffffu, fl, 1);
                const float u = __fsub_rn(f1, fl);
                const bool in = (g & 1) || g >= 6 || (u >= 0.0f && u < 1048576.0f);
                const unsigned good = __ballot_sync(0xffffffffu, ok && in) >> (lane & 24);
                const long long c = static_cast<long long>(in ? u : 0.0f) + 1;
                const long long cy = __shfl_down_sync(0xffffffffu, c, 2), cz = __shfl_down_sync(0xffffffffu, c, 4);
                if (g == 0) {
                    sm.st_s[k] = sv;
                    sm.st_b[k] = ((good & 63u) == 63u) ? c * cy * cz : LLONG_MAX;
                }
            }
            __syncthreads();

            // ----------------------------------------------------- layers
            int taken_before = 0;
            unsigned pass_no = 0;
#pragma unroll 1
            for (int l = 0; l < P.layers; ++l) {
                const int ml = sm.ml[l], kmax = sm.kmax[l];
                hav_layer_trace* tr = trace + (static_cast<long long>(j) * S + seg) * kMaxLayers + l;
                if (write_tr) {
                    tr->m_l = ml;
                    tr->k_max = kmax;
                    tr->k_star = 0;
                    tr->n_in = n - taken_before;
                    tr->iters = 0;
                    tr->accepted = 0;
                    tr->bounded = 0u;
                    tr->s_hi = sm.s_hi;
                    tr->s_star = 0.0f;
                }
                taken_before += ml;
                if (ml == 0 || err) continue;
                const bool fixed = P.fixed_s > 0.0f;
                const int steps = fixed ? 0 : P.t_max;
                const bool guided = (P.search == HAV_SEARCH_GUIDED);
                if (wid == 0) {
                    float hi = sm.s_hi, first = 0.0f;
                    int t = 0, up = 0;
                    if (guided && steps > 0) {
                        // guided start: the first size from the segment's previous search in
                        // this call (or from s_hi), doubling up from it while the counts stay
                        // too high; the same reading as the grid kernel's
                        const float g = (gm > 0) ? __fmul_rn(gs, __fsqrt_rn(__fdiv_rn(__int2float_rn(gm), __int2float_rn(ml))))
                                                 : __fdiv_rn(hi, __fsqrt_rn(__int2float_rn(ml)));
                        if (g > 0.0f && g < hi) {
                            first = g;
                            up = 1;
                        }
                    } else if (steps > 0) {
                        // The leading steps settled by an exact bound below m_l are taken
                        // without a pass, as in the grid kernel: the grid cells the
                        // bounding box spans, or an earlier layer's count at the same size
                        // s_hi / 2^(t+1) on a superset of the points; the trace keeps the
                        // smaller bound
                        static_assert(kMaxIters < 32, "one lane per step");
                        long long bd = LLONG_MAX;
                        float sv = 0.0f;
                        if (lane < steps) {
                            bd = sm.st_b[lane];
                            sv = sm.st_s[lane];
                            const int pk = sm.pre[lane];
                            if (pk >= 0 && pk < bd) bd = pk;
                        }
                        t = __ffs(~__ballot_sync(0xffffffffu, lane < steps && bd < ml)) - 1;
                        const float hs = __shfl_sync(0xffffffffu, sv, t > 0 ? t - 1 : 0);
                        if (t > 0) hi = hs;
                        if (rank == 0 && lane < t) {
                            tr->s[lane] = sv;
                            tr->K[lane] = bd;
                        }
                    }
                    if (lane == 0) {
                        sm.lo = 0.0f;
                        sm.hi = hi;
                        sm.first = first;
                        sm.up = up;
                        sm.pre_on = guided ? 0 : 1;  // every step so far had too few voxels (plain bisection)
                        sm.t = t;
                        sm.skipped = t;
                        sm.accepted = 0;
                        sm.err = 0;
                    }
                    __syncwarp();
                }

                // Section 3.3 search.  Every thread comes out with its size, s_star,
                // whether a count accepted it, and the selection's grid.
                float s_star = 0.0f;
                bool accepted = false;
                int sel = 4;
                if constexpr (Q == 1) {
                    // One size per pass, every warp deciding from the warps' counts.
                    // The last warp prepares the grids after both outcomes while the
                    // others count (it takes no points: its grids take as long).
                    constexpr int T = kST - 32;
                    const int t0 = (wid < kWarps - 1) ? tid : n;
                    static_assert(kPtsSmem <= 64 * T, "one bit per point of a thread");
                    __syncthreads();
                    float lo = 0.0f, hi = sm.hi;
                    bool up = sm.up != 0, pre = !guided;
                    int t = sm.t, par = 0, cur = 0;
                    if (t < steps) {
                        if (wid == kWarps - 1)
                            set_grids<kW>(0, 1, next_size(lo, hi, up, sm.first), P.aspect, n, area_words);
                        __syncthreads();
                        for (;;) {
                            const PassGrid& pg = sm.pg[cur];
                            const float sv = pg.sv;
                            const bool fits = pg.bg.ok != 0;  // (alike in every thread)
                            if (wid == kWarps - 1)  // outcome 0: too many voxels, 1: too few
                                set_grids<kW>(2 * (par ^ 1), 2,
                                          lane < 3 ? next_size(sv, hi, up, 0.0f) : next_size(lo, sv, false, 0.0f),
                                          P.aspect, n, area_words);
                            const unsigned won = __reduce_add_sync(0xffffffffu, count_pass<true, T, false>(pts, n, &pg, t0));
                            if (lane == 0) sm.wcnt[par][wid] = won;
                            __syncthreads();
                            const int K = static_cast<int>(
                                __reduce_add_sync(0xffffffffu, lane < kWarps ? sm.wcnt[par][lane] : 0u));
                            tm.mark(2, j, l, t);
                            if (tid == 0) {
                                sm.tr_s[t] = sv;
                                sm.tr_K[t] = K;
                            }
                            if (pre) {  // sv = s_hi / 2^(t+1): later layers of the level may reuse K
                                if (tid == 0) sm.pre[t] = K;
                                if (K >= ml) pre = false;
                            }
                            ++t;
                            // (a pass sets acc_err behind a barrier of its own (count_index), so
                            // what a warp reads here is this pass's and not a faster warp's next)
                            if (!fits || sm.acc_err) {
                                err = HAV_ERR_RANGE;
                                break;
                            }
                            if (K > kmax) {
                                lo = sv;
                            } else if (K < ml) {
                                hi = sv;
                                up = false;
                            } else {
                                accepted = true;
                                s_star = sv;
                                sel = cur;
                                break;
                            }
                            if (t >= steps) break;
                            par ^= 1;
                            cur = 2 * par + (K > kmax ? 0 : 1);
                        }
                    }
                    if (tid == 0) sm.t = t;
                    if (!accepted) {
                        s_star = fixed ? P.fixed_s : (P.t_max == 0 ? sm.s_hi : (lo > 0.0f ? lo : hi));
                        if (wid == 0) set_grids<kW>(4, 1, s_star, P.aspect, n, area_words);
                        __syncthreads();
                    }
                } else {
                    // CTA r of the cluster counts the size at node r of the subtree of
                    // steps below (lo, hi); every CTA then walks the subtree through the
                    // counts exactly as the sequential search does, up to its leaves or
                    // a node that was left out.  Warp 0 holds the search's state (alike
                    // in every CTA).
                    bool walk = false;
                    for (;;) {
                        if (wid == 0) {
                            float lo = sm.lo, hi = sm.hi, first = sm.first, ss = sm.s_hi;
                            bool up = sm.up != 0, acc = false;
                            int t = sm.t, serr = 0;
                            // lane c: node c of the subtree (heap order: child 2 c + 1 follows a
                            // count below m_l, 2 c + 2 one above k_max), its size and depth
                            const int depth = 31 - __clz(lane + 1);
                            if (walk) {
                                const float sv = sm.node_s[lane < kNodes ? lane : 0];
                                const unsigned long long c = sm.pass[(pass_no - 1u) & 1u][lane < kNodes ? lane : 0];
                                const int K = static_cast<int>(c & 0xffffffffull);
                                const unsigned flag = static_cast<unsigned>(c >> 32);
                                const bool counted = lane < kNodes && !(flag & 2u) && t + depth < steps;
                                const unsigned high = __ballot_sync(0xffffffffu, K > kmax && !(flag & 1u)),
                                               low = __ballot_sync(0xffffffffu, K < ml && !(flag & 1u)),
                                               cnt = __ballot_sync(0xffffffffu, counted);
                                // on the path: every ancestor was counted and its outcome led here
                                bool on = counted, left = true;
#pragma unroll 1
                                for (int x = lane + 1; x > 1; x >>= 1) {
                                    const int par = (x >> 1) - 1;
                                    on = on && ((cnt >> par) & 1u) && ((((x & 1) ? high : low) >> par) & 1u);
                                    left = left && !(x & 1);
                                }
                                const unsigned path = __ballot_sync(0xffffffffu, on);
                                const int last = 31 - __clz(path);  // (deeper nodes have larger numbers; the root is on it)
                                const unsigned ph = path & high, pl = path & low;
                                if (on) {
                                    sm.tr_s[t + depth] = sv;
                                    sm.tr_K[t + depth] = K;
                                    // s_hi / 2^(t+1): later layers of the level may reuse K
                                    if (left && sm.pre_on) sm.pre[t + depth] = K;
                                }
                                const float s_last = __shfl_sync(0xffffffffu, sv, last);
                                const int f_last = __shfl_sync(0xffffffffu, static_cast<int>(flag), last);
                                const float s_h = __shfl_sync(0xffffffffu, sv, ph ? 31 - __clz(ph) : 0),
                                            s_l = __shfl_sync(0xffffffffu, sv, pl ? 31 - __clz(pl) : 0);
                                if (f_last & 1) {
                                    serr = HAV_ERR_RANGE;
                                } else if (!(((high | low) >> last) & 1u)) {
                                    ss = s_last;
                                    acc = true;
                                }
                                if (ph) lo = s_h;
                                if (pl) {
                                    hi = s_l;
                                    up = false;
                                }
                                first = 0.0f;
#pragma unroll 1
                                for (int k = 0; k < __popc(path); ++k) tm.mark(2, j, l, t + k);
                                t += __popc(path);
                                __syncwarp();
                                if (lane == 0 && (pl != path)) sm.pre_on = 0;
                            }
                            const bool go = t < steps && !acc && !serr;
                            if (!go && !acc) ss = fixed ? P.fixed_s : (P.t_max == 0 ? sm.s_hi : (lo > 0.0f ? lo : hi));
                            __syncwarp();  // (every lane has read the state)
                            if (lane == 0) {
                                sm.lo = lo;
                                sm.hi = hi;
                                sm.first = first;
                                sm.up = up ? 1 : 0;
                                sm.t = t;
                                sm.s_star = ss;
                                sm.accepted = acc ? 1 : 0;
                                sm.err = serr;
                                sm.go = go ? 1 : 0;
                                sm.acc_err = 0u;
                            }
                            // this CTA's node and the root, or the selection's size
                            const float ns = cand_size(lo, hi, up, first, lane < kNodes ? lane : 0);
                            if (lane < kNodes) sm.node_s[lane] = ns;
                            const float sv = __shfl_sync(0xffffffffu, ns, (lane < 3 && rank < kNodes) ? rank : 0);
                            set_grids<kW>(go ? 0 : 4, go ? 2 : 1, go ? sv : ss, P.aspect, n, area_words);
                            if (lane == 0 && go) {
                                // left out: a step beyond the last, and a slower way to count
                                // than the root's (much finer sizes: the search seldom gets there)
                                const bool out = rank >= kNodes || t + (31 - __clz(rank + 1)) >= steps ||
                                                 sm.pg[0].mode > sm.pg[1].mode;
                                if (out) sm.pg[0].mode = kSkip;
                                if (out) sm.acc_err = 2u;
                                else if (!sm.pg[0].bg.ok) sm.acc_err = 1u;
                            }
                        }
                        __syncthreads();
                        if (!sm.go) break;
                        unsigned won = in_smem ? count_pass<true, kST, kW>(pts, n, sm.pg, tid)
                                               : count_pass<false, kST, kW>(stg, n, sm.pg, tid);
                        won = __reduce_add_sync(0xffffffffu, won);
                        if (lane == 0) sm.wcnt[0][wid] = won;
                        __syncthreads();
                        if (wid == 0) {
                            const unsigned long long v =
                                (static_cast<unsigned long long>(sm.acc_err) << 32) |
                                __reduce_add_sync(0xffffffffu, lane < kWarps ? sm.wcnt[0][lane] : 0u);
                            if (lane < Q) *at_rank<Q>(cl, &sm.pass[pass_no & 1u][rank], lane) = v;
                            __syncwarp();
                            cluster_arrive_release();
                        } else {
                            cluster_arrive_relaxed();  // (only warp 0 has something to publish)
                        }
                        cluster_wait();
                        ++pass_no;
                        walk = true;
                    }
                    s_star = sm.s_star;
                    accepted = sm.accepted != 0;
                    err = sm.err;
                }
                const BoxGrid& bg = sm.pg[sel].bg;
                if (rank == 0 && wid == 0) {
                    // the trace: the steps counted (the settled ones are there), behind them
                    __syncwarp();
                    const int t1 = sm.t, t0 = sm.skipped;
                    if (lane >= t0 && lane < t1) {
                        tr->s[lane] = sm.tr_s[lane];
                        tr->K[lane] = sm.tr_K[lane];
                    }
                    if (lane == 0) {
                        tr->iters = t1;
                        tr->bounded = t0 > 0 ? 0xffffffffu >> (32 - t0) : 0u;
                    }
                }
                if (!err) {
                    if (guided && P.t_max > 0 && !fixed) {  // the next search's guided start follows this one
                        gs = s_star;
                        gm = ml;
                    }
                    if (!bg.ok) err = HAV_ERR_RANGE;
                }
                if (err) {
                    if (write_tr) seg_fail(sh, gh, seg, err);
                    continue;
                }

                // ------------------------------ Section 3.2 selection at s*
                int part_log2 = 32 - __clz(2 * n - 1) - qlog2<Q>();  // nextpow2(2 n) / Q
                if (part_log2 < kMinCapLog2) part_log2 = kMinCapLog2;
                const int part = 1 << part_log2;
                unsigned long long* keys = reinterpret_cast<unsigned long long*>(area);
                unsigned long long* vals = keys + part;
                ulonglong2* rec = reinterpret_cast<ulonglong2*>(vals + part);
#pragma unroll 1
                for (int k = tid; k < part; k += kST)  // (both arrays: 16 bytes per slot)
                    reinterpret_cast<ulonglong2*>(area)[k] = make_ulonglong2(kEmptyKey, kEmptyVal);
                static_assert(kEmptyKey == kEmptyVal, "one fill for keys and values");
                if (tid < kCutBins) sm.own_hist[tid] = 0u;
                if (tid == kCutBins) {
                    sm.nlist = 0u;
                    sm.own_cand = 0u;
                }
                if (tid >= 96 && tid < 96 + Q) sm.bin_cnt[tid - 96] = 0;
                if (tid == 128) sm.acc_err = 0u;
                __syncthreads();
                unsigned ebits = 0;
                const unsigned mask = static_cast<unsigned>(part) - 1u;
                if constexpr (Q == 1) {
#pragma unroll 1
                    for (int i0 = tid - lane; i0 < n; i0 += kST) {  // (warp-uniform)
                        const int i = i0 + lane;
                        unsigned long long key = 0, packed = 0;
                        const bool in = i < n && select_key(P, pts[i], i, bg, &key, &packed, &ebits);
                        select_insert(sm, in, key, packed, keys, vals, mask, list, &ebits);
                    }
                } else {
                    // the share's points by the CTA that holds their voxel, as records
                    // (key, packed) that the owners fetch: into a region per owner, twice
                    // what it gets on average; where one overflows, counted and placed again
                    const int cap = min(2 * L / Q + 32, (static_cast<int>(area_words / 4) - part) / Q);
                    bool again = false;
#pragma unroll 1
                    for (int ph = 0; ph < 3; ++ph) {  // 0: regions; 1, 2: counts, exact places
#pragma unroll 1
                        for (int i = tid; i < L; i += kST) {
                            const float4 q = in_smem ? pts[a + i] : __ldcg(stg + a + i);
                            unsigned long long key, packed;
                            if (!select_key(P, q, a + i, bg, &key, &packed, &ebits)) continue;
                            const int own = voxel_rank<Q>(key);
                            const int pos = atomicAdd(&sm.bin_cnt[own], 1);
                            if (ph == 0 && pos >= cap) again = true;
                            else if (ph != 1) rec[(ph == 0 ? own * cap : 0) + pos] = make_ulonglong2(key, packed);
                        }
                        const bool redo = __syncthreads_or((ph == 0 && again) || ph == 1) != 0;
                        if (wid == 0) {
                            const int c = lane < Q ? sm.bin_cnt[lane] : 0;
                            const int off = ph == 0 ? lane * cap : warp_incl_scan(c) - c;
                            if (lane < Q) {
                                if (redo) sm.bin_cnt[lane] = ph == 0 ? 0 : off;
                                if (ph < 2) *at_rank<Q>(cl, &sm.rec[rank], lane) = make_int2(off, c);
                            }
                        }
                        if (!redo) break;
                        __syncthreads();
                    }
                    cl.sync();
                    int2 rr = (lane < Q) ? sm.rec[lane] : make_int2(0, 0);  // lane r: CTA r's records for this one
                    const int end = warp_incl_scan(rr.y);                  // ... end at this position of the whole
                    const int total = __shfl_sync(0xffffffffu, end, 31);
#pragma unroll 1
                    for (int i0 = tid - lane; i0 < total; i0 += kST) {  // (warp-uniform)
                        const int i = i0 + lane;
                        int r = 0;
#pragma unroll
                        for (int s2 = Q / 2; s2 > 0; s2 >>= 1)  // the CTA r with end[r - 1] <= i < end[r]
                            if (__shfl_sync(0xffffffffu, end, r + s2 - 1) <= i) r += s2;
                        const int e = __shfl_sync(0xffffffffu, end, r), c = __shfl_sync(0xffffffffu, rr.y, r),
                                  o = __shfl_sync(0xffffffffu, rr.x, r);
                        ulonglong2 kv = make_ulonglong2(0, 0);
                        if (i < total) kv = *at_rank<Q>(cl, rec + (o + i - (e - c)), r);
                        select_insert(sm, i < total, kv.x, kv.y, keys, vals, mask, list, &ebits);
                    }
                }
                if (ebits) atomicOr(&sm.acc_err, ebits);
                __syncthreads();
                // this CTA's histogram and errors into every CTA's copy
#pragma unroll 1
                for (int k = tid; k < kCutBins * Q; k += kST)
                    *at_rank<Q>(cl, &sm.hist[rank][k % kCutBins], k / kCutBins) = sm.own_hist[k % kCutBins];
                if (tid < Q) *at_rank<Q>(cl, &sm.errs[rank], tid) = sm.acc_err;
                csync<Q>(cl);
                tm.mark(3, j, l, 0);
                // K*, and the boundary bin: smallest b with (voxels in bins <= b) >= m_l
                if (wid == 0) {
                    static_assert(kCutBins == 64, "two bins per lane");
                    int h0 = 0, h1 = 0;
#pragma unroll
                    for (int r = 0; r < Q; ++r) {
                        const uint2 h = *reinterpret_cast<const uint2*>(&sm.hist[r][2 * lane]);
                        h0 += static_cast<int>(h.x);
                        h1 += static_cast<int>(h.y);
                    }
                    const int end = warp_incl_scan(h0 + h1);
                    const int before = end - h0 - h1;
                    if (before < ml && before + h0 >= ml) {
                        sm.cut_bin = 2 * lane;
                        sm.cut_below = before;
                    } else if (before + h0 < ml && end >= ml) {
                        sm.cut_bin = 2 * lane + 1;
                        sm.cut_below = before + h0;
                    }
                    const unsigned eb = __reduce_or_sync(0xffffffffu, lane < Q ? sm.errs[lane] : 0u);
                    if (lane == 31) {
                        sm.kstar = end;
                        sm.eb = eb;
                    }
                }
                __syncthreads();
                const int kstar = sm.kstar;
                if (write_tr) {
                    tr->k_star = kstar;
                    tr->accepted = accepted ? 1 : 0;
                    tr->s_star = s_star;
                }
                if (sm.eb) {
                    err = (sm.eb & 1u) ? HAV_ERR_RANGE : HAV_ERR_TABLE_FULL;
                    if (write_tr) seg_fail(sh, gh, seg, err);
                    continue;
                }

                // ----------------------------------- cut-off and taken marks
                const bool cut = kstar > ml;
                auto mark = [&](int g) {
                    if constexpr (Q == 1) reinterpret_cast<uint32_t*>(pts + g)[3] |= 0x80000000u;  // (one voxel, one writer)
                    else atomicOr(reinterpret_cast<uint32_t*>(stg + g) + 3, 0x80000000u);
                };
                const int nlist = static_cast<int>(sm.nlist);
#pragma unroll 1
                for (int k0 = 0; k0 < nlist; k0 += kST) {
                    const int k = k0 + tid;
                    const unsigned short sl = (k < nlist) ? list[k] : 0;
                    if (cut) __syncthreads();  // (the candidates go to the front of the list, behind the reads)
                    bool cand = false;
                    unsigned long long h = 0;
                    if (k < nlist) {
                        bool take = !cut;
                        if (cut) {
                            h = priority(keys[sl]);
                            const int hb = static_cast<int>(h >> (64 - kCutBits));
                            take = hb < sm.cut_bin;
                            cand = hb == sm.cut_bin;
                        }
                        if (take) mark(static_cast<int>(vals[sl] & 0xffffffffull));
                    }
                    if (cut) {
                        const int pos = warp_append(cand, &sm.own_cand);
                        if (pos >= 0) {
                            list[pos] = sl;
                            if (pos < kCandCap)
#pragma unroll 1
                                for (int r = 0; r < Q; ++r) *at_rank<Q>(cl, ch + rank * kCandCap + pos, r) = h;
                        }
                    }
                }
                if (cut) {
                    __syncthreads();
                    if (tid < Q) *at_rank<Q>(cl, &sm.ncand[rank], tid) = static_cast<int>(sm.own_cand);
                }
                csync<Q>(cl);
                tm.mark(4, j, l, 0);
                if (cut) {
                    // the boundary bin's candidates ranked exactly against the whole
                    // cluster's, a warp per candidate; the r smallest priorities are taken
                    const int c = static_cast<int>(sm.own_cand);
                    const int need = ml - sm.cut_below;
#pragma unroll 1
                    for (int f = wid; f < c; f += kWarps) {
                        const unsigned long long hf = priority(keys[list[f]]);
                        int rk = 0;
                        const int r = lane % Q;  // lanes of CTA r's candidates
                        const int cr = sm.ncand[r];
#pragma unroll 1
                        for (int k = lane / Q; k < cr; k += 32 / Q) {
                            // (beyond the received ones, from the CTA that holds them)
                            const unsigned long long hk =
                                (k < kCandCap) ? ch[r * kCandCap + k]
                                               : priority(at_rank<Q>(cl, keys, r)[at_rank<Q>(cl, list, r)[k]]);
                            rk += (hk < hf) ? 1 : 0;
                        }
                        rk = __reduce_add_sync(0xffffffffu, rk);
                        if (lane == 0 && rk < need) mark(static_cast<int>(vals[list[f]] & 0xffffffffull));
                    }
                    csync<Q>(cl);
                    tm.mark(5, j, l, 0);
                } else if (kstar < ml) {
                    // shortfall: untaken points in ascending level index until m_l
                    auto is_free = [&](int i) {
                        if constexpr (Q == 1) return !(reinterpret_cast<const uint32_t*>(pts + i)[3] >> 31);
                        else return !(__ldcg(reinterpret_cast<const uint32_t*>(stg + a + i) + 3) >> 31);
                    };
                    int cnt = 0;
#pragma unroll 1
                    for (int i = tid; i < L; i += kST) cnt += is_free(i) ? 1 : 0;
                    int tot;
                    scan_int(cnt, &tot);
                    if (tid < Q) *at_rank<Q>(cl, &sm.part_cnt[rank], tid) = tot;
                    csync<Q>(cl);
                    int before = 0;
#pragma unroll 1
                    for (int r2 = 0; r2 < rank; ++r2) before += sm.part_cnt[r2];
                    int budget = (ml - kstar) - before;
#pragma unroll 1
                    for (int i0 = 0; i0 < L && budget > 0; i0 += kST) {
                        const int i = i0 + tid;
                        const int free_pt = (i < L && is_free(i)) ? 1 : 0;
                        int chunk;
                        const int rk = scan_int(free_pt, &chunk);
                        if (free_pt && rk < budget) mark(a + i);
                        budget -= chunk;
                    }
                    csync<Q>(cl);
                    tm.mark(6, j, l, 0);
                }
                if (Q > 1 && in_smem && l + 1 < P.layers) {  // the copy in shared memory sees the marks
#pragma unroll 1
                    for (int i = tid; i < n; i += kST)
                        reinterpret_cast<uint32_t*>(pts + i)[3] = __ldcg(reinterpret_cast<const uint32_t*>(stg + i) + 3);
                }
                __syncthreads();
            }

            // ----------------------------------------------------- compaction
            // Segments in error take their first m points, as in the grid kernel.
            {
                long long obase = 0;  // this segment's first output position in the level array
#pragma unroll 1
                for (int s2 = 0; s2 < seg; ++s2) obase += P.m[j][s2];
                float4* nxt = reinterpret_cast<float4*>(ws + P.lay.ord[(j + 1) & 1]) + P.off0[seg];
                auto point = [&](int i) {
                    if constexpr (Q == 1) return pts[i];
                    else return __ldcg(stg + a + i);
                };
                auto kept = [&](int i, uint32_t w) { return err ? (a + i < m) : (w >> 31) != 0u; };
                int cnt = 0;
#pragma unroll 1
                for (int i = tid; i < L; i += kST) cnt += kept(i, __float_as_uint(point(i).w)) ? 1 : 0;
                int tot;
                scan_int(cnt, &tot);
                if (tid < Q) *at_rank<Q>(cl, &sm.part_cnt[rank], tid) = tot;
                csync<Q>(cl);
                tm.mark(7, j, 0, 0);
                int pos = 0;  // within the segment
#pragma unroll 1
                for (int r2 = 0; r2 < rank; ++r2) pos += sm.part_cnt[r2];
                int32_t* out = P.out[j] + obase;
                int32_t* orig_out = reinterpret_cast<int32_t*>(ws + P.lay.orig[j & 1]) + obase;
                const bool more = j + 1 < P.L;
                float mnv[3] = {INFINITY, INFINITY, INFINITY}, mxv[3] = {-INFINITY, -INFINITY, -INFINITY};
#pragma unroll 1
                for (int i0 = 0; i0 < L; i0 += kST) {
                    const int i = i0 + tid;
                    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (i < L) q = point(i);
                    const int keep = (i < L && kept(i, __float_as_uint(q.w))) ? 1 : 0;
                    int chunk;
                    const int rk = scan_int(keep, &chunk);
                    if (keep) {
                        if (pos + rk < m) {
                            const int o = static_cast<int>(__float_as_uint(q.w) & 0x7fffffffu);
                            out[pos + rk] = o;
                            if (P.keep_orig && !more) orig_out[pos + rk] = o;
                            if (more) {
                                q.w = __int_as_float(o);
                                // (Q = 1: in place, behind this round's reads)
                                if constexpr (Q == 1) pts[pos + rk] = q;
                                else __stcg(nxt + pos + rk, q);
                                mnv[0] = fminf(mnv[0], q.x);
                                mnv[1] = fminf(mnv[1], q.y);
                                mnv[2] = fminf(mnv[2], q.z);
                                mxv[0] = fmaxf(mxv[0], q.x);
                                mxv[1] = fmaxf(mxv[1], q.y);
                                mxv[2] = fmaxf(mxv[2], q.z);
                            }
                        } else {
                            seg_fail(sh, gh, seg, HAV_ERR_TABLE_FULL);  // cannot happen: every layer takes m_l
                        }
                    }
                    pos += chunk;
                }
                if (more) box_out<Q>(mnv, mxv, 0, rank);
                csync<Q>(cl);  // the next level reads the staged points and the boxes
                tm.mark(8, j, 0, 0);
            }
        }
        if (write_tr) {  // for a single-CTA launch that continues the chain
            sh[seg].guide_s = gs;
            sh[seg].guide_m = gm;
        }
    }
}

}  // namespace

// Sets a cluster kernel's launch attributes; the clusters that run at once, or -1.
template <int Q, bool kW>
static int set_up(cudaLaunchConfig_t* cfg) {
    int nc = 0;
    if (cudaFuncSetAttribute(hav_small_kernel<Q, kW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kSmallDyn)) != cudaSuccess)
        return -1;
    if (Q == 1) return 1;
    if (Q > 8 && cudaFuncSetAttribute(hav_small_kernel<Q, kW>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                     cudaSuccess)
        return -1;
    return cudaOccupancyMaxActiveClusters(&nc, hav_small_kernel<Q, kW>, cfg) == cudaSuccess ? nc : -1;
}

int small_clusters(int device, int q) {
    (void)device;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(q * 16));
    cfg.blockDim = dim3(kST);
    cfg.dynamicSmemBytes = kSmallDyn;
    if (q == 1) return set_up<1, false>(&cfg);
    if (q != 8 && q != 16) return -1;
    const int a = q == 8 ? set_up<8, false>(&cfg) : set_up<16, false>(&cfg);
    const int b = q == 8 ? set_up<8, true>(&cfg) : set_up<16, true>(&cfg);
    return a < b ? a : b;
}

int launch_small(const Plan& plan, int first_level, int q, int nclusters, cudaStream_t stream) {
    if (q != 8 && q != 16) return -1;
    // every level of the launch must fit its cluster's shared memory; sizes of 2^32
    // cells and more (kWide) are seldom met but near the points' own spacing, with
    // budgets of nearly all points (LiDAR scans of 16,384 points to 97 of 100 156 us
    // by kIndex, 91 by kWide; to 9/10 equal, of 24,000 151 and 97)
    bool wide = false;
    for (int j = first_level; j < plan.L; ++j)
#pragma unroll 1
        for (int s = 0; s < plan.S; ++s) {
            const long long n = (j == 0) ? plan.off0[s + 1] - plan.off0[s] : plan.m[j - 1][s];
            if (n > static_cast<long long>(kSmallMax)) return -1;
            wide = wide || (n > kWideMin && 8ll * plan.m[j][s] >= 7 * n);
        }
    int nc = nclusters < plan.S ? nclusters : plan.S;
    if (nc < 1) nc = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(q * nc));
    cfg.blockDim = dim3(kST);
    cfg.dynamicSmemBytes = kSmallDyn;
    cfg.stream = stream;
    const cudaError_t e =
        wide ? (q == 16 ? cudaLaunchKernelEx(&cfg, hav_small_kernel<16, true>, plan, first_level)
                        : cudaLaunchKernelEx(&cfg, hav_small_kernel<8, true>, plan, first_level))
             : (q == 16 ? cudaLaunchKernelEx(&cfg, hav_small_kernel<16, false>, plan, first_level)
                        : cudaLaunchKernelEx(&cfg, hav_small_kernel<8, false>, plan, first_level));
    return e == cudaSuccess ? 1 : -1;
}

int launch_solo(const Plan& plan, int first_level, int nblocks, cudaStream_t stream) {
    for (int j = first_level; j < plan.L; ++j)  // every level must fit one CTA
#pragma unroll 1
        for (int s = 0; s < plan.S; ++s) {
            const long long n = (j == 0) ? plan.off0[s + 1] - plan.off0[s] : plan.m[j - 1][s];
            if (n > static_cast<long long>(kSoloMax)) return -1;
        }
    int nc = nblocks < plan.S ? nblocks : plan.S;
    if (nc < 1) nc = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(nc));
    cfg.blockDim = dim3(kST);
    cfg.dynamicSmemBytes = kSmallDyn;
    cfg.stream = stream;
    return cudaLaunchKernelEx(&cfg, hav_small_kernel<1, false>, plan, first_level) == cudaSuccess ? 1 : -1;
}

}  // namespace havk
