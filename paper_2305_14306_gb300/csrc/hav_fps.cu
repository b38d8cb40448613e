// Farthest point sampling (Eq. 1 of Section 3.1), the comparator the paper
// measures HAVSampler against: clouds that fit the shared memory of one
// thread-block cluster on that cluster, many selected points per cluster
// barrier (a few selected points one per barrier); larger ones in one
// cooperative launch, one bounded grid barrier per selected point.
//
// Start at index 0; every point keeps its squared distance to the selected
// set (binary32, (dx*dx + dy*dy) + dz*dz without contraction); the next pick
// is the largest distance, ties to the lowest index; picked points are never
// picked again.

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "hav_device.cuh"
#include "hav_internal.h"

namespace cg = cooperative_groups;

namespace havk {
namespace {

constexpr int kFpsThreads = 1024;
constexpr size_t kFpsResidentBytes = 200 * 1024;  // shared memory for a block's resident points

// packed (distance bits, inverted index): the maximum is the farthest point,
// ties to the lowest index; picked points pack to 0 and never win
__device__ __forceinline__ unsigned long long fps_pack(float d2, int i) {
    return (static_cast<unsigned long long>(__float_as_uint(d2)) << 32) |
           static_cast<unsigned long long>(0xffffffffu - static_cast<unsigned>(i));
}

// kResident: the block's points and distances stay in shared memory (x, y,
// z, distance per point) for the whole run instead of being read from L2 in
// every round; the arithmetic and the picks are the same.
template <bool kResident>
__global__ void __launch_bounds__(kFpsThreads, 1)
    fps_kernel(const float* pts, int n, int m, int32_t* out, float* dist_g, unsigned long long* bmax, Barrier* bar,
               GlobalHdr* gh, int nblocks) {
    extern __shared__ float4 res[];
    __shared__ unsigned long long red[32];
    __shared__ int s_flag;
    __shared__ unsigned epoch;
    __shared__ int s_last;
    const int tid = threadIdx.x;
    if (tid == 0) epoch = 0u;
    const int chunk = (n + nblocks - 1) / nblocks;
    const int a = blockIdx.x * chunk;
    const int b = min(n, a + chunk);
    for (int i = a + tid; i < b; i += kFpsThreads) {
        if constexpr (kResident) res[i - a] = make_float4(pts[3ll * i], pts[3ll * i + 1], pts[3ll * i + 2], INFINITY);
        else dist_g[i] = INFINITY;
    }
    int last = 0;
    if (blockIdx.x == 0 && tid == 0) out[0] = 0;
    __syncthreads();
    for (int j = 1; j < m; ++j) {
        const float qx = pts[3ll * last], qy = pts[3ll * last + 1], qz = pts[3ll * last + 2];
        unsigned long long best = 0ull;
        for (int i = a + tid; i < b; i += kFpsThreads) {
            float px, py, pz, di;
            if constexpr (kResident) {
                const float4 r4 = res[i - a];
                px = r4.x;
                py = r4.y;
                pz = r4.z;
                di = r4.w;
            } else {
                di = dist_g[i];
            }
            if (i == last) {
                di = -1.0f;  // picked: never again
                if constexpr (kResident) res[i - a].w = di;
                else dist_g[i] = di;
            }
            if (di < 0.0f) continue;
            if constexpr (!kResident) {
                px = pts[3ll * i];
                py = pts[3ll * i + 1];
                pz = pts[3ll * i + 2];
            }
            const float dx = __fsub_rn(px, qx);
            const float dy = __fsub_rn(py, qy);
            const float dz = __fsub_rn(pz, qz);
            const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
            if (d2 < di) {
                di = d2;
                if constexpr (kResident) res[i - a].w = di;
                else dist_g[i] = di;
            }
            const unsigned long long k = fps_pack(di, i);
            best = k > best ? k : best;
        }
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, best, o);
            best = v > best ? v : best;
        }
        if ((tid & 31) == 0) red[tid >> 5] = best;
        __syncthreads();
        if (tid == 0) {
            unsigned long long bb = red[0];
            for (int w = 1; w < kFpsThreads / 32; ++w) bb = red[w] > bb ? red[w] : bb;
            bmax[(j & 1) * kMaxBlocks + blockIdx.x] = bb;
        }
        if (!grid_sync_impl(bar, gh, static_cast<unsigned>(nblocks), &epoch, &s_flag)) return;
        // every block finds the same maximum over the block maxima
        unsigned long long bb = 0ull;
        for (int k = tid; k < nblocks; k += kFpsThreads) {
            const unsigned long long v = bmax[(j & 1) * kMaxBlocks + k];
            bb = v > bb ? v : bb;
        }
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, bb, o);
            bb = v > bb ? v : bb;
        }
        if ((tid & 31) == 0) red[tid >> 5] = bb;
        __syncthreads();
        if (tid == 0) {
            unsigned long long m2 = red[0];
            for (int w = 1; w < kFpsThreads / 32; ++w) m2 = red[w] > m2 ? red[w] : m2;
            const int pick = static_cast<int>(0xffffffffu - static_cast<unsigned>(m2 & 0xffffffffull));
            s_last = (m2 != 0ull && pick >= 0 && pick < n) ? pick : 0;  // m <= n: an unpicked point exists
            if (blockIdx.x == 0) out[j] = s_last;
        }
        __syncthreads();
        last = s_last;
    }
}

constexpr int kFpsQ = 8;                  // CTAs of the one-pick cluster (portable size)
constexpr int kFpsQPoints = 4096;         // points one CTA of it holds
constexpr int kFpsClusterMax = kFpsQ * kFpsQPoints;

// a CTA's best candidate of a round with the point's coordinates
struct FpsCand {
    unsigned long long key;  // fps_pack of the CTA's farthest unpicked point
    float x, y, z, pad;
};

// Few picks of clouds of at most kFpsClusterMax points, one per cluster barrier:
// CTA r of one cluster holds points [r c, (r + 1) c), c = ceil(n / kFpsQ), with
// their distances in its shared memory.  Each round every CTA writes its best candidate into its own slot
// (two slots alternate), the cluster barrier publishes them, and every CTA
// takes the same maximum over the kFpsQ slots read through distributed shared
// memory; round j + 2 rewrites a slot only after every CTA has passed round
// j + 1's barrier, so no read of round j can see it.  The same arithmetic,
// ties and picks as fps_kernel.
__global__ void __cluster_dims__(kFpsQ, 1, 1) __launch_bounds__(kFpsThreads, 1)
    fps_cluster_kernel(const float* pts, int n, int m, int32_t* out) {
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ float4 res[];
    __shared__ unsigned long long red[32];
    __shared__ FpsCand cand[2];
    __shared__ float4 s_q;  // the last pick: x, y, z and its index bits
    const int tid = threadIdx.x;
    const int r = static_cast<int>(cl.block_rank());
    const int chunk = (n + kFpsQ - 1) / kFpsQ;
    const int a = r * chunk;
    const int b = min(n, a + chunk);
    for (int i = a + tid; i < b; i += kFpsThreads)
        res[i - a] = make_float4(pts[3 * i], pts[3 * i + 1], pts[3 * i + 2], INFINITY);
    if (r == 0 && tid == 0 && m > 0) out[0] = 0;
    float qx = 0.0f, qy = 0.0f, qz = 0.0f;
    if (n > 0) {
        qx = pts[0];
        qy = pts[1];
        qz = pts[2];
    }
    int last = 0;
    __syncthreads();
    for (int j = 1; j < m; ++j) {
        unsigned long long best = 0ull;
        for (int i = a + tid; i < b; i += kFpsThreads) {
            const float4 p4 = res[i - a];
            float di = p4.w;
            if (i == last) {
                di = -1.0f;  // picked: never again
                res[i - a].w = di;
            }
            if (di < 0.0f) continue;
            const float dx = __fsub_rn(p4.x, qx);
            const float dy = __fsub_rn(p4.y, qy);
            const float dz = __fsub_rn(p4.z, qz);
            const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
            if (d2 < di) {
                di = d2;
                res[i - a].w = di;
            }
            const unsigned long long k = fps_pack(di, i);
            best = k > best ? k : best;
        }
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, best, o);
            best = v > best ? v : best;
        }
        if ((tid & 31) == 0) red[tid >> 5] = best;
        __syncthreads();
        if (tid == 0) {
            unsigned long long bb = red[0];
            for (int w = 1; w < kFpsThreads / 32; ++w) bb = red[w] > bb ? red[w] : bb;
            FpsCand& c = cand[j & 1];
            c.key = bb;
            if (bb != 0ull) {  // this CTA's point: its coordinates travel with it
                const int g = static_cast<int>(0xffffffffu - static_cast<unsigned>(bb & 0xffffffffull));
                const float4 p4 = res[g - a];
                c.x = p4.x;
                c.y = p4.y;
                c.z = p4.z;
            }
        }
        cl.sync();
        if (tid == 0) {
            unsigned long long bk = 0ull;
            float bx = qx, by = qy, bz = qz;
            for (int q = 0; q < kFpsQ; ++q) {
                const FpsCand* c = cl.map_shared_rank(&cand[j & 1], q);
                const unsigned long long k = c->key;
                if (k > bk) {
                    bk = k;
                    bx = c->x;
                    by = c->y;
                    bz = c->z;
                }
            }
            const int pick = static_cast<int>(0xffffffffu - static_cast<unsigned>(bk & 0xffffffffull));
            const int s_last = (bk != 0ull && pick >= 0 && pick < n) ? pick : 0;  // m <= n: an unpicked point exists
            s_q = make_float4(bx, by, bz, __int_as_float(s_last));
            if (r == 0) out[j] = s_last;
        }
        __syncthreads();
        const float4 q4 = s_q;
        qx = q4.x;
        qy = q4.y;
        qz = q4.z;
        last = __float_as_int(q4.w);
    }
    cl.sync();  // no CTA leaves while another may still read its slots
}

// Clouds of up to kFpsMaxQ kFpsBatchPoints points: one cluster of Q CTAs picks many points
// per cluster barrier.  CTA r holds points r, r + Q, r + 2 Q, ... with their
// distances in its shared memory.  A round lists every point whose (distance,
// inverted index) key is at least a threshold and sends the list to every CTA.
// A point that is not listed stays below the threshold, as distances only
// shrink; so as long as the largest key among the listed points, lowered by the
// picks made meanwhile, is at least the threshold, it is the largest of all,
// and the next pick.  Every CTA finds these picks from the list alike, and then
// lowers its points' distances by all of them in one pass.
//
// The picks of a list, all at once (fps_resolve): in the order of their keys, a
// point that no earlier pick of the list comes nearer than its distance is a
// pick; the others are lowered.  Where a lowered point stays at or above the
// threshold, the picks end above its new key, as it may come next.  A list is
// resolved in as many steps as its longest chain of neighbours.
//
// The threshold follows the last pick's distance, as far below it as lately
// gave a list of 40 to 80 points; a list that is empty or too long is made
// again with another threshold (bisected between the two, on the whole key).
// A list gives about two thirds of its points as picks (16,384 uniform points
// to 4,096: about 110 lists).
//
// Measured on GB300: see launch_fps.
constexpr int kFpsBatchPoints = 12288;  // points one CTA holds (192 KB)
constexpr int kFpsListCap = 32;         // listed points per CTA
constexpr int kFpsList = 128;           // listed points of a round at most
constexpr int kFpsBatchThreads = 512;
static_assert(kFpsBatchThreads == 4 * kFpsList, "four threads rank a listed point");
constexpr int kFpsMaxQ = 16;

struct FpsBatchSmem {
    // by round parity: every CTA's listed points and counts, in every CTA's copy
    float4 pos[2][kFpsMaxQ][kFpsListCap];  // x, y, z, distance
    int idx[2][kFpsMaxQ][kFpsListCap];
    int cnt[2][kFpsMaxQ];
    unsigned mx[2][kFpsMaxQ];              // largest distance (bits + 1; 0: none left) of its unpicked points
    // the round's list, as received and in descending order of the keys; bit j of
    // near[i]: listed point j < i comes nearer to point i than its distance
    float4 c[kFpsList], s[kFpsList];
    unsigned long long key[kFpsList];
    int si[kFpsList];
    unsigned near[kFpsList][kFpsList / 32];
    float4 pick[kFpsList];                 // this round's picks
    int npick, own;
    unsigned wmax[kFpsBatchThreads / 32];
    float last;
};

__device__ __forceinline__ float fps_d2(const float4& p, const float4& q) {
    const float dx = __fsub_rn(p.x, q.x);
    const float dy = __fsub_rn(p.y, q.y);
    const float dz = __fsub_rn(p.z, q.z);
    return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

// The picks of one round from its list (above), at most `room` of them, into
// sm.pick and out; those of this CTA are marked in res.  The whole block calls
// it; its caller's barrier publishes what the first warp writes last.
template <int Q>
__device__ void fps_resolve(FpsBatchSmem& sm, int par, int total, unsigned long long thr, int room, int rank, float4* res,
                            int32_t* out) {
    constexpr int kW = kFpsList / 32;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid < kFpsList) {
        const int cnt = lane < Q ? sm.cnt[par][lane] : 0;
        const int end = warp_incl_scan(cnt);
        int r = 0;
#pragma unroll
        for (int s2 = Q / 2; s2 > 0; s2 >>= 1)  // the CTA r with end[r - 1] <= tid < end[r]
            if (__shfl_sync(0xffffffffu, end, r + s2 - 1) <= tid) r += s2;
        const int first = __shfl_sync(0xffffffffu, end - cnt, r);
        if (tid < total) {
            const float4 p = sm.pos[par][r][tid - first];
            sm.c[tid] = p;
            sm.key[tid] = fps_pack(p.w, sm.idx[par][r][tid - first]);
        }
    }
    __syncthreads();
    {
        const int e = tid >> 2;
        const unsigned long long k = e < total ? sm.key[e] : 0ull;
        int above = 0;
        for (int f = tid & 3; f < total; f += 4) above += sm.key[f] > k ? 1 : 0;
        above += __shfl_xor_sync(0xffffffffu, above, 1);
        above += __shfl_xor_sync(0xffffffffu, above, 2);
        if ((tid & 3) == 0 && e < total) {
            sm.s[above] = sm.c[e];
            sm.si[above] = static_cast<int>(0xffffffffu - static_cast<unsigned>(k & 0xffffffffull));
        }
    }
    __syncthreads();
    for (int i = wid; i < total; i += kFpsBatchThreads / 32) {
        const float4 p = sm.s[i];
#pragma unroll
        for (int u = 0; u < kW; ++u) {
            const int j = lane + 32 * u;
            const bool hit = j < i && fps_d2(p, sm.s[j]) < p.w;
            const unsigned b = __ballot_sync(0xffffffffu, hit);
            if (lane == 0) sm.near[i][u] = b;
        }
    }
    __syncthreads();
    if (wid != 0) return;
    // lane l: listed points l, l + 32, ...; decided and picked as bit sets
    unsigned nr[kW][kW], done[kW], picked[kW];
    float dist[kW];
#pragma unroll
    for (int u = 0; u < kW; ++u) {
        const int i = lane + 32 * u;
#pragma unroll
        for (int v = 0; v < kW; ++v) nr[u][v] = i < total ? sm.near[i][v] : 0u;
        dist[u] = i < total ? sm.s[i].w : 0.0f;
        done[u] = __ballot_sync(0xffffffffu, i >= total);
        picked[u] = 0u;
    }
    for (int step = 0; step < kFpsList; ++step) {  // (every step decides the first open point at least)
        unsigned d2[kW], p2[kW];
#pragma unroll
        for (int u = 0; u < kW; ++u) {
            unsigned open = 0u, hit = 0u;
#pragma unroll
            for (int v = 0; v < kW; ++v) {
                open |= nr[u][v] & ~done[v];
                hit |= nr[u][v] & picked[v];
            }
            // a near pick settles it at once, else every nearer point has to be decided
            d2[u] = __ballot_sync(0xffffffffu, open == 0u || hit != 0u);
            p2[u] = __ballot_sync(0xffffffffu, open == 0u && hit == 0u);
        }
        unsigned rest = 0u;
#pragma unroll
        for (int u = 0; u < kW; ++u) {
            picked[u] |= p2[u] & ~done[u];
            done[u] |= d2[u];
            rest |= ~done[u];
        }
        if (rest == 0u) break;
    }
    // the largest key a lowered point keeps, where it reaches the threshold
    unsigned stop = 0u;  // bits + 1 of its distance
#pragma unroll
    for (int u = 0; u < kW; ++u) {
        const int i = lane + 32 * u;
        if (i >= total || ((picked[u] >> lane) & 1u)) continue;
        const float4 p = sm.s[i];
        float w = p.w;
#pragma unroll
        for (int v = 0; v < kW; ++v)
            for (unsigned b = nr[u][v] & picked[v]; b; b &= b - 1u) w = fminf(w, fps_d2(p, sm.s[32 * v + __ffs(b) - 1]));
        if (fps_pack(w, sm.si[i]) >= thr) stop = max(stop, __float_as_uint(w) + 1u);
    }
    stop = __reduce_max_sync(0xffffffffu, stop);
    int before = 0;
#pragma unroll
    for (int u = 0; u < kW; ++u) {
        const bool take = ((picked[u] >> lane) & 1u) && __float_as_uint(dist[u]) + 1u > stop;
        const unsigned b = __ballot_sync(0xffffffffu, take);
        const int k = before + __popc(b & ((1u << lane) - 1u));
        if (take && k < room) {
            const int i = lane + 32 * u, g = sm.si[i];
            sm.pick[k] = sm.s[i];
            if (g % Q == rank) res[g / Q].w = -1.0f;  // picked: never again
            if (rank == 0) out[k] = g;
        }
        before += __popc(b);
    }
    __syncwarp();
    const int k = min(before, room);
    if (lane == 0) {
        sm.npick = k;
        sm.last = sm.pick[k - 1].w;
    }
}

template <int Q>
__global__ void __cluster_dims__(Q, 1, 1) __launch_bounds__(kFpsBatchThreads, 1)
    fps_batch_kernel(const float* pts, int n, int m, int32_t* out) {
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ float4 res[];
    __shared__ FpsBatchSmem sm;
    constexpr int T = kFpsBatchThreads;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int rank = static_cast<int>(cl.block_rank());
    const int mine = (n - rank + Q - 1) / Q;  // points rank, rank + Q, ...
    for (int i = tid; i < mine; i += T) {
        const float* p = pts + 3ll * (rank + static_cast<long long>(i) * Q);
        res[i] = make_float4(p[0], p[1], p[2], (i == 0 && rank == 0) ? -1.0f : INFINITY);
    }
    if (tid == 0) {
        sm.pick[0] = make_float4(pts[0], pts[1], pts[2], INFINITY);
        sm.npick = 1;
        sm.own = 0;
        if (rank == 0) out[0] = 0;
    }
    int j = 1, par = 0, k = 1;
    // the threshold; the largest that listed too many and the smallest that listed none
    unsigned long long thr = ~0ull, over = 0ull, none = ~0ull;
    bool have_over = false;
    float drop = 0.3f;
    cl.sync();  // every CTA runs before its memory is written to
    while (j < m) {
        // lower the distances by the last round's picks, list what reaches thr
        unsigned best = 0u;
#pragma unroll 1
        for (int i0 = tid; i0 < mine; i0 += 4 * T) {
            float4 p[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                p[u] = (i0 + u * T < mine) ? res[i0 + u * T] : make_float4(0.f, 0.f, 0.f, -1.0f);
#pragma unroll 2
            for (int q = 0; q < k; ++q) {
                const float4 pk = sm.pick[q];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float d2 = fps_d2(p[u], pk);
                    if (d2 < p[u].w) p[u].w = d2;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u * T;
                if (i >= mine || !(p[u].w >= 0.0f)) continue;
                if (k > 0) res[i].w = p[u].w;
                best = max(best, __float_as_uint(p[u].w) + 1u);
                const int g = rank + i * Q;
                if (fps_pack(p[u].w, g) >= thr) {
                    const int slot = atomicAdd(&sm.own, 1);
                    if (slot < kFpsListCap)
                        for (int r = 0; r < Q; ++r) {
                            *cl.map_shared_rank(&sm.pos[par][rank][slot], r) = p[u];
                            *cl.map_shared_rank(&sm.idx[par][rank][slot], r) = g;
                        }
                }
            }
        }
        best = __reduce_max_sync(0xffffffffu, best);
        if (lane == 0) sm.wmax[wid] = best;
        __syncthreads();
        if (wid == 0) {
            const unsigned b = __reduce_max_sync(0xffffffffu, lane < (T >> 5) ? sm.wmax[lane] : 0u);
            if (lane < Q) {
                *cl.map_shared_rank(&sm.cnt[par][rank], lane) = sm.own;
                *cl.map_shared_rank(&sm.mx[par][rank], lane) = b;
            }
            __syncwarp();
            if (lane == 0) sm.own = 0;
        }
        cl.sync();
        const int cr = lane < Q ? sm.cnt[par][lane] : 0;
        const int total = __reduce_add_sync(0xffffffffu, cr);
        const bool long_list = __any_sync(0xffffffffu, cr > kFpsListCap) || total > kFpsList;
        const unsigned mxb = __reduce_max_sync(0xffffffffu, lane < Q ? sm.mx[par][lane] : 0u);
        const int pp = par;
        par ^= 1;
        k = 0;
        if (total == 0) {
            // too high (or the first round): below the largest distance, or between the two
            none = min(none, thr);
            const float d = __uint_as_float(mxb - 1u);  // (m <= n: an unpicked point exists)
            if (have_over) thr = over + (none - over) / 2;
            else thr = static_cast<unsigned long long>(__float_as_uint(__fmul_rn(d, 1.0f - drop))) << 32;
            continue;
        }
        if (long_list) {
            over = thr;
            have_over = true;
            none = min(none, static_cast<unsigned long long>(mxb) << 32);
            thr = over + (none - over) / 2;
            drop *= 0.7f;
            continue;
        }
        fps_resolve<Q>(sm, pp, total, thr, min(m - j, kFpsList), rank, res, out + j);
        __syncthreads();
        k = sm.npick;
        j += k;
        // (a long list lowers it at every look, which suits a run of tied distances,
        // to 0 in the end; from there, and from far below what distinct distances
        // need, it has to come back)
        if (total < 40) drop = fminf(0.9f, drop * (drop < 1e-2f ? 2.0f : 1.25f) + 1e-7f);
        else if (total > 80) drop *= 0.8f;
        thr = static_cast<unsigned long long>(__float_as_uint(__fmul_rn(sm.last, 1.0f - drop))) << 32;
        have_over = false;
        none = ~0ull;
    }
    cl.sync();  // no CTA leaves while another may still write to it
}

}  // namespace

int fps_coresident_blocks(int device) {
    int sms = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return -1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fps_kernel<false>, kFpsThreads, 0) != cudaSuccess)
        return -1;
    long long nb = static_cast<long long>(sms) * per_sm;
    if (nb > kMaxBlocks) nb = kMaxBlocks;
    return static_cast<int>(nb);
}

template <int Q>
static bool launch_fps_batch(const float* points, int n, int m, int32_t* out, cudaStream_t stream) {
    const int chunk = (n + Q - 1) / Q;
    if (chunk > kFpsBatchPoints) return false;
    bool ok = cudaFuncSetAttribute(fps_batch_kernel<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   static_cast<int>(kFpsBatchPoints * sizeof(float4))) == cudaSuccess;
    if (Q > 8) ok = ok && cudaFuncSetAttribute(fps_batch_kernel<Q>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
                              cudaSuccess;
    if (ok) {
        cudaLaunchConfig_t cc = {};
        cc.gridDim = dim3(Q);
        cc.blockDim = dim3(kFpsBatchThreads);
        cc.dynamicSmemBytes = static_cast<size_t>(chunk < 1 ? 1 : chunk) * sizeof(float4);
        cc.stream = stream;
        if (cudaLaunchKernelEx(&cc, fps_batch_kernel<Q>, points, n, m, out) == cudaSuccess) return true;
    }
    (void)cudaGetLastError();  // a refused launch configuration leaves no sticky error
    return false;
}

static bool launch_fps_cluster(const float* points, int n, int m, int32_t* out, cudaStream_t stream) {
    if (n > kFpsClusterMax) return false;
    const int chunk = (n + kFpsQ - 1) / kFpsQ;
    if (cudaFuncSetAttribute(fps_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(kFpsQPoints * sizeof(float4))) == cudaSuccess) {
        cudaLaunchConfig_t cc = {};
        cc.gridDim = dim3(kFpsQ);
        cc.blockDim = dim3(kFpsThreads);
        cc.dynamicSmemBytes = static_cast<size_t>(chunk < 1 ? 1 : chunk) * sizeof(float4);
        cc.stream = stream;
        if (cudaLaunchKernelEx(&cc, fps_cluster_kernel, points, n, m, out) == cudaSuccess) return true;
    }
    (void)cudaGetLastError();  // a refused launch configuration leaves no sticky error
    return false;
}

int launch_fps(const float* points, int n, int m, int32_t* out, unsigned char* ws, const Layout& lay, int nblocks,
               cudaStream_t stream) {
    // scratch: the distance array in the first log array, block maxima in the phase-timer region
    float* dist = reinterpret_cast<float*>(ws + lay.dirty[0]);
    unsigned long long* bmax = reinterpret_cast<unsigned long long*>(ws + lay.ptimes);
    Barrier* bar = reinterpret_cast<Barrier*>(ws + lay.barrier);
    GlobalHdr* gh = reinterpret_cast<GlobalHdr*>(ws + lay.ghdr);
    // one cluster where its CTAs hold the points, of 16 CTAs or 8 (where the
    // device refuses the cluster, the grid form below).  Measured on GB300
    // against one pick per barrier (a cluster of 8 up to 32,768 points, the grid
    // form above): 16,384 uniform points to 4,096 7.14 -> 0.83 ms, a room of
    // 32,768 to 3,500 6.89 -> 0.79 ms, a LiDAR scan of 100,000 to 1,500 3.99 ->
    // 1.12 ms, 1,000 points to 500 0.78 -> 0.11 ms.  A round of about 40 picks
    // takes 7 us, a third of it the distances, the rest the list's short
    // sections between barriers
    //
    // Few picks go one by one: the first ones lie far apart, so that a list gives one
    // or two of them and its threshold is found anew for each.  Picks from which on
    // the lists win, 1,000 / 4,096 / 16,384 / 32,768 / 100,000 / 196,608 points of a
    // box and a room: 10-25 / 45 / 57 / 65 / 85-95 / 140; 8 picks take 21 / 21 / 22 /
    // 24 / 29 / 31 us one by one, 26 / 43 / 49 / 57 / 84 / 125 from lists.  (The line
    // lies at 20 / 46 / 52 / 60 / 92 / 140.)
    const bool few = m < n / 48 && m < 44 + n / 2048;
    if (few && launch_fps_cluster(points, n, m, out, stream)) return 1;
    if (!few && (launch_fps_batch<16>(points, n, m, out, stream) || launch_fps_batch<8>(points, n, m, out, stream)))
        return 1;
    // fewer blocks than points per block of work would only add barrier arrivals
    int nb = nblocks;
    const int want = (n + kFpsThreads - 1) / kFpsThreads;
    if (want < nb) nb = want < 1 ? 1 : want;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(nb));
    cfg.blockDim = dim3(kFpsThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    // the block's share resident in shared memory where it fits and the grid
    // stays co-resident with that much shared memory per block
    const long long chunk = (static_cast<long long>(n) + nb - 1) / nb;
    const size_t bytes = static_cast<size_t>(chunk) * sizeof(float4);
    bool resident = bytes <= kFpsResidentBytes &&
                    cudaFuncSetAttribute(fps_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(kFpsResidentBytes)) == cudaSuccess;
    if (resident) {
        int dev = 0, sms = 0, per_sm = 0;
        resident = cudaGetDevice(&dev) == cudaSuccess &&
                   cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
                   cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fps_kernel<true>, kFpsThreads, bytes) ==
                       cudaSuccess &&
                   static_cast<long long>(sms) * per_sm >= nb;
    }
    if (resident) {
        cfg.dynamicSmemBytes = bytes;
        return cudaLaunchKernelEx(&cfg, fps_kernel<true>, points, n, m, out, dist, bmax, bar, gh, nb) == cudaSuccess
                   ? 1
                   : -1;
    }
    return cudaLaunchKernelEx(&cfg, fps_kernel<false>, points, n, m, out, dist, bmax, bar, gh, nb) == cudaSuccess
               ? 1
               : -1;
}

}  // namespace havk
