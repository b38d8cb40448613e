// Grouping around sampled centres: the step after sampling in the
// sample-group-aggregate block (Section 3.1), the ball query of PointNet++.
// For centre j (point centres[j]) the nsample smallest indices k with
// (dx*dx + dy*dy) + dz*dz < radius*radius (binary32, no fusion), ascending;
// missing slots repeat the smallest.  The offsets p_k - c_j of every slot are
// written beside them (the gather of the block, fused).
//
// A uniform grid with cells of at least the radius (so every ball lies in the
// 3 x 3 x 3 cells around its centre's cell) is built by a counting sort of the
// points by cell, and within a cell by index in up to 64 steps: a cell's points
// with small indices come first.  One warp per centre then goes through those
// cells, all of them together, step by step of the indices, collects the
// qualifying indices in shared memory and stops at the first step after which
// it has nsample of them (every later index is larger); where the buffer
// fills, it is sorted and cut to the nsample smallest, the largest kept one
// then bounding the rest.  The result does not depend on the grid, only the
// work does.  Two kernels on the caller's stream: the grid build (one
// cooperative launch) and the query.
//
// What bounds it, at 65,536 centres among 1,048,576 points of a room, radius
// 0.2, nsample 32, on GB300 (times of one call, device):
//   build 42 us (from 51): five grid barriers of 1.3 to 2.5 us each, the counts
//     (1 M atomics, 4.5 us) and the scatter (1 M atomics that return, 12 us);
//   query 91 us (from 549): instructions.  A 27-cell neighbourhood holds some
//     6,000 points of which 2,000 qualify and 32 are asked for, so without the
//     steps nearly all of the work is thrown away (500 us of the query's time);
//     with 16 steps in place of 64 the call takes the same here and 162 us in
//     place of 99 for 4,096 centres of radius 0.8.  The points lie in cell order with their
//     indices (float4): the scan of a bucket is one coalesced load and no gather.
// The buckets (cells times steps) stay below four per point: beyond that the
// clearing and the scan of empty buckets cost more than shorter steps give
// (radius 0.05: 119 us with 2.4 M cells of 4 steps, 107 us of one).

#include <cuda_runtime.h>

#include "hav.h"
#include "hav_device.cuh"
#include "hav_internal.h"

namespace havk {
namespace {

constexpr int kBuildThreads = 1024;  // of the grid build
constexpr int kGrpMaxSample = 256;
constexpr int kScanItems = 16;                       // buckets per thread in the scan
constexpr int kStepsLog2 = 6;                        // index steps per cell at most (64)
constexpr long long kMaxCells = 1ll << 24;

struct GroupGrid {
    uint32_t box[6];  // ~enc(min xyz), enc(max xyz), atomicMax'ed
    float mn[3];
    float inv_h;
    int dims[3];
    int steps_log2;   // index steps per cell
    int step_shift;   // a point's step: its index >> step_shift
    int pad;
    long long cells;
};

__device__ __forceinline__ int axis_cell(float x, float mn, float inv_h, int dim) {
    const float t = __fmul_rn(__fsub_rn(x, mn), inv_h);
    int c = (t > 0.0f) ? static_cast<int>(t) : 0;
    return c < dim ? c : dim - 1;
}

__device__ __forceinline__ long long cell_of(const float* p, const GroupGrid& g, int c[3]) {
    for (int a = 0; a < 3; ++a) c[a] = axis_cell(p[a], g.mn[a], g.inv_h, g.dims[a]);
    return (static_cast<long long>(c[2]) * g.dims[1] + c[1]) * g.dims[0] + c[0];
}

// Cell size h >= radius (1 + 2^-10) and at least 1/256 of the largest
// extent, grown by 2^(1/3) until the grid has at most `budget` cells.  With
// at most 257 cells per axis the cell map t = (x - mn) * RN(1/h) is off by
// under 2^-12 cells, so two points closer than the radius (under 1 - 2^-10
// cells apart) never land more than one cell apart.
__device__ void setup_grid(GroupGrid* g, float radius, long long budget) {
    float ext = 0.0f, e[3];
    for (int a = 0; a < 3; ++a) {
        g->mn[a] = dec_f(~g->box[a]);
        const float mx = dec_f(g->box[3 + a]);
        e[a] = (mx >= g->mn[a]) ? __fsub_rn(mx, g->mn[a]) : 0.0f;
        ext = fmaxf(ext, e[a]);
        if (!(mx >= g->mn[a])) g->mn[a] = 0.0f;  // no finite point
    }
    float h = fmaxf(__fmul_rn(radius, 1.0009765625f), __fmul_rn(ext, 0.00390625f));
    if (!isfinite(h)) {  // an extent beyond binary32: one cell
        g->dims[0] = g->dims[1] = g->dims[2] = 1;
        g->inv_h = 0.0f;
        g->cells = 1;
        return;
    }
    long long cells = 0;
    for (int guard = 0; guard < 200; ++guard) {
        cells = 1;
        for (int a = 0; a < 3; ++a) {
            const long long d = static_cast<long long>(__fdiv_rn(e[a], h)) + 1;
            g->dims[a] = static_cast<int>(d);
            cells *= d;
        }
        if (cells <= budget) break;
        h = __fmul_rn(h, 1.2599210739135742f);
    }
    g->inv_h = __fdiv_rn(1.0f, h);
    g->cells = cells;
}

// f(i, x, y, z) for the points [0, n), spread over the grid; four points' loads
// in flight per thread.
template <typename F>
__device__ __forceinline__ void grid_points(const float* pts, long long n, F&& f) {
    const long long stride = static_cast<long long>(gridDim.x) * kBuildThreads;
#pragma unroll 1
    for (long long i0 = blockIdx.x * static_cast<long long>(kBuildThreads) + threadIdx.x; i0 < n; i0 += 4 * stride) {
        float p[4][3];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const long long i = i0 + k * stride < n ? i0 + k * stride : n - 1;
#pragma unroll
            for (int a = 0; a < 3; ++a) p[k][a] = __ldg(pts + 3 * i + a);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (i0 + k * stride < n) f(i0 + k * stride, p[k]);
    }
}

// The grid in one cooperative launch, its phases separated by grid barriers
// (bounded waits; a wait that gives up sets the abort flag, which the query
// honours): bounding box; set-up (every block alike) and cleared counts; cell
// counts; the total of each block's share of the buckets; the shares' scans; the
// scatter of the points with their indices.  Afterwards end[b] holds the end of
// bucket b = (cell << steps_log2) + step in sorted (its start is end[b - 1]).
__global__ void __launch_bounds__(kBuildThreads, 1)
    grp_build(const float* pts, long long n, float radius, long long budget, int max_steps_log2, GroupGrid* g,
              uint32_t* end, uint32_t* block_sums, float4* sorted, Barrier* bar, GlobalHdr* gh) {
    __shared__ GroupGrid sg;
    __shared__ unsigned epoch;
    __shared__ int flag;
    __shared__ uint32_t scratch[32];
    __shared__ float redf[6][32];
    const int tid = threadIdx.x;
    const unsigned nb = gridDim.x;
    const long long gtid = blockIdx.x * static_cast<long long>(kBuildThreads) + tid;
    const long long gstride = static_cast<long long>(nb) * kBuildThreads;
    if (tid == 0) epoch = 0u;
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    grid_points(pts, n, [&](long long, const float* p) {
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (isfinite(p[a])) {
                mn[a] = fminf(mn[a], p[a]);
                mx[a] = fmaxf(mx[a], p[a]);
            }
    });
    for (int a = 0; a < 3; ++a)
        for (int o = 16; o > 0; o >>= 1) {
            mn[a] = fminf(mn[a], __shfl_xor_sync(0xffffffffu, mn[a], o));
            mx[a] = fmaxf(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], o));
        }
    if ((tid & 31) == 0)
        for (int a = 0; a < 3; ++a) {
            redf[a][tid >> 5] = mn[a];
            redf[3 + a][tid >> 5] = mx[a];
        }
    __syncthreads();
    if (tid < 6) {
        float r = redf[tid][0];
        for (int w = 1; w < kBuildThreads / 32; ++w) r = (tid < 3) ? fminf(r, redf[tid][w]) : fmaxf(r, redf[tid][w]);
        if (isfinite(r)) atomicMax(&g->box[tid], (tid < 3) ? ~enc_f(r) : enc_f(r));
    }
    if (!grid_sync_impl(bar, gh, nb, &epoch, &flag)) return;

    if (tid == 0) {
        for (int a = 0; a < 6; ++a) sg.box[a] = ld_volatile_u(&g->box[a]);
        setup_grid(&sg, radius, budget);
        int lg = max_steps_log2, sh = 0;
        while (lg > 0 && (sg.cells << lg) > min(budget, 4 * n)) --lg;
        while (((n - 1) >> sh) >= (1ll << lg)) ++sh;
        sg.steps_log2 = lg;
        sg.step_shift = sh;
        if (blockIdx.x == 0) *g = sg;  // for the query
    }
    __syncthreads();
    const long long buckets = sg.cells << sg.steps_log2;
    for (long long i = gtid; i < buckets; i += gstride) end[i] = 0u;
    if (!grid_sync_impl(bar, gh, nb, &epoch, &flag)) return;
    const int lg = sg.steps_log2, sh = sg.step_shift;
    grid_points(pts, n, [&](long long i, const float* p) {
        int c[3];
        atomicAdd(&end[(cell_of(p, sg, c) << lg) + (i >> sh)], 1u);
    });
    if (!grid_sync_impl(bar, gh, nb, &epoch, &flag)) return;

    // this block's share of the buckets: its total, then, past the totals before
    // it, an exclusive scan in place (16 buckets per thread at a time)
    const long long share = ((buckets + nb - 1) / nb + 3) & ~3ll;
    const long long cb = share * blockIdx.x;
    const long long ce = (cb + share < buckets) ? cb + share : buckets;
    auto four = [&](long long i) {  // end[i, i + 4), what lies past the share as 0 (i and cb are multiples of 4)
        if (i + 4 <= ce) return *reinterpret_cast<const uint4*>(end + i);
        return make_uint4(i < ce ? end[i] : 0u, i + 1 < ce ? end[i + 1] : 0u, i + 2 < ce ? end[i + 2] : 0u, 0u);
    };
    uint32_t sum = 0;
#pragma unroll 4
    for (long long i = cb + 4 * tid; i < ce; i += 4 * kBuildThreads) {
        const uint4 v = four(i);
        sum += (v.x + v.y) + (v.z + v.w);
    }
    uint32_t run;
    block_excl_scan<uint32_t, kBuildThreads>(sum, &run, scratch);
    if (tid == 0) block_sums[blockIdx.x] = run;
    if (!grid_sync_impl(bar, gh, nb, &epoch, &flag)) return;

    uint32_t pre = 0;
    for (unsigned b = tid; b < blockIdx.x; b += kBuildThreads) pre += ld_volatile_u(&block_sums[b]);
    block_excl_scan<uint32_t, kBuildThreads>(pre, &run, scratch);
#pragma unroll 1
    for (long long t0 = cb; t0 < ce; t0 += kBuildThreads * kScanItems) {
        const long long i0 = t0 + static_cast<long long>(tid) * kScanItems;
        uint4 v[kScanItems / 4];
        uint32_t mine = 0, tot;
#pragma unroll
        for (int k = 0; k < kScanItems / 4; ++k) {
            v[k] = four(i0 + 4 * k);
            mine += (v[k].x + v[k].y) + (v[k].z + v[k].w);
        }
        uint32_t at = run + block_excl_scan<uint32_t, kBuildThreads>(mine, &tot, scratch);
#pragma unroll
        for (int k = 0; k < kScanItems / 4; ++k) {
            const long long i = i0 + 4 * k;
            const uint4 w = make_uint4(at, at + v[k].x, at + v[k].x + v[k].y, at + v[k].x + v[k].y + v[k].z);
            at = w.w + v[k].w;
            if (i + 4 <= ce) {
                *reinterpret_cast<uint4*>(end + i) = w;
            } else {
                if (i < ce) end[i] = w.x;
                if (i + 1 < ce) end[i + 1] = w.y;
                if (i + 2 < ce) end[i + 2] = w.z;
            }
        }
        run += tot;
    }
    if (!grid_sync_impl(bar, gh, nb, &epoch, &flag)) return;

    grid_points(pts, n, [&](long long i, const float* p) {
        int c[3];
        const uint32_t pos = atomicAdd(&end[(cell_of(p, sg, c) << lg) + (i >> sh)], 1u);
        if (pos < static_cast<uint32_t>(n))
            sorted[pos] = make_float4(p[0], p[1], p[2], __int_as_float(static_cast<int>(i)));
    });
}

// One warp per centre: the lanes test 32 candidates of the 27 cells at a time.
constexpr int kQueryWarps = 4;  // warps per block of the query
constexpr int kQueryBlocks = 40;  // blocks of the query per SM at most
constexpr int kCollect = 512;   // qualifying points a warp collects at most before it sorts and cuts them

// Ascending bitonic sort of buf[0, cnt) by one warp (cnt <= kCollect; the
// rest of the next power of two is padded with the largest index).
__device__ __forceinline__ void sort_prefix(int32_t* buf, int cnt, int lane) {
    int n2 = 32;
    while (n2 < cnt) n2 <<= 1;
    for (int e = cnt + lane; e < n2; e += 32) buf[e] = 0x7fffffff;
    __syncwarp();
    for (int k2 = 2; k2 <= n2; k2 <<= 1)
        for (int j2 = k2 >> 1; j2 > 0; j2 >>= 1) {
            for (int i = lane; i < n2; i += 32) {
                const int ixj = i ^ j2;
                if (ixj > i) {
                    const int32_t u = buf[i], w = buf[ixj];
                    if ((u > w) == ((i & k2) == 0)) {
                        buf[i] = w;
                        buf[ixj] = u;
                    }
                }
            }
            __syncwarp();
        }
}

// buf[0, cnt) ascending, cnt <= 32 U: U values per lane, value i in lane i % 32
// (bitonic; steps below 32 exchange between lanes, the others within a lane).
template <int U>
__device__ __forceinline__ void sort_lanes(int32_t* buf, int cnt, int lane) {
    int32_t v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = (lane + 32 * u < cnt) ? buf[lane + 32 * u] : 0x7fffffff;
#pragma unroll
    for (int k2 = 2; k2 <= 32 * U; k2 <<= 1)
#pragma unroll
        for (int j2 = k2 >> 1; j2 > 0; j2 >>= 1) {
            if (j2 >= 32) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int w = u ^ (j2 / 32);
                    if (w > u) {
                        const bool up = ((32 * u) & k2) == 0;
                        const int32_t lo = min(v[u], v[w]), hi = max(v[u], v[w]);
                        v[u] = up ? lo : hi;
                        v[w] = up ? hi : lo;
                    }
                }
            } else {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int32_t o = __shfl_xor_sync(0xffffffffu, v[u], j2);
                    const bool up = (((lane + 32 * u) & k2) == 0) == ((lane & j2) == 0);
                    v[u] = up ? min(v[u], o) : max(v[u], o);
                }
            }
        }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < U; ++u) buf[lane + 32 * u] = v[u];
    __syncwarp();
}

__global__ void __launch_bounds__(32 * kQueryWarps)
    grp_query(const float* pts, long long n, const int32_t* centres, long long m, float radius, int nsample,
              const GroupGrid* g, const uint32_t* end, const float4* sorted, int32_t* out_idx, float* out_xyz,
              int32_t* status, const GlobalHdr* gh) {
    __shared__ int32_t sbuf[kQueryWarps][kCollect];
    __shared__ int sfirst[kQueryWarps][32];
    if (ld_volatile(&gh->abort)) return;  // the build gave up (its status says so)
    const GroupGrid G = *g;
    const float r2 = __fmul_rn(radius, radius);
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const int wib = threadIdx.x >> 5;
    int32_t* buf = sbuf[wib];
    int* from = sfirst[wib];
    int cap = 64;
    while (cap < 2 * nsample && cap < kCollect) cap <<= 1;
    const int steps = 1 << G.steps_log2;
    const int ox = lane % 3 - 1, oy = lane / 3 % 3 - 1, oz = lane / 9 - 1;  // lane l < 27: cell l of the 27
    const long long warps = static_cast<long long>(gridDim.x) * kQueryWarps;
#pragma unroll 1
    for (long long j = blockIdx.x * static_cast<long long>(kQueryWarps) + wib; j < m; j += warps) {
        const int32_t ci = centres[j];
        int32_t* row = out_idx + j * nsample;
        if (ci < 0 || ci >= n) {
            if (lane == 0) atomicCAS(status, 0, static_cast<int>(HAV_ERR_INVALID));
            for (int s = lane; s < nsample; s += 32) row[s] = 0;
            if (out_xyz)
                for (int s = lane; s < 3 * nsample; s += 32) out_xyz[j * 3 * nsample + s] = 0.0f;
            continue;
        }
        const float cx = pts[3u * ci], cy = pts[3u * ci + 1], cz = pts[3u * ci + 2];  // (n < 2^30)
        const int x = axis_cell(cx, G.mn[0], G.inv_h, G.dims[0]) + ox, y = axis_cell(cy, G.mn[1], G.inv_h, G.dims[1]) + oy,
                  z = axis_cell(cz, G.mn[2], G.inv_h, G.dims[2]) + oz;
        const bool in = lane < 27 && x >= 0 && x < G.dims[0] && y >= 0 && y < G.dims[1] && z >= 0 && z < G.dims[2];
        // this lane's cell: its buckets from b0 (at most kMaxCells of them in all), its points [cur, stop) in sorted
        const int b0 = ((z * G.dims[1] + y) * G.dims[0] + x) << G.steps_log2;
        uint32_t cur = 0u, stop = 0u;
        if (in) {
            cur = b0 > 0 ? end[b0 - 1] : 0u;
            stop = end[b0 + steps - 1];
        }
        const int all = static_cast<int>(__reduce_add_sync(0xffffffffu, stop - cur));
        int cnt = 0, done = 0;  // qualifying indices collected, steps gone through
        int32_t top = 0x7fffffff;
        while (done < steps && cnt < nsample) {
            // the steps of this round: about 4 nsample candidates (a sixth to a third of
            // them qualify), then as many as before again; all where that is most of them
            int next = 2 * done;
            if (done == 0) {
                const float share = __fdividef(4.0f * nsample, static_cast<float>(all + 1));
                next = max(1, static_cast<int>(share * static_cast<float>(steps) + 0.5f));
            }
            if (next > steps || all <= 6 * nsample) next = steps;
            const uint32_t till = (next == steps || !in) ? stop : end[b0 + next - 1];
            const int len = static_cast<int>(till - cur);
            const int ends = warp_incl_scan(len);
            const int total = __shfl_sync(0xffffffffu, ends, 31);
            const int start = ends - len;
            // candidate e lies at sorted[from[i] + e], i the number of the cell's among those with candidates
            const unsigned some = __ballot_sync(0xffffffffu, len > 0);
            if (len > 0) from[__popc(some & below)] = static_cast<int>(cur) - start;
            __syncwarp();
            int before = -1;  // cells that start before this batch, less 1
            for (int e0 = 0; e0 < total; e0 += 32) {  // warp-uniform
                const int e = e0 + lane;
                const unsigned here = static_cast<unsigned>(start - e0);
                const unsigned starts = __reduce_or_sync(0xffffffffu, (len > 0 && here < 32u) ? 1u << here : 0u);
                int32_t k = 0;
                bool ok = false;
                if (e < total) {
                    const float4 q = sorted[from[before + __popc(starts & (below << 1 | 1u))] + e];
                    k = __float_as_int(q.w);
                    const float ex = __fsub_rn(q.x, cx), ey = __fsub_rn(q.y, cy), ez = __fsub_rn(q.z, cz);
                    const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
                    ok = d2 < r2 && k < top;
                }
                before += __popc(starts);
                // the qualifying indices, unsorted, into the warp's buffer; when it is
                // full it is sorted and cut to the nsample smallest, whose largest then
                // bounds every later index (indices are distinct)
                unsigned mask = __ballot_sync(0xffffffffu, ok);
                if (cnt + __popc(mask) > cap) {  // (warp-uniform)
                    __syncwarp();
                    sort_prefix(buf, cnt, lane);
                    if (cnt > nsample) cnt = nsample;
                    if (cnt == nsample) top = buf[nsample - 1];
                    ok = ok && k < top;
                    mask = __ballot_sync(0xffffffffu, ok);
                }
                if (ok) buf[cnt + __popc(mask & below)] = k;
                cnt += __popc(mask);
            }
            __syncwarp();  // from is rewritten for the next round
            cur = till;
            done = next;
        }
        if (cnt <= 32)
            sort_lanes<1>(buf, cnt, lane);
        else if (cnt <= 64)
            sort_lanes<2>(buf, cnt, lane);
        else if (cnt <= 128)
            sort_lanes<4>(buf, cnt, lane);
        else
            sort_prefix(buf, cnt, lane);
        if (cnt > nsample) cnt = nsample;
        if (cnt == 0) {  // unreachable: the centre is at distance 0
            if (lane == 0) buf[0] = ci;
            __syncwarp();
            cnt = 1;
        }
        for (int s = lane; s < nsample; s += 32) {
            const int32_t k = buf[s < cnt ? s : 0];
            row[s] = k;
            if (out_xyz) {
                float* o = out_xyz + (j * nsample + s) * 3;
                o[0] = __fsub_rn(pts[3u * k], cx);
                o[1] = __fsub_rn(pts[3u * k + 1], cy);
                o[2] = __fsub_rn(pts[3u * k + 2], cz);
            }
        }
        __syncwarp();  // the list is rewritten for the next centre
    }
}

// ------------------------------------------------------ spacing on the grid
// The Fig. 3 spacing of a large subset (hav_spacing): the subset's points are
// gathered (an invalid index or a non-finite coordinate as NaN: no distance
// involving such a point is ever below another, exactly as in the all-pairs
// search), the grid above is built over them (cells of 1/256 of the largest
// extent, grown to kSpacingCells per point at most), and one thread per point,
// in cell order, visits the 27 cells around its own; for the points that need
// more, the whole warp visits the shells of cells at Chebyshev distance 2, 3,
// ..., one point after another, until no cell farther out can hold a nearer
// point.  A point of a cell r + 1 or more shells away lies at least (r - 0.01)
// h away (the cell map is exact to far less than 0.01 cells), and a computed
// squared distance is within a relative 2^-20 of the exact one, so the search
// stops once best < ((r - 0.01) h)^2 (1 - 2^-20), every bound rounded down.
// Where a box of shells has more rows of cells than kRowCost-th of the subset's
// points, the warp scans the whole subset instead.
//
// Measured on GB300 (one call with its histogram): 262,144 points of a room 65
// us (174 with one thread per point through all shells and an index list in
// place of the points), of which gather 5, build 24, search 24, histogram 6;
// 65,536 of a LiDAR scan 308 us (3,743: its far returns, next to one another in
// cell order, searched thousands of rows of cells one by one).  The cells per
// point: 2 / 4 / 8 / 16 / 32 take 71 / 67 / 71 / 83 / 106 us on the room and
// 710 / 483 / 316 / 257 / 257 us on the scan, whose cells near the sensor are
// crowded; 8 is within 6 % of the best on the room.
constexpr int kRowCost = 8;  // a row of cells costs a warp about as much as so many points of a plain scan
constexpr int kSpacingThreads = 128;
constexpr long long kSpacingCells = 8;  // cells per point at most

__global__ void spacing_gather(const float* pts, long long n, const int32_t* idx, long long m, float* sub,
                               int32_t* status) {
    for (long long q = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; q < m;
         q += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int32_t i = idx[q];
        float x = NAN, y = NAN, z = NAN;
        if (i < 0 || i >= n) {
            atomicCAS(status, 0, static_cast<int>(HAV_ERR_INVALID));
        } else {
            x = pts[3ll * i];
            y = pts[3ll * i + 1];
            z = pts[3ll * i + 2];
            if (!(isfinite(x) && isfinite(y) && isfinite(z))) x = y = z = NAN;
        }
        sub[3 * q] = x;
        sub[3 * q + 1] = y;
        sub[3 * q + 2] = z;
    }
}

__device__ __forceinline__ float sq_dist(const float4& p, float x, float y, float z) {
    const float ex = __fsub_rn(p.x, x), ey = __fsub_rn(p.y, y), ez = __fsub_rn(p.z, z);
    return __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
}

__global__ void __launch_bounds__(kSpacingThreads)
    spacing_grid_query(long long m, const GroupGrid* g, const uint32_t* end, const float4* sorted, float* out_d2,
                       const GlobalHdr* gh) {
    if (ld_volatile(&gh->abort)) return;  // the build gave up (its status says so)
    const GroupGrid G = *g;
    // the cell width, rounded down and shrunk by 2^-20
    const float h = __fmul_rd(__fdiv_rd(1.0f, G.inv_h), 0.99999904632568359375f);
    const int lane = threadIdx.x & 31;
    // the points of cells [x0, x1] of the row that starts at cell `base`, side by side in sorted
    auto row = [&](int x0, int x1, long long base, uint32_t& a, uint32_t& b) {
        const long long c0 = base + (x0 > 0 ? x0 : 0), c1 = base + (x1 < G.dims[0] - 1 ? x1 : G.dims[0] - 1);
        a = (c0 > 0) ? end[c0 - 1] : 0u;
        b = end[c1];
    };
    // whether a point of cell c with `best` so far is done after shell r: every cell
    // visited, or none farther out can hold a nearer point
    auto enough = [&](const int c[3], int r, float best) {
        bool all = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) all = all && c[k] - r <= 0 && c[k] + r >= G.dims[k] - 1;
        const float bd = __fmul_rd(__fsub_rd(static_cast<float>(r), 0.01f), h);
        return all || best < __fmul_rd(__fmul_rd(bd, bd), 0.99999904632568359375f);
    };
    const long long stride = static_cast<long long>(gridDim.x) * kSpacingThreads;
    for (long long t0 = blockIdx.x * static_cast<long long>(kSpacingThreads) + threadIdx.x - lane; t0 < m;
         t0 += stride) {  // warp-uniform
        const uint32_t t = static_cast<uint32_t>(t0) + lane;
        const bool in = t < m;
        const float4 me = sorted[in ? t : 0];
        float best = INFINITY;
        int c[3] = {0, 0, 0};
        bool open = in && me.x == me.x;  // (a gathered point is NaN on every axis or on none)
        if (open) {
            const float p3[3] = {me.x, me.y, me.z};
            cell_of(p3, G, c);
            // shells 0 and 1: nine rows of three cells
            uint32_t a[9], b[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const int yc = c[1] + k % 3 - 1, zc = c[2] + k / 3 - 1;
                a[k] = b[k] = 0u;
                if (yc >= 0 && yc < G.dims[1] && zc >= 0 && zc < G.dims[2])
                    row(c[0] - 1, c[0] + 1, (static_cast<long long>(zc) * G.dims[1] + yc) * G.dims[0], a[k], b[k]);
            }
#pragma unroll
            for (int k = 0; k < 9; ++k)
#pragma unroll 4
                for (uint32_t q = a[k]; q < b[k]; ++q)
                    if (q != t) best = fminf(best, sq_dist(sorted[q], me.x, me.y, me.z));
            open = !enough(c, 1, best);
        }
        // the points left over, one after another: the warp's lanes share a shell's rows
        for (unsigned left = __ballot_sync(0xffffffffu, open); left; left &= left - 1) {
            const int l = __ffs(left) - 1;
            const uint32_t tl = static_cast<uint32_t>(t0) + l;
            const float x = __shfl_sync(0xffffffffu, me.x, l), y = __shfl_sync(0xffffffffu, me.y, l),
                        z = __shfl_sync(0xffffffffu, me.z, l);
            float bl = __shfl_sync(0xffffffffu, best, l);
            int cl[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) cl[k] = __shfl_sync(0xffffffffu, c[k], l);
            auto scan = [&](uint32_t a, uint32_t b) {
                for (uint32_t q = a; q < b; ++q)
                    if (q != tl) bl = fminf(bl, sq_dist(sorted[q], x, y, z));
            };
            for (int r0 = 1, r = 2;;) {  // shells r0 + 1 to r
                const int ylo = max(cl[1] - r, 0), yhi = min(cl[1] + r, G.dims[1] - 1);
                const int zlo = max(cl[2] - r, 0), zhi = min(cl[2] + r, G.dims[2] - 1);
                const int ny = yhi - ylo + 1, rows = ny * (zhi - zlo + 1);
                const bool whole = rows > m / kRowCost;  // the whole subset is less work
                if (whole) {
#pragma unroll 4
                    for (uint32_t q = lane; q < m; q += 32)
                        if (q != tl) bl = fminf(bl, sq_dist(sorted[q], x, y, z));
                } else {
                    for (int k = lane; k < rows; k += 32) {
                        const int zc = zlo + k / ny, yc = ylo + k % ny;
                        const long long base = (static_cast<long long>(zc) * G.dims[1] + yc) * G.dims[0];
                        uint32_t a, b;
                        if (abs(zc - cl[2]) > r0 || abs(yc - cl[1]) > r0) {
                            row(cl[0] - r, cl[0] + r, base, a, b);
                            scan(a, b);
                        } else {
                            if (cl[0] - r0 > 0) {
                                row(cl[0] - r, cl[0] - r0 - 1, base, a, b);
                                scan(a, b);
                            }
                            if (cl[0] + r0 < G.dims[0] - 1) {
                                row(cl[0] + r0 + 1, cl[0] + r, base, a, b);
                                scan(a, b);
                            }
                        }
                    }
                }
                // (squared distances are no less than 0: their bits are in their order)
                bl = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(bl)));
                if (whole || enough(cl, r, bl)) break;
                // on to the shell that the nearest so far needs, twice as far at most
                const float need = __fsqrt_rn(bl) * G.inv_h;
                r0 = r;
                r = need < static_cast<float>(2 * r) ? max(r + 1, static_cast<int>(need) + 1) : 2 * r;
            }
            if (lane == l) best = bl;
        }
        if (in) out_d2[__float_as_int(me.w)] = best;
    }
}

}  // namespace

int group_coresident_blocks(int device) {
    int sms = 0, per_sm = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return -1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, grp_build, kBuildThreads, 0) != cudaSuccess) return -1;
    if (per_sm < 1) return -1;
    return sms < kMaxBlocks ? sms : kMaxBlocks;  // one block per SM
}

// The larger of the two scratch areas for bucket counts, in words.
static long long count_area(unsigned char* ws, const Layout& lay, uint32_t** counts) {
    const long long cand = static_cast<long long>(sizeof(Cand)) * lay.cand_slots / 4;
    const long long logs = static_cast<long long>((lay.dirty[kTableSets - 1] - lay.dirty[0]) / 4) + lay.dirty_slots;
    *counts = reinterpret_cast<uint32_t*>(ws + (logs > cand ? lay.dirty[0] : lay.cand));
    const long long words = logs > cand ? logs : cand;
    return words < kMaxCells ? words : kMaxCells;
}

int launch_ball_query(const float* points, long long n, const int32_t* centres, long long m, float radius,
                      int nsample, int32_t* out_idx, float* out_xyz, unsigned char* ws, const Layout& lay,
                      int32_t* status, int nblocks, cudaStream_t stream) {
    if (nsample < 1 || nsample > kGrpMaxSample) return -1;
    // scratch: grid parameters and scan block sums in the phase-timer area, the
    // bucket counts in the candidate area or the fresh-insert logs (side by
    // side), whichever holds more, the sorted points in the staged points
    GroupGrid* g = reinterpret_cast<GroupGrid*>(ws + lay.ptimes);
    uint32_t* block_sums = reinterpret_cast<uint32_t*>(ws + lay.ptimes + 256);
    float4* sorted = reinterpret_cast<float4*>(ws + lay.ord[0]);
    uint32_t* counts;
    const long long budget = count_area(ws, lay, &counts);
    if (n > lay.max_points) return -1;
    static_assert(256 + 4 * kMaxBlocks <= 2 * 8 * kPhaseTimes, "scan scratch fits");
    if (cudaMemsetAsync(g, 0, sizeof(GroupGrid), stream) != cudaSuccess) return -1;
    Barrier* bar = reinterpret_cast<Barrier*>(ws + lay.barrier);  // zeroed by the caller
    GlobalHdr* gh = reinterpret_cast<GlobalHdr*>(ws + lay.ghdr);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(nblocks));
    cfg.blockDim = dim3(kBuildThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, grp_build, points, static_cast<long long>(n), radius, budget, kStepsLog2, g, counts,
                           block_sums, sorted, bar, gh) != cudaSuccess)
        return -1;
    long long qb = (m + kQueryWarps - 1) / kQueryWarps;
    if (qb > kQueryBlocks * nblocks) qb = kQueryBlocks * nblocks;
    grp_query<<<static_cast<unsigned>(qb < 1 ? 1 : qb), 32 * kQueryWarps, 0, stream>>>(
        points, n, centres, m, radius, nsample, g, counts, sorted, out_idx, out_xyz, status, gh);
    return cudaGetLastError() == cudaSuccess ? 2 : -1;
}

int launch_spacing_grid(const float* points, long long n, const int32_t* idx, long long m, float* out_d2,
                        unsigned char* ws, const Layout& lay, int32_t* status, int nblocks, cudaStream_t stream) {
    if (m < 2 || m > lay.max_points) return -1;
    // scratch as the ball query's, and the gathered subset in the second staged-point array
    GroupGrid* g = reinterpret_cast<GroupGrid*>(ws + lay.ptimes);
    uint32_t* block_sums = reinterpret_cast<uint32_t*>(ws + lay.ptimes + 256);
    float4* sorted = reinterpret_cast<float4*>(ws + lay.ord[0]);
    float* sub = reinterpret_cast<float*>(ws + lay.ord[1]);
    uint32_t* counts;
    long long budget = count_area(ws, lay, &counts);
    if (budget > kSpacingCells * m) budget = kSpacingCells * m;
    if (cudaMemsetAsync(g, 0, sizeof(GroupGrid), stream) != cudaSuccess) return -1;
    long long gb = (m + 255) / 256;
    if (gb > 65536) gb = 65536;
    spacing_gather<<<static_cast<unsigned>(gb), 256, 0, stream>>>(points, n, idx, m, sub, status);
    Barrier* bar = reinterpret_cast<Barrier*>(ws + lay.barrier);  // zeroed by the caller
    GlobalHdr* gh = reinterpret_cast<GlobalHdr*>(ws + lay.ghdr);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(nblocks));
    cfg.blockDim = dim3(kBuildThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    long long qb = (m + kSpacingThreads - 1) / kSpacingThreads;
    if (qb > 65536) qb = 65536;
    // (the smallest normal radius: the cells follow the extent alone)
    if (cudaLaunchKernelEx(&cfg, grp_build, static_cast<const float*>(sub), m, 1.17549435e-38f, budget, 0, g, counts,
                           block_sums, sorted, bar, gh) != cudaSuccess)
        return -1;
    spacing_grid_query<<<static_cast<unsigned>(qb), kSpacingThreads, 0, stream>>>(m, g, counts, sorted, out_d2, gh);
    return cudaGetLastError() == cudaSuccess ? 3 : -1;
}

}  // namespace havk
