// filter16.cu -- ch_filter16: the filter of Alg. 2 with a 16-direction
// polygon in place of the octagon.
//
// Among related work (Sec. 2) the paper cites a GPU filter over a convex
// polygon of 16 extreme points, without its directions.  Here they are the
// octagon's 8 (multiples of 45 degrees) and the 8 integer directions between
// them, (+-2, +-1) and (+-1, +-2), in counter-clockwise order from W:
//   k  0 W (-1, 0)   1 (-2,-1)   2 SW (-1,-1)   3 (-1,-2)
//      4 S ( 0,-1)   5 ( 1,-2)   6 SE ( 1,-1)   7 ( 2,-1)
//      8 E ( 1, 0)   9 ( 2, 1)  10 NE ( 1, 1)  11 ( 1, 2)
//     12 N ( 0, 1)  13 (-1, 2)  14 NW (-1, 1)  15 (-2, 1)
// V_k = argmax of a_k x + b_k y over the points, lowest index on ties.  A
// point strictly inside the polygon V_0..V_15 (strictly left of every edge of
// non-zero length; a polygon of zero area discards nothing) gets label 0;
// every other point the queue 1..4 of the quadrilateral rule over W = V_0,
// S = V_4, E = V_8, N = V_12 (as ch_filter).
//
// Launches: f16_init, the extremes (one streaming read), the labels (a second
// read), f16_output.  The extremes are tiled (f16_extremes: min / max of 8
// linear forms per warp tile, the winning tile rescanned for the lowest index)
// and the labels take 4 points per lane from a bulk-copy-fed shared-memory ring,
// with the octagon's inner region as a fast path (f16_labels).  Points that
// start 8 bytes past a 16-byte boundary have their first point taken alone, the
// tiles start behind it, and the label words are put together from two lanes
// (labels.cuh).  (Per-point kernels for such input: 143 us on 1e7 uniform
// points; these take 70.)
// Everything is exact: |a x + b y| < 3 * 2^24 fits int32 and every
// orientation product (< 2^48) int64.
#include "ch_internal.cuh"
#include "host.h"
#include "labels.cuh"
#include "octagon.cuh"
#include "tma.cuh"

#include <algorithm>
#include <climits>

namespace ch {
namespace {

constexpr int kF16Threads = 256;
constexpr int kF16Undecided = 4;
constexpr size_t kF16StreamSmemBytes = (size_t)(kF16Threads / 32) * kStages * kWarpTileF4 * sizeof(float4);   // the warps' rings
// Up to here the extremes pass leaves the points in L2 for the label pass (96 MB;
// 20 M points took 98 us a call evicted first, the two reads from HBM).
constexpr long long kF16Keep = 12ll << 20;
constexpr long long kF16PointsMax = 3ll << 20;   // a point per thread up to here (f16_extremes_points)
constexpr int kF16Bias = 1 << 26;   // makes every key positive below 2^27

struct F16Ctl {
    unsigned long long packed[16];  // (key + kF16Bias) << 32 | (0xFFFFFFFF - index): maxima
    int status;
    unsigned counts[4];
    // per direction (tile best, ~tile code)
    unsigned long long tile_packed[16];
    unsigned done;                  // last-arriver counter
    int ready;                      // the last block filled the fields below
    int vx[16], vy[16];             // the 16-gon's vertices
    Octagon oct;                    // octagon of the even directions, with its inner region
};
static_assert(kF16Threads == 256, "eight warps find the 16 directions' points");
static_assert(sizeof(F16Ctl) <= 4 * 4 * (size_t)kChainTile, "F16Ctl lives in the chain-tile scratch");

// a_k x + b_k y for direction k (a compile-time constant after unrolling)
__device__ __forceinline__ int key16(int k, int X, int Y) {
    switch (k) {
        case 0: return -X;
        case 1: return -2 * X - Y;
        case 2: return -X - Y;
        case 3: return -X - 2 * Y;
        case 4: return -Y;
        case 5: return X - 2 * Y;
        case 6: return X - Y;
        case 7: return 2 * X - Y;
        case 8: return X;
        case 9: return 2 * X + Y;
        case 10: return X + Y;
        case 11: return X + 2 * Y;
        case 12: return Y;
        case 13: return -X + 2 * Y;
        case 14: return -X + Y;
        default: return -2 * X + Y;
    }
}

__device__ __forceinline__ long long orient64(int ax, int ay, int bx, int by, int px, int py) {
    return (long long)(bx - ax) * (py - ay) - (long long)(by - ay) * (px - ax);
}

__device__ __forceinline__ unsigned long long max_u64(unsigned long long a, unsigned long long b) {
    return a > b ? a : b;
}

// ctl: the stream workspace's control block, whose status and abort flag
// the bounded waits of the streamed label pass use.
__global__ void f16_init(F16Ctl* c, Ctl* ctl) {
    const int t = threadIdx.x;
    if (t < 16) { c->packed[t] = 0ull; c->tile_packed[t] = 0ull; }
    if (t < 4) c->counts[t] = 0u;
    if (t == 0) { c->status = CH_OK; c->done = 0u; c->ready = 0; ctl->status = CH_OK; ctl->abort = 0; }
}

// ---------------------------------------------------------------------------
// Tiled extremes.  The 16 directions are the minima
// and maxima of 8 linear forms, biased to be non-negative below 2^26:
//   f0 = x, f1 = y, f2 = x + y, f3 = x - y + 2^24, f4 = 2x + y,
//   f5 = 2x - y + 2^24, f6 = x + 2y, f7 = x - 2y + 2^25.
// Direction k = (form, is_max): 0 W (f0, min), 1 (f4, min), 2 SW (f2, min),
// 3 (f6, min), 4 S (f1, min), 5 (f7, max), 6 SE (f3, max), 7 (f5, max),
// 8 E (f0, max), 9 (f4, max), 10 NE (f2, max), 11 (f6, max), 12 N (f1, max),
// 13 (f7, min), 14 NW (f3, min), 15 (f5, min).  Each lane keeps, per
// direction, its best tile value and the first warp tile reaching it (tiles
// rise within a lane); three-input float min / max on the bit patterns of
// the non-negative keys (which order like the integers) cut the per-point
// work.  The last block rescans each direction's winning tile for the lowest
// index, then builds what the label pass needs.
__device__ __forceinline__ int f16_form_of(int k) {
    constexpr int kForm[16] = {0, 4, 2, 6, 1, 7, 3, 5, 0, 4, 2, 6, 1, 7, 3, 5};
    return kForm[k];
}
__device__ __forceinline__ bool f16_is_max(int k) { return k >= 5 && k <= 12; }

__device__ __forceinline__ void f16_forms(int X, int Y, int (&f)[8]) {
    const int s = X + Y, d = X - Y + (1 << 24);
    f[0] = X; f[1] = Y; f[2] = s; f[3] = d;
    f[4] = X + s; f[5] = X + d; f[6] = s + Y; f[7] = d - Y + (1 << 24);
}

__device__ __forceinline__ int f16_max3(int a, int b, int c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(__int_as_float(a)), "f"(__int_as_float(b)), "f"(__int_as_float(c)));
    return __float_as_int(r);
}
__device__ __forceinline__ int f16_min3(int a, int b, int c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(__int_as_float(a)), "f"(__int_as_float(b)), "f"(__int_as_float(c)));
    return __float_as_int(r);
}

// One lane's 16 points of a warp tile (8 float4): per form the minimum and
// maximum; validity folded into *bad.
__device__ __forceinline__ void f16_tile_minmax(const float4* tile, int (&mn)[8], int (&mx)[8], bool& bad) {
#pragma unroll
    for (int j = 0; j < kLoadsPerLane; ++j) {
        const float4 v = tile[j * 32 + (threadIdx.x & 31)];
        const int X0 = __float2int_rn(v.x), Y0 = __float2int_rn(v.y);
        const int X1 = __float2int_rn(v.z), Y1 = __float2int_rn(v.w);
        bad |= (__int2float_rn(X0) != v.x) | (__int2float_rn(Y0) != v.y) |
               (__int2float_rn(X1) != v.z) | (__int2float_rn(Y1) != v.w) |
               ((((unsigned)X0 | (unsigned)Y0 | (unsigned)X1 | (unsigned)Y1) >> kCoordBits) != 0u);
        int a[8], b[8];
        f16_forms(X0 & (kCoordLimit - 1), Y0 & (kCoordLimit - 1), a);   // masked: keys stay in range on bad data
        f16_forms(X1 & (kCoordLimit - 1), Y1 & (kCoordLimit - 1), b);
#pragma unroll
        for (int f = 0; f < 8; ++f) {
            if (j == 0) {
                mn[f] = min(a[f], b[f]);
                mx[f] = max(a[f], b[f]);
            } else {
                mn[f] = f16_min3(mn[f], a[f], b[f]);
                mx[f] = f16_max3(mx[f], a[f], b[f]);
            }
        }
    }
}

__global__ void __launch_bounds__(kF16Threads, 2) f16_extremes(const float* __restrict__ pts, long long n, int head,
                                                               long long ntiles, int keep, F16Ctl* c, Ctl* ctl) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ unsigned long long s_bar[kF16Threads / 32][kStages];
    __shared__ unsigned long long s_m[kF16Threads / 32][16];
    __shared__ int s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long gwarp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    int best[16];
    unsigned code[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        best[k] = f16_is_max(k) ? -1 : INT_MAX;
        code[k] = 0u;
    }
    bool bad = false;
    const float2* p2 = reinterpret_cast<const float2*>(pts);
    const float4* p4 = reinterpret_cast<const float4*>(p2 + head);
    // single points in warp 0 of block 0: the unaligned head as tile code 0 and
    // the ragged tail (fewer than 512 points) as ntiles + 1
    auto scalar_range = [&](long long lo, long long hi, unsigned at) {
        for (long long i = lo + lane; i < hi; i += 32) {
            const float2 p = p2[i];
            const int X = __float2int_rn(p.x), Y = __float2int_rn(p.y);
            bad |= (__int2float_rn(X) != p.x) | (__int2float_rn(Y) != p.y) |
                   ((((unsigned)X | (unsigned)Y) >> kCoordBits) != 0u);
            int f[8];
            f16_forms(X & (kCoordLimit - 1), Y & (kCoordLimit - 1), f);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int tv = f[f16_form_of(k)];
                const bool better = f16_is_max(k) ? tv > best[k] : tv < best[k];
                best[k] = better ? tv : best[k];
                code[k] = better ? at : code[k];
            }
        }
    };
    if (gwarp == 0) scalar_range(0, head, 0u);
    WarpStream ws{reinterpret_cast<float4*>(dsm) + warp * kStages * kWarpTileF4, s_bar[warp], p4, gwarp, nwarps,
                  ntiles, lane, keep != 0};
    ws.start();
    for (long long j = 0;; ++j) {
        const long long t = gwarp + j * nwarps;
        if (t >= ntiles) break;
        const float4* cur = ws.acquire(j, ctl);
        if (!cur) {   // a copy never completed: the workspace status is CH_ETIMEOUT
            ws.drain(j);
            break;
        }
        int mn[8], mx[8];
        f16_tile_minmax(cur, mn, mx, bad);
        ws.release(j);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int tv = f16_is_max(k) ? mx[f16_form_of(k)] : mn[f16_form_of(k)];
            const bool better = f16_is_max(k) ? tv > best[k] : tv < best[k];
            best[k] = better ? tv : best[k];
            code[k] = better ? (unsigned)(t + 1) : code[k];
        }
    }
    if (gwarp == 0) scalar_range(head + ntiles * kWarpTilePts, n, (unsigned)(ntiles + 1));
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        // packed so that the maximum wins: the best value, then the lowest tile
        const bool any = f16_is_max(k) ? best[k] >= 0 : best[k] != INT_MAX;
        const unsigned hk = f16_is_max(k) ? (unsigned)best[k] : 0xFFFFFFFFu - (unsigned)best[k];
        unsigned long long m = any ? ((unsigned long long)hk << 32) | (0xFFFFFFFFu - code[k]) : 0ull;
#pragma unroll
        for (int o = 16; o; o >>= 1) m = max_u64(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
        if (lane == 0) s_m[warp][k] = m;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicCAS(&c->status, CH_OK, CH_ERANGE);
    if (threadIdx.x < 16) {
        unsigned long long m = 0ull;
        for (int w = 0; w < kF16Threads / 32; ++w) m = max_u64(m, s_m[w][threadIdx.x]);
        if (m) atomicMax(&c->tile_packed[threadIdx.x], m);
    }
    if (!last_block(&c->done, &s_last)) return;
    if (__syncthreads_or(*(volatile int*)&c->status != CH_OK || read_status(ctl) != CH_OK)) return;
    // lowest index of each direction's best value within its winning tile
    __shared__ unsigned long long s_best[16];
    __shared__ int s_val[16];
    __shared__ long long s_lo[16], s_hi[16];
    if (threadIdx.x < 16) {
        const int k = threadIdx.x;
        const unsigned long long pk = *(volatile unsigned long long*)&c->tile_packed[k];
        const unsigned hk = (unsigned)(pk >> 32), cd = 0xFFFFFFFFu - (unsigned)pk;
        s_val[k] = f16_is_max(k) ? (int)hk : (int)(0xFFFFFFFFu - hk);
        s_lo[k] = cd == 0u ? 0 : head + (long long)(cd - 1u) * kWarpTilePts;
        s_hi[k] = cd == 0u ? head : min(n, s_lo[k] + kWarpTilePts);
        s_best[k] = ~0ull;
    }
    __syncthreads();
    // two directions a warp, all loads of one in flight (one direction after the
    // other by the whole block was a chain of 16 loads' latencies, 15 us)
    for (int k = 2 * warp; k < 2 * warp + 2; ++k) {
        constexpr int kPer = kWarpTilePts / 32;
        float2 p[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const long long i = s_lo[k] + 32 * j + lane;
            p[j] = i < s_hi[k] ? p2[i] : make_float2(0.0f, 0.0f);
        }
        unsigned first = 0xFFFFFFFFu;
#pragma unroll
        for (int j = kPer - 1; j >= 0; --j) {
            int f[8];
            f16_forms(__float2int_rn(p[j].x), __float2int_rn(p[j].y), f);
            const int form = f16_form_of(k);
            int v = f[0];
#pragma unroll
            for (int q = 1; q < 8; ++q) v = q == form ? f[q] : v;
            if (s_lo[k] + 32 * j + lane < s_hi[k] && v == s_val[k]) first = (unsigned)(32 * j + lane);
        }
        first = __reduce_min_sync(0xFFFFFFFFu, first);
        if (lane == 0 && first != 0xFFFFFFFFu) s_best[k] = (unsigned long long)(s_lo[k] + first);
    }
    __syncthreads();
    if (threadIdx.x < 16) {
        const int k = threadIdx.x;
        const long long i = (long long)s_best[k];
        const float2 p = p2[i < n ? i : 0];
        const int key = key16(k, __float2int_rn(p.x), __float2int_rn(p.y));
        c->packed[k] = ((unsigned long long)(unsigned)(key + kF16Bias) << 32) | (0xFFFFFFFFu - (unsigned)i);
        c->vx[k] = __float2int_rn(p.x);
        c->vy[k] = __float2int_rn(p.y);
    }
    __syncthreads();
    // what the label pass needs beside the vertices: the octagon of the even
    // directions with its inner region (inside the 16-gon)
    __shared__ int s_vx[8], s_vy[8], s_id[8];
    __shared__ Octagon s_o;
    if (threadIdx.x < 8) {
        s_vx[threadIdx.x] = c->vx[2 * threadIdx.x];
        s_vy[threadIdx.x] = c->vy[2 * threadIdx.x];
        s_id[threadIdx.x] = (int)(0xFFFFFFFFu - (unsigned)(c->packed[2 * threadIdx.x] & 0xFFFFFFFFull));
    }
    __syncthreads();
    setup_octagon_block(s_o, s_vx, s_vy, s_id, true);
    copy_octagon(&c->oct, &s_o);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        c->ready = 1;
    }
}

// The label pass, fed by bulk copies as ch_filter's: each warp streams its warp
// tiles through a double-buffered shared-memory ring and labels 4 consecutive
// points per lane and round.  Points strictly inside the octagon's inner region
// are settled inline (that octagon lies inside the 16-gon), the others by the
// exact 16-edge test; the head and the ragged tail are labelled point by point
// by the first warp.
// Edge a -> b as a float function e(p) = A x + B y + C, positive left of the edge,
// its coefficients divided by the length |dx| + |dy|.  The factor 1 / length is off
// by 2 parts in 2^24, A and B (|A| + |B| = 1) by 3 and C (below 2^24) by 4, so by
// less than 3 and 4 in e; the two multiply-adds stay below 2^25 and round by 2 at
// most: e is off by less than kF16Tol, whatever the edge's length.  (With the
// octagon's one bound for all lengths a short edge left every point undecided: 20 M
// points of a triangle took 220 us, 157 now.)  A zero-length edge is a huge constant.
constexpr float kF16Tol = 16.0f;
__device__ __forceinline__ float4 f16_edge(int ax, int ay, int bx, int by) {
    const long long dx = bx - ax, dy = by - ay;
    const long long len = (dx < 0 ? -dx : dx) + (dy < 0 ? -dy : dy);
    if (len == 0) return make_float4(0.0f, 0.0f, kHugePositive, 0.0f);
    const float inv = 1.0f / __ll2float_rn(len);
    return make_float4((float)-dy * inv, (float)dx * inv, __ll2float_rn(dy * ax - dx * ay) * inv, 0.0f);
}
__device__ __forceinline__ float f16_value(const float4& e, float x, float y) { return fmaf(e.x, x, fmaf(e.y, y, e.z)); }

// The label from the edge functions in float: inside when surely left of every
// edge, else, when surely right of one (or the polygon has no area), the first
// quadrilateral edge it is surely right of while surely left of those before;
// kF16Undecided where the error bound leaves that open.  The exact test of 16
// int64 orientations decided every point outside the inner region before: 90 us a
// call on 2.2 M ring points, 52 now.
__device__ __forceinline__ int f16_label_float(float x, float y, const float4* e, bool none) {
    float m = kHugePositive;
#pragma unroll
    for (int k = 0; k < 16; ++k) m = fminf(m, f16_value(e[k], x, y));
    if (!none && m > kF16Tol) return -1;
    if (!none && m >= -kF16Tol) return kF16Undecided;
    int r = kF16Undecided;   // right of no edge: near
#pragma unroll
    for (int k = 3; k >= 0; --k) {
        const float v = f16_value(e[16 + k], x, y);
        r = v < -kF16Tol ? k : v <= kF16Tol ? (int)kF16Undecided : r;
    }
    return r;
}

// The polygon's and the quadrilateral's edges, for a block.
struct F16Poly {
    float4 e[20];            // the 16 edges' functions, then the quadrilateral's
    float2 v[16];            // the vertices,
    int vx[16], vy[16];
    int lab[16];             // and their labels: on the polygon, so outside
    int none;                // zero area: nothing is inside
    // The rest from vx and vy, by the first warp; a barrier before and after.
    __device__ __forceinline__ void set(int t) {
        if (t < 20) {
            const int a = t < 16 ? t : 4 * (t - 16), b = (t < 16 ? t + 1 : a + 4) & 15;
            e[t] = f16_edge(vx[a], vy[a], vx[b], vy[b]);
        }
        if (t < 16) {
            v[t] = make_float2((float)vx[t], (float)vy[t]);
            int r = -1;
            for (int q = 3; q >= 0; --q) {   // W->S, S->E, E->N, N->W
                const int a = 4 * q, b = (4 * q + 4) & 15;
                if (orient64(vx[a], vy[a], vx[b], vy[b], vx[t], vy[t]) < 0) r = q;
            }
            lab[t] = r;
        }
        if (t < 32) {
            const int k = t & 15, j = (k + 1) & 15;
            long long a2 = (long long)vx[k] * vy[j] - (long long)vx[j] * vy[k];
#pragma unroll
            for (int o = 8; o; o >>= 1) a2 += __shfl_xor_sync(0xFFFFFFFFu, a2, o);
            if (t == 0) none = a2 == 0 ? 1 : 0;
        }
    }
};

// The same where the bound leaves edges open: copies of a vertex have its label,
// the others take int64 orientations of those edges.  Out of line: most points are
// settled before, and the streaming loop stays small.  With all orientations exact,
// 5 M points with 60 % copies of a vertex took 140 us, 92 now.
static __device__ __noinline__ int f16_label_near(float x, float y, const F16Poly& p) {
    int at = -1;
#pragma unroll
    for (int k = 0; k < 16; ++k) at = x == p.v[k].x && y == p.v[k].y ? k : at;
    if (at >= 0) return p.lab[at];
    const int X = __float2int_rn(x), Y = __float2int_rn(y);
    unsigned open = 0u;   // not surely left of the edge
    bool inside = !p.none;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const float v = f16_value(p.e[k], x, y);
        open |= v <= kF16Tol ? 1u << k : 0u;
        inside = inside && v >= -kF16Tol;
    }
    for (; inside && open; open &= open - 1u) {
        const int a = __ffs((int)open) - 1, b = (a + 1) & 15;
        inside = orient64(p.vx[a], p.vy[a], p.vx[b], p.vy[b], X, Y) > 0;
    }
    if (inside) return -1;
    for (int q = 0; q < 4; ++q) {   // W->S, S->E, E->N, N->W
        const float v = f16_value(p.e[16 + q], x, y);
        const int a = 4 * q, b = (4 * q + 4) & 15;
        if (v < -kF16Tol || (v <= kF16Tol && orient64(p.vx[a], p.vy[a], p.vx[b], p.vy[b], X, Y) < 0)) return q;
    }
    return -1;
}

__global__ void __launch_bounds__(kF16Threads) f16_labels(const float* __restrict__ pts, long long n, int head,
                                                          long long ntiles, F16Ctl* c, Ctl* ctl, uint8_t* labels) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ F16Poly s_p;
    __shared__ Octagon s_o;
    __shared__ unsigned s_cnt[4];
    __shared__ unsigned long long s_bar[kF16Threads / 32][kStages];
    if (*(volatile int*)&c->status != CH_OK || !c->ready) return;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t < 16) {
        s_p.vx[t] = c->vx[t];
        s_p.vy[t] = c->vy[t];
    }
    if (t < 4) s_cnt[t] = 0u;
    copy_octagon(&s_o, &c->oct);
    __syncthreads();
    s_p.set(t);
    __syncthreads();
    const bool none = s_p.none != 0;
    const long long gwarp = ((long long)blockIdx.x * blockDim.x + t) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    unsigned cnt[4] = {0u, 0u, 0u, 0u};
    auto label = [&](float x, float y) {
        const int X = __float2int_rn(x), Y = __float2int_rn(y);
        int lab = -1;
        if (!in_inner_strict(s_o, X, Y)) {
            lab = f16_label_float(x, y, s_p.e, none);
            if (lab == kF16Undecided) lab = f16_label_near(x, y, s_p);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) cnt[q] += lab == q;
        return (uint32_t)(lab + 1);
    };
    const float4* p4 = reinterpret_cast<const float4*>(pts + 2 * head);
    const unsigned off = (unsigned)((uintptr_t)(labels + head) & 3u);   // of every tile's first label
    WarpStream ws{reinterpret_cast<float4*>(dsm) + warp * kStages * kWarpTileF4, s_bar[warp], p4, gwarp, nwarps,
                  ntiles, lane};
    ws.start();
    for (long long k = 0;; ++k) {
        const long long tile = gwarp + k * nwarps;
        if (tile >= ntiles) break;
        const float4* cur = ws.acquire(k, ctl);
        if (!cur) {   // a copy never completed: the workspace status is CH_ETIMEOUT
            ws.drain(k);
            break;
        }
        uint8_t* out = labels + head + tile * kWarpTilePts;
        uint32_t before = 0u;
#pragma unroll
        for (int r = 0; r < kWarpTilePts / 128; ++r) {
            const int q = r * 32 + lane;   // 4 points: float4 2q and 2q + 1 of the tile
            const float4 a = cur[2 * q], b = cur[2 * q + 1];
            const uint32_t word = label(a.x, a.y) | label(a.z, a.w) << 8 | label(b.x, b.y) << 16 | label(b.z, b.w) << 24;
            if (labels) store_labels(out, q, off, word, before);
        }
        ws.release(k);
    }
    if (gwarp == 0) {   // the head and the ragged tail
        const long long tail = head + ntiles * kWarpTilePts;
        for (long long j = lane; j < head + n - tail; j += 32) {
            const long long i = j < head ? j : tail + j - head;
            const float2 p = reinterpret_cast<const float2*>(pts)[i];
            const uint32_t lab = label(p.x, p.y);
            if (labels) labels[i] = (uint8_t)lab;
        }
    }
#pragma unroll
    for (int qd = 0; qd < 4; ++qd) {
        unsigned v = cnt[qd];
#pragma unroll
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        if (lane == 0 && v) atomicAdd(&s_cnt[qd], v);
    }
    __syncthreads();
    if (t < 4 && s_cnt[t]) atomicAdd(&c->counts[t], s_cnt[t]);
}

// Inputs of at most kF16PointsMax points: a point per thread, per-point maxima and
// labels.  Warp tiles of 512 points leave most of the chip idle there (uniform
// points: 37 us a call by points at 1 M, 45 and 50 by tiles at 2 M, 55 and 55 at
// 3 M, 72 and 63 at 5 M; of a ring 48 and 58, 58 and 69, 78 and 83).
__global__ void __launch_bounds__(kF16Threads) f16_extremes_points(const float2* __restrict__ pts, long long n,
                                                            F16Ctl* c) {
    __shared__ unsigned long long s_m[kF16Threads / 32][16];
    int best[16];
    unsigned arg[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        best[k] = INT_MIN;
        arg[k] = 0u;
    }
    bool bad = false;
    const long long stride = (long long)gridDim.x * blockDim.x;
    // indices rise within a thread, so a strict improvement keeps the lowest
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float2 p = __ldcs(pts + i);
        const bool ok = p.x >= 0.0f && p.x < 16777216.0f && p.x == rintf(p.x) && p.y >= 0.0f && p.y < 16777216.0f &&
                        p.y == rintf(p.y);
        bad |= !ok;
        const int X = ok ? __float2int_rz(p.x) : 0, Y = ok ? __float2int_rz(p.y) : 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int v = key16(k, X, Y);
            if (v > best[k]) {
                best[k] = v;
                arg[k] = (unsigned)i;
            }
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        // keys exceed -2^26, so INT_MIN marks a thread without points
        unsigned long long m = best[k] == INT_MIN
                                   ? 0ull
                                   : ((unsigned long long)(unsigned)(best[k] + kF16Bias) << 32) | (0xFFFFFFFFu - arg[k]);
#pragma unroll
        for (int o = 16; o; o >>= 1) m = max_u64(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
        if (lane == 0) s_m[warp][k] = m;
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicCAS(&c->status, CH_OK, CH_ERANGE);
    if (threadIdx.x < 16) {
        unsigned long long m = 0ull;
        for (int w = 0; w < kF16Threads / 32; ++w) m = max_u64(m, s_m[w][threadIdx.x]);
        if (m) atomicMax(&c->packed[threadIdx.x], m);
    }
}

__global__ void __launch_bounds__(kF16Threads) f16_labels_points(const float2* __restrict__ pts, long long n, F16Ctl* c,
                                                          uint8_t* labels) {
    __shared__ F16Poly s_p;
    __shared__ unsigned s_cnt[4];
    if (*(volatile int*)&c->status != CH_OK) return;   // set before this launch: the same for every block
    const int t = threadIdx.x;
    if (t < 16) {
        const unsigned idx = 0xFFFFFFFFu - (unsigned)(c->packed[t] & 0xFFFFFFFFull);
        const float2 v = (long long)idx < n ? pts[idx] : make_float2(0.0f, 0.0f);
        s_p.vx[t] = __float2int_rz(v.x);
        s_p.vy[t] = __float2int_rz(v.y);
    }
    if (t < 4) s_cnt[t] = 0u;
    __syncthreads();
    s_p.set(t);
    __syncthreads();
    const bool none = s_p.none != 0;
    unsigned cnt[4] = {0u, 0u, 0u, 0u};
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + t; i < n; i += stride) {
        const float2 p = __ldcs(pts + i);
        int r = f16_label_float(p.x, p.y, s_p.e, none);
        if (r == kF16Undecided) r = f16_label_near(p.x, p.y, s_p);
        if (labels) labels[i] = (uint8_t)(r + 1);
        if (r >= 0) cnt[r]++;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        unsigned v = cnt[q];
#pragma unroll
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        if ((t & 31) == 0 && v) atomicAdd(&s_cnt[q], v);
    }
    __syncthreads();
    if (t < 4 && s_cnt[t]) atomicAdd(&c->counts[t], s_cnt[t]);
}

__global__ void f16_output(const F16Ctl* c, const Ctl* ctl, int32_t* out_ext16, int64_t* out_counts4) {
    const int t = threadIdx.x;
    const int st = c->status != CH_OK ? c->status : ctl->status;
    if (t < 16) out_ext16[t] = st != CH_OK ? -1 : (int32_t)(0xFFFFFFFFu - (unsigned)(c->packed[t] & 0xFFFFFFFFull));
    if (t < 4 && out_counts4) out_counts4[t] = st != CH_OK ? (int64_t)st : (int64_t)c->counts[t];
}

}  // namespace
}  // namespace ch

using namespace ch;

extern "C" int ch_filter16(const float* pts, int64_t n, int32_t* out_ext16, uint8_t* out_labels,
                           int64_t* out_counts4, void* stream) {
    int st = check_points_args(pts, n);
    if (st != CH_OK) return st;
    if (!out_ext16) return CH_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    if (n == 0) {
        if (cudaMemsetAsync(out_ext16, 0xFF, 16 * sizeof(int32_t), s) != cudaSuccess) return CH_ECUDA;
        if (out_counts4 && cudaMemsetAsync(out_counts4, 0, 4 * sizeof(int64_t), s) != cudaSuccess)
            return CH_ECUDA;
        return CH_OK;
    }
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return CH_ECUDA;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return CH_ECUDA;
    char* base = nullptr;
    Layout L;
    if ((st = get_workspace(dev, s, n, &base, &L)) != CH_OK) return st;
    F16Ctl* c = reinterpret_cast<F16Ctl*>(base + L.off_cu);
    Ctl* ctl = reinterpret_cast<Ctl*>(base + L.off_ctl);
    const int head = ((uintptr_t)pts & 15u) != 0u ? 1 : 0;
    const long long ntiles = (n - head) / kWarpTilePts;
    const long long want = std::max(1ll, (ntiles + kF16Threads / 32 - 1) / (kF16Threads / 32));
    const bool lab = out_labels || out_counts4;
    f16_init<<<1, 32, 0, s>>>(c, ctl);
    if (n <= kF16PointsMax) {
        const float2* p2 = reinterpret_cast<const float2*>(pts);
        const int grid = (int)std::min<long long>((n + kF16Threads - 1) / kF16Threads, 4ll * sms);
        {
            ProfScope p("filter16_extremes", s);
            f16_extremes_points<<<grid, kF16Threads, 0, s>>>(p2, n, c);
        }
        if (lab) {
            ProfScope p("filter16_labels", s);
            f16_labels_points<<<grid, kF16Threads, 0, s>>>(p2, n, c, out_labels);
        }
        f16_output<<<1, 32, 0, s>>>(c, ctl, out_ext16, out_counts4);
        return cudaGetLastError() == cudaSuccess ? CH_OK : CH_ECUDA;
    }
    int occ_e = 0, occ_l = 0;
    const cudaFuncAttribute smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (cudaFuncSetAttribute(f16_extremes, smem, (int)kF16StreamSmemBytes) != cudaSuccess ||
        cudaFuncSetAttribute(f16_labels, smem, (int)kF16StreamSmemBytes) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_e, f16_extremes, kF16Threads, kF16StreamSmemBytes) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_l, f16_labels, kF16Threads, kF16StreamSmemBytes) !=
            cudaSuccess)
        return CH_ECUDA;
    {
        ProfScope p("filter16_extremes", s);
        const int grid = (int)std::min<long long>(want, (long long)sms * std::max(1, occ_e));
        f16_extremes<<<grid, kF16Threads, kF16StreamSmemBytes, s>>>(pts, n, head, ntiles, lab && n <= kF16Keep, c, ctl);
    }
    if (lab) {
        ProfScope p("filter16_labels", s);
        const int grid = (int)std::min<long long>(want, (long long)sms * std::max(1, occ_l));
        f16_labels<<<grid, kF16Threads, kF16StreamSmemBytes, s>>>(pts, n, head, ntiles, c, ctl, out_labels);
    }
    f16_output<<<1, 32, 0, s>>>(c, ctl, out_ext16, out_counts4);
    return cudaGetLastError() == cudaSuccess ? CH_OK : CH_ECUDA;
}
