// filter.cu -- the filtering stage of GPU heaphull (Alg. 2, GPUfilter) on sm_103a.
//
// Kernels (in launch order):
//   init_kernel     reset the per-call control block (calls with two reads; the
//                   sample pass does it itself).
//   sample_kernel   extremes of an evenly spaced sample of warp tiles; its last
//                   block builds the sample octagon (vertices are input points).
//   main_kernel     findExtremes (Alg. 2; Sec. 3) over every point: all 8
//                   directional extremes in one pass (the paper's second
//                   kernel finds the corner points by Manhattan distance to the
//                   bounding-box corners; that distance is x+y or x-y up to a
//                   constant, so one pass suffices), with the lowest index on
//                   ties.  In fused mode (ch_hull) the same pass also drops the
//                   points in the closed sample octagon and compacts the rest
//                   ("raw" survivors): one streaming read of the input instead
//                   of two.  When the raw survivors grow past a threshold
//                   (adversarial data such as points on a circle), the pass
//                   stops filtering and the second pass does it (two-pass mode).
//                   Its last block builds the octagon of the true extremes
//                   and the records of the chain end points.
//   dense_kernel    the main pass on dense data (an earlier pass's verdict):
//                   the star polygon (star.cuh), then one streaming read that
//                   validates the coordinates and drops the points strictly
//                   inside the polygon; the extremes are among the others.
//   (post.cu)       the classification of the survivors and the hull.
//   labels_kernel   ch_filter: the label array Q of Alg. 2 (paper rule).  On
//                   large inputs the main pass has left the points that may have
//                   a label other than 0, as in fused mode: one read of the
//                   points instead of two (1e8 normal points: 183 us a call
//                   against 288; 1.7 GB of needed traffic became 0.9).
#include "ch_internal.cuh"
#include "hullcore.cuh"
#include "launch.h"
#include "extremes.cuh"
#include "octagon.cuh"
#include "setup.cuh"
#include "star.cuh"
#include "tma.cuh"

#include "labels.cuh"

#include <climits>

namespace ch {

__global__ void init_kernel(Ctl* ctl, int mode) { reset_ctl(ctl, mode); }

// ---------------------------------------------------------------------------
// Sample pass: packed (key, other coordinate) maxima per direction; the other
// coordinate recovers the point (no index needed: the sample octagon only
// filters, and its vertices are input points).
__device__ __forceinline__ unsigned long long samp_pack(int d, int X, int Y) {
    const unsigned k = (unsigned)dir_key(d, X, Y);
    const unsigned aux = (d == W || d == E) ? (unsigned)Y : (unsigned)X;
    const unsigned hk = dir_is_max(d) ? k : 0xFFFFFFFFu - k;
    return ((unsigned long long)hk << 32) | aux;
}

// Density test of the block that built the octagon o (256 threads): kDensePts
// points spread over nspread warp tiles (tile(k), k < nspread); true when the
// share of them outside o would give the main pass more raw survivors than it
// gives up at (switch_at).  The points are loaded before the octagon is built,
// so that their latency is hidden.
constexpr int kDensePts = 2048;
struct DenseProbe {
    float2 p[kDensePts / 256];
    template <class Tile>
    __device__ __forceinline__ void load(const float4* p4, long long nspread, Tile tile) {
#pragma unroll
        for (int j = 0; j < kDensePts / 256; ++j) {
            const long long k = (long long)(j * 256 + threadIdx.x) * nspread / kDensePts;
            p[j] = __ldcg(reinterpret_cast<const float2*>(p4 + tile(k) * kWarpTileF4) +
                          (37 * threadIdx.x + 64 * j) % kWarpTilePts);
        }
    }
    __device__ __forceinline__ bool dense(const Octagon& o, long long n, unsigned switch_at) const {
        __shared__ unsigned s_out;
        __shared__ float s_e[24];
        if (threadIdx.x < 8) {
            s_e[3 * threadIdx.x] = o.oct[threadIdx.x].A;
            s_e[3 * threadIdx.x + 1] = o.oct[threadIdx.x].B;
            s_e[3 * threadIdx.x + 2] = o.oct[threadIdx.x].C;
        }
        if (threadIdx.x == 0) s_out = 0u;
        __syncthreads();
        unsigned out = 0u;
#pragma unroll
        for (int j = 0; j < kDensePts / 256; ++j)
            out += in_inner(o, __float2int_rn(p[j].x), __float2int_rn(p[j].y)) || pt_in_sample(p[j].x, p[j].y, s_e)
                       ? 0u
                       : 1u;
        out = __reduce_add_sync(0xFFFFFFFFu, out);
        if ((threadIdx.x & 31) == 0 && out) atomicAdd(&s_out, out);
        __syncthreads();
        return (long long)s_out * n > (long long)kDensePts * switch_at;
    }
    // ch_filter's region, in o.in_lo / o.in_hi: o's inner region, shrunk about its
    // centre to the largest scale of a probed point, so that about one point in
    // 2000 lies outside it and the octagon of the true extremes nearly always
    // contains it (checked by the main pass: finalize_block).  With one in 100
    // outside, the main pass took 178 us instead of 159 on 1e8 points and the
    // survivors' labels 18 instead of 12.  False when too many points lie
    // outside for one pass (more than switch_at of n).
    __device__ __forceinline__ bool label_region(Octagon& o, long long n, unsigned switch_at) const {
        __shared__ int s_t, s_b[8];
        __shared__ unsigned s_far;
        if (threadIdx.x == 0) {
            s_t = 0;
            s_far = 0u;
        }
        __syncthreads();
        const int lo0[4] = {o.vx[W], o.vy[S], o.vx[SW] + o.vy[SW], o.vx[NW] - o.vy[NW] + kCoordLimit};
        const int hi0[4] = {o.vx[E], o.vy[N], o.vx[NE] + o.vy[NE], o.vx[SE] - o.vy[SE] + kCoordLimit};
        const float cx = (float)((lo0[0] + hi0[0]) / 2), cy = (float)((lo0[1] + hi0[1]) / 2);
        const float c[4] = {cx, cy, cx + cy, cx - cy + (float)kCoordLimit};
        float m = 0.0f;
#pragma unroll
        for (int j = 0; j < kDensePts / 256; ++j) {
            const float f[4] = {p[j].x, p[j].y, p[j].x + p[j].y, p[j].x - p[j].y + (float)kCoordLimit};
#pragma unroll
            for (int k = 0; k < 4; ++k)
                m = fmaxf(m, (f[k] - c[k]) / (f[k] > c[k] ? (float)hi0[k] - c[k] : (float)lo0[k] - c[k]));
        }
        const int t = __reduce_max_sync(0xFFFFFFFFu, (int)ceilf(1024.0f * fminf(m, 1.0f)));
        if ((threadIdx.x & 31) == 0) atomicMax(&s_t, t);
        __syncthreads();
        if (threadIdx.x == 0) {
            int lo[4], hi[4];
            inner_bounds(lo0, hi0, s_t, lo, hi);
            for (int k = 0; k < 4; ++k) {
                o.in_lo[k] = s_b[k] = max(lo[k], o.in_lo[k]);
                o.in_hi[k] = s_b[4 + k] = min(hi[k], o.in_hi[k]);
            }
        }
        __syncthreads();
        unsigned far = 0u;
#pragma unroll
        for (int j = 0; j < kDensePts / 256; ++j)
            far += pt_in_inner(__float2int_rn(p[j].x), __float2int_rn(p[j].y), s_b) ? 0u : 1u;
        far = __reduce_add_sync(0xFFFFFFFFu, far);
        if ((threadIdx.x & 31) == 0 && far) atomicAdd(&s_far, far);
        __syncthreads();
        return (long long)s_far * n <= (long long)kDensePts * switch_at;
    }
};

__global__ void __launch_bounds__(256) sample_kernel(const float* __restrict__ pts, long long n, int head,
                                                     long long ntiles, Ctl* ctl, unsigned switch_at, int labels) {
    __shared__ unsigned long long s_red[8][8];
    __shared__ Octagon s_o;
    __shared__ int s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long gwarp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    if (blockIdx.x == 0) reset_ctl(ctl, 0);   // for the kernels that follow, and for this one's last block
    CH_TL(ctl, 1, 0);
    unsigned long long best[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) best[d] = 0ull;
    const long long nsamp = sample_tiles(ntiles);
    const float4* p4 = reinterpret_cast<const float4*>(pts + 2 * head);
    const unsigned long long pol = l2_evict_first();
    for (long long k = gwarp; k < nsamp; k += nwarps) {
        const long long t = k * ntiles / nsamp;
        const float4* base = p4 + t * kWarpTileF4 + lane;
        float4 v[kLoadsPerLane];
#pragma unroll
        for (int j = 0; j < kLoadsPerLane; ++j) v[j] = ld_stream_f4(base + j * 32, pol);
#pragma unroll
        for (int j = 0; j < kLoadsPerLane; ++j) {
            const int X0 = __float2int_rn(v[j].x), Y0 = __float2int_rn(v[j].y);
            const int X1 = __float2int_rn(v[j].z), Y1 = __float2int_rn(v[j].w);
#pragma unroll
            for (int d = 0; d < 8; ++d) {
                const unsigned long long a = samp_pack(d, X0, Y0), b = samp_pack(d, X1, Y1);
                const unsigned long long m = a > b ? a : b;
                best[d] = m > best[d] ? m : best[d];
            }
        }
    }
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        unsigned long long p = best[d];
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const unsigned long long q = __shfl_xor_sync(0xFFFFFFFFu, p, o);
            p = q > p ? q : p;
        }
        if (lane == 0) s_red[warp][d] = p;
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        unsigned long long m = 0ull;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = s_red[w][threadIdx.x] > m ? s_red[w][threadIdx.x] : m;
        if (m) atomicMax(&ctl->samp_packed[threadIdx.x], m);
    }
    CH_TL(ctl, 1, 1);
    if (!last_block(&ctl->blocks_done[0], &s_last)) return;
    CH_TL(ctl, 2, 0);
    CH_TRACE_DECL
    CH_TRACE_MARK();
    __shared__ int s_v[2][8];
    __shared__ int s_ok;
    const bool test = ntiles >= kStarMinTiles;
    DenseProbe probe;
    if (test) probe.load(p4, nsamp, [&](long long k) { return k * ntiles / nsamp; });
    if (threadIdx.x == 0) s_ok = nsamp > 0;
    __syncthreads();
    if (threadIdx.x < 8) {
        const int d = threadIdx.x;
        const unsigned long long p = *(volatile unsigned long long*)&ctl->samp_packed[d];
        ctl->samp_packed[d] = 0ull;   // at rest again
        if (p == 0ull) atomicAnd(&s_ok, 0);
        const unsigned hk = (unsigned)(p >> 32), aux = (unsigned)p;
        const int key = dir_is_max(d) ? (int)hk : (int)(0xFFFFFFFFu - hk);
        int x, y;
        switch (d) {
            case W: case E: x = key; y = (int)aux; break;
            case S: case N: y = key; x = (int)aux; break;
            case SW: case NE: x = (int)aux; y = key - x; break;
            default: x = (int)aux; y = x - (key - kCoordLimit); break;
        }
        s_v[0][d] = x;
        s_v[1][d] = y;
    }
    __syncthreads();
    CH_TRACE_MARK();
    if (!s_ok) {   // too few points to sample: run the two-pass path
        if (threadIdx.x == 0) ctl->mode = 1;
        return;
    }
    const int ext[8] = {-1, -1, -1, -1, -1, -1, -1, -1};
    setup_octagon_block(s_o, s_v[0], s_v[1], ext, true);
    CH_TRACE_MARK();

    if (s_o.discard_none) {
        if (threadIdx.x == 0) ctl->mode = 1;
        return;
    }
    if (labels) {   // ch_filter
        if (!test || !probe.label_region(s_o, n, switch_at)) {
            if (threadIdx.x == 0) ctl->mode = 1;
            return;
        }
        copy_octagon(&ctl->oct_s, &s_o);
        return;
    }
    copy_octagon(&ctl->oct_s, &s_o);
    // Dense data (points near a circle) goes to dense_kernel
    // from the start; the main pass would find out by writing switch_at raw
    // survivors, and all points would be read again.
    const bool dense = test && !s_o.discard_none && probe.dense(s_o, n, switch_at);
    __syncthreads();
    if (threadIdx.x == 0 && dense) {
        ctl->samp_dense = 1;
        ctl->mode = 1;
    }
    CH_TRACE_MARK();
    CH_TL(ctl, 2, 1);
    CH_TRACE_PRINT("sample-last");
}

// Strictly inside the inner region of the sample octagon: the tile's key
// extremes (or one point's keys) against the bounds, strict comparisons.
// Bounds are read from shared memory (lo = in[0..3], hi = in[4..7]) to keep
// them out of the streaming loop's registers.
__device__ __forceinline__ bool tile_in_inner(const int (&tk)[8], const int* in) {
    return tk[W] > in[0] && tk[E] < in[4] && tk[S] > in[1] && tk[N] < in[5] &&
           tk[SW] > in[2] && tk[NE] < in[6] && tk[NW] > in[3] && tk[SE] < in[7];
}


// Raw survivors are staged per warp in shared memory and written out in
// batches: one global atomic per batch instead of one per warp tile (a single
// contended counter otherwise serialises at L2).
constexpr int kWarpBuf = 256;
struct RawBuf {
    unsigned long long xy[kWarpBuf];
    unsigned idx[kWarpBuf];
};

// Warp-collective; returns the global raw count after this batch.
__device__ __forceinline__ unsigned flush_raw(RawBuf& b, unsigned& cnt, Ctl* ctl, uint64_t* raw_xy,
                                              uint32_t* raw_idx) {
    const int lane = threadIdx.x & 31;
    if (cnt == 0u) return 0u;
    unsigned base = 0u;
    if (lane == 0) base = atomicAdd(&ctl->count_raw, cnt);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    __syncwarp();
    for (unsigned i = lane; i < cnt; i += 32) {
        raw_xy[base + i] = b.xy[i];
        raw_idx[base + i] = b.idx[i];
    }
    __syncwarp();
    const unsigned after = base + cnt;
    cnt = 0u;
    return after;
}

// Warp-collective compaction of a lane's kept slots into the warp's buffer.
// get(s, idx, x, y) reads slot s; slots are unrolled so get indexes registers.
// Returns the global raw count when a batch was written out, else 0.
template <int kSlots, typename Get>
__device__ __forceinline__ unsigned emit_raw(unsigned keep, Get get, RawBuf& b, unsigned& cnt, Ctl* ctl,
                                             uint64_t* raw_xy, uint32_t* raw_idx) {
    const int lane = threadIdx.x & 31;
    const unsigned c = __popc(keep);
    unsigned incl, total;
    if constexpr (kSlots == 1) {
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, keep != 0u);
        incl = __popc(bal & lanemask_lt()) + c;
        total = __popc(bal);
    } else {
        incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += t;
        }
        total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
    if (total == 0u) return 0u;
    unsigned after = 0u;
    if (cnt + total > (unsigned)kWarpBuf) after = flush_raw(b, cnt, ctl, raw_xy, raw_idx);
    const bool direct = total > (unsigned)kWarpBuf;   // a dense tile: straight to global memory
    unsigned base = cnt;
    if (direct) {
        if (lane == 31) base = atomicAdd(&ctl->count_raw, total);
        base = __shfl_sync(0xFFFFFFFFu, base, 31);
        after = base + total;
    }
    unsigned pos = base + incl - c;
#pragma unroll
    for (int s = 0; s < kSlots; ++s) {
        if ((keep >> s) & 1u) {
            long long idx;
            float x, y;
            get(s, idx, x, y);
            const unsigned long long xy =
                ((unsigned long long)(unsigned)__float2int_rn(x) << 32) | (unsigned)__float2int_rn(y);
            if (direct) { raw_xy[pos] = xy; raw_idx[pos] = (uint32_t)idx; }
            else { b.xy[pos] = xy; b.idx[pos] = (unsigned)idx; }
            ++pos;
        }
    }
    __syncwarp();
    if (!direct) cnt += total;
    return after;
}

// Finalize of the main pass (whole block, the main pass's last block):
// lowest-index tie-break, octagon of the true extremes (-> s_o and ctl->oct),
// the chain end-point records.  The inner region of the true octagon is only
// searched in two-pass mode, where it settles most points of the second pass;
// raw survivors of the fused pass lie outside the sample octagon's inner
// region, so for them it would almost never apply.
__device__ __noinline__ void finalize_block(const float* __restrict__ pts, long long n, int head, Ctl* ctl,
                                            Octagon& s_o, uint32_t* keys, uint64_t* vals, bool labels) {
    __shared__ unsigned long long s_ext[8];
    __shared__ int s_G[8];
    __shared__ long long s_lo[8], s_hi[8];
    if (threadIdx.x < 8) {
        const int d = threadIdx.x;
        const unsigned long long pk = *(volatile unsigned long long*)&ctl->ext_packed[d];
        const unsigned code = 0xFFFFFFFFu - (unsigned)(pk & 0xFFFFFFFFull);
        const unsigned hi32 = (unsigned)(pk >> 32);
        s_G[d] = dir_is_max(d) ? (int)hi32 : (int)(0xFFFFFFFFu - hi32);
        long long lo, hi;
        if (code == 0u) { lo = 0; hi = head; }
        else { lo = head + (long long)(code - 1u) * kWarpTilePts; hi = min(n, lo + kWarpTilePts); }
        s_lo[d] = lo;
        s_hi[d] = hi;
        s_ext[d] = ~0ull;
    }
    __syncthreads();
    CH_TRACE_MARK();
    // One round of independent loads for all 8 directions (a tile has at
    // most kWarpTilePts points; blockDim.x >= kWarpTilePts / 2).
    {
        float2 p[8][2];
        bool valid[8][2];
#pragma unroll
        for (int d = 0; d < 8; ++d) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const long long i = s_lo[d] + threadIdx.x + (long long)h * blockDim.x;
                valid[d][h] = i < s_hi[d];
                p[d][h] = valid[d][h] ? reinterpret_cast<const float2*>(pts)[i] : make_float2(0.f, 0.f);
            }
        }
#pragma unroll
        for (int d = 0; d < 8; ++d) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const long long i = s_lo[d] + threadIdx.x + (long long)h * blockDim.x;
                if (valid[d][h] && dir_key(d, __float2int_rn(p[d][h].x), __float2int_rn(p[d][h].y)) == s_G[d])
                    atomicMin(&s_ext[d], (unsigned long long)i);
            }
        }
    }
    __syncthreads();
    bool bad = false;
    for (int d = 0; d < 8; ++d) bad |= s_ext[d] >= (unsigned long long)n;
    if (bad) {   // cannot happen for valid input; fail safe
        if (threadIdx.x == 0) set_status(ctl, CH_ECUDA);
        return;
    }
    __shared__ int s_vx[8], s_vy[8], s_id[8];
    if (threadIdx.x < 8) {
        const long long i = (long long)s_ext[threadIdx.x];
        s_id[threadIdx.x] = (int)i;
        s_vx[threadIdx.x] = __float2int_rn(pts[2 * i]);
        s_vy[threadIdx.x] = __float2int_rn(pts[2 * i + 1]);
    }
    __syncthreads();
    CH_TRACE_MARK();
    if (labels && threadIdx.x < 64 && *(volatile int*)&ctl->mode == 0) {
        // ch_filter: the region whose points the pass has labelled 0 has to lie
        // in the octagon (each corner left of each edge); else, all points anew
        const int k = threadIdx.x >> 3, a = threadIdx.x & 7, b = (a + 1) & 7;
        long long px, py;
        inner_corner(ctl->oct_s.in_lo, ctl->oct_s.in_hi, k, px, py);
        if (orient64(s_vx[a], s_vy[a], s_vx[b], s_vy[b], px, py) < 0) atomicExch(&ctl->mode, 1);
    }
    __syncthreads();
    setup_octagon_block(s_o, s_vx, s_vy, s_id, *(volatile int*)&ctl->mode != 0);
    CH_TRACE_MARK();
    end_records(s_vx, s_vy, s_id, ctl, keys, vals);
    __syncthreads();
    copy_octagon(&ctl->oct, &s_o);
    __syncthreads();
}

constexpr size_t kMainSmemBytes = (size_t)8 * kStages * kWarpTileF4 * sizeof(float4);

// With kLabels (ch_filter): the raw survivors are the points not strictly inside
// the region of the sample pass (oct_s's inner bounds).  two_pass: leave the
// points in L2 for a second pass.
template <bool kLabels>
__global__ void __launch_bounds__(256, 2) main_kernel(const float* __restrict__ pts, long long n, int head,
                                                      long long ntiles, Ctl* ctl, uint64_t* raw_xy,
                                                      uint32_t* raw_idx, unsigned switch_at, uint32_t* keys,
                                                      uint64_t* vals, int two_pass) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ int s_inner[8];
    __shared__ float s_edge[24];
    __shared__ unsigned long long s_red[8][8];
    __shared__ int s_mode;
    __shared__ RawBuf s_buf[8];
    __shared__ unsigned long long s_bar[8][kStages];
    __shared__ unsigned char s_q[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long gwarp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    CH_TL(ctl, 3, 0);
    if (!two_pass && *(volatile int*)&ctl->samp_dense && *(volatile int*)&ctl->star_final) return;   // dense_kernel's
    if (threadIdx.x == 0) s_mode = *(volatile int*)&ctl->mode;   // one read: uniform per block
    if (threadIdx.x < 4) {
        s_inner[threadIdx.x] = ctl->oct_s.in_lo[threadIdx.x];
        s_inner[4 + threadIdx.x] = ctl->oct_s.in_hi[threadIdx.x];
    }
    if (threadIdx.x < 8) {
        s_edge[3 * threadIdx.x] = ctl->oct_s.oct[threadIdx.x].A;
        s_edge[3 * threadIdx.x + 1] = ctl->oct_s.oct[threadIdx.x].B;
        s_edge[3 * threadIdx.x + 2] = ctl->oct_s.oct[threadIdx.x].C;
    }
    __syncthreads();
    bool filt = s_mode == 0;
    RawBuf& wbuf = s_buf[warp];
    unsigned wcnt = 0u;
    Track tr;
    track_init(tr);
    // Scalar ranges: the unaligned head point first and the ragged tail last,
    // so every lane visits tile codes in increasing order.
    auto scalar_range = [&](long long lo_i, long long hi_i, unsigned code) {
        int tk[8];
        bool any = false;
        for (long long b = lo_i; b < hi_i; b += 32) {
            const long long i = b + lane;
            unsigned keep = 0u;
            float x = 0.0f, y = 0.0f;
            if (i < hi_i) {
                x = pts[2 * i]; y = pts[2 * i + 1];
                int X, Y;
                convert_pt(x, y, X, Y, tr);
                tile_keys2(tk, X, Y, X, Y, !any);
                any = true;
                if (filt && !pt_in_inner(X, Y, s_inner) && (kLabels || !pt_in_sample(x, y, s_edge))) keep = 1u;
            }
            auto get = [&](int, long long& idx, float& px, float& py) { idx = i; px = x; py = y; };
            if (filt) emit_raw<1>(keep, get, wbuf, wcnt, ctl, raw_xy, raw_idx);
        }
        if (any) track_tile(tr, tk, code);
    };
    if (gwarp == 0 && head) scalar_range(0, head, 0u);
    // Warp tiles t = gwarp + k * nwarps stream through a double-buffered
    // shared-memory ring filled by bulk asynchronous copies (TMA).
    WarpStream ws{reinterpret_cast<float4*>(dsm) + warp * kStages * kWarpTileF4, s_bar[warp],
                  reinterpret_cast<const float4*>(pts + 2 * head), gwarp, nwarps, ntiles, lane, two_pass != 0};
    ws.start();
    for (long long k = 0;; ++k) {
        const long long t = gwarp + k * nwarps;
        if (t >= ntiles) break;
        const float4* cur = ws.acquire(k, ctl);
        if (!cur) {   // a copy never completed: status is CH_ETIMEOUT
            ws.drain(k);
            break;
        }
        int tk[8];
#pragma unroll
        for (int j = 0; j < kLoadsPerLane; ++j) {
            const float4 v = cur[j * 32 + lane];
            int X0, Y0, X1, Y1;
            convert_pt(v.x, v.y, X0, Y0, tr);
            convert_pt(v.z, v.w, X1, Y1, tr);
            tile_keys2(tk, X0, Y0, X1, Y1, j == 0);
        }
        track_tile(tr, tk, (unsigned)(t + 1));
        if (filt) {
            // Points strictly inside the inner region of the sample octagon
            // are strictly inside the hull; every other point is a raw
            // survivor, classified against the true octagon once its extremes
            // are known.  The 16 points of each lane whose tile test failed
            // are spread over the warp (two lane tiles per round) and tested
            // one per lane from the ring slot, so an outlier costs the warp
            // one round instead of a 16-point slow path on one lane.
            const bool inside = tile_in_inner(tk, s_inner);
            const unsigned fail = __ballot_sync(0xFFFFFFFFu, !inside);
            if (fail) {
                if (!inside) s_q[warp][__popc(fail & lanemask_lt())] = (unsigned char)lane;
                __syncwarp();
                const unsigned slots = 16u * (unsigned)__popc(fail);
                const float2* cur2 = reinterpret_cast<const float2*>(cur);
                unsigned upto = 0u;
                for (unsigned s0 = 0; s0 < slots; s0 += 32u) {
                    const unsigned s = s0 + (unsigned)lane;
                    unsigned keep = 0u;
                    float x = 0.0f, y = 0.0f;
                    long long idx = 0;
                    if (s < slots) {
                        // slot s: lane tile of rank s / 16, float4 (s / 2) % 8, half s % 2
                        const int ln = s_q[warp][s >> 4];
                        const int f2 = 2 * ((int)((s >> 1) & 7u) * 32 + ln) + (int)(s & 1u);
                        const float2 v = cur2[f2];
                        x = v.x;
                        y = v.y;
                        keep = (pt_in_inner(__float2int_rn(x), __float2int_rn(y), s_inner) ||
                                (!kLabels && pt_in_sample(x, y, s_edge))) ? 0u : 1u;
                        idx = head + t * kWarpTilePts + f2;
                    }
                    auto get = [&](int, long long& id, float& px, float& py) { id = idx; px = x; py = y; };
                    const unsigned a = emit_raw<1>(keep, get, wbuf, wcnt, ctl, raw_xy, raw_idx);
                    upto = a > upto ? a : upto;
                }
                __syncwarp();
                if (upto > switch_at) {   // dense data: leave filtering to the second pass
                    if (lane == 0) atomicExch(&ctl->mode, 1);
                    filt = false;
                }
            }
            if ((k & 7) == 7) {
                int m = 0;
                if (lane == 0) m = *(volatile int*)&ctl->mode;
                filt = filt && __shfl_sync(0xFFFFFFFFu, m, 0) == 0;
            }
        }
        ws.release(k);
    }
    // the ragged tail, 32 points per warp from the last warp down (one warp
    // taking all of it is a chain of up to 16 dependent loads)
    const long long tail = head + ntiles * kWarpTilePts + 32 * (nwarps - 1 - gwarp);
    if (tail < n) scalar_range(tail, min(n, tail + 32), (unsigned)(ntiles + 1));
    flush_raw(wbuf, wcnt, ctl, raw_xy, raw_idx);

    const bool err = tr.bad || (tr.orv >> kCoordBits) != 0u;
    if (__any_sync(0xFFFFFFFFu, err) && lane == 0) set_status(ctl, CH_ERANGE);
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        unsigned long long p = pack_best(d, tr.best[d], tr.code[d]);
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const unsigned long long q = __shfl_xor_sync(0xFFFFFFFFu, p, o);
            p = q > p ? q : p;
        }
        if (lane == 0) s_red[warp][d] = p;
    }
    __syncthreads();
    if (threadIdx.x < 8) {
        unsigned long long m = 0ull;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = s_red[w][threadIdx.x] > m ? s_red[w][threadIdx.x] : m;
        if (m) atomicMax(&ctl->ext_packed[threadIdx.x], m);
    }
    // The block that finishes last builds the octagon of the true extremes.
    // Every bulk copy of this block has completed (or was drained), so the
    // ring's shared memory is free for it.
    CH_TL(ctl, 3, 1);
    if (!last_block(&ctl->blocks_done[1], &s_mode)) return;
    CH_TL(ctl, 4, 0);
    CH_TRACE_DECL
    CH_TRACE_MARK();
    if (__syncthreads_or(read_status(ctl) != CH_OK)) return;
    // A call without a sample pass (two_pass) finds out here whether the data
    // are dense, against the octagon of the true extremes.
    const bool test = !kLabels && two_pass && ntiles >= kStarMinTiles;
    DenseProbe probe;
    if (test)
        probe.load(reinterpret_cast<const float4*>(pts + 2 * head), kDensePts / 4,
                   [&](long long k) { return k * ntiles / (kDensePts / 4); });
    Octagon& o = *reinterpret_cast<Octagon*>(dsm);
    finalize_block(pts, n, head, ctl, o, keys, vals, kLabels);
    if (test && read_status(ctl) == CH_OK && !o.discard_none && probe.dense(o, n, switch_at)) {
        copy_octagon(&ctl->oct_s, &o);
        if (threadIdx.x == 0) {
            ctl->samp_dense = 1;
            ctl->oct_ready = 1;
        }
    }
    CH_TRACE_PRINT("finalize");
    CH_TL(ctl, 4, 1);
}

// ---------------------------------------------------------------------------
// The main pass on dense data (points near a circle, Table V), one launch of one
// block per SM with waits between its phases (claim_item, wait_phase):
//   1. the angular bins of the star polygon (star.cuh), per block in shared
//      memory: a warp tile per warp, spread over the input.  Every point
//      outside oct_s goes to its angular bin around that octagon's centre c,
//      where an atomicMax keeps the point farthest from c (its squared
//      distance, truncated, above its index), unless its key is no larger than
//      the bin's already.  (Bins shared by all blocks in L2 took 37 us: most of
//      the first points of every block met there as atomics.)
//   2. every block merges its share of the bins and re-reads their points, one
//      block makes the polygon of them (star_polygon), every block finds its
//      share of the bins' radius bounds;
//   3. one streaming read of all points.  A point closer to c than its bin's
//      radius bound is strictly inside the polygon; the others wait in a
//      per-warp queue and go 32 at a time through the exact wedge test; what
//      that leaves are the raw survivors, classified by the post pass.  A point
//      strictly inside the polygon is interior to the hull, so it reaches no
//      extreme: the 8 extremes are tracked over the raw survivors alone.  Every
//      coordinate is validated.
// Without a polygon (its checks failed) the main pass and the post pass read
// all points.  Before, the main pass's full tracking (143 us on 1e8 points)
// ran beside 1, every block of the post pass did 2 (90 us) and the post pass 3
// with integer distances (400 us).
// One warp tile: bins (in shared memory) the points outside the octagon.
__device__ __forceinline__ void star_tile_pass(const float4* __restrict__ p4, long long t, int head, const int* s_in,
                                               const float* s_edge, int cx, int cy, unsigned long long* bins,
                                               unsigned long long pol) {
    const int lane = threadIdx.x & 31;
    const float4* base = p4 + t * kWarpTileF4 + lane;
    constexpr int kHalf = kLoadsPerLane / 2;   // half a tile's loads in flight keeps the registers low
#pragma unroll 1
    for (int j0 = 0; j0 < kLoadsPerLane; j0 += kHalf) {
        float4 v[kHalf];
#pragma unroll
        for (int j = 0; j < kHalf; ++j) v[j] = ld_stream_f4(base + (j0 + j) * 32, pol);
#pragma unroll
        for (int j = 0; j < kHalf; ++j) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float x = h ? v[j].z : v[j].x, y = h ? v[j].w : v[j].y;
                const int X = __float2int_rn(x), Y = __float2int_rn(y);
                if (pt_in_inner(X, Y, s_in) || pt_in_sample(x, y, s_edge)) continue;
                const int dx = X - cx, dy = Y - cy;
                const unsigned long long d2 = (unsigned long long)((long long)dx * dx + (long long)dy * dy);
                const unsigned idx = (unsigned)(head + t * kWarpTilePts + 2 * ((j0 + j) * 32 + lane) + h);
                const unsigned long long key = ((d2 >> 17) << 32) | idx;
                unsigned long long* bin = bins + star_bin(dx, dy);
                if (key > *(volatile unsigned long long*)bin) atomicMax(bin, key);
            }
        }
    }
}

constexpr int kDenseThreads = 1024;
constexpr int kDenseF4 = kWarpTileF4 / 2;   // float4 of a warp's ring tile: 32 warps' rings fit
constexpr int kDenseQueue = 64;   // < 32 waiting + 32 added per step
constexpr int kDenseBuf = 64;     // raw survivors staged per warp
struct DenseWarp {
    unsigned long long xy[kDenseBuf];
    unsigned raw_idx[kDenseBuf];
    float2 p[kDenseQueue];
    unsigned idx[kDenseQueue];
    unsigned cnt;                 // raw survivors staged
    int best[8];                  // the warp's extreme keys so far and the
    unsigned code[8];             // first tile where each occurred
};
// Shared memory: the radius bounds, the warps' buffers, their rings of tiles;
// first of all, in the block that makes it, the polygon and star_polygon's work
// area.  The exact tests read the polygon from L2: few points take them.
constexpr size_t kDenseWarpOff = sizeof(float) * kStarBins;
constexpr size_t kDenseRingOff = (kDenseWarpOff + (kDenseThreads / 32) * sizeof(DenseWarp) + 127) / 128 * 128;
constexpr size_t kDenseWorkOff = (sizeof(StarPoly) + 15) / 16 * 16;
constexpr size_t kDenseStream = kDenseRingOff + (size_t)(kDenseThreads / 32) * kStages * kDenseF4 * sizeof(float4);
constexpr size_t kDenseBuild = kDenseWorkOff + sizeof(unsigned long long) * kStarBins;
constexpr size_t kDenseSmemBytes = kDenseStream > kDenseBuild ? kDenseStream : kDenseBuild;
static_assert(kDenseSmemBytes <= 224 * 1024 && sizeof(StarPoly) % 16 == 0, "one block's shared memory");

__device__ __forceinline__ void dense_flush(DenseWarp& w, unsigned cnt, Ctl* ctl, uint64_t* raw_xy, uint32_t* raw_idx) {
    const int lane = threadIdx.x & 31;
    if (cnt == 0u) return;
    unsigned base = 0u;
    if (lane == 0) base = atomicAdd(&ctl->count_raw, cnt);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    for (unsigned i = lane; i < cnt; i += 32) {
        raw_xy[base + i] = w.xy[i];
        raw_idx[base + i] = w.raw_idx[i];
    }
    __syncwarp();
}

// Packed pairs of floats (x, y).
__device__ __forceinline__ unsigned long long f2_pack(float x, float y) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float2 f2_unpack(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Warp-collective, out of line: the queued points [first, first + count),
// count <= 32.
__device__ __noinline__ void dense_drain(const StarPoly& P, int cx, int cy, DenseWarp& w, unsigned first,
                                         unsigned count, int head, Ctl* ctl, uint64_t* raw_xy, uint32_t* raw_idx) {
    const int lane = threadIdx.x & 31;
    const bool valid = (unsigned)lane < count;
    const float2 p = valid ? w.p[first + lane] : make_float2(0.0f, 0.0f);
    const unsigned idx = valid ? w.idx[first + lane] : 0u;
    const int X = __float2int_rn(p.x), Y = __float2int_rn(p.y);
    const bool keep = valid && !star_inside_exact(X - cx, Y - cy, star_bin(p.x - (float)cx, p.y - (float)cy), P);
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, keep);
    if (!bal) return;
    // tile code as in extremes.cuh: 0 = head, t + 1 = body tile t or the tail
    const unsigned code = idx < (unsigned)head ? 0u : (idx - (unsigned)head) / (unsigned)kWarpTilePts + 1u;
    bool better = false;
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        const int key = dir_key(d, X, Y), b = w.best[d];
        better |= dir_is_max(d) ? key > b : key < b;
        better |= key == b && code < w.code[d];
    }
    if (__any_sync(0xFFFFFFFFu, keep && better)) {
        __syncwarp();
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            const unsigned key = (unsigned)dir_key(d, X, Y);
            const unsigned m = dir_is_max(d) ? __reduce_max_sync(0xFFFFFFFFu, keep ? key : 0u)
                                             : __reduce_min_sync(0xFFFFFFFFu, keep ? key : 0xFFFFFFFFu);
            const unsigned c = __reduce_min_sync(0xFFFFFFFFu, keep && key == m ? code : 0xFFFFFFFFu);
            if (lane == 0) {
                const int b = w.best[d];
                const bool up = dir_is_max(d) ? (int)m > b : (int)m < b;
                if (up || ((int)m == b && c < w.code[d])) {
                    w.best[d] = (int)m;
                    w.code[d] = c;
                }
            }
        }
    }
    unsigned cnt = w.cnt;
    if (cnt + (unsigned)__popc(bal) > (unsigned)kDenseBuf) {
        dense_flush(w, cnt, ctl, raw_xy, raw_idx);
        cnt = 0u;
    }
    if (keep) {
        const unsigned pos = cnt + __popc(bal & lanemask_lt());
        w.xy[pos] = ((unsigned long long)(unsigned)X << 32) | (unsigned)Y;
        w.raw_idx[pos] = idx;
    }
    __syncwarp();
    if (lane == 0) w.cnt = cnt + (unsigned)__popc(bal);
    __syncwarp();
}

__global__ void __launch_bounds__(kDenseThreads, 1) dense_kernel(const float* __restrict__ pts, long long n, int head,
                                                                 long long ntiles, Ctl* ctl, unsigned long long* bins,
                                                                 StarPoly* poly, uint64_t* raw_xy, uint32_t* raw_idx,
                                                                 uint32_t* keys, uint64_t* vals) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ unsigned long long s_red[kDenseThreads / 32][8];
    __shared__ unsigned long long s_bar[kDenseThreads / 32][kStages];
    __shared__ int s_flag, s_in[8], s_K0;
    __shared__ unsigned s_scan[kDenseThreads / 32];
    __shared__ float s_edge[24];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kWarps = kDenseThreads / 32;
    if (tid == 0) s_flag = *(volatile int*)&ctl->samp_dense && read_status(ctl) == CH_OK;
    __syncthreads();
    if (!s_flag) return;
    const Octagon& os = ctl->oct_s;
    const int cx = (os.vx[W] + os.vx[E]) / 2, cy = (os.vy[S] + os.vy[N]) / 2;
    const float4* p4 = reinterpret_cast<const float4*>(pts + 2 * head);
    unsigned long long* merged = bins + (size_t)gridDim.x * kStarBins;
    unsigned item;   // of the phase at hand
    {   // 1. bins
        if (tid < 4) {
            s_in[tid] = os.in_lo[tid];
            s_in[4 + tid] = os.in_hi[tid];
        }
        if (tid < 8) {
            s_edge[3 * tid] = os.oct[tid].A;
            s_edge[3 * tid + 1] = os.oct[tid].B;
            s_edge[3 * tid + 2] = os.oct[tid].C;
        }
        unsigned long long* mine = reinterpret_cast<unsigned long long*>(dsm);
        const long long nt = min(ntiles, (long long)gridDim.x * kWarps);
        item = claim_item(ctl, kDenseBins);
        while (item < gridDim.x) {   // gridDim.x shares
            const unsigned g = item;
            for (int b = tid; b < kStarBins; b += kDenseThreads) mine[b] = 0ull;
            __syncthreads();
            const long long k = g + (long long)gridDim.x * warp;
            if (k < nt)
                star_tile_pass(p4, ((2 * k + 1) * ntiles) / (2 * nt), head, s_in, s_edge, cx, cy, mine, l2_evict_first());
            __syncthreads();
            for (int b = tid; b < kStarBins; b += kDenseThreads) bins[(size_t)g * kStarBins + b] = mine[b];
            item = finish_and_claim(ctl, kDenseBins, gridDim.x);
        }
        CH_TL(ctl, 7, 1);
        if (!wait_phase(ctl, kDenseBins, gridDim.x, kDenseMerge, &item)) return;
    }
    auto make_polygon = [&]() {
        StarPoly& M = *reinterpret_cast<StarPoly*>(dsm);
        unsigned long long* work = reinterpret_cast<unsigned long long*>(dsm + kDenseWorkOff);
        constexpr int kPer = kStarBins / kDenseThreads;
        unsigned long long v[kPer];
        int c = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            v[i] = __ldcg(merged + tid * kPer + i);
            c += v[i] != 0ull;
        }
        int o = star_scan<kDenseThreads>(c, s_scan, &s_K0);
#pragma unroll
        for (int i = 0; i < kPer; ++i)
            if (v[i]) work[o++] = v[i];
        __syncthreads();
        CH_TL(ctl, 9, 1);
        const int K0 = s_K0;
        const int K = star_polygon<kDenseThreads>(work, K0, M, ctl);
        __syncthreads();
        for (int j = tid; K && j < K + 2; j += kDenseThreads) poly->v[j] = M.v[j];
        for (int j = tid; K && j < kStarBins; j += kDenseThreads) poly->tbl[j] = M.tbl[j];
        if (tid == 0) {
            ctl->star_k = K ? K0 : 0;
            ctl->star_edges = K;
            ctl->star_cx = cx;
            ctl->star_cy = cy;
            ctl->star_final = K ? 1 : 0;
        }
        CH_TL(ctl, 8, 1);
    };
    // 2. polygon: the blocks merge the bins and re-read their points, the one that
    // finishes last makes the polygon of them, the blocks find the bins' radius bounds
    {
        // 64 consecutive bins at a time, 16 threads each over the blocks' bins
        constexpr int kSlots = 64, kGroups = kDenseThreads / kSlots;
        constexpr unsigned kItems = kStarBins / kSlots;
        unsigned long long* part = reinterpret_cast<unsigned long long*>(dsm);
        const int slot = tid % kSlots, grp = tid / kSlots;
        while (item < kItems) {
            const int b0 = (int)item * kSlots;
            unsigned long long key = 0ull;
            for (int g = grp; g < (int)gridDim.x; g += kGroups) {
                const unsigned long long x = __ldcg(bins + (size_t)g * kStarBins + b0 + slot);
                key = x > key ? x : key;
            }
            part[tid] = key;
            __syncthreads();
            if (tid < kSlots) {
#pragma unroll
                for (int g = 1; g < kGroups; ++g) key = part[g * kSlots + tid] > key ? part[g * kSlots + tid] : key;
                merged[b0 + tid] = star_vertex(key, star_point(key, pts, n), b0 + tid, cx, cy);
            }
            bool last;
            item = finish_and_claim(ctl, kDenseMerge, kItems, &last);
            if (!last) continue;
            CH_TL(ctl, 14, 1);
            make_polygon();
            finish_items(ctl, kDensePoly, 1u, 1u);
        }
    }
    if (!wait_phase(ctl, kDensePoly, 1u, kDenseRadius, &item)) return;
    const int K = *(volatile int*)&ctl->star_edges;   // the same for all from here on
    if (!K) return;
    {   // kStarWindow threads per bin, an edge of its window each
        constexpr int kSlots = kDenseThreads / kStarWindow;
        constexpr unsigned kItems = kStarBins / kSlots;
        const int k = tid % kStarWindow;
        while (item < kItems) {
            const int b = (int)item * kSlots + tid / kStarWindow;
            int first, count;
            star_window(poly->tbl, K, b, first, count);
            unsigned r = 0xFFFFFFFFu;
            if (k < count && count <= kStarWindow) {
                const int e = first + k < K ? first + k : first + k - K;
                r = star_edge_radius(poly->v[e], poly->v[e + 1]);
            }
#pragma unroll
            for (int d = kStarWindow / 2; d; d >>= 1) r = min(r, __shfl_xor_sync(0xFFFFFFFFu, r, d));
            if (k == 0) poly->thr[b] = star_threshold(count <= kStarWindow ? r : 0u);
            item = finish_and_claim(ctl, kDenseRadius, kItems);
        }
        if (!wait_phase(ctl, kDenseRadius, kItems)) return;
    }
    CH_TL(ctl, 12, 1);
    // 3. the filter
    float* thr = reinterpret_cast<float*>(dsm);
    for (int j = tid; j < kStarBins / 4; j += kDenseThreads)
        reinterpret_cast<float4*>(thr)[j] = __ldcg(reinterpret_cast<const float4*>(poly->thr) + j);
    DenseWarp& w = reinterpret_cast<DenseWarp*>(dsm + kDenseWarpOff)[warp];
    if (lane == 0) w.cnt = 0u;
    if (lane < 8) {
        w.best[lane] = dir_is_max(lane) ? INT_MIN : INT_MAX;
        w.code[lane] = 0u;
    }
    __syncthreads();
    CH_TL(ctl, 3, 0);
    const long long first = ((long long)blockIdx.x * kDenseThreads + tid) >> 5;
    const long long stride = ((long long)gridDim.x * kDenseThreads) >> 5;
    unsigned qn = 0u;   // points queued (warp-uniform)
    unsigned bad = 0u;  // bits of the differences that a valid coordinate leaves at zero
    float lowest = 0.0f, highest = 0.0f;
    const unsigned long long away = f2_pack(-16777216.0f, -16777216.0f), back = f2_pack(16777216.0f, 16777216.0f);
    const unsigned long long minus_c = f2_pack(-(float)cx, -(float)cy);
    // Checks a point and tells whether the radius bound settles it.  A
    // coordinate is an integer, or at least 2^23 in magnitude, when adding and
    // taking away 2^24 leaves it alone (an infinity or NaN does not); with the
    // range check this is convert_pt's validity without integer conversions.
    auto undecided = [&](float x, float y) __attribute__((always_inline)) {
        const unsigned long long p = f2_pack(x, y);
        const float2 r = f2_unpack(f2_add(f2_add(p, away), back));
        bad |= __float_as_uint(__fsub_rn(r.x, x)) | __float_as_uint(__fsub_rn(r.y, y));
        asm("min.f32 %0, %0, %1, %2;" : "+f"(lowest) : "f"(x), "f"(y));
        asm("max.f32 %0, %0, %1, %2;" : "+f"(highest) : "f"(x), "f"(y));
        const float2 d = f2_unpack(f2_add(p, minus_c));   // exact
        return !(star_d2(d.x, d.y) < thr[star_bin(d.x, d.y)]);
    };
    const long long nt = ntiles * (kWarpTileF4 / kDenseF4);
    WarpStreamT<kDenseF4> ws{reinterpret_cast<float4*>(dsm + kDenseRingOff) + warp * kStages * kDenseF4, s_bar[warp], p4,
                             first, stride, nt, lane};
    ws.start();
    for (long long k = 0;; ++k) {
        const long long t = first + k * stride;
        if (t >= nt) break;
        const float4* cur = ws.acquire(k, ctl);
        if (!cur) {   // a copy never completed: status is CH_ETIMEOUT
            ws.drain(k);
            break;
        }
        unsigned mask = 0u;   // the lane's undecided points: bit 2 j + half
#pragma unroll
        for (int j = 0; j < kDenseF4 / 32; ++j) {
            const float4 p = cur[j * 32 + lane];
            if (undecided(p.x, p.y)) mask |= 1u << (2 * j);
            if (undecided(p.z, p.w)) mask |= 2u << (2 * j);
        }
        // queued, a point per lane and step (few lanes have more than one or
        // two of 8); full rounds of 32 go through the exact test
        const float2* cur2 = reinterpret_cast<const float2*>(cur);
        for (unsigned bal; (bal = __ballot_sync(0xFFFFFFFFu, mask != 0u)) != 0u;) {
            if (mask) {
                const int s = __ffs((int)mask) - 1, f2 = 64 * (s >> 1) + 2 * lane + (s & 1);
                mask &= mask - 1u;
                const unsigned pos = qn + __popc(bal & lanemask_lt());
                w.p[pos] = cur2[f2];
                w.idx[pos] = (unsigned)(head + t * (2 * kDenseF4)) + (unsigned)f2;
            }
            qn += __popc(bal);
            __syncwarp();
            if (qn >= 32u) {
                qn -= 32u;
                dense_drain(*poly, cx, cy, w, qn, 32u, head, ctl, raw_xy, raw_idx);
            }
        }
        ws.release(k);
    }
    if (qn) dense_drain(*poly, cx, cy, w, 0u, qn, head, ctl, raw_xy, raw_idx);
    // the unaligned head point, and the ragged tail by 32 points per warp
    const long long tail = head + ntiles * kWarpTilePts + 32 * (stride - 1 - first);
    const long long ranges[2][2] = {{0, first == 0 ? head : 0}, {tail, min(n, tail + 32)}};
    for (int rg = 0; rg < 2; ++rg) {
        const long long i = ranges[rg][0] + lane, cnt = ranges[rg][1] - ranges[rg][0];
        if (cnt <= 0) continue;
        __syncwarp();
        if (lane < cnt) {
            w.p[lane] = reinterpret_cast<const float2*>(pts)[i];
            w.idx[lane] = (unsigned)i;
            undecided(w.p[lane].x, w.p[lane].y);   // the checks
        }
        __syncwarp();
        dense_drain(*poly, cx, cy, w, 0u, (unsigned)cnt, head, ctl, raw_xy, raw_idx);
    }
    const bool err = bad != 0u || lowest < 0.0f || highest >= (float)kCoordLimit;
    if (__any_sync(0xFFFFFFFFu, err) && lane == 0) set_status(ctl, CH_ERANGE);
    dense_flush(w, w.cnt, ctl, raw_xy, raw_idx);
    if (lane < 8) s_red[warp][lane] = pack_best(lane, w.best[lane], w.code[lane]);
    __syncthreads();
    if (tid < 8) {
        unsigned long long m = 0ull;
        for (int k = 0; k < kDenseThreads / 32; ++k) m = s_red[k][tid] > m ? s_red[k][tid] : m;
        if (m) atomicMax(&ctl->ext_packed[tid], m);
    }
    CH_TL(ctl, 3, 1);
    if (!last_block(&ctl->blocks_done[1], &s_flag)) return;
    if (__syncthreads_or(read_status(ctl) != CH_OK)) return;
    if (tid == 0) ctl->mode = 0;   // the post pass classifies the raw survivors
    __syncthreads();
    if (!*(volatile int*)&ctl->oct_ready) finalize_block(pts, n, head, ctl, *reinterpret_cast<Octagon*>(dsm), keys, vals, false);
}

// ---------------------------------------------------------------------------
// ch_filter: the label array Q of Alg. 2 and the queue sizes (paper rule).
// The label of one point: -1 inside the octagon's inner region or the octagon,
// else its queue.
__device__ __forceinline__ int label_of(float x, float y, const Octagon& o) {
    const int X = __float2int_rn(x), Y = __float2int_rn(y);
    return in_inner_strict(o, X, Y) ? -1 : classify_paper_slow(x, y, &o);
}

// After a fused main pass (mode 0): every label 0, 16 bytes a store, a share of
// the words per item.  Not beside the main pass's reads (181 us a call on 1e8
// points, 183 here, 191 by a kernel of its own): the caller's labels stay as they
// are when that pass meets a bad coordinate.  Whole block.
__device__ __forceinline__ void zero_labels(uint8_t* labels, long long n, Ctl* ctl) {
    const long long lead = min(n, (long long)((16u - ((uintptr_t)labels & 15u)) & 15u)), words = (n - lead) / 16;
    int4* w = reinterpret_cast<int4*>(labels + lead);
    for (unsigned it; (it = claim_item(ctl, kLabelZero)) < gridDim.x;) {
        const long long end = words * (it + 1) / gridDim.x;
        for (long long j = words * it / gridDim.x + threadIdx.x; j < end; j += blockDim.x) __stcs(w + j, make_int4(0, 0, 0, 0));
        if (it == 0u && threadIdx.x < 16) {   // what the words leave at each end
            if (threadIdx.x < lead) labels[threadIdx.x] = 0;
            if (threadIdx.x < n - lead - 16 * words) labels[lead + 16 * words + threadIdx.x] = 0;
        }
        finish_items(ctl, kLabelZero, 1u, gridDim.x);
    }
}

// After a fused main pass (mode 0) every label is set to 0, then the raw
// survivors' labels, one per thread.  Else all points: up to
// kPointsMax one per thread, above each warp streams its warp tiles (512 points, behind the unaligned head point)
// through a double-buffered shared-memory ring, as the main pass does, and
// labels 4 consecutive points per lane and round; the label array's words
// (aligned, whatever its address and the head) are put together from two
// lanes' labels.  The head and the ragged tail (fewer than 512 points) are
// labelled point by point by the first warp.
constexpr size_t kLabStreamSmemBytes = (size_t)8 * kStages * kWarpTileF4 * sizeof(float4);

__global__ void __launch_bounds__(256) labels_kernel(const float* __restrict__ pts, long long n, int head,
                                                     long long ntiles, Ctl* ctl, const uint64_t* raw_xy,
                                                     const uint32_t* raw_idx, uint8_t* labels) {
    extern __shared__ __align__(128) unsigned char dsm[];
    __shared__ Octagon s_o;
    __shared__ unsigned s_cnt[4];
    __shared__ unsigned long long s_bar[8][kStages];
    if (__syncthreads_or(read_status(ctl) != CH_OK)) return;   // (a wait below may set it meanwhile)
    copy_octagon(&s_o, &ctl->oct);
    if (threadIdx.x < 4) s_cnt[threadIdx.x] = 0u;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long gwarp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    unsigned c[4] = {0u, 0u, 0u, 0u};
    auto count = [&](int lab) { c[0] += lab == 0; c[1] += lab == 1; c[2] += lab == 2; c[3] += lab == 3; };
    if (ctl->mode == 0) {
        // the first survivor's loads are in flight while the zeros go out
        const long long m = ctl->count_raw;
        long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        uint64_t xy = i < m ? __ldcs(raw_xy + i) : 0ull;
        uint32_t id = i < m ? __ldcs(raw_idx + i) : 0u;
        if (labels) zero_labels(labels, n, ctl);
        bool zeroed = !labels;
        do {
            int lab = -1;
            if (i < m) lab = classify_paper_slow((float)(int)(xy >> 32), (float)(int)(unsigned)xy, &s_o);
            if (!zeroed && !wait_phase(ctl, kLabelZero, gridDim.x)) return;
            zeroed = true;
            if (labels && lab >= 0) labels[id] = (uint8_t)(lab + 1);
            count(lab);
            i += 32 * nwarps;
            xy = i < m ? __ldcs(raw_xy + i) : 0ull;
            id = i < m ? __ldcs(raw_idx + i) : 0u;
        } while (i < m);
    } else if (n <= kPointsMax) {
        for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 32 * nwarps) {
            const float2 p = reinterpret_cast<const float2*>(pts)[i];
            const int lab = label_of(p.x, p.y, s_o);
            if (labels) labels[i] = (uint8_t)(lab + 1);
            count(lab);
        }
    } else {
        const float4* p4 = reinterpret_cast<const float4*>(pts + 2 * head);
        const unsigned off = (unsigned)((uintptr_t)(labels + head) & 3u);   // of every tile's first label
        WarpStream ws{reinterpret_cast<float4*>(dsm) + warp * kStages * kWarpTileF4, s_bar[warp], p4, gwarp, nwarps,
                      ntiles, lane};
        ws.start();
        for (long long k = 0;; ++k) {
            const long long t = gwarp + k * nwarps;
            if (t >= ntiles) break;
            const float4* cur = ws.acquire(k, ctl);
            if (!cur) {   // a copy never completed: status is CH_ETIMEOUT
                ws.drain(k);
                break;
            }
            uint8_t* out = labels + head + t * kWarpTilePts;
            uint32_t before = 0u;   // lane 0: the previous round's last word
#pragma unroll
            for (int r = 0; r < kWarpTilePts / 128; ++r) {
                const int q = r * 32 + lane;   // 4 points: float4 2q and 2q + 1 of the tile
                const float4 a = cur[2 * q], b = cur[2 * q + 1];
                const float xs[4] = {a.x, a.z, b.x, b.z}, ys[4] = {a.y, a.w, b.y, b.w};
                uint32_t word = 0u;
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int lab = label_of(xs[m], ys[m], s_o);
                    word |= (uint32_t)(lab + 1) << (8 * m);
                    count(lab);
                }
                if (labels) store_labels(out, q, off, word, before);
            }
            ws.release(k);
        }
        if (gwarp == 0) {   // the head and the ragged tail
            const long long tail = head + ntiles * kWarpTilePts;
            for (long long j = lane; j < head + n - tail; j += 32) {
                const long long i = j < head ? j : tail + j - head;
                const float2 p = reinterpret_cast<const float2*>(pts)[i];
                const int lab = label_of(p.x, p.y, s_o);
                if (labels) labels[i] = (uint8_t)(lab + 1);
                count(lab);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        unsigned v = c[r];
#pragma unroll
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        if (lane == 0 && v) atomicAdd(&s_cnt[r], v);
    }
    __syncthreads();
    if (threadIdx.x < 4 && s_cnt[threadIdx.x]) atomicAdd(&ctl->counts4[threadIdx.x], s_cnt[threadIdx.x]);
}

__global__ void filter_output_kernel(const Ctl* ctl, long long n, int32_t* out_ext8, int64_t* out_counts4) {
    const int t = threadIdx.x;
    const int st = read_status(ctl);
    if (t < 8 && out_ext8) out_ext8[t] = (n == 0 || st != CH_OK) ? -1 : ctl->oct.ext[t];
    if (t < 4 && out_counts4) out_counts4[t] = (st != CH_OK) ? (int64_t)st : (int64_t)ctl->counts4[t];
}

// ---------------------------------------------------------------------------
// Host launchers
void launch_init(Ctl* ctl, int mode, cudaStream_t s) { init_kernel<<<1, 256, 0, s>>>(ctl, mode); }

void launch_sample(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, unsigned switch_at, int grid,
                   cudaStream_t s, int labels) {
    sample_kernel<<<grid, 256, 0, s>>>(pts, n, head, ntiles, ctl, switch_at, labels);
}

void launch_main(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, uint64_t* raw_xy,
                 uint32_t* raw_idx, unsigned switch_at, uint32_t* keys, uint64_t* vals, int two_pass, int grid,
                 cudaStream_t s) {
    main_kernel<false><<<grid, 256, kMainSmemBytes, s>>>(pts, n, head, ntiles, ctl, raw_xy, raw_idx, switch_at, keys,
                                                         vals, two_pass);
}

void launch_main_labels(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, uint64_t* raw_xy,
                        uint32_t* raw_idx, unsigned switch_at, uint32_t* keys, uint64_t* vals, int two_pass, int grid,
                        cudaStream_t s) {
    main_kernel<true><<<grid, 256, kMainSmemBytes, s>>>(pts, n, head, ntiles, ctl, raw_xy, raw_idx, switch_at, keys,
                                                        vals, two_pass);
}

void launch_dense(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, void* bins, void* poly,
                  uint64_t* raw_xy, uint32_t* raw_idx, uint32_t* keys, uint64_t* vals, int sms, cudaStream_t s) {
    dense_kernel<<<sms, kDenseThreads, kDenseSmemBytes, s>>>(pts, n, head, ntiles, ctl, (unsigned long long*)bins,
                                                             (StarPoly*)poly, raw_xy, raw_idx, keys, vals);
}

size_t star_bins_bytes(int sms) { return sizeof(unsigned long long) * kStarBins * ((size_t)sms + 1); }
size_t star_poly_bytes() { return sizeof(StarPoly); }

void launch_labels(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, const uint64_t* raw_xy,
                   const uint32_t* raw_idx, uint8_t* labels, int grid, cudaStream_t s) {
    labels_kernel<<<grid, 256, kLabStreamSmemBytes, s>>>(pts, n, head, ntiles, ctl, raw_xy, raw_idx, labels);
}

void launch_filter_output(const Ctl* ctl, long long n, int32_t* out_ext8, int64_t* out_counts4, cudaStream_t s) {
    filter_output_kernel<<<1, 32, 0, s>>>(ctl, n, out_ext8, out_counts4);
}

long long sample_tiles_host(long long ntiles) { return sample_tiles(ntiles); }

cudaError_t configure_filter_kernels() {
    const cudaFuncAttribute smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(main_kernel<false>, smem, (int)kMainSmemBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(main_kernel<true>, smem, (int)kMainSmemBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(dense_kernel, smem, (int)kDenseSmemBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(labels_kernel, smem, (int)kLabStreamSmemBytes);
    return e;
}

cudaError_t occupancy_filter(int* main_k, int* labels) {
    int a = 0, b = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, main_kernel<false>, 256, kMainSmemBytes);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, main_kernel<true>, 256, kMainSmemBytes);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(labels, labels_kernel, 256, kLabStreamSmemBytes);
    *main_k = a < b ? a : b;   // one grid size for both
    return e;
}

}  // namespace ch
