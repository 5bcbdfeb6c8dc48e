// post.cu -- the loop of Alg. 1/2 after findExtremes, on the survivors.
//
// post_kernel classifies, against the octagon of the true extremes (hull
// rule, findQueue by the quadrilateral rule), either the raw survivors of the
// fused main pass or, in two-pass mode, every point; kept points become sort
// records (queue | u, v | index).  The block that finishes last adds the
// records of the support-line end points and, when the records are few,
// computes the hull itself (quickhull rounds over the queues), so the
// large-survivor path that follows finds ctl->done set and exits at once.
#include "ch_internal.cuh"
#include "extremes.cuh"
#include "hullcore.cuh"
#include "launch.h"
#include "octagon.cuh"
#include "partition.cuh"
#include "records.cuh"
#include "setup.cuh"

#include <climits>

namespace ch {

constexpr int kPostThreads = 512;
static_assert(kPostThreads % 128 == 0, "mid_hull splits the block in four");
static_assert(kSmallMax + 16 <= kQueueCap, "small_kernel's queues fit a block");

// Records are staged per warp in shared memory; a full buffer goes out with
// one atomic on the record counter, and at the end the block's remainders go
// out together with one atomic (a single counter hit once per warp batch
// serialises at L2).
constexpr int kRecBuf = 256;
struct RecBuf {
    unsigned long long val[kRecBuf];
    unsigned key[kRecBuf];
};

__device__ __forceinline__ void rec_flush_warp(RecBuf& b, unsigned& cnt, Ctl* ctl, uint32_t* keys, uint64_t* vals) {
    const int lane = threadIdx.x & 31;
    unsigned base = 0u;
    if (lane == 0) base = atomicAdd(&ctl->count, cnt);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    for (unsigned i = lane; i < cnt; i += 32) {
        keys[base + i] = b.key[i];
        vals[base + i] = b.val[i];
    }
    __syncwarp();
    cnt = 0u;
}

// Warp-collective: stages one classified point per lane (r = -1 for none).
// Records per queue are counted per lane in `tally`.
__device__ __forceinline__ void post_stage(int r, int X, int Y, unsigned idx, const Octagon& o, RecBuf& b,
                                           unsigned& cnt, Ctl* ctl, uint32_t* keys, uint64_t* vals,
                                           QueueTally& tally) {
    bool keep = r >= 0;
    if (!__any_sync(0xFFFFFFFFu, keep)) return;
    if (reduce_on_line(o, keep, X, Y, idx, ctl)) keep = false;
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, keep);
    if (!bal) return;
    if (cnt + (unsigned)__popc(bal) > (unsigned)kRecBuf) rec_flush_warp(b, cnt, ctl, keys, vals);
    tally.add(keep, r);
    if (keep) {
        uint32_t u, v;
        queue_frame(r, X, Y, u, v);
        const unsigned pos = cnt + __popc(bal & lanemask_lt());
        b.key[pos] = make_key(r, u);
        b.val[pos] = make_val(v, idx);
    }
    cnt += __popc(bal);
    __syncwarp();
}

// Warp-collective: classifies one point per lane (valid = false for none) and
// stages it; folds the tally (one add per lane and call).
__device__ __forceinline__ void post_point(bool valid, float x, float y, unsigned idx, const Octagon& o, RecBuf& b,
                                           unsigned& cnt, Ctl* ctl, uint32_t* keys, uint64_t* vals,
                                           QueueTally& tally) {
    int r = -1, X = 0, Y = 0;
    if (valid) {
        X = __float2int_rn(x);
        Y = __float2int_rn(y);
        r = classify_hull(x, y, o);
    }
    post_stage(r, X, Y, idx, o, b, cnt, ctl, keys, vals, tally);
    tally.fold();
}

// Whole block: the warps' staged records go out with one atomic.
__device__ void rec_flush_block(RecBuf& b, unsigned cnt, Ctl* ctl, uint32_t* keys, uint64_t* vals) {
    __shared__ unsigned s_off[kPostThreads / 32];
    __shared__ unsigned s_base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) s_off[warp] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned tot = 0u;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            const unsigned c = s_off[w];
            s_off[w] = tot;
            tot += c;
        }
        s_base = tot ? atomicAdd(&ctl->count, tot) : 0u;
    }
    __syncthreads();
    const unsigned base = s_base + s_off[warp];
    for (unsigned i = lane; i < cnt; i += 32) {
        keys[base + i] = b.key[i];
        vals[base + i] = b.val[i];
    }
}

// The block's records per queue (lane tallies) into ctl->rec_q.
__device__ __forceinline__ void flush_queue_counts(QueueTally& tally, Ctl* ctl) {
    __shared__ unsigned s_q[4];
    if (threadIdx.x < 4) s_q[threadIdx.x] = 0u;
    __syncthreads();
    tally.fold();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const unsigned w = tally.warp_total(q);
        if ((threadIdx.x & 31) == 0 && w) atomicAdd(&s_q[q], w);
    }
    __syncthreads();
    if (threadIdx.x < 4 && s_q[threadIdx.x]) atomicAdd(&ctl->rec_q[threadIdx.x], s_q[threadIdx.x]);
}

// The block that finished last: support-line records, then the hull of few
// records (at most kMidCap: quickhull rounds, else the sort-based mid_hull), or
// the path of the large-survivor part.  On dense data (an earlier pass's verdict,
// or more than a quarter of the points kept) the records are near the hull, mostly
// vertices, and past kNearHullRec of them the rounds take longer than the queues,
// a block each: calls on 300 and 700 points of a ring 51 and 78 us by the rounds,
// 35 and 36 by the queues (with 60 % copies of a vertex 26 and 27, 26 and 49; the
// line lies between).  The sort takes what neither a block nor the tiles are for: a
// queue too large for a block among few records in all.  Every other record is
// already in keys/vals and in the per-queue counts.
constexpr unsigned kNearHullRec = 512;

__device__ void post_last_block(const float* __restrict__ pts, long long n, Ctl* ctl, const Octagon& o,
                                uint32_t* keys, uint64_t* vals, unsigned* tiles, int32_t* out_idx, int64_t* out_n,
                                char* dyn, bool dense) {
    __shared__ unsigned long long s_lep[8];
    __shared__ uint64_t s_lval[8];
    __shared__ unsigned s_lkey[8];
    __shared__ int s_lpos[8];
    __shared__ unsigned s_m, s_total;
    __shared__ int s_mv, s_path;
    const int tid = threadIdx.x;
    CH_TRACE_DECL
    CH_TRACE_MARK();
    // one round of loads: line end points and the record count
    if (tid < 8) s_lep[tid] = *(volatile unsigned long long*)&ctl->line_ep[tid];
    if (tid == 8) s_m = *(volatile unsigned*)&ctl->count;
    __syncthreads();
    if (tid < 8) s_lpos[tid] = line_record(o, tid, s_lep[tid], s_lkey[tid], s_lval[tid]) ? 1 : -1;
    __syncthreads();
    if (tid == 0) {
        unsigned m = s_m;
        for (int t = 0; t < 8; ++t)
            if (s_lpos[t] > 0) s_lpos[t] = (int)m++;
        s_total = m;
        ctl->count = m;
    }
    __syncthreads();
    const unsigned total = s_total;
    const bool near_hull = dense || 4ll * total > n;
    const bool small = total <= (near_hull ? kNearHullRec : (unsigned)kMidCap);
    if (tid < 8 && s_lpos[tid] >= 0) {
        keys[s_lpos[tid]] = s_lkey[tid];
        vals[s_lpos[tid]] = s_lval[tid];
        if (!small) atomicAdd(&ctl->rec_q[s_lkey[tid] >> kKeyBits], 1u);
    }
    if (!small) {   // the large-survivor path follows
        __syncthreads();
        if (tid == 0) {
            unsigned most = 0u;
            for (int r = 0; r < 4; ++r) most = max(most, *(volatile unsigned*)&ctl->rec_q[r]);
            const int path = most <= (unsigned)kQueueCap ? kPathQueues
                             : *(volatile int*)&ctl->star_final || total > 4u * (unsigned)kQueueCap ? kPathTiles : kPathSort;
            ctl->path = s_path = path;
            ctl->bk_state = path == kPathSort ? 2 : 1;
        }
        __syncthreads();
        if (s_path == kPathTiles)   // large_kernel counts the records of each group of u there
            for (int g = tid; g < kPtGroups; g += blockDim.x) tiles[g] = 0u;
        return;
    }
    __syncthreads();      // also makes this block's line records visible to it
    QhSmem& q = *reinterpret_cast<QhSmem*>(dyn);
    for (unsigned i = tid; i < total; i += blockDim.x) {
        const uint32_t k = __ldcg(keys + i);
        const uint64_t w = __ldcg(vals + i);
        q.ru[i] = (int)(k & kKeyMask);
        q.rv[i] = (int)(w >> 31);
        q.ri[i] = (int)(w & 0x7FFFFFFFull);
        q.rs[i] = (int)(k >> kKeyBits);
    }
    __syncthreads();
    CH_TRACE_MARK();
    const bool ok = qh_chains(q, (int)total, &s_mv);
    CH_TRACE_MARK();
    if (ok) {
        stitch_cycle(q.ru, q.rv, q.ri, s_mv, q.rs, ctl, n, out_idx, out_n);
    } else {
        __syncthreads();
        mid_hull(keys, vals, (int)total, pts, n, ctl, out_idx, out_n, dyn);
    }
    if (tid == 0) ctl->done = 1;
    CH_TRACE_MARK();
#ifdef CH_TRACE
    if (tid == 0) printf("[post] records %u raw %u mv %d ok %d\n", total, ctl->count_raw, s_mv, (int)ok);
#endif
    CH_TRACE_PRINT("post-last");
}

constexpr size_t cmax(size_t a, size_t b) { return a > b ? a : b; }

// Dynamic shared memory: the warps' record buffers while points are
// classified; the last block's hull reuses it.
constexpr size_t kPostSmemBytes =
    cmax(cmax(kMidSmemBytes, sizeof(QhSmem)), (kPostThreads / 32) * sizeof(RecBuf));

__global__ void __launch_bounds__(kPostThreads, 1) post_kernel(const float* __restrict__ pts, long long n, int head,
                                                               long long ntiles, Ctl* ctl, const uint64_t* raw_xy,
                                                               const uint32_t* raw_idx, uint32_t* keys,
                                                               uint64_t* vals, unsigned* tiles, int32_t* out_idx,
                                                               int64_t* out_n) {
    extern __shared__ __align__(16) char dyn[];
    __shared__ Octagon s_o;
    __shared__ int s_flag, s_mode, s_dense;
    __shared__ unsigned s_nraw;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    CH_TL(ctl, 5, 0);
    if (tid == 0) {
        s_flag = read_status(ctl);
        s_mode = *(volatile int*)&ctl->mode;
        s_nraw = *(volatile unsigned*)&ctl->count_raw;
        // (small inputs take two passes whatever the data)
        s_dense = *(volatile int*)&ctl->samp_dense || (s_mode == 1 && n > kTwoPassMax);
    }
    copy_octagon(&s_o, &ctl->oct);
    __syncthreads();
    if (s_flag != CH_OK) {   // data error or timeout of an earlier stage
        if (blockIdx.x == 0 && tid == 0) { *out_n = s_flag; ctl->done = 1; }
        return;
    }
    RecBuf& rb = reinterpret_cast<RecBuf*>(dyn)[warp];
    unsigned rc = 0u;
    QueueTally tally;
    if (s_mode == 1) {   // two-pass mode: every point
        // n < 2^31, so step and point numbers fit in 32 bits
        const unsigned gwarp = (blockIdx.x * blockDim.x + tid) >> 5;
        const unsigned nwarps = (gridDim.x * blockDim.x) >> 5;
        const float4* p4 = reinterpret_cast<const float4*>(pts + 2 * head);
        const unsigned long long pol = l2_evict_first();
        // one float4 (two points, classified together) per step with the
        // loads of the next kAhead steps in flight: a rolled loop keeps the
        // classification code small.  Steps run over this warp's tiles,
        // kLoadsPerLane float4 per tile.
        constexpr int kAhead = 8;
        const unsigned total = (unsigned)ntiles * kLoadsPerLane;
        const unsigned sstep = nwarps * kLoadsPerLane;
        auto next_step = [&](unsigned st) {
            return (st % kLoadsPerLane == kLoadsPerLane - 1) ? st + sstep - (kLoadsPerLane - 1) : st + 1;
        };
        unsigned s = gwarp * kLoadsPerLane, sl = s;   // sl: the step of the newest load
        float4 q[kAhead];
#pragma unroll
        for (int a = 0; a < kAhead; ++a) {
            q[a] = sl < total ? ld_stream_f4(p4 + sl * 32 + lane, pol) : make_float4(0.f, 0.f, 0.f, 0.f);
            sl = next_step(sl);
        }
#pragma unroll 1
        while (s < total) {
            const float4 v = q[0];
#pragma unroll
            for (int a = 0; a + 1 < kAhead; ++a) q[a] = q[a + 1];
            q[kAhead - 1] = sl < total ? ld_stream_f4(p4 + sl * 32 + lane, pol) : make_float4(0.f, 0.f, 0.f, 0.f);
            sl = next_step(sl);
            const unsigned i0 = (unsigned)head + (s / kLoadsPerLane) * kWarpTilePts + 64u * (s % kLoadsPerLane) +
                                2u * lane;
            const int X0 = __float2int_rn(v.x), Y0 = __float2int_rn(v.y);
            const int X1 = __float2int_rn(v.z), Y1 = __float2int_rn(v.w);
            int r0 = classify_hull_fast(v.x, v.y, X0, Y0, s_o);
            int r1 = classify_hull_fast(v.z, v.w, X1, Y1, s_o);
            if (r0 == kUndecided) r0 = classify_hull_slow(v.x, v.y, &s_o);
            if (r1 == kUndecided) r1 = classify_hull_slow(v.z, v.w, &s_o);
            post_stage(r0, X0, Y0, i0, s_o, rb, rc, ctl, keys, vals, tally);
            post_stage(r1, X1, Y1, i0 + 1u, s_o, rb, rc, ctl, keys, vals, tally);
            if (s % kLoadsPerLane == kLoadsPerLane - 1) tally.fold();   // at most 2 kLoadsPerLane adds
            s = next_step(s);
        }
        // the unaligned head point, and the ragged tail by 32 points per warp
        const long long tail = head + ntiles * kWarpTilePts + 32ll * (nwarps - 1u - gwarp);
        const long long ranges[2][2] = {{0, gwarp == 0 ? head : 0}, {tail, min(n, tail + 32)}};
        for (int rg = 0; rg < 2; ++rg) {
            if (ranges[rg][0] >= ranges[rg][1]) continue;
            const long long i = ranges[rg][0] + lane;
            const bool valid = i < ranges[rg][1];
            float x = 0.0f, y = 0.0f;
            if (valid) { x = pts[2 * i]; y = pts[2 * i + 1]; }
            post_point(valid, x, y, (unsigned)i, s_o, rb, rc, ctl, keys, vals, tally);
        }
    } else {   // fused mode: the raw survivors of the main pass
        // the next point's loads in flight while one is classified
        const unsigned nraw = s_nraw;
        const unsigned stride = gridDim.x * blockDim.x;
        unsigned i = blockIdx.x * blockDim.x + warp * 32 + lane;
        unsigned long long nxy = i < nraw ? __ldcs(raw_xy + i) : 0ull;
        unsigned nidx = i < nraw ? __ldcs(raw_idx + i) : 0u;
        for (; i - lane < nraw; i += stride) {
            const bool valid = i < nraw;
            const float x = (float)(unsigned)(nxy >> 32), y = (float)(unsigned)(nxy & 0xFFFFFFFFull);
            const unsigned idx = nidx;
            if (i + stride < nraw) {
                nxy = __ldcs(raw_xy + i + stride);
                nidx = __ldcs(raw_idx + i + stride);
            }
            post_point(valid, x, y, idx, s_o, rb, rc, ctl, keys, vals, tally);
        }
    }
    rec_flush_block(rb, rc, ctl, keys, vals);
    flush_queue_counts(tally, ctl);
    CH_TL(ctl, 5, 1);
    if (!last_block(&ctl->blocks_done[2], &s_flag)) return;
    CH_TL(ctl, 6, 0);
    post_last_block(pts, n, ctl, s_o, keys, vals, tiles, out_idx, out_n, dyn, s_dense != 0);
    CH_TL(ctl, 6, 1);
}

// ---------------------------------------------------------------------------
// Inputs of at most kSmallMax points: one block does the work of the init, main
// and post kernels (their launches and the two grids' last blocks are most of
// such a call: 39 us of device time for 1000 uniform points, 21 in one block;
// 3000: 39 and 25; 8000: 41 and 38; past that the grid is the faster).
__global__ void __launch_bounds__(kPostThreads, 1) small_kernel(const float* __restrict__ pts, int n, Ctl* ctl,
                                                                uint32_t* keys, uint64_t* vals, int32_t* out_idx,
                                                                int64_t* out_n) {
    extern __shared__ __align__(16) char dyn[];
    __shared__ Octagon s_o;
    __shared__ unsigned long long s_best[8];
    __shared__ int s_vx[8], s_vy[8], s_id[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float2* p2 = reinterpret_cast<const float2*>(pts);
    reset_ctl(ctl, 1);
    if (tid < 8) s_best[tid] = 0ull;
    __syncthreads();
    // extremes with the lowest index on ties; validity of every coordinate
    unsigned long long best[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) best[d] = 0ull;
    bool bad = false;
    for (int i = tid; i < n; i += kPostThreads) {
        const float2 p = __ldg(p2 + i);
        const int X = __float2int_rn(p.x), Y = __float2int_rn(p.y);
        bad |= (__int2float_rn(X) != p.x) | (__int2float_rn(Y) != p.y) |
               ((((unsigned)X | (unsigned)Y) >> kCoordBits) != 0u);
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            const unsigned k = (unsigned)dir_key(d, X, Y);
            const unsigned long long w =
                ((unsigned long long)(dir_is_max(d) ? k : 0xFFFFFFFFu - k) << 32) | (0xFFFFFFFFu - (unsigned)i);
            best[d] = w > best[d] ? w : best[d];
        }
    }
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        unsigned long long w = best[d];
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xFFFFFFFFu, w, o);
            w = v > w ? v : w;
        }
        if (lane == 0) atomicMax(&s_best[d], w);
    }
    if (__syncthreads_or(bad)) {
        if (tid == 0) {
            set_status(ctl, CH_ERANGE);
            *out_n = CH_ERANGE;
            ctl->done = 1;
        }
        return;
    }
    if (tid < 8) {
        const int i = (int)(0xFFFFFFFFu - (unsigned)s_best[tid]);
        s_id[tid] = i;
        s_vx[tid] = __float2int_rn(p2[i].x);
        s_vy[tid] = __float2int_rn(p2[i].y);
    }
    __syncthreads();
    setup_octagon_block(s_o, s_vx, s_vy, s_id, false);   // a point per thread and step: no inner region needed
    end_records(s_vx, s_vy, s_id, ctl, keys, vals);
    copy_octagon(&ctl->oct, &s_o);
    RecBuf& rb = reinterpret_cast<RecBuf*>(dyn)[warp];
    unsigned rc = 0u;
    QueueTally tally;
    for (int i = tid; i - lane < n; i += kPostThreads) {
        const bool valid = i < n;
        const float2 p = valid ? __ldg(p2 + i) : make_float2(0.0f, 0.0f);
        post_point(valid, p.x, p.y, (unsigned)i, s_o, rb, rc, ctl, keys, vals, tally);
    }
    __syncthreads();   // the end records are counted
    rec_flush_block(rb, rc, ctl, keys, vals);
    flush_queue_counts(tally, ctl);
    __syncthreads();
    // (at most kSmallMax + 16 records: every queue fits a block, so no tiles)
    post_last_block(pts, n, ctl, s_o, keys, vals, nullptr, out_idx, out_n, dyn, false);
}

// ---------------------------------------------------------------------------
void launch_small(const float* pts, long long n, Ctl* ctl, uint32_t* keys, uint64_t* vals, int32_t* out_idx,
                  int64_t* out_n, cudaStream_t s) {
    small_kernel<<<1, kPostThreads, kPostSmemBytes, s>>>(pts, (int)n, ctl, keys, vals, out_idx, out_n);
}

void launch_post(const float* pts, long long n, int head, long long ntiles, Ctl* ctl, const uint64_t* raw_xy,
                 const uint32_t* raw_idx, uint32_t* keys, uint64_t* vals, unsigned* tiles, int32_t* out_idx,
                 int64_t* out_n, int grid, cudaStream_t s) {
    post_kernel<<<grid, kPostThreads, kPostSmemBytes, s>>>(pts, n, head, ntiles, ctl, raw_xy, raw_idx, keys, vals, tiles,
                                                          out_idx, out_n);
}

cudaError_t configure_post_kernel() {
    const cudaError_t e =
        cudaFuncSetAttribute(small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPostSmemBytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(post_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPostSmemBytes);
}

cudaError_t occupancy_post(int* blocks) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, post_kernel, kPostThreads, kPostSmemBytes);
}

}  // namespace ch
