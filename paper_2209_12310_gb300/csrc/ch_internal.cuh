// ch_internal.cuh -- device-side data layout and helpers shared by the CUDA
// translation units of libconvhull (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include "ch.h"

namespace ch {

// ---------------------------------------------------------------------------
// Geometry of the input domain.  Coordinates are integers in [0, 2^24), so
// x + y < 2^25 and every orientation product is below 2^50 (exact in int64).
// ---------------------------------------------------------------------------
constexpr int kCoordBits = 24;
constexpr int kCoordLimit = 1 << kCoordBits;
constexpr int kKeyBits = 25;                  // bits of the per-queue sort key u
constexpr uint32_t kKeyMask = (1u << kKeyBits) - 1;
constexpr int kSortBits = 27;                 // queue (2 bits) | u (25 bits)
constexpr int kDigitBits = 9;                 // 3 LSD passes of 9 bits
constexpr int kDigits = 1 << kDigitBits;
constexpr int kSortPasses = 3;

// Streaming passes: a warp tile is 256 float4 = 512 points (8 float4 / lane).
constexpr int kLoadsPerLane = 8;
constexpr int kWarpTileF4 = 32 * kLoadsPerLane;
constexpr int kWarpTilePts = 2 * kWarpTileF4;

// Onesweep radix sort tile: 256 threads x 16 keys.
constexpr int kSortThreads = 256;
constexpr int kSortItems = 16;
constexpr int kSortTile = kSortThreads * kSortItems;

// Hull stage tile: 256 threads x 16 sorted records.
constexpr int kChainThreads = 256;
constexpr int kChainItems = 16;
constexpr int kChainTile = kChainThreads * kChainItems;
constexpr int kMergeSmemCap = 8192;           // chain points a global merge keeps on chip
// Large-survivor path of the single hull (queues.cu): records of a queue that
// one block reduces to its chain, and the ways a call can take.
constexpr int kQueueCap = 10240;
enum Path { kPathNone = 0, kPathQueues, kPathTiles, kPathSort };
// Bucketed large-survivor path of a batch (batched_large.cu): records per
// bucket on average, chain vertices a bucket may keep, bucket chains per
// chain-kernel tile.
constexpr int kBkAvg = 256;
constexpr int kBkNearHull = 64;   // records per bucket when a star polygon filtered them
constexpr int kBkChain = 32;
constexpr int kBkGroup = kChainTile / kBkChain;
// Buckets of a queue of cnt records: about kBkAvg records each, and at least
// 7 cnt^(1/3) (at most one per 8 records).  The queue chain of cnt records
// on a thin ring (the ring workload: width 64 at radius 2^23) has about
// 54 cnt^(1/3) vertices, so a bucket holds about 8 of them and its chain
// stays within kBkChain; a set whose chains still overflow takes the
// single-hull path.  kBkMinQ bounds the floor (7 cnt^(1/3) - cnt / kBkAvg
// stays below 115), for the workspace bounds.
constexpr int kBkMinQ = 256;

__host__ __device__ __forceinline__ unsigned bk_buckets_for(unsigned cnt) {
    unsigned nb = (cnt + kBkAvg - 1) / kBkAvg;
    unsigned ring = (unsigned)(7.0f * cbrtf((float)cnt)) + 1u;
    ring = ring < (unsigned)kBkMinQ ? ring : (unsigned)kBkMinQ;
    const unsigned lo = (cnt / 8u < ring) ? cnt / 8u : ring;
    nb = nb > lo ? nb : lo;
    return nb > 0u ? nb : 1u;
}
constexpr int kSampleTiles = 1024;            // warp tiles read by the sample pass (512k points)
// Star polygon of dense data (star.cuh): angular bins around a centre.
constexpr int kStarBins = 8192;
constexpr int kStarBlocks = 160;              // blocks of dense_kernel at most
constexpr long long kStarMinTiles = 128;      // inputs below this many warp tiles get no star polygon
// Inputs of at most this many points take two passes: the extremes first, without
// a sample, and the second read from L2.  Past it a sample and one pass are the
// faster (uniform points: 68 us by two passes and 71 by one at 2.0 M, 75 and 66 at
// 2.5 M, 86 and 72 at 4.2 M).
constexpr long long kTwoPassMax = 1 << 21;
constexpr long long kSmallMax = 8192;   // one block finds the records of so few points (small_kernel)
// The label passes take a point per thread up to here, above warp tiles of 512
// points (which leave most of the chip idle on small inputs).
constexpr long long kPointsMax = 1 << 21;
// ch_filter: up to kFilterTwoPassMax points two reads (the second from L2 while the
// points are 64 MB at most), above one and a sample before it, which only pays when
// nearly all points lie inside the sample's region (8.5 M uniform points 62 us by
// two reads and 67 by one, 16.7 M 84 and 80, 1e8 288 and 183; of a triangle, which
// is read twice all the same, 79 and 88, 124 and 134).
constexpr long long kFilterKeepMax = 1 << 23;
constexpr long long kFilterTwoPassMax = 1 << 24;
constexpr int kMaxLevels = 32;

// Warp tiles read by the sample pass: about 1/32 of the input, at most
// kSampleTiles, at least min(ntiles, 64).
__host__ __device__ __forceinline__ long long sample_tiles(long long ntiles) {
    long long s = ntiles / 32;
    if (s < 64) s = ntiles < 64 ? ntiles : 64;
    return s < kSampleTiles ? s : kSampleTiles;
}

// Float edge-function error bound: |e_float - e_exact| < 2^28 for every edge
// and query point of the domain (see octagon setup in filter.cu).
constexpr float kEdgeTol = 268435456.0f;      // 2^28
constexpr float kHugePositive = 1.0e30f;      // "always inside" coefficient of a skipped edge

constexpr unsigned kSpinLimit = 1u << 20;     // polls of a bounded wait (of a phase: without progress)

constexpr int kJoinRounds = 8;                // rounds that join a queue's tile chains, at most

// Phases of dense_kernel, large_kernel, sort_kernel and labels_kernel whose end their blocks
// wait for (claim_item, wait_phase).
enum Phase {
    kDenseBins = 0, kDenseMerge, kDensePoly, kDenseRadius,
    kLargeHist, kLargeCut, kLargePart, kLargeChains, kLargeJoin,
    kSortHist = kLargeJoin + kJoinRounds, kSortPass, kLabelZero = kSortPass + kSortPasses, kPhases
};

// Directions of the 8 extremes in counter-clockwise octagon order.
enum Dir { W = 0, SW, S, SE, E, NE, N, NW };

// Edge function  e(p) = A*px + B*py + C  equals orient(a, b, p) (positive when
// p is left of a->b); exact data kept for the ambiguous band |e| <= kEdgeTol.
struct Edge {
    float A, B, C;
    int ax, ay, dx, dy;  // origin and direction (dx = dy = 0: skipped edge)
};

struct Octagon {
    int vx[8], vy[8];    // vertices W, SW, S, SE, E, NE, N, NW
    int ext[8];          // their indices (-1 for a sample octagon)
    Edge oct[8];         // octagon edges V[k] -> V[k+1]
    Edge quad[4];        // W->S, S->E, E->N, N->W (queue rule)
    int in_lo[4], in_hi[4];   // inner region: x, y, x+y, x-y+2^24 bounds (empty if lo > hi)
    int discard_none;    // octagon of zero area: nothing is discarded
    int pad[3];
};

// Small-path limits: the last block of a pass finishes the hull itself when
// the survivors are few.
constexpr int kMidCap = 8192;           // sort records one block turns into the hull

// Per-call control block in device memory.
struct Ctl {
    unsigned long long ext_packed[8];   // (key, ~tile) packed maxima of pass 1
    unsigned long long samp_packed[8];  // (key, other coordinate) maxima of the sample pass
    int status;                         // CH_OK or a negative ch_status
    int abort;                          // set by a timed-out wait; all waits give up
    unsigned int count;                 // sort records (the 8 extreme records first)
    unsigned int count_raw;             // raw survivors of the fused pass
    unsigned int epoch;                 // onesweep status epoch (incremented per call)
    int mode;                           // 0: fused single pass, 1: two streaming passes
    int done;                           // the hull has been written by a small-path block
    unsigned int blocks_done[4];        // last-arriver counters (sample, main, post, a batched set's queues)
    unsigned int digit_hist[kSortPasses][kDigits];   // sort path only (sort_kernel)
    unsigned int rec_q[4];              // records per queue
    unsigned int reg_end[4];            // chain length of queue r (large_kernel, bt_queue_chain)
    unsigned int counts4[4];            // survivors per queue (ch_filter)
    unsigned long long line_ep[8];      // end points of survivors on the 4 axis support lines
    int bk_state;                       // large-survivor path: 0 unused, 1 queues / tiles / buckets, 2 full sort
    int path;                           // the single hull's large-survivor path (Path)
    unsigned int q_tile[5];             // path tiles: tiles of queue r are [q_tile[r], q_tile[r + 1])
    int samp_dense;                     // dense data (oct_s: an octagon of input points): dense_kernel's
    int oct_ready;                      // the octagon of the true extremes and the end-point records stand
    int skip;                           // batched: nothing for bt_filter (empty, failed, classified, or bt_dense's)
    int star_k;                         // the polygon's vertices, the dropped ones included
    int star_edges;                     // dense_kernel: the polygon's vertices in use (0: none)
    int star_final;                     // a polygon was built and accepted
    int star_cx, star_cy;               // its centre (vertices are stored relative to it)
    Octagon oct;                        // octagon of the true extremes
    Octagon oct_s;                      // octagon of a sample's extremes
    unsigned int claimed[kPhases];      // items of a phase that blocks have taken,
    unsigned int finished[kPhases];     // and finished
    unsigned int beat;                  // progress within long items
    unsigned int joins_done;            // large_kernel: queues whose chain stands
    unsigned int join_n[kJoinRounds + 1][4];   // large_kernel: points of each queue's tile chains,
                                        // and after each round that joins them
    unsigned int roots_done;            // sort_kernel: queue roots of the merge tree
#if defined(CH_TRACE) || defined(CH_TIMELINE)
    unsigned long long tl[24][2];       // debug builds: first start / last end per phase (%globaltimer)
#endif
};

// Optional phase tracing of single-block kernels (debug builds with
// -DCH_TRACE): thread 0 stamps %globaltimer and prints the deltas.
#ifdef CH_TRACE
__shared__ unsigned long long s_trace_t[24];
__shared__ int s_trace_n;
#define CH_TRACE_DECL if (threadIdx.x == 0) s_trace_n = 0;
#define CH_TRACE_MARK() do { if (threadIdx.x == 0 && s_trace_n >= 0 && s_trace_n < 24) { unsigned long long _t; \
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(_t)); s_trace_t[s_trace_n++] = _t; } } while (0)
#define CH_TRACE_PRINT(tag) do { if (threadIdx.x == 0) { printf("[trace %s]", tag); \
    for (int _i = 1; _i < s_trace_n; ++_i) printf(" %llu", s_trace_t[_i] - s_trace_t[_i - 1]); printf("\n"); } } while (0)
#else
#define CH_TRACE_DECL
#define CH_TRACE_MARK() do { } while (0)
#define CH_TRACE_PRINT(tag) do { } while (0)
#endif
// Debug builds (-DCH_TRACE or -DCH_TIMELINE): grid-wide phase timeline, the
// first start and the last end of each phase in ctl->tl.
#if defined(CH_TRACE) || defined(CH_TIMELINE)
#define CH_TL(ctl, slot, end) do { if (threadIdx.x == 0) { unsigned long long _t; \
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(_t)); \
    if (end) atomicMax(&(ctl)->tl[slot][1], _t); else atomicMin(&(ctl)->tl[slot][0], _t); } } while (0)
#else
#define CH_TL(ctl, slot, end) do { } while (0)
#endif

// ---------------------------------------------------------------------------
// Small helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long orient64(long long ax, long long ay, long long bx,
                                              long long by, long long px, long long py) {
    return (bx - ax) * (py - ay) - (by - ay) * (px - ax);
}

// L2 policy for data read once per call (the input points): evicted first,
// so streaming 100s of MB does not flush the workspace, the control block and
// the kernels' code out of L2.
__device__ __forceinline__ unsigned long long l2_evict_first() {
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

__device__ __forceinline__ unsigned long long l2_evict_normal() {
    unsigned long long pol;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

__device__ __forceinline__ float4 ld_stream_f4(const float4* p, unsigned long long pol) {
    float4 r;
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.f32 {%0,%1,%2,%3}, [%4], %5;"
        : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w)
        : "l"(p), "l"(pol));
    return r;
}

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Last-arriver election: returns true in exactly one block, after every other
// block of the grid has finished (and made its writes visible).
__device__ __forceinline__ bool last_block(unsigned* counter, int* s_flag) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) *s_flag = (atomicAdd(counter, 1u) == gridDim.x - 1);
    __syncthreads();
    if (!*s_flag) return false;
    __threadfence();
    if (threadIdx.x == 0) *counter = 0u;
    return true;
}

__device__ __forceinline__ void set_status(Ctl* ctl, int st) {
    atomicCAS(&ctl->status, CH_OK, st);
}

// One poll of a bounded wait on a flag another block sets: false to poll
// again (after a short sleep); true to give up, after kSpinLimit polls or
// when another wait already gave up (then status CH_ETIMEOUT and the abort
// flag are set, and the caller leaves the wait).
__device__ __forceinline__ bool spin_give_up(unsigned& spins, Ctl* ctl) {
    if (++spins > kSpinLimit || ((spins & 63u) == 0u && *(volatile int*)&ctl->abort)) {
        set_status(ctl, CH_ETIMEOUT);
        atomicExch(&ctl->abort, 1);
        return true;
    }
    __nanosleep(64);
    return false;
}

// Work of a phase that the whole grid shares.  Running blocks claim its items
// one at a time until none is left and then wait for the phase's end, so a wait
// is only ever for items that running blocks hold: it ends whatever share of the
// grid is resident.  (Cooperative launches with grid barriers instead started
// only once every SM was free, so that one block of another stream's kernel
// held up the whole call, and a kernel that waited for the call's result never
// saw it.)  All four: whole block.
__device__ __forceinline__ unsigned claim_item(Ctl* ctl, int phase) {
    __shared__ unsigned s_item;
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(&ctl->claimed[phase], 1u);
    __syncthreads();
    return s_item;
}

// The block's writes for n items stand; true in the one block that finishes the
// phase's last (it sees the writes of all).
__device__ __forceinline__ bool finish_items(Ctl* ctl, int phase, unsigned n, unsigned items) {
    __shared__ int s_end;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_end = atomicAdd(&ctl->finished[phase], n) + n == items;
        __threadfence();
    }
    __syncthreads();
    return s_end != 0;
}

// The same for one item, and the claim of the phase's next one, whose latency is
// the same (one after the other on both sides of every phase: 4 us more on a dense
// hull's three phases).  *last: as finish_items returns.
__device__ __forceinline__ unsigned finish_and_claim(Ctl* ctl, int phase, unsigned items, bool* last = nullptr) {
    __shared__ unsigned s_next, s_end;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned before = atomicAdd(&ctl->finished[phase], 1u);
        s_next = atomicAdd(&ctl->claimed[phase], 1u);
        s_end = before + 1u == items;
        if (last && s_end) __threadfence();
    }
    __syncthreads();
    if (last) *last = s_end != 0u;
    return s_next;
}

// Bounded: false when the wait gave up (status CH_ETIMEOUT), after kSpinLimit
// polls in which no item of the phase was taken or finished and no block
// reported progress within one (ctl->beat).  Meanwhile claims an item of phase
// next, to be worked on after the wait.
__device__ __forceinline__ bool wait_phase(Ctl* ctl, int phase, unsigned items, int next = -1, unsigned* item = nullptr) {
    __shared__ int s_ok;
    __shared__ unsigned s_claim;
    __syncthreads();
    if (threadIdx.x == 0) {
        if (item) s_claim = atomicAdd(&ctl->claimed[next], 1u);
        volatile unsigned *claimed = &ctl->claimed[phase], *finished = &ctl->finished[phase], *beat = &ctl->beat;
        unsigned spins = 0u, seen = 0u;
        s_ok = 1;
        while (*finished < items) {
            if (spin_give_up(spins, ctl)) {
                s_ok = 0;
                break;
            }
            if ((spins & 1023u) == 0u) {
                const unsigned now = *claimed + *finished + *beat;
                if (now != seen) spins = 0u;
                seen = now;
            }
        }
        __threadfence();
    }
    __syncthreads();
    if (item) *item = s_claim;
    return s_ok != 0;
}

__device__ __forceinline__ int read_status(const Ctl* ctl) {
    return *(volatile const int*)&ctl->status;
}

// Queue-frame coordinates of a survivor.  For queue r the chain from its
// start extreme to its end extreme is strictly increasing in u, and among
// points of equal u only the one of minimum v can be a hull vertex.  Every
// map (x, y) -> (u, v) is a rotation by a multiple of 90 degrees plus 45,
// scaled by sqrt(2): orientation-preserving, so cross products keep their sign.
//   r = 0 (W->S):  u = x - y + 2^24,      v = x + y
//   r = 1 (S->E):  u = x + y,             v = y - x + 2^24
//   r = 2 (E->N):  u = y - x + 2^24,      v = 2^25 - 2 - x - y
//   r = 3 (N->W):  u = 2^25 - 2 - x - y,  v = x - y + 2^24
__device__ __forceinline__ void queue_frame(int r, int x, int y, uint32_t& u, uint32_t& v) {
    const int off = kCoordLimit;
    const int top = 2 * kCoordLimit - 2;
    switch (r) {
        case 0: u = (uint32_t)(x - y + off); v = (uint32_t)(x + y); break;
        case 1: u = (uint32_t)(x + y); v = (uint32_t)(y - x + off); break;
        case 2: u = (uint32_t)(y - x + off); v = (uint32_t)(top - x - y); break;
        default: u = (uint32_t)(top - x - y); v = (uint32_t)(x - y + off); break;
    }
}

__device__ __forceinline__ uint32_t make_key(int r, uint32_t u) { return ((uint32_t)r << kKeyBits) | u; }
__device__ __forceinline__ uint64_t make_val(uint32_t v, uint32_t idx) {
    return ((uint64_t)v << 31) | (uint64_t)idx;
}

}  // namespace ch
