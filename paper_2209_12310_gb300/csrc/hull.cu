// hull.cu -- the large-survivor path by sort: the radix sort (sort.cuh) and the
// hull of the sorted survivors, in one launch.
//
// The paper ends with "for i = 1..4: CH <- CH U hull(Q_i, n_i)" (Alg. 1): one
// hull per queue, joined.  Here every queue r is a chain from quad vertex r
// to quad vertex r+1 that is strictly monotone in the queue-frame coordinate u
// (see queue_frame), and its hull chain is Andrew's lower chain (Table I) in
// the (u, v) frame:
//   sort_kernel    the digit histograms, the three passes; then queue
//                  boundaries from the top-digit histogram; per tile
//                  of 4096 records: keep the minimum-(v, index)
//                  record of every run of equal u (only it can be a vertex),
//                  build per-thread chains, merge them pairwise in shared
//                  memory, then merge tiles pairwise up a binary tree: the
//                  block that completes a pair (second arrival on an atomic
//                  counter) performs that merge, so no block ever waits;
//                  the block completing the fourth queue root joins the
//                  chains (stitch_core: collinear junction vertices dropped,
//                  degenerate cases, rotation to the lex-smallest vertex).
// As one kernel the path costs a call that does not take it one empty launch.
//
// Merging two chains A, B (all u of A below all u of B): a_k (k > 0) stays iff
// every b in B is strictly left of a_{k-1} -> a_k; b_l (l < |B|-1) stays iff
// every a in A is strictly left of b_l -> b_{l+1}.  Both predicates hold on a
// prefix of A / a suffix of B, and "every b" reduces to the minimum of a
// linear function over the convex chain B, found by binary search.
#include "ch_internal.cuh"
#include "hullcore.cuh"
#include "launch.h"
#include "merge.cuh"
#include "sort.cuh"

#include <climits>

namespace ch {

// ---------------------------------------------------------------------------
struct HullBufs {
    const uint32_t* keys;   // sorted records
    const uint64_t* vals;
    int* cu;                // chain storage: tile c at [c*kChainTile, ...)
    int* cv;
    int* ci;
    int* clen;
    int* counters;          // merge-tree arrival counters (zero at rest)
    int ctcap;
    int* vbuf;              // stitch scratch (2 * records ints)
    int* kbuf;              // stitch scratch (records ints)
    int* xbuf;              // stitch coordinates (records ints each)
    int* ybuf;
    const float* pts;
    long long n;
    int32_t* out_idx;
    int64_t* out_n;
};

static_assert(kSortThreads == kChainThreads, "one block shape");

__global__ void __launch_bounds__(kChainThreads) sort_kernel(Ctl* ctl, uint32_t* kA, uint64_t* vA, uint32_t* kB,
                                                             uint64_t* vB, unsigned long long* status, HullBufs hb) {
    extern __shared__ int smem[];
    int* su = smem;
    int* sv = su + kMergeSmemCap;
    int* si = sv + kMergeSmemCap;
    __shared__ int s_len[kChainThreads];
    __shared__ int s_red[4];
    __shared__ int s_old;
    __shared__ unsigned s_qn[4], s_q0[5], s_tb[5];
    __shared__ uint64_t s_behind;   // of the run at a tile's end, minimum behind the tile
    __shared__ int s_mv[kChainThreads / 2][3];   // per pair: destination, source, count

    if (*(volatile int*)&ctl->done) return;
    bool go = !__syncthreads_or(read_status(ctl) != CH_OK);   // (a wait below may set it meanwhile)
    if (go) {
        if (*(volatile int*)&ctl->bk_state != 2) return;
        SortSmem& sm = *reinterpret_cast<SortSmem*>(smem);
        go = wait_phase(ctl, kSortHist, sort_hist(reinterpret_cast<unsigned(*)[kDigits]>(smem), kA, ctl));
        if (go) go = wait_phase(ctl, kSortPass, onesweep(sm, kA, vA, kB, vB, ctl, status, 0));
        if (go) go = wait_phase(ctl, kSortPass + 1, onesweep(sm, kB, vB, kA, vA, ctl, status, 1));
        if (go) go = wait_phase(ctl, kSortPass + 2, onesweep(sm, kA, vA, kB, vB, ctl, status, 2));
    }
    if (__syncthreads_or(!go || read_status(ctl) != CH_OK)) {   // a wait gave up: report it
        if (threadIdx.x == 0) *hb.out_n = read_status(ctl);
        return;
    }
    const int tid = threadIdx.x;
    // Queue r holds the top-pass digits [128 r, 128 (r + 1)), so its size is a
    // sum of that histogram.
    if (tid < 4) s_qn[tid] = 0u;
    __syncthreads();
    for (int d = tid; d < kDigits; d += blockDim.x) {
        const unsigned c = ctl->digit_hist[kSortPasses - 1][d];
        if (c) atomicAdd(&s_qn[d >> (kDigitBits - 2)], c);
    }
    __syncthreads();
    if (tid == 0) {
        const unsigned per = (unsigned)kChainTile;
        unsigned q = 0, tb = 0;
        for (int r = 0; r < 4; ++r) {
            s_q0[r] = q;
            s_tb[r] = tb;
            q += s_qn[r];
            tb += (s_qn[r] + per - 1) / per;
        }
        s_q0[4] = q;
        s_tb[4] = tb;
    }
    __syncthreads();
    const unsigned total_tiles = s_tb[4];
    const unsigned nrec = ctl->count;
    const int seg = kChainItems;      // shared-memory slot per leaf chain
    const int nseg = kChainThreads;   // leaf chains per tile

    for (unsigned c = blockIdx.x; c < total_tiles; c += gridDim.x) {
        CH_MG_DECL
        int r = 0;
        while (r < 3 && c >= s_tb[r + 1]) ++r;
        const unsigned rb = s_tb[r];
        const unsigned ct = s_tb[r + 1] - rb;
        const unsigned t_local = c - rb;
        const unsigned q0 = s_q0[r], q1 = s_q0[r + 1];
        const unsigned ts = q0 + t_local * (unsigned)kChainTile;
        const unsigned te = min(q1, ts + (unsigned)kChainTile);

        // 1) run reduction + per-thread chain (records [ts + 16 tid, +16)).
        // A run (records of equal queue and u) belongs to the thread with its
        // first record; where it goes on, the threads behind tell what they hold
        // of it, and the block reads together what lies behind the tile (one
        // thread alone took 1.1 ms for 12,000 copies of a point).
        {
            const int sbase = tid * kChainItems;
            const unsigned p0 = ts + tid * kChainItems;
            const int have = p0 < te ? (int)min((unsigned)kChainItems, te - p0) : 0;
            uint64_t* lead = reinterpret_cast<uint64_t*>(su + kChainTile);   // minimum of the thread's first run
            int* leadk = sv + kChainTile;                                   // its key, -1 for none
            int* whole = si + kChainTile;                                   // all of the thread's records
            uint32_t k[kChainItems];
            uint64_t w[kChainItems];
#pragma unroll
            for (int m = 0; m < kChainItems; ++m) {
                k[m] = m < have ? hb.keys[p0 + m] : 0u;
                w[m] = m < have ? hb.vals[p0 + m] : ~0ull;
            }
            {
                uint64_t best = w[0];
                bool in = have > 0;
#pragma unroll
                for (int m = 1; m < kChainItems; ++m) {
                    in = in && m < have && k[m] == k[0];
                    best = in && w[m] < best ? w[m] : best;
                }
                lead[tid] = best;
                leadk[tid] = have ? (int)k[0] : -1;
                whole[tid] = in && have == kChainItems;
            }
            // behind the tile: the run that reaches its end, when it began in it
            if (tid == 0) s_behind = ~0ull;
            __syncthreads();
            const uint32_t last = hb.keys[te - 1u];
            if (te < q1 && hb.keys[te] == last && (ts == q0 || hb.keys[ts - 1u] != last)) {
                uint64_t best = ~0ull;
                constexpr int kU = 4;
                bool more = true;
                for (unsigned p = te; more; p += kU * kChainThreads) {
#pragma unroll
                    for (int e = 0; e < kU; ++e) {
                        const unsigned i = p + e * kChainThreads + tid;
                        const bool in = i < q1 && hb.keys[i] == last;
                        if (in) best = min(best, hb.vals[i]);
                        else more = false;
                    }
                    more = __syncthreads_and(more);
                }
                atomicMin(reinterpret_cast<unsigned long long*>(&s_behind), (unsigned long long)best);
                __syncthreads();
            }
            int sp = 0;
            uint64_t best = ~0ull;
            const uint32_t before = have && p0 != q0 ? hb.keys[p0 - 1u] : 0u;
#pragma unroll
            for (int m = 0; m < kChainItems; ++m) {
                if (m >= have) break;
                const bool first = m ? k[m] != k[m - 1] : p0 == q0 || k[0] != before;
                if (first) best = w[m];
                else best = best < w[m] ? best : w[m];
                const bool ends = m + 1 < kChainItems && m + 1 < have && k[m + 1] != k[m];
                if (!ends && m + 1 < have) continue;
                // the run that begins the thread's records belongs to a thread before
                bool own = p0 == q0 || k[m] != before;
                if (!own) continue;
                if (!ends) {   // goes on behind the thread's records?
                    int t = tid + 1;
                    bool on = true;
                    while (on && t < kChainThreads && leadk[t] == (int)k[m]) {
                        best = min(best, lead[t]);
                        on = whole[t] != 0;
                        ++t;
                    }
                    if (on && k[m] == last) best = min(best, s_behind);
                }
                const int pu = (int)(k[m] & kKeyMask);
                const int pv = (int)(best >> 31);
                const int pi = (int)(best & 0x7FFFFFFFull);
                while (sp >= 2 && cross_uv(su[sbase + sp - 2], sv[sbase + sp - 2], su[sbase + sp - 1],
                                           sv[sbase + sp - 1], pu, pv) <= 0)
                    --sp;
                su[sbase + sp] = pu; sv[sbase + sp] = pv; si[sbase + sp] = pi;
                ++sp;
            }
            s_len[tid] = sp;
        }
        __syncthreads();
        CH_MG(0);
        const TreeBufs tb{hb.cu, hb.cv, hb.ci, hb.clen, hb.counters, hb.ctcap};
        const bool root = tile_merge_climb(su, sv, si, s_len, s_mv, seg, nseg, tb, c, rb, ct, t_local, s_red, &s_old);
        __syncthreads();
        if (!root) continue;
        // 5) the block completing the fourth queue root joins the chains.
        __threadfence();
        __syncthreads();
        if (tid == 0) s_old = (int)atomicAdd(&ctl->roots_done, 1u);
        __syncthreads();
        if (s_old != 3) continue;
        __threadfence();
        int off[5];
        off[0] = 0;
        for (int q = 0; q < 4; ++q) off[q + 1] = off[q] + __ldcg(hb.clen + s_tb[q]) - 1;
        const int m = off[4];
        if (m < 0 || m > (int)nrec) {   // inconsistent state: report, never read out of range
            if (tid == 0) { set_status(ctl, CH_ECUDA); *hb.out_n = CH_ECUDA; }
            return;
        }
        // the cycle's coordinates from the chains' frames (no reads of the
        // points), into the sort/scatter buffers, free by now
        for (int q = 0; q < 4; ++q) {
            const size_t o = (size_t)s_tb[q] * kChainTile;
            for (int j = tid; j < off[q + 1] - off[q]; j += blockDim.x) {
                int x, y;
                frame_to_xy(q, __ldcg(hb.cu + o + j), __ldcg(hb.cv + o + j), x, y);
                hb.vbuf[off[q] + j] = __ldcg(hb.ci + o + j);
                hb.xbuf[off[q] + j] = x;
                hb.ybuf[off[q] + j] = y;
            }
        }
        __syncthreads();
        const int* X = hb.xbuf;
        const int* Y = hb.ybuf;
        CH_MG(7);
        stitch_core(hb.vbuf, m, hb.kbuf, hb.vbuf + m,
                    [&](int p, long long& x, long long& y) { x = __ldcg(X + p); y = __ldcg(Y + p); }, hb.n, ctl,
                    hb.out_idx, hb.out_n);
        CH_MG(8);
        return;
    }
}

// ---------------------------------------------------------------------------
#ifdef CH_PHASEPROF
}  // namespace ch
extern "C" int ch_phase_read_merge(unsigned long long* out16) {
    return cudaMemcpyFromSymbol(out16, ch::g_mg_phase, sizeof(unsigned long long) * 16) == cudaSuccess ? 0 : -4;
}
extern "C" int ch_phase_reset_merge(void) {
    unsigned long long z[16] = {};
    return cudaMemcpyToSymbol(ch::g_mg_phase, z, sizeof(z)) == cudaSuccess ? 0 : -4;
}
namespace ch {
#endif

size_t chain_smem_bytes() { return (size_t)3 * kMergeSmemCap * sizeof(int); }

void launch_sort(Ctl* ctl, uint32_t* kA, uint64_t* vA, uint32_t* kB, uint64_t* vB, unsigned long long* status, int* cu,
                 int* cv, int* ci, int* clen, int* counters, int ctcap, const float* pts, long long n, int32_t* out_idx,
                 int64_t* out_n, int grid, cudaStream_t s) {
    // the A buffers are free once the records are sorted into B, and B once
    // its chains are built: the stitch's scratch
    const HullBufs hb{kB, vB, cu, cv, ci, clen, counters, ctcap, (int*)vA, (int*)kA, (int*)kB, (int*)vB, pts, n, out_idx,
                      out_n};
    sort_kernel<<<grid, kChainThreads, chain_smem_bytes(), s>>>(ctl, kA, vA, kB, vB, status, hb);
}

cudaError_t configure_hull_kernels() {
    return cudaFuncSetAttribute(sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)chain_smem_bytes());
}

cudaError_t occupancy_sort(int* b) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(b, sort_kernel, kChainThreads, chain_smem_bytes());
}

}  // namespace ch
