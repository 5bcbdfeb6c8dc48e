// setup.cuh -- what the kernels that begin a hull share: the reset of the control
// block and the records of the octagon's vertices.
#pragma once

#include "ch_internal.cuh"
#include "octagon.cuh"

namespace ch {

// ---------------------------------------------------------------------------
// Resets the per-call control block (one block).  The fields that the sample
// pass itself gathers in (samp_packed, blocks_done[0]) are at rest between
// calls: its last block leaves them at zero.
__device__ __forceinline__ void reset_ctl(Ctl* ctl, int mode) {
    const int t = threadIdx.x;
    if (t < 8) {
        ctl->ext_packed[t] = 0ull;
        ctl->line_ep[t] = (t & 1) ? 0ull : ~0ull;   // even: minimum slot, odd: maximum slot
    }
    if (t < 4) {
        ctl->counts4[t] = 0u;
        ctl->rec_q[t] = 0u;
        if (t) ctl->blocks_done[t] = 0u;
    }
    if (t < 4 * (kJoinRounds + 1)) (&ctl->join_n[0][0])[t] = 0u;
    if (t < kPhases) {
        ctl->claimed[t] = 0u;
        ctl->finished[t] = 0u;
    }
    if (t == 0) {
        ctl->status = CH_OK;
        ctl->abort = 0;
        ctl->count = 8u;
        ctl->count_raw = 0u;
        ctl->epoch += 1u;
        ctl->mode = mode;
        ctl->done = 0;
        ctl->bk_state = 0;
        ctl->path = kPathNone;
        ctl->beat = 0u;
        ctl->joins_done = 0u;
        ctl->roots_done = 0u;
        ctl->samp_dense = 0;
        ctl->oct_ready = 0;
        ctl->star_k = 0;
        ctl->star_final = 0;
    }
    unsigned* h = &ctl->digit_hist[0][0];
    for (int i = t; i < kSortPasses * kDigits; i += blockDim.x) h[i] = 0u;
#if defined(CH_TRACE) || defined(CH_TIMELINE)
    if (t < 24) { ctl->tl[t][0] = ~0ull; ctl->tl[t][1] = 0ull; }
#endif
}

// The records of the extremes (vx, vy, id: shared memory), by the block's first 12
// threads: slots 0 .. 7 and, past ctl->count, the others.
__device__ __forceinline__ void end_records(const int* s_vx, const int* s_vy, const int* s_id, Ctl* ctl, uint32_t* keys,
                                            uint64_t* vals) {
    if (threadIdx.x < 12) {
        // Threads 0..7: chain end points (queue r runs from quad vertex r to
        // r+1).  Threads 8..11: the diagonal extreme of queue r, when it lies
        // strictly right of the quad edge (the hull rule drops every point of
        // the closed octagon, vertices included, so the vertices that can be
        // hull vertices get their own record; on the edge it cannot be one).
        const int lane = threadIdx.x;
        int r, d;
        bool emit = true;
        if (lane < 8) {
            r = lane >> 1;
            d = (lane & 1) ? ((2 * r + 2) & 7) : 2 * r;
        } else {
            r = lane - 8;
            d = 2 * r + 1;
            const int a = 2 * r, b = (2 * r + 2) & 7;
            emit = orient64(s_vx[a], s_vy[a], s_vx[b], s_vy[b], s_vx[d], s_vy[d]) < 0;
        }
        if (emit) {
            uint32_t u, v;
            queue_frame(r, s_vx[d], s_vy[d], u, v);
            const uint32_t key = make_key(r, u);
            const unsigned pos = lane < 8 ? (unsigned)lane : atomicAdd(&ctl->count, 1u);
            keys[pos] = key;
            vals[pos] = make_val(v, (uint32_t)s_id[d]);
            atomicAdd(&ctl->rec_q[r], 1u);
        }
    }
}

}  // namespace ch
