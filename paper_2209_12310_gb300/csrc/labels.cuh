// labels.cuh -- the stores of the label passes (ch_filter, ch_filter16).
#pragma once

#include <cstdint>

namespace ch {

// Warp-collective: the labels 4 q .. 4 q + 3 of a warp tile (q = 32 r + lane in
// round r; `word` holds the lane's four, lowest first) into out, the tile's
// first label, off bytes past a 4-byte boundary, by aligned words: the last off
// labels of the lane before and the first 4 - off of the lane's own.  The
// tile's first and last bytes share their words with the neighbouring tiles and
// go alone.  `before`: the previous round's words, kept by the caller (any
// value before round 0).
__device__ __forceinline__ void store_labels(uint8_t* out, int q, unsigned off, uint32_t word, uint32_t& before) {
    if (off == 0u) {
        __stcs(reinterpret_cast<uint32_t*>(out) + q, word);
        return;
    }
    const int lane = (int)(threadIdx.x & 31u);
    const uint32_t up = __shfl_up_sync(0xFFFFFFFFu, word, 1);
    const uint32_t prev = lane == 0 ? before : up;
    if (q > 0) {
        __stcs(reinterpret_cast<uint32_t*>(out - off) + q, __funnelshift_l(prev, word, 8u * off));
    } else {
        for (unsigned b = 0u; b < 4u - off; ++b) out[b] = (uint8_t)(word >> (8u * b));
    }
    before = __shfl_sync(0xFFFFFFFFu, word, 31);
    if (q == kWarpTilePts / 4 - 1)
        for (unsigned b = 4u - off; b < 4u; ++b) out[4 * q + b] = (uint8_t)(word >> (8u * b));
}

}  // namespace ch
