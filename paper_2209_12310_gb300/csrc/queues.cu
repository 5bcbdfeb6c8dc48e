// queues.cu -- hull of many survivors without a full sort.
//
// The post pass leaves the records in no order, counted per queue, and picks
// one of three ways (post_last_block):
//   queues  every queue fits one block: a block per queue sorts the queue by u
//           and reduces it to its lower chain in shared memory (qchain.cuh);
//   tiles   the u range of each queue is cut into tiles of some thousand
//           records, which a block each reduces the same way, and a block per
//           queue reduces its tiles' chains, joined in u order, to its chain
//           (all blocks in rounds, when those outgrow shared memory);
//   sort    the radix sort and the merge tree (sort.cuh, hull.cu), also when a
//           tile's chain outgrows shared memory.
// The lower chain of a set of points equals the lower chain of the chains of
// any partition of it into u ranges, joined in u order.
//
// large_kernel is one launch for the first two ways: its blocks share the phases
// of the tiles (count, cut, move, reduce) by claimed items and wait for their
// ends (claim_item, wait_phase).  As one kernel it costs a call that needs none of
// it one empty launch.
#include "ch_internal.cuh"
#include "host.h"
#include "hullcore.cuh"
#include "launch.h"
#include "partition.cuh"
#include "qchain.cuh"

namespace ch {

constexpr int kQGroups = 1024;          // equal u ranges of a queue
// Records of a tile on average: as many tiles as blocks, or twice, three times
// ... as many while a tile would have more than kTileMost (the density of near-
// hull records varies by a quarter around its average along a queue).
constexpr unsigned kTileMost = 6000;
constexpr int kLargeThreads = 1024;
using QcQueue = QcSmem<kQueueCap, 4096>;
static_assert(4 * kQGroups == kPtGroups, "groups of the four queues; as many tiles at most");

// u ranges of the queues (every record of queue r has u between its two quad
// vertices); the same float arithmetic in every kernel, monotone in u.
struct QMap {
    int lo[4], hi[4];
    float scale[4];
};

__device__ __forceinline__ void q_map(const Octagon& o, QMap& m) {   // threads 0 .. 3
    const int r = threadIdx.x;
    if (r < 4) {
        uint32_t ulo, uhi, v;
        queue_frame(r, o.vx[2 * r], o.vy[2 * r], ulo, v);
        queue_frame(r, o.vx[(2 * r + 2) & 7], o.vy[(2 * r + 2) & 7], uhi, v);
        m.lo[r] = (int)ulo;
        m.hi[r] = (int)uhi;
        m.scale[r] = (float)kQGroups / (float)((int)uhi - (int)ulo + 1);
    }
}

__device__ __forceinline__ unsigned q_group(const QMap& m, uint32_t key) {
    const int r = (int)(key >> kKeyBits);
    const int g = (int)((float)((int)(key & kKeyMask) - m.lo[r]) * m.scale[r]);
    return (unsigned)(r * kQGroups + max(0, min(kQGroups - 1, g)));
}

struct LargeArgs {
    Ctl* ctl;
    const uint32_t* keys;    // the records
    const uint64_t* vals;
    uint32_t* kB;            // the records by tile; then scratch and
    uint64_t* vB;            // the queues' chains (u, v)
    unsigned *ghist, *gtile, *tbeg, *tcur;   // kPtGroups each
    unsigned* seg[2];        // as many: ghist and gtile again, once the tiles stand
    int* tlen;
    int *cu, *cv, *ci;       // the tiles' chains; then (cu) the queues' chains (index)
    long long n;
    int32_t* out_idx;
    int64_t* out_n;
};

// Records per group (shared-memory counts, then one atomic per group that
// occurs), by chunks of the records, as many as blocks unless those grow long.
// Returns whether this block finished the last chunk.
struct TileHistSmem {
    unsigned h[kPtGroups];     // records per group; in the cut, per tile
    unsigned beg[kPtGroups];
    unsigned q0[5], tb[5];
    int tmp[33];
};

__device__ bool tile_hist(const LargeArgs& a, TileHistSmem& sm, const QMap& m) {
    const int tid = threadIdx.x;
    const unsigned n = a.ctl->count;
    const unsigned chunk = min(64u, (n - 1u) / (gridDim.x * kLargeThreads) + 1u) * kLargeThreads;
    const unsigned chunks = (n - 1u) / chunk + 1u;
    constexpr int kU = 4;
    bool last = false;
    for (unsigned c = claim_item(a.ctl, kLargeHist); c < chunks; c = finish_and_claim(a.ctl, kLargeHist, chunks, &last)) {
        for (int g = tid; g < kPtGroups; g += kLargeThreads) sm.h[g] = 0u;
        __syncthreads();
        const unsigned end = min(n, (c + 1u) * chunk);
        for (unsigned i0 = c * chunk + tid; i0 < end; i0 += kLargeThreads * kU) {
            uint32_t k[kU];
#pragma unroll
            for (int j = 0; j < kU; ++j)
                if (i0 + j * kLargeThreads < end) k[j] = __ldcg(a.keys + i0 + j * kLargeThreads);
#pragma unroll
            for (int j = 0; j < kU; ++j)
                if (i0 + j * kLargeThreads < end) atomicAdd(&sm.h[q_group(m, k[j])], 1u);
        }
        __syncthreads();
        for (int g = tid; g < kPtGroups; g += kLargeThreads)
            if (sm.h[g]) atomicAdd(&a.ghist[g], sm.h[g]);
    }
    return last;
}

// One block cuts the tiles: gtile maps a group to its tile, tile t's records go
// to tbeg[t] on.
__device__ void tile_cut(const LargeArgs& a, TileHistSmem& sm) {
    const int tid = threadIdx.x;
    Ctl* ctl = a.ctl;
    constexpr int kE = kPtGroups / kLargeThreads;   // groups per thread, all of one queue
    unsigned c[kE], sum = 0u;
#pragma unroll
    for (int e = 0; e < kE; ++e) {
        c[e] = __ldcg(a.ghist + tid * kE + e);
        sum += c[e];
    }
    int tot;
    unsigned run = (unsigned)block_excl_scan((int)sum, sm.tmp, &tot);
    if (tid % (kQGroups / kE) == 0) sm.q0[tid / (kQGroups / kE)] = run;
    if (tid == 0) sm.q0[4] = (unsigned)tot;
    for (int t = tid; t < kPtGroups; t += kLargeThreads) {
        sm.h[t] = 0u;
        sm.beg[t] = 0xFFFFFFFFu;
    }
    __syncthreads();
    const unsigned n = (unsigned)tot;
    const unsigned rounds = (n + gridDim.x * kTileMost - 1) / (gridDim.x * kTileMost);
    // at most kPtGroups - 92 tiles (more records: larger tiles, in pieces)
    const unsigned target = max(n / (gridDim.x * rounds) + 1u, n / (unsigned)(kPtGroups - 96) + 1u);
    if (tid == 0) {
        unsigned t = 0u;
        for (int r = 0; r < 4; ++r) {
            sm.tb[r] = t;
            t += (sm.q0[r + 1] - sm.q0[r]) / target + 1u;
        }
        sm.tb[4] = t;
        for (int r = 0; r < 5; ++r) ctl->q_tile[r] = sm.tb[r];
    }
    __syncthreads();
    const int r = tid / (kQGroups / kE);
#pragma unroll
    for (int e = 0; e < kE; ++e) {
        const unsigned t = sm.tb[r] + (run - sm.q0[r]) / target;
        a.gtile[tid * kE + e] = t;
        if (c[e]) {
            atomicMin(&sm.beg[t], run);
            atomicAdd(&sm.h[t], c[e]);
        }
        run += c[e];
    }
    __syncthreads();
    for (unsigned t = tid; t < sm.tb[4]; t += kLargeThreads) {
        const unsigned b = sm.h[t] ? sm.beg[t] : 0u;   // a tile that a large group skipped is empty
        a.tbeg[t] = b;
        a.tcur[t] = b;
    }
}

// Records into their tiles' ranges; tcur[t] ends up at the end of tile t.
struct TilePartSmem {
    PartSmem p;
    unsigned short gtile[kPtGroups];
};

// item: claimed already.  Returns the number of the phase's items.
__device__ unsigned tile_part(const LargeArgs& a, TilePartSmem& sm, const QMap& m, unsigned item) {
    static_assert(kLargeThreads == kPtThreads, "partition block");
    const int tid = threadIdx.x;
    for (int g = tid; g < kPtGroups; g += kPtThreads) sm.gtile[g] = (unsigned short)__ldcg(a.gtile + g);
    const unsigned n = a.ctl->count, nt = *(volatile unsigned*)&a.ctl->q_tile[4];
    const unsigned parts = (n - 1u) / kPtTile + 1u;
    __syncthreads();
    for (unsigned p = item; p < parts; p = finish_and_claim(a.ctl, kLargePart, parts)) {
        const unsigned i0 = p * kPtTile;
        partition_tile(
            sm.p, a.keys, a.vals, i0, min((unsigned)kPtTile, n - i0), nt,
            [&](uint32_t key) { return (unsigned)sm.gtile[q_group(m, key)]; },
            [&](unsigned g, unsigned cnt) { return atomicAdd(&a.tcur[g], cnt); }, a.kB, a.vB);
    }
    return parts;
}

// The tiles' lower chains, to [tbeg[t], tbeg[t] + tlen[t]) of cu / cv / ci
// (u, v, index).  A tile with more records than the block holds goes in
// pieces: the records after the first piece are tested against the chain so far
// as they are read, and only those that it leaves (few, unless the records are
// mostly vertices; none of a vertex's copies) are sorted with it.  (Every piece
// sorted whole, a million points with 600,000 copies of one hull vertex took
// 23 ms; see tile_read.)  When the chain fills the block, the call goes to the
// sort.
constexpr int kReadU = 2;                                         // records per thread and step
constexpr int kCarry = QcQueue::kCap - kReadU * kLargeThreads;    // vertices carried at most

// Reads the tile's records from c0 on (at beg + c0, cnt in all), while a step's
// fit the block; q.a and q.si [0, len) hold the chain so far, what it leaves goes
// behind.  Returns the number of points in q.a, *next the first record not read.
__device__ int tile_read(const LargeArgs& a, QcQueue& q, unsigned beg, unsigned cnt, unsigned c0, int len, unsigned* next) {
    __shared__ int s_fill;
    constexpr int T = kLargeThreads, U = kReadU;
    const int tid = threadIdx.x, lane = tid & 31;
    uint32_t k[U];
    uint64_t w[U];
    auto load = [&]() {
#pragma unroll
        for (int e = 0; e < U; ++e) {
            const unsigned j = c0 + e * T + tid;
            k[e] = j < cnt ? __ldcg(a.kB + beg + j) & kKeyMask : 0u;
            w[e] = j < cnt ? __ldcg(a.vB + beg + j) : 0ull;
        }
    };
    if (tid == 0) s_fill = len;
    load();
    int fill = len;
    for (unsigned step = 0u; c0 < cnt && fill <= QcQueue::kCap - U * T; ++step) {
        unsigned long long x[U];
        int id[U];
        bool keep[U];
#pragma unroll
        for (int e = 0; e < U; ++e) {
            x[e] = qc_pack(k[e], (unsigned)(w[e] >> 31), (1u << kQcPosBits) - 1u);   // no slot of a vertex
            id[e] = (int)(w[e] & 0x7FFFFFFFull);
            keep[e] = c0 + e * T + tid < cnt;
        }
        c0 += U * T;
        load();   // the next step's, while this one's are tested
        __syncthreads();   // s_fill and q.a [0, len) stand
#pragma unroll
        for (int e = 0; e < U; ++e) {
            keep[e] = keep[e] && qc_beside(x[e], id[e], q.a, len, q.si);
            // of a warp's copies of one point, the lowest index
            unsigned bal = __ballot_sync(0xFFFFFFFFu, keep[e]);
            if (bal == 0u) continue;
            if (keep[e]) {
                const unsigned same = __match_any_sync(bal, x[e]);
                keep[e] = (unsigned)id[e] == __reduce_min_sync(same, (unsigned)id[e]);
            }
            bal = __ballot_sync(0xFFFFFFFFu, keep[e]);
            int pos = 0;
            if (lane == 0) pos = atomicAdd(&s_fill, __popc(bal));
            pos = __shfl_sync(0xFFFFFFFFu, pos, 0) + __popc(bal & lanemask_lt());
            if (keep[e]) {
                q.a[pos] = (x[e] & ~((1ull << kQcPosBits) - 1ull)) | (unsigned)pos;
                q.si[pos] = id[e];
            }
        }
        __syncthreads();
        fill = s_fill;
        if (tid == 0 && (step & 63u) == 63u) atomicAdd(&a.ctl->beat, 1u);
    }
    __syncthreads();
    *next = min(c0, cnt);
    return fill;
}

__device__ void tile_chains(const LargeArgs& a, QcQueue& q, unsigned item) {
    const int tid = threadIdx.x;
    constexpr int T = kLargeThreads, kCap = QcQueue::kCap, kPer = kCap / T;
    static_assert(kCap % T == 0, "carried points per thread");
    const unsigned nt = *(volatile unsigned*)&a.ctl->q_tile[4];
    for (unsigned t = item; t < nt; t = finish_and_claim(a.ctl, kLargeChains, nt)) {
        const unsigned beg = __ldcg(a.tbeg + t), cnt = __ldcg(a.tcur + t) - beg;
        unsigned long long *src = q.a, *dst = q.b;
        int len = 0;
        for (unsigned c0 = 0; c0 < cnt;) {
            int n;
            if (len == 0) {
                n = (int)min(cnt, (unsigned)kCap);
#pragma unroll 5
                for (int j = tid; j < n; j += T) {
                    const uint32_t k = __ldcg(a.kB + beg + j);
                    const uint64_t w = __ldcg(a.vB + beg + j);
                    q.a[j] = qc_pack(k & kKeyMask, (unsigned)(w >> 31), (unsigned)j);
                    q.si[j] = (int)(w & 0x7FFFFFFFull);
                }
                c0 = (unsigned)n;
            } else {   // the chain so far in slots 0 .. len - 1
                unsigned long long w[kPer];
                int id[kPer];
#pragma unroll
                for (int e = 0; e < kPer; ++e) {
                    const int j = e * T + tid;
                    w[e] = j < len ? src[j] : 0ull;
                    id[e] = j < len ? q.si[qc_pos(w[e])] : 0;
                }
                __syncthreads();
#pragma unroll
                for (int e = 0; e < kPer; ++e) {
                    const int j = e * T + tid;
                    if (j < len) {
                        q.a[j] = qc_pack((unsigned)qc_u(w[e]), (unsigned)qc_v(w[e]), (unsigned)j);
                        q.si[j] = id[e];
                    }
                }
                src = q.a;
                dst = q.b;
                n = tile_read(a, q, beg, cnt, c0, len, &c0);
            }
            __syncthreads();
            if (n > len) {
                // the buckets span the points' own range, which is the tile's
                int lo = INT_MAX, hi = INT_MIN;
                for (int j = tid; j < n; j += T) {
                    lo = min(lo, qc_u(q.a[j]));
                    hi = max(hi, qc_u(q.a[j]));
                }
                lo = block_reduce<int>(lo, [](int x, int y) { return min(x, y); }, q.tmp);
                hi = block_reduce<int>(hi, [](int x, int y) { return max(x, y); }, q.tmp);
                n = qc_sort<T>(q, n, lo, hi);
                src = q.a;
                dst = q.b;
                len = qc_eliminate<T>(src, dst, n, q.tmp);
            }
            if (tid == 0) atomicAdd(&a.ctl->beat, 1u);   // a tile can hold any share of the records
            if (len > kCarry && c0 < cnt) {   // no room for the rest
                if (tid == 0) a.ctl->bk_state = 2;
                len = 0;
                break;
            }
        }
        for (int j = tid; j < len; j += T) {
            const unsigned long long w = src[j];
            a.cu[beg + j] = qc_u(w);
            a.cv[beg + j] = qc_v(w);
            a.ci[beg + j] = q.si[qc_pos(w)];
        }
        if (tid == 0) {
            a.tlen[t] = len;
            int r = 0;
            while (r < 3 && t >= *(volatile unsigned*)&a.ctl->q_tile[r + 1]) ++r;
            atomicAdd(&a.ctl->join_n[0][r], (unsigned)len);
        }
    }
}

// Joining the tile chains needs no sort and keeps the indices in global
// memory: a larger capacity in the same shared memory.
struct QcJoin {
    static constexpr int kCap = 13000;
    unsigned long long a[kCap], b[kCap];
    unsigned off[kPtGroups];   // tile chains' places in the queue
    int tmp[33];
};
// Tile chains of a queue that are too long for one block, joined by all blocks in
// rounds.  The queues' points, in u order, are cut into segments; a block
// reduces a segment, with the point before and the point after it as fixed ends,
// to its lower chain (what that drops lies on or above a segment between two
// input points), and the next round cuts at other places.  A round that drops
// nothing has found every three neighbours turning strictly left: the chains
// stand.  (Of a circle's points a few at the tiles' ends go in the first round.
// 4e6 points 1.15 ms a call with the radix sort and the merge tree as the way out,
// 0.45 now; 2e7 3.4 and 1.26.)
// Round j reads the tiles' chains (j = 0), else what round j - 1 left, a segment's
// points at its place (cu / cv / ci after odd rounds, vB / kB after even ones), its
// count in seg[(j - 1) & 1].
struct JoinPlan {
    unsigned n[4], first[5];   // points and first segment of each queue
    unsigned shift;            // the first segment is shorter by this much
    __device__ __forceinline__ void set(const Ctl* ctl, int j, unsigned size) {
        shift = (j & 1) ? size / 2u : 0u;
        first[0] = 0u;
        for (int r = 0; r < 4; ++r) {
            n[r] = __ldcg(&ctl->join_n[j][r]);
            first[r + 1] = first[r] + (n[r] + shift + size - 1u) / size;
        }
    }
    __device__ __forceinline__ unsigned low(unsigned k, unsigned size) const { return k ? k * size - shift : 0u; }
};
constexpr unsigned kJoinLeast = 2048, kJoinMost = 8192;   // points of a segment
static_assert(kJoinMost + 2 <= QcQueue::kCap && QcQueue::kBuckets >= kPtGroups, "a segment's points, the pieces' places");

// Segment k of queue r in round j.
__device__ void join_segment(const LargeArgs& a, QcQueue& q, const JoinPlan& p, const JoinPlan& was, int j, int r,
                             unsigned k, unsigned size, unsigned pre) {
    constexpr int T = kLargeThreads, kE = kPtGroups / T;
    const int tid = threadIdx.x;
    Ctl* ctl = a.ctl;
    // the places of the pieces that round j - 1 left of the queue
    const unsigned t0 = j ? was.first[r] : __ldcg(&ctl->q_tile[r]);
    const unsigned np = (j ? was.first[r + 1] : __ldcg(&ctl->q_tile[r + 1])) - t0;
    const unsigned* lens = j ? a.seg[(j - 1) & 1] : reinterpret_cast<const unsigned*>(a.tlen);
    unsigned c[kE], sum = 0u;
#pragma unroll
    for (int e = 0; e < kE; ++e) {
        const unsigned t = tid * kE + e;
        c[e] = t < np ? __ldcg(lens + t0 + t) : 0u;
        sum += c[e];
    }
    int tot;
    unsigned run = (unsigned)block_excl_scan((int)sum, q.tmp, &tot);
#pragma unroll
    for (int e = 0; e < kE; ++e) {
        q.cnt[tid * kE + e] = run;
        run += c[e];
    }
    __syncthreads();
    const unsigned lo = p.low(k, size), hi = min(p.n[r], (k + 1u) * size - p.shift);
    const unsigned left = lo ? 1u : 0u, right = hi < p.n[r] ? 1u : 0u;
    const int m = (int)(hi - lo + left + right);
    for (int x = tid; x < m; x += T) {
        const unsigned i = lo - left + x;
        unsigned b = 0u, e = np;   // the last piece that begins at or before i (empty ones begin where the next does)
        while (e - b > 1u) {
            const unsigned mid = (b + e) >> 1;
            if (q.cnt[mid] <= i) b = mid;
            else e = mid;
        }
        unsigned u, v;
        int id;
        if (j & 1) {
            const size_t at = (size_t)pre + was.low(b, size) + (i - q.cnt[b]);
            const uint64_t w = __ldcg(a.vB + at);
            u = (unsigned)(w >> kKeyBits);
            v = (unsigned)(w & kKeyMask);
            id = (int)__ldcg(a.kB + at);
        } else {
            const size_t at = (j ? (size_t)pre + was.low(b, size) : (size_t)__ldcg(a.tbeg + t0 + b)) + (i - q.cnt[b]);
            u = (unsigned)__ldcg(a.cu + at);
            v = (unsigned)__ldcg(a.cv + at);
            id = __ldcg(a.ci + at);
        }
        q.a[x] = qc_pack(u, v, (unsigned)x);
        q.si[x] = id;
    }
    __syncthreads();
    unsigned long long *src = q.a, *dst = q.b;
    const int len = qc_eliminate<T>(src, dst, m, q.tmp) - (int)(left + right);   // the ends stay
    for (int x = tid; x < len; x += T) {
        const unsigned long long w = src[x + left];
        const size_t at = (size_t)pre + lo + x;
        if (j & 1) {
            a.cu[at] = qc_u(w);
            a.cv[at] = qc_v(w);
            a.ci[at] = q.si[qc_pos(w)];
        } else {
            a.vB[at] = w >> kQcPosBits;
            a.kB[at] = (uint32_t)q.si[qc_pos(w)];
        }
    }
    if (tid == 0) {
        a.seg[j & 1][p.first[r] + k] = (unsigned)len;
        atomicAdd(&ctl->join_n[j + 1][r], (unsigned)len);
    }
}

// All blocks.  Returns the last round in the one block that finished it (the
// queues' chains are at their places, without gaps), else -1; *go is false when a
// wait gave up.
__device__ int join_rounds(const LargeArgs& a, QcQueue& q, const unsigned (&pre)[5], bool* go) {
    __shared__ JoinPlan s_p[2];
    __shared__ unsigned s_size;
    const int tid = threadIdx.x;
    Ctl* ctl = a.ctl;
    if (tid == 0) {
        unsigned n = 0u;
        for (int r = 0; r < 4; ++r) n += __ldcg(&ctl->join_n[0][r]);
        s_size = max(kJoinLeast, min(kJoinMost, (n / gridDim.x + 2u) & ~1u));
    }
    __syncthreads();
    const unsigned size = s_size;
    for (int j = 0; j < kJoinRounds; ++j) {
        JoinPlan &p = s_p[j & 1], &was = s_p[(j & 1) ^ 1];
        if (tid == 0) p.set(ctl, j, size);
        __syncthreads();
        const unsigned items = p.first[4];
        bool last = false;
        if (items <= (unsigned)kPtGroups) {
            for (unsigned it; (it = claim_item(ctl, kLargeJoin + j)) < items;) {
                const int r = it >= p.first[2] ? (it >= p.first[3] ? 3 : 2) : (it >= p.first[1] ? 1 : 0);
                join_segment(a, q, p, was, j, r, it - p.first[r], size, pre[r]);
                last = finish_items(ctl, kLargeJoin + j, 1u, items);
            }
            if (!wait_phase(ctl, kLargeJoin + j, items)) {
                *go = false;
                return -1;
            }
        } else {   // too many points: the sort
            last = blockIdx.x == 0;
        }
        unsigned before = 0u, after = 0u;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            before += p.n[r];
            after += __ldcg(&ctl->join_n[j + 1][r]);
        }
        if (items <= (unsigned)kPtGroups && before == after) return last ? j : -1;
        if (items > (unsigned)kPtGroups || j + 1 == kJoinRounds) {
            if (last && tid == 0) ctl->bk_state = 2;   // the sort takes over (its input is untouched)
            return -1;
        }
    }
    return -1;
}

constexpr size_t large_max(size_t x, size_t y) { return x > y ? x : y; }
constexpr size_t kLargeSmem = large_max(large_max(sizeof(QcJoin), sizeof(QcQueue)),
                                        large_max(sizeof(TileHistSmem), sizeof(TilePartSmem)));
static_assert(kLargeSmem <= 226 * 1024 && QcJoin::kCap < (1 << kQcPosBits), "one block's shared memory");

// Blocks 0 .. 3 end with a queue each: its chain from its records (path queues)
// or from its tiles' chains (path tiles, while they fit), left at the queue's
// records' place in vB (u, v) and cu (index; each queue's own tiles' chains lie
// there, consumed by then); the block that finishes last joins the four.  Longer
// tile chains are all blocks' work (join_rounds).
__global__ void __launch_bounds__(kLargeThreads, 1) large_kernel(LargeArgs a) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ QMap s_m;
    __shared__ int s_path, s_way, s_n, s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, qq = blockIdx.x;
    constexpr int T = kLargeThreads;
    Ctl* ctl = a.ctl;
    if (tid == 0) {
        s_path = *(volatile int*)&ctl->bk_state == 1 && read_status(ctl) == CH_OK ? *(volatile int*)&ctl->path
                                                                                  : kPathNone;
        s_n = 0;
    }
    __syncthreads();
    const int path = s_path;
    if (path != kPathTiles && (path != kPathQueues || qq >= 4)) return;
    CH_TL(ctl, 13, 0);
    q_map(ctl->oct, s_m);
    __syncthreads();
    if (path == kPathTiles) {
        TileHistSmem& h = *reinterpret_cast<TileHistSmem*>(s_dyn);
        if (tile_hist(a, h, s_m)) {
            tile_cut(a, h);
            finish_items(ctl, kLargeCut, 1u, 1u);
        }
        unsigned item;
        bool go = wait_phase(ctl, kLargeCut, 1u, kLargePart, &item);
        CH_TL(ctl, 16, 1);
        if (go)
            go = wait_phase(ctl, kLargePart, tile_part(a, *reinterpret_cast<TilePartSmem*>(s_dyn), s_m, item), kLargeChains,
                            &item);
        CH_TL(ctl, 17, 1);
        if (go) {
            tile_chains(a, *reinterpret_cast<QcQueue*>(s_dyn), item);
            CH_TL(ctl, 18, 1);
            go = wait_phase(ctl, kLargeChains, *(volatile unsigned*)&ctl->q_tile[4]);
        }
        if (!go) {
            if (tid == 0) *a.out_n = CH_ETIMEOUT;
            return;
        }
        // What follows is the same for every block: the totals stand, and a tile's
        // chain that outgrew its block has set bk_state before the phase's end (one
        // read per block: its warps too).
        if (tid == 0) {
            bool fit = true;
            for (int r = 0; r < 4; ++r) fit = fit && __ldcg(&ctl->join_n[0][r]) <= (unsigned)QcJoin::kCap;
            s_way = *(volatile int*)&ctl->bk_state != 1 ? kPathSort : fit ? kPathQueues : kPathTiles;
        }
        __syncthreads();
        if (s_way == kPathSort || (s_way == kPathQueues && qq >= 4)) return;
    }
    const uint32_t* keys = a.keys;
    const uint64_t* vals = a.vals;
    const unsigned* tbeg = a.tbeg;
    const int *tlen = a.tlen, *cu = a.cu, *cv = a.cv, *ci = a.ci;
    uint64_t* vout = a.vB;
    int* iout = a.cu;
    unsigned* scratch = a.kB;
    const long long n = a.n;
    int32_t* out_idx = a.out_idx;
    int64_t* out_n = a.out_n;
    unsigned pre[5];   // records of the queues before each queue
    pre[0] = 0u;
#pragma unroll
    for (int r = 0; r < 4; ++r) pre[r + 1] = pre[r] + ctl->rec_q[r];
    unsigned long long *src, *dst;
    int len = 0, round = -1;
    if (path == kPathTiles && s_way == kPathTiles) {   // too long for a block each
        bool go = true;
        round = join_rounds(a, *reinterpret_cast<QcQueue*>(s_dyn), pre, &go);
        if (!go && tid == 0) *out_n = CH_ETIMEOUT;
        if (round < 0) return;
    } else if (path == kPathQueues) {
        QcQueue& q = *reinterpret_cast<QcQueue*>(s_dyn);
        const unsigned m = ctl->count;
        qc_gather<T, 4>(keys, vals, m, qq, q, &s_n);
        CH_TL(ctl, 19, 1);
        const int cnt = min(s_n, QcQueue::kCap);   // rec_q[qq], the two end points among them
        const int left = qc_sort<T>(q, cnt, s_m.lo[qq], s_m.hi[qq]);
        CH_TL(ctl, 20, 1);
        src = q.a;
        dst = q.b;
        len = qc_eliminate<T>(src, dst, left, q.tmp);
        for (int j = tid; j < len; j += T) {
            vout[pre[qq] + j] = src[j] >> kQcPosBits;
            iout[pre[qq] + j] = q.si[qc_pos(src[j])];
        }
    } else {
        QcJoin& q = *reinterpret_cast<QcJoin*>(s_dyn);
        const unsigned t0 = *(volatile unsigned*)&ctl->q_tile[qq], nt = *(volatile unsigned*)&ctl->q_tile[qq + 1] - t0;
        constexpr int kE = kPtGroups / T;
        unsigned c[kE], sum = 0u;
#pragma unroll
        for (int e = 0; e < kE; ++e) {
            const unsigned t = tid * kE + e;
            c[e] = t < nt ? (unsigned)__ldcg(tlen + t0 + t) : 0u;
            sum += c[e];
        }
        int tot;
        unsigned run = (unsigned)block_excl_scan((int)sum, q.tmp, &tot);
#pragma unroll
        for (int e = 0; e < kE; ++e) {
            q.off[tid * kE + e] = run;
            run += c[e];
        }
        __syncthreads();
        for (unsigned t = warp; t < nt; t += T / 32) {
            const unsigned o = q.off[t], l = (unsigned)__ldcg(tlen + t0 + t), b = __ldcg(tbeg + t0 + t);
            for (unsigned j = lane; j < l; j += 32) {
                q.a[o + j] = qc_pack((unsigned)__ldcg(cu + b + j), (unsigned)__ldcg(cv + b + j), o + j);
                scratch[pre[qq] + o + j] = (unsigned)__ldcg(ci + b + j);
            }
        }
        __syncthreads();
        CH_TL(ctl, 19, 1);
        src = q.a;
        dst = q.b;
        len = qc_eliminate<T>(src, dst, tot, q.tmp);
        for (int j = tid; j < len; j += T) {
            vout[pre[qq] + j] = src[j] >> kQcPosBits;
            iout[pre[qq] + j] = (int)scratch[pre[qq] + qc_pos(src[j])];
        }
    }
    CH_TL(ctl, 21, 1);
    if (round < 0) {
        if (tid == 0) ctl->reg_end[qq] = (unsigned)len;
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            s_last = atomicAdd(&ctl->joins_done, 1u) == 3u;
            __threadfence();
        }
        __syncthreads();
        if (!s_last) return;
    }
    CH_TL(ctl, 22, 1);
    const unsigned* lens = round < 0 ? ctl->reg_end : ctl->join_n[round + 1];
    const bool spread = round >= 0 && (round & 1);   // in cu, cv, ci
    const int* idx = round < 0 ? iout : spread ? ci : (const int*)a.kB;
    int off[5];
    off[0] = 0;
    for (int r = 0; r < 4; ++r) off[r + 1] = off[r] + max((int)__ldcg(lens + r) - 1, 0);
    auto get = [&](int r, int j, int& pu, int& pv, int& pi) {
        if (spread) {
            pu = __ldcg(cu + pre[r] + j);
            pv = __ldcg(cv + pre[r] + j);
        } else {
            const uint64_t x = __ldcg(vout + pre[r] + j);
            pu = (int)(x >> kKeyBits);
            pv = (int)(x & kKeyMask);
        }
        pi = __ldcg(idx + pre[r] + j);
    };
    if (off[4] > kStitchLong) {
        stitch_long(off, get, n, ctl, out_idx, out_n);
    } else {   // few vertices, or a degenerate cycle: one warp, in shared memory
        int* X = reinterpret_cast<int*>(s_dyn);
        int *Y = X + kStitchLong, *V = Y + kStitchLong, *tmp = V + kStitchLong;
        for (int p = tid; p < off[4]; p += T) {
            const int r = p >= off[2] ? (p >= off[3] ? 3 : 2) : (p >= off[1] ? 1 : 0);
            int pu, pv;
            get(r, p - off[r], pu, pv, V[p]);
            frame_to_xy(r, pu, pv, X[p], Y[p]);
        }
        __syncthreads();
        stitch_cycle(X, Y, V, off[4], tmp, ctl, n, out_idx, out_n);
    }
    if (tid == 0) ctl->done = 1;
    CH_TL(ctl, 13, 1);
}

// ---------------------------------------------------------------------------
void launch_large(Ctl* ctl, const uint32_t* kA, const uint64_t* vA, uint32_t* kB, uint64_t* vB, unsigned* tiles, int* cu,
                  int* cv, int* ci, long long n, int32_t* out_idx, int64_t* out_n, int grid, cudaStream_t s) {
    const LargeArgs a{ctl, kA, vA, kB, vB, tiles, tiles + kPtGroups, tiles + 2 * kPtGroups, tiles + 3 * kPtGroups,
                      {tiles, tiles + kPtGroups}, (int*)(tiles + 4 * kPtGroups), cu, cv, ci, n, out_idx, out_n};
    large_kernel<<<grid, kLargeThreads, kLargeSmem, s>>>(a);
}

size_t tiles_bytes() { return sizeof(unsigned) * 5 * (size_t)kPtGroups; }

cudaError_t configure_large_kernel() {
    return cudaFuncSetAttribute(large_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLargeSmem);
}

}  // namespace ch
