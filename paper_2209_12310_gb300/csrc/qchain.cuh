// qchain.cuh -- a queue's lower chain from its unsorted records by one block:
// a bucket sort by u in shared memory, then elimination rounds; and the stitch
// of four long queue chains.
//
// Elimination: a point on or above the segment between two other input points
// of its queue (one on either side in u) is no strict vertex of the lower
// chain, whatever becomes of those two.  So in one round every thread takes a
// run of consecutive points, with the point before and the point after the run
// as fixed context, and reduces it to the lower chain of the run and its
// context (Andrew's scan, Table I); the runs that are left are packed together
// and the next round cuts them at other places.  A round that removes nothing
// has found every triple of neighbours turning strictly left: the chain is
// convex, hence the lower chain.  Points near the hull (what a star polygon
// leaves of dense data) need a few rounds.  Where long parts of two chains hide
// each other the rounds are bounded by doubling the runs, up to one run that
// holds every point.
//
// This replaces, for queues that fit, a warp's quickhull per bucket of 16
// records and a tree of pairwise merges: those are chains of dependent
// shared-memory searches with a few lanes at work (1.0 + 2.1 ms of a 7.5 ms
// batch of 4096 sets), while a round here is a short scan on every thread.
#pragma once

#include "ch_internal.cuh"
#include "hullcore.cuh"

namespace ch {

// A point of a chain under construction: u, v (25 bits each) and its slot in
// the index array (14 bits).  The words order by (u, v).
constexpr int kQcPosBits = 14;
constexpr unsigned long long kQcPad = ~0ull;   // sorts last; u never has all bits set

__device__ __forceinline__ unsigned long long qc_pack(unsigned u, unsigned v, unsigned pos) {
    return ((unsigned long long)u << (kKeyBits + kQcPosBits)) | ((unsigned long long)v << kQcPosBits) | pos;
}
__device__ __forceinline__ int qc_u(unsigned long long w) { return (int)(w >> (kKeyBits + kQcPosBits)); }
__device__ __forceinline__ int qc_v(unsigned long long w) { return (int)(w >> kQcPosBits) & (int)kKeyMask; }
__device__ __forceinline__ int qc_pos(unsigned long long w) { return (int)(w & ((1ull << kQcPosBits) - 1ull)); }

// CAP points at most (below 2^14), NB buckets at most.
template <int CAP, int NB>
struct QcSmem {
    static_assert(CAP <= (1 << kQcPosBits) - 1 && NB % 32 == 0, "slots and buckets");
    static constexpr int kCap = CAP, kBuckets = NB;
    unsigned long long a[CAP], b[CAP];   // contiguous: the bitonic sort uses both
    int si[CAP];                         // index of the point in slot p
    unsigned cnt[NB];
    int tmp[33];
    int big;
};

// Order by (u, v), then by the lowest index, then by slot (a record can occur
// twice: the two ends of a support line with one survivor).
__device__ __forceinline__ bool qc_less(unsigned long long x, unsigned long long y, const int* si) {
    const unsigned long long kx = x >> kQcPosBits, ky = y >> kQcPosBits;
    if (kx != ky) return kx < ky;
    if (x == kQcPad || y == kQcPad) return false;
    const int ix = si[qc_pos(x)], iy = si[qc_pos(y)];
    return ix != iy ? ix < iy : x < y;
}

// Queue qq's records among keys / vals [0, m) into q.a and q.si, U per thread in
// flight; *s_n (shared, 0 at the call) receives their number (those past q's
// capacity are left out).  Whole block of T threads.  One atomic per warp and
// step: with one per ballot, the block's 32 U on one word took longer than the
// loads (25,000 cycles for 32,000 records).  This and the sort's cheaper ranks:
// the queues of 4096 mixed sets 458 -> 354 us.
template <int T, int U, class Q>
__device__ __forceinline__ void qc_gather(const uint32_t* keys, const uint64_t* vals, unsigned m, int qq, Q& q,
                                          int* s_n) {
    const int tid = threadIdx.x, lane = tid & 31;
    for (unsigned j0 = 0; j0 < m; j0 += T * U) {
        uint32_t k[U];
        uint64_t w[U];
        bool own[U];
#pragma unroll
        for (int e = 0; e < U; ++e) {
            const unsigned j = j0 + e * T + tid;
            k[e] = j < m ? __ldcg(keys + j) : 0u;
            own[e] = j < m && (int)(k[e] >> kKeyBits) == qq;
        }
#pragma unroll
        for (int e = 0; e < U; ++e) w[e] = own[e] ? __ldcg(vals + j0 + e * T + tid) : 0ull;
        int mine = 0;
#pragma unroll
        for (int e = 0; e < U; ++e) mine += __popc(__ballot_sync(0xFFFFFFFFu, own[e]));
        int pos = 0;
        if (lane == 0 && mine) pos = atomicAdd(s_n, mine);
        pos = __shfl_sync(0xFFFFFFFFu, pos, 0);
#pragma unroll
        for (int e = 0; e < U; ++e) {
            const unsigned bal = __ballot_sync(0xFFFFFFFFu, own[e]);
            const int at = pos + __popc(bal & lanemask_lt());
            if (own[e] && at < Q::kCap) {
                q.a[at] = qc_pack(k[e] & kKeyMask, (unsigned)(w[e] >> 31), (unsigned)at);
                q.si[at] = (int)(w[e] & 0x7FFFFFFFull);
            }
            pos += __popc(bal);
        }
    }
    __syncthreads();
}

// Whether point w can still be a strict vertex beside the lower chain of some of
// its queue's points: not when it lies on or above an edge, or above a vertex.  A
// copy of a vertex goes too, its index kept at the vertex if it is lower.
__device__ __forceinline__ bool qc_beside(unsigned long long w, int id, const unsigned long long* chain, int len, int* si) {
    const int u = qc_u(w), v = qc_v(w);
    int lo = 0, hi = len;   // the first vertex with no smaller u
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (qc_u(chain[mid]) < u) lo = mid + 1;
        else hi = mid;
    }
    if (lo == len) return true;
    const unsigned long long c = chain[lo];
    const int cu = qc_u(c), cv = qc_v(c);
    if (cu == u) {
        if (v != cv) return v < cv;
        if (qc_pos(c) == qc_pos(w)) return true;   // the vertex itself
        if (id < si[qc_pos(c)]) atomicMin(&si[qc_pos(c)], id);
        return false;
    }
    if (lo == 0) return true;
    const unsigned long long p = chain[lo - 1];
    return (long long)(cu - qc_u(p)) * (v - qc_v(p)) < (long long)(cv - qc_v(p)) * (u - qc_u(p));
}

// The P words of s in order, P a power of two (a bitonic network).  Whole block.
template <int T>
__device__ __forceinline__ void qc_bitonic(unsigned long long* s, int P, const int* si) {
    for (int k = 2; k <= P; k <<= 1)
        for (int d = k >> 1; d > 0; d >>= 1) {
            for (int i = threadIdx.x; i < P; i += T) {
                const int l = i ^ d;
                if (l > i) {
                    const unsigned long long x = s[i], y = s[l];
                    const bool up = (i & k) == 0;
                    if (up ? qc_less(y, x, si) : qc_less(x, y, si)) {
                        s[i] = y;
                        s[l] = x;
                    }
                }
            }
            __syncthreads();
        }
}

// The lower chain of the n >= 1 points in src, ordered by (u, v), the first of
// equal points with their lowest index:
// returns its length; src points at it (the two buffers change roles).  Of
// points of equal u only the first can be a vertex: the others are skipped
// where they follow it.  Whole block of T threads.  Runs have an odd length,
// so that the lanes of a warp read different banks.
constexpr int kQcRun = 5;      // points of a run at least
constexpr int kQcSteady = 8;   // rounds before the runs grow (twofold every second round)

template <int T>
__device__ int qc_eliminate(unsigned long long*& src, unsigned long long*& dst, int n, int* s_tmp) {
    const int tid = threadIdx.x;
    int least = kQcRun;
    for (int round = 0;; ++round) {
        if (round > kQcSteady && (round & 1) && least < n) least = 2 * least + 1;
        // odd rounds cut half a run later (T - 1 whole runs still hold all points)
        const int c = max(least, (n + T - 2) / (T - 1)) | 1;
        const int shift = (round & 1) ? c / 2 : 0;
        const long long l0 = (long long)tid * c - shift;
        const int lo = (int)max(0ll, min((long long)n, l0)), hi = (int)max(0ll, min((long long)n, l0 + c));
        const bool some = lo < hi, ctx = some && lo > 0, after = some && hi < n;
        const unsigned long long left = ctx ? src[lo - 1] : 0ull, right = after ? src[hi] : 0ull;
        __syncthreads();   // every context is read before the runs are rewritten
        // the stack: the context if there is one, then src[lo .. lo + cnt), the
        // points kept; its top (tu, tv) and the edge that leads there (eu, ev)
        // stay in registers
        int cnt = 0;
        const int below = ctx ? 1 : 0;
        int tu = ctx ? qc_u(left) : -1, tv = qc_v(left), eu = 0, ev = 0;
        auto pop_before = [&](int u, int v) {
            while (cnt + below >= 2 && (long long)eu * (v - tv) <= (long long)ev * (u - tu)) {
                --cnt;
                tu -= eu;
                tv -= ev;
                if (cnt + below >= 2) {   // the edge that leads to the new top
                    const unsigned long long w = cnt >= 2 ? src[lo + cnt - 2] : left;
                    eu = tu - qc_u(w);
                    ev = tv - qc_v(w);
                }
            }
        };
        for (int j = lo; j < hi; ++j) {
            const unsigned long long w = src[j];
            const int u = qc_u(w), v = qc_v(w);
            if (u == tu) continue;
            pop_before(u, v);
            src[lo + cnt] = w;
            ++cnt;
            eu = u - tu;
            ev = v - tv;
            tu = u;
            tv = v;
        }
        if (after && qc_u(right) != tu) pop_before(qc_u(right), qc_v(right));
        int tot;
        const int off = block_excl_scan(cnt, s_tmp, &tot);
        if (tot == n) return n;   // nothing removed: convex
        for (int j = 0; j < cnt; ++j) dst[off + j] = src[lo + j];
        __syncthreads();
        unsigned long long* t = src;
        src = dst;
        dst = t;
        n = tot;
    }
}

// Drops, of the n > kQcSample points of q.a, those that the lower chain of
// kQcSample of them rules out; returns how many are left.  Whole block.
constexpr int kQcSample = 512;

template <int T, class Q>
__device__ __noinline__ int qc_thin(Q& q, int n) {
    static_assert(Q::kCap % T == 0 && Q::kCap >= 2 * kQcSample, "points per thread; the sample and its chain in b");
    constexpr int kPer = Q::kCap / T;
    const int tid = threadIdx.x;
    for (int j = tid; j < kQcSample; j += T) q.b[j] = q.a[(int)((long long)j * n / kQcSample)];
    __syncthreads();
    qc_bitonic<T>(q.b, kQcSample, q.si);
    unsigned long long *src = q.b, *dst = q.b + kQcSample;
    const int len = qc_eliminate<T>(src, dst, kQcSample, q.tmp);
    unsigned long long w[kPer];
    unsigned kept = 0u;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
        const int j = e * T + tid;
        w[e] = j < n ? q.a[j] : 0ull;
        if (j < n && qc_beside(w[e], q.si[qc_pos(w[e])], src, len, q.si)) kept |= 1u << e;
    }
    int tot;
    int at = block_excl_scan(__popc(kept), q.tmp, &tot);   // its barriers: every word is read
#pragma unroll
    for (int e = 0; e < kPer; ++e)
        if ((kept >> e) & 1u) q.a[at++] = w[e];
    __syncthreads();
    return tot;
}

// The n points of q.a (u in [lo, hi]) in order, in place, less some that are no
// vertices; returns how many are left.  Whole block of T threads.  Buckets of
// equal width in u hold about two points each; every point
// counts the points of its bucket before it (independent loads, where an
// insertion sort per bucket is a chain of them: records that a polygon leaves
// can crowd a few buckets by the hundred; by words, not indices: with qc_less this
// loop was 23,000 of the sort's 32,000 cycles for 8000 points).  When some bucket holds more than kQcBucket,
// the points are thinned first (copies of one vertex all share a bucket) and the
// buckets span what is left; still crowded, the whole array goes through a
// bitonic sort.
constexpr unsigned kQcBucket = 512;
static_assert(kQcBucket >= kQcSample, "crowded: more points than the sample");

template <int T, class Q>
__device__ int qc_sort(Q& q, int n, int lo, int hi) {
    const int tid = threadIdx.x;
    int nb;
    float scale;
    auto bucket = [&](unsigned long long w) { return max(0, min(nb - 1, (int)((float)(qc_u(w) - lo) * scale))); };
    for (int turn = 0;; ++turn) {
        nb = min(Q::kBuckets, n / 2 + 1);
        scale = (float)nb / (float)(hi - lo + 1);
        for (int b = tid; b < nb; b += T) q.cnt[b] = 0u;
        if (tid == 0) q.big = 0;
        __syncthreads();
        for (int j = tid; j < n; j += T) atomicAdd(&q.cnt[bucket(q.a[j])], 1u);
        __syncthreads();
        const int per = (nb + T - 1) / T, b0 = min(nb, tid * per), b1 = min(nb, b0 + per);
        unsigned sum = 0u, most = 0u;
        for (int b = b0; b < b1; ++b) {
            sum += q.cnt[b];
            most = max(most, q.cnt[b]);
        }
        if (most > kQcBucket) q.big = 1;
        int tot;
        unsigned run = (unsigned)block_excl_scan((int)sum, q.tmp, &tot);
        if (!q.big) {   // block-uniform: set before the scan's barriers
            for (int b = b0; b < b1; ++b) {
                const unsigned c = q.cnt[b];
                q.cnt[b] = run;
                run += c;
            }
            __syncthreads();
            break;
        }
        __syncthreads();   // read by all before the next turn writes it
        if (turn == 0) {
            n = qc_thin<T>(q, n);
            lo = INT_MAX;
            hi = INT_MIN;
            for (int j = tid; j < n; j += T) {
                lo = min(lo, qc_u(q.a[j]));
                hi = max(hi, qc_u(q.a[j]));
            }
            lo = block_reduce<int>(lo, [](int x, int y) { return min(x, y); }, q.tmp);
            hi = block_reduce<int>(hi, [](int x, int y) { return max(x, y); }, q.tmp);
            continue;
        }
        int P = 1;
        while (P < n) P <<= 1;   // n <= CAP < 2^14 <= 2 CAP words in a and b
        for (int j = n + tid; j < P; j += T) q.a[j] = kQcPad;
        __syncthreads();
        qc_bitonic<T>(q.a, P, q.si);
        return n;
    }
    for (int j = tid; j < n; j += T) {
        const unsigned long long w = q.a[j];
        q.b[atomicAdd(&q.cnt[bucket(w)], 1u)] = w;
    }
    __syncthreads();
    for (int j = tid; j < n; j += T) {
        const unsigned long long w = q.b[j];
        const int b = bucket(w);   // cnt[b] is now the end of bucket b
        const int s = b ? (int)q.cnt[b - 1] : 0, e = (int)q.cnt[b];
        int r = s, same = 0;   // same: points of equal (u, v), this one among them
        for (int i = s; i < e; ++i) {
            const unsigned long long x = q.b[i];
            r += x < w ? 1 : 0;
            same += ((x ^ w) >> kQcPosBits) == 0ull ? 1 : 0;
        }
        if (same > 1) {   // the first of them, which can be a vertex, takes the lowest index
            unsigned long long first = w;
            for (int i = s; i < e; ++i) {
                const unsigned long long x = q.b[i];
                if (((x ^ w) >> kQcPosBits) == 0ull && x < first) first = x;
            }
            if (first != w) atomicMin(&q.si[qc_pos(first)], q.si[qc_pos(w)]);
        }
        q.a[r] = w;
    }
    __syncthreads();
    return n;
}

// ---------------------------------------------------------------------------
// Joins four queue chains into the output: the cycle of the chains without
// their last points, off[q] the position of queue q's first point, m = off[4]
// > kStitchLong in all; get(q, j, u, v, i) reads point j of chain q.  Each
// chain is strictly convex and the cycle has an area (a degenerate input's
// chains have two points at most), so only the chains' first points can fail
// to be strict vertices, and the lexicographically smallest vertex is the
// first or the second of queue 0 (W, or the lower end of the line x = xmin).
// So each position's place in the output follows from the at most four
// positions dropped: one pass, no scan.  Whole block.
constexpr int kStitchLong = 64;

template <class Get>
__device__ void stitch_long(const int (&off)[5], Get get, long long n, Ctl* ctl, int32_t* out_idx, int64_t* out_n) {
    __shared__ int s_drop[4], s_bad, s_start;
    const int tid = threadIdx.x, m = off[4];
    auto locate = [&](int p, int& q, int& j) {
        q = p >= off[2] ? (p >= off[3] ? 3 : 2) : (p >= off[1] ? 1 : 0);
        j = p - off[q];
    };
    auto xy = [&](int p, long long& x, long long& y) {
        int q, j, u, v, i, X, Y;
        locate(p, q, j);
        get(q, j, u, v, i);
        frame_to_xy(q, u, v, X, Y);
        x = X;
        y = Y;
    };
    if (tid == 0) s_bad = 0;
    __syncthreads();
    if (tid < 4) {
        s_drop[tid] = INT_MAX;
        const int p = off[tid];
        if (off[tid + 1] > p) {   // queue tid has a point in the cycle
            long long ax, ay, bx, by, cx, cy;
            xy(p == 0 ? m - 1 : p - 1, ax, ay);
            xy(p, bx, by);
            xy(p + 1 == m ? 0 : p + 1, cx, cy);
            const long long tr = orient64(ax, ay, bx, by, cx, cy);
            if (tr < 0) s_bad = 1;   // internal consistency check
            if (tr <= 0) s_drop[tid] = p;
        }
    }
    __syncthreads();
    const int d0 = s_drop[0], d1 = s_drop[1], d2 = s_drop[2], d3 = s_drop[3];
    auto dropped_before = [&](int p) { return (d0 < p) + (d1 < p) + (d2 < p) + (d3 < p); };
    auto dropped = [&](int p) { return p == d0 || p == d1 || p == d2 || p == d3; };
    const int h = m - dropped_before(INT_MAX);
    if (tid == 0) {
        unsigned long long best = ~0ull;
        int start = 0;
        for (int e = -2; e < 4; ++e) {
            const int p = e < 0 ? m + e : e;
            if (dropped(p)) continue;
            long long x, y;
            xy(p, x, y);
            const unsigned long long k = xy_key(x, y);
            if (k < best) {
                best = k;
                start = p - dropped_before(p);
            }
        }
        s_start = start;
        if (s_bad || h > n) set_status(ctl, CH_ECUDA);
    }
    __syncthreads();
    if (h > n) {   // cannot happen for a correct hull; never write past out_idx
        if (tid == 0) *out_n = CH_ECUDA;
        return;
    }
    const int start = s_start;
    for (int p = tid; p < m; p += blockDim.x) {
        if (dropped(p)) continue;
        int q, j, u, v, i;
        locate(p, q, j);
        get(q, j, u, v, i);
        const int r = p - dropped_before(p) - start;
        out_idx[r < 0 ? r + h : r] = i;
    }
    if (tid == 0) {
        const int st = read_status(ctl);
        *out_n = st == CH_OK ? (int64_t)h : (int64_t)st;
    }
}

}  // namespace ch
