// star.cuh -- a star-shaped filter polygon for dense data, and its point tests.
//
// When most points survive the octagon (points near a circle, the worst case
// of Table V), the octagon leaves a rim of width ~0.08 R that holds almost
// every point.  A polygon with thousands of vertices that are input points
// hugs the hull far closer.  It is built from a sample: around a centre c,
// the sample is split into kStarBins angular bins and each bin keeps its point
// farthest from c (dense_kernel); one block then builds the polygon (star_finish):
// it gathers the bins' points, drops reflex vertices, which only enlarges the
// polygon, checks it exactly, and builds the lookup tables of the point tests.
//
// Why dropping points strictly inside it is exact: every vertex is an input
// point, and the polygon is star-shaped around c with every wedge
// (c, V_j, V_j+1) turning counter-clockwise by less than pi and the wedges
// winding once around c (checked exactly).  So it is the union of the
// triangles (c, V_j, V_j+1), each inside the hull of the input; a point in its
// interior is in the interior of the hull, no hull vertex, and so are all its
// duplicates.  The tests below drop a point only when they prove that it lies
// strictly inside; any doubt keeps it.
#pragma once

#include "ch_internal.cuh"

namespace ch {

// The finished polygon:
//   v    vertices relative to c (|.| < 2^24: every orientation is exact in
//        int64), counter-clockwise, the first two repeated after the last;
//   tbl  per bin, the last vertex whose bin comes before it (K - 1 if none);
//   thr  per bin, a bound on the squared distance from c as floats compute it:
//        let r be an integer radius no larger than the distance from c to the
//        line of any edge whose wedge can hold points of the bin (star_window);
//        a point of the bin closer to c than r is strictly inside.
//        thr is r^2 less 5 parts in 2^24, rounded down, and star_d2 is at most
//        2 parts in 2^24 below d^2: star_d2 < thr proves d < r.  (0 when no
//        bound was found.)
struct StarPoly {
    int2 v[kStarBins + 2];
    unsigned short tbl[kStarBins];
    float thr[kStarBins];
};

// Angular bin of an offset (dx, dy) from c (integers below 2^24, exact as
// floats): a pseudo-angle in [0, 4) that grows with the angle (1 - dx / (|dx| +
// |dy|) above, 3 + dx / (|dx| + |dy|) below), scaled to kStarBins bins and
// rounded to the nearest (adding 2^23 leaves the integer in the low bits).
// Float rounding may move a point near a bin boundary to the neighbouring
// bin; no test relies on the bin being right to within one bin.
__device__ __forceinline__ int star_bin(float dx, float dy) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fabsf(dx) + fabsf(dy)));
    const float w = copysignf(fmaf(dx, r, 1.0f), dy);
    return __float_as_int(fmaf(w, -(float)(kStarBins / 4), 8388608.0f + (float)(kStarBins / 2))) & (kStarBins - 1);
}
__device__ __forceinline__ int star_bin(int dx, int dy) { return star_bin((float)dx, (float)dy); }

// Squared distance in floats: two roundings, at most 2 parts in 2^24 low.
__device__ __forceinline__ float star_d2(float dx, float dy) { return fmaf(dx, dx, dy * dy); }

// orient(c, v, p) for v, p given relative to c.
__device__ __forceinline__ long long star_orient_c(int2 v, int px, int py) {
    return (long long)v.x * py - (long long)v.y * px;
}

// Exact test: true only when p = c + (px, py) is strictly inside.  The bin's
// table entry j names the last vertex before the bin; p lies in wedge j
// (V_j, V_j+1) or, when it is past V_j+1, in wedge j+1 (V_j+1's bin may be
// p's own).  The chosen wedge is verified on both spokes, then p must be
// strictly left of the wedge's edge.
__device__ __forceinline__ bool star_inside_exact(int px, int py, int b, const StarPoly& P) {
    const int j = P.tbl[b];
    const int2 a = P.v[j], m = P.v[j + 1], z = P.v[j + 2];
    const bool past_m = star_orient_c(m, px, py) > 0;
    const bool spoke_ok = past_m ? star_orient_c(z, px, py) <= 0 : star_orient_c(a, px, py) >= 0;
    const int2 e0 = past_m ? m : a, e1 = past_m ? z : m;
    const long long side =
        (long long)(e1.x - e0.x) * (py - e0.y) - (long long)(e1.y - e0.y) * (px - e0.x);
    return spoke_ok && side > 0;
}

// Fast test: true when p = c + (dx, dy) lies closer to c than its bin's
// radius bound, hence strictly inside; false says nothing.
__device__ __forceinline__ bool star_inside_fast(float dx, float dy, int b, const StarPoly& P) {
    return star_d2(dx, dy) < P.thr[b];
}

// Full test: the bin's radius bound, then the exact wedge test.
__device__ __forceinline__ bool star_inside(int px, int py, const StarPoly& P) {
    const int b = star_bin(px, py);
    return star_inside_fast((float)px, (float)py, b, P) || star_inside_exact(px, py, b, P);
}

// The largest integer r with r^2 <= o^2 / l2: the distance from c to an edge
// line with orient(c, A, B) = o and |B - A|^2 = l2 (0 < o < 2^50,
// 0 < l2 < 2^52; the distance is below 2^25), rounded down.  A float estimate
// (four roundings of 2^-24 each: off by less than 8) takes one Newton step on
// the exact 128-bit residual, then single steps while they improve it.  Every
// loop is bounded; leaving one early only lowers the result, and 0 means no
// bound.
__device__ __forceinline__ unsigned star_line_radius(long long o, long long l2) {
    typedef unsigned __int128 u128;
    const unsigned long long ul = (unsigned long long)l2;
    const u128 oo = (u128)(unsigned long long)o * (unsigned long long)o;
    const float root = sqrtf((float)l2);
    const float rf = (float)o / root;
    if (rf < 16.0f) return 0u;   // too close to c to be of use
    unsigned long long r = (unsigned long long)rf;
    {
        // residual / (2 r l2), below 10 in magnitude
        const u128 rr = (u128)(r * r) * ul;
        const bool over = rr > oo;
        const u128 e = over ? rr - oo : oo - rr;
        const float ef = fmaf(__ull2float_rn((unsigned long long)(e >> 64)), 18446744073709551616.0f,
                              __ull2float_rn((unsigned long long)e));
        const float step = ef / (2.0f * rf * (float)l2);
        r = over ? r - (unsigned long long)ceilf(step) : r + (unsigned long long)floorf(step);
    }
    for (int it = 0; it < 4 && (u128)(r * r) * ul > oo; ++it) --r;
    if ((u128)(r * r) * ul > oo) return 0u;
    for (int it = 0; it < 4 && (u128)((r + 1ull) * (r + 1ull)) * ul <= oo; ++it) ++r;
    return (unsigned)r;
}

// Bound on star_d2 for radius r (see StarPoly).
__device__ __forceinline__ float star_threshold(unsigned r) {
    return __fmul_rd(__ull2float_rd((unsigned long long)r * r), 1.0f - 5.0f / 16777216.0f);
}

// Block-wide exclusive scan of one count per thread (warp shuffles, then the
// warp totals in s, one word per warp); returns the thread's offset and
// leaves the total in *total.
template <int T>
__device__ __forceinline__ int star_scan(int c, unsigned* s, int* total) {
    constexpr int kWarps = T / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned incl = (unsigned)c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s[warp] = incl;
    __syncthreads();
    unsigned sums = lane < kWarps ? s[lane] : 0u;   // every warp scans the warps' totals
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(0xFFFFFFFFu, sums, o);
        if (lane >= o) sums += u;
    }
    if (threadIdx.x == 31) *total = (int)sums;
    const unsigned before = __shfl_sync(0xFFFFFFFFu, sums, (warp + 31) & 31);
    __syncthreads();
    return (int)((warp ? before : 0u) + incl - (unsigned)c);
}

// A vertex under construction: (dx, dy) relative to c, biased by 2^24 (25 bits
// each), and its bin (13 bits).
static_assert(kStarBins == 1 << 13, "a vertex's bin has 13 bits");
__device__ __forceinline__ unsigned long long star_pack(int dx, int dy, int b) {
    return ((unsigned long long)(unsigned)(dx + kCoordLimit) << 38) |
           ((unsigned long long)(unsigned)(dy + kCoordLimit) << 13) | (unsigned)b;
}
__device__ __forceinline__ int2 star_xy(unsigned long long w) {
    return make_int2((int)(w >> 38) - kCoordLimit, (int)((w >> 13) & 0x1FFFFFFull) - kCoordLimit);
}

// Drops the reflex and flat vertices of the polygon of the n points in src
// (counter-clockwise around c, cyclic), until a round drops none or kStarRounds
// rounds are done; returns the vertices left, src points at them.  A vertex m
// between a and z goes when orient(a, m, z) <= 0 and a and z turn by less than
// pi around c: it then lies in the hull of c, a and z, whatever becomes of a
// and z.  So every thread takes a run of consecutive vertices, with the vertex
// before and the one after it as fixed context, through Andrew's scan, and the
// runs that are left are packed together and cut at other places in the next
// round (qc_eliminate's rounds, cyclic).  Dropping such vertices only enlarges
// the polygon, towards the hull of its points.  Whole block of T threads.
constexpr int kStarRounds = 12;

template <int T>
__device__ int star_eliminate(unsigned long long*& src, unsigned long long*& dst, int n, unsigned* s_scan,
                              int* s_tot) {
    const int tid = threadIdx.x;
    for (int round = 0; round < kStarRounds && n > 3; ++round) {
        const int c = max(5, (n + T - 2) / (T - 1)) | 1;
        const int shift = (round & 1) ? c / 2 : 0;
        const int l0 = tid * c - shift;
        const int lo = max(0, min(n, l0)), hi = max(0, min(n, l0 + c));
        const bool some = lo < hi;
        const int2 left = star_xy(some ? src[lo > 0 ? lo - 1 : n - 1] : 0ull);
        const int2 right = star_xy(some ? src[hi < n ? hi : 0] : 0ull);
        __syncthreads();   // every context is read before the runs are rewritten
        int2 top = left, sec = left;
        int cnt = 0;   // vertices kept: src[lo .. lo + cnt)
        auto pop_before = [&](int2 w) {
            while (cnt > 0) {
                const long long turn =
                    (long long)(top.x - sec.x) * (w.y - sec.y) - (long long)(top.y - sec.y) * (w.x - sec.x);
                if (turn > 0 || star_orient_c(sec, w.x, w.y) <= 0) break;
                --cnt;
                top = sec;
                sec = cnt >= 2 ? star_xy(src[lo + cnt - 2]) : left;
            }
        };
        for (int j = lo; j < hi; ++j) {
            const unsigned long long w = src[j];
            const int2 p = star_xy(w);
            pop_before(p);
            src[lo + cnt] = w;
            ++cnt;
            sec = top;
            top = p;
        }
        if (some) pop_before(right);
        const int off = star_scan<T>(cnt, s_scan, s_tot);
        const int tot = *s_tot;
        __syncthreads();   // read by all before the next scan writes it
        if (tot == n) break;
        for (int j = 0; j < cnt; ++j) dst[off + j] = src[lo + j];
        __syncthreads();
        unsigned long long* t = src;
        src = dst;
        dst = t;
        n = tot;
    }
    return n;
}

// The vertex of bin b: its packed farthest point's index (key, 0 for an empty
// bin) names a point of the input; that point, if it is a valid coordinate and
// falls in that bin again (so every vertex is an input point of this call,
// whatever the bins held), as a word of star_pack, else 0 (no word of a vertex).
__device__ __forceinline__ unsigned long long star_vertex(unsigned long long key, float2 p, int b, int cx, int cy) {
    const int X = __float2int_rn(p.x), Y = __float2int_rn(p.y);
    const bool valid = key != 0ull && __int2float_rn(X) == p.x && __int2float_rn(Y) == p.y &&
                       ((unsigned)(X | Y) >> kCoordBits) == 0u;
    return valid && star_bin(X - cx, Y - cy) == b ? star_pack(X - cx, Y - cy, b) : 0ull;
}
__device__ __forceinline__ float2 star_point(unsigned long long key, const float* __restrict__ pts, long long n) {
    const long long idx = (long long)(unsigned)key;
    return key != 0ull && idx < n ? __ldcg(reinterpret_cast<const float2*>(pts) + idx) : make_float2(-1.0f, -1.0f);
}

// The polygon of the K0 vertices in work (shared memory, in bin order), all T
// threads of the block: star_eliminate, the checks, then v and tbl of P (shared
// memory; its first kStarBins words double as the second work area).  Returns
// its vertices (the same in every thread), or 0 when the checks fail.
template <int T>
__device__ int star_polygon(unsigned long long* work, int K0, StarPoly& P, Ctl* ctl) {
    (void)ctl;   // debug timeline only
    constexpr int kPer = kStarBins / T;
    static_assert(sizeof(P.v) >= sizeof(unsigned long long) * kStarBins, "the second work area fits in the vertices");
    __shared__ unsigned s_scan[T / 32];
    __shared__ int s_K, s_bad, s_cross, s_last[T / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t == 0) { s_bad = 0; s_cross = 0; }
    __syncthreads();
    if (K0 < 3) return 0;
    unsigned long long *src = work, *dst = reinterpret_cast<unsigned long long*>(P.v);
    const int K = star_eliminate<T>(src, dst, K0, s_scan, &s_K);
    CH_TL(ctl, 10, 1);
    if (src != work) {   // the list must sit in work before P is written over it
        for (int i = t; i < K; i += T) work[i] = src[i];
        __syncthreads();
    }
    // every wedge turns counter-clockwise by less than pi, and exactly one edge
    // crosses the ray from c along +x (the wedges wind once)
    int bad = 0, cross = 0;
    for (int j = t; j < K; j += T) {
        const int2 a = star_xy(work[j]), b = star_xy(work[j + 1 == K ? 0 : j + 1]);
        bad |= star_orient_c(a, b.x, b.y) <= 0;
        cross += (a.y < 0 && b.y >= 0) ? 1 : 0;
    }
    if (bad) atomicOr(&s_bad, 1);
    if (cross) atomicAdd(&s_cross, cross);
    __syncthreads();
    const bool ok = K >= 3 && !s_bad && s_cross == 1;
    if (!ok) return 0;
    // the vertices; the bin table by a running maximum over the bins' vertices
    // (thr holds them meanwhile, no vertex as -1)
    int* mark = reinterpret_cast<int*>(P.thr);
    for (int j = t; j < K + 2; j += T) P.v[j] = star_xy(work[j < K ? j : j - K]);
    for (int b = t; b < kStarBins; b += T) mark[b] = -1;
    __syncthreads();
    for (int j = t; j < K; j += T) mark[(int)(work[j] & (kStarBins - 1))] = j;
    __syncthreads();
    {
        int m[kPer], best = -1;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            m[i] = mark[t * kPer + i];
            best = max(best, m[i]);
        }
        int incl = best;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl = max(incl, u);
        }
        if (lane == 31) s_last[warp] = incl;
        int run = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
        if (lane == 0) run = -1;
        __syncthreads();
        for (int w = 0; w < warp; ++w) run = max(run, s_last[w]);
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            P.tbl[t * kPer + i] = (unsigned short)(run < 0 ? K - 1 : run);
            run = max(run, m[i]);
        }
    }
    __syncthreads();
    CH_TL(ctl, 11, 1);
    return K;
}

// The line radius of edge (a, c2), vertices relative to c turning counter-clockwise.
__device__ __forceinline__ unsigned star_edge_radius(int2 a, int2 c2) {
    const long long o = (long long)a.x * c2.y - (long long)a.y * c2.x;   // > 0 (checked)
    const long long dx = (long long)c2.x - a.x, dy = (long long)c2.y - a.y;
    return star_line_radius(o, dx * dx + dy * dy);
}

// The edges whose wedges can hold points of bin b of a polygon of K vertices:
// [first, first + count), cyclic.  A point's or a vertex's computed bin is off
// by far less than a bin at its boundaries, so the last vertex before bin b - 1
// and the first one from bin b + 2 on enclose the bin.
constexpr int kStarWindow = 8;   // edges of a bin's window at most; a longer one gets no bound
template <class Tbl>
__device__ __forceinline__ void star_window(Tbl tbl, int K, int b, int& first, int& count) {
    first = (int)tbl[(b - 1) & (kStarBins - 1)];
    int last = (int)tbl[(b + 2) & (kStarBins - 1)];   // the edge from the last vertex before bin b + 2
    count = (last >= first ? last - first : last - first + K) + 1;
}

// Builds the whole polygon in P (shared memory), all T threads of one block,
// from bins (bins[b]: the packed farthest point of bin b, or 0) around c = (cx,
// cy); work: kStarBins words of shared memory.  Returns the number of points it
// was made of (the same in every thread) when it passed its checks and P is
// ready, else 0; leaves the bins as they are.  With kSharedBins the bins are in
// this block's shared memory and may share their bytes with work: every bin is
// read before the first write to it.
template <int T, bool kSharedBins = false>
__device__ int star_finish(const unsigned long long* bins, const float* __restrict__ pts, long long n, int cx, int cy,
                           unsigned long long* work, StarPoly& P, Ctl* ctl) {
    static_assert(T % 32 == 0 && T >= 256 && T <= 1024, "block size");
    constexpr int kPer = kStarBins / T;   // bins per thread: at most 32
    static_assert(kPer <= 16, "gather registers");
    __shared__ unsigned s_scan2[T / 32];
    __shared__ int s_K0;
    const int t = threadIdx.x;
    // bins [t kPer, (t + 1) kPer): all their keys, then all their points, in
    // flight at once
    unsigned kept = 0u;
    unsigned long long w[kPer];
    {
#pragma unroll
        for (int i = 0; i < kPer; ++i) w[i] = kSharedBins ? bins[t * kPer + i] : __ldcg(bins + t * kPer + i);
        float2 p[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) p[i] = star_point(w[i], pts, n);
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            w[i] = star_vertex(w[i], p[i], t * kPer + i, cx, cy);
            if (w[i]) kept |= 1u << i;
        }
    }
    const int off = star_scan<T>(__popc(kept), s_scan2, &s_K0);
#pragma unroll
    for (int i = 0; i < kPer; ++i)
        if ((kept >> i) & 1u) work[off + __popc(kept & ((1u << i) - 1u))] = w[i];
    __syncthreads();
    CH_TL(ctl, 9, 1);
    const int K0 = s_K0;
    const int K = star_polygon<T>(work, K0, P, ctl);
    if (!K) return 0;
    // each edge's line radius (work is free again), then per bin the smallest
    // of its window
    unsigned* er = reinterpret_cast<unsigned*>(work);
    for (int e = t; e < K; e += T) er[e] = star_edge_radius(P.v[e], P.v[e + 1]);
    __syncthreads();
    CH_TL(ctl, 12, 1);
    for (int b = t; b < kStarBins; b += T) {
        int first, count;
        star_window(P.tbl, K, b, first, count);
        unsigned m = 0u;
        if (count <= kStarWindow) {
            m = er[first];
            for (int k = 1; k < count; ++k) m = min(m, er[first + k < K ? first + k : first + k - K]);
        }
        P.thr[b] = star_threshold(m);
    }
    __syncthreads();
    return K0;
}

}  // namespace ch
