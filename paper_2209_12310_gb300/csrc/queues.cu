// queues.cu -- hull of many survivors without a full sort.
//
// The post pass leaves the records in no order, counted per queue, and picks
// one of three ways (post_last_block):
//   queues  every queue fits one block: queue_kernel, a block per queue, sorts
//           the queue by u and reduces it to its lower chain in shared memory
//           (qchain.cuh);
//   tiles   the u range of each queue is cut into tiles of about kTileTarget
//           records: tile_hist_kernel counts the records of kQGroups equal u
//           ranges per queue and its last block joins neighbouring ranges into
//           tiles; tile_part_kernel moves the records into their tiles' ranges
//           (partition.cuh); tile_chain_kernel reduces each tile to its lower
//           chain by the same block sort and elimination; queue_kernel then
//           reduces each queue's tile chains, joined in u order, to its chain;
//   sort    the radix sort and the merge tree (sort.cu, hull.cu), also when
//           a tile's or a queue's chain outgrows shared memory.
// The lower chain of a set of points equals the lower chain of the chains of
// any partition of it into u ranges, joined in u order.
#include "ch_internal.cuh"
#include "host.h"
#include "hullcore.cuh"
#include "launch.h"
#include "partition.cuh"
#include "qchain.cuh"

namespace ch {

constexpr int kQGroups = 1024;          // equal u ranges of a queue
constexpr unsigned kTileTarget = 1280;  // records of a tile on average: half of what its block holds
constexpr int kTileThreads = 256;
constexpr int kQueueThreads = 1024;
using QcTile = QcSmem<2560, 1024>;
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

// The call takes path p and no earlier stage failed.
__device__ __forceinline__ bool on_path(Ctl* ctl, int p) {
    return *(volatile int*)&ctl->path == p && *(volatile int*)&ctl->bk_state == 1 && read_status(ctl) == CH_OK;
}

// Records per group; the block that finishes last cuts the tiles: gtile maps a
// group to its tile, tile t's records go to [tbeg[t], tbeg[t + 1]).
__global__ void __launch_bounds__(kPtThreads, 1) tile_hist_kernel(Ctl* ctl, const uint32_t* keys, unsigned* ghist,
                                                                  unsigned* gtile, unsigned* tbeg, unsigned* tcur) {
    __shared__ unsigned s_h[kPtGroups];   // records per group; then per tile
    __shared__ unsigned s_beg[kPtGroups];
    __shared__ unsigned s_q0[5], s_tb[5];
    __shared__ QMap s_m;
    __shared__ int s_go, s_last, s_tmp[33];
    const int tid = threadIdx.x;
    if (tid == 0) s_go = on_path(ctl, kPathTiles);
    __syncthreads();
    if (!s_go) return;
    q_map(ctl->oct, s_m);
    for (int g = tid; g < kPtGroups; g += kPtThreads) s_h[g] = 0u;
    __syncthreads();
    const unsigned n = ctl->count;
    const unsigned stride = gridDim.x * kPtThreads;
    constexpr int kU = 4;
    for (unsigned i0 = blockIdx.x * kPtThreads + tid; i0 < n; i0 += stride * kU) {
        uint32_t k[kU];
#pragma unroll
        for (int j = 0; j < kU; ++j)
            if (i0 + j * stride < n) k[j] = __ldcs(keys + i0 + j * stride);
#pragma unroll
        for (int j = 0; j < kU; ++j)
            if (i0 + j * stride < n) atomicAdd(&s_h[q_group(s_m, k[j])], 1u);
    }
    __syncthreads();
    for (int g = tid; g < kPtGroups; g += kPtThreads)
        if (s_h[g]) atomicAdd(&ghist[g], s_h[g]);
    if (!last_block(&ctl->blocks_done[2], &s_last)) return;
    __syncthreads();
    constexpr int kE = kPtGroups / kPtThreads;   // groups per thread, all of one queue
    unsigned c[kE], sum = 0u;
#pragma unroll
    for (int e = 0; e < kE; ++e) {
        c[e] = __ldcg(ghist + tid * kE + e);
        ghist[tid * kE + e] = 0u;   // at rest again
        sum += c[e];
    }
    int tot;
    unsigned run = (unsigned)block_excl_scan((int)sum, s_tmp, &tot);
    if (tid % (kQGroups / kE) == 0) s_q0[tid / (kQGroups / kE)] = run;
    if (tid == 0) s_q0[4] = (unsigned)tot;
    for (int t = tid; t < kPtGroups; t += kPtThreads) {
        s_h[t] = 0u;
        s_beg[t] = 0xFFFFFFFFu;
    }
    __syncthreads();
    const unsigned target = max(kTileTarget, n / (unsigned)(kPtGroups - 96));   // at most kPtGroups - 92 tiles
    if (tid == 0) {
        unsigned t = 0u;
        for (int r = 0; r < 4; ++r) {
            s_tb[r] = t;
            t += (s_q0[r + 1] - s_q0[r]) / target + 1u;
        }
        s_tb[4] = t;
        for (int r = 0; r < 5; ++r) ctl->q_tile[r] = s_tb[r];
    }
    __syncthreads();
    const int r = tid / (kQGroups / kE);
#pragma unroll
    for (int e = 0; e < kE; ++e) {
        const unsigned t = s_tb[r] + (run - s_q0[r]) / target;
        gtile[tid * kE + e] = t;
        if (c[e]) {
            atomicMin(&s_beg[t], run);
            atomicAdd(&s_h[t], c[e]);
        }
        run += c[e];
    }
    __syncthreads();
    for (unsigned t = tid; t < s_tb[4]; t += kPtThreads) {
        const unsigned b = s_h[t] ? s_beg[t] : 0u;   // a tile that a large group skipped is empty
        tbeg[t] = b;
        tcur[t] = b;
    }
}

// Records into their tiles' ranges; tcur[t] ends up at the end of tile t.
struct TilePartSmem {
    PartSmem p;
    unsigned short gtile[kPtGroups];
};

__global__ void __launch_bounds__(kPtThreads, 1) tile_part_kernel(Ctl* ctl, const uint32_t* kin, const uint64_t* vin,
                                                                  const unsigned* gtile, unsigned* tcur,
                                                                  uint32_t* kout, uint64_t* vout) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    TilePartSmem& sm = *reinterpret_cast<TilePartSmem*>(s_dyn);
    __shared__ QMap s_m;
    __shared__ int s_go;
    const int tid = threadIdx.x;
    if (tid == 0) s_go = on_path(ctl, kPathTiles);
    __syncthreads();
    if (!s_go) return;
    q_map(ctl->oct, s_m);
    for (int g = tid; g < kPtGroups; g += kPtThreads) sm.gtile[g] = (unsigned short)gtile[g];
    __syncthreads();
    const unsigned n = ctl->count, nt = ctl->q_tile[4];
    for (unsigned i0 = blockIdx.x * kPtTile; i0 < n; i0 += gridDim.x * kPtTile)
        partition_tile(
            sm.p, kin, vin, i0, min((unsigned)kPtTile, n - i0), nt,
            [&](uint32_t key) { return (unsigned)sm.gtile[q_group(s_m, key)]; },
            [&](unsigned g, unsigned cnt) { return atomicAdd(&tcur[g], cnt); }, kout, vout);
}

// Each tile's lower chain, to [tbeg[t], tbeg[t] + tlen[t]) of cu / cv / ci
// (u, v, index).  A tile with more records than the block holds goes in
// pieces, the chain so far taken along with each; when that chain fills the
// block, the call goes to the sort.
__global__ void __launch_bounds__(kTileThreads) tile_chain_kernel(Ctl* ctl, const uint32_t* keys, const uint64_t* vals,
                                                                  const unsigned* tbeg, const unsigned* tend, int* cu,
                                                                  int* cv, int* ci, int* tlen) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    QcTile& q = *reinterpret_cast<QcTile*>(s_dyn);
    __shared__ int s_go;
    __shared__ unsigned s_tile, s_nt;
    const int tid = threadIdx.x;
    constexpr int kCap = QcTile::kCap, kCarry = kCap * 3 / 4, kPer = kCap / kTileThreads;
    static_assert(kCap % kTileThreads == 0, "carried points per thread");
    if (tid == 0) {
        s_go = on_path(ctl, kPathTiles);
        s_nt = ctl->q_tile[4];
    }
    __syncthreads();
    if (!s_go) return;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_tile = atomicAdd(&ctl->tile_ctr[3], 1u);   // the sort's passes use 0 .. 2
        __syncthreads();
        const unsigned t = s_tile;
        if (t >= s_nt) return;
        const unsigned beg = tbeg[t], cnt = tend[t] - beg;
        unsigned long long *src = q.a, *dst = q.b;
        int len = 0;
        for (unsigned c0 = 0; c0 < cnt;) {
            const int take = (int)min(cnt - c0, (unsigned)(kCap - len));
            if (len) {   // the carried chain first, in slots 0 .. len - 1
                unsigned long long w[kPer];
                int id[kPer];
#pragma unroll
                for (int e = 0; e < kPer; ++e) {
                    const int j = e * kTileThreads + tid;
                    w[e] = j < len ? src[j] : 0ull;
                    id[e] = j < len ? q.si[qc_pos(w[e])] : 0;
                }
                __syncthreads();
#pragma unroll
                for (int e = 0; e < kPer; ++e) {
                    const int j = e * kTileThreads + tid;
                    if (j < len) {
                        q.a[j] = qc_pack((unsigned)qc_u(w[e]), (unsigned)qc_v(w[e]), (unsigned)j);
                        q.si[j] = id[e];
                    }
                }
            }
#pragma unroll 5
            for (int j = tid; j < take; j += kTileThreads) {
                const uint32_t k = __ldcs(keys + beg + c0 + j);
                const uint64_t w = __ldcs(vals + beg + c0 + j);
                q.a[len + j] = qc_pack(k & kKeyMask, (unsigned)(w >> 31), (unsigned)(len + j));
                q.si[len + j] = (int)(w & 0x7FFFFFFFull);
            }
            __syncthreads();
            // the buckets span the points' own range, which is the tile's
            int lo = INT_MAX, hi = INT_MIN;
            for (int j = tid; j < len + take; j += kTileThreads) {
                lo = min(lo, qc_u(q.a[j]));
                hi = max(hi, qc_u(q.a[j]));
            }
            lo = block_reduce<int>(lo, [](int x, int y) { return min(x, y); }, q.tmp);
            hi = block_reduce<int>(hi, [](int x, int y) { return max(x, y); }, q.tmp);
            qc_sort<kTileThreads>(q, len + take, lo, hi);
            src = q.a;
            dst = q.b;
            len = qc_eliminate<kTileThreads>(src, dst, len + take, q.tmp);
            c0 += (unsigned)take;
            if (len > kCarry && c0 < cnt) {   // no room for the rest
                if (tid == 0) ctl->bk_state = 2;
                len = 0;
                break;
            }
        }
        for (int j = tid; j < len; j += kTileThreads) {
            const unsigned long long w = src[j];
            cu[beg + j] = qc_u(w);
            cv[beg + j] = qc_v(w);
            ci[beg + j] = q.si[qc_pos(w)];
        }
        if (tid == 0) tlen[t] = len;
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
constexpr size_t kQueueSmem = sizeof(QcJoin) > sizeof(QcQueue) ? sizeof(QcJoin) : sizeof(QcQueue);
static_assert(kQueueSmem <= 226 * 1024 && QcJoin::kCap < (1 << kQcPosBits), "one block's shared memory");

// Block q: queue q's chain from its records (path queues) or its tiles' chains
// (path tiles), left at the queue's records' place in (vout, iout); the block
// that finishes last joins the four.
__global__ void __launch_bounds__(kQueueThreads, 1) queue_kernel(Ctl* ctl, const uint32_t* keys, const uint64_t* vals,
                                                                 const unsigned* tbeg, const int* tlen, const int* cu,
                                                                 const int* cv, const int* ci, uint64_t* vout,
                                                                 int* iout, unsigned* scratch, long long n,
                                                                 int32_t* out_idx, int64_t* out_n) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ QMap s_m;
    __shared__ int s_path, s_n, s_last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, qq = blockIdx.x;
    constexpr int T = kQueueThreads;
    if (tid == 0) {
        s_path = on_path(ctl, kPathQueues) ? kPathQueues : on_path(ctl, kPathTiles) ? kPathTiles : 0;
        s_n = 0;
    }
    __syncthreads();
    const int path = s_path;
    if (!path) return;
    q_map(ctl->oct, s_m);
    unsigned pre[5];   // records of the queues before each queue
    pre[0] = 0u;
#pragma unroll
    for (int r = 0; r < 4; ++r) pre[r + 1] = pre[r] + ctl->rec_q[r];
    unsigned long long *src, *dst;
    int len = 0;
    bool ok = true;
    if (path == kPathQueues) {
        QcQueue& q = *reinterpret_cast<QcQueue*>(s_dyn);
        const unsigned m = ctl->count;
        constexpr int kU = 4;   // records per thread in flight
        for (unsigned j0 = 0; j0 < m; j0 += T * kU) {
            uint32_t k[kU];
            uint64_t w[kU];
            bool own[kU];
#pragma unroll
            for (int e = 0; e < kU; ++e) {
                const unsigned j = j0 + e * T + tid;
                k[e] = j < m ? __ldcg(keys + j) : 0u;
                own[e] = j < m && (int)(k[e] >> kKeyBits) == qq;
            }
#pragma unroll
            for (int e = 0; e < kU; ++e) w[e] = own[e] ? __ldcg(vals + j0 + e * T + tid) : 0ull;
#pragma unroll
            for (int e = 0; e < kU; ++e) {
                const unsigned bal = __ballot_sync(0xFFFFFFFFu, own[e]);
                if (!bal) continue;
                int pos = 0;
                if (lane == 0) pos = atomicAdd(&s_n, __popc(bal));
                pos = __shfl_sync(0xFFFFFFFFu, pos, 0) + __popc(bal & lanemask_lt());
                if (own[e] && pos < QcQueue::kCap) {
                    q.a[pos] = qc_pack(k[e] & kKeyMask, (unsigned)(w[e] >> 31), (unsigned)pos);
                    q.si[pos] = (int)(w[e] & 0x7FFFFFFFull);
                }
            }
        }
        __syncthreads();
        const int cnt = min(s_n, QcQueue::kCap);   // rec_q[qq], the two end points among them
        qc_sort<T>(q, cnt, s_m.lo[qq], s_m.hi[qq]);
        src = q.a;
        dst = q.b;
        len = qc_eliminate<T>(src, dst, cnt, q.tmp);
        for (int j = tid; j < len; j += T) {
            vout[pre[qq] + j] = src[j] >> kQcPosBits;
            iout[pre[qq] + j] = q.si[qc_pos(src[j])];
        }
    } else {
        QcJoin& q = *reinterpret_cast<QcJoin*>(s_dyn);
        const unsigned t0 = ctl->q_tile[qq], nt = ctl->q_tile[qq + 1] - t0;
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
        ok = tot <= QcJoin::kCap;
        if (ok) {
            for (unsigned t = warp; t < nt; t += T / 32) {
                const unsigned o = q.off[t], l = (unsigned)__ldcg(tlen + t0 + t), b = tbeg[t0 + t];
                for (unsigned j = lane; j < l; j += 32) {
                    q.a[o + j] = qc_pack((unsigned)__ldcg(cu + b + j), (unsigned)__ldcg(cv + b + j), o + j);
                    scratch[pre[qq] + o + j] = (unsigned)__ldcg(ci + b + j);
                }
            }
            __syncthreads();
            src = q.a;
            dst = q.b;
            len = qc_eliminate<T>(src, dst, tot, q.tmp);
            for (int j = tid; j < len; j += T) {
                vout[pre[qq] + j] = src[j] >> kQcPosBits;
                iout[pre[qq] + j] = (int)scratch[pre[qq] + qc_pos(src[j])];
            }
        }
    }
    if (tid == 0) {
        ctl->reg_end[qq] = ok ? (unsigned)len : 0u;
        if (!ok) ctl->bk_state = 2;   // the sort takes over (its input is untouched)
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        s_last = atomicAdd(&ctl->blocks_done[3], 1u) == 3u;
        if (s_last) ctl->blocks_done[3] = 0u;
        __threadfence();
        if (*(volatile int*)&ctl->bk_state != 1) s_last = 0;
    }
    __syncthreads();
    if (!s_last) return;
    int off[5];
    off[0] = 0;
    for (int r = 0; r < 4; ++r) off[r + 1] = off[r] + max((int)__ldcg(&ctl->reg_end[r]) - 1, 0);
    auto get = [&](int r, int j, int& pu, int& pv, int& pi) {
        const uint64_t x = __ldcg(vout + pre[r] + j);
        pu = (int)(x >> kKeyBits);
        pv = (int)(x & kKeyMask);
        pi = __ldcg(iout + pre[r] + j);
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
}

// ---------------------------------------------------------------------------
void launch_tiles(Ctl* ctl, uint32_t* kA, uint64_t* vA, uint32_t* kB, uint64_t* vB, unsigned* tiles, int* cu, int* cv,
                  int* ci, int sms, cudaStream_t s) {
    unsigned *ghist = tiles, *gtile = ghist + kPtGroups, *tbeg = gtile + kPtGroups, *tcur = tbeg + kPtGroups;
    int* tlen = (int*)(tcur + kPtGroups);
    { ProfScope p("bk_hist", s); tile_hist_kernel<<<sms, kPtThreads, 0, s>>>(ctl, kA, ghist, gtile, tbeg, tcur); }
    {
        ProfScope p("bk_part1", s);
        tile_part_kernel<<<sms, kPtThreads, sizeof(TilePartSmem), s>>>(ctl, kA, vA, gtile, tcur, kB, vB);
    }
    {
        ProfScope p("bk_hull", s);
        tile_chain_kernel<<<4 * sms, kTileThreads, sizeof(QcTile), s>>>(ctl, kB, vB, tbeg, tcur, cu, cv, ci, tlen);
    }
}

size_t tiles_bytes() { return sizeof(unsigned) * 5 * (size_t)kPtGroups; }

void launch_queues(Ctl* ctl, const uint32_t* kA, const uint64_t* vA, uint32_t* kB, uint64_t* vB, unsigned* tiles,
                   int* cu, int* cv, int* ci, long long n, int32_t* out_idx, int64_t* out_n, cudaStream_t s) {
    ProfScope p("queues", s);
    unsigned* tbeg = tiles + 2 * kPtGroups;
    // the tile chains are consumed into shared memory and kB before the
    // queue's chain is written to vB and cu (each queue to its own records'
    // place, where only its own tiles' chains lie)
    queue_kernel<<<4, kQueueThreads, kQueueSmem, s>>>(ctl, kA, vA, tbeg, (const int*)(tbeg + 2 * kPtGroups), cu, cv,
                                                      ci, vB, cu, kB, n, out_idx, out_n);
}

cudaError_t configure_queue_kernels() {
    cudaError_t e = cudaFuncSetAttribute(tile_part_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(TilePartSmem));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(tile_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(QcTile));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(queue_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQueueSmem);
}

}  // namespace ch
