// api.cu -- C ABI entry points (ch.h): argument checks, workspace management,
// launch sequences and device-timed kernel statistics.
#include "ch_internal.cuh"
#include "launch.h"
#include "host.h"

#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

namespace ch {

// ---------------------------------------------------------------------------
// Device information (SM count, resident blocks per SM of every kernel).
struct DevInfo {
    int sms = 0;
    int occ_main = 1, occ_post = 1, occ_lab = 1, occ_sort = 1;
};

static std::mutex g_mu;
static std::map<int, DevInfo> g_dev;

static int device_info(int dev, DevInfo* out) {
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_dev.find(dev);
    if (it != g_dev.end()) { *out = it->second; return CH_OK; }
    DevInfo di;
    if (cudaDeviceGetAttribute(&di.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return CH_ECUDA;
    if (configure_hull_kernels() != cudaSuccess) return CH_ECUDA;
    if (configure_filter_kernels() != cudaSuccess) return CH_ECUDA;
    if (configure_post_kernel() != cudaSuccess) return CH_ECUDA;
    if (configure_large_kernel() != cudaSuccess) return CH_ECUDA;
    if (occupancy_filter(&di.occ_main, &di.occ_lab) != cudaSuccess) return CH_ECUDA;
    if (occupancy_post(&di.occ_post) != cudaSuccess) return CH_ECUDA;
    if (occupancy_sort(&di.occ_sort) != cudaSuccess) return CH_ECUDA;
    di.occ_main = std::max(1, di.occ_main);
    di.occ_post = std::max(1, di.occ_post);
    di.occ_lab = std::max(1, di.occ_lab);
    di.occ_sort = std::max(1, di.occ_sort);
    g_dev[dev] = di;
    *out = di;
    return CH_OK;
}

// ---------------------------------------------------------------------------
// Workspace layout for one hull of up to n points.
static size_t align_up(size_t x, size_t a = 256) { return (x + a - 1) / a * a; }

Layout make_layout(long long n) {
    Layout L{};
    L.cap = n + 16;
    L.sort_tiles = (L.cap + kSortTile - 1) / kSortTile;
    L.ctcap = (L.cap + kChainTile - 1) / kChainTile + 4;   // chain tiles of the sorted records
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t r = o;
        o = align_up(o + bytes);
        return r;
    };
    // zeroed at allocation: the control block, the sort's look-back status
    // words and the merge tree's arrival counters (each kernel leaves them in that
    // state for the next call)
    L.off_ctl = take(sizeof(Ctl));
    L.off_status = take(8 * (size_t)kDigits * L.sort_tiles);
    L.off_counters = take(4 * (size_t)kMaxLevels * L.ctcap);
    L.zero_bytes = o;
    L.off_tiles = take(tiles_bytes());
    // inputs that dense_kernel can take (device-independent: at most kStarBlocks
    // blocks of it run)
    const bool star = n / kWarpTilePts >= kStarMinTiles;
    L.off_star_poly = take(star ? star_poly_bytes() : 0);
    L.off_kA = take(4 * (size_t)L.cap);
    L.off_kB = take(4 * (size_t)L.cap);
    L.off_vA = take(8 * (size_t)L.cap);
    L.off_vB = take(8 * (size_t)L.cap);
    L.off_cu = take(4 * (size_t)L.ctcap * kChainTile);
    L.off_cv = take(4 * (size_t)L.ctcap * kChainTile);
    L.off_ci = take(4 * (size_t)L.ctcap * kChainTile);
    // dense_kernel's bins, done with before the first chain is stored
    L.off_star_bins = L.off_cu;
    if (star) o = std::max(o, align_up(L.off_cu + star_bins_bytes(kStarBlocks)));
    L.off_clen = take(4 * (size_t)L.ctcap);
    L.total = o;
    return L;
}

struct Workspace {
    char* base = nullptr;
    size_t bytes = 0;
    long long n_cap = -1;
    // staging for the host-buffer entry point
    char* stage = nullptr;
    size_t stage_bytes = 0;
};

static std::map<std::pair<int, cudaStream_t>, Workspace> g_ws;

void drop_graphs(int dev, cudaStream_t s);

static int grow_workspace(Workspace& ws, long long n, cudaStream_t s, int dev) {
    if (n <= ws.n_cap) return CH_OK;
    drop_graphs(dev, s);
    const long long want = std::max(n, (long long)(ws.n_cap > 0 ? ws.n_cap + ws.n_cap / 4 : n));
    const Layout L = make_layout(want);
    if (ws.base) {
        cudaStreamSynchronize(s);
        cudaFree(ws.base);
        ws.base = nullptr;
        ws.bytes = 0;
        ws.n_cap = -1;
    }
    void* p = nullptr;
    if (cudaMalloc(&p, L.total) != cudaSuccess) {
        cudaGetLastError();
        return CH_ENOMEM;
    }
    if (cudaMemsetAsync(p, 0, L.zero_bytes, s) != cudaSuccess) {
        cudaFree(p);
        return CH_ECUDA;
    }
    ws.base = (char*)p;
    ws.bytes = L.total;
    ws.n_cap = want;
    return CH_OK;
}

int get_workspace(int dev, cudaStream_t s, long long n, char** base, Layout* L) {
    std::lock_guard<std::mutex> lk(g_mu);
    Workspace& ws = g_ws[std::make_pair(dev, s)];
    const int st = grow_workspace(ws, n, s, dev);
    if (st != CH_OK) return st;
    *base = ws.base;
    *L = make_layout(ws.n_cap);
    return CH_OK;
}

static void free_workspace(Workspace& w, cudaStream_t s) {
    cudaStreamSynchronize(s);
    if (w.base) cudaFree(w.base);
    if (w.stage) cudaFree(w.stage);
    w = Workspace();
}

void release_stream_workspace(int dev, cudaStream_t s) {
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_ws.find(std::make_pair(dev, s));
    drop_batched_graphs(dev, s);
    release_batched_stream(dev, s);
    if (it == g_ws.end()) return;
    drop_graphs(dev, s);
    free_workspace(it->second, s);
    g_ws.erase(it);
}

static int get_stage(int dev, cudaStream_t s, size_t bytes, char** out) {
    std::lock_guard<std::mutex> lk(g_mu);
    Workspace& ws = g_ws[std::make_pair(dev, s)];
    if (ws.stage_bytes < bytes) {
        if (ws.stage) {
            cudaStreamSynchronize(s);
            cudaFree(ws.stage);
            ws.stage = nullptr;
            ws.stage_bytes = 0;
        }
        void* p = nullptr;
        const size_t want = std::max(bytes, ws.stage_bytes + ws.stage_bytes / 4);
        if (cudaMalloc(&p, want) != cudaSuccess) {
            cudaGetLastError();
            return CH_ENOMEM;
        }
        ws.stage = (char*)p;
        ws.stage_bytes = want;
    }
    *out = ws.stage;
    return CH_OK;
}

// ---------------------------------------------------------------------------
// Device-timed statistics: CUDA events recorded on the launching stream.
struct ProfPending {
    const char* name;
    cudaEvent_t a, b;
};
static bool g_prof = false;
static std::mutex g_prof_mu;
static std::vector<ProfPending> g_pending;
static std::vector<cudaEvent_t> g_event_pool;
static std::map<std::string, std::pair<long long, double>> g_acc;
static std::vector<std::string> g_names;   // stable storage for names returned to callers

bool prof_enabled() { return g_prof; }

static cudaEvent_t take_event() {
    if (!g_event_pool.empty()) {
        cudaEvent_t e = g_event_pool.back();
        g_event_pool.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
}

ProfScope::ProfScope(const char* name, cudaStream_t s) : name_(name), s_(s), a_(nullptr) {
    if (!g_prof) return;
    std::lock_guard<std::mutex> lk(g_prof_mu);
    a_ = take_event();
    cudaEventRecord((cudaEvent_t)a_, s_);
}

ProfScope::~ProfScope() {
    if (!a_) return;
    std::lock_guard<std::mutex> lk(g_prof_mu);
    cudaEvent_t b = take_event();
    cudaEventRecord(b, s_);
    g_pending.push_back(ProfPending{name_, (cudaEvent_t)a_, b});
}

static void prof_drain() {
    for (auto& p : g_pending) {
        cudaEventSynchronize(p.b);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, p.a, p.b);
        auto& acc = g_acc[p.name];
        acc.first += 1;
        acc.second += ms;
        g_event_pool.push_back(p.a);
        g_event_pool.push_back(p.b);
    }
    g_pending.clear();
}

// ---------------------------------------------------------------------------
// The launch sequence of one hull (n >= 1) on an allocated workspace: one chain
// of kernels, each of which returns at once when the call does not need it (the
// dense part on sparse data, the main pass on dense data, the large-survivor
// paths not taken).  What a call may need beyond the sparse path is packed in
// three kernels whose blocks wait for one another inside: an empty launch costs
// about 2 us, and a conditional graph node about 7 (measured on 65,537 points:
// 50 us a call with one such node, 57 with two).
static int enqueue_hull_direct(const float* pts, long long n, int32_t* out_idx, int64_t* out_n, cudaStream_t s,
                               int dev, char* base, const Layout& L) {
    DevInfo di;
    const int st = device_info(dev, &di);
    if (st != CH_OK) return st;
    Ctl* ctl = (Ctl*)(base + L.off_ctl);
    uint32_t *kA = (uint32_t*)(base + L.off_kA), *kB = (uint32_t*)(base + L.off_kB);
    uint64_t *vA = (uint64_t*)(base + L.off_vA), *vB = (uint64_t*)(base + L.off_vB);
    unsigned* tiles = (unsigned*)(base + L.off_tiles);
    const int head = ((uintptr_t)pts & 15u) != 0u ? 1 : 0;
    const long long ntiles = (n - head) / kWarpTilePts;
    const long long samples = sample_tiles_host(ntiles);
    const int grid_sample = (int)std::max<long long>(1, std::min<long long>(256, (samples + 7) / 8));
    // Raw survivors live in the B buffers until the post pass has turned them
    // into sort records in the A buffers.
    const unsigned switch_at = (unsigned)std::max<long long>(1 << 16, n >> 5);
    const bool dense = ntiles >= kStarMinTiles && n > kSmallMax;   // large enough for a star polygon
    // Inputs that stay in L2 take two passes: the extremes, then the filter
    // against their octagon.  Larger ones take one, with a sample's octagon.
    const bool two_pass = n <= kTwoPassMax;
    const bool one_block = n <= kSmallMax;   // one block does it all up to the large-survivor paths
    if (one_block) {
        ProfScope p("small", s);
        launch_small(pts, n, ctl, kA, vA, out_idx, out_n, s);
    } else if (two_pass) {
        { ProfScope p("init", s); launch_init(ctl, 1, s); }
        ProfScope p("main_filter", s);
        launch_main(pts, n, head, ntiles, ctl, nullptr, nullptr, switch_at, kA, vA, 1, di.sms * di.occ_main, s);
    } else {
        ProfScope p("sample", s);
        launch_sample(pts, n, head, ntiles, ctl, dense ? switch_at : 0xFFFFFFFFu, grid_sample, s);
    }
    if (dense) {
        ProfScope p("dense_filter", s);
        launch_dense(pts, n, head, ntiles, ctl, base + L.off_star_bins, base + L.off_star_poly, vB, kB, kA, vA,
                     std::min(di.sms, kStarBlocks), s);
    }
    if (!two_pass) {
        ProfScope p("main_filter", s);
        launch_main(pts, n, head, ntiles, ctl, vB, kB, switch_at, kA, vA, 0, di.sms * di.occ_main, s);
    }
    if (!one_block) {
        ProfScope p("post", s);
        launch_post(pts, n, head, ntiles, ctl, vB, kB, kA, vA, tiles, out_idx, out_n, di.sms * di.occ_post, s);
    }
    int *cu = (int*)(base + L.off_cu), *cv = (int*)(base + L.off_cv), *ci = (int*)(base + L.off_ci);
    const bool large = n + 16 > kQueueCap;   // else every queue fits a block
    {
        ProfScope p("large", s);
        launch_large(ctl, kA, vA, kB, vB, tiles, cu, cv, ci, n, out_idx, out_n, large ? di.sms : 4, s);
    }
    if (large) {
        ProfScope p("sort", s);
        launch_sort(ctl, kA, vA, kB, vB, (unsigned long long*)(base + L.off_status), cu, cv, ci,
                    (int*)(base + L.off_clen), (int*)(base + L.off_counters), (int)L.ctcap, pts, n, out_idx, out_n,
                    di.sms * di.occ_sort, s);
    }
    return cudaGetLastError() == cudaSuccess ? CH_OK : CH_ECUDA;
}

// ---------------------------------------------------------------------------
// CUDA-graph cache.  A call repeated with the same (device, stream, points,
// n, outputs, workspace) replays one captured graph instead of separate
// launches.  The first call of a key runs directly; the second captures the
// sequence on a private stream and instantiates it; later ones replay it.
// Disabled while profiling (per-kernel events) and when the caller's stream
// is itself being captured (the launches then become part of that graph).
struct GraphKey {
    int dev;
    cudaStream_t s;
    const void* pts;
    long long n;
    const void* out_idx;
    const void* out_n;
    const void* ws;
    bool operator<(const GraphKey& o) const {
        if (dev != o.dev) return dev < o.dev;
        if (s != o.s) return s < o.s;
        if (pts != o.pts) return pts < o.pts;
        if (n != o.n) return n < o.n;
        if (out_idx != o.out_idx) return out_idx < o.out_idx;
        if (out_n != o.out_n) return out_n < o.out_n;
        return ws < o.ws;
    }
};
struct GraphEntry {
    cudaGraphExec_t exec = nullptr;
    int seen = 0;
    unsigned long long last_use = 0;
};
static std::mutex g_graph_mu;
static std::map<GraphKey, GraphEntry> g_graphs;
static unsigned long long g_graph_clock = 0;
static constexpr size_t kGraphCacheMax = 64;

static void drop_graphs_locked(int dev, cudaStream_t s) {
    for (auto it = g_graphs.begin(); it != g_graphs.end();) {
        if (it->first.dev == dev && it->first.s == s) {
            if (it->second.exec) cudaGraphExecDestroy(it->second.exec);
            it = g_graphs.erase(it);
        } else {
            ++it;
        }
    }
}

void drop_graphs(int dev, cudaStream_t s) {
    std::lock_guard<std::mutex> lk(g_graph_mu);
    drop_graphs_locked(dev, s);
}

int enqueue_hull_nograph(const float* pts, long long n, int32_t* out_idx, int64_t* out_n, cudaStream_t s,
                         int dev) {
    char* base = nullptr;
    Layout L;
    const int st = get_workspace(dev, s, n, &base, &L);
    if (st != CH_OK) return st;
    return enqueue_hull_direct(pts, n, out_idx, out_n, s, dev, base, L);
}

int enqueue_hull(const float* pts, long long n, int32_t* out_idx, int64_t* out_n, cudaStream_t s, int dev) {
    DevInfo di;
    int st = device_info(dev, &di);
    if (st != CH_OK) return st;
    // The workspace must exist (and keep its address) before a graph names it.
    char* base = nullptr;
    Layout L;
    st = get_workspace(dev, s, n, &base, &L);
    if (st != CH_OK) return st;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (g_prof || cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone)
        return enqueue_hull_direct(pts, n, out_idx, out_n, s, dev, base, L);
    const GraphKey key{dev, s, pts, n, out_idx, out_n, base};
    cudaGraphExec_t exec = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_graph_mu);
        GraphEntry& e = g_graphs[key];
        e.last_use = ++g_graph_clock;
        if (e.exec) exec = e.exec;
        else if (e.seen++ == 0) return enqueue_hull_direct(pts, n, out_idx, out_n, s, dev, base, L);
    }
    if (exec) return cudaGraphLaunch(exec, s) == cudaSuccess ? CH_OK : CH_ECUDA;
    // Second call of this key: capture on a private stream, then replay.
    cudaStream_t cs = nullptr;
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
        cudaGetLastError();
        return enqueue_hull_direct(pts, n, out_idx, out_n, s, dev, base, L);
    }
    cudaGraph_t graph = nullptr;
    bool ok = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
        st = enqueue_hull_direct(pts, n, out_idx, out_n, cs, dev, base, L);
        ok = cudaStreamEndCapture(cs, &graph) == cudaSuccess && st == CH_OK && graph;
    }
    if (ok) ok = cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess;
    if (graph) cudaGraphDestroy(graph);
    cudaStreamDestroy(cs);
    if (!ok) {
        cudaGetLastError();
        return enqueue_hull_direct(pts, n, out_idx, out_n, s, dev, base, L);
    }
    {
        std::lock_guard<std::mutex> lk(g_graph_mu);
        if (g_graphs.size() > kGraphCacheMax) {   // evict the least recently used entry
            auto victim = g_graphs.begin();
            for (auto it = g_graphs.begin(); it != g_graphs.end(); ++it)
                if (it->second.last_use < victim->second.last_use) victim = it;
            if (victim->second.exec) cudaGraphExecDestroy(victim->second.exec);
            g_graphs.erase(victim);
        }
        g_graphs[key].exec = exec;
    }
    return cudaGraphLaunch(exec, s) == cudaSuccess ? CH_OK : CH_ECUDA;
}

int check_points_args(const float* pts, long long n) {
    if (n < 0 || n > CH_MAX_POINTS) return CH_EINVAL;
    if (n > 0 && !pts) return CH_EINVAL;
    if (((uintptr_t)pts & 7u) != 0u) return CH_EINVAL;
    return CH_OK;
}

}  // namespace ch

using namespace ch;

extern "C" {

int ch_hull(const float* pts, int64_t n, int32_t* out_idx, int64_t* out_n, void* stream) {
    int st = check_points_args(pts, n);
    if (st != CH_OK) return st;
    if (!out_n || (n > 0 && !out_idx)) return CH_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    if (n == 0) return cudaMemsetAsync(out_n, 0, sizeof(int64_t), s) == cudaSuccess ? CH_OK : CH_ECUDA;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return CH_ECUDA;
    return enqueue_hull(pts, n, out_idx, out_n, s, dev);
}

int ch_filter(const float* pts, int64_t n, int32_t* out_ext8, uint8_t* out_labels, int64_t* out_counts4,
              void* stream) {
    int st = check_points_args(pts, n);
    if (st != CH_OK) return st;
    if (!out_ext8) return CH_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    if (n == 0) {
        if (cudaMemsetAsync(out_ext8, 0xFF, 8 * sizeof(int32_t), s) != cudaSuccess) return CH_ECUDA;
        if (out_counts4 && cudaMemsetAsync(out_counts4, 0, 4 * sizeof(int64_t), s) != cudaSuccess)
            return CH_ECUDA;
        return CH_OK;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return CH_ECUDA;
    DevInfo di;
    if ((st = device_info(dev, &di)) != CH_OK) return st;
    char* base = nullptr;
    Layout L;
    if ((st = get_workspace(dev, s, n, &base, &L)) != CH_OK) return st;
    Ctl* ctl = (Ctl*)(base + L.off_ctl);
    const int head = (((uintptr_t)pts & 15u) != 0u) ? 1 : 0;
    const long long ntiles = (n - head) / kWarpTilePts;
    uint32_t* kA = (uint32_t*)(base + L.off_kA);
    uint64_t* vA = (uint64_t*)(base + L.off_vA);
    uint32_t* kB = (uint32_t*)(base + L.off_kB);
    uint64_t* vB = (uint64_t*)(base + L.off_vB);
    const bool lab = out_labels || out_counts4;
    // One read of the points, which finds those of a region inside a sample's
    // octagon (label 0) and leaves the others for labels_kernel; inputs that stay
    // in L2, or want no labels: the extremes first.
    const bool fused = lab && n > kFilterTwoPassMax;
    const unsigned switch_at = fused ? (unsigned)(n >> 5) : 0xFFFFFFFFu;
    if (fused) {
        ProfScope p("sample", s);
        const int grid = (int)std::min<long long>(256, (sample_tiles_host(ntiles) + 7) / 8);
        launch_sample(pts, n, head, ntiles, ctl, switch_at, grid, s, 1);
    } else {
        ProfScope p("init", s);
        launch_init(ctl, 1, s);
    }
    {
        ProfScope p("main_filter", s);
        launch_main_labels(pts, n, head, ntiles, ctl, vB, kB, switch_at, kA, vA, lab && n <= kFilterKeepMax,
                           di.sms * di.occ_main, s);
    }
    if (lab) {
        ProfScope p("labels", s);
        launch_labels(pts, n, head, ntiles, ctl, vB, kB, out_labels, di.sms * di.occ_lab, s);
    }
    launch_filter_output(ctl, n, out_ext8, out_counts4, s);
    return cudaGetLastError() == cudaSuccess ? CH_OK : CH_ECUDA;
}

int ch_hull_host(const float* pts, int64_t n, int32_t* out_idx, int64_t* out_n, void* stream) {
    int st = check_points_args(pts, n);
    if (st != CH_OK) return st;
    if (!out_n || (n > 0 && !out_idx)) return CH_EINVAL;
    if (n == 0) { *out_n = 0; return CH_OK; }
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return CH_ECUDA;
    const size_t pts_bytes = align_up(8 * (size_t)n), idx_bytes = align_up(4 * (size_t)n);
    char* stage = nullptr;
    if ((st = get_stage(dev, s, pts_bytes + idx_bytes + 256, &stage)) != CH_OK) return st;
    float* dpts = (float*)stage;
    int32_t* didx = (int32_t*)(stage + pts_bytes);
    int64_t* dn = (int64_t*)(stage + pts_bytes + idx_bytes);
    if (cudaMemcpyAsync(dpts, pts, 8 * (size_t)n, cudaMemcpyHostToDevice, s) != cudaSuccess) return CH_ECUDA;
    if ((st = enqueue_hull(dpts, n, didx, dn, s, dev)) != CH_OK) return st;
    int64_t h = 0;
    if (cudaMemcpyAsync(&h, dn, sizeof(int64_t), cudaMemcpyDeviceToHost, s) != cudaSuccess) return CH_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return CH_ECUDA;
    *out_n = h;
    if (h > 0) {
        if (cudaMemcpyAsync(out_idx, didx, 4 * (size_t)h, cudaMemcpyDeviceToHost, s) != cudaSuccess)
            return CH_ECUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess) return CH_ECUDA;
    }
    return CH_OK;
}

int ch_reserve(int64_t n, int32_t k, void* stream) {
    if (n < 0 || k < 0) return CH_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return CH_ECUDA;
    DevInfo di;
    int st = device_info(dev, &di);
    if (st != CH_OK) return st;
    char* base;
    Layout L;
    st = get_workspace(dev, (cudaStream_t)stream, std::max<int64_t>(n, 1), &base, &L);
    if (st != CH_OK) return st;
    return reserve_batched(dev, (cudaStream_t)stream, n, k);
}

size_t ch_workspace_bytes(int64_t n) { return n < 0 ? 0 : make_layout(n).total; }

int ch_hull_counters(void* stream, int64_t* out, int cap) {
    if (!out || cap < 0) return CH_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return CH_ECUDA;
    char* base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        auto it = g_ws.find(std::make_pair(dev, s));
        if (it == g_ws.end() || !it->second.base) return CH_EINVAL;
        base = it->second.base;
    }
    Ctl c;
    if (cudaMemcpyAsync(&c, base, sizeof(Ctl), cudaMemcpyDeviceToHost, s) != cudaSuccess) return CH_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return CH_ECUDA;
    const int64_t v[] = {
        (int64_t)c.count_raw,
        (int64_t)c.count,
        (int64_t)(c.mode || c.star_final),
        (int64_t)(c.bk_state == 2 ? 2 : c.bk_state == 1 ? 1 : 0),
        (int64_t)c.status,
        (int64_t)(c.star_final ? c.star_k : 0),
    };
    const int nv = (int)(sizeof(v) / sizeof(v[0]));
    for (int i = 0; i < nv && i < cap; ++i) out[i] = v[i];
    return nv;
}

#if defined(CH_TRACE) || defined(CH_TIMELINE)
// Debug builds: the phase timeline of the most recent call on the first
// workspace (%globaltimer ns; 24 phases, first start and last end of each).
int ch_trace_timeline(unsigned long long* out48) {
    std::lock_guard<std::mutex> lk(g_mu);
    if (g_ws.empty() || !g_ws.begin()->second.base) return CH_EINVAL;
    Ctl c;
    if (cudaMemcpy(&c, g_ws.begin()->second.base, sizeof(Ctl), cudaMemcpyDeviceToHost) != cudaSuccess) return CH_ECUDA;
    for (int i = 0; i < 24; ++i) {
        out48[2 * i] = c.tl[i][0];
        out48[2 * i + 1] = c.tl[i][1];
    }
    return CH_OK;
}
#endif

int ch_release(void) {
    {
        std::lock_guard<std::mutex> lk(g_graph_mu);
        for (auto& kv : g_graphs)
            if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
        g_graphs.clear();
    }
    std::lock_guard<std::mutex> lk(g_mu);
    for (auto& kv : g_ws) free_workspace(kv.second, kv.first.second);
    g_ws.clear();
    release_batched();
    return CH_OK;
}

const char* ch_strerror(int status) {
    switch (status) {
        case CH_OK: return "ok";
        case CH_PENDING: return "pending";
        case CH_EINVAL: return "invalid argument";
        case CH_ERANGE: return "coordinate outside the integer domain [0, 2^24)";
        case CH_ENOMEM: return "out of memory or over budget";
        case CH_ECUDA: return "CUDA error";
        case CH_ETIMEOUT: return "device wait timed out";
        case CH_EBUSY: return "busy, retry";
        default: return "unknown status";
    }
}

int ch_profile_enable(int on) {
    std::lock_guard<std::mutex> lk(g_prof_mu);
    g_prof = on != 0;
    return CH_OK;
}

int ch_profile_reset(void) {
    std::lock_guard<std::mutex> lk(g_prof_mu);
    prof_drain();
    g_acc.clear();
    return CH_OK;
}

int ch_profile_read(const char** names, int64_t* launches, double* total_ms, int cap) {
    std::lock_guard<std::mutex> lk(g_prof_mu);
    prof_drain();
    g_names.clear();
    for (auto& kv : g_acc) g_names.push_back(kv.first);
    int i = 0;
    for (auto& kv : g_acc) {
        if (i < cap) {
            if (names) names[i] = g_names[i].c_str();
            if (launches) launches[i] = kv.second.first;
            if (total_ms) total_ms[i] = kv.second.second;
        }
        ++i;
    }
    return (int)g_acc.size();
}

}  // extern "C"
