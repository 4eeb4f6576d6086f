// htd_api.cu -- the extern "C" entry points declared in include/htruss.h.
//
// Every call runs on a stream private to the handle (a CUDA graph can be captured on it)
// and is ordered against the caller's stream with two events: the private stream waits
// for the caller's prior work, and the caller's stream waits for the call's work.
#include <algorithm>
#include <climits>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <vector>

#include "htd_internal.h"

struct htd_graph {
    htd::Handle H;
};

namespace htd {

namespace {
thread_local std::string g_last_error;
thread_local int64_t g_launches = 0;
constexpr int kRoundsPerGraph = 16;  // rounds of one launch each phase
constexpr int kSlotsPerGraph = 4;    // slots with the cluster round kernel
}  // namespace

void set_last_error(const std::string &msg) { g_last_error = msg; }

namespace {
constexpr uint64_t kPoolKeeps = (uint64_t)512 << 20;
// Larger blocks are cudaMalloc's: mapping 8.6 GB through the pool took 6 ms, through cudaMalloc
// a fraction of one.
constexpr size_t kLargeBytes = (size_t)64 << 20;
constexpr size_t kStatusKeeps = 32;
std::mutex g_mem_mutex;
// Pools and pinned blocks end with their context (cudaDeviceReset): they are used only in it.
struct PinnedStatus {
    int device;
    uint64_t context;
    DevStatus *p;
};
std::map<std::pair<int, uint64_t>, cudaMemPool_t> g_pool;  // by device and context
std::vector<PinnedStatus> g_status;
std::set<void *> g_large;
thread_local int64_t g_fail_alloc = 0;
thread_local bool g_no_helpers = false;
thread_local int32_t g_wait_polls = 0;
thread_local uint64_t g_context = 0;  // of the thread's present call
}  // namespace

uint64_t current_context() {
    using GetId = int (*)(void *, unsigned long long *);
    static const GetId get_id = [] {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &fn, 12000, cudaEnableDefault, &found) != cudaSuccess)
            fn = nullptr;
        return found == cudaDriverEntryPointSuccess ? reinterpret_cast<GetId>(fn) : nullptr;
    }();
    unsigned long long id = 0;
    return get_id && get_id(nullptr, &id) == 0 ? (uint64_t)id : 0;
}

void dev_free(void *p, cudaStream_t s) {
    if (!p) return;
    {
        std::lock_guard<std::mutex> lk(g_mem_mutex);
        if (g_large.erase(p) == 0) {
            cudaFreeAsync(p, s);
            return;
        }
    }
    cudaStreamSynchronize(s);
    cudaFree(p);
}

namespace {
cudaError_t alloc_bytes(void **p, size_t bytes, cudaStream_t s) {
    if (g_fail_alloc > 0 && --g_fail_alloc == 0) bytes = (size_t)1 << 50;  // more than any device has
    if (bytes >= kLargeBytes) {
        const cudaError_t e = cudaMalloc(p, bytes);
        if (e == cudaSuccess) {
            std::lock_guard<std::mutex> lk(g_mem_mutex);
            g_large.insert(*p);
        }
        return e;
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t context = g_context;
    cudaMemPool_t pool;
    {
        std::lock_guard<std::mutex> lk(g_mem_mutex);
        const auto own = g_pool.find({dev, context});
        if (own == g_pool.end()) {
            cudaMemPoolProps props;
            std::memset(&props, 0, sizeof(props));
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            e = cudaMemPoolCreate(&pool, &props);
            uint64_t keeps = kPoolKeeps;
            if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keeps);
            if (e != cudaSuccess) return e;
            g_pool[{dev, context}] = pool;
        } else {
            pool = own->second;
        }
    }
    return cudaMallocFromPoolAsync(p, bytes, pool, s);
}
}  // namespace

cudaError_t dev_alloc_bytes(void **p, size_t bytes, cudaStream_t s) {
    const cudaError_t e = alloc_bytes(p, bytes, s);
    // the caller gets it: left behind, the next launch's check would report it once more
    if (e != cudaSuccess) (void)cudaGetLastError();
    return e;
}

uint64_t call_context() { return g_context; }

htd_status enter_call(cudaStream_t user) {
    g_context = current_context();
    if (g_context == 0) {  // a thread's first call: the runtime has not bound its context yet
        (void)cudaFree(nullptr);
        g_context = current_context();
    }
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const cudaError_t e = cudaStreamIsCapturing(user, &cap);
    if (e == cudaSuccess && cap == cudaStreamCaptureStatusNone) return HTD_OK;
    if (e != cudaSuccess) (void)cudaGetLastError();
    set_last_error("htd: the caller's stream is being captured into a graph; these calls read results on the host");
    return HTD_ECUDA;
}

DevStatus *take_status_host() {
    const uint64_t context = g_context;
    {
        std::lock_guard<std::mutex> lk(g_mem_mutex);
        for (size_t i = g_status.size(); i-- > 0;) {
            if (g_status[i].context != context) continue;
            DevStatus *p = g_status[i].p;
            g_status.erase(g_status.begin() + i);
            return p;
        }
    }
    DevStatus *p = nullptr;
    if (cudaMallocHost(reinterpret_cast<void **>(&p), sizeof(DevStatus)) == cudaSuccess) return p;
    (void)cudaGetLastError();
    return nullptr;
}

void give_status_host(DevStatus *p) {
    if (!p) return;
    int device = 0;
    const uint64_t context = current_context();
    cudaGetDevice(&device);
    {
        std::lock_guard<std::mutex> lk(g_mem_mutex);
        // full of blocks of the device's other contexts: most likely ended, and the blocks with them
        if (g_status.size() >= kStatusKeeps)
            for (size_t i = g_status.size(); i-- > 0;)
                if (g_status[i].device == device && g_status[i].context != context)
                    g_status.erase(g_status.begin() + i);
        if (g_status.size() < kStatusKeeps) {
            g_status.push_back(PinnedStatus{device, context, p});
            return;
        }
    }
    cudaFreeHost(p);
}

htd_status trim_memory(int device) {
    const uint64_t context = current_context();
    std::lock_guard<std::mutex> lk(g_mem_mutex);
    cudaError_t e = cudaSuccess;
    const auto own = g_pool.find({device, context});
    if (own != g_pool.end()) e = cudaMemPoolTrimTo(own->second, 0);
    for (size_t i = g_status.size(); i-- > 0;) {
        if (g_status[i].context != context) continue;
        cudaFreeHost(g_status[i].p);
        g_status.erase(g_status.begin() + i);
    }
    if (e == cudaSuccess) return HTD_OK;
    (void)cudaGetLastError();
    set_last_error(std::string("htd_trim_memory: ") + cudaGetErrorString(e));
    return HTD_ECUDA;
}

cudaError_t raise_smem_limit(const void *func, size_t bytes) {
    static std::mutex mu;
    static std::map<std::pair<int, const void *>, std::pair<uint64_t, size_t>> limit;  // (context, bytes)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t context = g_context;
    std::lock_guard<std::mutex> lk(mu);
    auto &cur = limit[{dev, func}];
    if (cur.first == context && cur.second >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) cur = {context, bytes};
    return e;
}
bool test_no_helpers() { return g_no_helpers; }
int32_t test_wait_polls() { return g_wait_polls; }
GraphDev *graph_dev(htd_graph *g) { return &g->H.g; }
std::atomic<int32_t> &peels_in_flight(int device) {
    static std::atomic<int32_t> counts[64];
    return counts[device & 63];
}

void set_shared_device(htd_graph *g, int32_t peers) {
    g->H.shared_device = true;
    g->H.peers = peers;
}
void add_launches(int64_t k) { g_launches += k; }

}  // namespace htd

using htd::Handle;
using htd::set_last_error;

#define API_CHECK(...)                                                              \
    do {                                                                             \
        cudaError_t _e = (__VA_ARGS__);                                                     \
        if (_e != cudaSuccess) {                                                     \
            set_last_error(std::string(#__VA_ARGS__) + ": " + cudaGetErrorString(_e));      \
            return (_e == cudaErrorMemoryAllocation) ? HTD_ENOMEM : HTD_ECUDA;       \
        }                                                                            \
    } while (0)

#define API_TRY(expr)                        \
    do {                                     \
        htd_status _s = (expr);              \
        if (_s != HTD_OK) return _s;         \
    } while (0)

namespace {

// The handle's stream goes on after what is on the caller's.
htd_status follow_caller(Handle *H, cudaStream_t user) {
    API_CHECK(cudaEventRecord(H->ev_in, user));
    API_CHECK(cudaStreamWaitEvent(H->pstream, H->ev_in, 0));
    return HTD_OK;
}

htd_status begin_call(Handle *H, cudaStream_t user) {
    API_CHECK(cudaSetDevice(H->g.device));
    API_TRY(htd::enter_call(user));
    return follow_caller(H, user);
}

htd_status end_call(Handle *H, cudaStream_t user) {
    API_CHECK(cudaEventRecord(H->ev_out, H->pstream));
    API_CHECK(cudaStreamWaitEvent(user, H->ev_out, 0));
    API_CHECK(cudaStreamSynchronize(H->pstream));
    return HTD_OK;
}

void destroy_graph(Handle *H) {
    if (H->graph_exec) cudaGraphExecDestroy(H->graph_exec);
    if (H->graph_exec_timed) cudaGraphExecDestroy(H->graph_exec_timed);
    H->graph_exec = nullptr;
    H->graph_exec_timed = nullptr;
    H->graph_h = 0;
    H->graph_rounds = 0;
}

htd_status check_status_err(const htd::DevStatus *st) {
    if (st->err & htd::kErrBarrierTimeout) {
        set_last_error("htd_truss_decompose: a wait between blocks of the round kernel gave up");
        return HTD_ETIMEOUT;
    }
    if (st->err) {
        set_last_error("htd: device-side consistency check failed (code " +
                       std::to_string(st->err) + ")");
        return HTD_ECUDA;
    }
    return HTD_OK;
}

htd_status prepare_work(Handle *H, int32_t h, bool incremental, bool tiny = false) {
    if (H->w.status && (H->w.h != h || H->w.lost_tiny != tiny)) destroy_graph(H);
    return htd::ensure_work(H, h, incremental, tiny);
}

}  // namespace

namespace htd {
htd_status h_support_run(Handle *H, int32_t h, int32_t *sup_dev, cudaStream_t user) {
    API_TRY(begin_call(H, user));
    API_TRY(prepare_work(H, h, false));
    H->w.twin = false;
    H->w.dense_balls = false;  // h-support alone streams the smaller form of each ball
    H->w.inc3 = false;
    int64_t launches = 0;
    const htd_status ip = initial_pass(H, h, H->pstream, &launches, nullptr, true);
    g_launches += launches;
    API_TRY(ip);
    if (H->g.m > 0)
        API_CHECK(cudaMemcpyAsync(sup_dev, H->w.sup, H->g.m * 4, cudaMemcpyDeviceToDevice, H->pstream));
    API_CHECK(cudaMemcpyAsync(H->w.status_host, H->w.status, sizeof(DevStatus), cudaMemcpyDeviceToHost,
                              H->pstream));
    API_TRY(end_call(H, user));
    if (H->w.status_host->pool_next > 0) H->w.support_words = H->w.status_host->pool_next;
    if (H->w.status_host->pool_next > H->w.pool_words) H->w.status_host->err |= kErrBallCapacity;
    return check_status_err(H->w.status_host);
}
}  // namespace htd

extern "C" {

// For tests of what a call leaves behind when memory runs out: the calling thread's k-th
// device allocation from now on fails (0: none).  Returns how many the previous setting still
// lacked, 0 if it took effect.
int64_t htd_test_fail_alloc(int64_t k) {
    const int64_t left = htd::g_fail_alloc;
    htd::g_fail_alloc = k;
    return left;
}

// For tests: no helper cluster of the calling thread's peels takes part from now on, as on a device
// with no room for them.
void htd_test_no_helpers(int32_t on) { htd::g_no_helpers = on != 0; }

// For tests: waits between the clusters of the calling thread's round kernels give up after so many
// polls (0: the ordinary limit).
void htd_test_wait_polls(int32_t polls) { htd::g_wait_polls = polls; }

const char *htd_status_string(htd_status s) {
    switch (s) {
        case HTD_OK: return "ok";
        case HTD_EINVAL: return "invalid argument";
        case HTD_ENOMEM: return "device memory allocation failed";
        case HTD_ECUDA: return "CUDA error";
        case HTD_ETIMEOUT: return "peel exceeded its round cap, or a wait in it gave up";
        case HTD_EOVERFLOW: return "graph too large for 32-bit adjacency offsets";
        case HTD_EUNSUPPORTED: return "graph too large for shared-memory balls";
    }
    return "unknown status";
}

const char *htd_last_error(void) { return htd::g_last_error.c_str(); }

int64_t htd_kernel_launch_count(void) { return htd::g_launches; }

void htd_graph_free(htd_graph *g) {
    if (!g) return;
    Handle *H = &g->H;
    cudaSetDevice(H->g.device);
    if (H->pstream) cudaStreamSynchronize(H->pstream);
    destroy_graph(H);
    htd::free_work(H);
    htd::free_graph_dev(&H->g, H->pstream);
    // what the pool does not keep goes back to the device now
    if (H->pstream) cudaStreamSynchronize(H->pstream);
    for (cudaEvent_t e : H->round_events) cudaEventDestroy(e);
    H->round_events.clear();
    if (H->ev_in) cudaEventDestroy(H->ev_in);
    if (H->ev_out) cudaEventDestroy(H->ev_out);
    if (H->pstream) cudaStreamDestroy(H->pstream);
    delete g;
}

htd_status htd_trim_memory(void) {
    int dev = 0;
    API_CHECK(cudaGetDevice(&dev));
    return htd::trim_memory(dev);
}

htd_status htd_build_csr(int32_t n, const int32_t *src, const int32_t *dst, int64_t m_in,
                         int inputs_on_device, void *stream, htd_graph **out) {
    if (!out) {
        set_last_error("htd_build_csr: out is NULL");
        return HTD_EINVAL;
    }
    *out = nullptr;
    if (n < 0 || m_in < 0 || (m_in > 0 && (!src || !dst))) {
        set_last_error("htd_build_csr: bad n, m_in or NULL endpoint array");
        return HTD_EINVAL;
    }
    if (n > HTD_MAX_N) {
        set_last_error("htd_build_csr: n exceeds HTD_MAX_N");
        return HTD_EUNSUPPORTED;
    }
    if (2 * m_in >= (int64_t)INT32_MAX) {
        set_last_error("htd_build_csr: 2*m_in >= 2^31");
        return HTD_EOVERFLOW;
    }
    cudaStream_t user = static_cast<cudaStream_t>(stream);
    API_TRY(htd::enter_call(user));
    htd_graph *G = new htd_graph();
    Handle *H = &G->H;
    htd_status st = HTD_OK;
    int32_t *dsrc = nullptr, *ddst = nullptr;
    int64_t launches = 0;
    auto fail = [&](htd_status s) {
        htd::dev_free(dsrc, H->pstream);
        htd::dev_free(ddst, H->pstream);
        htd_graph_free(G);
        return s;
    };
    {
        cudaError_t e = cudaGetDevice(&H->g.device);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&H->num_sms, cudaDevAttrMultiProcessorCount,
                                                         H->g.device);
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&H->pstream, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&H->ev_in, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&H->ev_out, cudaEventDisableTiming);
        if (e != cudaSuccess) {
            set_last_error(std::string("htd_build_csr: ") + cudaGetErrorString(e));
            return fail(HTD_ECUDA);
        }
    }
    st = follow_caller(H, user);
    if (st != HTD_OK) return fail(st);
    const int32_t *s_dev = src, *d_dev = dst;
    if (!inputs_on_device && m_in > 0) {
        cudaError_t e = htd::dev_alloc(&dsrc, m_in, H->pstream);
        if (e == cudaSuccess) e = htd::dev_alloc(&ddst, m_in, H->pstream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(dsrc, src, m_in * sizeof(int32_t), cudaMemcpyHostToDevice, H->pstream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(ddst, dst, m_in * sizeof(int32_t), cudaMemcpyHostToDevice, H->pstream);
        if (e != cudaSuccess) {
            set_last_error(std::string("htd_build_csr: input copy: ") + cudaGetErrorString(e));
            return fail(e == cudaErrorMemoryAllocation ? HTD_ENOMEM : HTD_ECUDA);
        }
        s_dev = dsrc;
        d_dev = ddst;
    }
    st = htd::build_csr_device(n, s_dev, d_dev, m_in, H->pstream, &H->g, &launches);
    htd::g_launches += launches;
    if (st != HTD_OK) return fail(st);
    st = end_call(H, user);
    if (st != HTD_OK) return fail(st);
    htd::dev_free(dsrc, H->pstream);
    htd::dev_free(ddst, H->pstream);
    *out = G;
    return HTD_OK;
}

htd_status htd_graph_info(const htd_graph *g, int32_t *n, int64_t *m) {
    if (!g) {
        set_last_error("htd_graph_info: NULL handle");
        return HTD_EINVAL;
    }
    if (n) *n = g->H.g.n;
    if (m) *m = g->H.g.m;
    return HTD_OK;
}

htd_status htd_edges(const htd_graph *g, int32_t *eu_dev, int32_t *ev_dev, void *stream) {
    if (!g || (g->H.g.m > 0 && (!eu_dev || !ev_dev))) {
        set_last_error("htd_edges: NULL argument");
        return HTD_EINVAL;
    }
    Handle *H = const_cast<Handle *>(&g->H);
    cudaStream_t user = static_cast<cudaStream_t>(stream);
    API_TRY(begin_call(H, user));
    if (H->g.m > 0) {
        API_CHECK(cudaMemcpyAsync(eu_dev, H->g.eu, H->g.m * 4, cudaMemcpyDeviceToDevice, H->pstream));
        API_CHECK(cudaMemcpyAsync(ev_dev, H->g.ev, H->g.m * 4, cudaMemcpyDeviceToDevice, H->pstream));
    }
    return end_call(H, user);
}

htd_status htd_csr(const htd_graph *g, int32_t *row_ptr_dev, int32_t *col_dev,
                   int32_t *slot_eid_dev, void *stream) {
    if (!g) {
        set_last_error("htd_csr: NULL handle");
        return HTD_EINVAL;
    }
    Handle *H = const_cast<Handle *>(&g->H);
    cudaStream_t user = static_cast<cudaStream_t>(stream);
    API_TRY(begin_call(H, user));
    const int64_t n = H->g.n, m = H->g.m;
    if (row_ptr_dev)
        API_CHECK(cudaMemcpyAsync(row_ptr_dev, H->g.row_ptr, (n + 1) * 4, cudaMemcpyDeviceToDevice,
                                  H->pstream));
    if (col_dev && m > 0)
        API_CHECK(cudaMemcpyAsync(col_dev, H->g.col, 2 * m * 4, cudaMemcpyDeviceToDevice, H->pstream));
    if (slot_eid_dev && m > 0)
        API_CHECK(cudaMemcpyAsync(slot_eid_dev, H->g.slot_eid, 2 * m * 4, cudaMemcpyDeviceToDevice,
                                  H->pstream));
    return end_call(H, user);
}

htd_status htd_h_support(htd_graph *g, int32_t h, int32_t *sup_dev, void *stream) {
    if (!g || h < 1 || h > HTD_MAX_H || (g->H.g.m > 0 && !sup_dev)) {
        set_last_error("htd_h_support: NULL argument or h outside [1, HTD_MAX_H]");
        return HTD_EINVAL;
    }
    const htd_status st = htd::h_support_run(&g->H, h, sup_dev, static_cast<cudaStream_t>(stream));
    htd::trim_support(&g->H);
    return st;
}

htd_status htd_truss_decompose_ex(htd_graph *g, int32_t h, uint32_t flags, int32_t *truss_dev,
                                  int32_t *stamp_dev, htd_stats *stats, void *stream) {
    if (!g || h < 1 || h > HTD_MAX_H || (g->H.g.m > 0 && !truss_dev)) {
        set_last_error("htd_truss_decompose: NULL argument or h outside [1, HTD_MAX_H]");
        return HTD_EINVAL;
    }
    Handle *H = &g->H;
    htd::PeelWork &w = H->w;
    cudaStream_t user = static_cast<cudaStream_t>(stream);
    const bool timing = (flags & HTD_OPT_TIMING) != 0;
    const bool graphs_wanted = (flags & HTD_OPT_NO_GRAPH) == 0;
    htd_stats local;
    std::memset(&local, 0, sizeof(local));
    local.h = h;
    int64_t launches = 0;
    int64_t launches_counted = 0;
    // adds the launches enqueued since the last call to the thread's counter
    auto count_launches = [&]() {
        htd::g_launches += launches - launches_counted;
        launches_counted = launches;
    };

    API_TRY(begin_call(H, user));
    bool incremental = (flags & HTD_OPT_REBUILD) == 0;
    {
        // the incremental peel's membership tests take one load on a dense ball, a binary
        // search on a compact one: keep every ball dense when the n x n bits fit comfortably.
        // At h = 3 the incremental rounds need two dense ball sets (radius 2 and 3).
        size_t free_b = 0, total_b = 0;
        API_CHECK(cudaMemGetInfo(&free_b, &total_b));
        const double Wp = (double)(((H->g.n + 31) / 32 + 3) & ~3);
        const double dense_bytes = 4.0 * (double)H->g.n * (Wp > 0 ? Wp : 4.0);
        const bool fits = dense_bytes <= (double)free_b / 4 && dense_bytes < 4.0 * (double)((int64_t)1 << 33);
        if (h == 3 && ((flags & HTD_OPT_COMPACT_BALLS) != 0 || !(2.0 * dense_bytes <= (double)free_b / 3) ||
                       dense_bytes >= 4.0 * (double)((int64_t)1 << 33)))
            incremental = false;
        API_TRY(prepare_work(H, h, incremental, (flags & HTD_OPT_TINY_LOSS_TABLE) != 0));
        incremental = w.incremental;
        w.dense_balls = incremental && (h == 3 || ((flags & HTD_OPT_COMPACT_BALLS) == 0 && fits));
        // (beside other peels a quarter of what these have left: their admission counts twins.
        // 4,096 graphs in 42 unions of up to 262,144 vertices 21.2 s without, 13.4 s with)
        API_TRY(htd::ensure_twin(H, (int64_t)(free_b / (H->shared_device ? 4 : 8))));
    }
    {
        htd_status ip = htd::initial_pass(H, h, H->pstream, &launches, timing ? &local : nullptr, false);
        if (ip == HTD_OK) ip = htd::initial_pass_r2(H, H->pstream, &launches);
        htd::g_launches += launches;
        launches_counted = launches;
        API_TRY(ip);
    }
    API_CHECK(cudaMemcpyAsync(w.status_host, w.status, sizeof(htd::DevStatus), cudaMemcpyDeviceToHost,
                              H->pstream));
    API_CHECK(cudaStreamSynchronize(H->pstream));
    API_TRY(check_status_err(w.status_host));

    const htd::PeelInFlight in_flight(H->g.device);
    // a slot with the cluster round kernel holds many rounds
    const int R = incremental && w.twin ? htd::kSlotsPerGraph : htd::kRoundsPerGraph;
    const bool persistent = incremental && h <= 2 && (flags & HTD_OPT_PERSISTENT_ROUNDS) != 0;
    if (persistent && w.status_host->alive > 0) {
        // one cooperative launch runs up to kPersistentSlots round slots; the host checks the
        // status block between launches
        constexpr int kPersistentSlots = 4096;
        const int64_t slot_cap = H->g.m + w.status_host->st_ball_total / 2 + 2;
        const int64_t launch_cap = slot_cap / kPersistentSlots + 3;
        cudaEvent_t p0 = nullptr, p1 = nullptr;
        API_CHECK(cudaEventCreate(&p0));
        API_CHECK(cudaEventCreate(&p1));
        int64_t nlaunch = 0;
        htd_status ps = HTD_OK;
        while (ps == HTD_OK && w.status_host->alive > 0) {
            if (++nlaunch > launch_cap) {
                set_last_error("htd_truss_decompose: no progress within the slot cap");
                ps = HTD_ETIMEOUT;
                break;
            }
            if (cudaEventRecord(p0, H->pstream) != cudaSuccess) ps = HTD_ECUDA;
            if (ps == HTD_OK) ps = htd::launch_persistent_rounds(H, H->pstream, kPersistentSlots, &launches);
            if (ps == HTD_OK && cudaEventRecord(p1, H->pstream) != cudaSuccess) ps = HTD_ECUDA;
            count_launches();
            if (ps != HTD_OK) break;
            if (cudaMemcpyAsync(w.status_host, w.status, sizeof(htd::DevStatus),
                                cudaMemcpyDeviceToHost, H->pstream) != cudaSuccess ||
                cudaStreamSynchronize(H->pstream) != cudaSuccess) {
                set_last_error(std::string("htd_truss_decompose: ") +
                               cudaGetErrorString(cudaGetLastError()));
                ps = HTD_ECUDA;
                break;
            }
            float ms = 0.f;
            if (cudaEventElapsedTime(&ms, p0, p1) == cudaSuccess) {
                local.ms_round_kernel += ms;
                local.round_kernel_launches += 1;
            }
            ps = check_status_err(w.status_host);
        }
        cudaEventDestroy(p0);
        cudaEventDestroy(p1);
        if (ps != HTD_OK) return ps;
        const htd::DevStatus *sh = w.status_host;
        local.ms_select = sh->st_phase_ns[0] * 1e-6f;
        local.ms_find = sh->st_phase_ns[1] * 1e-6f;
        local.ms_update = sh->st_phase_ns[3] * 1e-6f;
        local.ms_minreduce = sh->st_phase_ns[4] * 1e-6f;
        local.timed_slots = sh->st_slots;
    } else if (w.status_host->alive > 0) {
        // Graph path: R rounds per graph launch.  With HTD_OPT_TIMING a second graph with an
        // external event record at every phase boundary runs every kTimedEvery-th batch (the
        // events would otherwise slow every round); per-launch averages come from those.
        constexpr int kTimedEvery = 16;
        // slots that hold many rounds are launched directly: capturing and instantiating a graph
        // costs more than the few slots of a peel save
        const bool use_graph = graphs_wanted && !w.twin;
        const bool by_events = timing && !incremental;  // incremental rounds time themselves
        if (by_events && H->round_events.empty()) {
            H->round_events.resize(htd::kRoundEvents * R, nullptr);
            for (auto &e : H->round_events) API_CHECK(cudaEventCreate(&e));
        }
        auto capture = [&](cudaGraphExec_t *exec, cudaEvent_t *ev, bool timed) -> htd_status {
            cudaGraph_t graph = nullptr;
            API_CHECK(cudaStreamBeginCapture(H->pstream, cudaStreamCaptureModeThreadLocal));
            int64_t per_graph = 0;
            htd_status cs = HTD_OK;
            for (int r = 0; r < R && cs == HTD_OK; r++)
                cs = htd::enqueue_round(H, H->pstream, &per_graph, ev ? ev + htd::kRoundEvents * r : nullptr,
                                        timed, w.twin);
            cudaError_t ce = cudaStreamEndCapture(H->pstream, &graph);
            if (cs != HTD_OK) {
                if (graph) cudaGraphDestroy(graph);
                return cs;
            }
            if (ce != cudaSuccess) {
                set_last_error(std::string("htd: graph capture: ") + cudaGetErrorString(ce));
                return HTD_ECUDA;
            }
            ce = cudaGraphInstantiate(exec, graph, 0);
            cudaGraphDestroy(graph);
            if (ce != cudaSuccess) {
                *exec = nullptr;
                set_last_error(std::string("htd: graph instantiate: ") + cudaGetErrorString(ce));
                return HTD_ECUDA;
            }
            H->graph_launches = per_graph;
            return HTD_OK;
        };
        // the captured kernel arguments fix h, the round variant and the ball layout
        if (use_graph && (!H->graph_exec || H->graph_h != h || H->graph_incremental != incremental ||
                          H->graph_dense != w.dense_balls || H->graph_shared != H->shared_device || H->graph_twin != w.twin)) {
            destroy_graph(H);
            API_TRY(capture(&H->graph_exec, nullptr, false));
            H->graph_h = h;
            H->graph_rounds = R;
            H->graph_incremental = incremental;
            H->graph_dense = w.dense_balls;
            H->graph_shared = H->shared_device;
            H->graph_twin = w.twin;
        }
        if (use_graph && timing && !H->graph_exec_timed)
            API_TRY(capture(&H->graph_exec_timed, by_events ? H->round_events.data() : nullptr, true));
        // every active round removes at least one edge, so m/R + 2 batches always suffice
        const int64_t round_cap = H->g.m + 2 * R + 2;
        // continued incremental rounds handle at least one new lost pair per slot, and a
        // pair is lost at most once (sum of ball sizes / 2 pairs in all)
        const int64_t batch_cap =
            (H->g.m + (incremental ? w.status_host->st_ball_total / 2 + 1 : 0)) / (w.twin ? 1 : R) + 3;
        int64_t batches = 0;
        int cluster_reads = 0;  // reads of the status before slots with the cluster round kernel
        int continued = 0;      // reads in a row that found a round of several batches
        bool timing_ok = by_events;
        while (w.status_host->alive > 0) {
            if (++batches > batch_cap) {
                set_last_error("htd_truss_decompose: no progress within the batch cap");
                return HTD_ETIMEOUT;
            }
            const bool timed = timing_ok && (batches % kTimedEvery == 1);
            const int64_t slots_before = w.status_host->st_slots;
            if (use_graph) {
                const bool second = timed || (timing && incremental);
                API_CHECK(cudaGraphLaunch(second ? H->graph_exec_timed : H->graph_exec, H->pstream));
                launches += H->graph_launches;
            } else {
                // the first slot often ends a small peel: one, then more at a time.  A round that has
                // taken several batches is the phase launches', and so are the next ones: in each
                // slot the cluster round kernel would return at once (128-slot tables, ER
                // n = 2,000 at h = 2: 49 ms with it, 35 without)
                const bool by_cluster = w.twin && w.status_host->cont == 0;
                // (such a round often needs one batch more: two slots, then more at a time, and one
                // with the cluster kernel for what comes after it)
                const bool in_batches = w.twin && !by_cluster;
                const int slots = by_cluster   ? std::min(R, ++cluster_reads)
                                  : in_batches ? std::min(htd::kRoundsPerGraph, 2 << std::min(continued, 3)) + 1
                                               : htd::kRoundsPerGraph;
                continued = in_batches ? continued + 1 : 0;
                for (int r = 0; r < slots; r++) {
                    API_TRY(htd::enqueue_round(H, H->pstream, &launches,
                                               timed ? &H->round_events[htd::kRoundEvents * r] : nullptr,
                                               timing, by_cluster || (in_batches && r == slots - 1)));
                }
            }
            count_launches();
            API_CHECK(cudaMemcpyAsync(w.status_host, w.status, sizeof(htd::DevStatus),
                                      cudaMemcpyDeviceToHost, H->pstream));
            API_CHECK(cudaStreamSynchronize(H->pstream));
            API_TRY(check_status_err(w.status_host));
            const bool halted = w.status_host->halt != 0;
            if (halted) {
                // an h = 3 round ran out of room: finish it by rebuilds, then go on (the
                // batch's sampled events then cover idle rounds and are not used)
                API_TRY(htd::recover_round_h3(H, H->pstream, &launches));
                count_launches();
                API_CHECK(cudaMemcpyAsync(w.status_host, w.status, sizeof(htd::DevStatus),
                                          cudaMemcpyDeviceToHost, H->pstream));
                API_CHECK(cudaStreamSynchronize(H->pstream));
                API_TRY(check_status_err(w.status_host));
            }
            if (timed && !halted) {
                // only the slots that ran a round (or a batch of one) count; those after the
                // last round are no-ops
                const int64_t active = std::min<int64_t>(R, w.status_host->st_slots - slots_before);
                for (int r = 0; r < active && timing_ok; r++) {
                    float t[htd::kRoundEvents - 1];
                    for (int q = 0; q + 1 < htd::kRoundEvents; q++) {
                        if (cudaEventElapsedTime(&t[q], H->round_events[htd::kRoundEvents * r + q],
                                                 H->round_events[htd::kRoundEvents * r + q + 1]) !=
                            cudaSuccess) {
                            (void)cudaGetLastError();  // not sticky: report "no timing" instead
                            timing_ok = false;
                            break;
                        }
                    }
                    if (!timing_ok) break;
                    local.ms_select += t[0];
                    local.ms_find += t[1];
                    local.ms_remove += t[2];
                    local.ms_ball += t[3];
                    local.ms_update += t[4];
                    local.ms_minreduce += t[5];
                    local.timed_slots += 1;
                }
                if (!timing_ok) local.timed_slots = -1;
            }
            if (w.status_host->round > round_cap) {
                set_last_error("htd_truss_decompose: round cap exceeded");
                return HTD_ETIMEOUT;
            }
        }
        if (timing && incremental) {
            // as at the event-timed rounds: detection | radius-3 tests in the "remove" place
            const unsigned long long *ns = w.status_host->st_phase_ns;
            local.ms_select = ns[0] * 1e-6f;
            local.ms_remove = (h == 3 ? ns[1] : 0) * 1e-6f;
            local.ms_find = (h == 3 ? ns[2] : ns[1]) * 1e-6f;
            local.ms_update = ns[3] * 1e-6f;
            local.ms_minreduce = ns[4] * 1e-6f;
            local.timed_slots = w.status_host->st_slots;
        }
    }
    const int64_t m = H->g.m;
    if (m > 0) {
        API_CHECK(cudaMemcpyAsync(truss_dev, w.truss, m * 4, cudaMemcpyDeviceToDevice, H->pstream));
        if (stamp_dev)
            API_CHECK(cudaMemcpyAsync(stamp_dev, w.stamp, m * 4, cudaMemcpyDeviceToDevice, H->pstream));
    }
    API_TRY(end_call(H, user));
    if (stats) {
        const htd::DevStatus *s = w.status_host;
        local.rounds = s->round;
        local.levels = s->levels;
        local.max_truss = s->max_k;
        local.hsup_evals = m + s->st_recomputed;
        local.pairs_tested = s->st_pairs;
        local.pairs_lost = s->st_lost;
        local.member_tests = s->st_tests;
        local.incremental = incremental ? 1 : 0;
        local.slots = s->st_slots;
        local.levels = s->levels;
        local.ball_builds = H->g.n + s->st_candidates;
        local.balls_changed = s->st_changed;
        local.frontier_edges = s->st_frontier;
        local.alg_bytes_ball = (double)s->st_bytes_ball + (double)w.or_bytes;
        local.alg_bytes_hsup = (double)s->st_bytes_hsup;
        local.alg_bytes_hsup_initial = (double)s->st_bytes_hsup_init;
        local.alg_bytes_detect = (double)s->st_bytes_detect;
        local.alg_bytes_update = (double)s->st_bytes_update;
        local.kernel_launches = launches;
        local.ball_pool_bytes = (w.pool_used + (w.inc3 ? (int64_t)H->g.n * w.Wpad : 0)) * 4;
        local.pairs3_tested = s->st_c3_pairs;
        local.pairs2_lost = s->st_lost2;
        local.rounds_rebuilt = s->st_recovered;
        *stats = local;
    }
    return HTD_OK;
}

htd_status htd_hindex_decompose_ex(htd_graph *g, int32_t h, int32_t sweeps, int32_t max_iter,
                                   uint32_t flags, int32_t *truss_dev, int32_t *hval_dev,
                                   htd_hindex_stats *stats, void *stream) {
    if (!g || h < 1 || h > HTD_MAX_H || sweeps < 1 || sweeps > 4096 || (flags & ~HTD_HX_PRUNE) != 0u ||
        ((flags & HTD_HX_PRUNE) && sweeps != 1)) {
        set_last_error("htd_hindex_decompose: NULL handle, h outside [1, HTD_MAX_H], sweeps outside "
                       "[1, 4096], unknown flags, or pruning with sweeps != 1");
        return HTD_EINVAL;
    }
    Handle *H = &g->H;
    cudaStream_t user = static_cast<cudaStream_t>(stream);
    API_TRY(begin_call(H, user));
    const htd_status hs = htd::hindex_run(g, H, h, sweeps, max_iter, (flags & HTD_HX_PRUNE) != 0u, truss_dev,
                                          hval_dev, stats, H->pstream);
    htd::trim_support(H);
    API_TRY(hs);
    return end_call(H, user);
}

htd_status htd_hindex_decompose(htd_graph *g, int32_t h, int32_t sweeps, int32_t max_iter,
                                int32_t *truss_dev, int32_t *hval_dev, htd_hindex_stats *stats,
                                void *stream) {
    return htd_hindex_decompose_ex(g, h, sweeps, max_iter, 0u, truss_dev, hval_dev, stats, stream);
}

htd_status htd_truss_decompose(htd_graph *g, int32_t h, int32_t *truss_dev, int32_t *stamp_dev,
                               htd_stats *stats, void *stream) {
    return htd_truss_decompose_ex(g, h, 0u, truss_dev, stamp_dev, stats, stream);
}

htd_status htd_truss_decompose_host(int32_t n, const int32_t *src_host, const int32_t *dst_host,
                                    int64_t m_in, int32_t h, int32_t *eu_host, int32_t *ev_host,
                                    int32_t *truss_host, int64_t *m_out, htd_stats *stats,
                                    void *stream) {
    if (!m_out || (m_in > 0 && (!src_host || !dst_host || !eu_host || !ev_host || !truss_host)) ||
        h < 1 || h > HTD_MAX_H) {
        set_last_error("htd_truss_decompose_host: NULL argument or bad h");
        return HTD_EINVAL;
    }
    htd_graph *g = nullptr;
    API_TRY(htd_build_csr(n, src_host, dst_host, m_in, 0, stream, &g));
    Handle *H = &g->H;
    const int64_t m = H->g.m;
    int32_t *truss_dev = nullptr;
    htd_status st = HTD_OK;
    cudaStream_t user = static_cast<cudaStream_t>(stream);
    if (htd::dev_alloc(&truss_dev, m, user) != cudaSuccess) {
        set_last_error("htd_truss_decompose_host: output allocation failed");
        htd_graph_free(g);
        return HTD_ENOMEM;
    }
    st = htd_truss_decompose(g, h, truss_dev, nullptr, stats, stream);
    if (st == HTD_OK && m > 0) {
        cudaError_t e = cudaMemcpyAsync(eu_host, H->g.eu, m * 4, cudaMemcpyDeviceToHost, user);
        if (e == cudaSuccess) e = cudaMemcpyAsync(ev_host, H->g.ev, m * 4, cudaMemcpyDeviceToHost, user);
        if (e == cudaSuccess) e = cudaMemcpyAsync(truss_host, truss_dev, m * 4, cudaMemcpyDeviceToHost, user);
        if (e == cudaSuccess) e = cudaStreamSynchronize(user);
        if (e != cudaSuccess) {
            set_last_error(std::string("htd_truss_decompose_host: copy back: ") + cudaGetErrorString(e));
            st = HTD_ECUDA;
        }
    }
    if (st == HTD_OK) *m_out = m;
    htd::dev_free(truss_dev, user);
    htd_graph_free(g);
    return st;
}

}  // extern "C"
