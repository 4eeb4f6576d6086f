// htd_hindex.cu -- the paper's own parallel method on the device: the higher-order H-index
// iteration of Sec. 4 (Definition of the h-hop reachable path key, Theorems 3 and 4,
// Algorithm 2, asynchronous updating).
//
// With H^(0)(e) = sup_G(e,h), order n computes for every edge e = (u,v)
//     H^(n)(e) = H({ min(P(u,w), P(v,w)) : w in N_G(u,h) ∩ N_G(v,h) }),
// where H(S) is the largest y such that at least y members of S are >= y, and P(a,b), the
// h-hop reachable path key, is the largest over paths from a to b of at most h edges of
// the smallest H^(n-1) on the path.  The iteration stops at the first order that changes
// nothing, and then t(e,h) = H(e) + 2 (Theorem 4).  Readings (as in the oracle): paths have
// at most h edges and may use e itself; the common h-neighbourhood is that of the whole
// graph G, which never changes.
//
// GPU form.  The graph is fixed, so every vertex's closed ball B(x,h) is kept as a sorted
// member list, taken from the balls the h-support pass (H^(0)) has just built.  An order is
// two kernels, one block per vertex each, with that vertex's ball in shared memory as an
// n-bit set and, per word, the rank of its first member: a member's place in the list is then
// two shared-memory reads.  (Binary searches in the lists, about ten dependent loads for every
// relaxation and every common member, made an order 12 ms on DC-SBM 50k at h = 2.)
//   k_hx_pathkeys  P(x, .) over the members of B(x,h) by h rounds of hop-limited relaxation
//                  (round r extends paths of at most r-1 edges by one edge);
//   k_hx_edges     the edges the vertex owns (the endpoint with the larger ball), one warp
//                  each: the other endpoint's members are streamed against the set, the values
//                  min(P(u,w), P(v,w)) of the common ones gathered in a per-warp buffer, and
//                  H(.) found by the monotone test "at least y values >= y", down from the
//                  old key in growing steps (keys never increase), then by bisection.
// Synchronous orders (Algorithm 2) write the new keys to a second array.  With pruning
// (Lemma 4), from the second order on an edge keeps its key without being computed when no
// edge near it fell across that key in the previous order: per vertex, the range of the
// fallen edges' values (lowest new, highest old) is spread h-1 hops, and an edge whose two
// endpoints' ranges do not straddle its key is skipped (the range hull is a conservative
// form of the lemma's per-edge conditions, so the result is unchanged); path keys are then
// computed only at the endpoints of the edges still listed.  The asynchronous
// form splits every sweep into S sub-sweeps over consecutive edge-id ranges: a sub-sweep
// recomputes the path keys of the vertices its edges touch from the current keys and
// writes its edges' keys in place, so later sub-sweeps already use them (the paper's
// asynchronous updating, by blocks of edges).  Keys never increase, so both forms reach
// the same fixed point.
#include <algorithm>
#include <climits>
#include <cstring>
#include <string>
#include <vector>

#include "htd_internal.h"
#include "htd_scan.cuh"

namespace htd {
namespace {

constexpr int kBlock = 256;

// Sorted member lists of every vertex, block per vertex, from the stored balls (dense words,
// or sorted (word index, word) pairs).
__global__ void __launch_bounds__(kBlock) k_hx_members(int32_t n, int32_t W, const uint32_t *__restrict__ pool,
                                                      const int64_t *__restrict__ ball_off,
                                                      const int32_t *__restrict__ ball_nw,
                                                      const int64_t *__restrict__ off,
                                                      int32_t *__restrict__ members) {
    __shared__ int32_t s_scan[kBlock / 32];
    for (int x = blockIdx.x; x < n; x += gridDim.x) {
        const int nw = ball_nw[x], count = nw < 0 ? W : nw;
        const uint32_t *words = pool + ball_off[x];
        int64_t base = off[x];
        for (int i0 = 0; i0 < count; i0 += kBlock) {
            const int i = i0 + threadIdx.x;
            int w = i;
            uint32_t v = 0u;
            if (i < count) {
                if (nw < 0) {
                    v = words[i];
                } else {
                    w = (int)words[2 * i];
                    v = words[2 * i + 1];
                }
            }
            int tot;
            int at = block_exclusive_scan<kBlock, int>(__popc(v), &tot, s_scan);
            while (v) {
                const int b = __ffs(v) - 1;
                v &= v - 1u;
                members[base + at++] = (w << 5) + b;
            }
            base += tot;
        }
    }
}

// Index of z in the sorted list m[0..len), or -1.
__device__ __forceinline__ int find_member(const int32_t *__restrict__ m, int len, int z) {
    int lo = 0, hi = len - 1;
    while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        const int v = m[mid];
        if (v == z) return mid;
        if (v < z) lo = mid + 1;
        else hi = mid - 1;
    }
    return -1;
}

// A vertex's ball in shared memory: the n-bit set and, for every word that holds members,
// the rank of its first one (the list is sorted, so that member knows its own rank).  Where
// the two do not fit (words == 0), places are found by binary search in the list.
struct BallIndex {
    uint32_t *bits;
    int32_t *rank;
    const int32_t *m;  // member list
    int32_t len;
    int32_t words;

    __device__ void clear_all() {
        for (int i = threadIdx.x; i < words; i += blockDim.x) bits[i] = 0u;
        __syncthreads();
    }
    __device__ void load(const int32_t *list, int n) {
        m = list;
        len = n;
        if (words == 0) return;
        for (int j = threadIdx.x; j < len; j += blockDim.x) {
            const int z = m[j], w = z >> 5;
            atomicOr(bits + w, 1u << (z & 31));
            if (j == 0 || (m[j - 1] >> 5) != w) rank[w] = j;
        }
        __syncthreads();
    }
    // after a barrier; the next load needs one more
    __device__ void unload() {
        if (words == 0) return;
        for (int j = threadIdx.x; j < len; j += blockDim.x) bits[m[j] >> 5] = 0u;
    }
    __device__ __forceinline__ int find(int z) const {
        if (words == 0) return find_member(m, len, z);
        const uint32_t v = bits[z >> 5], below = (1u << (z & 31)) - 1u;
        return (v >> (z & 31)) & 1u ? rank[z >> 5] + __popc(v & below) : -1;
    }
};

// P(x, .) for the vertices of `list` (all vertices if null; `count`, or *dcount of them), block
// per vertex.  The values are kept in shared memory while they fit pcap entries, else in P;
// `prev` is the block's scratch of maxb entries (the values of the previous round, h >= 3).
__global__ void __launch_bounds__(kBlock) k_hx_pathkeys(const int32_t *__restrict__ list, int32_t count,
                                                       const int32_t *__restrict__ dcount, int32_t h,
                                                       const int32_t *__restrict__ row_ptr,
                                                       const int32_t *__restrict__ col,
                                                       const int32_t *__restrict__ slot_eid,
                                                       const int32_t *__restrict__ key,
                                                       const int64_t *__restrict__ off,
                                                       const int32_t *__restrict__ members,
                                                       int32_t *__restrict__ P, int32_t *prev_all,
                                                       int64_t maxb, int32_t words, int32_t pcap) {
    extern __shared__ __align__(16) uint32_t smem[];
    BallIndex ball;
    ball.bits = smem;
    ball.rank = reinterpret_cast<int32_t *>(smem + words);
    ball.words = words;
    int32_t *const sp = reinterpret_cast<int32_t *>(smem + 2 * words);
    int32_t *prev = prev_all + (int64_t)blockIdx.x * maxb;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (dcount) count = *dcount;
    ball.clear_all();
    for (int i = blockIdx.x; i < count; i += gridDim.x) {
        const int x = list ? list[i] : i;
        const int64_t o = off[x];
        const int len = (int)(off[x + 1] - o);
        int32_t *const p = len <= pcap ? sp : P + o;
        for (int j = threadIdx.x; j < len; j += blockDim.x) p[j] = -1;
        ball.load(members + o, len);
        __syncthreads();
        const int rb = row_ptr[x], re = row_ptr[x + 1];
        // round 1: the edges of x
        if (threadIdx.x == 0) p[ball.find(x)] = INT_MAX;
        for (int s = rb + threadIdx.x; s < re; s += blockDim.x) p[ball.find(col[s])] = key[slot_eid[s]];
        __syncthreads();
        // every neighbour of a vertex within r-1 <= h-1 edges of x is a member of the ball
        for (int r = 2; r <= h; r++) {
            if (r > 2) {
                for (int j = threadIdx.x; j < len; j += blockDim.x) prev[j] = p[j];
                __syncthreads();
            }
            // one warp per vertex reached within r-1 edges (r = 2: the row of x says which,
            // and with what value); its lanes walk that vertex's row
            const int sources = r == 2 ? re - rb : len;
            for (int j = wid; j < sources; j += nw) {
                const int pv = r == 2 ? key[slot_eid[rb + j]] : prev[j];
                if (pv < 0) continue;
                const int y = r == 2 ? col[rb + j] : members[o + j];
                const int ye = row_ptr[y + 1];
                for (int s = row_ptr[y] + lane; s < ye; s += 32) {
                    const int iz = ball.find(col[s]);
                    const int c = min(pv, key[slot_eid[s]]);
                    if (c > p[iz]) atomicMax(&p[iz], c);
                }
            }
            __syncthreads();
        }
        if (len <= pcap)
            for (int j = threadIdx.x; j < len; j += blockDim.x) P[o + j] = p[j];
        ball.unload();
        __syncthreads();
    }
}

// Work items of k_hx_edges: every kItemSlots adjacency slots of the vertices of `list` (all
// vertices if null), so that a hub's edges are spread over many blocks.
constexpr int kItemSlots = 64;

__global__ void k_hx_items(const int32_t *__restrict__ list, int32_t count, const int32_t *__restrict__ dcount,
                           const int32_t *__restrict__ row_ptr, int2 *__restrict__ items, int32_t *nitems) {
    if (dcount) count = *dcount;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const int x = list ? list[i] : i;
        const int rb = row_ptr[x], nch = (row_ptr[x + 1] - rb + kItemSlots - 1) / kItemSlots;
        if (nch == 0) continue;
        const int first = atomicAdd(nitems, nch);
        for (int c = 0; c < nch; c++) items[first + c] = make_int2(x, rb + c * kItemSlots);
    }
}

// New keys of the listed edges: those of [e0, e1), or with `emark` those with emark[e] ==
// stamp.  A block takes an item (a vertex and a run of its slots) at a time from a queue, its
// warps the listed edges that vertex owns.  vals: the warp's buffer of maxd.
__global__ void __launch_bounds__(kBlock) k_hx_edges(const int2 *__restrict__ items, const int32_t *__restrict__ nitems,
                                                    int32_t *queue, int64_t e0, int64_t e1,
                                                    const int32_t *__restrict__ emark, int32_t stamp,
                                                    const int32_t *__restrict__ row_ptr,
                                                    const int32_t *__restrict__ col,
                                                    const int32_t *__restrict__ slot_eid,
                                                    const int64_t *__restrict__ off,
                                                    const int32_t *__restrict__ members,
                                                    const int32_t *__restrict__ P,
                                                    const int32_t *key_in, int32_t *key_out,
                                                    int32_t *vals_all, int64_t maxd,
                                                    unsigned long long *changed, int32_t words, int32_t pcap) {
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ int32_t s_slot[kItemSlots], s_n, s_next, s_item;
    BallIndex ball;
    ball.bits = smem;
    ball.rank = reinterpret_cast<int32_t *>(smem + words);
    ball.words = words;
    int32_t *const sp = reinterpret_cast<int32_t *>(smem + 2 * words);
    const int lane = threadIdx.x & 31;
    int32_t *vals = vals_all + ((int64_t)blockIdx.x * (kBlock / 32) + (threadIdx.x >> 5)) * maxd;
    unsigned long long nchg = 0;
    const int count = *nitems;
    ball.clear_all();
    for (;;) {
        if (threadIdx.x == 0) {
            s_item = atomicAdd(queue, 1);
            s_n = s_next = 0;
        }
        __syncthreads();
        const int it = s_item;
        if (it >= count) break;
        const int2 item = items[it];
        const int u = item.x;
        const int64_t ou = off[u];
        const int lu = (int)(off[u + 1] - ou);
        const int sl = item.y + threadIdx.x;
        if (threadIdx.x < kItemSlots && sl < row_ptr[u + 1]) {
            const int v = col[sl], e = slot_eid[sl];
            const bool listed = emark ? emark[e] == stamp : e >= e0 && e < e1;
            const int lv = (int)(off[v + 1] - off[v]);
            // the endpoint with the larger ball owns the edge: the smaller list is streamed
            if (listed && (lu > lv || (lu == lv && u < v))) s_slot[atomicAdd(&s_n, 1)] = sl;
        }
        __syncthreads();
        const int owned = s_n;
        if (owned > 0) {
            const int32_t *pu = P + ou;
            if (lu <= pcap) {
                for (int j = threadIdx.x; j < lu; j += blockDim.x) sp[j] = pu[j];
                pu = sp;
            }
            ball.load(members + ou, lu);
            __syncthreads();
            for (;;) {
                int k = 0;
                if (lane == 0) k = atomicAdd(&s_next, 1);
                k = __shfl_sync(0xffffffffu, k, 0);
                if (k >= owned) break;
                const int s = s_slot[k], v = col[s], e = slot_eid[s];
                const int64_t ov = off[v];
                const int lv = (int)(off[v + 1] - ov);
                const int32_t *mv = members + ov, *pv = P + ov;
                int cnt = 0;
                for (int j0 = 0; j0 < lv; j0 += 32) {
                    const int j = j0 + lane;
                    int val = -1;
                    if (j < lv) {
                        const int w = mv[j];
                        const int iu = (w != u && w != v) ? ball.find(w) : -1;
                        if (iu >= 0) val = min(pu[iu], pv[j]);
                    }
                    const unsigned b = __ballot_sync(0xffffffffu, val >= 0);
                    if (val >= 0) vals[cnt + __popc(b & lanemask_lt())] = val;
                    cnt += __popc(b);
                }
                __syncwarp();
                // H = largest y in [0, cnt] with at least y values >= y; it is at most the old key
                const int old = key_in[e];
                int lo = 0, hi = cnt + 1, step = 1, mid = min(old, cnt);
                while (hi - lo > 1) {
                    int c = 0;
                    for (int j = lane; j < cnt; j += 32) c += vals[j] >= mid;
                    c = warp_sum(c);
                    if (c >= mid) {
                        lo = mid;
                        if (mid == old) break;  // keys never increase
                        step = 0;
                    } else {
                        hi = mid;
                    }
                    if (step > 0) {
                        mid = max(hi - step, (lo + hi) >> 1);
                        step *= 2;
                    } else {
                        mid = (lo + hi) >> 1;
                    }
                }
                if (lane == 0) {
                    if (lo != old) nchg++;
                    key_out[e] = lo;
                }
                __syncwarp();
            }
            __syncthreads();
            ball.unload();
        }
        __syncthreads();
    }
    if (lane == 0 && nchg) atomicAdd(changed, nchg);
}

// Vertices touched by the edges [e0, e1) (both endpoints), each listed once.
__global__ void k_hx_touch(int64_t e0, int64_t e1, const int32_t *__restrict__ eu,
                           const int32_t *__restrict__ ev, int32_t stamp, int32_t *mark,
                           int32_t *list, int32_t *count) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = e0 + blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); i0 < e1; i0 += stride) {
        const int64_t i = i0 + (threadIdx.x & 31);
        const int a = i < e1 ? eu[i] : 0, b = i < e1 ? ev[i] : 0;
        warp_append(i < e1 && atomicExch(&mark[a], stamp) != stamp, a, count, list);
        warp_append(i < e1 && atomicExch(&mark[b], stamp) != stamp, b, count, list);
    }
}

// Pruning, step 1: per vertex, the range of the values that fell at its edges in the
// previous order: hi = largest H^(n-2), lo = smallest H^(n-1) over its edges that changed.
__global__ void k_hx_fall(int64_t m, const int32_t *__restrict__ eu, const int32_t *__restrict__ ev,
                          const int32_t *__restrict__ kold, const int32_t *__restrict__ kcur,
                          int32_t *hi, int32_t *lo) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const int a = kold[e], b = kcur[e];
        if (a == b) continue;
        atomicMax(&hi[eu[e]], a);
        atomicMin(&lo[eu[e]], b);
        atomicMax(&hi[ev[e]], a);
        atomicMin(&lo[ev[e]], b);
    }
}

// Pruning, step 2 (h-1 times): one hop of spreading, warp per vertex: the range of x
// becomes the hull of the ranges of x and its neighbours.
__global__ void __launch_bounds__(kBlock) k_hx_spread(int32_t n, const int32_t *__restrict__ row_ptr,
                                                     const int32_t *__restrict__ col,
                                                     const int32_t *__restrict__ hi_in,
                                                     const int32_t *__restrict__ lo_in,
                                                     int32_t *__restrict__ hi_out, int32_t *__restrict__ lo_out) {
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = gw; x < n; x += nwarps) {
        int h = lane == 0 ? hi_in[x] : -1, l = lane == 0 ? lo_in[x] : INT_MAX;
        for (int s = row_ptr[x] + lane; s < row_ptr[x + 1]; s += 32) {
            const int y = col[s];
            h = max(h, hi_in[y]);
            l = min(l, lo_in[y]);
        }
        for (int o = 16; o > 0; o >>= 1) {
            h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
            l = min(l, __shfl_xor_sync(0xffffffffu, l, o));
        }
        if (lane == 0) {
            hi_out[x] = h;
            lo_out[x] = l;
        }
    }
}

// Pruning, step 3: an edge e = (u,v) with T = H^(n-1)(e) is listed for computation (emark =
// stamp) when the hull [min(lo(u), lo(v)), max(hi(u), hi(v))] of the fallen values near it
// straddles T (some value went from >= T to < T); otherwise H^(n)(e) = T (Lemma 4).  The
// endpoints of listed edges are listed once each (mark holds the stamp of the order).
__global__ void k_hx_select(int64_t m, const int32_t *__restrict__ eu, const int32_t *__restrict__ ev,
                            const int32_t *__restrict__ kcur, const int32_t *__restrict__ hi,
                            const int32_t *__restrict__ lo, int32_t *knew, int32_t *emark,
                            int32_t *ecount, int32_t stamp, int32_t *mark, int32_t *vlist,
                            int32_t *vcount) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); i0 < m; i0 += stride) {
        const int64_t e = i0 + (threadIdx.x & 31);
        int u = 0, v = 0;
        bool listed = false;
        if (e < m) {
            u = eu[e];
            v = ev[e];
            const int T = kcur[e];
            const int l = min(lo[u], lo[v]), hh = max(hi[u], hi[v]);
            listed = l < T && T <= hh;
            if (listed) emark[e] = stamp;
            else knew[e] = T;
        }
        const unsigned b = __ballot_sync(0xffffffffu, listed);
        if ((threadIdx.x & 31) == 0 && b) atomicAdd(ecount, __popc(b));
        const bool fu = listed && atomicExch(&mark[u], stamp) != stamp;
        const bool fv = listed && atomicExch(&mark[v], stamp) != stamp;
        warp_append(fu, u, vcount, vlist);
        warp_append(fv, v, vcount, vlist);
    }
}

// t(e,h) = H(e) + 2 at the fixed point (Theorem 4).
__global__ void k_hx_truss(int64_t m, const int32_t *__restrict__ hv, int32_t *__restrict__ t) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
        t[e] = hv[e] + 2;
}

#define HX_CHECK(...)                                                               \
    do {                                                                             \
        cudaError_t _e = (__VA_ARGS__);                                              \
        if (_e != cudaSuccess) {                                                     \
            set_last_error(std::string("htd_hindex_decompose: ") + #__VA_ARGS__ + ": " + \
                           cudaGetErrorString(_e));                                   \
            st = (_e == cudaErrorMemoryAllocation) ? HTD_ENOMEM : HTD_ECUDA;         \
            goto done;                                                               \
        }                                                                            \
    } while (0)

}  // namespace

htd_status hindex_run(htd_graph *G, Handle *H, int32_t h, int32_t sweeps, int32_t max_iter, bool prune,
                      int32_t *truss_dev, int32_t *hval_dev, htd_hindex_stats *stats, cudaStream_t s) {
    GraphDev &g = H->g;
    const int64_t n = g.n, m = g.m;
    htd_status st = HTD_OK;
    int32_t *members = nullptr, *P = nullptr, *prev = nullptr, *vals = nullptr;
    int32_t *key = nullptr, *key2 = nullptr, *mark = nullptr, *vlist = nullptr;
    int32_t *kold = nullptr, *hi = nullptr, *lo = nullptr, *hi2 = nullptr, *lo2 = nullptr;
    int32_t *emark = nullptr;
    int64_t *off = nullptr;
    // edges changed in the order; vertices and edges listed
    struct Counters {
        unsigned long long changed;
        int32_t vertices, edges;
        int32_t items, queue;  // of the order's edge kernel
    };
    static_assert(sizeof(Counters) <= sizeof(DevStatus), "read through the handle's pinned status block");
    Counters *dctr = nullptr, *hctr = nullptr;
    cudaEvent_t t0 = nullptr, t1 = nullptr;
    htd_hindex_stats loc;
    std::memset(&loc, 0, sizeof(loc));
    loc.h = h;
    loc.sweeps = sweeps;
    loc.pruned = prune ? 1 : 0;
    int64_t launches = 0;
    PeelWork &w = H->w;
    const int W = (int)std::max<int64_t>(1, (n + 31) / 32);
    int occ_p = 0, occ_e = 0, grid_p = 0, grid_e = 0;
    int64_t total = 0, maxb = 0;
    std::vector<int32_t> hsizes;
    // the ball index (set and ranks) where it leaves room for two blocks an SM, and path keys
    // of up to kPathCap members beside it
    constexpr int32_t kPathCap = 4096;
    const int32_t words = 8 * (int64_t)W <= 90 * 1024 ? W : 0;
    const size_t smem = 8 * (size_t)words + 4 * (size_t)kPathCap;
    if (m == 0) goto finish;
    HX_CHECK(cudaEventCreate(&t0));
    HX_CHECK(cudaEventCreate(&t1));
    HX_CHECK(cudaEventRecord(t0, s));
    {
        // H^(0) = sup(e,h), the h-support of every edge (the initial step of Algorithm 2)
        HX_CHECK(dev_alloc(&key, m, s));
        HX_CHECK(dev_alloc(&key2, m, s));
        htd_status hs = h_support_run(H, h, key, s);
        if (hs != HTD_OK) {
            st = hs;
            goto done;
        }
    }
    hctr = reinterpret_cast<Counters *>(w.status_host);  // the h-support pass is done with it
    HX_CHECK(raise_smem_limit((const void *)k_hx_pathkeys, smem));
    HX_CHECK(raise_smem_limit((const void *)k_hx_edges, smem));
    HX_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_p, k_hx_pathkeys, kBlock, smem));
    HX_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_e, k_hx_edges, kBlock, smem));
    if (occ_p < 1 || occ_e < 1) {
        set_last_error("htd_hindex_decompose: no resident block fits");
        st = HTD_ECUDA;
        goto done;
    }
    grid_p = H->num_sms * std::min(occ_p, 8);
    grid_e = H->num_sms * std::min(occ_e, 8);
    // member lists from the balls the h-support pass left in the handle's scratch
    HX_CHECK(dev_alloc(&off, n + 1, s));
    HX_CHECK(scan_exclusive<int32_t, int64_t>(w.ball_size, off, n, w.scan_tmp, s, &launches));
    hsizes.resize(n);
    HX_CHECK(cudaMemcpyAsync(&total, off + n, 8, cudaMemcpyDeviceToHost, s));
    HX_CHECK(cudaMemcpyAsync(hsizes.data(), w.ball_size, n * 4, cudaMemcpyDeviceToHost, s));
    HX_CHECK(cudaStreamSynchronize(s));
    for (int64_t x = 0; x < n; x++) maxb = std::max<int64_t>(maxb, hsizes[x]);
    loc.ball_entries = total;
    HX_CHECK(dev_alloc(&members, total, s));
    HX_CHECK(dev_alloc(&P, total, s));
    k_hx_members<<<(unsigned)std::min<int64_t>(n, H->num_sms * 8), kBlock, 0, s>>>((int32_t)n, w.W, w.pool, w.ball_off,
                                                                         w.ball_nw, off, members);
    launches++;
    HX_CHECK(cudaGetLastError());
    {
        // one block per vertex at most; prev is only read from the third round on
        grid_p = (int)std::min<int64_t>(grid_p, n);
        grid_e = (int)std::min<int64_t>(grid_e, n);
        HX_CHECK(dev_alloc(&prev, (h >= 3 ? (int64_t)grid_p : 1) * std::max<int64_t>(maxb, 1), s));
        HX_CHECK(dev_alloc(&vals, (int64_t)grid_e * (kBlock / 32) * std::max<int64_t>(maxb, 1), s));
        HX_CHECK(dev_alloc(&dctr, 1, s));
        HX_CHECK(dev_alloc(&mark, n, s));
        HX_CHECK(dev_alloc(&vlist, n, s));
        HX_CHECK(cudaMemsetAsync(mark, 0xff, n * 4, s));
        if (prune) {
            HX_CHECK(dev_alloc(&kold, m, s));
            HX_CHECK(dev_alloc(&hi, n, s));
            HX_CHECK(dev_alloc(&lo, n, s));
            HX_CHECK(dev_alloc(&hi2, n, s));
            HX_CHECK(dev_alloc(&lo2, n, s));
            HX_CHECK(dev_alloc(&emark, m, s));
            HX_CHECK(cudaMemsetAsync(emark, 0xff, m * 4, s));
        }
        const int64_t prev_stride = h >= 3 ? maxb : 0;
        auto pathkeys = [&](const int32_t *list, int32_t count, const int32_t *dcount) {
            k_hx_pathkeys<<<grid_p, kBlock, smem, s>>>(list, count, dcount, h, g.row_ptr, g.col, g.slot_eid, key, off,
                                                       members, P, prev, prev_stride, words, kPathCap);
            launches++;
        };
        // dctr->items and ->queue are zero
        auto edges = [&](const int32_t *list, int32_t count, const int32_t *dcount, int64_t e0, int64_t e1,
                         const int32_t *marks, int32_t stamp, int32_t *out) {
            k_hx_items<<<H->num_sms * 2, kBlock, 0, s>>>(list, count, dcount, g.row_ptr, w.items, &dctr->items);
            k_hx_edges<<<grid_e, kBlock, smem, s>>>(w.items, &dctr->items, &dctr->queue, e0, e1, marks, stamp,
                                                    g.row_ptr, g.col, g.slot_eid, off, members, P, key, out, vals,
                                                    maxb, &dctr->changed, words, kPathCap);
            launches += 2;
        };
        // every order before the fixed point lowers at least one key (Theorem 3): the sum
        // of H^(0) plus one orders always suffice
        std::vector<int32_t> k0(m);
        HX_CHECK(cudaMemcpyAsync(k0.data(), key, m * 4, cudaMemcpyDeviceToHost, s));
        HX_CHECK(cudaStreamSynchronize(s));
        int64_t cap = 1;
        for (int64_t e = 0; e < m; e++) cap += k0[e];
        const int S = std::max(1, sweeps);
        int32_t stamp = 0;
        int32_t it = 0;
        bool converged = false;
        while (!converged && (max_iter < 0 || it < max_iter) && it < cap) {
            HX_CHECK(cudaMemsetAsync(dctr, 0, sizeof(Counters), s));
            const bool pruned = S == 1 && prune && it > 0;
            if (pruned) {
                // Lemma 4: list the edges that can still fall (key = H^(n-1), kold = H^(n-2))
                HX_CHECK(cudaMemsetAsync(hi, 0xff, n * 4, s));
                HX_CHECK(cudaMemsetAsync(lo, 0x7f, n * 4, s));
                k_hx_fall<<<H->num_sms * 4, kBlock, 0, s>>>(m, g.eu, g.ev, kold, key, hi, lo);
                launches++;
                for (int r = 1; r < h; r++) {
                    k_hx_spread<<<H->num_sms * 8, kBlock, 0, s>>>((int32_t)n, g.row_ptr, g.col, hi, lo, hi2, lo2);
                    launches++;
                    std::swap(hi, hi2);
                    std::swap(lo, lo2);
                }
                k_hx_select<<<H->num_sms * 4, kBlock, 0, s>>>(m, g.eu, g.ev, key, hi, lo, key2, emark, &dctr->edges,
                                                             stamp, mark, vlist, &dctr->vertices);
                launches++;
                pathkeys(vlist, 0, &dctr->vertices);
                edges(vlist, 0, &dctr->vertices, 0, m, emark, stamp, key2);
                stamp++;
            } else if (S == 1) {
                pathkeys(nullptr, (int32_t)n, nullptr);
                edges(nullptr, (int32_t)n, nullptr, 0, m, nullptr, 0, key2);
                loc.edge_evals += m;
                loc.vertex_evals += n;
            } else {
                for (int j = 0; j < S; j++) {
                    const int64_t e0 = m * j / S, e1 = m * (j + 1) / S;
                    if (e1 <= e0) continue;
                    HX_CHECK(cudaMemsetAsync(&dctr->vertices, 0, sizeof(Counters) - sizeof(dctr->changed), s));
                    k_hx_touch<<<H->num_sms * 2, kBlock, 0, s>>>(e0, e1, g.eu, g.ev, stamp++, mark, vlist,
                                                                &dctr->vertices);
                    launches++;
                    HX_CHECK(cudaMemcpyAsync(hctr, dctr, sizeof(Counters), cudaMemcpyDeviceToHost, s));
                    HX_CHECK(cudaStreamSynchronize(s));
                    pathkeys(vlist, hctr->vertices, nullptr);
                    edges(vlist, hctr->vertices, nullptr, e0, e1, nullptr, 0, key);
                    loc.edge_evals += e1 - e0;
                    loc.vertex_evals += hctr->vertices;
                }
            }
            HX_CHECK(cudaGetLastError());
            HX_CHECK(cudaMemcpyAsync(hctr, dctr, sizeof(Counters), cudaMemcpyDeviceToHost, s));
            HX_CHECK(cudaStreamSynchronize(s));
            if (pruned) {
                loc.edge_evals += hctr->edges;
                loc.vertex_evals += hctr->vertices;
            }
            if (S == 1) {
                if (prune) std::swap(kold, key);  // H^(n-2) <- H^(n-1) <- H^(n)
                std::swap(key, key2);
            }
            it++;
            if (hctr->changed == 0) converged = true;
        }
        loc.iterations = it;
        loc.converged = converged ? 1 : 0;
    }
    if (hval_dev) HX_CHECK(cudaMemcpyAsync(hval_dev, key, m * 4, cudaMemcpyDeviceToDevice, s));
    if (truss_dev) {
        k_hx_truss<<<H->num_sms * 2, kBlock, 0, s>>>(m, key, truss_dev);
        launches++;
        HX_CHECK(cudaGetLastError());
    }
    HX_CHECK(cudaEventRecord(t1, s));
    HX_CHECK(cudaEventSynchronize(t1));
    {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, t0, t1);
        loc.ms_total = ms;
    }
finish:
    loc.kernel_launches = launches;
    if (stats) *stats = loc;
    add_launches(launches);
done:
    dev_free(off, s);
    dev_free(members, s);
    dev_free(P, s);
    dev_free(prev, s);
    dev_free(vals, s);
    dev_free(key, s);
    dev_free(key2, s);
    dev_free(mark, s);
    dev_free(vlist, s);
    dev_free(kold, s);
    dev_free(hi, s);
    dev_free(lo, s);
    dev_free(hi2, s);
    dev_free(lo2, s);
    dev_free(emark, s);
    dev_free(dctr, s);
    if (t0) cudaEventDestroy(t0);
    if (t1) cudaEventDestroy(t1);
    return st;
}

}  // namespace htd
