// htd_peel.cu -- h-hop balls, h-support and level-synchronous peeling on the device.
//
// Notation (Sec. 2): B(x,h) = x plus every vertex within distance h of x over the alive
// edges, so N(x,h) = B(x,h) \ {x} and, for an alive edge e = (u,v),
//     sup(e,h) = |N(u,h) ∩ N(v,h)| = |B(u,h) ∩ B(v,h)| - 2            (Def. 2, Def. 3)
// because u and v lie in both balls.
//
// Balls are materialised per vertex as n-bit sets, stored either dense (W words) or as a
// sorted list of (word index, word) pairs when that is at most W words; the choice is
// remade at every rebuild and always fits the storage reserved by the first build,
// because balls only shrink as edges are removed.
//
// One peel round (Sec. 3, Algorithm 1 with every edge of level k removed together):
//   select     F = alive edges with sup <= k-2 (k = max(k, min alive sup + 2));
//   candidates vertices within distance h-1 of an endpoint of F, before removal: only
//              their balls can lose members (a lost shortest path of length <= h runs
//              through a removed edge, so its start is within h-1 of that edge);
//   remove     t(e) = k, stamp(e) = round, the edge's two adjacency slots are marked dead;
//   rebuild    every candidate's ball; a ball that shrank marks its vertex "changed";
//   recompute  sup(e) for every alive edge with a changed endpoint (sup depends only on
//              the two balls), owned by one endpoint so each edge is computed once;
//   reduce     min alive sup and alive count; the host polls them between graph launches.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include "htd_internal.h"
#include "htd_round.cuh"
#include "htd_scan.cuh"

namespace htd {
namespace {

constexpr int kBlock = 256;
constexpr int kNWarps = kBlock / 32;
constexpr int kItemChunk = 64;  // adjacency slots per h-support work item

enum BallMode { kModeCount = 0, kModeStore = 1, kModeRebuild = 2 };

struct BallArgs {
    int32_t n, W, Wpad, h;
    int32_t count_bytes;
    int32_t force_dense;  // store every ball dense whatever its size
    const int32_t *row_ptr;
    const int32_t *col_live;
    const int32_t *deg_alive;
    uint32_t *pool;
    uint32_t *pool_new;   // nullable: a second copy of every dense ball stored
    int64_t *ball_off;
    int32_t *ball_need;
    int32_t *ball_size;
    int32_t *ball_nw;
    int2 *ball_meta;
    const int32_t *cand_list;
    int32_t *changed_list;
    int32_t *changed_stamp;
    int32_t *bfs_lists;
    int64_t bfs_list_len;
    // Adjacency rows as n-bit sets (nullable; h = 2, first build only): a neighbour of degree
    // or_deg or more is expanded by ORing its row, row_of[y] (null: row y).
    const uint32_t *rows;
    const int32_t *row_of;
    int32_t or_deg;
    int32_t bump;           // storage is taken from the pool in the order of completion; the pool
                            // has room for all of it (bound_storage, or an earlier pass)
    const uint32_t *inner;  // k_ball_or: dense balls of radius h - 1, row x at x * Wpad
    DevStatus *st;
};

// Sets bit z of the block's n-bit set; returns true if this thread set it first.
__device__ __forceinline__ bool set_member(uint32_t *bits, int32_t z) {
    const uint32_t m = 1u << (z & 31);
    uint32_t *w = bits + (z >> 5);
    if (*(volatile uint32_t *)w & m) return false;
    return (atomicOr(w, m) & m) == 0u;
}

// Load-balanced expansion of up to kBlock frontier vertices (one per thread, -1 = none):
// every alive neighbour z of them is set in `bits`; if `next` is non-null, vertices set
// for the first time are appended to it.  Consecutive threads read consecutive slots.
__device__ __forceinline__ void expand_chunk(int32_t y, const int32_t *__restrict__ row_ptr,
                                             const int32_t *__restrict__ col_live,
                                             uint32_t *bits, int32_t *s_off, int32_t *s_beg,
                                             int32_t *s_scan, int32_t *next,
                                             int32_t *next_cnt) {
    int beg = 0, len = 0;
    if (y >= 0) {
        beg = row_ptr[y];
        len = row_ptr[y + 1] - beg;
    }
    int total;
    const int off = block_exclusive_scan<kBlock, int>(len, &total, s_scan);
    s_off[threadIdx.x] = off;
    s_beg[threadIdx.x] = beg;
    __syncthreads();
    for (int t = threadIdx.x; t < total; t += kBlock) {
        int lo = 0, hi = kBlock - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (s_off[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        const int z = col_live[s_beg[lo] + (t - s_off[lo])];
        bool fresh = false;
        if (z >= 0) fresh = set_member(bits, z);
        if (next) warp_append(fresh, z, next_cnt, next);
    }
    __syncthreads();
}

// Stores B(x,h) from the block's n-bit set: its size and form, then dense or as (word index,
// word) pairs (kModeCount: only the storage it needs; kModeRebuild: only if it shrank).
template <int MODE>
__device__ __forceinline__ void store_ball(const BallArgs &a, int x, uint32_t *bits, int32_t *s_wsz,
                                           int32_t *s_wnz, int64_t *s_off64) {
    DevStatus *st = a.st;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int W = a.W;
    const int seg = ((W + kNWarps - 1) / kNWarps + 31) & ~31;
    uint4 *bits4 = reinterpret_cast<uint4 *>(bits);
    // ball size and non-zero words, per warp segment of words
    const int w0 = wid * seg, w1 = min(W, w0 + seg);
    int sz = 0, nz = 0;
#pragma unroll 4
    for (int i = w0 + lane; i < w1; i += 32) {
        const uint32_t w = bits[i];
        sz += __popc(w);
        nz += (w != 0u);
    }
    sz = warp_sum(sz);
    nz = warp_sum(nz);
    if (lane == 0) {
        s_wsz[wid] = sz;
        s_wnz[wid] = nz;
    }
    __syncthreads();
    int size = 0, nzw = 0, wbase = 0;
#pragma unroll
    for (int j = 0; j < kNWarps; j++) {
        size += s_wsz[j];
        nzw += s_wnz[j];
        if (j < wid) wbase += s_wnz[j];
    }
    const bool dense = a.force_dense || 2 * nzw > W;
    const int stor = dense ? a.Wpad : ((2 * nzw + 3) & ~3);
    bool store = true;
    if (MODE == kModeCount) {
        if (threadIdx.x == 0) a.ball_need[x] = stor;
        store = false;
    } else if (MODE == kModeRebuild) {
        const int old = a.ball_size[x];
        if (size == old) store = false;
        else if (size > old) {
            if (threadIdx.x == 0) atomicOr(&st->err, kErrBallGrew);
            store = false;
        }
    }
    if (store) {
        int64_t off, cap = stor;
        if (MODE == kModeStore && a.bump) {
            if (threadIdx.x == 0) *s_off64 = (int64_t)atomicAdd((unsigned long long *)&st->pool_next,
                                                                (unsigned long long)stor);
            __syncthreads();
            off = *s_off64;
            if (threadIdx.x == 0) a.ball_off[x] = off;
        } else {
            off = a.ball_off[x];
            cap = a.ball_off[x + 1] - off;
        }
        if (stor > cap) {
            if (threadIdx.x == 0) atomicOr(&st->err, kErrBallCapacity);
        } else if (dense) {
            uint4 *dst = reinterpret_cast<uint4 *>(a.pool + off);
#pragma unroll 4
            for (int i = threadIdx.x; i < (a.Wpad >> 2); i += kBlock) dst[i] = bits4[i];
            if (a.pool_new) {
                uint4 *twin = reinterpret_cast<uint4 *>(a.pool_new + off);
                for (int i = threadIdx.x; i < (a.Wpad >> 2); i += kBlock) twin[i] = bits4[i];
            }
        } else {
            uint2 *dst = reinterpret_cast<uint2 *>(a.pool + off);
            int run = wbase;
#pragma unroll 4
            for (int i0 = w0; i0 < w1; i0 += 32) {
                const int i = i0 + lane;
                const uint32_t w = (i < w1) ? bits[i] : 0u;
                const unsigned bal = __ballot_sync(0xffffffffu, w != 0u);
                if (w != 0u) dst[run + __popc(bal & lanemask_lt())] = make_uint2((uint32_t)i, w);
                run += __popc(bal);
            }
        }
        if (threadIdx.x == 0 && stor <= cap) {
            if (MODE == kModeStore) atomicAdd((unsigned long long *)&st->st_ball_total,
                                              (unsigned long long)size);
            a.ball_size[x] = size;
            a.ball_nw[x] = dense ? -1 : nzw;
            a.ball_meta[x] = make_int2((int)(off >> 2), dense ? -1 : nzw);
            if (MODE == kModeRebuild) {
                a.changed_stamp[x] = st->round;
                a.changed_list[atomicAdd(&st->nchanged, 1)] = x;
            }
        }
    }
}

// Builds B(x,h) for a list of vertices, one vertex per block at a time (work queue).
//   kModeCount:   records the storage words the ball needs (first pass);
//   kModeStore:   stores the ball at its reserved offset (second pass);
//   kModeRebuild: rebuilds a peel candidate; stores it and marks x changed iff it shrank.
// The builds are bound by the expansions (about 160 G adjacency slots/s).  On hub graphs most
// of them expand the same few rows: with the rows of degree W/16 and more as n-bit sets
// (L2-resident: 988 rows, 32 MB on R-MAT 18) their share becomes W/4 16-byte loads each.
// Four blocks per SM leave the compiler registers for loads in flight (R-MAT 8,192 by rebuilds
// at h = 2 825 -> 790 ms; it takes 32 registers when left to itself).
template <int MODE>
__global__ void __launch_bounds__(kBlock, 4) k_ball(BallArgs a) {
    extern __shared__ __align__(16) uint32_t bits[];
    __shared__ int32_t s_scan[kNWarps];
    __shared__ int32_t s_off[kBlock], s_beg[kBlock];
    __shared__ int32_t s_item;
    __shared__ int32_t s_cnt[2];
    __shared__ int32_t s_wsz[kNWarps], s_wnz[kNWarps];
    __shared__ unsigned long long s_bytes;
    __shared__ int64_t s_off64;
    __shared__ int32_t s_or[kBlock], s_nor;
    const bool by_rows = MODE != kModeRebuild && a.rows != nullptr && a.h == 2;

    DevStatus *st = a.st;
    int count;
    int32_t *queue;
    if (MODE == kModeRebuild) {
        if (st->alive == 0) return;
        count = 0;
        for (int j = 0; j < a.h && j < kMaxH; j++) count += st->cand_cnt[j];
        queue = &st->q_ball;
    } else {
        count = a.n;
        queue = (MODE == kModeCount) ? &st->q_count : &st->q_store;
    }
    const int lane = threadIdx.x & 31;
    int32_t *lists[2] = {nullptr, nullptr};
    if (a.h >= 3) {
        lists[0] = a.bfs_lists + (int64_t)blockIdx.x * 2 * a.bfs_list_len;
        lists[1] = lists[0] + a.bfs_list_len;
    }
    if (threadIdx.x == 0) s_bytes = 0ull;
    unsigned long long bytes = 0ull;  // per-thread share of the algorithmic bytes

    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(queue, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= count) break;
        const int x = (MODE == kModeRebuild) ? a.cand_list[it] : it;

        uint4 *bits4 = reinterpret_cast<uint4 *>(bits);
#pragma unroll 4
        for (int i = threadIdx.x; i < (a.Wpad >> 2); i += kBlock) bits4[i] = make_uint4(0, 0, 0, 0);
        if (threadIdx.x == 0) {
            s_cnt[0] = 0;
            s_cnt[1] = 0;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            atomicOr(&bits[x >> 5], 1u << (x & 31));
            if (a.count_bytes && a.h >= 2) bytes += 8ull + 4ull * (unsigned)a.deg_alive[x];
        }
        // depth 1 (x's alive neighbours) and depth 2 (their neighbours)
        const int rb = a.row_ptr[x], re = a.row_ptr[x + 1];
        for (int c = rb; c < re; c += kBlock) {
            const int s = c + threadIdx.x;
            int y = -1;
            if (s < re) {
                y = a.col_live[s];
                if (y < 0) y = -1;
            }
            if (y >= 0) {
                set_member(bits, y);
                if (a.count_bytes && a.h >= 2) bytes += 8ull + 4ull * (unsigned)a.deg_alive[y];
            }
            if (a.h >= 2) {
                if (by_rows) {
                    // hubs among the neighbours are set aside: their rows are ORed in below
                    if (threadIdx.x == 0) s_nor = 0;
                    __syncthreads();
                    if (y >= 0 && a.row_ptr[y + 1] - a.row_ptr[y] >= a.or_deg) {
                        const int r = a.row_of ? a.row_of[y] : y;
                        if (r >= 0) {
                            s_or[atomicAdd(&s_nor, 1)] = r;
                            y = -1;
                        }
                    }
                }
                expand_chunk(y, a.row_ptr, a.col_live, bits, s_off, s_beg, s_scan,
                             a.h >= 3 ? lists[0] : nullptr, &s_cnt[0]);
                if (by_rows && s_nor > 0) {
                    const int W4 = a.Wpad >> 2, nor = s_nor;
                    const uint4 *rows4 = reinterpret_cast<const uint4 *>(a.rows);
                    for (int i = threadIdx.x; i < W4; i += kBlock) {
                        uint4 v = bits4[i];
                        for (int k = 0; k < nor; k++) {
                            const uint4 r = rows4[(int64_t)s_or[k] * W4 + i];
                            v.x |= r.x;
                            v.y |= r.y;
                            v.z |= r.z;
                            v.w |= r.w;
                        }
                        bits4[i] = v;
                    }
                    __syncthreads();
                }
            }
        }
        // depth 3..h from the level lists
        for (int d = 3; d <= a.h; d++) {
            const int cur = (d - 3) & 1, nxt = cur ^ 1;
            __syncthreads();
            const int ncur = s_cnt[cur];
            __syncthreads();
            if (threadIdx.x == 0) s_cnt[nxt] = 0;
            __syncthreads();
            for (int c = 0; c < ncur; c += kBlock) {
                const int i = c + threadIdx.x;
                const int y = (i < ncur) ? lists[cur][i] : -1;
                if (a.count_bytes && y >= 0) bytes += 8ull + 4ull * (unsigned)a.deg_alive[y];
                expand_chunk(y, a.row_ptr, a.col_live, bits, s_off, s_beg, s_scan,
                             d < a.h ? lists[nxt] : nullptr, &s_cnt[nxt]);
            }
        }
        __syncthreads();

        store_ball<MODE>(a, x, bits, s_wsz, s_wnz, &s_off64);
        __syncthreads();
    }
    if (a.count_bytes) {
        unsigned long long b = bytes;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
        if (lane == 0 && b) atomicAdd(&s_bytes, b);
        __syncthreads();
        if (threadIdx.x == 0 && s_bytes) atomicAdd(&st->st_bytes_ball, s_bytes);
    }
}

// B(x,h) for every vertex as the OR of its own and its neighbours' dense balls of radius
// h - 1, one vertex per block at a time: 2m rows of W words are read, coalesced, whatever the
// radius, where the search by levels of k_ball visits every slot of every vertex within h - 1.
// Four blocks per SM leave the compiler registers for the rows' loads: DC-SBM 200k at h = 3
// 22.5 -> 19.6 ms, R-MAT 16 6.7 -> 5.8 ms for the whole h-support.
__global__ void __launch_bounds__(kBlock, 4) k_ball_or(BallArgs a) {
    extern __shared__ __align__(16) uint32_t bits[];
    __shared__ int32_t s_item, s_row[kBlock];
    __shared__ int32_t s_wsz[kNWarps], s_wnz[kNWarps];
    __shared__ int64_t s_off64;
    DevStatus *st = a.st;
    uint4 *bits4 = reinterpret_cast<uint4 *>(bits);
    const uint4 *in4 = reinterpret_cast<const uint4 *>(a.inner);
    const int W4 = a.Wpad >> 2;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(&st->q_store, 1);
        __syncthreads();
        const int x = s_item;
        if (x >= a.n) break;
        const int rb = a.row_ptr[x], re = a.row_ptr[x + 1];
        for (int c = rb; c == rb || c < re; c += kBlock) {
            const int cnt = min(kBlock, re - c);
            if (threadIdx.x < cnt) s_row[threadIdx.x] = a.col_live[c + threadIdx.x];
            __syncthreads();
            for (int i = threadIdx.x; i < W4; i += kBlock) {
                uint4 v = c == rb ? in4[(int64_t)x * W4 + i] : bits4[i];
#pragma unroll 4
                for (int k = 0; k < cnt; k++) {
                    const uint4 r = in4[(int64_t)s_row[k] * W4 + i];
                    v.x |= r.x;
                    v.y |= r.y;
                    v.z |= r.z;
                    v.w |= r.w;
                }
                bits4[i] = v;
            }
            __syncthreads();
        }
        store_ball<kModeStore>(a, x, bits, s_wsz, s_wnz, &s_off64);
        __syncthreads();
    }
}

// Offsets of dense balls: x * Wpad.
__global__ void k_dense_offsets(int64_t n, int64_t Wpad, int64_t *__restrict__ off) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x <= n; x += (int64_t)gridDim.x * blockDim.x)
        off[x] = x * Wpad;
}

// Upper bounds of the ball sizes, for storage without a counting pass: |B(x,1)| = degree + 1, and
// |B(x,r)| is at most the sum of |B(y,r-1)| over the neighbours y of x (1 without any).  Sums stop
// at `cap`, from which on a ball may be dense.  One warp per vertex.
__global__ void __launch_bounds__(kBlock) k_ball_bound(int32_t n, int32_t cap, const int32_t *__restrict__ row_ptr,
                                                      const int32_t *__restrict__ col,
                                                      const int32_t *__restrict__ inner,
                                                      int32_t *__restrict__ bound) {
    const int lane = threadIdx.x & 31, nwarps = gridDim.x * (blockDim.x >> 5);
    for (int x = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < n; x += nwarps) {
        const int rb = row_ptr[x], re = row_ptr[x + 1];
        int sum = 0;
        if (!inner) {
            sum = re - rb + 1;
        } else {
            for (int s0 = rb; s0 < re && sum < cap; s0 += 128) {
                int v = 0;  // 128 values of at most `cap`, about n / 32
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int s = s0 + 32 * j + lane;
                    if (s < re) v += inner[col[s]];
                }
                sum += __reduce_add_sync(0xffffffffu, v);
            }
            sum = max(sum, 1);
        }
        if (lane == 0) bound[x] = min(sum, cap);
    }
}

// Storage of balls of at most the given sizes: dense, or a (word index, word) pair per member.  A
// ball is stored as pairs when these take at most its W words, and a word holds a member at least,
// so that store_ball never takes more (tests/test_ball_bound.py).
__global__ void __launch_bounds__(kBlock) k_bound_words(int32_t n, int32_t Wpad, const int32_t *__restrict__ bound,
                                                       DevStatus *st) {
    unsigned long long words = 0ull;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += gridDim.x * blockDim.x)
        words += (unsigned)min(Wpad, (2 * bound[x] + 3) & ~3);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) words += __shfl_xor_sync(0xffffffffu, words, o);
    if ((threadIdx.x & 31) == 0 && words) atomicAdd((unsigned long long *)&st->ball_bound, words);
}

// Vertices of degree `deg` and more get a row (at most `cap` of them); the others none.
__global__ void k_or_rows(int32_t n, const int32_t *__restrict__ row_ptr, int32_t deg, int32_t cap,
                          int32_t *__restrict__ row_of, int32_t *__restrict__ list, int32_t *__restrict__ count) {
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += gridDim.x * blockDim.x) {
        int r = -1;
        if (row_ptr[x + 1] - row_ptr[x] >= deg) {
            r = atomicAdd(count, 1);
            if (r < cap) list[r] = x;
            else r = -1;
        }
        row_of[x] = r;
    }
}

struct HsupArgs {
    int32_t n, W, Wpad;
    int32_t initial;
    int32_t count_bytes;
    const int32_t *row_ptr;
    const int32_t *col_live;
    const int32_t *slot_eid;
    const uint32_t *pool;
    const int64_t *ball_off;
    const int32_t *ball_size;
    const int32_t *ball_nw;
    const int32_t *changed_stamp;
    const int2 *items;
    int32_t *sup;
    DevStatus *st;
};

// h-support of the edges of each work item (vertex x, run of x's adjacency slots).  The
// block loads B(x,h) into shared memory as a dense set; each warp takes one slot, and if
// x owns the edge it streams the other endpoint's stored ball against it:
//   sup(e) = popc(B(x) & B(y)) - 2.
// Ownership: x owns (x,y) if y's ball did not change this round, else the endpoint with
// the larger stored ball owns it (ties: smaller id).  In the initial pass every ball
// counts as changed, so each edge is computed exactly once.
// Bound by the rows it streams.  Four loads in flight at six blocks per SM: R-MAT 18 at h = 2
// 17.1 -> 16.9 ms for the whole h-support, DC-SBM 40k at h = 3 1.49 -> 1.41 ms; at five blocks R-MAT
// 18 takes 14.7 ms, but graphs of short balls 5% more (ER n = 200,000 at h = 2 2.90 -> 3.04 ms).
__global__ void __launch_bounds__(kBlock, 6) k_hsup(HsupArgs a) {
    extern __shared__ __align__(16) uint32_t bits[];
    __shared__ int32_t s_item;
    __shared__ unsigned long long s_bytes;
    __shared__ int32_t s_owned;
    DevStatus *st = a.st;
    if (!a.initial && st->alive == 0) return;
    const int nitems = st->nitems;
    const int round = st->round;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int W = a.W;
    uint4 *bits4 = reinterpret_cast<uint4 *>(bits);
    const uint4 *pool4 = reinterpret_cast<const uint4 *>(a.pool);
    const uint2 *pool2 = reinterpret_cast<const uint2 *>(a.pool);
    if (threadIdx.x == 0) {
        s_bytes = 0ull;
        s_owned = 0;
    }
    unsigned long long bytes = 0ull;
    int owned = 0;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(&st->q_items, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= nitems) break;
        const int2 item = a.items[it];
        const int x = item.x;
        const int nwx = a.ball_nw[x];
        const int64_t offx = a.ball_off[x];
        if (nwx < 0) {
            for (int i = threadIdx.x; i < (a.Wpad >> 2); i += kBlock) bits4[i] = pool4[(offx >> 2) + i];
        } else {
            for (int i = threadIdx.x; i < (a.Wpad >> 2); i += kBlock) bits4[i] = make_uint4(0, 0, 0, 0);
            __syncthreads();
            for (int j = threadIdx.x; j < nwx; j += kBlock) {
                const uint2 p = pool2[(offx >> 1) + j];
                bits[p.x] = p.y;
            }
        }
        __syncthreads();
        const int storx = nwx < 0 ? W : 2 * nwx;
        const int s1 = min(a.row_ptr[x + 1], item.y + kItemChunk);
        for (int s = item.y + wid; s < s1; s += kNWarps) {
            const int y = a.col_live[s];
            if (y < 0) continue;
            const bool ychanged = a.initial || a.changed_stamp[y] == round;
            const int nwy = a.ball_nw[y];
            const int story = nwy < 0 ? W : 2 * nwy;
            const bool own = !ychanged || storx > story || (storx == story && x < y);
            if (!own) continue;
            const int64_t offy = a.ball_off[y];
            int cnt = 0;
            if (nwy < 0) {
                const uint4 *p = pool4 + (offy >> 2);
#pragma unroll 4
                for (int i = lane; i < (a.Wpad >> 2); i += 32) {
                    const uint4 v = p[i];
                    const uint4 b = bits4[i];
                    cnt += __popc(v.x & b.x) + __popc(v.y & b.y) + __popc(v.z & b.z) +
                           __popc(v.w & b.w);
                }
            } else {
                const uint2 *p = pool2 + (offy >> 1);
#pragma unroll 4
                for (int j = lane; j < nwy; j += 32) {
                    const uint2 v = p[j];
                    cnt += __popc(bits[v.x] & v.y);
                }
            }
            cnt = warp_sum(cnt);
            if (lane == 0) {
                a.sup[a.slot_eid[s]] = cnt - 2;
                owned++;
                if (a.count_bytes)
                    bytes += 4ull * (unsigned)(story) + 12ull;
            }
        }
        if (a.count_bytes && threadIdx.x == 0) bytes += 4ull * (unsigned)storx;
        __syncthreads();
    }
    if (lane == 0 && owned) atomicAdd(&s_owned, owned);
    if (a.count_bytes) {
        unsigned long long b = bytes;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
        if (lane == 0 && b) atomicAdd(&s_bytes, b);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (a.count_bytes && s_bytes) {
            atomicAdd(&st->st_bytes_hsup, s_bytes);
            if (a.initial) atomicAdd(&st->st_bytes_hsup_init, s_bytes);
        }
        if (!a.initial && s_owned) atomicAdd((unsigned long long *)&st->st_recomputed,
                                             (unsigned long long)s_owned);
    }
}

// Work items for k_hsup: every vertex of `list` (all vertices if list is null) gets one
// item per kItemChunk adjacency slots.  One atomic per warp.
__global__ void k_make_items(const int32_t *__restrict__ list, int32_t initial, int32_t n,
                             const int32_t *__restrict__ row_ptr, int2 *__restrict__ items,
                             DevStatus *st) {
    if (!initial && st->alive == 0) return;
    const int count = list ? st->nchanged : n;
    const int lane = threadIdx.x & 31;
    const int stride = gridDim.x * blockDim.x;
    for (int i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < count; i0 += stride) {
        const int i = i0 + lane;
        int x = -1, rb = 0, nch = 0;
        if (i < count) {
            x = list ? list[i] : i;
            rb = row_ptr[x];
            nch = (row_ptr[x + 1] - rb + kItemChunk - 1) / kItemChunk;
        }
        int incl = nch;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const int tot = __shfl_sync(0xffffffffu, incl, 31);
        int base = 0;
        if (lane == 31 && tot) base = atomicAdd(&st->nitems, tot);
        base = __shfl_sync(0xffffffffu, base, 31);
        const int first = base + incl - nch;
        for (int c = 0; c < nch; c++) items[first + c] = make_int2(x, rb + c * kItemChunk);
    }
}

__global__ void k_select(const int32_t *__restrict__ sup, int64_t m, DevStatus *st,
                         int32_t *__restrict__ frontier) {
    if (st->alive == 0 || st->cont) return;  // a continued round keeps its frontier
    const int thr = st->k - 2;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); e0 < m; e0 += stride) {
        const int64_t e = e0 + (threadIdx.x & 31);
        const bool p = e < m && sup[e] <= thr;
        warp_append(p, (int32_t)e, &st->nF, frontier);
    }
}

__device__ __forceinline__ void cand_mark(bool pred, int32_t w, int round, int level,
                                          int base, int32_t *cand_stamp, int32_t *cand_list,
                                          DevStatus *st) {
    bool fresh = pred && atomicExch(&cand_stamp[w], round) != round;
    warp_append(fresh, w, &st->cand_cnt[level], cand_list + base);
}

// Depth 0 of the candidate search: both endpoints of every frontier edge.
__global__ void k_cand_init(const int32_t *__restrict__ frontier, const int32_t *__restrict__ eu,
                            const int32_t *__restrict__ ev, DevStatus *st,
                            int32_t *__restrict__ cand_stamp, int32_t *__restrict__ cand_list) {
    if (st->alive == 0) return;
    const int nF = st->nF, round = st->round;
    const int stride = gridDim.x * blockDim.x;
    for (int i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < nF; i0 += stride) {
        const int i = i0 + (threadIdx.x & 31);
        const bool p = i < nF;
        const int e = p ? frontier[i] : 0;
        cand_mark(p, p ? eu[e] : 0, round, 0, 0, cand_stamp, cand_list, st);
        cand_mark(p, p ? ev[e] : 0, round, 0, 0, cand_stamp, cand_list, st);
    }
}

// Depth d of the candidate search (alive edges, frontier still present): one warp per
// vertex found at depth d-1.
// with_removed: also follow the slots removed in the current round (the pre-removal graph
// after the round's frontier is already gone: the h = 3 recovery).
__global__ void k_cand_expand(int32_t d, const int32_t *__restrict__ row_ptr,
                              const int32_t *__restrict__ col, const int32_t *__restrict__ col_live,
                              int32_t with_removed, DevStatus *st,
                              int32_t *__restrict__ cand_stamp, int32_t *__restrict__ cand_list) {
    if (st->alive == 0) return;
    int start = 0;
    for (int j = 0; j < d - 1; j++) start += st->cand_cnt[j];
    const int len = st->cand_cnt[d - 1];
    const int out_base = start + len;
    const int round = st->round;
    const int lane = threadIdx.x & 31;
    const int nwarps = gridDim.x * (blockDim.x >> 5);
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < len; i += nwarps) {
        const int w = cand_list[start + i];
        const int rb = row_ptr[w], re = row_ptr[w + 1];
        for (int s0 = rb; s0 < re; s0 += 32) {
            const int s = s0 + lane;
            int z = (s < re) ? col_live[s] : -1;
            if (with_removed && s < re && z == -(round + 1)) z = col[s];
            cand_mark(z >= 0, z >= 0 ? z : 0, round, d, out_base, cand_stamp, cand_list, st);
        }
    }
}

__global__ void k_remove(const int32_t *__restrict__ frontier, DevStatus *st,
                         const int32_t *__restrict__ eu, const int32_t *__restrict__ ev,
                         const int32_t *__restrict__ slot_lo, const int32_t *__restrict__ slot_hi,
                         int32_t *__restrict__ sup, int32_t *__restrict__ truss,
                         int32_t *__restrict__ stamp, int32_t *__restrict__ col_live,
                         int32_t *__restrict__ deg_alive, const int32_t *__restrict__ hub_slot,
                         uint32_t *__restrict__ hub_bits, int32_t Wpad) {
    if (st->alive == 0 || st->cont) return;  // a continued round removed its frontier already
    const int nF = st->nF, k = st->k, round = st->round;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nF; i += gridDim.x * blockDim.x)
    {
        const int e = frontier[i];
        remove_edge(e, k, round, eu[e], ev[e], slot_lo[e], slot_hi[e], sup, truss, stamp, col_live,
                    deg_alive, false, hub_slot, hub_bits, Wpad);
    }
}

// The records the incremental rounds read instead of chasing pointers: per edge (u, v, its
// two slots) and both rows' bounds, per adjacency slot (neighbour, its row's bounds, edge).
__global__ void k_make_records(int64_t m, const int32_t *__restrict__ row_ptr,
                               const int32_t *__restrict__ eu, const int32_t *__restrict__ ev,
                               const int32_t *__restrict__ slot_lo, const int32_t *__restrict__ slot_hi,
                               int4 *__restrict__ erec, int4 *__restrict__ srec) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const int u = eu[e], v = ev[e], lo = slot_lo[e], hi = slot_hi[e];
        const int rbu = row_ptr[u], reu = row_ptr[u + 1], rbv = row_ptr[v], rev = row_ptr[v + 1];
        erec[2 * e] = make_int4(u, v, lo, hi);
        erec[2 * e + 1] = make_int4(rbu, reu, rbv, rev);
        srec[lo] = make_int4(v, rbv, rev, (int)e);
        srec[hi] = make_int4(u, rbu, reu, (int)e);
    }
}

// Alive-adjacency n-bit sets of the high-degree vertices (all edges alive), block per hub.
// hub_list null: vertex x is hub x.  count (nullable): the number of hubs, at most nhub of them, as a device value.
__global__ void __launch_bounds__(kBlock) k_hub_init(const int32_t *__restrict__ hub_list, int32_t nhub,
                                                    const int32_t *__restrict__ count,
                                                    const int32_t *__restrict__ row_ptr,
                                                    const int32_t *__restrict__ col,
                                                    uint32_t *__restrict__ hub_bits, int32_t Wpad) {
    const int hubs = count ? min(nhub, *count) : nhub;
    for (int hb = blockIdx.x; hb < hubs; hb += gridDim.x) {
        uint32_t *bits = hub_bits + (int64_t)hb * Wpad;
        for (int i = threadIdx.x; i < Wpad; i += kBlock) bits[i] = 0u;
        __syncthreads();
        const int x = hub_list ? hub_list[hb] : hb;
        for (int s = row_ptr[x] + threadIdx.x; s < row_ptr[x + 1]; s += kBlock) {
            const int y = col[s];
            atomicOr(bits + (y >> 5), 1u << (y & 31));
        }
        __syncthreads();
    }
}

// Minimum alive h-support and alive count; the last block to finish closes the round.
__global__ void __launch_bounds__(kBlock) k_minreduce(const int32_t *__restrict__ sup, int64_t m,
                                                      DevStatus *st, int32_t initial) {
    if (!initial && st->alive == 0) return;
    minreduce_body<kNWarps>(sup, m, st, initial);
}

__global__ void k_init_deg(int32_t n, const int32_t *__restrict__ row_ptr,
                           int32_t *__restrict__ deg_alive) {
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += gridDim.x * blockDim.x)
        deg_alive[x] = row_ptr[x + 1] - row_ptr[x];
}

#define HTD_CHECK(...)                                                              \
    do {                                                                             \
        cudaError_t _e = (__VA_ARGS__);                                                     \
        if (_e != cudaSuccess) {                                                     \
            set_last_error(std::string(#__VA_ARGS__) + ": " + cudaGetErrorString(_e));      \
            return (_e == cudaErrorMemoryAllocation) ? HTD_ENOMEM : HTD_ECUDA;       \
        }                                                                            \
    } while (0)

// Degree from which ORing a vertex's n-bit row beats expanding its slots: a row costs W/4
// 16-byte loads, a slot about 60 cycles per 32 of them (R-MAT 18, W = 8,192: 512 gave 5.5 ms
// by the model of 160 G slots/s and 12 TB/s, 256 6.3 ms, 1,024 7.4 ms).
int32_t or_degree(const PeelWork &w) { return std::max(64, w.W / 16); }

BallArgs ball_args(Handle *H) {
    PeelWork &w = H->w;
    GraphDev &g = H->g;
    BallArgs a;
    a.n = g.n;
    a.W = w.W;
    a.Wpad = w.Wpad;
    a.h = w.h;
    a.count_bytes = 1;
    a.force_dense = w.dense_balls ? 1 : 0;
    a.row_ptr = g.row_ptr;
    a.col_live = w.col_live;
    a.deg_alive = w.deg_alive;
    a.pool = w.pool;
    a.pool_new = w.twin ? w.pool_new : nullptr;
    a.ball_off = w.ball_off;
    a.ball_need = w.ball_need;
    a.ball_size = w.ball_size;
    a.ball_nw = w.ball_nw;
    a.ball_meta = w.ball_meta;
    a.cand_list = w.cand_list;
    a.changed_list = w.changed_list;
    a.changed_stamp = w.changed_stamp;
    a.bfs_lists = w.bfs_lists;
    a.bfs_list_len = w.bfs_list_len;
    a.rows = nullptr;
    a.row_of = nullptr;
    a.or_deg = or_degree(w);
    a.bump = 0;
    a.inner = nullptr;
    a.st = w.status;
    return a;
}

HsupArgs hsup_args(Handle *H, int initial) {
    PeelWork &w = H->w;
    GraphDev &g = H->g;
    HsupArgs a;
    a.n = g.n;
    a.W = w.W;
    a.Wpad = w.Wpad;
    a.initial = initial;
    a.count_bytes = 1;
    a.row_ptr = g.row_ptr;
    a.col_live = w.col_live;
    a.slot_eid = g.slot_eid;
    a.pool = w.pool;
    a.ball_off = w.ball_off;
    a.ball_size = w.ball_size;
    a.ball_nw = w.ball_nw;
    a.changed_stamp = w.changed_stamp;
    a.items = w.items;
    a.sup = w.sup;
    a.st = w.status;
    return a;
}

}  // namespace

void free_work(Handle *H) {
    PeelWork &w = H->w;
    const cudaStream_t s = H->pstream;
    dev_free(w.pool, s);
    dev_free(w.ball_off, s);
    dev_free(w.ball_need, s);
    dev_free(w.ball_size, s);
    dev_free(w.ball_nw, s);
    dev_free(w.ball_meta, s);
    dev_free(w.col_live, s);
    dev_free(w.deg_alive, s);
    dev_free(w.sup, s);
    dev_free(w.truss, s);
    dev_free(w.stamp, s);
    dev_free(w.frontier, s);
    dev_free(w.cand_list, s);
    dev_free(w.cand_stamp, s);
    dev_free(w.changed_list, s);
    dev_free(w.changed_stamp, s);
    dev_free(w.items, s);
    dev_free(w.bfs_lists, s);
    dev_free(w.lost_keys, s);
    dev_free(w.lost, s);
    dev_free(w.edge_touch, s);
    dev_free(w.hub_slot, s);
    dev_free(w.hub_list, s);
    dev_free(w.hub_bits, s);
    dev_free(w.pitems, s);
    dev_free(w.uitems, s);
    dev_free(w.win, s);
    dev_free(w.erec, s);
    dev_free(w.srec, s);
    dev_free(w.scan_tmp, s);
    dev_free(w.pool2, s);
    dev_free(w.pool_new, s);
    dev_free(w.or_rows, s);
    dev_free(w.dense_off, s);
    dev_free(w.or_row_of, s);
    dev_free(w.or_list, s);
    dev_free(w.pool2_new, s);
    dev_free(w.ball_size2, s);
    dev_free(w.ball_nw2, s);
    dev_free(w.ball_meta2, s);
    dev_free(w.changed_list2, s);
    dev_free(w.changed_stamp2, s);
    dev_free(w.lost2_keys, s);
    dev_free(w.lost2, s);
    dev_free(w.c3items, s);
    dev_free(w.touch2, s);
    dev_free(w.status, s);
    give_status_host(w.status_host);
    w = PeelWork{};
}

void drop_graphs(Handle *H);
namespace {
htd_status ensure_work_impl(Handle *H, int32_t h, bool incremental, bool tiny_table);
}  // namespace

// The captured round graphs hold the scratch pointers: dropped whenever the scratch goes.
void drop_graphs(Handle *H) {
    if (H->graph_exec) cudaGraphExecDestroy(H->graph_exec);
    if (H->graph_exec_timed) cudaGraphExecDestroy(H->graph_exec_timed);
    H->graph_exec = nullptr;
    H->graph_exec_timed = nullptr;
    H->graph_h = 0;
    H->graph_rounds = 0;
}

// Allocates (or reuses) the scratch of an h-support pass / peel; on failure nothing of it
// is kept (the handle stays usable for a later attempt).
htd_status ensure_work(Handle *H, int32_t h, bool incremental, bool tiny_table) {
    const htd_status st = ensure_work_impl(H, h, incremental, tiny_table);
    if (st != HTD_OK) {
        drop_graphs(H);
        free_work(H);
    }
    return st;
}

namespace {
// Scratch every pass at this h needs.
htd_status alloc_base(Handle *H, int32_t h) {
    PeelWork &w = H->w;
    const int64_t n = H->g.n, m = H->g.m;
    w.h = h;
    w.W = (int32_t)((n + 31) / 32);
    if (w.W < 1) w.W = 1;
    w.Wpad = (w.W + 3) & ~3;
    w.smem_ball = (size_t)w.Wpad * 4;
    w.smem_hsup = (size_t)w.Wpad * 4;
    HTD_CHECK(raise_smem_limit((const void *)k_ball<kModeCount>, w.smem_ball));
    HTD_CHECK(raise_smem_limit((const void *)k_ball<kModeStore>, w.smem_ball));
    HTD_CHECK(raise_smem_limit((const void *)k_ball<kModeRebuild>, w.smem_ball));
    HTD_CHECK(raise_smem_limit((const void *)k_ball_or, w.smem_ball));
    HTD_CHECK(raise_smem_limit((const void *)k_hsup, w.smem_hsup));
    int occ_ball = 0, occ_hsup = 0;
    HTD_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_ball, k_ball<kModeRebuild>,
                                                            kBlock, w.smem_ball));
    HTD_CHECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_hsup, k_hsup, kBlock,
                                                            w.smem_hsup));
    if (occ_ball < 1 || occ_hsup < 1) {
        set_last_error("htd: an n-bit ball does not fit in shared memory");
        return HTD_EUNSUPPORTED;
    }
    w.grid_ball = H->num_sms * occ_ball;
    w.grid_hsup = H->num_sms * occ_hsup;
    w.grid_edges = H->num_sms * 4;
    HTD_CHECK(dev_alloc(&w.ball_off, n + 1, H->pstream));
    HTD_CHECK(dev_alloc(&w.ball_need, n, H->pstream));
    HTD_CHECK(dev_alloc(&w.ball_size, n, H->pstream));
    HTD_CHECK(dev_alloc(&w.ball_nw, n, H->pstream));
    HTD_CHECK(dev_alloc(&w.ball_meta, n, H->pstream));
    HTD_CHECK(dev_alloc(&w.col_live, 2 * m, H->pstream));
    HTD_CHECK(dev_alloc(&w.deg_alive, n, H->pstream));
    HTD_CHECK(dev_alloc(&w.sup, m, H->pstream));
    HTD_CHECK(dev_alloc(&w.truss, m, H->pstream));
    HTD_CHECK(dev_alloc(&w.stamp, m, H->pstream));
    HTD_CHECK(dev_alloc(&w.frontier, m, H->pstream));
    HTD_CHECK(dev_alloc(&w.cand_list, n, H->pstream));
    HTD_CHECK(dev_alloc(&w.cand_stamp, n, H->pstream));
    HTD_CHECK(dev_alloc(&w.changed_list, n, H->pstream));
    HTD_CHECK(dev_alloc(&w.changed_stamp, n, H->pstream));
    w.items_cap = n + (2 * m + kItemChunk - 1) / kItemChunk + 1;
    HTD_CHECK(dev_alloc(&w.items, w.items_cap, H->pstream));
    if (h >= 3) {
        w.bfs_list_len = n > 0 ? n : 1;
        HTD_CHECK(dev_alloc(&w.bfs_lists, (int64_t)w.grid_ball * 2 * w.bfs_list_len, H->pstream));
    }
    HTD_CHECK(dev_alloc_bytes(&w.scan_tmp, scan_temp_bytes(n + 1), H->pstream));
    HTD_CHECK(dev_alloc(&w.status, 1, H->pstream));
    w.status_host = take_status_host();
    if (!w.status_host) {
        set_last_error("htd: pinned status block allocation failed");
        return HTD_ENOMEM;
    }
    return HTD_OK;
}

htd_status ensure_work_impl(Handle *H, int32_t h, bool incremental, bool tiny_table) {
    PeelWork &w = H->w;
    GraphDev &g = H->g;
    incremental = incremental && h <= 3;
    if (w.status && w.h == h && (!incremental || (w.lost_keys && w.lost_tiny == tiny_table))) {
        w.incremental = incremental;
        w.inc3 = incremental && h == 3;
        return HTD_OK;
    }
    // scratch of an h-support pass at the same h only lacks the incremental rounds' part
    const bool base_ready = w.status && w.h == h && !w.lost_keys;
    if (w.status && !base_ready) {
        // the per-block BFS lists and the ball storage depend on h: rebuild everything
        drop_graphs(H);
        free_work(H);
    }
    const int64_t n = g.n, m = g.m;
    if (!base_ready) {
        const htd_status bs = alloc_base(H, h);
        if (bs != HTD_OK) return bs;
    }
    if (incremental) {
        // a round's lost pairs: half of a power-of-two table of 8 x (2m) slots (>= 2^12)
        // sized to stay L2-resident (at most 2^22 slots, 32 MiB); larger rounds run in batches
        // h = 3 rounds lose many more radius-3 pairs: a table up to 2^24 slots
        const int64_t cap_max = (int64_t)1 << (h == 3 ? 24 : 22);
        int64_t cap = 4096;
        while (cap < 4 * m * (h == 3 ? 4 : 1) && cap < cap_max) cap <<= 1;
        if (tiny_table) cap = 128;  // forces rounds to run in many batches
        w.lost_tiny = tiny_table;
        w.lost_cap = cap;
        w.lost_max = cap / 2;
        HTD_CHECK(dev_alloc(&w.lost_keys, cap, H->pstream));
        HTD_CHECK(dev_alloc(&w.lost, 2 * w.lost_max, H->pstream));
        HTD_CHECK(dev_alloc(&w.edge_touch, n, H->pstream));
        // work items of the loss detection and of the support updates (per batch)
        // (sized with the graph: 2m adjacency slots)
        w.pitems_cap = std::min<int64_t>((int64_t)1 << 22, std::max<int64_t>(4096, 2 * m));
        // adjacency slots the updates of one batch may visit
        w.upd_budget = std::min<int64_t>((int64_t)1 << 30, std::max<int64_t>(1 << 16, 256 * m));
        w.uitems_cap = 2 * w.lost_max + w.upd_budget / 32 + 1024;
        HTD_CHECK(dev_alloc(&w.pitems, 2 * w.pitems_cap, H->pstream));
        HTD_CHECK(dev_alloc(&w.uitems, w.uitems_cap, H->pstream));
        w.win_cap = std::min<int64_t>(m, (int64_t)1 << 15);
        HTD_CHECK(dev_alloc(&w.win, 2 * w.win_cap, H->pstream));
        HTD_CHECK(dev_alloc(&w.erec, 2 * m, H->pstream));
        HTD_CHECK(dev_alloc(&w.srec, 2 * m, H->pstream));
        if (h == 3) {
            // radius-2 balls (dense) with their own metadata, the round's radius-2 losses and
            // the radius-3 candidate items
            if (!w.pool2) HTD_CHECK(dev_alloc(&w.pool2, n * (int64_t)w.Wpad, H->pstream));
            if (!w.ball_size2) HTD_CHECK(dev_alloc(&w.ball_size2, n, H->pstream));
            if (!w.ball_nw2) HTD_CHECK(dev_alloc(&w.ball_nw2, n, H->pstream));
            if (!w.ball_meta2) HTD_CHECK(dev_alloc(&w.ball_meta2, n, H->pstream));
            HTD_CHECK(dev_alloc(&w.changed_list2, n, H->pstream));
            HTD_CHECK(dev_alloc(&w.changed_stamp2, n, H->pstream));
            HTD_CHECK(dev_alloc(&w.touch2, n, H->pstream));
            int64_t cap2 = 4096;
            while (cap2 < 4 * m && cap2 < ((int64_t)1 << 22)) cap2 <<= 1;
            if (tiny_table) cap2 = 128;
            w.lost2_cap = cap2;
            w.lost2_max = cap2 / 2;
            HTD_CHECK(dev_alloc(&w.lost2_keys, cap2, H->pstream));
            HTD_CHECK(dev_alloc(&w.lost2, 2 * w.lost2_max, H->pstream));
            w.c3items_cap = tiny_table ? 256
                                       : std::min<int64_t>((int64_t)1 << 25, std::max<int64_t>(1 << 16, 8 * m));
            HTD_CHECK(dev_alloc(&w.c3items, w.c3items_cap, H->pstream));
        }
        // alive-adjacency n-bit sets: every vertex of degree >= T, the smallest power of two
        // for which they fit in min(16 GiB, a quarter of the free device memory)
        size_t free_b = 0, total_b = 0;
        HTD_CHECK(cudaMemGetInfo(&free_b, &total_b));
        const int64_t budget_words = std::min<int64_t>((int64_t)1 << 32, (int64_t)(free_b / 16));
        if (n * w.Wpad <= budget_words) {
            // T = 1: every vertex gets a set (isolated ones too), set x at row x, no lists needed
            w.nhub = (int32_t)n;
            w.hub_min_deg = 1;
        } else {
            std::vector<int32_t> rp(n + 1);
            HTD_CHECK(cudaMemcpyAsync(rp.data(), g.row_ptr, (n + 1) * sizeof(int32_t), cudaMemcpyDeviceToHost,
                                      H->pstream));
            HTD_CHECK(cudaStreamSynchronize(H->pstream));
            int32_t T = 2;
            for (;; T *= 2) {
                int64_t cnt = 0;
                for (int64_t x = 0; x < n; x++) cnt += (rp[x + 1] - rp[x] >= T);
                if (cnt * w.Wpad <= budget_words || T > (1 << 24)) break;
            }
            std::vector<int32_t> slot(n, -1), list;
            for (int64_t x = 0; x < n; x++)
                if (rp[x + 1] - rp[x] >= T) {
                    slot[x] = (int32_t)list.size();
                    list.push_back((int32_t)x);
                }
            w.nhub = (int32_t)list.size();
            w.hub_min_deg = T;
            HTD_CHECK(dev_alloc(&w.hub_slot, n, H->pstream));
            HTD_CHECK(cudaMemcpyAsync(w.hub_slot, slot.data(), n * sizeof(int32_t), cudaMemcpyHostToDevice,
                                      H->pstream));
            if (w.nhub > 0) {
                HTD_CHECK(dev_alloc(&w.hub_list, w.nhub, H->pstream));
                HTD_CHECK(cudaMemcpyAsync(w.hub_list, list.data(), w.nhub * sizeof(int32_t),
                                          cudaMemcpyHostToDevice, H->pstream));
            }
            HTD_CHECK(cudaStreamSynchronize(H->pstream));  // the lists are on this function's stack
        }
        if (w.nhub > 0) {
            HTD_CHECK(dev_alloc(&w.hub_bits, (int64_t)w.nhub * w.Wpad, H->pstream));
        }
    }
    w.incremental = incremental;
    w.inc3 = incremental && h == 3;
    return HTD_OK;
}

}  // namespace

// Takes the twin ball matrices into use if they are there or can be had: every ball dense,
// an alive-adjacency set at every vertex, and the copies no larger than `budget` bytes.
// Without them the rounds keep the batch's losses in hash sets (same results).  In the cluster round
// kernel they took R-MAT 16 at h = 2 from 886 to 800 ms and ER n = 2,000 from 1.83 to 1.61 ms; the
// budget only keeps a peel from taking most of the device.
htd_status ensure_twin(Handle *H, int64_t budget) {
    PeelWork &w = H->w;
    const int64_t n = H->g.n, words = n * (int64_t)w.Wpad;
    w.twin = false;
    if (!w.incremental || !w.dense_balls || n == 0 || w.nhub != n || w.hub_min_deg != 1) return HTD_OK;
    const int copies = w.inc3 ? 2 : 1;
    if (!w.pool_new && copies * words * 4 > budget) return HTD_OK;
    if (!w.pool_new) {
        cudaError_t e = dev_alloc(&w.pool_new, words, H->pstream);
        if (e == cudaSuccess && copies == 2) e = dev_alloc(&w.pool2_new, words, H->pstream);
        if (e != cudaSuccess) {
            dev_free(w.pool_new, H->pstream);
            w.pool_new = nullptr;
            return HTD_OK;
        }
    }
    w.twin = true;
    return HTD_OK;
}

namespace {

// Adjacency rows of the high-degree vertices as n-bit sets, built once per handle: at most
// 512 MiB of them (more would not stay in L2, where the builds read them).
htd_status ensure_or_rows(Handle *H, cudaStream_t s, int64_t *launches) {
    PeelWork &w = H->w;
    GraphDev &g = H->g;
    if (w.or_rows) return HTD_OK;
    const int64_t deg = or_degree(w);
    const int32_t cap = (int32_t)std::max<int64_t>(
        1, std::min<int64_t>(2 * g.m / deg + 1, ((int64_t)512 << 20) / (4 * (int64_t)w.Wpad)));
    cudaError_t e = dev_alloc(&w.or_row_of, g.n, H->pstream);
    if (e == cudaSuccess) e = dev_alloc(&w.or_list, (int64_t)cap + 1, H->pstream);
    if (e == cudaSuccess) e = dev_alloc(&w.or_rows, (int64_t)cap * w.Wpad, H->pstream);
    if (e != cudaSuccess) {  // no room: every row is expanded
        dev_free(w.or_row_of, H->pstream);
        dev_free(w.or_list, H->pstream);
        w.or_row_of = nullptr;
        w.or_list = nullptr;
        w.or_rows = nullptr;
        return HTD_OK;
    }
    int32_t *count = w.or_list + cap;
    HTD_CHECK(cudaMemsetAsync(count, 0, sizeof(int32_t), s));
    k_or_rows<<<std::min<int64_t>((g.n + kBlock - 1) / kBlock, H->num_sms * 8), kBlock, 0, s>>>(
        g.n, g.row_ptr, (int32_t)deg, cap, w.or_row_of, w.or_list, count);
    k_hub_init<<<std::min(cap, H->num_sms * 8), kBlock, 0, s>>>(w.or_list, cap, count, g.row_ptr, g.col, w.or_rows,
                                                            w.Wpad);
    *launches += 2;
    HTD_CHECK(cudaGetLastError());
    return HTD_OK;
}

// Radius-3 balls as ORs of the neighbours' radius-2 rows (2m rows of W words, about 6 TB/s)
// against the search by levels (about the sum of squared degrees x the mean degree slots, 60
// G/s): DC-SBM 200k 10 ms against 32 ms; ER of mean degree 8 at n = 200,000 6.7 ms against 2.
bool or_beats_search(const Handle *H) {
    const GraphDev &g = H->g;
    const double rows = 8.0 * (double)g.m * (double)H->w.Wpad;
    const double slots = std::min((double)g.deg2, (double)g.n * (double)g.n) * (2.0 * (double)g.m / (double)g.n);
    return rows < 100.0 * slots;
}

void destroy_rounds(Handle *H) {
    for (cudaGraphExec_t *e : {&H->graph_exec, &H->graph_exec_timed}) {
        if (*e) cudaGraphExecDestroy(*e);
        *e = nullptr;
    }
}

// Radius-2 balls of every vertex, stored dense in pool2 with their own sizes.
htd_status build_inner(Handle *H, cudaStream_t s, int64_t *launches) {
    PeelWork &w = H->w;
    BallArgs b2 = ball_args(H);
    b2.h = 2;
    b2.count_bytes = 0;
    b2.force_dense = 1;
    b2.pool = w.pool2;
    b2.pool_new = w.twin ? w.pool2_new : nullptr;
    if (w.dense_off) b2.ball_off = w.dense_off;
    if (w.incremental && w.nhub == H->g.n && w.hub_min_deg == 1) b2.rows = w.hub_bits;
    b2.ball_size = w.ball_size2;
    b2.ball_nw = w.ball_nw2;
    b2.ball_meta = w.ball_meta2;
    b2.changed_list = w.changed_list2;
    b2.changed_stamp = w.changed_stamp2;
    b2.bfs_lists = nullptr;
    HTD_CHECK(cudaMemsetAsync(&w.status->q_store, 0, sizeof(int32_t), s));
    k_ball<kModeStore><<<w.grid_ball, kBlock, w.smem_ball, s>>>(b2);
    (*launches)++;
    HTD_CHECK(cudaGetLastError());
    return HTD_OK;
}

// The dense radius-2 balls for it: those of the incremental peel, or (h-support) a pool of
// their own where they fit an eighth of the free memory.  Where one of the arrays cannot be had
// the search by levels, which needs none of them, does the work (inner_ready stays false).
htd_status ensure_inner(Handle *H, cudaStream_t s, int64_t *launches, size_t free_b) {
    PeelWork &w = H->w;
    const int64_t n = H->g.n, words = n * (int64_t)w.Wpad;
    w.inner_ready = false;
    if (!w.pool2 && (double)words * 4 > (double)free_b / 8) return HTD_OK;
    auto have = [&](auto **p, int64_t count) {
        if (*p) return true;
        if (dev_alloc(p, count, H->pstream) == cudaSuccess) return true;
        *p = nullptr;
        return false;
    };
    if (!have(&w.pool2, words) || !have(&w.ball_size2, n) || !have(&w.ball_nw2, n) || !have(&w.ball_meta2, n))
        return HTD_OK;
    if (!w.dense_off) {
        if (!have(&w.dense_off, n + 1)) return HTD_OK;
        k_dense_offsets<<<std::min<int64_t>((n + kBlock) / kBlock, H->num_sms * 8), kBlock, 0, s>>>(n, w.Wpad,
                                                                                                w.dense_off);
        (*launches)++;
    }
    const htd_status rs = build_inner(H, s, launches);
    w.inner_ready = rs == HTD_OK;
    return rs;
}

// Words that the balls of an h-support pass take at most.
htd_status bound_storage(Handle *H, int32_t h, cudaStream_t s, int64_t *launches, int64_t *words) {
    PeelWork &w = H->w;
    GraphDev &g = H->g;
    const int grid = (int)std::min<int64_t>(((int64_t)g.n * 32 + kBlock - 1) / kBlock, H->num_sms * 8);
    int32_t *bound = w.ball_need, *inner = w.cand_list;  // neither is in use yet
    for (int r = 1; r <= h; r++) {
        std::swap(bound, inner);
        k_ball_bound<<<grid, kBlock, 0, s>>>(g.n, w.Wpad, g.row_ptr, g.col, r > 1 ? inner : nullptr, bound);
    }
    k_bound_words<<<std::min<int64_t>((g.n + kBlock - 1) / kBlock, H->num_sms * 8), kBlock, 0, s>>>(g.n, w.Wpad, bound,
                                                                                            w.status);
    *launches += h + 1;
    HTD_CHECK(cudaGetLastError());
    HTD_CHECK(cudaMemcpyAsync(words, &w.status->ball_bound, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    HTD_CHECK(cudaStreamSynchronize(s));
    return HTD_OK;
}

}  // namespace

// What an h-support pass held beyond its balls goes back where it is more than a 32nd of the
// device's memory (room that later peels, of this handle and others, look for): the radius-2 rows
// that radius-3 balls were made of, and a pool taken by the bound that came out much too large.
// Up to there a repeated call saves taking them again (DC-SBM 200k at h = 3, 5 GB of rows: 4 ms of
// 23).  Scratch of a peel on the handle stays.
void trim_support(Handle *H) {
    PeelWork &w = H->w;
    if (w.lost_keys || w.keep_bytes <= 0) return;
    const int64_t rows = w.pool2 ? 4 * H->g.n * (int64_t)w.Wpad : 0;
    const int64_t spare = w.pool ? 4 * (w.pool_words - w.support_words) : 0;
    if (rows + spare <= w.keep_bytes) return;
    if (w.pool2) {
        dev_free(w.pool2, H->pstream);
        w.pool2 = nullptr;
        w.inner_ready = false;
    }
    if (spare > w.keep_bytes) {
        destroy_rounds(H);
        dev_free(w.pool, H->pstream);
        w.pool = nullptr;
        w.pool_words = 0;
    }
}

// Initial pass: every vertex's ball and every edge's h-support, then the first min reduction.
// Leaves the status ready for round 0 (support_only: the supports are all that is wanted).
htd_status initial_pass(Handle *H, int32_t h, cudaStream_t s, int64_t *launches,
                        htd_stats *timing, bool support_only) {
    PeelWork &w = H->w;
    GraphDev &g = H->g;
    const int64_t n = g.n, m = g.m;
    w.inner_ready = false;
    w.or_bytes = 0;
    H->cluster_launches = 0;
    std::memset(w.status_host, 0, sizeof(DevStatus));
    w.status_host->k = 2;
    w.status_host->min_acc = INT_MAX;
    w.status_host->overflow_unit = INT_MAX;
    w.status_host->unit_span = INT_MAX;
    w.status_host->pitems_cap = (int32_t)w.pitems_cap;
    HTD_CHECK(cudaMemcpyAsync(w.status, w.status_host, sizeof(DevStatus), cudaMemcpyHostToDevice, s));
    if (m > 0)
        HTD_CHECK(cudaMemcpyAsync(w.col_live, g.col, 2 * m * sizeof(int32_t),
                                  cudaMemcpyDeviceToDevice, s));
    HTD_CHECK(cudaMemsetAsync(w.cand_stamp, 0xff, (n > 0 ? n : 1) * sizeof(int32_t), s));
    HTD_CHECK(cudaMemsetAsync(w.changed_stamp, 0xff, (n > 0 ? n : 1) * sizeof(int32_t), s));
    HTD_CHECK(cudaMemsetAsync(w.stamp, 0xff, (m > 0 ? m : 1) * sizeof(int32_t), s));
    if (w.incremental) {
        HTD_CHECK(cudaMemsetAsync(w.edge_touch, 0xff, (n > 0 ? n : 1) * sizeof(int32_t), s));
        if (!w.twin) HTD_CHECK(cudaMemsetAsync(w.lost_keys, 0xff, w.lost_cap * sizeof(unsigned long long), s));
        if (w.inc3) {
            if (!w.twin)
                HTD_CHECK(cudaMemsetAsync(w.lost2_keys, 0xff, w.lost2_cap * sizeof(unsigned long long), s));
            HTD_CHECK(cudaMemsetAsync(w.changed_stamp2, 0xff, (n > 0 ? n : 1) * sizeof(int32_t), s));
            HTD_CHECK(cudaMemsetAsync(w.touch2, 0xff, (n > 0 ? n : 1) * sizeof(int32_t), s));
        }
        if (m > 0) {
            k_make_records<<<std::min<int64_t>((m + kBlock - 1) / kBlock, H->num_sms * 8), kBlock, 0, s>>>(
                m, g.row_ptr, g.eu, g.ev, g.slot_lo, g.slot_hi, w.erec, w.srec);
            (*launches)++;
        }
        if (w.nhub > 0) {
            k_hub_init<<<std::min(w.nhub, H->num_sms * 8), kBlock, 0, s>>>(w.hub_list, w.nhub, nullptr, g.row_ptr,
                                                                        g.col, w.hub_bits, w.Wpad);
            (*launches)++;
        }
    }
    if (n > 0) {
        k_init_deg<<<std::min<int64_t>((n + kBlock - 1) / kBlock, H->num_sms * 8), kBlock, 0, s>>>(
            (int32_t)n, g.row_ptr, w.deg_alive);
        (*launches)++;
    }
    BallArgs ba = ball_args(H);
    cudaEvent_t e0 = nullptr, e1 = nullptr, e2 = nullptr, e3 = nullptr;
    if (timing) {
        HTD_CHECK(cudaEventCreate(&e0));
        HTD_CHECK(cudaEventCreate(&e1));
        HTD_CHECK(cudaEventCreate(&e2));
        HTD_CHECK(cudaEventCreate(&e3));
    }
    if (n > 0) {
        if (support_only && h == 2) {
            const htd_status rs = ensure_or_rows(H, s, launches);
            if (rs != HTD_OK) return rs;
            ba.rows = w.or_rows;
            ba.row_of = w.or_row_of;
        } else if (w.incremental && w.nhub == n && w.hub_min_deg == 1) {
            ba.rows = w.hub_bits;  // alive-adjacency sets, every edge alive
        }
        // Storage: dense balls have fixed places; h-support alone takes places as the balls are
        // done, from a pool with room for them: all dense where that is 64 MiB at most, else by an
        // upper bound, from the second call on what they took.  Where that is more than a quarter
        // of the free memory a first pass counts.
        int64_t total = n * (int64_t)w.Wpad;
        size_t free_b = 0, total_b = 0;
        if (support_only) {
            HTD_CHECK(cudaMemGetInfo(&free_b, &total_b));
            w.keep_bytes = (int64_t)(total_b / 32);
            if (w.support_words > 0) {
                total = w.support_words;
            } else if (total > ((int64_t)1 << 24)) {
                int64_t words = 0;
                const htd_status bs = bound_storage(H, h, s, launches, &words);
                if (bs != HTD_OK) return bs;
                total = std::min(total, words);
            }
        }
        const bool room = total <= w.pool_words || (double)total * 4 <= (double)free_b / 4;
        auto take_pool = [&]() -> cudaError_t {
            if (total <= w.pool_words) return cudaSuccess;
            dev_free(w.pool, s);
            w.pool = nullptr;
            w.pool_words = 0;
            destroy_rounds(H);  // the captured rounds hold the old pool pointer
            const cudaError_t e = dev_alloc(&w.pool, total, H->pstream);
            if (e == cudaSuccess) w.pool_words = total;
            else w.pool = nullptr;
            return e;
        };
        if (w.dense_balls) {
            k_dense_offsets<<<std::min<int64_t>((n + kBlock) / kBlock, H->num_sms * 8), kBlock, 0, s>>>(n, w.Wpad,
                                                                                                    w.ball_off);
            (*launches)++;
        } else if (support_only && room && total < ((int64_t)1 << 33)) {
            if (take_pool() == cudaSuccess) ba.bump = 1;
        }
        if (!w.dense_balls && !ba.bump) {
            k_ball<kModeCount><<<w.grid_ball, kBlock, w.smem_ball, s>>>(ba);
            (*launches)++;
            HTD_CHECK(cudaGetLastError());
            HTD_CHECK(scan_exclusive<int32_t, int64_t>(w.ball_need, w.ball_off, n, w.scan_tmp, s, launches));
            HTD_CHECK(cudaMemcpyAsync(&total, w.ball_off + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
            HTD_CHECK(cudaStreamSynchronize(s));
            w.support_words = total;
        }
        if (total >= ((int64_t)1 << 33)) {
            set_last_error("htd: h-hop balls need more than 32 GiB of storage");
            return HTD_EUNSUPPORTED;
        }
        HTD_CHECK(take_pool());
        ba.pool = w.pool;
        w.pool_used = total;
        // radius 3 from the dense radius-2 balls, where their rows cost less than the search
        const uint32_t *inner = nullptr;
        if (h == 3 && (ba.bump || w.inc3) && or_beats_search(H)) {
            const htd_status rs = ensure_inner(H, s, launches, free_b);
            if (rs != HTD_OK) return rs;
            inner = w.inner_ready ? w.pool2 : nullptr;
            HTD_CHECK(cudaMemsetAsync(&w.status->q_store, 0, sizeof(int32_t), s));
        }
        if (timing) HTD_CHECK(cudaEventRecord(e0, s));
        if (inner) {
            ba.inner = inner;
            w.or_bytes = 4 * (int64_t)w.W * (n + 2 * m);  // every row once, and once per adjacency slot
            k_ball_or<<<w.grid_ball, kBlock, w.smem_ball, s>>>(ba);
        } else {
            k_ball<kModeStore><<<w.grid_ball, kBlock, w.smem_ball, s>>>(ba);
        }
        if (timing) HTD_CHECK(cudaEventRecord(e1, s));
        (*launches)++;
        HTD_CHECK(cudaGetLastError());
        k_make_items<<<std::min<int64_t>((n + kBlock - 1) / kBlock, H->num_sms * 8), kBlock, 0, s>>>(
            nullptr, 1, (int32_t)n, g.row_ptr, w.items, w.status);
        (*launches)++;
        HsupArgs ha = hsup_args(H, 1);
        if (timing) HTD_CHECK(cudaEventRecord(e2, s));
        k_hsup<<<w.grid_hsup, kBlock, w.smem_hsup, s>>>(ha);
        if (timing) HTD_CHECK(cudaEventRecord(e3, s));
        (*launches)++;
        HTD_CHECK(cudaGetLastError());
    }
    k_minreduce<<<w.grid_edges, kBlock, 0, s>>>(w.sup, m, w.status, 1);
    (*launches)++;
    HTD_CHECK(cudaGetLastError());
    if (timing) {
        HTD_CHECK(cudaStreamSynchronize(s));
        float a = 0.f, b = 0.f;
        if (n > 0) {
            HTD_CHECK(cudaEventElapsedTime(&a, e0, e1));
            HTD_CHECK(cudaEventElapsedTime(&b, e2, e3));
            timing->ms_initial_ball += a;
            timing->ms_initial_hsup += b;
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        cudaEventDestroy(e2);
        cudaEventDestroy(e3);
    }
    return HTD_OK;
}

// Enqueues one peel round.  evs (nullable) = kRoundEvents events at the phase boundaries:
//   rebuild:     | select | candidates | remove | ball rebuild | items + h-support | reduce |
//   (incremental rounds add their phase times to the status block instead, with `timer`)
htd_status enqueue_round(Handle *H, cudaStream_t s, int64_t *launches, cudaEvent_t *evs, bool timer,
                         bool by_cluster) {
    PeelWork &w = H->w;
    GraphDev &g = H->g;
    const int64_t m = g.m;
    const int gsmall = H->num_sms * 4;
    if (w.incremental) return enqueue_incremental_round(H, s, launches, timer, by_cluster);
    // inside a stream capture an ordinary record only orders nodes; an external record
    // node really records the event each time the graph runs, so it can be timed
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (evs) HTD_CHECK(cudaStreamIsCapturing(s, &cap));
    const unsigned rec_flags = (cap == cudaStreamCaptureStatusActive) ? cudaEventRecordExternal : 0u;
    auto mark = [&](int i) {
        if (evs) cudaEventRecordWithFlags(evs[i], s, rec_flags);
    };
    mark(0);
    k_select<<<w.grid_edges, kBlock, 0, s>>>(w.sup, m, w.status, w.frontier);
    mark(1);
    k_cand_init<<<gsmall, kBlock, 0, s>>>(w.frontier, g.eu, g.ev, w.status, w.cand_stamp, w.cand_list);
    *launches += 2;
    for (int d = 1; d < w.h; d++) {
        k_cand_expand<<<gsmall * 2, kBlock, 0, s>>>(d, g.row_ptr, g.col, w.col_live, 0, w.status,
                                                     w.cand_stamp, w.cand_list);
        (*launches)++;
    }
    mark(2);
    k_remove<<<gsmall, kBlock, 0, s>>>(w.frontier, w.status, g.eu, g.ev, g.slot_lo, g.slot_hi,
                                       w.sup, w.truss, w.stamp, w.col_live, w.deg_alive, nullptr,
                                       nullptr, 0);
    (*launches)++;
    mark(3);
    BallArgs ba = ball_args(H);
    k_ball<kModeRebuild><<<w.grid_ball, kBlock, w.smem_ball, s>>>(ba);
    mark(4);
    k_make_items<<<gsmall, kBlock, 0, s>>>(w.changed_list, 0, g.n, g.row_ptr, w.items, w.status);
    HsupArgs ha = hsup_args(H, 0);
    k_hsup<<<w.grid_hsup, kBlock, w.smem_hsup, s>>>(ha);
    mark(5);
    k_minreduce<<<w.grid_edges, kBlock, 0, s>>>(w.sup, m, w.status, 0);
    mark(6);
    *launches += 4;
    HTD_CHECK(cudaGetLastError());
    return HTD_OK;
}

// Radius-2 balls of the incremental h = 3 peel, unless the radius-3 balls were made of them.
htd_status initial_pass_r2(Handle *H, cudaStream_t s, int64_t *launches) {
    if (!H->w.inc3 || H->g.n == 0 || H->w.inner_ready) return HTD_OK;
    return build_inner(H, s, launches);
}

namespace {

// Clears what a halted h = 3 round recorded (its pair sets are emptied by the caller) and
// the queue heads the rebuild kernels use.
__global__ void k_recover_reset(DevStatus *st) {
    st->halt = 0;
    st->nlost = 0;
    st->nlost2 = 0;
    st->npitems = 0;
    st->nuitems = 0;
    st->nc3items = 0;
    st->upd_work = 0;
    st->touched = 0;
    st->overflow_unit = INT_MAX;
    for (int j = 0; j < kMaxH; j++) st->cand_cnt[j] = 0;
    st->q_ball = 0;
    st->nchanged = 0;
    st->nitems = 0;
    st->q_items = 0;
    st->st_recovered++;
}

__global__ void k_reset_rebuild_queue(DevStatus *st) {
    st->q_ball = 0;
    st->nchanged = 0;
}

}  // namespace

// Finishes a halted round of the incremental h = 3 peel.  Its frontier is already removed
// (slots marked with the round) and nothing else of the round was applied: balls and
// supports are those of before the round.  Every vertex within distance 2 of a frontier
// endpoint in the pre-removal graph is a candidate: its radius-2 ball (if within distance
// 1) and its radius-3 ball are rebuilt, and the supports of the alive edges at vertices
// whose radius-3 ball shrank are recomputed; the min reduction then closes the round.
htd_status recover_round_h3(Handle *H, cudaStream_t s, int64_t *launches) {
    PeelWork &w = H->w;
    GraphDev &g = H->g;
    const int gsmall = H->num_sms * 4;
    if (!w.twin) {
        HTD_CHECK(cudaMemsetAsync(w.lost_keys, 0xff, w.lost_cap * sizeof(unsigned long long), s));
        HTD_CHECK(cudaMemsetAsync(w.lost2_keys, 0xff, w.lost2_cap * sizeof(unsigned long long), s));
    }
    k_recover_reset<<<1, 1, 0, s>>>(w.status);
    k_cand_init<<<gsmall, kBlock, 0, s>>>(w.frontier, g.eu, g.ev, w.status, w.cand_stamp, w.cand_list);
    *launches += 2;
    for (int d = 1; d < 3; d++) {
        k_cand_expand<<<gsmall * 2, kBlock, 0, s>>>(d, g.row_ptr, g.col, w.col_live, 1, w.status,
                                                     w.cand_stamp, w.cand_list);
        (*launches)++;
    }
    // radius 2: candidates of depth 0..1 (the rebuild counts the first h levels)
    BallArgs b2 = ball_args(H);
    b2.h = 2;
    b2.count_bytes = 0;
    b2.force_dense = 1;
    b2.pool = w.pool2;
    b2.pool_new = w.twin ? w.pool2_new : nullptr;
    b2.ball_size = w.ball_size2;
    b2.ball_nw = w.ball_nw2;
    b2.ball_meta = w.ball_meta2;
    b2.changed_list = w.changed_list2;
    b2.changed_stamp = w.changed_stamp2;
    b2.bfs_lists = nullptr;
    k_ball<kModeRebuild><<<w.grid_ball, kBlock, w.smem_ball, s>>>(b2);
    k_reset_rebuild_queue<<<1, 1, 0, s>>>(w.status);
    // radius 3 and the supports it changes
    BallArgs b3 = ball_args(H);
    k_ball<kModeRebuild><<<w.grid_ball, kBlock, w.smem_ball, s>>>(b3);
    k_make_items<<<gsmall, kBlock, 0, s>>>(w.changed_list, 0, g.n, g.row_ptr, w.items, w.status);
    HsupArgs ha = hsup_args(H, 0);
    k_hsup<<<w.grid_hsup, kBlock, w.smem_hsup, s>>>(ha);
    k_minreduce<<<w.grid_edges, kBlock, 0, s>>>(w.sup, g.m, w.status, 0);
    *launches += 6;
    HTD_CHECK(cudaGetLastError());
    return HTD_OK;
}

}  // namespace htd
