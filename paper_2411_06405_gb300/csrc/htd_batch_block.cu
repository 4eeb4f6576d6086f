// htd_batch_block.cu -- the batched decomposition of many small graphs in one persistent
// launch: one block owns one graph at a time and runs every peel round of it inside the
// kernel (Sec. 3 peeling, level-synchronous), then takes the next graph from a queue.
//
// For a graph of L <= kBlockMaxN vertices every closed ball is an L-bit row of W = L/32
// words, kept for every radius r = 1..h (B(x,1) = x plus its alive neighbours).  Balls of
// radius r are ORs of balls of radius r-1:  B(x,r) = OR over z in {x} ∪ N(x) of B(z,r-1),  and
//     sup(e,h) = |B(u,h) ∩ B(v,h)| - 2                                   (Def. 2, Def. 3).
// A round takes the minimum alive support (k = max(k, min + 2)), removes every alive edge
// with sup <= k-2 (t(e) = k), and brings the rest up to date exactly:
//   * candidates C: the vertices within h-1 of a removed edge's endpoint before the round,
//     i.e. the OR of the endpoints' B(.,h-1) rows taken before any row changes (only their
//     balls can lose members: a lost path of at most h edges runs through a removed edge);
//   * the removed edges leave the radius-1 rows; then radius 2..h is recomputed for C, one
//     radius after the other (radius r only reads radius r-1, which is already final);
//   * every alive edge at a vertex whose radius-h row changed gets its support recomputed.
// A round is a chain of short steps over a few thousand words, so a block holds everything in
// shared memory where it fits (about 600 vertices at h = 3: rows, 16-bit neighbour lists with
// the dead slots marked, edge endpoints, supports), runs 1,024 threads, and lists the
// candidates, changed vertices and affected edges before it works on them.  Larger graphs keep
// the same arrays in the block's global scratch.  (256 threads with everything in global
// memory, walking slot -> edge -> support -> row for every neighbour: 101 ms against 12.8 ms
// for 256 graphs of 50 to 600 vertices.)
// Graphs are taken largest first so that the long ones start early.
#include <algorithm>
#include <climits>
#include <cstring>
#include <string>
#include <vector>

#include "htd_internal.h"

namespace htd {

namespace {

constexpr int kBB = 1024;  // threads per block
constexpr int kBBWarps = kBB / 32;
constexpr uint16_t kDead = 0xffff;  // neighbour slot of a removed edge
constexpr int64_t kBlockSmem = 220 * 1024;  // arrays of a graph a block keeps in shared memory

// Reads of the union arrays a block needs for its graph (global ids; the graph's vertices are
// [v0, v0 + L) and its edges [e0, e0 + m) of the union).
struct BlockGraphDesc {
    const int32_t *row_ptr;
    const int32_t *col;
    const int32_t *eu;
    const int32_t *ev;
    const int32_t *slot_lo;
    const int32_t *slot_hi;
    int32_t *out;       // t(e,h) of the graph's edges, in the union's (canonical) order
    int64_t e0, m;
    int32_t v0, L, h;
    int32_t global;     // the arrays are in the block's global scratch
};

// A graph's working arrays, in this order, each from a multiple of 16 bytes on.
struct BlockLayout {
    int64_t rows, sup, ends, list, nbr, rp, vl, bytes;
    __host__ __device__ static int64_t up(int64_t b) { return (b + 15) & ~(int64_t)15; }
    __host__ __device__ BlockLayout(int64_t L, int64_t m, int h) {
        const int64_t W = (L + 31) >> 5;
        int64_t at = 0;
        rows = at;                      // h x L x W words
        at = up(at + 4 * h * L * W);
        sup = at;                       // m supports (INT_MAX: removed)
        at = up(at + 4 * m);
        ends = at;                      // m x (u, v)
        at = up(at + 4 * m);
        list = at;                      // m: the round's removed, then affected edges
        at = up(at + 4 * m);
        nbr = at;                       // 2m neighbours
        at = up(at + 4 * m);
        rp = at;                        // L + 1 row offsets
        at = up(at + 4 * (L + 1));
        vl = at;                        // L: endpoints, then candidates
        at = up(at + 2 * L);
        bytes = at;
    }
};

// Lists the members of an L-bit set (W words), in no order; *count is zero before.
__device__ __forceinline__ void bb_list(const uint32_t *set, int W, uint16_t *out, int32_t *count) {
    for (int w = threadIdx.x; w < W; w += kBB) {
        uint32_t v = set[w];
        if (!v) continue;
        int at = atomicAdd(count, __popc(v));
        while (v) {
            out[at++] = (uint16_t)((w << 5) + __ffs(v) - 1);
            v &= v - 1u;
        }
    }
}

// |bu ∩ bv| - 2 by a group of G lanes (every lane of the group returns it).
template <int G>
__device__ __forceinline__ int bb_support(const uint32_t *bu, const uint32_t *bv, int W) {
    int c = 0;
    for (int w = threadIdx.x & (G - 1); w < W; w += G) c += __popc(bu[w] & bv[w]);
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    return c - 2;
}

// Supports of the n edges of `list` (edges 0..n-1 if null), G lanes each.
template <int G>
__device__ __forceinline__ void bb_supports(const int32_t *list, int n, const ushort2 *ends, const uint32_t *rh,
                                            int W, int32_t *sup) {
    const int g = threadIdx.x / G;
    for (int i0 = 0; i0 < n; i0 += kBB / G) {  // whole warps: the groups' shuffles need every lane
        const int i = i0 + g;
        const int e = i < n ? (list ? list[i] : i) : 0;
        const ushort2 uv = ends[e];
        const int s = bb_support<G>(rh + (int64_t)uv.x * W, rh + (int64_t)uv.y * W, W);
        if (i < n && (threadIdx.x & (G - 1)) == 0) sup[e] = s;
    }
}

__global__ void __launch_bounds__(kBB, 1) k_batch_block(const BlockGraphDesc *__restrict__ gd, int32_t count,
                                                        unsigned char *scratch, int64_t stride, int32_t *queue,
                                                        unsigned long long *rounds_total) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t E[kBlockMaxN / 32], C[kBlockMaxN / 32], CH[kBlockMaxN / 32];
    __shared__ int32_t s_g, s_min[2], s_nf, s_nv, s_na;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (;;) {
        if (tid == 0) s_g = atomicAdd(queue, 1);
        __syncthreads();
        const int gi = s_g;
        __syncthreads();
        if (gi >= count) break;
        const BlockGraphDesc G = gd[gi];
        const int L = G.L, h = G.h, W = (L + 31) >> 5, m = (int)G.m;
        const BlockLayout lay(L, G.m, h);
        unsigned char *base = G.global ? scratch + (int64_t)blockIdx.x * stride : smem;
        uint32_t *const rows = reinterpret_cast<uint32_t *>(base + lay.rows);
        int32_t *const sup = reinterpret_cast<int32_t *>(base + lay.sup);
        ushort2 *const ends = reinterpret_cast<ushort2 *>(base + lay.ends);
        int32_t *const list = reinterpret_cast<int32_t *>(base + lay.list);
        uint16_t *const nbr = reinterpret_cast<uint16_t *>(base + lay.nbr);
        int32_t *const rp = reinterpret_cast<int32_t *>(base + lay.rp);
        uint16_t *const vl = reinterpret_cast<uint16_t *>(base + lay.vl);
        const int64_t rad = (int64_t)L * W;  // words of one radius
        uint32_t *const rh = rows + (int64_t)(h - 1) * rad;
        const int32_t s0 = G.row_ptr[G.v0];
        // lanes to words of a row: several vertices per warp while a row is shorter than one
        const int per = W < 32 ? 32 / W : 1;
        const int vi = W < 32 ? lane / W : 0, w0 = W < 32 ? lane % W : lane;
        // B(.,r) of the vertices `ids` (all if null) from the rows of radius r - 1; changed
        // vertices of the last radius are marked in CH
        auto build = [&](int r, const uint16_t *ids, int n, bool mark) {
            const uint32_t *in = rows + (int64_t)(r - 2) * rad;
            uint32_t *out = rows + (int64_t)(r - 1) * rad;
            if (vi < per) {
                for (int i = wid * per + vi; i < n; i += kBBWarps * per) {
                    const int x = ids ? ids[i] : i;
                    const int b = rp[x], e = rp[x + 1];
                    for (int w = w0; w < W; w += 32) {
                        uint32_t acc = in[(int64_t)x * W + w];
#pragma unroll 4
                        for (int s = b; s < e; s++) {
                            const int z = nbr[s];
                            if (z != kDead) acc |= in[(int64_t)z * W + w];
                        }
                        uint32_t *const dst = out + (int64_t)x * W + w;
                        if (mark && acc != *dst) atomicOr(&CH[x >> 5], 1u << (x & 31));
                        *dst = acc;
                    }
                }
            }
            __syncthreads();
        };
        auto supports = [&](const int32_t *l, int n) {
            if (W <= 32) bb_supports<8>(l, n, ends, rh, W, sup);
            else bb_supports<32>(l, n, ends, rh, W, sup);
            __syncthreads();
        };
        // the graph's arrays, and radius 1: x and its neighbours
        for (int x = tid; x <= L; x += kBB) rp[x] = G.row_ptr[G.v0 + x] - s0;
        for (int s = tid; s < 2 * m; s += kBB) nbr[s] = (uint16_t)(G.col[s0 + s] - G.v0);
        for (int e = tid; e < m; e += kBB)
            ends[e] = make_ushort2((uint16_t)(G.eu[G.e0 + e] - G.v0), (uint16_t)(G.ev[G.e0 + e] - G.v0));
        for (int64_t i = tid; i < rad; i += kBB) rows[i] = 0u;
        __syncthreads();
        for (int x = wid; x < L; x += kBBWarps) {
            uint32_t *r1 = rows + (int64_t)x * W;
            if (lane == 0) atomicOr(&r1[x >> 5], 1u << (x & 31));
            for (int s = rp[x] + lane; s < rp[x + 1]; s += 32) atomicOr(&r1[nbr[s] >> 5], 1u << (nbr[s] & 31));
        }
        __syncthreads();
        for (int r = 2; r <= h; r++) build(r, nullptr, L, false);
        supports(nullptr, m);
        int k = 2, round = 0;
        if (tid == 0) s_min[0] = s_min[1] = INT_MAX;
        __syncthreads();
        for (; round <= m; round++) {
            // level: k = max(k, min alive sup + 2)
            int mn = INT_MAX;
            for (int e = tid; e < m; e += kBB) mn = min(mn, sup[e]);
            mn = __reduce_min_sync(0xffffffffu, mn);
            if (lane == 0 && mn != INT_MAX) atomicMin(&s_min[round & 1], mn);
            for (int w = tid; w < W; w += kBB) E[w] = C[w] = CH[w] = 0u;
            if (tid == 0) s_nf = s_nv = s_na = 0;
            __syncthreads();
            mn = s_min[round & 1];
            if (tid == 0) s_min[(round & 1) ^ 1] = INT_MAX;
            if (mn == INT_MAX) break;  // every edge removed
            k = max(k, mn + 2);
            // remove the frontier: every alive edge with sup <= k - 2 (t = k)
            for (int e = tid; e < m; e += kBB) {
                if (sup[e] > k - 2) continue;
                const ushort2 uv = ends[e];
                G.out[e] = k;
                sup[e] = INT_MAX;
                list[atomicAdd(&s_nf, 1)] = e;
                atomicOr(&E[uv.x >> 5], 1u << (uv.x & 31));
                atomicOr(&E[uv.y >> 5], 1u << (uv.y & 31));
                nbr[G.slot_lo[G.e0 + e] - s0] = kDead;
                nbr[G.slot_hi[G.e0 + e] - s0] = kDead;
            }
            __syncthreads();
            // candidates: endpoints (h = 1) or the OR of their radius h-1 rows, before any
            // row changes
            const uint32_t *cand = E;
            if (h > 1) {
                bb_list(E, W, vl, &s_nv);
                __syncthreads();
                const uint32_t *in = rows + (int64_t)(h - 2) * rad;
                if (vi < per) {
                    for (int i = wid * per + vi; i < s_nv; i += kBBWarps * per)
                        for (int w = w0; w < W; w += 32) {
                            const uint32_t v = in[(int64_t)vl[i] * W + w];
                            if (v & ~C[w]) atomicOr(&C[w], v);
                        }
                }
                cand = C;
                __syncthreads();
                if (tid == 0) s_nv = 0;
                __syncthreads();
                bb_list(C, W, vl, &s_nv);
            }
            // the removed edges leave the radius-1 rows
            const int nf = s_nf;
            for (int i = tid; i < nf; i += kBB) {
                const ushort2 uv = ends[list[i]];
                atomicAnd(&rows[(int64_t)uv.x * W + (uv.y >> 5)], ~(1u << (uv.y & 31)));
                atomicAnd(&rows[(int64_t)uv.y * W + (uv.x >> 5)], ~(1u << (uv.x & 31)));
            }
            __syncthreads();
            // radius 2..h of the candidates, from the already updated radius below; at h = 1 the
            // endpoints' rows are the changed ones
            for (int r = 2; r <= h; r++) build(r, vl, s_nv, r == h);
            const uint32_t *changed = h > 1 ? CH : cand;
            // supports of the alive edges at a changed vertex
            for (int e = tid; e < m; e += kBB) {
                if (sup[e] == INT_MAX) continue;
                const ushort2 uv = ends[e];
                if (((changed[uv.x >> 5] >> (uv.x & 31)) | (changed[uv.y >> 5] >> (uv.y & 31))) & 1u)
                    list[atomicAdd(&s_na, 1)] = e;
            }
            __syncthreads();
            supports(list, s_na);
        }
        if (tid == 0) atomicAdd(rounds_total, (unsigned long long)round);
        __syncthreads();
    }
}

}  // namespace

// Decomposes the graphs (device pointers inside the descriptors) with one block per graph in a
// single launch.  Shared memory and scratch are sized from the largest graphs.
htd_status batch_block_run(const std::vector<BlockGraphDescHost> &graphs, cudaStream_t s,
                           int num_sms, int64_t *rounds_out) {
    if (graphs.empty()) return HTD_OK;
    std::vector<BlockGraphDesc> gd(graphs.size());
    int64_t smem = 0, stride = 0;
    for (size_t i = 0; i < graphs.size(); i++) {
        const BlockGraphDescHost &g = graphs[i];
        const int64_t bytes = BlockLayout(g.L, g.m, g.h).bytes;
        const bool global = bytes > kBlockSmem;
        if (global) stride = std::max(stride, (bytes + 255) & ~(int64_t)255);
        else smem = std::max(smem, bytes);
        gd[i] = BlockGraphDesc{g.row_ptr, g.col, g.eu, g.ev, g.slot_lo, g.slot_hi, g.out,
                               g.e0, g.m, g.v0, g.L, g.h, global ? 1 : 0};
    }
    // largest graphs first
    std::sort(gd.begin(), gd.end(), [](const BlockGraphDesc &a, const BlockGraphDesc &b) {
        return a.m * (int64_t)a.h > b.m * (int64_t)b.h;
    });
    int occ = 0;
    cudaError_t e = raise_smem_limit((const void *)k_batch_block, (size_t)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_batch_block, kBB, (size_t)smem);
    if (e != cudaSuccess || occ < 1) {
        set_last_error("batched blocks: no resident block fits");
        return HTD_ECUDA;
    }
    // every block that can be resident, bounded by the graphs and by the scratch
    size_t free_b = 0, total_b = 0;
    cudaMemGetInfo(&free_b, &total_b);
    int64_t grid = std::min<int64_t>((int64_t)num_sms * occ, (int64_t)gd.size());
    if (stride > 0) grid = std::max<int64_t>(1, std::min<int64_t>(grid, (int64_t)(free_b / 2) / stride));
    BlockGraphDesc *d_gd = nullptr;
    unsigned char *scratch = nullptr;
    unsigned long long *d_ctr = nullptr;  // rounds, then the queue head
    htd_status st = HTD_OK;
    if (stride > 0) e = dev_alloc(&scratch, grid * stride, s);
    if (e == cudaSuccess) e = dev_alloc(&d_gd, (int64_t)gd.size(), s);
    if (e == cudaSuccess) e = dev_alloc(&d_ctr, 2, s);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_gd, gd.data(), gd.size() * sizeof(BlockGraphDesc), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_ctr, 0, 16, s);
    if (e == cudaSuccess) {
        k_batch_block<<<(unsigned)grid, kBB, (size_t)smem, s>>>(d_gd, (int32_t)gd.size(), scratch, stride,
                                                                reinterpret_cast<int32_t *>(d_ctr + 1), d_ctr);
        add_launches(1);
        e = cudaGetLastError();
    }
    unsigned long long hr = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hr, d_ctr, 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        set_last_error(std::string("batched blocks: ") + cudaGetErrorString(e));
        st = e == cudaErrorMemoryAllocation ? HTD_ENOMEM : HTD_ECUDA;
    }
    if (rounds_out) *rounds_out = (int64_t)hr;
    dev_free(scratch, s);
    dev_free(d_gd, s);
    dev_free(d_ctr, s);
    return st;
}

}  // namespace htd
