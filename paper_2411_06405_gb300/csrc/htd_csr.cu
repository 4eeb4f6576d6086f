// htd_csr.cu -- normalise an undirected edge list and build the CSR + edge ids.
//
// Graph model of Sec. 2 (simple undirected graph): self-loops are dropped, each pair is
// stored in both rows, every row is sorted and deduplicated (which merges duplicate and
// reversed pairs), and edge e is the e-th pair (u,v), u < v, in lexicographic order.
//
// Steps (all on the device; two host synchronisations, to size the outputs and to read
// the error flag and m):
//   1. count row lengths (ids checked against [0,n));     2. scan -> raw row offsets;
//   3. scatter both directions;                           4. sort + unique each row by size
//      class: <= 256 (one warp, register bitonic), <= 4096 (one block, shared-memory
//      bitonic), larger (one block, n-bit shared-memory set read back in order), counting
//      its neighbours and those above the row id;
//   5. one scan of both counts, packed, -> row_ptr and the first edge id of each row;
//   6. one thread per slot: compacted column, edge id, endpoints.
// Steps 5 and 6 read sorted raw rows, so hub rows are spread over every block (a warp per row
// left them to single warps: on R-MAT 18 compaction and edge ids took 745 us, one thread per
// slot 95 us).
#include <cstdio>

#include "htd_internal.h"
#include "htd_scan.cuh"

namespace htd {
namespace {

constexpr int kBlock = 256;
constexpr int kWarpMax = 256;  // longest row one warp sorts
constexpr int kMedMax = 4096;

// Row length and number of neighbours above the row id, as one 64-bit value (both sums of a
// scan fit 31 bits).
__device__ __forceinline__ int64_t pack_row(int len, int above) { return (int64_t)above << 32 | len; }
__host__ __device__ __forceinline__ int row_len(int64_t v) { return (int)(v & 0xffffffff); }
__host__ __device__ __forceinline__ int row_above(int64_t v) { return (int)(v >> 32); }

__global__ void k_csr_count(const int32_t *__restrict__ src, const int32_t *__restrict__ dst,
                            int64_t m_in, int32_t n, int32_t *__restrict__ deg,
                            int32_t *__restrict__ err) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m_in;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t a = src[i], b = dst[i];
        if (a < 0 || a >= n || b < 0 || b >= n) {
            atomicOr(err, 1);
            continue;
        }
        if (a == b) continue;
        atomicAdd(&deg[a], 1);
        atomicAdd(&deg[b], 1);
    }
}

__global__ void k_csr_scatter(const int32_t *__restrict__ src, const int32_t *__restrict__ dst,
                              int64_t m_in, int32_t n, const int32_t *__restrict__ off,
                              int32_t *__restrict__ fill, int32_t *__restrict__ colraw) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m_in;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t a = src[i], b = dst[i];
        if (a < 0 || a >= n || b < 0 || b >= n || a == b) continue;
        int pa = atomicAdd(&fill[a], 1);
        colraw[off[a] + pa] = b;
        int pb = atomicAdd(&fill[b], 1);
        colraw[off[b] + pb] = a;
    }
}

// Sorts and deduplicates a row of at most 32 * K entries with one warp, in registers: entry
// 32 * k + lane is v[k], so exchanges at distance 32 and more stay within the lane.
template <int K>
__device__ __forceinline__ void warp_sort_row(int x, int b, int len, int32_t *__restrict__ colraw,
                                              int64_t *__restrict__ rows) {
    const int lane = threadIdx.x & 31;
    int v[K];
#pragma unroll
    for (int k = 0; k < K; k++) v[k] = 32 * k + lane < len ? colraw[b + 32 * k + lane] : INT_MAX;
#pragma unroll
    for (int s = 2; s <= 32 * K; s <<= 1) {
#pragma unroll
        for (int j = s >> 1; j > 0; j >>= 1) {
#pragma unroll
            for (int k = 0; k < K; k++) {
                const bool up = ((32 * k + lane) & s) == 0;
                if (j >= 32) {
                    const int o = k ^ (j >> 5);
                    if (o > k) {
                        const int lo = min(v[k], v[o]), hi = max(v[k], v[o]);
                        v[k] = up ? lo : hi;
                        v[o] = up ? hi : lo;
                    }
                } else {
                    const int p = __shfl_xor_sync(0xffffffffu, v[k], j);
                    v[k] = (((lane & j) == 0) == up) ? min(v[k], p) : max(v[k], p);
                }
            }
        }
    }
    int at = 0, above = 0, last = -1;  // last: the entry before v[k] of lane 0
#pragma unroll
    for (int k = 0; k < K; k++) {
        int prev = __shfl_up_sync(0xffffffffu, v[k], 1);
        if (lane == 0) prev = last;
        last = __shfl_sync(0xffffffffu, v[k], 31);
        const bool keep = v[k] != INT_MAX && v[k] != prev;
        const unsigned bal = __ballot_sync(0xffffffffu, keep);
        if (keep) colraw[b + at + __popc(bal & lanemask_lt())] = v[k];
        at += __popc(bal);
        above += __popc(__ballot_sync(0xffffffffu, keep && v[k] > x));
    }
    if (lane == 0) rows[x] = pack_row(at, above);
}

// Rows of length <= 256: one warp each.  Longer rows are listed for the block kernels.
__global__ void k_row_sort_warp(int32_t n, const int32_t *__restrict__ off,
                                int32_t *__restrict__ colraw, int64_t *__restrict__ rows,
                                int32_t *__restrict__ med_list, int32_t *__restrict__ med_cnt,
                                int32_t *__restrict__ big_list, int32_t *__restrict__ big_cnt) {
    const int lane = threadIdx.x & 31;
    const int nwarps = gridDim.x * (blockDim.x >> 5);
    for (int x = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; x < n; x += nwarps) {
        const int b = off[x], len = off[x + 1] - b;
        if (len > kWarpMax) {
            if (lane == 0) {
                if (len <= kMedMax) med_list[atomicAdd(med_cnt, 1)] = x;
                else big_list[atomicAdd(big_cnt, 1)] = x;
            }
        } else if (len > 128) {
            warp_sort_row<8>(x, b, len, colraw, rows);
        } else if (len > 64) {
            warp_sort_row<4>(x, b, len, colraw, rows);
        } else if (len > 32) {
            warp_sort_row<2>(x, b, len, colraw, rows);
        } else {
            warp_sort_row<1>(x, b, len, colraw, rows);
        }
    }
}

// Rows of length 257..4096: one block each, bitonic sort in shared memory.
__global__ void __launch_bounds__(kBlock)
k_row_sort_block(const int32_t *__restrict__ list, const int32_t *__restrict__ cnt,
                 const int32_t *__restrict__ off, int32_t *__restrict__ colraw,
                 int64_t *__restrict__ rows_out) {
    __shared__ int32_t buf[kMedMax];
    __shared__ int32_t scratch[kBlock / 32];
    const int rows = *cnt;
    for (int r = blockIdx.x; r < rows; r += gridDim.x) {
        const int x = list[r];
        const int b = off[x], len = off[x + 1] - b;
        int P = 64;
        while (P < len) P <<= 1;
        for (int i = threadIdx.x; i < P; i += kBlock) buf[i] = (i < len) ? colraw[b + i] : INT_MAX;
        __syncthreads();
        for (int k = 2; k <= P; k <<= 1) {
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int i = threadIdx.x; i < (P >> 1); i += kBlock) {
                    int a = 2 * i - (i & (j - 1));
                    int c = a + j;
                    bool ascending = (a & k) == 0;
                    int va = buf[a], vc = buf[c];
                    if ((va > vc) == ascending) {
                        buf[a] = vc;
                        buf[c] = va;
                    }
                }
                __syncthreads();
            }
        }
        // unique + ordered compaction: thread t owns items [t*per, (t+1)*per)
        const int per = (len + kBlock - 1) / kBlock;
        const int lo = threadIdx.x * per, hi = min(len, lo + per);
        int keep = 0, above = 0;
        for (int p = lo; p < hi; p++) {
            const bool first = p == 0 || buf[p] != buf[p - 1];
            keep += first;
            above += first && buf[p] > x;
        }
        above = block_sum<kBlock, int>(above, scratch);
        int total;
        int pos = block_exclusive_scan<kBlock, int>(keep, &total, scratch);
        for (int p = lo; p < hi; p++) {
            if (p == 0 || buf[p] != buf[p - 1]) colraw[b + pos++] = buf[p];
        }
        if (threadIdx.x == 0) rows_out[x] = pack_row(total, above);
        __syncthreads();
    }
}

// Rows longer than 4096: one block each; the row is set into an n-bit shared-memory set
// and read back in increasing id order, which sorts and deduplicates it.
__global__ void __launch_bounds__(kBlock)
k_row_sort_bitset(const int32_t *__restrict__ list, const int32_t *__restrict__ cnt,
                  const int32_t *__restrict__ off, int32_t *__restrict__ colraw,
                  int64_t *__restrict__ rows_out, int32_t W) {
    extern __shared__ uint32_t bits[];
    __shared__ int32_t scratch[kBlock / 32];
    __shared__ int32_t warp_base[kBlock / 32];
    constexpr int NW = kBlock / 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // word segment of each warp, a multiple of 32 words
    const int seg = ((W + NW - 1) / NW + 31) & ~31;
    const int rows = *cnt;
    for (int r = blockIdx.x; r < rows; r += gridDim.x) {
        const int x = list[r];
        const int b = off[x], len = off[x + 1] - b;
        for (int i = threadIdx.x; i < W; i += kBlock) bits[i] = 0u;
        __syncthreads();
        for (int i = threadIdx.x; i < len; i += kBlock) {
            int v = colraw[b + i];
            atomicOr(&bits[v >> 5], 1u << (v & 31));
        }
        __syncthreads();
        const int w0 = wid * seg, w1 = min(W, w0 + seg);
        int c = 0, above = 0;
        for (int i = w0 + lane; i < w1; i += 32) {
            const uint32_t word = bits[i];
            c += __popc(word);
            if (i > (x >> 5)) above += __popc(word);
            else if (i == (x >> 5)) above += __popc(word & ~((2u << (x & 31)) - 1u));
        }
        c = warp_sum(c);
        above = block_sum<kBlock, int>(above, scratch);
        int total;
        int ex = block_exclusive_scan<kBlock, int>(lane == 0 ? c : 0, &total, scratch);
        if (lane == 0) warp_base[wid] = ex;
        __syncthreads();
        int run = warp_base[wid];
        for (int i0 = w0; i0 < w1; i0 += 32) {
            int i = i0 + lane;
            uint32_t word = (i < w1) ? bits[i] : 0u;
            int pc = __popc(word);
            int incl = pc;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            int pos = run + incl - pc;
            while (word) {
                int bit = __ffs(word) - 1;
                word &= word - 1;
                colraw[b + pos++] = i * 32 + bit;
            }
            run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (threadIdx.x == 0) rows_out[x] = pack_row(total, above);
        __syncthreads();
    }
}

// row_ptr from the packed scan, and the sum of the squared degrees.
__global__ void k_row_ptr(int32_t n, const int64_t *__restrict__ rows, const int64_t *__restrict__ first,
                          int32_t *__restrict__ row_ptr, unsigned long long *__restrict__ deg2) {
    unsigned long long squares = 0ull;
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x <= n; x += gridDim.x * blockDim.x) {
        row_ptr[x] = row_len(first[x]);
        const unsigned len = x < n ? (unsigned)row_len(rows[x]) : 0u;
        squares += (unsigned long long)len * len;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) squares += __shfl_xor_sync(0xffffffffu, squares, o);
    if ((threadIdx.x & 31) == 0 && squares) atomicAdd(deg2, squares);
}

constexpr int kSlotsPerBlock = 4 * kBlock;

// Adjacency slots and edges, one thread per slot.  `rows` and `first`: length and neighbours
// above the id of each row, and their exclusive sums (first slot, first edge id).  The rows a
// block's slots lie in are found once; a thread searches among those.
__global__ void __launch_bounds__(kBlock) k_slots(int32_t n, int32_t two_m, const int32_t *__restrict__ off,
                                                 const int32_t *__restrict__ colraw,
                                                 const int64_t *__restrict__ rows,
                                                 const int64_t *__restrict__ first,
                                                 const int32_t *__restrict__ row_ptr,
                                                 int32_t *__restrict__ col, int32_t *__restrict__ slot_eid,
                                                 int32_t *__restrict__ eu, int32_t *__restrict__ ev,
                                                 int32_t *__restrict__ slot_lo, int32_t *__restrict__ slot_hi) {
    __shared__ int32_t s_row[2];
    // last row starting at or before s, in [lo, hi]
    auto row_of = [&](int s, int lo, int hi) {
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (row_ptr[mid] <= s) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    };
    for (int64_t b = (int64_t)blockIdx.x * kSlotsPerBlock; b < two_m; b += (int64_t)gridDim.x * kSlotsPerBlock) {
        if (threadIdx.x < 2)
            s_row[threadIdx.x] = row_of((int)min((int64_t)two_m - 1, b + threadIdx.x * (kSlotsPerBlock - 1)), 0, n - 1);
        __syncthreads();
        const int r0 = s_row[0], r1 = s_row[1];
#pragma unroll
        for (int k = 0; k < kSlotsPerBlock / kBlock; k++) {
            const int64_t sl = b + k * kBlock + threadIdx.x;
            if (sl >= two_m) break;
            const int s = (int)sl, x = row_of(s, r0, r1);
            const int64_t fx = first[x], lx = rows[x];
            const int j = s - row_len(fx);
            const int y = colraw[off[x] + j];
            col[s] = y;
            if (y > x) {
                const int e = row_above(fx) + j - (row_len(lx) - row_above(lx));
                eu[e] = x;
                ev[e] = y;
                slot_eid[s] = e;
                slot_lo[e] = s;
            } else {
                // place of x among the neighbours of y above y
                const int64_t fy = first[y], ly = rows[y];
                const int32_t *up = colraw + off[y] + (row_len(ly) - row_above(ly));
                int lo = 0, hi = row_above(ly) - 1;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (up[mid] < x) lo = mid + 1;
                    else hi = mid;
                }
                const int e = row_above(fy) + lo;
                slot_eid[s] = e;
                slot_hi[e] = s;
            }
        }
        __syncthreads();
    }
}

int grid_for(int64_t work, int per_block, int cap) {
    int64_t g = (work + per_block - 1) / per_block;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

}  // namespace

void free_graph_dev(GraphDev *g, cudaStream_t s) {
    for (void *p : {(void *)g->row_ptr, (void *)g->col, (void *)g->slot_eid, (void *)g->eu, (void *)g->ev,
                    (void *)g->slot_lo, (void *)g->slot_hi})
        dev_free(p, s);
    *g = GraphDev{};
}

#define HTD_TRY(...)                                                                   \
    do {                                                                                \
        cudaError_t _e = (__VA_ARGS__);                                                        \
        if (_e != cudaSuccess) {                                                        \
            set_last_error(std::string(#__VA_ARGS__) + ": " + cudaGetErrorString(_e));         \
            st = (_e == cudaErrorMemoryAllocation) ? HTD_ENOMEM : HTD_ECUDA;            \
            goto done;                                                                  \
        }                                                                               \
    } while (0)

htd_status build_csr_device(int32_t n, const int32_t *src, const int32_t *dst, int64_t m_in,
                            cudaStream_t s, GraphDev *out, int64_t *launches) {
    htd_status st = HTD_OK;
    GraphDev g;
    int dev = 0;
    int nsm = 0;
    int32_t *deg = nullptr, *off = nullptr, *fill = nullptr, *colraw = nullptr;
    int32_t *lists = nullptr, *counters = nullptr;
    int64_t *rows = nullptr, *first = nullptr;
    unsigned long long *deg2 = nullptr;
    void *tmp = nullptr;
    int32_t host_ctr[4] = {0, 0, 0, 0};
    int64_t nn = n > 0 ? n : 1;
    int64_t raw_slots = 2 * m_in;
    const int W = (n + 31) / 32;
    const size_t smem_big = (size_t)((W + 3) & ~3) * sizeof(uint32_t);
    int64_t totals = 0;  // slots and edges, packed
    int32_t two_m = 0;

    HTD_TRY(cudaGetDevice(&dev));
    HTD_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    g.device = dev;
    g.n = n;
    HTD_TRY(dev_alloc(&deg, nn, s));
    HTD_TRY(dev_alloc(&off, (nn + 1), s));
    HTD_TRY(dev_alloc(&fill, nn, s));
    HTD_TRY(dev_alloc(&colraw, raw_slots, s));
    HTD_TRY(dev_alloc(&rows, nn, s));
    HTD_TRY(dev_alloc(&first, nn + 1, s));
    HTD_TRY(dev_alloc(&lists, 2 * nn, s));
    HTD_TRY(dev_alloc(&counters, 6, s));
    deg2 = reinterpret_cast<unsigned long long *>(counters + 4);
    HTD_TRY(dev_alloc_bytes(&tmp, scan_temp_bytes(nn + raw_slots), s));
    HTD_TRY(dev_alloc(&g.row_ptr, (nn + 1), s));
    HTD_TRY(cudaMemsetAsync(deg, 0, nn * sizeof(int32_t), s));
    HTD_TRY(cudaMemsetAsync(fill, 0, nn * sizeof(int32_t), s));
    HTD_TRY(cudaMemsetAsync(counters, 0, 6 * sizeof(int32_t), s));

    if (m_in > 0) {
        int gb = grid_for(m_in, kBlock, nsm * 8);
        k_csr_count<<<gb, kBlock, 0, s>>>(src, dst, m_in, n, deg, counters + 2);
        (*launches)++;
    }
    HTD_TRY(scan_exclusive<int32_t, int32_t>(deg, off, n, tmp, s, launches));
    if (m_in > 0) {
        int gb = grid_for(m_in, kBlock, nsm * 8);
        k_csr_scatter<<<gb, kBlock, 0, s>>>(src, dst, m_in, n, off, fill, colraw);
        (*launches)++;
    }
    if (n > 0) {
        int gw = grid_for((int64_t)n * 32, kBlock, nsm * 16);
        k_row_sort_warp<<<gw, kBlock, 0, s>>>(n, off, colraw, rows, lists, counters, lists + nn,
                                              counters + 1);
        k_row_sort_block<<<nsm * 4, kBlock, 0, s>>>(lists, counters, off, colraw, rows);
        if (smem_big > 48 * 1024) {
            HTD_TRY(raise_smem_limit((const void *)k_row_sort_bitset, smem_big));
        }
        k_row_sort_bitset<<<nsm, kBlock, smem_big, s>>>(lists + nn, counters + 1, off, colraw,
                                                        rows, W);
        *launches += 3;
    }
    HTD_TRY(cudaGetLastError());
    HTD_TRY(scan_exclusive<int64_t, int64_t>(rows, first, n, tmp, s, launches));
    k_row_ptr<<<grid_for((int64_t)n + 1, kBlock, nsm * 8), kBlock, 0, s>>>(n, rows, first, g.row_ptr, deg2);
    (*launches)++;
    HTD_TRY(cudaMemcpyAsync(&totals, first + n, sizeof(totals), cudaMemcpyDeviceToHost, s));
    HTD_TRY(cudaMemcpyAsync(host_ctr, counters, 4 * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    HTD_TRY(cudaStreamSynchronize(s));
    if (host_ctr[2] != 0) {
        set_last_error("htd_build_csr: vertex id outside [0, n)");
        st = HTD_EINVAL;
        goto done;
    }
    two_m = row_len(totals);
    g.m = two_m / 2;
    {
        int64_t mm = g.m > 0 ? g.m : 1;
        HTD_TRY(dev_alloc(&g.col, 2 * mm, s));
        HTD_TRY(dev_alloc(&g.slot_eid, 2 * mm, s));
        HTD_TRY(dev_alloc(&g.eu, mm, s));
        HTD_TRY(dev_alloc(&g.ev, mm, s));
        HTD_TRY(dev_alloc(&g.slot_lo, mm, s));
        HTD_TRY(dev_alloc(&g.slot_hi, mm, s));
    }
    if (two_m > 0) {
        k_slots<<<grid_for(two_m, kSlotsPerBlock, nsm * 16), kBlock, 0, s>>>(n, two_m, off, colraw, rows, first,
                                                                            g.row_ptr, g.col, g.slot_eid, g.eu, g.ev,
                                                                            g.slot_lo, g.slot_hi);
        (*launches)++;
    }
    HTD_TRY(cudaMemcpyAsync(&g.deg2, deg2, sizeof(g.deg2), cudaMemcpyDeviceToHost, s));
    HTD_TRY(cudaGetLastError());
    HTD_TRY(cudaStreamSynchronize(s));

done:
    dev_free(deg, s);
    dev_free(off, s);
    dev_free(fill, s);
    dev_free(colraw, s);
    dev_free(rows, s);
    dev_free(first, s);
    dev_free(lists, s);
    dev_free(counters, s);
    dev_free(tmp, s);
    if (st != HTD_OK) {
        cudaStreamSynchronize(s);
        free_graph_dev(&g, s);
        return st;
    }
    *out = g;
    return HTD_OK;
}

}  // namespace htd
