// htd_loss.cu -- exact incremental h-support updates for h <= 3 and the kernels that run the rounds.
//
// For h <= 2 the members a removal can take out of a ball are few and can be listed: an
// old path of length <= h that used a removed edge (a,b) is a-b itself, x-a-b with x in
// N(a), or a-b-w with w in N(b).  So after removing the frontier F of a round the only
// vertex pairs that can stop being within distance h of each other are
//     {a,b}, {a,z} for z in N_old(b) \ {a}, and {b,z} for z in N_old(a) \ {b}
// for every (a,b) in F (for h = 1 only {a,b}).  Each such pair is tested in the new graph
// (adjacent, or for h = 2 a common alive neighbour); a pair that fails is "lost": each
// endpoint leaves the other's ball (distance is symmetric).  Lost pairs are deduplicated
// in an open-addressing hash set, or, where memory allows a second copy of the ball matrix
// (the "twin"), by clearing the pair's bits there: the twin is then the matrix of B_new.
//
// The h-support of an alive edge (x,y), x < y, then drops by exactly
//     |L(x) ∩ B_old(y)| + |L(y) ∩ B_new(x)|,
// where L(v) = B_old(v) \ B_new(v) (Def. 3: sup = |B(x) ∩ B(y)| - 2, and a member that
// leaves B(x) ∩ B(y) either leaves B(x), or stays in B(x) and leaves B(y)).  The first
// term is counted against the stored balls before the lost members are cleared, the
// second after.  Every step is exact integer arithmetic; no ball is rebuilt.
//
// A round whose lost pairs outgrow the table is processed in batches: the deltas of
// successive batches telescope (each is taken between the stored balls before and after
// that batch), and a pair whose stored bit is already clear was handled by an earlier
// batch of the same round, so it is skipped.  Detection records the first frontier edge
// side it could not finish; the next round slot resumes there without selecting anew.
#include <algorithm>
#include <climits>
#include <cstdint>

#include "htd_internal.h"
#include "htd_round.cuh"

namespace htd {
namespace {

constexpr int kBlock = 256;
constexpr unsigned long long kEmpty = ~0ull;

struct LossArgs {
    int64_t m;
    const int32_t *slot_lo;
    const int32_t *slot_hi;
    int32_t *truss;
    int32_t *stamp_w;
    int32_t *frontier_w;
    int32_t *col_live_w;
    int32_t *deg_alive_w;
    uint32_t *hub_bits_w;
    int32_t h;
    int32_t lost_max;
    unsigned cap_mask;
    const int32_t *row_ptr;
    const int32_t *col;
    const int32_t *col_live;
    const int32_t *slot_eid;
    const int32_t *eu;
    const int32_t *ev;
    const int32_t *frontier;
    const int32_t *stamp;
    uint32_t *pool;
    const int64_t *ball_off;
    const int32_t *ball_nw;
    const int2 *ball_meta;
    int32_t *ball_size;
    unsigned long long *keys;
    int4 *lost;
    int32_t *sup;
    int32_t *vtouch;
    const int32_t *deg_alive;
    const int32_t *hub_slot;
    const uint32_t *hub_bits;
    int32_t Wpad;
    int32_t dense_all;  // every ball dense at pool + x * Wpad (no metadata lookup)
    int32_t hub_all;    // every vertex has its alive-adjacency set, at row x
    int32_t pitems_cap;
    int4 *pitems;       // two per item: (edge side, first slot, x, y), (row x, end, row y, end)
    int32_t uitems_cap;
    int4 *uitems;
    long long upd_budget;
    DevStatus *st;
    // h = 3: radius-2 balls and the round's radius-2 losses
    int32_t h3;         // incremental h = 3 round: overflows halt the round (host rebuild)
    uint32_t *pool2;    // dense radius-2 balls, row x at x * Wpad
    int32_t *ball_size2;
    unsigned long long *keys2;
    unsigned cap2_mask;
    int4 *lost2;
    int32_t lost2_max;
    int32_t c3items_cap;
    int4 *c3items;
    int32_t *touch2;    // h = 3: round in which the vertex last lost a radius-2 member
    // Twin ball matrices (null without): pool and pool2 hold the balls of before the batch,
    // these the same minus the batch's losses so far.
    uint32_t *pool_new;
    uint32_t *pool2_new;
    int32_t cluster;    // the slot starts with the cluster round kernel
    int32_t launch;     // its number, from 1, among the launches of that kernel in this peel
    int32_t wait_polls; // cluster round kernel: polls without progress after which a wait gives up
    int32_t no_helpers; // cluster round kernel: helpers end at once (a test of a busy device)
    int32_t max_split;  // phase launches: log2 of the warps one detection item may take
    int32_t timer;      // add the time of each phase to the status block
    int32_t win_cap;    // cluster round kernel: edges its window and next-frontier lists hold
    int32_t *win;
    int32_t *next;
    const int4 *erec;   // per edge: (u, v, slot in u's row, slot in v's row), (row u, row v)
    const int4 *srec;   // per adjacency slot: (neighbour, its row, its row's end, edge)
};

__device__ __forceinline__ unsigned long long pair_key(int p, int q) {
    const unsigned a = (unsigned)min(p, q), b = (unsigned)max(p, q);
    return ((unsigned long long)a << 32) | b;
}

// First slot of the pair {p,q} in a table of mask + 1 slots: multiplicative hashing (Knuth) of
// both ids in 32 bits.  (With a 64-bit mix of the key, its two wide multiplications were a
// third of the instructions of a support update that probes.)
__device__ __forceinline__ unsigned pair_slot(int p, int q, unsigned mask) {
    unsigned x = (unsigned)min(p, q) * 0x9e3779b1u + (unsigned)max(p, q) * 0x85ebca6bu;
    x ^= x >> 15;
    return x & mask;
}

// Status fields are written by other blocks between the phases of the persistent kernel:
// read them through the memory system, never from a register copy.
template <typename T>
__device__ __forceinline__ T vload(const T &x) {
    return *(const volatile T *)&x;
}

// A batch limit was reached at edge side u: h <= 2 resumes the round there in the next slot;
// an h = 3 round halts and the host finishes it by rebuilds.
__device__ __forceinline__ void overflow_at(const LossArgs &a, RoundCtr *c, int u) {
    if (a.h3) atomicOr(&c->halt, 1);
    else atomicMin(&c->overflow_unit, u);
}

// Round kernels do nothing once the peel is over or a round halted, and a phase launch of a
// slot with the cluster round kernel only runs from the phase that kernel left to it.
__device__ __forceinline__ bool round_idle(const LossArgs &a, RoundStage phase) {
    if (vload(a.st->alive) == 0 || vload(a.st->halt) != 0) return true;
    if (!a.cluster) return false;
    const int stage = vload(a.st->stage);
    return stage == kStageNone || stage > phase;
}

// Alive-adjacency set of p if p has one (high degree), else null.
__device__ __forceinline__ const uint32_t *hub_set(const LossArgs &a, int p, unsigned &reads) {
    if (a.hub_all) return a.hub_bits + (int64_t)p * a.Wpad;
    reads++;
    const int hs = a.hub_slot[p];
    return hs >= 0 ? a.hub_bits + (int64_t)hs * a.Wpad : nullptr;
}

__device__ __forceinline__ bool bit_of(const uint32_t *m, int Wpad, int row, int col) {
    return (m[(int64_t)row * Wpad + (col >> 5)] >> (col & 31)) & 1u;
}

// Is q an alive neighbour of p?  One bit of p's alive-adjacency set when p has one, else a
// binary search in p's sorted row and the alive mark.  `reads` counts the 4-byte words
// touched (algorithmic bytes = 4 x reads).
__device__ __forceinline__ bool alive_adjacent_set(const LossArgs &a, const uint32_t *pset, int p,
                                                   int q, unsigned &reads) {
    if (pset) {
        reads++;
        return (pset[q >> 5] >> (q & 31)) & 1u;
    }
    int lo = a.row_ptr[p], hi = a.row_ptr[p + 1] - 1;
    reads += 2;
    while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        const int v = __ldg(a.col + mid);
        reads++;
        if (v == q) {
            reads++;
            return a.col_live[mid] >= 0;
        }
        if (v < q) lo = mid + 1;
        else hi = mid - 1;
    }
    return false;
}

// Short rows are scanned by one lane; pairs whose shorter row is longer go to the warp.
constexpr int kInlineScan = 8;

enum PairState { kKept = 0, kLost = 1, kHard = 2 };

// Test of the non-adjacent pair {p,q} (h = 2) in the alive graph by one lane: p's row
// [rb, re) is the shorter one; a common alive neighbour is looked for when it is at most
// kInlineScan long, longer rows are left to the warp (kHard).
template <bool kTwin>
__device__ __forceinline__ int pair_quick(const LossArgs &a, int rb, int re, int q, unsigned &reads) {
    // with q's set every scanned neighbour costs one read; without it, a binary search
    if (re - rb > kInlineScan) return kHard;
    const uint32_t *qset = kTwin ? a.hub_bits + (int64_t)q * a.Wpad : hub_set(a, q, reads);
    // four slots at a time: their loads (and their set lookups) are independent
    for (int s0 = rb; s0 < re; s0 += 4) {
        int y[4];
#pragma unroll
        for (int j = 0; j < 4; j++) y[j] = (s0 + j < re) ? a.col_live[s0 + j] : -1;
        bool hit = false;
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (y[j] >= 0) {
                if (kTwin) hit |= (qset[y[j] >> 5] >> (y[j] & 31)) & 1u;
                else hit |= alive_adjacent_set(a, qset, q, y[j], reads);
            }
        reads += (unsigned)min(4, re - s0);
        if (hit) return kKept;
    }
    return kLost;
}

// Inclusive prefix sum over the warp.
template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Rows up to this long are walked by eight lanes, four rows side by side, longer ones by the
// whole warp.
constexpr int kShortRow = 64;

// Walks the rows [rb, re) of the warp's hard pairs (lanes with state == kHard; q the other
// endpoint): a pair is kept at its first alive neighbour y with test(q, y).  Short rows: four
// at a time, eight lanes each, 16 slots per row and step; long rows: one at a time, 128
// slots per step.  Laying the rows end to end, as warp_walk3 does, keeps more lanes busy but
// issues about 150 instructions per 128 slots against 25 per 64 here, and the walks of the
// h = 2 rounds are bound by what they issue (R-MAT 16, h = 2: 601 ms against 640 ms).  Whole
// warps call it.
template <typename Test>
__device__ __forceinline__ void warp_walk(const LossArgs &a, int &state, int rb, int re, int q, unsigned &reads,
                                          Test test) {
    __shared__ uint8_t s_lane[32][32];  // per warp: the lanes of its short rows
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const bool hard = state == kHard;
    unsigned kept = 0u;
    unsigned todo = __ballot_sync(full, hard && re - rb > kShortRow);
    while (todo) {
        const int l = __ffs(todo) - 1;
        todo &= todo - 1u;
        const int b = __shfl_sync(full, rb, l), e = __shfl_sync(full, re, l), ql = __shfl_sync(full, q, l);
        for (int s = b + lane; s - lane < e; s += 128) {
            int y[4];
            bool hit = false;
#pragma unroll
            for (int j = 0; j < 4; j++) y[j] = s + 32 * j < e ? a.col_live[s + 32 * j] : -1;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                if (y[j] >= 0) {
                    reads++;
                    hit |= test(ql, y[j]);
                }
            }
            if (__any_sync(full, hit)) {
                kept |= 1u << l;
                break;
            }
        }
    }
    const bool mine = hard && re - rb <= kShortRow;
    const unsigned shorts = __ballot_sync(full, mine);
    const int count = __popc(shorts);
    if (count) {
        if (mine) s_lane[wid][__popc(shorts & lanemask_lt())] = (uint8_t)lane;
        __syncwarp();
        for (int r0 = 0; r0 < count; r0 += 4) {
            const int r = r0 + (lane >> 3);
            const int src = r < count ? s_lane[wid][r] : 0;
            const int b = __shfl_sync(full, rb, src), e = __shfl_sync(full, re, src), ql = __shfl_sync(full, q, src);
            int s = b + (lane & 7);
            bool done = r >= count;
            while (__any_sync(full, !done && s - (lane & 7) < e)) {
                const int y0 = !done && s < e ? a.col_live[s] : -1;
                const int y1 = !done && s + 8 < e ? a.col_live[s + 8] : -1;
                bool hit = false;
                if (y0 >= 0) hit = test(ql, y0);
                if (y1 >= 0) hit |= test(ql, y1);
                reads += (y0 >= 0) + (y1 >= 0);
                const unsigned hits = __ballot_sync(full, hit);
                done = done || ((hits >> (lane & 24)) & 0xffu) != 0u;
                s += 16;
            }
            kept |= __reduce_or_sync(full, done && r < count ? 1u << src : 0u);
        }
        __syncwarp();
    }
    if (hard) state = ((kept >> lane) & 1u) ? kKept : kLost;
}

// Hard pairs at h = 2: a common alive neighbour ([rb, re): the endpoint with the shorter row).
template <bool kTwin>
__device__ __forceinline__ void warp_hard_pairs(const LossArgs &a, int &state, int rb, int re, int q,
                                                unsigned &reads) {
    warp_walk(a, state, rb, re, q, reads, [&](int qo, int y) -> bool {
        if (kTwin) return bit_of(a.hub_bits, a.Wpad, qo, y);
        return alive_adjacent_set(a, hub_set(a, qo, reads), qo, y, reads);
    });
}

// Is w in the stored ball of z (dense words, or sorted (word index, word) pairs)?
// `reads` counts 4-byte words: two of metadata plus the words probed.
__device__ __forceinline__ bool ball_contains_meta(const LossArgs &a, int2 meta, int w,
                                                   unsigned &reads) {
    const int nw = meta.y;
    const int64_t off = (int64_t)(unsigned)meta.x << 2;
    const uint32_t bit = 1u << (w & 31);
    const uint32_t wi = (uint32_t)(w >> 5);
    if (nw < 0) {
        reads++;
        return (a.pool[off + wi] & bit) != 0u;
    }
    const uint2 *p = reinterpret_cast<const uint2 *>(a.pool + off);
    int lo = 0, hi = nw - 1;
    while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        const uint2 v = p[mid];
        reads += 2;
        if (v.x == wi) return (v.y & bit) != 0u;
        if (v.x < wi) lo = mid + 1;
        else hi = mid - 1;
    }
    return false;
}

__device__ __forceinline__ bool ball_contains(const LossArgs &a, int z, int w, unsigned &reads) {
    if (a.dense_all) {
        reads++;
        return (a.pool[(int64_t)z * a.Wpad + (w >> 5)] >> (w & 31)) & 1u;
    }
    reads += 2;
    return ball_contains_meta(a, a.ball_meta[z], w, reads);
}

// The lost-pair records of a round: two lists take turns, since the cluster round kernel clears
// one round's from the balls while it records the next one's.
__device__ __forceinline__ int4 *lost_list(const LossArgs &a, int round) {
    return a.lost + (round & 1) * (int64_t)a.lost_max;
}
__device__ __forceinline__ int4 *lost2_list(const LossArgs &a, int round) {
    return a.lost2 + (round & 1) * (int64_t)a.lost2_max;
}

// Is the pair {p,q} in the table of the batch's lost pairs?  `probes` counts its slots read.
__device__ __forceinline__ bool in_pair_set(const unsigned long long *keys, unsigned mask, int p, int q,
                                            unsigned &probes) {
    const unsigned long long key = pair_key(p, q);
    unsigned slot = pair_slot(p, q, mask);
    for (unsigned probe = 0; probe <= mask; probe++) {
        const unsigned long long k = keys[slot];
        probes++;
        if (k == key) return true;
        if (k == kEmpty) return false;
        slot = (slot + 1) & mask;
    }
    return false;
}

// Records the lost pairs {x, z} of a warp (lanes with want == true; all lanes call it; the
// stored bit of each is set: a pair whose bit is clear was handled by an earlier batch of
// this round).  [rbx, rex) and [rbz, rez) are the endpoints' rows.  Each record and its
// update work (both rows are visited by the support updates) are reserved against the batch
// limits with one atomic per warp and counter; a pair that does not fit marks its edge side
// u as the point where the next slot of this round resumes.  New pairs go into the lost-pair
// set, and their update items (runs of 32 slots of each endpoint's row) are written: by
// their own lane when few, else by the warp.  Also counts, once per round and vertex, the
// alive edges whose support the round brings up to date (every alive edge at an endpoint of
// a lost pair).
// r2: radius-2 losses of an h = 3 round (recorded only: they change no support).
// kTwin: the pair is new if its bit is still set in the twin matrix, which is cleared.
// counted: where the new pairs and the alive edges at them are added up (a phase launch keeps
// them per block: every warp's atomic to one global word was a quarter of its same-address ones).
template <bool r2, bool kTwin>
__device__ __forceinline__ void record_lost_warp(const LossArgs &a, RoundCtr *ctr, int round, bool want,
                                                 int x, int z, int rbx, int rex, int rbz, int rez, int u,
                                                 unsigned long long *counted) {
    constexpr int kOwnItems = 8;
    const int lane = threadIdx.x & 31;
    const long long work = (want && !r2) ? (long long)(rex - rbx) + (rez - rbz) : 0ll;
    const unsigned wantb = __ballot_sync(0xffffffffu, want);
    if (wantb == 0u) return;
    const long long wincl = warp_incl_scan(work);
    const int rank = __popc(wantb & lanemask_lt());
    const long long wtot = __shfl_sync(0xffffffffu, wincl, 31);
    long long wbase = 0;
    unsigned ibase = 0u;
    if (lane == 0) {
        if (!r2)
            wbase = (long long)atomicAdd((unsigned long long *)&ctr->upd_work, (unsigned long long)wtot);
        ibase = atomicAdd(r2 ? &ctr->nlost2 : &ctr->nlost, (unsigned)__popc(wantb));
    }
    wbase = __shfl_sync(0xffffffffu, wbase, 0);
    ibase = __shfl_sync(0xffffffffu, ibase, 0);
    int4 *const lostv = r2 ? lost2_list(a, round) : lost_list(a, round);
    unsigned long long *const keys = r2 ? a.keys2 : a.keys;
    const unsigned cmask = r2 ? a.cap2_mask : a.cap_mask;
    const unsigned lmax = (unsigned)(r2 ? a.lost2_max : a.lost_max);
    int rec_idx = -1;
    if (want) {
        const unsigned idx = ibase + (unsigned)rank;
        if (idx >= lmax || (!r2 && wbase + wincl > a.upd_budget)) {
            overflow_at(a, ctr, u);
            if (idx < lmax) lostv[idx] = make_int4(-1, -1, -1, 0);
        } else {
            int4 rec = make_int4(-1, -1, -1, 0);  // null record: the pair is already held
            if (kTwin) {
                uint32_t *const twin = r2 ? a.pool2_new : a.pool_new;
                // another warp may be recording the pair from its other end: the bit in the
                // smaller id's row decides
                const int lo = min(x, z), hi = max(x, z);
                const uint32_t bit = 1u << (hi & 31);
                if (atomicAnd(twin + (int64_t)lo * a.Wpad + (hi >> 5), ~bit) & bit) {
                    atomicAnd(twin + (int64_t)hi * a.Wpad + (lo >> 5), ~(1u << (lo & 31)));
                    rec = make_int4(lo, hi, 0, 0);
                }
            } else {
                const unsigned long long key = pair_key(x, z);
                unsigned slot = pair_slot(x, z, cmask);
                for (unsigned probe = 0; probe <= cmask; probe++) {
                    const unsigned long long prev = atomicCAS(keys + slot, kEmpty, key);
                    if (prev == kEmpty) {
                        rec = make_int4(min(x, z), max(x, z), (int)slot, 0);
                        break;
                    }
                    if (prev == key) break;
                    slot = (slot + 1) & cmask;
                }
            }
            lostv[idx] = rec;
            if (rec.x >= 0) rec_idx = (int)idx;
            if (r2 && !kTwin) {
                // B2_new(v) differs from the stored B2(v) only at vertices marked here
                a.touch2[x] = round;
                a.touch2[z] = round;
            }
        }
    }
    if (r2) return;  // radius-2 losses change no support directly
    // update items: direction 0 = v0 = min loses v1, direction 1 = v1 loses v0
    int v0 = 0, v1 = 0, rb0 = 0, re0 = 0, rb1 = 0, re1 = 0, n0 = 0, n1 = 0;
    unsigned touched = 0u;
    if (rec_idx >= 0) {
        const unsigned dx = (unsigned)a.deg_alive[x], dz = (unsigned)a.deg_alive[z];
        if (atomicExch(a.vtouch + x, round) != round) touched += dx;
        if (atomicExch(a.vtouch + z, round) != round) touched += dz;
        const bool xf = x < z;
        v0 = xf ? x : z;
        v1 = xf ? z : x;
        rb0 = xf ? rbx : rbz;
        re0 = xf ? rex : rez;
        rb1 = xf ? rbz : rbx;
        re1 = xf ? rez : rex;
        n0 = (re0 - rb0 + 31) >> 5;
        n1 = (re1 - rb1 + 31) >> 5;
    }
    const int nincl = warp_incl_scan(n0 + n1);
    int nbase = 0;
    if (lane == 31 && nincl) nbase = atomicAdd(&ctr->nuitems, nincl);
    nbase = __shfl_sync(0xffffffffu, nbase, 31);
    const int base = nbase + nincl - (n0 + n1);
    if (rec_idx >= 0 && n0 + n1 <= kOwnItems) {
        for (int c = 0; c < n0 + n1 && base + c < a.uitems_cap; c++)
            a.uitems[base + c] = (c < n0) ? make_int4(rb0 + 32 * c, v0, v1, re0)
                                          : make_int4(rb1 + 32 * (c - n0), v1, v0, re1);
    }
    unsigned big = __ballot_sync(0xffffffffu, rec_idx >= 0 && n0 + n1 > kOwnItems);
    while (big) {
        const int l = __ffs(big) - 1;
        big &= big - 1;
        const int b = __shfl_sync(0xffffffffu, base, l);
        const int c0 = __shfl_sync(0xffffffffu, n0, l), c1 = __shfl_sync(0xffffffffu, n1, l);
        const int w0 = __shfl_sync(0xffffffffu, v0, l), w1 = __shfl_sync(0xffffffffu, v1, l);
        const int b0 = __shfl_sync(0xffffffffu, rb0, l), e0 = __shfl_sync(0xffffffffu, re0, l);
        const int b1 = __shfl_sync(0xffffffffu, rb1, l), e1 = __shfl_sync(0xffffffffu, re1, l);
        for (int c = lane; c < c0 + c1 && b + c < a.uitems_cap; c += 32)
            a.uitems[b + c] = (c < c0) ? make_int4(b0 + 32 * c, w0, w1, e0)
                                       : make_int4(b1 + 32 * (c - c0), w1, w0, e1);
    }
    touched = __reduce_add_sync(0xffffffffu, touched);
    const unsigned long long recorded = __popc(__ballot_sync(0xffffffffu, rec_idx >= 0));
    if (lane == 0 && recorded) atomicAdd(counted, recorded << kLostShift | touched);
}

// Pair enumeration of edge side u = (edge F[u/2], side u%2): side 0 of (a,b) pairs a with
// {b} and with N_old(b) \ {a} (slots start-1 .. re-1 of b's row, start-1 standing for b);
// side 1 pairs b with N_old(a) \ {b}.  For h = 1 only {a,b}.
struct UnitInfo {
    int x, y, start, stop;
    int4 rows;  // (row x, end, row y, end)
};

__device__ __forceinline__ UnitInfo unit_info(const LossArgs &a, int u) {
    UnitInfo r;
    const int e = a.frontier[u >> 1];
    const int side = u & 1;
    const int4 ends = a.erec[2 * (int64_t)e], rows = a.erec[2 * (int64_t)e + 1];
    r.x = side ? ends.y : ends.x;
    r.y = side ? ends.x : ends.y;
    r.rows = side ? make_int4(rows.z, rows.w, rows.x, rows.y) : rows;
    r.start = (side == 0) ? r.rows.z - 1 : r.rows.z;
    r.stop = (a.h < 2) ? r.rows.z : r.rows.w;
    return r;
}

// Detection item i: <= 32 pairs of edge side u from slot `first` on (u < 0: empty).
__device__ __forceinline__ void write_pitem(const LossArgs &a, int i, int u, int first, int x, int y, int4 rows) {
    a.pitems[2 * (int64_t)i] = make_int4(u, first, x, y);
    a.pitems[2 * (int64_t)i + 1] = rows;
}

// Place of the first of a warp's `tot` detection items (the value of lane 31 counts; all lanes call it).
__device__ __forceinline__ long long reserve_pitems(RoundCtr *ctr, int tot) {
    long long base = 0;
    if ((threadIdx.x & 31) == 31 && tot)
        base = (long long)atomicAdd((unsigned long long *)&ctr->npitems, (unsigned long long)tot);
    return __shfl_sync(0xffffffffu, base, 31);
}

// Items of the frontier's remaining edge sides, of at most 32 pairs (one warp each), so a hub
// row is spread over many warps.  Sides beyond unit_span, or that do not fit the item list, are
// left to the next slot of the round (resume point).  (Dense graphs: without the span the sides
// that fitted were spread over all of them, the resume point moved by a few sides a slot or not
// at all, and a round could take every slot a peel is given.)
__device__ void ph_pair_items(const LossArgs &a) {
    DevStatus *st = a.st;
    const int all = 2 * vload(st->nF), u0 = vload(st->unit_begin);
    const int units = (int)min((int64_t)all, (int64_t)u0 + vload(st->unit_span));
    const int lane = threadIdx.x & 31;
    if (units < all && blockIdx.x == 0 && threadIdx.x == 0) overflow_at(a, st, units);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t b = u0 + blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); b < units; b += stride) {
        const int u = (int)min(b + lane, (int64_t)units);
        int nch = 0, start = 0, x = 0, y = 0;
        int4 rows = make_int4(0, 0, 0, 0);
        if (u < units) {
            const UnitInfo r = unit_info(a, u);
            start = r.start;
            x = r.x;
            y = r.y;
            rows = r.rows;
            nch = (r.stop - r.start + 31) >> 5;
        }
        int incl = nch;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const int tot = __shfl_sync(0xffffffffu, incl, 31);
        const long long at = reserve_pitems(st, tot) + incl - nch;
        const int first = (int)min(at, (long long)a.pitems_cap);
        const bool fits = at + nch <= a.pitems_cap;
        if (!fits && nch) overflow_at(a, st, u);
        // a lane writes its one item, the whole warp the others (a hub row has hundreds)
        if (nch == 1 && first < a.pitems_cap) write_pitem(a, first, fits ? u : -1, start, x, y, rows);
        unsigned todo = __ballot_sync(0xffffffffu, nch > 1);
        while (todo) {
            const int l = __ffs(todo) - 1;
            todo &= todo - 1;
            const int f = __shfl_sync(0xffffffffu, first, l), c_n = __shfl_sync(0xffffffffu, nch, l);
            const int ul = __shfl_sync(0xffffffffu, u, l), sl = __shfl_sync(0xffffffffu, start, l);
            const int xl = __shfl_sync(0xffffffffu, x, l), yl = __shfl_sync(0xffffffffu, y, l);
            const int4 rl = make_int4(__shfl_sync(0xffffffffu, rows.x, l), __shfl_sync(0xffffffffu, rows.y, l),
                                      __shfl_sync(0xffffffffu, rows.z, l), __shfl_sync(0xffffffffu, rows.w, l));
            const bool fl = __shfl_sync(0xffffffffu, fits, l);
            for (int c = lane; c < c_n && f + c < a.pitems_cap; c += 32)
                write_pitem(a, f + c, fl ? ul : -1, sl + 32 * c, xl, yl, rl);
        }
    }
}

// Warps that share one detection item: with few items, 2^split_log2 warps take the same
// item and every 2^split_log2-th of its pairs, so that the walks of its hard pairs run side
// by side instead of one after the other in one warp (the median round of R-MAT 16 at h = 2
// has 79 items for 6,000 resident warps).
// Where the counters a warp's records reserve from are in global memory, more than 2^2 warps
// per item cost more in same-address atomics than their walks save.
__device__ __forceinline__ int split_log2(int nitems, int nwarps, int most) {
    int lg = 0;
    while (lg < most && nitems <= (nwarps >> (lg + 1))) lg++;
    return lg;
}

// Loss detection at h = 1: an item is one removed edge, whose endpoints are no longer adjacent.
// 2^lg items per warp, one per lane: as few as keep every warp busy, as many as there are
// for the atomics that reserve records, one set per warp (ER n = 400,000, 1.6 M edges in one
// round: 9.6 ms with one item per warp).
template <bool kTwin>
__device__ __forceinline__ void detect_edges(const LossArgs &a, RoundCtr *ctr, int gw, int nwarps, int nitems,
                                             int round, unsigned &pairs, unsigned &reads,
                                             unsigned long long *counted) {
    const int lane = threadIdx.x & 31;
    int lg = 0;
    while (lg < 5 && (nitems >> lg) > nwarps) lg++;
    for (int w = gw; w << lg < nitems; w += nwarps) {
        const int i = (w << lg) + lane;
        int4 item = make_int4(-1, 0, 0, 0), rows = make_int4(0, 0, 0, 0);
        if (lane < 1 << lg && i < nitems) {
            item = a.pitems[2 * (int64_t)i];
            rows = a.pitems[2 * (int64_t)i + 1];
        }
        // edges past an overflow are redone by the next slot of the round
        bool lost = item.x >= 0 && item.x <= vload(ctr->overflow_unit);
        if (lost) {
            pairs++;
            // an earlier batch may have recorded the pair
            if (kTwin) lost = bit_of(a.pool_new, a.Wpad, item.z, item.w);
            else lost = ball_contains(a, item.z, item.w, reads);
            reads += kTwin;
        }
        record_lost_warp<false, kTwin>(a, ctr, round, lost, item.z, item.w, rows.x, rows.y, rows.z, rows.w, item.x,
                                       counted);
    }
}

// Loss detection, one warp per item: lane i tests the pair of slot item.y + i.  A pair is
// kept if its endpoints are adjacent or (h = 2) share an alive neighbour; the pairs whose
// test needs a longer row scan are walked by the whole warp together.
template <bool r2, bool kTwin>
__device__ __forceinline__ void detect_items(const LossArgs &a, RoundCtr *ctr, int gw, int nwarps,
                                             int nitems, int max_split, int round, unsigned &pairs,
                                             unsigned &reads, unsigned long long *counted) {
    if (!r2 && a.h < 2) {
        detect_edges<kTwin>(a, ctr, gw, nwarps, nitems, round, pairs, reads, counted);
        return;
    }
    const int lane = threadIdx.x & 31;
    const int lg = split_log2(nitems, nwarps, max_split), split = 1 << lg;
    for (int w = gw; w < nitems << lg; w += nwarps) {
        const int4 item = a.pitems[2 * (int64_t)(w >> lg)], rows = a.pitems[2 * (int64_t)(w >> lg) + 1];
        const int u = item.x, x = item.z;
        // sides past an overflow are redone by the next slot of the round: skip them now
        if (u < 0 || u > vload(ctr->overflow_unit)) continue;
        const int sl = item.y + lane;
        int z = -1, rbz = 0, rez = 0;
        if (sl < rows.w && (lane & (split - 1)) == (w & (split - 1))) {
            if (sl < rows.z) {
                z = item.w;
                rbz = rows.z;
                rez = rows.w;
            } else {
                // an old neighbour: alive, or removed in this round
                const int4 s = a.srec[sl];
                const int cl = a.col_live[sl];
                reads += 5;
                if (s.x != x && (cl >= 0 || cl == -(round + 1))) {
                    z = s.x;
                    rbz = s.y;
                    rez = s.z;
                }
            }
        }
        // kept if adjacent, or if the stored bit is clear (an earlier batch, or in the twin
        // matrix another warp, recorded the pair): in the twin both words are in x's rows, so
        // their loads go out together; else only a pair about to be recorded looks it up
        int state = kKept, p = rows.x, pe = rows.y, q = z;
        if (z >= 0) {
            pairs++;
            const int64_t at = (int64_t)x * a.Wpad + (z >> 5);
            bool adjacent, held = true;
            if (kTwin) {
                const uint32_t stored = r2 ? a.pool2_new[at] : a.pool_new[at];
                adjacent = (a.hub_bits[at] >> (z & 31)) & 1u;
                held = (stored >> (z & 31)) & 1u;
                reads += 2;
            } else {
                const bool xs = rows.y - rows.x < rez - rbz;  // the longer row's set, if it has one
                adjacent = alive_adjacent_set(a, hub_set(a, xs ? z : x, reads), xs ? z : x, xs ? x : z, reads);
            }
            if (held && !adjacent) {
                if (rez - rbz < pe - p) {  // p: the shorter row
                    p = rbz;
                    pe = rez;
                    q = x;
                }
                state = pair_quick<kTwin>(a, p, pe, q, reads);
            }
        }
        if (__any_sync(0xffffffffu, state == kHard)) warp_hard_pairs<kTwin>(a, state, p, pe, q, reads);
        if (!kTwin && state == kLost && !(r2 ? bit_of(a.pool2, a.Wpad, x, z) : ball_contains(a, x, z, reads)))
            state = kKept;
        record_lost_warp<r2, kTwin>(a, ctr, round, state == kLost, x, z, rows.x, rows.y, rbz, rez, u, counted);
    }
}

template <bool r2, bool kTwin>
__device__ __forceinline__ void ph_detect(const LossArgs &a) {
    __shared__ unsigned long long s_pairs, s_reads, s_counted;
    DevStatus *st = a.st;
    if (threadIdx.x == 0) {
        s_pairs = 0ull;
        s_reads = 0ull;
        s_counted = 0ull;
    }
    __syncthreads();
    const int nitems = (int)min(vload(st->npitems), (long long)a.pitems_cap), round = vload(st->round);
    const int lane = threadIdx.x & 31;
    unsigned lane_pairs = 0u, lane_reads = 0u;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = gridDim.x * (blockDim.x >> 5);
    detect_items<r2, kTwin>(a, st, gw, nwarps, nitems, a.max_split, round, lane_pairs, lane_reads, &s_counted);
    unsigned long long pairs = lane_pairs, reads_total = lane_reads;
    for (int o = 16; o > 0; o >>= 1) {
        pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
        reads_total += __shfl_xor_sync(0xffffffffu, reads_total, o);
    }
    if (lane == 0 && pairs) {
        atomicAdd(&s_pairs, pairs);
        atomicAdd(&s_reads, reads_total);
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_pairs) {
        atomicAdd((unsigned long long *)&st->st_pairs, s_pairs);
        atomicAdd(&st->st_bytes_detect, 4ull * s_reads);
    }
    if (threadIdx.x == 0 && s_counted) atomicAdd((unsigned long long *)&st->touched, s_counted);
}

// Support updates, one warp per item (a directed loss v loses w, and <= 32 of v's slots),
// both orientations in one pass: an edge (v,z) with v < z loses w from B(v) ∩ B(z) iff w in
// B_old(z); with v > z iff w in B_new(z) = B_old(z) minus this batch's losses.  Distance is
// symmetric, so w in B(z) is tested as z in B(w) (all lanes read one ball, at increasing z).
// kWindow (the cluster round kernel): an edge whose support falls to win_hi joins the window,
// one whose support falls to thr the next frontier.
template <bool kWindow>
__device__ __forceinline__ void lower_support(const LossArgs &a, WindowCtr *wctr, int eid, int win_hi, int thr) {
    if (!kWindow) {
        atomicSub(a.sup + eid, 1);
        return;
    }
    // supports fall by one at a time: exactly one update takes the edge across
    const int old = atomicSub(a.sup + eid, 1);
    if (old == win_hi + 1) {
        const int i = atomicAdd(&wctr->nwin, 1);
        if (i < a.win_cap) a.win[i] = eid;
    }
    if (old == thr + 1) {
        const int i = atomicAdd(&wctr->nnext, 1);
        if (i < a.win_cap) a.next[i] = eid;
    }
}

// What a lane counts over its update items: the updates are bound by the instructions they
// issue, so bytes follow from the counts afterwards.
struct DeltaStats {
    unsigned tests = 0u, hits = 0u, probes = 0u, member_reads = 0u;
    __device__ unsigned bytes(bool twin) const {
        return 4u * (twin ? tests : member_reads) + 8u * hits + 8u * probes;
    }
};

// Algorithmic bytes of an update item beside its lanes': itself and 32 row slots.  (A batch may
// have 50 M items: their bytes pass 2^32.)
constexpr unsigned long long kItemBytes = 16ull + 4ull * 32ull;

// A directed loss (v loses w) tests z in B_old(w) or z in B_new(w), by the order of v and z: with
// the twin matrices that is one bit of either, else a bit and, for B_new, a probe of the lost-pair
// set.  In the cluster round kernel block `blk` of `nblks` takes a contiguous share of the items
// (an item and the next often test the same ball row), its warps every (blockDim / 32)-th of it,
// two at a time.  The phase launches, whose rounds are larger, deal runs of four to the warps of
// the whole grid: with the shares above, two at a time, R-MAT 18 with 16 M edges at h = 1 took
// 182 us a round for them instead of 141, R-MAT 16 at h = 2 11.2 instead of 10.2.
template <bool kWindow, bool kTwin>
__device__ __forceinline__ void delta_items_in(const LossArgs &a, WindowCtr *wctr, int blk, int nblks, int nitems,
                                               int win_hi, int thr, DeltaStats &ds) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    // items in flight per warp: their loads are interleaved
    constexpr int U = kWindow ? 2 : 4;
    const int share = (nitems + nblks - 1) / nblks;
    const int first = kWindow ? min(nitems, blk * share) + wid : U * (blk * wpb + wid);
    const int last = kWindow ? min(nitems, blk * share + share) : nitems;
    const int step = kWindow ? U * wpb : U * wpb * nblks, next = kWindow ? wpb : 1;
    for (int it0 = first; it0 < last; it0 += step) {
        int4 item[U];  // (first slot, v, w, end of v's row)
#pragma unroll
        for (int j = 0; j < U; j++) {
            const int it = it0 + j * next;
            item[j] = (it < last) ? a.uitems[it] : make_int4(0, 0, 0, 0);
        }
        int z[U], eid[U];
        bool drop[U];
#pragma unroll
        for (int j = 0; j < U; j++) {
            const int sl = item[j].x + lane;
            const bool ok = sl < item[j].w;
            z[j] = ok ? a.col_live[sl] : -1;
            eid[j] = ok ? a.slot_eid[sl] : 0;
        }
#pragma unroll
        for (int j = 0; j < U; j++) {
            drop[j] = false;
            if (z[j] >= 0) {
                ds.tests++;
                if (kTwin)
                    drop[j] = bit_of(item[j].y < z[j] ? a.pool : a.pool_new, a.Wpad, item[j].z, z[j]);
                else
                    drop[j] = ball_contains(a, item[j].z, z[j], ds.member_reads);
            }
        }
#pragma unroll
        for (int j = 0; j < U; j++) {
            if (!kTwin && drop[j] && item[j].y > z[j])
                drop[j] = !in_pair_set(a.keys, a.cap_mask, item[j].z, z[j], ds.probes);
            if (drop[j]) {
                lower_support<kWindow>(a, wctr, eid[j], win_hi, thr);
                ds.hits++;
            }
        }
    }
}

template <bool kWindow, bool kTwin>
__device__ __forceinline__ void delta_items(const LossArgs &a, WindowCtr *wctr, int blk, int nblks, int nitems,
                                            int win_hi, int thr, unsigned &tests, unsigned &bytes) {
    DeltaStats ds;
    delta_items_in<kWindow, kTwin>(a, wctr, blk, nblks, nitems, win_hi, thr, ds);
    tests = ds.tests;
    bytes = ds.bytes(kTwin);
}

template <bool kTwin>
__device__ __forceinline__ void ph_delta(const LossArgs &a) {
    __shared__ unsigned long long s_tests, s_bytes;
    DevStatus *st = a.st;
    const int nitems = min(vload(st->nuitems), a.uitems_cap);
    if (threadIdx.x == 0) {
        s_tests = 0ull;
        s_bytes = blockIdx.x == 0 ? kItemBytes * nitems : 0ull;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    unsigned lane_tests = 0u, lane_bytes = 0u;
    delta_items<false, kTwin>(a, nullptr, blockIdx.x, gridDim.x, nitems, 0, 0, lane_tests, lane_bytes);
    unsigned long long tests = lane_tests, bytes_total = lane_bytes;
    for (int o = 16; o > 0; o >>= 1) {
        tests += __shfl_xor_sync(0xffffffffu, tests, o);
        bytes_total += __shfl_xor_sync(0xffffffffu, bytes_total, o);
    }
    if (lane == 0 && (tests || bytes_total)) {
        atomicAdd(&s_tests, tests);
        atomicAdd(&s_bytes, bytes_total);
    }
    __syncthreads();
    if (threadIdx.x == 0 && (s_tests || s_bytes)) {
        atomicAdd((unsigned long long *)&st->st_tests, s_tests);
        atomicAdd(&st->st_bytes_update, s_bytes);
    }
}

// Clears every lost member from the stored balls (each record's bits are set) and empties
// the hash slots.
// Thread t of nt.
__device__ __forceinline__ void apply_lost(const LossArgs &a, int t, int nt, int nlost, int round) {
    const int4 *const lost = lost_list(a, round);
    for (int d = t; d < 2 * nlost; d += nt) {
        const int4 L = lost[d >> 1];
        if (L.x < 0) continue;
        const int v = (d & 1) ? L.y : L.x;
        const int w = (d & 1) ? L.x : L.y;
        const uint32_t bit = 1u << (w & 31);
        const uint32_t wi = (uint32_t)(w >> 5);
        uint32_t *word = nullptr;
        if (a.dense_all) {
            word = a.pool + (int64_t)v * a.Wpad + wi;
        } else {
            const int2 meta = a.ball_meta[v];
            const int nw = meta.y;
            const int64_t off = (int64_t)(unsigned)meta.x << 2;
            if (nw < 0) {
                word = a.pool + off + wi;
            } else {
                const uint2 *p = reinterpret_cast<const uint2 *>(a.pool + off);
                int lo = 0, hi = nw - 1;
                while (lo <= hi) {
                    const int mid = (lo + hi) >> 1;
                    const uint32_t idx = p[mid].x;
                    if (idx == wi) {
                        word = a.pool + off + 2 * (int64_t)mid + 1;
                        break;
                    }
                    if (idx < wi) lo = mid + 1;
                    else hi = mid - 1;
                }
            }
        }
        if (word) {
            atomicAnd(word, ~bit);
            atomicSub(a.ball_size + v, 1);
        }
        if ((d & 1) == 0 && !a.pool_new) a.keys[L.z] = kEmpty;
    }
}

__device__ void ph_apply(const LossArgs &a) {
    apply_lost(a, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, (int)min(vload(a.st->nlost), (unsigned)a.lost_max),
               vload(a.st->round));
}

// ---- h = 3 -------------------------------------------------------------------------------
//
// At h = 3 the supports are taken on radius-3 balls B3 while radius-2 balls B2 are kept
// beside them.  Removing F can only separate pairs that had a path of at most 3 edges
// through a removed edge (a,b), i.e. pairs {p,q} with p in B(a,i), q in B(b,2-i) before the
// removal, i = 0, 1, 2:  {a} x B2_old(b),  N_old(a) x N_old(b),  B2_old(a) x {b}.  A
// candidate still in B3_old(p) stays within distance 3 iff q is in B2_new(z) for z = p or
// for some alive neighbour z of p (or, symmetrically, of q).  B2_new is the stored B2 minus
// this round's radius-2 losses, which the radius-2 detection (the h = 2 rule, recorded in
// their own pair set) has listed first.  Radius-3 losses then take the support deltas of
// the h = 2 rounds unchanged, on B3.

// q in B2_new(z): a bit of the twin matrix, or the stored radius-2 bit unless this round lost
// the pair (the pair set is probed only for vertices that lost a radius-2 member this round).
template <bool kTwin>
__device__ __forceinline__ bool in_b2_new(const LossArgs &a, int z, int q, int round, unsigned &reads) {
    reads++;
    if (kTwin) return bit_of(a.pool2_new, a.Wpad, z, q);
    if (!bit_of(a.pool2, a.Wpad, z, q)) return false;
    if (z == q) return true;
    reads++;
    if (a.touch2[z] != round) return true;
    unsigned probes = 0u;
    const bool lost = in_pair_set(a.keys2, a.cap2_mask, z, q, probes);
    reads += 2 * probes;
    return !lost;
}

// Position of the k-th (0-based) set bit of v (k < popc(v)).
__device__ __forceinline__ int nth_set_bit(uint32_t v, int k) {
    for (; k > 0; k--) v &= v - 1u;
    return __ffs(v) - 1;
}

// Words of a B2 row one radius-3 candidate item scans: at most 128 candidates, so that one
// item never holds up its launch (one GB300, DC-SBM n = 200,000 at h = 3: 3.7 s per
// decomposition with 4 words, 4.2 s with 16, 5.1 s with 32; 2 words made more rounds
// overflow the item list).
constexpr int kC3Words = 4;
// Range items one warp tests per step (kC3Words lanes each).
constexpr int kC3Groups = 32 / kC3Words;
static_assert(32 % kC3Words == 0, "range items must tile a warp");

// Radius-3 candidate items of the round's frontier.  For each frontier edge F[f] = (a,b):
//   (a, row b, word range) and (b, row a, word range): {a} x B2_old(b) and {b} x B2_old(a),
//     2 * nch items per edge, not stored: item index i < 2 * nch * |F| is frontier edge
//     i / (2 nch), side (i % (2 nch)) / nch, word chunk i % nch (c3_range_item);
//   (p, row b, 32 slots) for every old neighbour p != b of a: N_old(a) x N_old(b), written
//     by one warp per frontier edge into the item list.
// Item layout: (x, y, first word | first slot, -1 - end word | end slot).  A round whose
// items (both kinds) exceed the list's capacity halts.
__device__ __forceinline__ int c3_chunks(const LossArgs &a) { return (a.Wpad + kC3Words - 1) / kC3Words; }

__device__ __forceinline__ int4 c3_range_item(const LossArgs &a, int i, int nch) {
    const int f = i / (2 * nch), r = i - f * 2 * nch;
    const int side = r >= nch, ch = side ? r - nch : r;
    const int e = a.frontier[f];
    const int ea = a.eu[e], eb = a.ev[e];
    const int w0 = ch * kC3Words, w1 = min(a.Wpad, w0 + kC3Words);
    return side ? make_int4(eb, ea, w0, -1 - w1) : make_int4(ea, eb, w0, -1 - w1);
}

__device__ __forceinline__ void c3_items(const LossArgs &a, RoundCtr *ctr, int gw, int nwarps, int nF,
                                         int round) {
    const int lane = threadIdx.x & 31;
    const long long nA = 2ll * c3_chunks(a) * nF;
    if (nA > a.c3items_cap) {
        if (gw == 0 && lane == 0) atomicOr(&ctr->halt, 1);
        return;
    }
    for (int i = gw; i < nF; i += nwarps) {
        const int e = a.frontier[i];
        const int ea = a.eu[e], eb = a.ev[e];
        const int rba = a.row_ptr[ea], rea = a.row_ptr[ea + 1];
        const int rbb = a.row_ptr[eb], reb = a.row_ptr[eb + 1];
        const int nb = (reb - rbb + 31) >> 5;
        for (int s0 = rba; s0 < rea; s0 += 32) {
            const int sl = s0 + lane;
            int p = -1;
            if (sl < rea) {
                const int c = a.col[sl], cl = a.col_live[sl];
                if (c != eb && (cl >= 0 || cl == -(round + 1))) p = c;
            }
            const int cnt = p >= 0 ? nb : 0;
            const int incl = warp_incl_scan(cnt);
            const int tot = __shfl_sync(0xffffffffu, incl, 31);
            long long b2 = 0;
            if (lane == 31 && tot)
                b2 = (long long)atomicAdd((unsigned long long *)&ctr->nc3items, (unsigned long long)tot);
            b2 = __shfl_sync(0xffffffffu, b2, 31);
            if (nA + b2 + tot > a.c3items_cap) {
                if (lane == 0 && tot) atomicOr(&ctr->halt, 1);
                continue;
            }
            const int first = (int)b2 + incl - cnt;
            for (int c = 0; c < cnt; c++)
                a.c3items[first + c] = make_int4(p, eb, rbb + 32 * c, min(reb, rbb + 32 * (c + 1)));
        }
    }
}

// Common walk of the warp's hard radius-3 pairs (lanes with state == kHard): [rb, re) is the
// row of one endpoint, t the other one; the pair is kept at the first alive neighbour y in
// the row with t in B2_new(y).  The rows are laid end to end and walked 128 slots per step,
// each lane finding the pair its slot belongs to by a binary search over the lanes' running
// row lengths; the walk skips kept pairs.  (Eight lanes per row, as in warp_walk, makes the
// many long rows wait for one another: R-MAT 4096 at h = 3 23 ms against 16 ms.)  Called by
// whole warps.
template <bool kTwin>
__device__ __forceinline__ void warp_walk3(const LossArgs &a, int &state, int rb, int re, int t, int round,
                                           unsigned &reads) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool hard = state == kHard;
    const int len = hard ? re - rb : 0;
    const int incl = warp_incl_scan(len);
    const int excl = incl - len;
    const int total = __shfl_sync(full, incl, 31);
    unsigned pending = __ballot_sync(full, hard);
    unsigned kept = 0u;
    for (int base = 0; base < total && pending; base += 128) {
        int y[4], own[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int idx = base + 32 * j + lane;
            int o = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(full, incl, o + step - 1) <= idx) o += step;
            o = min(o, 31);
            const int ex = __shfl_sync(full, excl, o), rbo = __shfl_sync(full, rb, o);
            own[j] = o;
            y[j] = (idx < total && ((pending >> o) & 1u)) ? a.col_live[rbo + idx - ex] : -1;
        }
        unsigned hits = 0u;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int to = __shfl_sync(full, t, own[j]);
            if (y[j] >= 0) {
                reads++;
                if (in_b2_new<kTwin>(a, y[j], to, round, reads)) hits |= 1u << own[j];
            }
        }
        hits = __reduce_or_sync(full, hits);
        kept |= hits;
        pending &= ~hits;
    }
    if (hard) state = ((kept >> lane) & 1u) ? kKept : kLost;
}

// Decides the lanes' radius-3 candidate pairs {p,q} (q < 0: none; q is in B3_old(p) and not in
// B2_new(p)) in the new graph and records the lost ones with their support-update items.
// Whole warps.
template <bool kTwin>
__device__ __forceinline__ void decide_pairs3(const LossArgs &a, RoundCtr *ctr, int p, int q, int round,
                                              unsigned &reads, unsigned long long *counted) {
    int state = kKept, rb = 0, re = 0, t = q, rbp = 0, rep = 0, rbq = 0, req = 0;
    if (q >= 0) {
        state = kHard;
        rbp = a.row_ptr[p];
        rep = a.row_ptr[p + 1];
        rbq = a.row_ptr[q];
        req = a.row_ptr[q + 1];
        reads += 6;
        const bool walk_q = a.deg_alive[q] < a.deg_alive[p];  // the shorter alive row
        rb = walk_q ? rbq : rbp;
        re = walk_q ? req : rep;
        t = walk_q ? p : q;
    }
    if (!__any_sync(0xffffffffu, q >= 0)) return;
    warp_walk3<kTwin>(a, state, rb, re, t, round, reads);
    record_lost_warp<false, kTwin>(a, ctr, round, state == kLost, p, q, rbp, rep, rbq, req, 0, counted);
}

// Radius-3 loss tests, one warp per candidate item: nA range items, then the stored ones.
template <bool kTwin>
__device__ __forceinline__ void test3_items(const LossArgs &a, RoundCtr *ctr, int gw, int nwarps, int nA,
                                            int nitems, int round, unsigned &pairs, unsigned &reads,
                                            unsigned long long *counted) {
    const int lane = threadIdx.x & 31;
    const int nch = c3_chunks(a);
    // pairs another warp has recorded already are not candidates
    const uint32_t *const b3 = kTwin ? a.pool_new : a.pool;
    // {x} x B2_old(y) restricted to B3_old(x), kC3Groups range items per warp and step: the
    // lanes of group g hold the words of item (step * kC3Groups + g) * nwarps + warp (items
    // of one warp step lie far apart, so their candidate counts average out), and the
    // step's candidates are dealt out 32 at a time by a warp prefix sum
    for (int s0 = 0; s0 * kC3Groups * nwarps < nA; s0++) {
        const int it = (s0 * kC3Groups + lane / kC3Words) * nwarps + gw;
        int x = -1, wi = 0;
        uint32_t bits = 0u;
        if (it < nA) {
            const int4 item = c3_range_item(a, it, nch);
            x = item.x;
            wi = item.z + lane % kC3Words;
            if (wi < -1 - item.w) {
                const int64_t ax = (int64_t)x * a.Wpad + wi;
                bits = a.pool2[(int64_t)item.y * a.Wpad + wi] & b3[ax];
                reads += 2;
                if (wi == (x >> 5)) bits &= ~(1u << (x & 31));
                pairs += __popc(bits);
                // pairs within distance 2 still are kept: one word decides 32 of them
                if (kTwin) bits &= ~a.pool2_new[ax];
            }
        }
        const int cnt = __popc(bits);
        const int incl = warp_incl_scan(cnt);
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int idx = t0 + lane;
            // owner lane: the number of lanes whose candidates end at or before idx
            int o = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(0xffffffffu, incl, o + step - 1) <= idx) o += step;
            o = min(o, 31);
            const uint32_t ob = __shfl_sync(0xffffffffu, bits, o);
            const int ex = __shfl_sync(0xffffffffu, incl - cnt, o);
            const int ow = __shfl_sync(0xffffffffu, wi, o), ox = __shfl_sync(0xffffffffu, x, o);
            int q = -1;
            if (idx < total) q = (ow << 5) + nth_set_bit(ob, idx - ex);
            if (!kTwin && q >= 0 && in_b2_new<kTwin>(a, ox, q, round, reads)) q = -1;
            decide_pairs3<kTwin>(a, ctr, ox, q, round, reads, counted);
        }
    }
    // {x} x N_old(y) for the 32 slots of a stored item, restricted to B3_old(x): one per warp
    for (int it = nA + gw; it < nitems; it += nwarps) {
        const int4 item = a.c3items[it - nA];
        const int x = item.x;
        const int sl = item.z + lane;
        int q = -1;
        if (sl < item.w) {
            const int c = a.col[sl], cl = a.col_live[sl];
            reads += 2;
            if (c != x && (cl >= 0 || cl == -(round + 1))) {
                reads++;
                const bool in3 = bit_of(b3, a.Wpad, x, c), in2 = in_b2_new<kTwin>(a, x, c, round, reads);
                pairs += in3;
                if (in3 && !in2) q = c;
            }
        }
        decide_pairs3<kTwin>(a, ctr, x, q, round, reads, counted);
    }
}

template <bool kTwin>
__device__ __forceinline__ void ph_test3(const LossArgs &a) {
    __shared__ unsigned long long s_pairs, s_reads, s_counted;
    DevStatus *st = a.st;
    if (threadIdx.x == 0) {
        s_pairs = 0ull;
        s_reads = 0ull;
        s_counted = 0ull;
    }
    __syncthreads();
    // a round whose items passed the capacity has halted (this kernel is then idle), so
    // both counts fit the list here
    const long long nA64 = 2ll * c3_chunks(a) * vload(st->nF);
    if (nA64 > a.c3items_cap) return;
    const int nA = (int)nA64;
    const int nitems = nA + (int)min(vload(st->nc3items), (long long)a.c3items_cap - nA);
    const int lane = threadIdx.x & 31;
    unsigned lane_pairs = 0u, lane_reads = 0u;
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = gridDim.x * (blockDim.x >> 5);
    const int round = vload(st->round);
    test3_items<kTwin>(a, st, gw, nwarps, nA, nitems, round, lane_pairs, lane_reads, &s_counted);
    unsigned long long pairs = lane_pairs, reads_total = lane_reads;
    for (int o = 16; o > 0; o >>= 1) {
        pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
        reads_total += __shfl_xor_sync(0xffffffffu, reads_total, o);
    }
    if (lane == 0 && pairs) {
        atomicAdd(&s_pairs, pairs);
        atomicAdd(&s_reads, reads_total);
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_pairs) {
        atomicAdd((unsigned long long *)&st->st_c3_pairs, s_pairs);
        atomicAdd(&st->st_bytes_detect, 4ull * s_reads);
    }
    if (threadIdx.x == 0 && s_counted) atomicAdd((unsigned long long *)&st->touched, s_counted);
}

// Clears the round's radius-2 losses from the stored B2 (and their pair-set slots).
__device__ __forceinline__ void apply_lost2(const LossArgs &a, int t, int nt, int nlost, int round,
                                            unsigned &real) {
    const int4 *const lost = lost2_list(a, round);
    for (int d = t; d < 2 * nlost; d += nt) {
        const int4 L = lost[d >> 1];
        if (L.x < 0) continue;
        const int v = (d & 1) ? L.y : L.x;
        const int w = (d & 1) ? L.x : L.y;
        const uint32_t bit = 1u << (w & 31);
        atomicAnd(a.pool2 + (int64_t)v * a.Wpad + (w >> 5), ~bit);
        atomicSub(a.ball_size2 + v, 1);
        if ((d & 1) == 0) {
            if (!a.pool_new) a.keys2[L.z] = kEmpty;
            real++;
        }
    }
}

__device__ void ph_apply2(const LossArgs &a) {
    DevStatus *st = a.st;
    unsigned lane_real = 0u;
    apply_lost2(a, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x,
                (int)min(vload(st->nlost2), (unsigned)a.lost2_max), vload(st->round), lane_real);
    unsigned long long real = lane_real;
    for (int o = 16; o > 0; o >>= 1) real += __shfl_xor_sync(0xffffffffu, real, o);
    if ((threadIdx.x & 31) == 0 && real) atomicAdd((unsigned long long *)&st->st_lost2, real);
}

// One candidate edge per lane (p: it joins the frontier): warp-aggregated frontier slot,
// removal (the removal step of Algorithm 1) and the detection items of its two edge sides.  Whole
// warps call it.
__device__ __forceinline__ void select_one(const LossArgs &a, RoundCtr *ctr, bool p, int e, int k,
                                           int round) {
    const int lane = threadIdx.x & 31;
    const unsigned bal = __ballot_sync(0xffffffffu, p);
    if (bal == 0u) return;
    int4 ends = make_int4(0, 0, 0, 0), rows = make_int4(0, 0, 0, 0);
    if (p) {
        ends = a.erec[2 * (int64_t)e];
        rows = a.erec[2 * (int64_t)e + 1];
    }
    int base = 0;
    if (lane == 0) base = atomicAdd(&ctr->nF, __popc(bal));
    base = __shfl_sync(0xffffffffu, base, 0);
    const int pos = base + __popc(bal & lanemask_lt());
    int n0 = 0, n1 = 0;
    if (p) {
        a.frontier_w[pos] = e;
        remove_edge(e, k, round, ends.x, ends.y, ends.z, ends.w, a.sup, a.truss, a.stamp_w, a.col_live_w,
                    a.deg_alive_w, a.hub_all, a.hub_slot, a.hub_bits_w, a.Wpad);
        // side 0: eu with {ev} and N_old(ev); side 1: ev with N_old(eu); h = 1: {eu,ev}
        n0 = (a.h < 2) ? 1 : (rows.w - rows.z + 1 + 31) >> 5;
        n1 = (a.h < 2) ? 0 : (rows.y - rows.x + 31) >> 5;
    }
    const int incl = warp_incl_scan(n0 + n1);
    const long long at = reserve_pitems(ctr, incl) + incl - (n0 + n1);
    const int first = (int)min(at, (long long)a.pitems_cap);
    const bool fits0 = at + n0 <= a.pitems_cap, fits1 = at + n0 + n1 <= a.pitems_cap;
    if (p && !fits0) overflow_at(a, ctr, 2 * pos);
    if (p && n1 && !fits1) overflow_at(a, ctr, 2 * pos + 1);
    // few items are written by their own lane, a hub row's by the whole warp
    constexpr int kOwnItems = 4;
    auto write = [&](int c, int n0w, int f, int posw, int4 ew, int4 rw, bool f0, bool f1) {
        if (c < n0w)
            write_pitem(a, f + c, f0 ? 2 * posw : -1, rw.z - 1 + 32 * c, ew.x, ew.y, rw);
        else
            write_pitem(a, f + c, f1 ? 2 * posw + 1 : -1, rw.x + 32 * (c - n0w), ew.y, ew.x,
                        make_int4(rw.z, rw.w, rw.x, rw.y));
    };
    if (p && n0 + n1 <= kOwnItems)
        for (int c = 0; c < n0 + n1 && first + c < a.pitems_cap; c++) write(c, n0, first, pos, ends, rows, fits0, fits1);
    unsigned todo = __ballot_sync(0xffffffffu, p && n0 + n1 > kOwnItems);
    while (todo) {
        const int l = __ffs(todo) - 1;
        todo &= todo - 1;
        const int f = __shfl_sync(0xffffffffu, first, l), pl = __shfl_sync(0xffffffffu, pos, l);
        const int c0 = __shfl_sync(0xffffffffu, n0, l), c1 = __shfl_sync(0xffffffffu, n1, l);
        const int4 el = make_int4(__shfl_sync(0xffffffffu, ends.x, l), __shfl_sync(0xffffffffu, ends.y, l), 0, 0);
        const int4 rl = make_int4(__shfl_sync(0xffffffffu, rows.x, l), __shfl_sync(0xffffffffu, rows.y, l),
                                  __shfl_sync(0xffffffffu, rows.z, l), __shfl_sync(0xffffffffu, rows.w, l));
        const bool l0 = __shfl_sync(0xffffffffu, fits0, l), l1 = __shfl_sync(0xffffffffu, fits1, l);
        for (int c = lane; c < c0 + c1 && f + c < a.pitems_cap; c += 32) write(c, c0, f, pl, el, rl, l0, l1);
    }
}

// Phase 1 of an incremental round: every alive edge with h-support <= k-2 joins F and is
// removed at once (the selection and removal steps of Algorithm 1), and the loss detection items of its two edge
// sides are written.  A continued round only writes the items of its remaining sides.
__device__ void ph_select_items(const LossArgs &a) {
    DevStatus *st = a.st;
    if (vload(st->cont)) {
        ph_pair_items(a);
        return;
    }
    const int k = vload(st->k), round = vload(st->round), thr = k - 2;
    const int lane = threadIdx.x & 31;
    const int64_t stride = 4 * (int64_t)gridDim.x * blockDim.x;
    // four coalesced loads per thread per step, issued before any of them is used
    for (int64_t e0 = 4 * (blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31)); e0 < a.m;
         e0 += stride) {
        int sv[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const int64_t e = e0 + 32 * j + lane;
            sv[j] = (e < a.m) ? a.sup[e] : INT_MAX;
        }
#pragma unroll
        for (int j = 0; j < 4; j++) select_one(a, st, sv[j] <= thr, (int)(e0 + 32 * j + lane), k, round);
    }
}

// Programmatic dependent launch: a phase kernel may be scheduled while the previous one
// still runs; it waits here until that grid has completed and its writes are visible, then
// lets the next phase be scheduled in turn.  (Without a programmatic launch the wait
// returns at once.)
__device__ __forceinline__ void phase_entry() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Phases of a round whose time the status block adds up (st_phase_ns).
enum TimedPhase { kTimeSelect = 0, kTimeDetect, kTimeTest3, kTimeDelta, kTimeReduce };

// With a.timer: a phase launch starts, which ends the time of phase `done` (-1: the slot
// begins).  One thread of the launch calls it; launches of a slot follow one another.
__device__ __forceinline__ void phase_clock(const LossArgs &a, int done) {
    if (!a.timer || blockIdx.x != 0 || threadIdx.x != 0) return;
    const unsigned long long t = global_ns();
    if (done >= 0) a.st->st_phase_ns[done] += t - a.st->st_phase_start;
    a.st->st_phase_start = t;
}

// Resident blocks per SM a phase kernel is compiled for: left to itself the compiler gives up
// loads in flight for more blocks, which the small rounds have no use for.
constexpr int kPhaseBlocks = 4;
// The two scans over all edges use fewer blocks: the reduction's per-block atomics all hit the
// same few counters.
constexpr int kScanBlocks = 2;

// One launch per phase (the rounds of a CUDA graph).
__global__ void __launch_bounds__(kBlock, kScanBlocks) k_inc_select(LossArgs a) {
    phase_entry();
    if (round_idle(a, kStageSelect)) return;
    phase_clock(a, -1);
    ph_select_items(a);
}
template <bool kTwin>
__global__ void __launch_bounds__(kBlock, kPhaseBlocks) k_loss_detect(LossArgs a) {
    phase_entry();
    if (round_idle(a, kStageDetect)) return;
    phase_clock(a, kTimeSelect);
    ph_detect<false, kTwin>(a);
}
// h = 3: the radius-2 detection and the round's radius-3 candidate items
template <bool kTwin>
__global__ void __launch_bounds__(kBlock, kPhaseBlocks) k_loss_detect3(LossArgs a) {
    phase_entry();
    if (round_idle(a, kStageDetect)) return;
    phase_clock(a, kTimeSelect);
    ph_detect<true, kTwin>(a);
    c3_items(a, a.st, (blockIdx.x * blockDim.x + threadIdx.x) >> 5, gridDim.x * (blockDim.x >> 5),
             vload(a.st->nF), vload(a.st->round));
}
template <bool kTwin>
__global__ void __launch_bounds__(kBlock, kPhaseBlocks) k_loss3_test(LossArgs a) {
    phase_entry();
    if (round_idle(a, kStageTest3)) return;
    phase_clock(a, kTimeDetect);
    ph_test3<kTwin>(a);
}
template <bool kTwin>
__global__ void __launch_bounds__(kBlock, kPhaseBlocks) k_loss_delta(LossArgs a) {
    phase_entry();
    if (round_idle(a, kStageDelta)) return;
    phase_clock(a, a.h3 ? kTimeTest3 : kTimeDetect);
    ph_delta<kTwin>(a);
}
// Bound by the loads of its scan.  Two blocks per SM, which is what the scans are launched with,
// leave registers for 16 of them a thread: 16 M supports 62 -> 29 us, 0.5 M 11.2 -> 9.9.
__global__ void __launch_bounds__(kBlock, kScanBlocks) k_loss_apply_reduce(LossArgs a) {
    phase_entry();
    if (round_idle(a, kStageDelta)) return;
    phase_clock(a, kTimeDelta);
    ph_apply(a);
    if (a.h3) ph_apply2(a);
    if (minreduce_body<kBlock / 32>(a.sup, a.m, a.st, 0) && a.timer)
        a.st->st_phase_ns[kTimeReduce] += global_ns() - a.st->st_phase_start;
}

constexpr int kPBlock = 512;  // threads per block of the persistent kernel

// Persistent round kernel (cooperative launch, every block resident): runs up to
// `max_slots` round slots, each the four phases of an incremental round separated by grid
// barriers, and stops early once no edge is alive or an error is flagged.  Block 0 adds
// the time of each phase to the status block.
__global__ void __launch_bounds__(kPBlock, 2) k_rounds_persistent(LossArgs a, int max_slots) {
    DevStatus *st = a.st;
    const bool timer = blockIdx.x == 0 && threadIdx.x == 0;
    unsigned long long t_prev = timer ? global_ns() : 0ull;
    auto phase_done = [&](int p) -> bool {
        if (!grid_barrier(st)) return false;
        if (timer) {
            const unsigned long long t = global_ns();
            st->st_phase_ns[p] += t - t_prev;
            t_prev = t;
        }
        return true;
    };
    for (int slot = 0; slot < max_slots; slot++) {
        if (vload(st->alive) == 0 || vload(st->err) != 0) break;
        ph_select_items(a);
        if (!phase_done(kTimeSelect)) return;
        if (a.pool_new) ph_detect<false, true>(a);
        else ph_detect<false, false>(a);
        if (!phase_done(kTimeDetect)) return;
        if (a.pool_new) ph_delta<true>(a);
        else ph_delta<false>(a);
        if (!phase_done(kTimeDelta)) return;
        // clearing the lost members touches balls and hash slots only; the reduction reads
        // supports only, and its last block closes the round after every block did both
        ph_apply(a);
        minreduce_body<kPBlock / 32>(a.sup, a.m, st, 0);
        if (!phase_done(kTimeReduce)) return;
    }
}

// ---- small rounds in one thread-block cluster --------------------------------------------
//
// Most rounds are small (R-MAT 16 at h = 2: 8 frontier edges and 12K update items in the
// median), and a round of separate launches then costs its launches, two scans of every
// support and a dozen dependent loads behind each launch.  This kernel runs such rounds in
// ONE cluster of up to 16 blocks: the phases are split by hardware cluster barriers, the
// round's counters sit in the shared memory of the cluster's first block, and the frontier
// comes from a window instead of a scan.  It needs the twin ball matrices.
// What bounds it: a round is a chain of about fifteen dependent L2 loads (290 cycles each) and
// five cluster barriers (600 cycles, more behind stores); the updates and the walks of the
// detection are bound by the instructions 16 SMs issue (IPC 1.2 of them, DRAM 12 GB/s).
// 1,024 threads a block, 16 blocks: with 512 threads the selection is faster (5.4 -> 4.0 us
// a round) and the updates slower (15.7 -> 22 us).
// One decomposition, one launch per phase -> this kernel: ER n = 2,000 at h = 2 4.3 -> 1.95 ms,
// R-MAT 16 at h = 2 920 -> 590 ms (a round 50 -> 31 us), DC-SBM 40k at h = 3 1,640 -> 1,070 ms.
//
// Frontier: the edges the last round's updates took to the level (exactly one update sees
// each crossing, since supports fall one at a time), else from the window.
// Window: the list of edges whose support was at most win_hi when the list was built from a
// full scan, plus every edge whose support has fallen to win_hi since.  While an alive edge is in it, the
// smallest alive support is its smallest; when none is left it is rebuilt.
//
// A phase with more work than one cluster does quickly is shared with helpers: further
// clusters of the same launch, which wait for jobs in global memory (bounded waits).  A
// launch beside others on the device takes its share of the room, and may have no helpers.
// A round that is too large even so is left, at the phase where it shows, to the phase
// launches that follow in the slot (RoundStage); their state is the same.
constexpr int kCBlock = 1024;        // threads per block
constexpr int kCMaxBlocks = 16;      // blocks per cluster (the non-portable size)
constexpr int kWinPerThread = 2;     // window edges each thread holds
constexpr int kCRounds = 1024;       // rounds per launch
// Work of a phase: the leader cluster runs up to kHelp... units alone and shares more with the
// helpers that have started; more than kMost... with all of a launch's helpers, kAlone... with none
// and in proportion between them, is left to the phase launches.  On a busy device helpers start
// late or not at all (with none, R-MAT 16 with 4 M edges at h = 1 took 462 ms by the limits of a
// launch with all of them, 200 by these; 167 with helpers).  Sharing costs about 5 us of hand-over and turns the counters' shared-memory atomics
// into global ones: with helpers from 256 detection items on, ER n = 2,000 detects in 12 us a round
// instead of 7; without helpers R-MAT 16 at h = 2 takes 800 ms instead of 640.
constexpr int kHelpDetect = 1024, kAloneDetect = 4096, kMostDetect = 1 << 16;     // detection items
constexpr int kHelpTest3 = 1 << 14, kAloneTest3 = 1 << 17, kMostTest3 = 1 << 20;  // radius-3 items
constexpr int kHelpDelta = 16384, kAloneDelta = 65536, kMostDelta = 1 << 21;       // update items
// Polls (of about a microsecond) without any progress on the other side after which a helper gives
// up waiting for a job, or the leader for its helpers: some minutes, which no phase within the limits
// above takes.  Counted in polls, so that time in which the device runs others does not count.
constexpr int kWaitPolls = 1 << 27;

__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ unsigned cluster_blocks() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

// The address of `p` (this block's shared memory) in the block of rank `rank`.
template <typename T>
__device__ __forceinline__ T *cluster_map(T *p, unsigned rank) {
    unsigned long long r;
    asm("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(reinterpret_cast<unsigned long long>(p)), "r"(rank));
    return reinterpret_cast<T *>(r);
}

enum ClusterStat { kStatPairs = 0, kStatReads, kStatTests, kStatBytes, kStatLost, kStatTouched, kStatC3,
                   kStatLost2, kNumStats };

// Adds the warp's sum of v to the block's counter.
__device__ __forceinline__ void stat_add(unsigned long long *s_stat, int which, unsigned v) {
    const unsigned s = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(s_stat + which, (unsigned long long)s);
}

__device__ __forceinline__ unsigned long long load_acquire(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void store_release(unsigned long long *p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// The phases helpers can share, as one call by block `blk` of `nblks`.  Consecutive detection
// and candidate items go to different blocks.
template <bool kH3>
__device__ __forceinline__ void shared_phase(const LossArgs &a, RoundCtr *ctr, WindowCtr *wctr,
                                             unsigned long long *s_stat, int phase, int blk, int nblks,
                                             int max_split, const HelperJob &job) {
    const int gw = (threadIdx.x >> 5) * nblks + blk, nwarps = nblks * (kCBlock / 32);
    if (phase == kStageDetect) {
        unsigned pairs = 0u, reads = 0u;
        detect_items<kH3, true>(a, ctr, gw, nwarps, job.nitems, max_split, job.round, pairs, reads,
                                (unsigned long long *)&ctr->touched);
        if (kH3) c3_items(a, ctr, nwarps - 1 - gw, nwarps, job.nF, job.round);  // the warps with fewest items first
        stat_add(s_stat, kStatPairs, pairs);
        stat_add(s_stat, kStatReads, reads);
    } else if (kH3 && phase == kStageTest3) {
        unsigned pairs = 0u, reads = 0u;
        test3_items<true>(a, ctr, gw, nwarps, 2 * c3_chunks(a) * job.nF, job.nitems, job.round, pairs, reads,
                          (unsigned long long *)&ctr->touched);
        stat_add(s_stat, kStatC3, pairs);
        stat_add(s_stat, kStatReads, reads);
    } else {
        unsigned tests = 0u, bytes = 0u;
        delta_items<true, true>(a, wctr, blk, nblks, job.nitems, job.win_hi, job.thr, tests, bytes);
        stat_add(s_stat, kStatTests, tests);
        stat_add(s_stat, kStatBytes, bytes);
        if (blk == 0 && threadIdx.x == 0) atomicAdd(s_stat + kStatBytes, kItemBytes * job.nitems);
    }
}

__device__ __forceinline__ void flush_stats(DevStatus *st, unsigned long long *s_stat) {
    const int tid = threadIdx.x;
    if (tid < kNumStats && s_stat[tid]) {
        unsigned long long *const out[kNumStats] = {
            (unsigned long long *)&st->st_pairs, &st->st_bytes_detect, (unsigned long long *)&st->st_tests,
            &st->st_bytes_update, (unsigned long long *)&st->st_lost, (unsigned long long *)&st->st_recomputed,
            (unsigned long long *)&st->st_c3_pairs, (unsigned long long *)&st->st_lost2};
        atomicAdd(out[tid], tid == kStatReads ? 4ull * s_stat[tid] : s_stat[tid]);
    }
}

// A helper block: registers, then takes its share of every job whose helper count covers its
// number, until the leader of launch `epoch` has finished.  A job word is (launch, job
// number, helper blocks); a block that is not needed reads nothing else of the job.
template <bool kH3>
__device__ __forceinline__ void helper_blocks(const LossArgs &a, unsigned long long epoch, int nblk,
                                           unsigned long long *s_stat) {
    __shared__ unsigned long long s_word;
    DevStatus *st = a.st;
    unsigned long long seen = (epoch << 40);
    int id = 0;
    if (threadIdx.x == 0) {
        atomicMax(&st->cl_reg, epoch << 32);
        id = (int)(atomicAdd(&st->cl_reg, 1ull) & 0xffffffffull);
    }
    for (;;) {
        if (threadIdx.x == 0) {
            unsigned long long word = 0ull;  // 0: stop
            for (int polls = 0, beat = vload(st->cl_beat);; polls++) {
                const unsigned long long w = load_acquire(&st->cl_job);
                if ((w >> 16) > (seen >> 16) && (w >> 40) == epoch) {
                    seen = w;
                    if (id < (int)(w & 0xffffull)) {
                        word = w;
                        break;
                    }
                }
                if (load_acquire(&st->cl_exit) > epoch) break;
                if (polls >= a.wait_polls) {
                    const int now = vload(st->cl_beat);
                    if (now == beat) {
                        atomicOr(&st->err, kErrBarrierTimeout);
                        break;
                    }
                    beat = now;
                    polls = 0;
                }
                __nanosleep(64);
            }
            __threadfence();
            s_word = word ? (word & 0xffffull) | ((unsigned long long)id << 32) : 0ull;
        }
        __syncthreads();
        const unsigned long long w = s_word;
        if (w == 0ull) break;
        const int blocks = nblk + (int)(w & 0xffffffffull), me = nblk + (int)(w >> 32);
        HelperJob job;
        job.phase = vload(st->cl_work.phase);
        job.nitems = vload(st->cl_work.nitems);
        job.nF = vload(st->cl_work.nF);
        job.round = vload(st->cl_work.round);
        job.win_hi = vload(st->cl_work.win_hi);
        job.thr = vload(st->cl_work.thr);
        shared_phase<kH3>(a, &st->cl_ctr, &st->cl_wctr, s_stat, job.phase, me, blocks, 2, job);
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(&st->cl_done, 1ull);
        }
    }
    __syncthreads();
    flush_stats(st, s_stat);
}

template <bool kH3>
__global__ void __launch_bounds__(kCBlock, 1) k_rounds_cluster(const __grid_constant__ LossArgs a) {
    __shared__ int s_leads, s_helpers, s_failed;
    __shared__ RoundCtr s_ctr[2];
    __shared__ WindowCtr s_wctr;
    __shared__ int s_min[3];
    __shared__ unsigned long long s_stat[kNumStats];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    DevStatus *st = a.st;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const unsigned rank = cluster_rank(), nblk = cluster_blocks();
    const bool lead = rank == 0 && tid == 0;
    const int nwarps = (int)nblk * (kCBlock / 32);
    const int gw = wid * (int)nblk + (int)rank;  // consecutive items go to different blocks
    const int nthreads = (int)nblk * kCBlock, gt = (int)rank * kCBlock + tid;
    const int win_cap = a.win_cap;
    // The first cluster of a launch to start leads; the others help.  Helpers that start late
    // (or never, while the device is busy) are not waited for.
    const unsigned long long epoch = (unsigned long long)a.launch;
    const int nclusters = (int)(gridDim.x / nblk);
    if (nclusters > 1) {
        if (lead) s_leads = atomicMax(&st->cl_lead, epoch) < epoch;
        cluster_sync();
        const bool leads = *(volatile int *)cluster_map(&s_leads, 0) != 0;
        cluster_sync();
        if (!leads) {
            if (a.no_helpers) return;
            if (tid < kNumStats) s_stat[tid] = 0ull;
            __syncthreads();
            helper_blocks<kH3>(a, epoch, (int)nblk, s_stat);
            return;
        }
    }
    if (vload(st->alive) == 0 || vload(st->halt) != 0 || vload(st->err) != 0 || vload(st->cont)) {
        cluster_sync();
        if (lead) {
            if (vload(st->cont)) st->stage = kStageSelect;  // a round of several batches: the launches'
            store_release(&st->cl_exit, epoch + 1);
        }
        return;
    }
    unsigned long long job_seq = 0ull, done_base = 0ull;
    if (lead) done_base = load_acquire(&st->cl_done);
    // the counters of the round and of the one before it take turns
    RoundCtr *const ctrs = cluster_map(&s_ctr[0], 0);
    WindowCtr *const wctr = cluster_map(&s_wctr, 0);
    auto reset_ctr = [&](RoundCtr *c) {
        *c = RoundCtr{};
        c->overflow_unit = INT_MAX;
    };
    if (tid == 0) {
        reset_ctr(&s_ctr[0]);
        reset_ctr(&s_ctr[1]);
        s_wctr = WindowCtr{};
        s_failed = 0;
        for (int j = 0; j < 3; j++) s_min[j] = INT_MAX;
        for (int j = 0; j < kNumStats; j++) s_stat[j] = 0ull;
    }
    int k = vload(st->k), round = vload(st->round), levels = vload(st->levels);
    int last_k = vload(st->last_k), max_k = vload(st->max_k);
    long long alive = vload(st->alive);
    const int first_round = round;
    long long removed = 0;
    int win_hi = 0, width = 8, buf = 0, stage = kStageNone;
    bool applied = true, rebuild = true;
    unsigned long long t_prev = a.timer && lead ? global_ns() : 0ull;
    auto clock = [&](int phase) {
        if (!a.timer || !lead) return;
        const unsigned long long t = global_ns();
        st->st_phase_ns[phase] += t - t_prev;
        t_prev = t;
    };
    auto count_round = [&](const RoundCtr *c) {
        s_stat[kStatTouched] += (unsigned long long)c->touched & kTouchedMask;
        s_stat[kStatLost] += (unsigned long long)c->touched >> kLostShift;
    };
    // smallest value the blocks put into s_min[buf] before the last barrier; the buffer used
    // two reductions ago is reset (a barrier lies between its readers and this point, and
    // another one before its next use)
    auto cluster_min = [&]() -> int {
        int v = lane < (int)nblk ? *(volatile int *)cluster_map(&s_min[buf], lane) : INT_MAX;
        v = __reduce_min_sync(0xffffffffu, v);
        if (tid == 0) s_min[(buf + 2) % 3] = INT_MAX;
        buf = (buf + 1) % 3;
        return v;
    };
    // The previous round's lost members leave the balls.  Nothing before the next updates reads
    // the old balls (h = 3: before the radius-3 tests), so this goes beside the detection, whose
    // chain of loads hides it.
    auto apply_previous = [&]() {
        if (applied) return;
        const RoundCtr *const prev = ctrs + ((round & 1) ^ 1);
        const int t = nthreads - 1 - gt;  // the warps with fewest detection items first
        apply_lost(a, t, nthreads, (int)min(vload(prev->nlost), (unsigned)a.lost_max), round - 1);
        if (kH3) {
            unsigned real = 0u;
            apply_lost2(a, t, nthreads, (int)min(vload(prev->nlost2), (unsigned)a.lost2_max), round - 1, real);
            stat_add(s_stat, kStatLost2, real);
        }
        applied = true;
    };
    // One phase over `work` units, by the leader cluster alone or with the helpers that have
    // started.  Counters of a shared phase are in global memory (a helper cannot reach the
    // leader's shared memory): copied there before and back after.  Ends with a barrier, unless
    // the work is too much (kLeft: nothing was done).
    enum { kDone = 0, kLeft, kFailed };  // kFailed: the helpers did not finish in time (an error is set)
    auto run_phase = [&](int phase, RoundCtr *ctr, HelperJob job, long long work, int help, int alone,
                         int most) -> int {
        int helpers = 0;
        if (nclusters == 1) {
            if (work > alone) return kLeft;
        } else if (work > help) {
            if (lead) {
                const unsigned long long reg = load_acquire(&st->cl_reg);
                const int started = (reg >> 32) == epoch ? (int)(reg & 0xffffull) : 0;
                const long long room = alone + (long long)(most - alone) * started / ((nclusters - 1) * (int)nblk);
                s_helpers = work > room ? -1 : started;
                if (s_helpers > 0) {
                    job.phase = phase;
                    st->cl_work = job;
                    st->cl_ctr = *ctr;
                    st->cl_wctr = *wctr;
                    job_seq++;
                    store_release(&st->cl_job, (epoch << 40) | (job_seq << 16) | (unsigned)s_helpers);
                }
            }
            cluster_sync();
            helpers = *(volatile int *)cluster_map(&s_helpers, 0);
            if (helpers < 0) return kLeft;
        }
        if (helpers == 0) {
            shared_phase<kH3>(a, ctr, wctr, s_stat, phase, (int)rank, (int)nblk, 5, job);
            cluster_sync();
            return kDone;
        }
        const int blocks = (int)nblk + helpers;
        shared_phase<kH3>(a, &st->cl_ctr, &st->cl_wctr, s_stat, phase, (int)rank, blocks, 2, job);
        cluster_sync();
        if (lead) {
            done_base += (unsigned)helpers;
            unsigned long long last = 0ull;
            for (int polls = 0;; polls++) {
                const unsigned long long done = load_acquire(&st->cl_done);
                if (done >= done_base) break;
                if (done != last) {
                    last = done;
                    polls = 0;
                }
                if (polls >= a.wait_polls || vload(st->err) != 0) {
                    atomicOr(&st->err, kErrBarrierTimeout);
                    s_failed = 1;
                    break;
                }
            }
            __threadfence();
            RoundCtr c;
            const int *from = reinterpret_cast<const int *>(&st->cl_ctr);
            int *to = reinterpret_cast<int *>(&c);
            for (int j = 0; j < (int)(sizeof(RoundCtr) / sizeof(int)); j++) to[j] = vload(from[j]);
            *ctr = c;
            wctr->nwin = vload(st->cl_wctr.nwin);
            wctr->nnext = vload(st->cl_wctr.nnext);
        }
        cluster_sync();
        // (not s_helpers: the leader may be in the next phase already and write it)
        return *(volatile int *)cluster_map(&s_failed, 0) ? kFailed : kDone;
    };
    cluster_sync();
    for (;;) {
        RoundCtr *const ctr = ctrs + (round & 1), *const prev = ctrs + ((round & 1) ^ 1);
        // the frontier: the edges the last updates took to the level, if any; else it comes
        // from the window
        const int nnext = rebuild || round - first_round >= kCRounds ? 0 : vload(wctr->nnext);
        const bool direct = nnext > 0 && nnext <= win_cap;
        int we[kWinPerThread];
        bool take[kWinPerThread];
        const int32_t *const list = direct ? a.next : a.win;
        int nlist = direct ? nnext : min(vload(wctr->nwin), win_cap);
        auto load_list = [&]() {
#pragma unroll
            for (int j = 0; j < kWinPerThread; j++) {
                const int i = (lane + 32 * j) * nwarps + gw;
                we[j] = i < nlist ? list[i] : -1;
                take[j] = direct && we[j] >= 0;
            }
        };
        load_list();
        if (!direct) {
            int mn = INT_MAX;
            const bool rebuilt = rebuild;
            while (rebuild) {
                cluster_sync();  // the old window is no longer read
                if (lead) wctr->nwin = 0;
                cluster_sync();
                win_hi = k - 2 + width;
                int lmin = INT_MAX;
                const int64_t stride = 4 * (int64_t)nthreads;
                // a full window ends the scan: where every round has a larger frontier than it
                // holds, whole scans at each width by one cluster cost more than the round (R-MAT
                // 18 with 16 M edges at h = 1: 912 -> 838 ms)
                bool full = false;
                for (int64_t e0 = 4 * ((int64_t)gt & ~31ll); e0 < a.m && !full; e0 += stride) {
                    int sv[4];
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const int64_t e = e0 + 32 * j + lane;
                        sv[j] = (e < a.m) ? a.sup[e] : INT_MAX;
                    }
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        lmin = min(lmin, sv[j]);
                        const unsigned bal = __ballot_sync(0xffffffffu, sv[j] <= win_hi);
                        if (bal) {
                            int base = 0;
                            if (lane == 0) base = atomicAdd(&wctr->nwin, __popc(bal));
                            base = __shfl_sync(0xffffffffu, base, 0) + __popc(bal & lanemask_lt());
                            if (sv[j] <= win_hi && base < win_cap) a.win[base] = (int)(e0 + 32 * j + lane);
                            full = __any_sync(0xffffffffu, base >= win_cap);
                        }
                    }
                }
                lmin = __reduce_min_sync(0xffffffffu, lmin);
                if (lane == 0 && lmin != INT_MAX) atomicMin(&s_min[buf], lmin);
                cluster_sync();
                mn = cluster_min();
                nlist = vload(wctr->nwin);
                if (nlist > win_cap) {
                    // the scan stopped there: its minimum is not that of all edges
                    if (width == 0) {  // a frontier larger than the window
                        stage = kStageSelect;
                        break;
                    }
                    width >>= 2;
                    continue;
                }
                if (mn == INT_MAX) {
                    alive = 0;
                    break;
                }
                k = max(k, mn + 2);
                if (nlist > 0) {
                    rebuild = false;
                    if (nlist < win_cap / 16) width = min(2 * width + 1, 1 << 20);
                }
            }
            if (rebuild) break;  // nothing alive, or left to the launches
            if (rebuilt) load_list();
            // the window's supports and their minimum
            int ws[kWinPerThread];
            int lmin = INT_MAX;
#pragma unroll
            for (int j = 0; j < kWinPerThread; j++) {
                ws[j] = we[j] >= 0 ? a.sup[we[j]] : INT_MAX;
                lmin = min(lmin, ws[j]);
            }
            lmin = __reduce_min_sync(0xffffffffu, lmin);
            if (lane == 0 && lmin != INT_MAX) atomicMin(&s_min[buf], lmin);
            const bool spilled = vload(wctr->nwin) > win_cap;
            cluster_sync();
            mn = cluster_min();
            if (spilled) {  // crossings did not fit the list
                width >>= 2;
                rebuild = true;
                continue;
            }
            if (mn == INT_MAX) {
                if (alive == 0) break;
                rebuild = true;
                continue;
            }
            if (round - first_round >= kCRounds) break;
            k = max(k, mn + 2);
#pragma unroll
            for (int j = 0; j < kWinPerThread; j++) take[j] = ws[j] <= k - 2;
        }
        // selection and removal, and the detection items of the frontier's edge sides
#pragma unroll
        for (int j = 0; j < kWinPerThread; j++) select_one(a, ctr, take[j], we[j], k, round);
        cluster_sync();
        clock(kTimeSelect);
        // Every block takes the decisions of this loop alike: between two barriers they read
        // only counters that nothing changes before the next one (overflow marks, which the
        // phase now starting may set, are read where no phase sets them).
        const int nF = vload(ctr->nF);
        const long long npitems = vload(ctr->npitems);
        if (lead) *(volatile int *)&st->cl_beat = round + 1;  // for the helpers: rounds go on
        if (lead) wctr->nnext = 0;  // read by all before the barrier, used again after the next
        const long long nA = kH3 ? 2ll * c3_chunks(a) * nF : 0ll;
        if (npitems > a.pitems_cap || nA > (nclusters > 1 ? kMostTest3 : kAloneTest3)) {
            stage = kStageDetect;
            break;
        }
        HelperJob job;
        job.phase = 0;
        job.nitems = (int)npitems;
        job.nF = nF;
        job.round = round;
        job.win_hi = win_hi;
        job.thr = k - 2;
        apply_previous();
        int got = run_phase(kStageDetect, ctr, job, npitems, kHelpDetect, kAloneDetect, kMostDetect);
        if (got != kDone) {
            if (got == kLeft) stage = kStageDetect;
            break;
        }
        clock(kTimeDetect);
        if (kH3) {
            // too many items, or no room for the items or the radius-2 losses (a halt)
            const long long nc3 = vload(ctr->nc3items);
            if (nA + nc3 > a.c3items_cap || vload(ctr->nlost2) > (unsigned)a.lost2_max) {
                stage = kStageTest3;
                break;
            }
            job.nitems = (int)(nA + nc3);
            got = run_phase(kStageTest3, ctr, job, nA + nc3, kHelpTest3, kAloneTest3, kMostTest3);
            if (got != kDone) {
                if (got == kLeft) stage = kStageTest3;
                break;
            }
            clock(kTimeTest3);
        }
        if (lead) {  // the round before is done with
            count_round(prev);
            reset_ctr(prev);
        }
        const int nuitems = vload(ctr->nuitems);
        if (vload(ctr->overflow_unit) != INT_MAX || (kH3 && vload(ctr->halt) != 0)) {
            stage = kStageDelta;
            break;
        }
        job.nitems = nuitems;
        got = run_phase(kStageDelta, ctr, job, nuitems, kHelpDelta, kAloneDelta, kMostDelta);
        if (got != kDone) {
            if (got == kLeft) stage = kStageDelta;
            break;
        }
        clock(kTimeDelta);
        // the round's bookkeeping (round_finalize's, kept by every thread alike)
        if (k != last_k) {
            levels++;
            last_k = k;
        }
        max_k = max(max_k, k);
        round++;
        removed += nF;
        alive -= nF;
        applied = false;
    }
    apply_previous();
    cluster_sync();
    if (lead) {
        // a round left unfinished keeps its counters (`touched` among them: its closing
        // launch adds them), the last finished one only adds its touched edges
        RoundCtr *const ctr = ctrs + (round & 1), *const prev = ctrs + ((round & 1) ^ 1);
        count_round(prev);
        if (stage <= kStageSelect) reset_ctr(ctr);
        *static_cast<RoundCtr *>(st) = *ctr;
    }
    __syncthreads();
    flush_stats(st, s_stat);
    if (lead) {
        st->k = k;
        st->round = round;
        st->levels = levels;
        st->last_k = last_k;
        st->max_k = max_k;
        st->alive = alive;
        st->st_frontier += removed;
        st->st_slots += round - first_round;
        st->stage = stage;
        st->unit_begin = 0;
        if (a.timer) st->st_phase_start = global_ns();
        store_release(&st->cl_exit, epoch + 1);
    }
}

LossArgs loss_args(Handle *H) {
    PeelWork &w = H->w;
    GraphDev &g = H->g;
    LossArgs a;
    a.h = w.h;
    a.lost_max = (int32_t)w.lost_max;
    a.cap_mask = (unsigned)(w.lost_cap - 1);
    a.row_ptr = g.row_ptr;
    a.col = g.col;
    a.col_live = w.col_live;
    a.slot_eid = g.slot_eid;
    a.eu = g.eu;
    a.ev = g.ev;
    a.frontier = w.frontier;
    a.stamp = w.stamp;
    a.pool = w.pool;
    a.ball_off = w.ball_off;
    a.ball_nw = w.ball_nw;
    a.ball_meta = w.ball_meta;
    a.ball_size = w.ball_size;
    a.keys = w.lost_keys;
    a.lost = w.lost;
    a.sup = w.sup;
    a.vtouch = w.edge_touch;
    a.deg_alive = w.deg_alive;
    a.pitems_cap = (int32_t)w.pitems_cap;
    a.pitems = w.pitems;
    a.uitems_cap = (int32_t)w.uitems_cap;
    a.uitems = w.uitems;
    a.upd_budget = w.upd_budget;
    a.hub_slot = w.hub_slot;
    a.hub_bits = w.hub_bits;
    a.Wpad = w.Wpad;
    a.dense_all = w.dense_balls ? 1 : 0;
    a.hub_all = (w.nhub == g.n && w.hub_min_deg == 1) ? 1 : 0;
    a.m = g.m;
    a.slot_lo = g.slot_lo;
    a.slot_hi = g.slot_hi;
    a.truss = w.truss;
    a.stamp_w = w.stamp;
    a.frontier_w = w.frontier;
    a.col_live_w = w.col_live;
    a.deg_alive_w = w.deg_alive;
    a.hub_bits_w = w.hub_bits;
    a.st = w.status;
    a.h3 = w.inc3 ? 1 : 0;
    a.pool2 = w.pool2;
    a.ball_size2 = w.ball_size2;
    a.keys2 = w.lost2_keys;
    a.cap2_mask = w.lost2_cap > 0 ? (unsigned)(w.lost2_cap - 1) : 0u;
    a.lost2 = w.lost2;
    a.lost2_max = (int32_t)w.lost2_max;
    a.c3items_cap = (int32_t)w.c3items_cap;
    a.c3items = w.c3items;
    a.touch2 = w.touch2;
    a.pool_new = w.twin ? w.pool_new : nullptr;
    a.pool2_new = w.twin ? w.pool2_new : nullptr;
    a.cluster = 0;
    a.launch = 0;
    a.wait_polls = test_wait_polls() > 0 ? test_wait_polls() : kWaitPolls;
    a.no_helpers = test_no_helpers() ? 1 : 0;
    a.max_split = H->shared_device ? 0 : 2;  // beside others, idle warps are theirs
    a.timer = 0;
    a.win_cap = 0;
    a.win = w.win;
    a.next = w.win + w.win_cap;
    a.erec = w.erec;
    a.srec = w.srec;
    return a;
}

}  // namespace

// Launches the persistent round kernel once (at most max_slots round slots).  The grid is
// every block that can be resident at once, as a cooperative launch requires.
htd_status launch_persistent_rounds(Handle *H, cudaStream_t s, int max_slots, int64_t *launches) {
    LossArgs a = loss_args(H);
    static thread_local int grid_cached = 0, dev_cached = -1;
    if (grid_cached == 0 || dev_cached != H->g.device) {
        int occ = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_rounds_persistent,
                                                                      kPBlock, 0);
        if (e != cudaSuccess || occ < 1) {
            set_last_error("persistent round kernel: no resident block fits");
            return HTD_ECUDA;
        }
        grid_cached = std::min(H->num_sms * occ, 64 * 32);  // the grid barrier's limit
        dev_cached = H->g.device;
    }
    void *args[] = {&a, &max_slots};
    cudaError_t e = cudaLaunchCooperativeKernel((const void *)k_rounds_persistent, dim3(grid_cached),
                                                dim3(kPBlock), args, 0, s);
    (*launches)++;
    if (e != cudaSuccess) {
        set_last_error(std::string("persistent round kernel: ") + cudaGetErrorString(e));
        return HTD_ECUDA;
    }
    return HTD_OK;
}

namespace {

// Blocks of one full wave of a phase kernel (every block resident at once), per device.
struct PhaseGrids {
    int device = -1;
    uint64_t context = 0;
    int detect = 0, detect3 = 0, delta = 0, test3 = 0;
    int cluster = 0;   // blocks of a cluster of the cluster round kernel (0: none fits the device)
    int clusters = 0;  // clusters of a launch that has the device to itself
};

using PhaseKernel = void (*)(LossArgs);

// Launch configuration of the cluster round kernel: `clusters` clusters of `blocks` blocks.
struct ClusterLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    ClusterLaunch(int clusters, int blocks, cudaStream_t s, bool pdl) {
        cfg.gridDim = dim3((unsigned)(clusters * blocks));
        cfg.blockDim = dim3(kCBlock);
        cfg.stream = s;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)blocks;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = pdl ? 2 : 1;
    }
};

// The largest cluster both forms of the kernel can run as on this device: 16 blocks (which
// needs the non-portable size), else 8, else none.
// *resident: clusters of that size the whole device holds at once.
int cluster_size(int *resident) {
    for (int blocks = kCMaxBlocks; blocks >= 8; blocks /= 2) {
        bool fits = true;
        *resident = INT_MAX;
        for (PhaseKernel kern : {PhaseKernel(k_rounds_cluster<false>), PhaseKernel(k_rounds_cluster<true>)}) {
            if (blocks > 8)
                fits = fits && cudaFuncSetAttribute((const void *)kern, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                                    1) == cudaSuccess;
            ClusterLaunch c(1, blocks, nullptr, false);
            int n = 0;
            fits = fits && cudaOccupancyMaxActiveClusters(&n, (const void *)kern, &c.cfg) == cudaSuccess && n > 0;
            *resident = std::min(*resident, n);
        }
        if (fits) return blocks;
        (void)cudaGetLastError();
    }
    *resident = 0;
    return 0;
}

template <bool kTwin>
htd_status phase_grids(Handle *H, PhaseGrids &pg) {
    const uint64_t context = call_context();
    if (pg.device == H->g.device && pg.context == context) return HTD_OK;
    int od = 0, od3 = 0, ou = 0, ot = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&od, k_loss_detect<kTwin>, kBlock, 0) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&od3, k_loss_detect3<kTwin>, kBlock, 0) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ou, k_loss_delta<kTwin>, kBlock, 0) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ot, k_loss3_test<kTwin>, kBlock, 0) != cudaSuccess ||
        od < 1 || od3 < 1 || ou < 1 || ot < 1) {
        set_last_error("incremental round: no resident block fits");
        return HTD_ECUDA;
    }
    pg.detect = H->num_sms * od;
    pg.detect3 = H->num_sms * od3;
    pg.delta = H->num_sms * ou;
    pg.test3 = H->num_sms * ot;
    int resident = 0;
    pg.cluster = cluster_size(&resident);
    // one cluster's room stays free, so that another stream's leader can start beside it
    pg.clusters = std::max(1, resident - 1);
    pg.device = H->g.device;
    pg.context = context;
    return HTD_OK;
}

// One phase launch; `pdl` lets it be scheduled before the previous kernel on the stream
// has finished (it waits in phase_entry).
cudaError_t launch_phase(void (*kernel)(LossArgs), int grid, cudaStream_t s, bool pdl,
                         const LossArgs &a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kBlock);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

template <bool kTwin>
cudaError_t launch_slot(Handle *H, LossArgs &a, cudaStream_t s, int64_t *launches, bool by_cluster) {
    static thread_local PhaseGrids pg;
    if (phase_grids<kTwin>(H, pg) != HTD_OK) return cudaErrorInvalidConfiguration;
    const bool pdl = true;
    a.cluster = (pg.cluster > 0 && kTwin && by_cluster) ? 1 : 0;
    a.win_cap = (int32_t)std::min<int64_t>(H->w.win_cap, (int64_t)pg.cluster * kCBlock * kWinPerThread);
    const int grid_scan = H->num_sms * kScanBlocks;
    cudaError_t e = cudaSuccess;
    if (a.cluster) {
        // Peels of several threads share the room for clusters: helpers of one keep the leader of
        // another waiting until their launch ends (eight threads, DC-SBM 40k at h = 2: 52.6 ms a
        // peel with five helpers each, 28.5 ms with this; 49.2 ms with one launch per phase).  The
        // share follows the peels in flight from launch to launch, so that a peel which began
        // alone makes room for the ones that join it (seven threads joining R-MAT 16 at h = 2: their
        // slowest peel 290-342 ms with a share kept for the whole peel, 139-189 with this, 248 with
        // one launch per phase).  (Job words hold 24 bits of the number.)
        const int peels = std::max({H->peers, (int32_t)peels_in_flight(H->g.device).load(), 1});
        a.launch = ++H->cluster_launches;
        const int clusters = a.launch < (1 << 24) ? std::max(1, pg.clusters / peels) : 1;
        ClusterLaunch c(clusters, pg.cluster, s, pdl);
        e = cudaLaunchKernelEx(&c.cfg, a.h3 ? k_rounds_cluster<true> : k_rounds_cluster<false>, a);
        *launches += 1;
    }
    if (e == cudaSuccess) e = launch_phase(k_inc_select, grid_scan, s, pdl, a);
    if (a.h3) {
        // select | radius-2 detection + radius-3 items | radius-3 tests | updates | reduce
        if (e == cudaSuccess) e = launch_phase(k_loss_detect3<kTwin>, pg.detect3, s, pdl, a);
        if (e == cudaSuccess) e = launch_phase(k_loss3_test<kTwin>, pg.test3, s, pdl, a);
    } else {
        if (e == cudaSuccess) e = launch_phase(k_loss_detect<kTwin>, pg.detect, s, pdl, a);
    }
    if (e == cudaSuccess) e = launch_phase(k_loss_delta<kTwin>, pg.delta, s, pdl, a);
    if (e == cudaSuccess) e = launch_phase(k_loss_apply_reduce, grid_scan, s, pdl, a);
    *launches += a.h3 ? 5 : 4;
    return e;
}

}  // namespace

// Enqueues one slot of incremental rounds: with the twin matrices the cluster round kernel,
// then the launches of one round, which run from the phase that kernel left to them.  Every
// launch is programmatic (it overlaps the previous one's tail).
htd_status enqueue_incremental_round(Handle *H, cudaStream_t s, int64_t *launches, bool timer, bool by_cluster) {
    LossArgs a = loss_args(H);
    a.timer = timer ? 1 : 0;
    cudaError_t e = H->w.twin ? launch_slot<true>(H, a, s, launches, by_cluster)
                              : launch_slot<false>(H, a, s, launches, false);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_last_error(std::string("enqueue_incremental_round: ") + cudaGetErrorString(e));
        return HTD_ECUDA;
    }
    return HTD_OK;
}

}  // namespace htd
