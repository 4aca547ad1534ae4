// Per-user epilogues of the fused product kernels.
//
// Both product passes see approximate scores v ~ u.p with a proven error bound E
// (|v - u.p| <= E for every pair of the tile).  One thread owns one user row of
// the tile and consumes it 32 columns at a time.
//
// Threshold pass (K2, Definition 1).  The thread keeps a min-heap of the k largest
// lower bounds v - E seen so far; its root L never exceeds tau_u, because k items
// have u.p >= L.  Any item with u.p >= tau_u has v + E >= u.p >= L, so keeping every
// item with v >= L - E as a candidate (with its upper bound v + E) keeps all of
// S_k(u) and every item tied with t_u.  Candidates whose upper bound fell below the
// current L can never be needed and are compacted away when the list fills.
//
// Counting pass (K5, Eq. 1).  v > tau_u + E proves u.p > tau_u (member); v < tau_u - E
// proves u.p < tau_u (not a member); anything between is queued for exact rescoring.
#pragma once

#include "common.cuh"

namespace rkm {

// Heap element j of user-thread t lives at heap[j * BU + t] (conflict-free per warp).
__device__ __forceinline__ void heap_replace_root(float* heap, int t, int k, float v) {
    int j = 0;
    while (true) {
        int l = 2 * j + 1;
        if (l >= k) break;
        int c = l;
        float cv = heap[l * BU + t];
        int r = l + 1;
        if (r < k) {
            float rv = heap[r * BU + t];
            if (rv < cv) { c = r; cv = rv; }
        }
        if (cv >= v) break;
        heap[j * BU + t] = cv;
        j = c;
    }
    heap[j * BU + t] = v;
}

static __device__ __noinline__ int compact_candidates(Cand* c, int cnt, float L) {
    // Keep the candidates whose upper bound still reaches the bound L <= tau_u.
    int w = 0;
    for (int r = 0; r < cnt; ++r) {
        Cand x = c[r];
        if (x.ub >= L) c[w++] = x;
    }
    return w;
}

struct SelState {
    float L;     // heap root once the heap holds k lower bounds (-inf while it fills)
    int hn;      // lower bounds held in the heap (<= k)
    float Lw;    // warm-start bound of this group (-inf if none)
    float Lx;    // a lower bound of tau_u published by the other epilogue group (or -inf)
    float thr;   // max(L, Lw, Lx) - E of the current tile, rounded down
    int cnt;     // candidates stored
    unsigned long long* pub;  // where this group publishes its bound for the other (null: none)
    unsigned tag;             // user tile the published bound belongs to
    int mark;    // first candidate not yet offered to the heap (-1 after a compaction)
    float Em;    // largest error bound of the tiles since
};

// The best lower bound of tau_u this group knows.
__device__ __forceinline__ float sel_bound(const SelState& s) { return fmaxf(fmaxf(s.L, s.Lw), s.Lx); }

// A published bound: (user tile << 32) | bits of the bound, written and read as one 64-bit
// word so a reader never mixes a bound with the tag of another user tile.
__device__ __forceinline__ void publish_bound(unsigned long long* p, unsigned tag, float L) {
    *reinterpret_cast<volatile unsigned long long*>(p) =
        ((unsigned long long)tag << 32) | (unsigned long long)__float_as_uint(L);
}

__device__ __forceinline__ float read_bound(const unsigned long long* p, unsigned tag) {
    const unsigned long long x = *reinterpret_cast<const volatile unsigned long long*>(p);
    return ((unsigned)(x >> 32) == tag) ? __uint_as_float((unsigned)(x & 0xffffffffull)) : -INFINITY;
}

// Min-heap order over heap[0 .. k) of user-thread t (bottom-up construction).
__device__ __forceinline__ void heapify(float* heap, int t, int k) {
    for (int i = k / 2 - 1; i >= 0; --i) {
        const float v = heap[i * BU + t];
        int j = i;
        while (true) {
            const int l = 2 * j + 1;
            if (l >= k) break;
            int c = l;
            float cv = heap[l * BU + t];
            if (l + 1 < k) {
                const float rv = heap[(l + 1) * BU + t];
                if (rv < cv) { c = l + 1; cv = rv; }
            }
            if (cv >= v) break;
            heap[j * BU + t] = cv;
            j = c;
        }
        heap[j * BU + t] = v;
    }
}

// Record a value that reached the threshold: store it as a candidate (with its upper bound).  Its
// lower bound enters the heap later (sel_merge): any k lower bounds held in the heap make its root
// a valid lower bound of tau_u, so delaying or skipping an admission is sound.
__device__ __forceinline__ void sel_insert(float v, int pos, float E, SelState& s, Cand* mycand, int cap,
                                           DevStatus* st) {
    if (s.cnt >= cap) {
        s.cnt = compact_candidates(mycand, s.cnt, sel_bound(s));
        s.mark = -1;
    }
    if (s.cnt < cap) {
        Cand c;
        c.ub = __fadd_ru(v, E);
        c.pos = pos;
        mycand[s.cnt++] = c;
    } else {
        st->cand_overflow = 1u;
    }
}

// A lower bound of u.p for a candidate recorded with ub = RU(v + E) in a tile whose products
// have error bound E: v >= ub - E - ulp(ub), so u.p >= v - E >= ub - 2E - ulp(ub) (the ulp
// taken as |ub| 2^-23 + 2^-149, every step rounded down).
__device__ __forceinline__ float cand_lower(float ub, float E) {
    const float d = __fadd_ru(__fmul_ru(fabsf(ub), 0x1p-23f), 0x1p-149f);
    return __fsub_rd(__fsub_rd(__fsub_rd(ub, E), E), d);
}

// A selector offers its candidates to the heap after MERGE_TILES of its tiles, or once some row of
// the warp has MERGE_HITS new ones.
constexpr int MERGE_TILES = 8;
constexpr int MERGE_HITS = 2;

// Deferred admissions: the lower bounds of the candidates recorded since the last call enter the
// heap with every lane of the warp stepping through its own list together (the heap is built at
// most once per lane, in one place, instead of at the hit that completes it).  Candidates are read
// back four at a time, so that a step waits for one read instead of four.  Skipping admissions
// is sound (see sel_insert), so a list that a compaction moved admits nothing.
__device__ __forceinline__ void sel_merge(SelState& s, const Cand* mycand, float* heap, int t, int k, bool active) {
    const float E = s.Em;
    int j = s.mark;
    const int j1 = s.cnt;
    s.mark = s.cnt;
    s.Em = 0.f;
    if (!active || j < 0 || j >= j1) return;
    const float L0 = sel_bound(s);
    bool filled = false;
    while (j < j1 && s.hn < k) {
        float ub[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) ub[i] = j + i < j1 ? mycand[j + i].ub : -INFINITY;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (s.hn == k || j >= j1) break;
            const float lb = cand_lower(ub[i], E);
            if (lb > L0) {
                heap[s.hn * BU + t] = lb;
                if (++s.hn == k) filled = true;
            }
            ++j;
        }
    }
    if (filled) {
        heapify(heap, t, k);
        s.L = heap[t];
    }
    while (j < j1) {
        float ub[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) ub[i] = j + i < j1 ? mycand[j + i].ub : -INFINITY;
#pragma unroll 1
        for (int i = 0; i < 4 && j < j1; ++i, ++j) {
            const float lb = cand_lower(i == 0 ? ub[0] : i == 1 ? ub[1] : i == 2 ? ub[2] : ub[3], E);
            if (lb > sel_bound(s)) {
                heap_replace_root(heap, t, k, lb);
                s.L = heap[t];
            }
        }
    }
    if (s.hn == k && s.pub) publish_bound(s.pub, s.tag, fmaxf(s.L, s.Lw));
}

// x = v[c] for a run-time c in [0, 32): a five-level select tree (no local memory).
__device__ __forceinline__ float select32(const float (&v)[32], int c) {
    float l1[16], l2[8], l3[4], l4[2];
#pragma unroll
    for (int i = 0; i < 16; ++i) l1[i] = (c & 1) ? v[2 * i + 1] : v[2 * i];
#pragma unroll
    for (int i = 0; i < 8; ++i) l2[i] = (c & 2) ? l1[2 * i + 1] : l1[2 * i];
#pragma unroll
    for (int i = 0; i < 4; ++i) l3[i] = (c & 4) ? l2[2 * i + 1] : l2[2 * i];
#pragma unroll
    for (int i = 0; i < 2; ++i) l4[i] = (c & 8) ? l3[2 * i + 1] : l3[2 * i];
    return (c & 16) ? l4[1] : l4[0];
}

// Maxima of the four 8-column groups of a chunk.
__device__ __forceinline__ void group_max8(const float (&v)[32], float (&g)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
        g[q] = fmax3f(fmax3f(v[8 * q], v[8 * q + 1], v[8 * q + 2]), fmax3f(v[8 * q + 3], v[8 * q + 4], v[8 * q + 5]),
                      fmaxf(v[8 * q + 6], v[8 * q + 7]));
}

// Bit c of the result is set when v[c] >= thr, for the 8-column groups whose maximum g[q]
// reaches thr in some lane of the warp (all 32 lanes must call it).
__device__ __forceinline__ unsigned hit_mask(const float (&v)[32], const float (&g)[4], bool active, float thr) {
    unsigned mask = 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const bool hq = active && g[q] >= thr;
        if (__any_sync(0xffffffffu, hq) && hq) {
#pragma unroll
            for (int j = 0; j < 8; ++j) mask |= (v[8 * q + j] >= thr ? 1u : 0u) << (8 * q + j);
        }
    }
    return mask;
}

// Threshold-pass epilogue of one 32-column chunk, called when the pair vote of the product
// kernel found a value reaching some lane's threshold.  Must be called by all 32 lanes of the
// warp: a maximum tree and a vote skip a chunk without hits; 8-column groups in which some
// lane reaches its threshold are compared element by element, and the hits are inserted one
// by one through a single call site.  `active` masks lanes without a valid user.
__device__ __forceinline__ void sel_chunk(const float (&v)[32], bool active, int pos0, int64_t m,
                                          float E, SelState& s, Cand* mycand, int cap, DevStatus* st) {
    float g[4];
    group_max8(v, g);
    const float mx = fmax3f(g[0], g[1], fmaxf(g[2], g[3]));
    if (!__any_sync(0xffffffffu, active && mx >= s.thr)) return;
    if (pos0 + 32 <= m && !__any_sync(0xffffffffu, active && s.cnt + 32 > cap)) {
        // Room for the whole chunk and no column past the items: the columns of each 8-column
        // group with a hit are compared and stored in place, without a branch per hit.
        Cand* p = mycand + s.cnt;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool hq = active && g[q] >= s.thr;
            if (!__any_sync(0xffffffffu, hq)) continue;
            const float thr = hq ? s.thr : INFINITY;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float x = v[8 * q + j];
                if (hq && x >= thr) {
                    Cand c;
                    c.ub = __fadd_ru(x, E);
                    c.pos = pos0 + 8 * q + j;
                    *p++ = c;
                }
            }
        }
        s.cnt = (int)(p - mycand);
        return;
    }
    unsigned mask = hit_mask(v, g, active, s.thr);
    while (mask) {
        const int c = __ffs(mask) - 1;
        mask &= mask - 1u;
        const float x = select32(v, c);
        // s.thr only grows, so skipping values now below it is still sound.
        if (x >= s.thr && pos0 + c < m) sel_insert(x, pos0 + c, E, s, mycand, cap, st);
    }
}

// Band pairs of one warp on their way to the queue in global memory: pushed one by one they cost
// a global atomic with its round trip each, while the accumulator was held.
constexpr int BAND_STAGE = 128;  // pairs per warp in shared memory
struct BandStage {
    int2* q;  // this warp's [BAND_STAGE]
    int n;    // pairs staged (the same in every lane)
};

// Append the staged pairs to the band queue (all 32 lanes).
__device__ __forceinline__ void band_flush(BandStage& b, int2* __restrict__ band, unsigned band_cap, DevStatus* st) {
    if (b.n == 0) return;
    const int lane = threadIdx.x & 31;
    __syncwarp();
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(&st->band_count, (unsigned)b.n);
    base = __shfl_sync(0xffffffffu, base, 0);
    for (int j = lane; j < b.n; j += 32) {
        if (base + j < band_cap) band[base + j] = b.q[j];
        else st->band_overflow = 1u;
    }
    b.n = 0;
    __syncwarp();
}

// Counting-pass epilogue of one 32-column chunk; same calling rule as sel_chunk.
// cnt_s: per-column member counters of the tile (shared memory), indexed by column.  A lane's
// values become two bit masks (at least lo, above hi), so no value has to be picked out of the
// registers again: members are one shared-memory increment per bit, the others go to the stage.
// Cycles in hits per tile and warp over the first 8,192 items, where most are, with a value selected
// and a queue atomic per pair -> so: 500K users, d = 64 3,750 -> 2,440; 200K, d = 96 4,410 -> 2,900;
// 100K, FP8 10,400 -> 4,870.
__device__ __forceinline__ void count_chunk(const float (&v)[32], bool active, int col0, int pos0,
                                            int64_t mlim, float hi, float lo, int* cnt_s,
                                            int u_orig, BandStage& stage, int2* band, unsigned band_cap,
                                            DevStatus* st) {
    float g[4];
    group_max8(v, g);
    unsigned reach = 0u, above = 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (!__any_sync(0xffffffffu, active && g[q] >= lo)) continue;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            reach |= (v[8 * q + j] >= lo ? 1u : 0u) << (8 * q + j);
            above |= (v[8 * q + j] > hi ? 1u : 0u) << (8 * q + j);
        }
    }
    if (!active) reach = 0u;
    if (pos0 + 32 > mlim) reach &= pos0 < mlim ? (1u << (int)(mlim - pos0)) - 1u : 0u;
    unsigned members = reach & above, open = reach & ~above;
    while (members) {
        atomicAdd(&cnt_s[col0 + __ffs(members) - 1], 1);
        members &= members - 1u;
    }
    const unsigned lt_mask = (1u << (threadIdx.x & 31)) - 1u;
    for (unsigned with; (with = __ballot_sync(0xffffffffu, open != 0u)) != 0u;) {
        if (open) {
            stage.q[stage.n + __popc(with & lt_mask)] = make_int2(u_orig, pos0 + __ffs(open) - 1);
            open &= open - 1u;
        }
        stage.n += __popc(with);
        if (stage.n > BAND_STAGE - 32) band_flush(stage, band, band_cap, st);
    }
}

// Bitonic network over N registers in descending order, from merges of SIZE on.
template <int N, int SIZE, int STRIDE = SIZE / 2>
__device__ __forceinline__ void sort_desc(float (&v)[N]) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int j = i ^ STRIDE;
        if (j > i) {
            const float hi = fmaxf(v[i], v[j]), lo = fminf(v[i], v[j]);
            const bool desc = (i & SIZE) == 0;
            v[i] = desc ? hi : lo;
            v[j] = desc ? lo : hi;
        }
    }
    if constexpr (STRIDE > 1) sort_desc<N, SIZE, STRIDE / 2>(v);
    else if constexpr (SIZE < N) sort_desc<N, SIZE * 2>(v);
}

// Warm-start bound from COLS columns of one accumulator row held in TMEM: the maxima of
// the NG column groups of width COLS/NG, sorted by a bitonic network in registers; the k-th
// largest (k <= NG) minus E bounds tau_u from below, because k distinct items reach it.
// Columns at or beyond m count as -inf.  Returns -inf when fewer than k groups are valid.
template <int NG, int COLS, typename LoadChunk>
__device__ __forceinline__ float warm_bound(LoadChunk load, int pos0, int64_t m, int k, float E) {
    constexpr int GW = COLS / NG;  // group width
    float g[NG];
#pragma unroll
    for (int c0 = 0; c0 < COLS; c0 += 32) {
        float v[32];
        load(c0, v);
#pragma unroll
        for (int q = 0; q < 32 / GW; ++q) {
            float x = -INFINITY;
#pragma unroll
            for (int j = 0; j < GW; ++j)
                if (pos0 + c0 + q * GW + j < m) x = fmaxf(x, v[q * GW + j]);
            g[(c0 / GW) + q] = x;
        }
    }
    sort_desc<NG, 2>(g);
    float kth = -INFINITY;
#pragma unroll
    for (int j = 0; j < NG; ++j)
        if (j == k - 1) kth = g[j];
    return (kth == -INFINITY) ? -INFINITY : __fsub_rd(kth, E);
}

}  // namespace rkm
