// Exact rescoring: K3 (exact tau_u, t_u and S_k(u) from the candidate lists, Definition 1),
// K6 (exact membership of the counting pass's band pairs, Eq. 1) and K8 (scores as the
// histogram of S_k(u), the first Section 2.2 baseline).
//
// Exact inner products.  When every row is on the grid 2^e * q / 4096, u.p equals
// 2^(e_u + e_p - 24) * sum_j q_u[j] q_p[j], an integer sum scaled exactly into FP64.
// Otherwise u.p is the left-to-right FP64 sum of the exact FP64 products of the FP32 inputs.
//
// Both kernels gather one row per candidate (or two per pair) and are bound by the latency of
// those gathers and by issue slots, so rows are read by groups of eight lanes, 128 contiguous
// bytes at a time, and the eight lanes' partial sums of eight rows are folded together (7
// exchanges for 32 rows).  FP64 runs at 2 lanes per SM and clock on sm_103, so off the grid no
// candidate is summed in FP64 to be ranked: an FP32 sum with a proven error bound ranks it, FP64
// decides only between candidates whose FP32 sums are too close, and the FP64 value of tau_u
// itself is formed for up to 32 users at a time, one per lane.  Against one lane per candidate
// and a ranking of all of them by shuffles, measured on GB300:
//   K3, grid      500K users x 100K items, d = 64,  k = 25         1.87 -> 0.76 ms
//   K3, grid      2M x 500K,               d = 128, k = 10         4.11 -> 2.4 ms
//   K3, FP8 band  100K x 50K,              d = 128, k = 10         4.77 -> 0.90 ms
//   K3, off grid  480K x 17.8K,            d = 200, k = 10         32.0 -> 1.58 ms
//   K3, off grid  130K x 30K,              d = 100, k = 50, lists  11.0 -> 1.29 ms
//   K6, off grid  2.2M pairs, d = 200: 2.39 -> 0.93 ms;  grid, 8.1M pairs, d = 128: 2.1 -> 1.1 ms
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.h"

namespace rkm {

namespace {

constexpr int EX_WARPS = 4;             // warps per block of K3
constexpr int BAND_WARPS = 4;           // and of K6
constexpr int EX_CHUNK = 192;           // candidates a warp collects before it scores them
constexpr int EX_ENTRIES = EX_CHUNK + KMAX;  // and the best k of the chunks before

// FP32 -> FP64 by bit arithmetic (the conversion instruction shares the slow FP64 pipe); zero,
// subnormal, infinite and NaN values take the instruction.
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), mag = b & 0x7fffffffu;
    if (mag - 0x00800000u >= 0x7f000000u) return (double)x;
    return __hiloint2double((int)((b & 0x80000000u) | ((mag >> 3) + 0x38000000u)), (int)(b << 29));
}

// Columns c .. c+3 of an FP32 row (zero at and beyond d); `vec`: rows_aligned.
__device__ __forceinline__ float4 load4(const float* __restrict__ row, int c, int d, bool vec) {
    if (vec) return c < d ? *reinterpret_cast<const float4*>(row + c) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 v;
    v.x = (c < d) ? row[c] : 0.f;
    v.y = (c + 1 < d) ? row[c + 1] : 0.f;
    v.z = (c + 2 < d) ? row[c + 2] : 0.f;
    v.w = (c + 3 < d) ? row[c + 3] : 0.f;
    return v;
}

// Rows that are whole 16-byte pieces on 16-byte boundaries.
__device__ __forceinline__ bool rows_aligned(const float* X, int64_t ld, int d) {
    return ((reinterpret_cast<uintptr_t>(X) & 15u) == 0u) && ((ld & 3) == 0) && ((d & 3) == 0);
}

// Left-to-right FP64 sum of one (user, item) pair by a lane; the lanes of a warp form 32 at once,
// and the FP64 chain is what this costs.  Columns past d are zero in both rows and change nothing.
__device__ __forceinline__ double dot_f64(const ExactData& x, int64_t u, int64_t i, bool vec_u, bool vec_p) {
    const float* a = x.U + u * x.ldu;
    const float* b = x.P + i * x.ldp;
    double s = 0.0;
#pragma unroll 2
    for (int c = 0; c < x.d; c += 4) {
        const float4 p = load4(a, c, x.d, vec_u), q = load4(b, c, x.d, vec_p);
        s = fma(widen(p.x), widen(q.x), s);
        s = fma(widen(p.y), widen(q.y), s);
        s = fma(widen(p.z), widen(q.z), s);
        s = fma(widen(p.w), widen(q.w), s);
    }
    return s + 0.0;  // -0.0 -> +0.0
}

__device__ __forceinline__ double key_to_double(unsigned long long k) {
    unsigned long long b = (k & 0x8000000000000000ull) ? (k ^ 0x8000000000000000ull) : ~k;
    return __longlong_as_double((long long)b);
}

// double_key of acc * 2^t in integer arithmetic (|acc| <= 2^33; the exponents of FP32 rows keep
// the value a normal double).
__device__ __forceinline__ unsigned long long grid_key(long long acc, int t) {
    if (acc == 0) return 0x8000000000000000ull;
    const unsigned long long m = (unsigned long long)(acc < 0 ? -acc : acc);
    const int lz = __clzll((long long)m);
    const unsigned long long bits =
        ((unsigned long long)(1023 + 63 - lz + t) << 52) + ((m << (lz - 11)) & 0xfffffffffffffull);
    return acc < 0 ? ~(bits | 0x8000000000000000ull) : (bits | 0x8000000000000000ull);
}

// FP32 round-to-nearest of acc * 2^t (a monotone function of it; may underflow or overflow).
__device__ __forceinline__ float grid_float(long long acc, int t) {
    const float f = fmaf((float)(int)(acc >> 10), 1024.f, (float)((int)acc & 1023));
    return (t >= -100 && t <= 100) ? f * __int_as_float((t + 127) << 23) : ldexpf(f, t);
}

// Sums over the eight lanes of a group: a[j] is this lane's part of row j; lane `sub` of the
// group returns the whole of row sub.  Integer parts are at most 2^29 in magnitude (32
// products of grid codes), so the first stage stays in 32 bits.
__device__ __forceinline__ long long fold8(const int (&a)[8], int lane) {
    const bool h4 = lane & 4, h2 = lane & 2, h1 = lane & 1;
    int r[4];
    long long q[2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        r[i] = (h4 ? a[i + 4] : a[i]) + __shfl_xor_sync(0xffffffffu, h4 ? a[i] : a[i + 4], 4);
#pragma unroll
    for (int i = 0; i < 2; ++i)
        q[i] = (long long)(h2 ? r[i + 2] : r[i]) + __shfl_xor_sync(0xffffffffu, h2 ? r[i] : r[i + 2], 2);
    return (h1 ? q[1] : q[0]) + __shfl_xor_sync(0xffffffffu, h1 ? q[0] : q[1], 1);
}

__device__ __forceinline__ float fold8(const float (&a)[8], int lane) {
    const bool h4 = lane & 4, h2 = lane & 2, h1 = lane & 1;
    float r[4], q[2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        r[i] = (h4 ? a[i + 4] : a[i]) + __shfl_xor_sync(0xffffffffu, h4 ? a[i] : a[i + 4], 4);
#pragma unroll
    for (int i = 0; i < 2; ++i)
        q[i] = (h2 ? r[i + 2] : r[i]) + __shfl_xor_sync(0xffffffffu, h2 ? r[i] : r[i + 2], 2);
    return (h1 ? q[1] : q[0]) + __shfl_xor_sync(0xffffffffu, h1 ? q[0] : q[1], 1);
}

__device__ __forceinline__ void fma4(float4& s, const float4& a, const float4& b) {
    s.x = fmaf(a.x, b.x, s.x);
    s.y = fmaf(a.y, b.y, s.y);
    s.z = fmaf(a.z, b.z, s.z);
    s.w = fmaf(a.w, b.w, s.w);
}

// Bound of |w - u.p| for the FP32 sums below: each of a lane's four chains is at most eight
// FMAs (d <= 256 over eight lanes of four columns), joined by two additions and three folds, so
// the error is at most gamma_13 sum|u p| <= gamma_13 ||u|| ||p|| (Higham, "Accuracy and Stability
// of Numerical Algorithms", Section 3.1); 2^-20 = 16 * 2^-24 also covers the rounding of the FP64
// reference sum, and 2^-140 underflow.  Item norms are bounded by the end of the bucket of the first
// item tile's largest: the order inside a bucket is free, and subnormal norms share buckets that are
// wide for their size (all below 2^-133 one), so no factor of that largest norm would do.
__device__ __forceinline__ float f32_bound(const ExactData& x, int64_t u) {
    const float pn = bucket_end(*x.pmax);
    return __fmaf_ru(__fmul_ru(x.unrm[u], 0x1p-20f), pn, 0x1p-140f);
}

// Working set of one warp.
struct ExactWarp {
    unsigned long long key[EX_ENTRIES];  // exact keys (off the grid: of the entries that need one)
    float w[EX_ENTRIES];                 // FP32 score: rounded exact (grid) or with error bound
    int id[EX_ENTRIES];                  // original item id
    uint8_t rank[EX_ENTRIES];            // rank of the entries that exact_ranks ordered
    union {
        int4 codes[32];  // user row: per 8 codes q = 128 h + l the bytes h (two words), l (two words)
        float f[256];    // user row, zero padded
    } row;
    int kth;         // t_u (off the grid)
    unsigned more;   // best_of_many: candidates scored
    int bad;         // best_of_many: some score was not finite
};
static_assert(EX_CHUNK % 32 == 0 && EX_CHUNK - 32 >= 2 * KMAX, "a full chunk holds 2k candidates");
static_assert(EX_ENTRIES <= 256, "ranks are bytes");

// Bytes h_j = q_j >> 7 (in [-32, 32]) and l_j = q_j & 127 of four codes, so that a 16 x 8 bit
// dot product (dp2a) takes item codes as they are stored.
__device__ __forceinline__ void split_codes(int q01, int q23, int& h, int& l) {
    const int a = (int)(int16_t)q01, b = q01 >> 16, c = (int)(int16_t)q23, d = q23 >> 16;
    h = ((a >> 7) & 255) | (((b >> 7) & 255) << 8) | (((c >> 7) & 255) << 16) | (int)((unsigned)(d >> 7) << 24);
    l = (a & 127) | ((b & 127) << 8) | ((c & 127) << 16) | ((d & 127) << 24);
}

// Scores of entries [n0, n) of S against the warp's user row on the grid: writes S.w and the
// integer sums to S.key (KEYS: their exact keys).
template <bool KEYS>
__device__ __forceinline__ void score_grid(const ExactData& x, ExactWarp& S, int n0, int n, int eu, int lane) {
    const int sub = lane & 7, grp = lane >> 3, vecs = x.dq >> 3;
    for (int b0 = n0; b0 < n; b0 += 32) {
        int a[8];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            int hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
            if (b0 + half * 16 < n) {
                const int4* p[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int c = b0 + (half * 4 + t) * 4 + grp;
                    p[t] = reinterpret_cast<const int4*>(x.qp + (int64_t)S.id[c < n ? c : n - 1] * x.dq);
                }
                for (int v = sub; v < vecs; v += 8) {
                    int4 q[4];
#pragma unroll
                    for (int t = 0; t < 4; ++t) q[t] = p[t][v];
                    const int4 r = S.row.codes[v];
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        hi[t] = __dp2a_hi(q[t].y, r.x, __dp2a_lo(q[t].x, r.x, hi[t]));
                        hi[t] = __dp2a_hi(q[t].w, r.y, __dp2a_lo(q[t].z, r.y, hi[t]));
                        lo[t] = __dp2a_hi(q[t].y, r.z, __dp2a_lo(q[t].x, r.z, lo[t]));
                        lo[t] = __dp2a_hi(q[t].w, r.w, __dp2a_lo(q[t].z, r.w, lo[t]));
                    }
                }
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) a[half * 4 + t] = 128 * hi[t] + lo[t];
        }
        __syncwarp();
        const long long acc = fold8(a, lane);
        const int c = b0 + sub * 4 + grp;
        if (c < n) {
            const int t = eu + x.ep[S.id[c]] - 24;
            S.key[c] = KEYS ? grid_key(acc, t) : (unsigned long long)acc;
            S.w[c] = grid_float(acc, t);
        }
    }
    __syncwarp();
}

// The same in FP32 (error at most f32_bound); returns true when some score is not finite.
template <bool VEC>
__device__ __forceinline__ bool score_f32(const ExactData& x, ExactWarp& S, int n0, int n, int lane) {
    const int sub = lane & 7, grp = lane >> 3;
    bool bad = false;
    for (int b0 = n0; b0 < n; b0 += 32) {
        float a[8];
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            float4 s[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) s[t] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (b0 + half * 16 < n) {
                const float* p[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int c = b0 + (half * 4 + t) * 4 + grp;
                    p[t] = x.P + (int64_t)S.id[c < n ? c : n - 1] * x.ldp;
                }
                for (int c0 = sub * 4; c0 < x.d; c0 += 32) {
                    float4 q[4];
#pragma unroll
                    for (int t = 0; t < 4; ++t) q[t] = load4(p[t], c0, x.d, VEC);
                    const float4 r = *reinterpret_cast<const float4*>(&S.row.f[c0]);
#pragma unroll
                    for (int t = 0; t < 4; ++t) fma4(s[t], r, q[t]);
                }
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) a[half * 4 + t] = (s[t].x + s[t].y) + (s[t].z + s[t].w);
        }
        __syncwarp();
        const float w = fold8(a, lane);
        const int c = b0 + sub * 4 + grp;
        if (c < n) {
            S.w[c] = w;
            bad |= !(fabsf(w) < INFINITY);
        }
    }
    __syncwarp();
    return __any_sync(0xffffffffu, bad);
}

// Values v[r * 32 + lane] (R registers per lane) sorted in descending order by a bitonic network.
template <int R>
__device__ __forceinline__ void sort_desc(float (&v)[R], int lane) {
#pragma unroll
    for (int size = 2; size <= 32 * R; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride >= 32) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int o = r ^ (stride >> 5);
                    if (o > r) {
                        const bool desc = ((r * 32) & size) == 0;
                        const float hi = fmaxf(v[r], v[o]), lo = fminf(v[r], v[o]);
                        v[r] = desc ? hi : lo;
                        v[o] = desc ? lo : hi;
                    }
                }
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float o = __shfl_xor_sync(0xffffffffu, v[r], stride);
                    const bool desc = size >= 32 ? ((r * 32) & size) == 0 : (lane & size) == 0;
                    v[r] = desc == ((lane & stride) == 0) ? fmaxf(v[r], o) : fminf(v[r], o);
                }
            }
        }
    }
}

// The k-th largest of the scores S.w[0 .. n), 1 <= k <= n.  Up to 64 are sorted in registers (15
// or 21 exchanges; half the time of counting by ballot, measured at 24 and 47 scores); for more,
// a bisection counts them by ballot in a short loop (a network of 128 overran the instruction
// cache: 2.0 against 1.5 ms at 130K users with 90 scores each).
__device__ __forceinline__ float kth_score(const ExactWarp& S, int n, int k, int lane) {
    if (n <= 32) {
        float v[1] = {lane < n ? S.w[lane] : -INFINITY};
        sort_desc(v, lane);
        return __shfl_sync(0xffffffffu, v[0], k - 1);
    }
    if (n <= 64) {
        float v[2] = {S.w[lane], 32 + lane < n ? S.w[32 + lane] : -INFINITY};
        sort_desc(v, lane);
        return __shfl_sync(0xffffffffu, k > 32 ? v[1] : v[0], (k - 1) & 31);
    }
    unsigned mn = 0xffffffffu, mx = 0u;
    for (int j = lane; j < n; j += 32) {
        const unsigned b = float_key(S.w[j]);
        mn = min(mn, b);
        mx = max(mx, b);
    }
    // At least k scores reach lo, fewer than k reach hi.
    unsigned lo = __reduce_min_sync(0xffffffffu, mn), hi = __reduce_max_sync(0xffffffffu, mx) + 1u;
    while (hi - lo > 1u) {
        const unsigned mid = lo + ((hi - lo) >> 1);
        const float T = key_float(mid);
        int c = 0;
        for (int j = 0; j < n; j += 32) c += __popc(__ballot_sync(0xffffffffu, j + lane < n && S.w[j + lane] >= T));
        if (c < k) {
            hi = mid;
        } else {
            lo = mid;
            if (c == k) break;
        }
    }
    // The smallest score that reaches lo (lo itself when the bisection ran out on a tie).
    const float T = key_float(lo);
    mn = 0xffffffffu;
    for (int j = lane; j < n; j += 32)
        if (S.w[j] >= T) mn = min(mn, float_key(S.w[j]));
    return key_float(__reduce_min_sync(0xffffffffu, mn));
}

// Moves the entries of [0, n) whose score reaches `cut` to the front; returns how many.
__device__ __forceinline__ int keep_from(ExactWarp& S, bool keys, int n, float cut, int lane) {
    const unsigned lt_mask = (1u << lane) - 1u;
    int out = 0;
    for (int j0 = 0; j0 < n; j0 += 32) {
        const int j = j0 + lane;
        const float w = j < n ? S.w[j] : 0.f;
        const int id = j < n ? S.id[j] : 0;
        unsigned long long key = 0ull;
        if (keys && j < n) key = S.key[j];
        const bool take = j < n && w >= cut;
        const unsigned mask = __ballot_sync(0xffffffffu, take);
        // Every lane has read its entry (the ballot orders it before the writes), and writes
        // go to slots at or before the ones read in this round.
        if (take) {
            const int slot = out + __popc(mask & lt_mask);
            S.w[slot] = w;
            S.id[slot] = id;
            if (keys) S.key[slot] = key;
        }
        out += __popc(mask);
        __syncwarp();
    }
    return out;
}

// Entries of [0, n) surely before one of score wa (gt), and surely or possibly before it (ge,
// itself included): scores more than tol apart decide.
__device__ __forceinline__ void rank_bounds(const ExactWarp& S, int n, float wa, float tol, int& gt, int& ge) {
    const float hi = __fadd_ru(wa, tol), lo = __fsub_rd(wa, tol);
    const float4* w4 = reinterpret_cast<const float4*>(S.w);
    gt = 0;
    ge = 0;
    for (int b = 0; b < n; b += 4) {
        const float4 v = w4[b >> 2];
        gt += (v.x > hi) + (v.y > hi) + (v.z > hi) + (v.w > hi);
        ge += (v.x >= lo) + (v.y >= lo) + (v.z >= lo) + (v.w >= lo);
    }
}

__device__ __forceinline__ void pad_scores(ExactWarp& S, int n, int lane) {
    if (lane < ((4 - (n & 3)) & 3)) S.w[n + lane] = -INFINITY;  // rank_bounds reads four at a time
    __syncwarp();
}

// Exact rank of every entry of [0, n) under (score desc, id asc), into S.rank: entries within tol
// of each other are ordered by their exact keys, which off the grid are computed here for the
// entries that need them (tol covers both errors; the test that picks them is an eighth wider
// than the other, more than its rounding, so both entries of every close pair have their key).
// The user's row is in S.row.  S.w is padded.
__device__ __forceinline__ void exact_ranks(const ExactData& x, ExactWarp& S, bool grid, bool vec, int n, float tol,
                                         int lane) {
    for (int a = lane; a < n; a += 32) {
        int gt, ge;
        rank_bounds(S, n, S.w[a], 1.125f * tol, gt, ge);
        const bool alone = ge - gt == 1;
        S.rank[a] = (uint8_t)(alone ? gt : 255);
        if (!grid && !alone) {
            // Left-to-right FP64 sum; columns past d are zero in both rows and change nothing.
            const float* row = x.P + (int64_t)S.id[a] * x.ldp;
            double s = 0.0;
#pragma unroll 2
            for (int c = 0; c < x.d; c += 4) {
                const float4 q = load4(row, c, x.d, vec), r = *reinterpret_cast<const float4*>(&S.row.f[c]);
                s = fma(widen(r.x), widen(q.x), s);
                s = fma(widen(r.y), widen(q.y), s);
                s = fma(widen(r.z), widen(q.z), s);
                s = fma(widen(r.w), widen(q.w), s);
            }
            S.key[a] = double_key(s + 0.0);
        }
    }
    __syncwarp();
    for (int a = lane; a < n; a += 32) {
        if (S.rank[a] != 255) continue;
        const float wa = S.w[a], hi = __fadd_ru(wa, tol), lo = __fsub_rd(wa, tol);
        const unsigned long long ka = S.key[a];
        const int ia = S.id[a];
        int rank = 0;
        for (int b = 0; b < n; ++b) {
            const float wb = S.w[b];
            if (wb > hi) {
                ++rank;
            } else if (b != a && wb >= lo) {
                const unsigned long long kb = S.key[b];
                rank += kb > ka || (kb == ka && S.id[b] < ia);
            }
        }
        S.rank[a] = (uint8_t)rank;
    }
    __syncwarp();
}

// Cuts the n > k entries that FP32 left to exactly the k best (order not kept).
__device__ __forceinline__ void cut_exactly(const ExactData& x, ExactWarp& S, bool grid, bool vec, int n, int k,
                                         float tol, int lane) {
    exact_ranks(x, S, grid, vec, n, tol, lane);
    int out = 0;
    for (int j0 = 0; j0 < n; j0 += 32) {
        const int j = j0 + lane;
        const bool take = j < n && S.rank[j] < k;
        const float w = j < n ? S.w[j] : 0.f;
        const int id = j < n ? S.id[j] : 0;
        const unsigned long long key = j < n ? S.key[j] : 0ull;
        const unsigned mask = __ballot_sync(0xffffffffu, take);
        if (take) {
            const int slot = out + __popc(mask & ((1u << lane) - 1u));
            S.w[slot] = w;
            S.id[slot] = id;
            S.key[slot] = key;
        }
        out += __popc(mask);
        __syncwarp();
    }
}

// The users' candidate lists (nseg segments of cap slots each).
struct CandLists {
    const Cand* cand;
    const int* cand_cnt;
    const unsigned* lfin_key;
    int cap, nseg;
    const int* item_perm;
};

// A threshold on the upper bounds that k to `most` candidates of list row u reach, by bisection
// over their keys between L and the largest; +inf when ties leave none.
__device__ __forceinline__ float bound_threshold(const CandLists& l, int64_t u, float L, int k, int most, int lane) {
    const Cand* list = l.cand + u * (int64_t)l.nseg * l.cap;
    unsigned lo = float_key(L), hi = 0u;
    for (bool first = true;; first = false) {
        const unsigned T = first ? 0u : lo + ((hi - lo) >> 1);
        int c = 0;
        unsigned mx = 0u;
        for (int s = 0; s < l.nseg; ++s) {
            const int cnt = l.cand_cnt[u * l.nseg + s];
#pragma unroll 4
            for (int j = lane; j < cnt; j += 32) {
                const unsigned b = float_key(list[s * (int64_t)l.cap + j].ub);
                c += b >= T;
                mx = b > mx ? b : mx;
            }
        }
        if (first) {
            hi = __reduce_max_sync(0xffffffffu, mx);
        } else {
            c = __reduce_add_sync(0xffffffffu, c);
            if (c < k) hi = T;
            else if (c > most) lo = T;
            else return key_float(T);
        }
        if (hi <= lo || hi - lo == 1u) return INFINITY;
    }
}

// Appends to S.id[n ..) the ids of the candidates of list row u with lo <= ub < hi (hi = inf: no
// limit), 32 at a time from (seg, base) on, until the lists are exhausted (seg >= nseg) or the
// count passes `full`; returns the count.  Two segments are read as one list, and 128 entries and
// then their ids are in flight at once (the two dependent reads are what this waits for).
__device__ __forceinline__ int collect(const ExactData& x, const CandLists& l, ExactWarp& S, int64_t u, float lo,
                                       float hi, int n, int full, int& seg, int& base, int lane, DevStatus* st) {
    const unsigned lt_mask = (1u << lane) - 1u;
    while (seg < l.nseg) {
        const int c0 = l.cand_cnt[u * l.nseg + seg];
        const int total = c0 + (seg + 1 < l.nseg ? l.cand_cnt[u * l.nseg + seg + 1] : 0);
        const Cand* c = l.cand + (u * l.nseg + seg) * (int64_t)l.cap;
        for (; base < total; base += 128) {
            Cand r[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int j = base + t * 32 + lane;
                r[t].ub = -INFINITY;
                r[t].pos = -1;
                if (j < total) r[t] = c[j < c0 ? j : j - c0 + l.cap];
            }
            int io[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                bool keep = r[t].ub >= lo && (r[t].ub < hi || hi == INFINITY) && base + t * 32 + lane < total;
                keep = keep && RKM_DCHECK(r[t].pos >= 0 && (x.m_items == 0 || r[t].pos < x.m_items), st);
                io[t] = keep ? l.item_perm[r[t].pos] : -1;
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                if (base + t * 32 >= total) break;
                if (n > full) {
                    base += t * 32;
                    return n;
                }
                const unsigned mask = __ballot_sync(0xffffffffu, io[t] >= 0);
                if (mask == 0u) continue;
                if (io[t] >= 0) S.id[n + __popc(mask & lt_mask)] = io[t];
                n += __popc(mask);
            }
        }
        seg += 2;
        base = 0;
    }
    return n;
}

// The k best of a user with more than a chunk of candidates (a wide guard band, as on the FP8
// path), at the front of S with exact keys on the grid; returns how many are left (k, or more
// where FP32 cannot tell the last ones).  The candidates with the k to 2k largest upper bounds
// are scored first: their k-th score bounds tau_u far better than L, and only the others whose
// upper bound reaches it are scored at all (546 candidates per user became 99 at 100K x 50K,
// d = 128, k = 10, FP8).
__device__ __forceinline__ int best_of_many(const ExactData& x, bool grid, const CandLists& l, ExactWarp& S, int k,
                                         DevStatus* st, int64_t u, bool vec, int lane, float L, int eu,
                                         float err) {
    bool bad = !(err < INFINITY);
    unsigned scored = 0;
    float T = bound_threshold(l, u, L, k, 2 * k > 48 ? 2 * k : 48, lane);
    int seg = 0, base = 0, n0 = 0;
    int n = collect(x, l, S, u, T < INFINITY ? T : L, INFINITY, 0, EX_CHUNK - 32, seg, base, lane, st);
    if (T < INFINITY) {  // the rest follow from the start of the lists
        seg = 0;
        base = 0;
    }
    for (;;) {
        __syncwarp();
        scored += (unsigned)(n - n0);
        if (grid) {
            score_grid<true>(x, S, n0, n, eu, lane);
        } else {
            bad |= vec ? score_f32<true>(x, S, n0, n, lane) : score_f32<false>(x, S, n0, n, lane);
            if (bad)
                for (int j = lane; j < n; j += 32) S.w[j] = 0.f;
            __syncwarp();
        }
        const float tol = grid ? 0.f : bad ? INFINITY : 2.f * err;
        const float wk = kth_score(S, n, k, lane);
        n0 = keep_from(S, true, n, __fsub_rd(wk, tol), lane);
        if (seg >= l.nseg) break;
        if (n0 > k) {
            pad_scores(S, n0, lane);
            cut_exactly(x, S, grid, vec, n0, k, tol, lane);
            n0 = k;
        }
        // k items reach the k-th score (less its error), so tau_u does.
        L = fmaxf(L, __fsub_rd(wk, grid ? __fmaf_ru(fabsf(wk), 0x1p-23f, 0x1p-149f) : tol));
        n = collect(x, l, S, u, L, T, n0, n0 + EX_CHUNK - 32, seg, base, lane, st);
        if (n == n0) break;
    }
    if (lane == 0) {
        S.more = scored;
        S.bad = bad;
    }
    __syncwarp();
    return n0;
}

// Exact tau_u, t_u (and S_k(u) when topk != null) of the user of list row u; one warp per
// user, all 32 lanes call it.  On the grid tau is written here; otherwise t_u is returned (by
// every lane) for the FP64 sum that the caller forms for many users at once, or -1.
// Candidates whose upper bound is below the final lower bound L of tau_u are dropped.
__device__ __forceinline__ int exact_user(const ExactData& x, bool grid, const CandLists& l, ExactWarp& S, int k,
                                          double* __restrict__ tau, int* __restrict__ tid, int* __restrict__ topk,
                                          DevStatus* st, int64_t u, int64_t uo, bool vec, int lane,
                                          unsigned& scored) {
    const float L = key_float(l.lfin_key[u]);
    // user row
    __syncwarp();
    int eu = 0;
    float err = 0.f;
    if (grid) {
        eu = x.eu[uo];
        if (lane < (x.dq >> 3)) {
            const int4 q = reinterpret_cast<const int4*>(x.qu + uo * x.dq)[lane];
            int4 r;
            split_codes(q.x, q.y, r.x, r.z);
            split_codes(q.z, q.w, r.y, r.w);
            S.row.codes[lane] = r;
        }
    } else {
        const float* a = x.U + uo * x.ldu;
#pragma unroll
        for (int j = 0; j < 256; j += 32)
            if (j < x.d) S.row.f[j + lane] = (j + lane < x.d) ? a[j + lane] : 0.f;
        err = f32_bound(x, uo);
    }
    // Off the grid, a score or bound that is not finite orders nothing: the scores are then all
    // set equal and the exact keys decide.
    bool bad = !(err < INFINITY), keyed = false;
    int seg = 0, base = 0;
    int n = collect(x, l, S, u, L, INFINITY, 0, EX_CHUNK - 32, seg, base, lane, st);
    if (seg < l.nseg) {
        n = best_of_many(x, grid, l, S, k, st, u, vec, lane, L, eu, err);
        scored += S.more;
        bad = S.bad != 0;
        keyed = grid;
    } else {
        if (n < k) {
            if (lane == 0) st->internal_error = 1u;
            return -1;
        }
        __syncwarp();
        scored += (unsigned)n;
        if (grid) {
            score_grid<false>(x, S, 0, n, eu, lane);
        } else {
            bad |= vec ? score_f32<true>(x, S, 0, n, lane) : score_f32<false>(x, S, 0, n, lane);
            if (bad)
                for (int j = lane; j < n; j += 32) S.w[j] = 0.f;
            __syncwarp();
        }
    }
    const float tol = grid ? 0.f : bad ? INFINITY : 2.f * err;
    auto emit = [&](int rank, int a) {
        const int id = S.id[a];
        if (topk) topk[uo * (int64_t)k + rank] = id;
        if (rank == k - 1) {
            tid[uo] = id;
            if (!grid) S.kth = id;
            else tau[uo] = key_to_double(keyed ? S.key[a] : grid_key((long long)S.key[a], eu + x.ep[id] - 24));
        }
    };
    const float wk = kth_score(S, n, k, lane), cut = __fsub_rd(wk, tol);
    bool close = false;
    if (topk) {
        n = keep_from(S, grid, n, cut, lane);  // the k best, and those too close to tell
        pad_scores(S, n, lane);
        for (int a = lane; a < n; a += 32) {
            int gt, ge;
            rank_bounds(S, n, S.w[a], tol, gt, ge);
            if (ge - gt != 1) close = true;
            else if (gt < k) emit(gt, a);
        }
        close = __any_sync(0xffffffffu, close);
    } else {
        // t_u alone: the entry within tol of the k-th largest score, if there is only one.
        const float up = __fadd_ru(wk, tol);
        int near = 0, at = -1;
        for (int j = 0; j < n; j += 32) {
            const float w = j + lane < n ? S.w[j + lane] : 0.f;
            const bool here = j + lane < n && w >= cut && w <= up;
            near += __popc(__ballot_sync(0xffffffffu, here));
            if (here) at = j + lane;
        }
        close = near > 1;
        if (!close && at >= 0) emit(k - 1, at);
    }
    if (close) {
        if (grid && !keyed) {
            for (int a = lane; a < n; a += 32)
                S.key[a] = grid_key((long long)S.key[a], eu + x.ep[S.id[a]] - 24);
            __syncwarp();
            keyed = true;
        }
        pad_scores(S, n, lane);
        exact_ranks(x, S, grid, vec, n, tol, lane);
        for (int a = lane; a < n; a += 32) {
            const int rank = S.rank[a];
            if (topk ? rank < k : rank == k - 1) emit(rank, a);
        }
    }
    __syncwarp();
    return S.kth;
}

// K3.  A warp takes `per` list rows in turn, one user at a time; off the grid the FP64 values of
// their thresholds are then formed together, one user per lane.  Eight blocks of four warps per SM
// (64 registers, some spilled) beat seven and nine over the four measured forms; functions
// called out of line cost more (1.0 against 0.84 ms at 500K x 100K) than they save in instruction
// cache.
__global__ void __launch_bounds__(32 * EX_WARPS, 8)
    k_exact_tau(const __grid_constant__ ExactData x, const CandLists l, int64_t n, int k, int per, double* __restrict__ tau,
                int* __restrict__ tid, int* __restrict__ topk, DevStatus* st, const int* __restrict__ uperm) {
    __shared__ __align__(16) ExactWarp work[EX_WARPS];
    const int lane = threadIdx.x & 31;
    ExactWarp& S = work[threadIdx.x >> 5];
    const bool grid = *x.off_grid == 0u;
    const bool vec = rows_aligned(x.P, x.ldp, x.d), vec_u = rows_aligned(x.U, x.ldu, x.d);
    const int64_t warps = (int64_t)gridDim.x * EX_WARPS;
    unsigned scored = 0;
    for (int64_t u0 = ((int64_t)blockIdx.x * EX_WARPS + (threadIdx.x >> 5)) * per; u0 < n; u0 += warps * per) {
        int my_u = -1, my_i = -1;
        for (int j = 0; j < per && u0 + j < n; ++j) {
            const int64_t u = u0 + j;
            const int64_t uo = uperm ? (int64_t)uperm[u] : u;  // row of the lists -> original user
            if (!RKM_DCHECK(uo >= 0 && (x.n_users == 0 || uo < x.n_users), st)) continue;
            const int i = exact_user(x, grid, l, S, k, tau, tid, topk, st, u, uo, vec, lane, scored);
            if (lane == j && i >= 0) {
                my_u = (int)uo;
                my_i = i;
            }
        }
        if (!grid && my_u >= 0) tau[my_u] = dot_f64(x, my_u, my_i, vec_u, vec);
    }
    if (lane == 0 && scored) atomicAdd(&st->cand_total, (unsigned long long)scored);
}

// The same over the users of many problems: global user g belongs to the last job whose
// user_begin is <= g.  A warp's users may span problems; its pending FP64 sums are formed when
// the problem changes.
__global__ void __launch_bounds__(32 * EX_WARPS, 8)
    k_exact_tau_multi(const BatchJob* __restrict__ jobs, int count, int64_t total_users, int per) {
    __shared__ __align__(16) ExactWarp work[EX_WARPS];
    const int lane = threadIdx.x & 31;
    ExactWarp& S = work[threadIdx.x >> 5];
    const int64_t warps = (int64_t)gridDim.x * EX_WARPS;
    for (int64_t g0 = ((int64_t)blockIdx.x * EX_WARPS + (threadIdx.x >> 5)) * per; g0 < total_users;
         g0 += warps * per) {
        const int64_t g1 = (g0 + per < total_users) ? g0 + per : total_users;
        for (int64_t g = g0; g < g1;) {
            int lo = 0, hi = count;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (jobs[mid].user_begin <= g) lo = mid; else hi = mid;
            }
            const BatchJob& J = jobs[lo];
            const int64_t end = (J.user_begin + J.n < g1) ? J.user_begin + J.n : g1;
            const bool grid = *J.x.off_grid == 0u;
            const bool vec = rows_aligned(J.x.P, J.x.ldp, J.x.d), vec_u = rows_aligned(J.x.U, J.x.ldu, J.x.d);
            const CandLists l{J.cand, J.cand_cnt, J.lfin, J.cap, J.nseg, J.item_perm};
            int my_u = -1, my_i = -1;
            unsigned scored = 0;
            for (int j = 0; g < end; ++g, ++j) {
                const int64_t u = g - J.user_begin;
                const int i = exact_user(J.x, grid, l, S, J.k, J.tau, J.tid, nullptr, J.st, u, u, vec, lane, scored);
                if (lane == j && i >= 0) {
                    my_u = (int)u;
                    my_i = i;
                }
            }
            if (!grid && my_u >= 0) J.tau[my_u] = dot_f64(J.x, my_u, my_i, vec_u, vec);
            if (lane == 0 && scored) atomicAdd(&J.st->cand_total, (unsigned long long)scored);
        }
    }
}

// K6.  The pairs of one warp that FP32 could not decide.  Kept small: a counting CTA leaves about
// 10 KB of shared memory and a quarter of the registers of its SM free, and the band pairs of
// one serving batch must fit there beside the counting pass of another (with 47 KB of staging
// per block the serving loop was 12 % slower).
struct BandWarp {
    int u[64], io[64], pos[64];
};

// Exact membership of band pairs [st->band_done, min(st->band_count, cap)), 32 to a warp,
// warp `first` of `stride`; members add one to their item's count.  On the grid the integer
// sums decide.  Otherwise an FP32 sum decides the pairs whose distance to tau_u exceeds its
// error bound, and the rest (the pairs of t_u itself among them) are collected until a warp has
// 32 for the FP64 sums.
__device__ __forceinline__ void band_pairs(const ExactData& x, const int2* __restrict__ band, unsigned band_cap,
                                           const int* __restrict__ item_perm, const double* __restrict__ tau,
                                           const int* __restrict__ tid, bool new_items, int* __restrict__ counts,
                                           const DevStatus* st, unsigned first, unsigned stride, BandWarp& S) {
    const int lane = threadIdx.x & 31, sub = lane & 7, grp = lane >> 3;
    const bool grid = *x.off_grid == 0u;
    const bool vec = rows_aligned(x.P, x.ldp, x.d) && rows_aligned(x.U, x.ldu, x.d);
    const int home = (lane & 3) * 8 + (lane >> 2);  // lane that holds the folded sum of pair `lane`
    const unsigned begin = st->band_done;
    unsigned end = st->band_count;
    if (end > band_cap) end = band_cap;
    int queued = 0;
    // FP64 decision of the queued pairs [q0, q0 + 32) (fewer at the end).
    auto decide = [&](int q0, int cnt) {
        __syncwarp();
        const bool mine = lane < cnt;
        const int u = mine ? S.u[q0 + lane] : -1, io = mine ? S.io[q0 + lane] : -1;
        const int pos = mine ? S.pos[q0 + lane] : 0;
        if (mine) {
            const double s = dot_f64(x, u, io, vec, vec), t = tau[u];
            if (s > t || (!new_items && s == t && io <= tid[u])) atomicAdd(&counts[pos], 1);
        }
    };
    for (uint64_t e0 = (uint64_t)begin + 32ull * first; e0 < end; e0 += 32ull * stride) {
        const int cnt = (end - e0 < 32u) ? (int)(end - e0) : 32;
        const bool mine = lane < cnt;
        const int2 b = mine ? band[e0 + lane] : make_int2(0, 0);
        bool ok = mine && RKM_DCHECK(b.x >= 0 && (x.n_users == 0 || b.x < x.n_users) && b.y >= 0 &&
                                         (x.m_items == 0 || b.y < x.m_items),
                                     const_cast<DevStatus*>(st));
        const int u = ok ? b.x : 0, io = ok ? item_perm[b.y] : 0;
        const double t = ok ? tau[u] : 0.0;
        if (grid) {
            const int tsc = ok ? x.eu[u] + x.ep[io] - 24 : 0;
            const int vecs = x.dq >> 3;
            int a[8];
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                int s[4] = {0, 0, 0, 0};
                const int4 *pu[4], *pi[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int src = (half * 4 + j) * 4 + grp;
                    const int ur = __shfl_sync(0xffffffffu, u, src), ir = __shfl_sync(0xffffffffu, io, src);
                    pu[j] = reinterpret_cast<const int4*>(x.qu + (int64_t)ur * x.dq);
                    pi[j] = reinterpret_cast<const int4*>(x.qp + (int64_t)ir * x.dq);
                }
                if (half * 16 < cnt) {
                    for (int v = sub; v < vecs; v += 8) {
                        int4 qa[4], qb[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            qa[j] = pu[j][v];
                            qb[j] = pi[j][v];
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int aw[4] = {qa[j].x, qa[j].y, qa[j].z, qa[j].w};
                            const int bw[4] = {qb[j].x, qb[j].y, qb[j].z, qb[j].w};
#pragma unroll
                            for (int h = 0; h < 4; ++h)
                                s[j] += (int)(int16_t)aw[h] * (int)(int16_t)bw[h] + (aw[h] >> 16) * (bw[h] >> 16);
                        }
                    }
                }
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 4; ++j) a[half * 4 + j] = s[j];
            }
            const long long acc = __shfl_sync(0xffffffffu, fold8(a, lane), home);
            if (ok) {
                const double s = key_to_double(grid_key(acc, tsc));
                if (s > t || (!new_items && s == t && io <= tid[u])) atomicAdd(&counts[b.y], 1);
            }
        } else {
            float a[8];
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                float4 s[4];
                const float *pu[4], *pi[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int src = (half * 4 + j) * 4 + grp;
                    const int ur = __shfl_sync(0xffffffffu, u, src), ir = __shfl_sync(0xffffffffu, io, src);
                    pu[j] = x.U + (int64_t)ur * x.ldu;
                    pi[j] = x.P + (int64_t)ir * x.ldp;
                    s[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
                if (half * 16 < cnt) {
                    for (int c0 = sub * 4; c0 < x.d; c0 += 32) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) fma4(s[j], load4(pu[j], c0, x.d, vec), load4(pi[j], c0, x.d, vec));
                    }
                }
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 4; ++j) a[half * 4 + j] = (s[j].x + s[j].y) + (s[j].z + s[j].w);
            }
            const float w = __shfl_sync(0xffffffffu, fold8(a, lane), home);
            bool open = false;
            if (ok) {
                const float err = f32_bound(x, u);
                const double lo = (double)__fsub_rd(w, err), hi = (double)__fadd_ru(w, err);
                if (!(fabsf(w) < INFINITY)) open = true;  // an FP32 overflow decides nothing
                else if (lo > t) atomicAdd(&counts[b.y], 1);
                else open = !(hi < t);
            }
            const unsigned mask = __ballot_sync(0xffffffffu, open);
            if (open) {
                const int slot = queued + __popc(mask & ((1u << lane) - 1u));
                S.u[slot] = u;
                S.io[slot] = io;
                S.pos[slot] = b.y;
            }
            queued += __popc(mask);
            if (queued >= 32) {
                queued -= 32;
                decide(queued, 32);
            }
        }
    }
    if (queued > 0) decide(0, queued);
}

__global__ void __launch_bounds__(32 * BAND_WARPS, 8)
    k_band_rescore(const __grid_constant__ ExactData x, const int2* __restrict__ band, unsigned band_cap,
                   const int* __restrict__ item_perm, const double* __restrict__ tau, const int* __restrict__ tid,
                   bool new_items, int* __restrict__ counts, const DevStatus* st) {
    __shared__ BandWarp work[BAND_WARPS];
    const int w = threadIdx.x >> 5;
    band_pairs(x, band, band_cap, item_perm, tau, tid, new_items, counts, st, blockIdx.x * BAND_WARPS + w,
               gridDim.x * BAND_WARPS, work[w]);
}

// Band rescoring of job blockIdx.y (catalogue items: ties at tau_u are decided by t_u).
__global__ void __launch_bounds__(32 * BAND_WARPS) k_band_rescore_multi(const BatchJob* __restrict__ jobs) {
    __shared__ BandWarp work[BAND_WARPS];
    const int w = threadIdx.x >> 5;
    const BatchJob& J = jobs[blockIdx.y];
    band_pairs(J.x, J.band, J.band_cap, J.item_perm, J.tau, J.tid, false, J.counts, J.st, blockIdx.x * BAND_WARPS + w,
               gridDim.x * BAND_WARPS, work[w]);
}

// Zero the counts of job blockIdx.y and its band counters.
__global__ void k_batch_reset(const BatchJob* __restrict__ jobs) {
    const BatchJob& J = jobs[blockIdx.y];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < J.m; i += (int64_t)gridDim.x * blockDim.x)
        J.counts[i] = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        J.st->band_count = 0u;
        J.st->band_done = 0u;
    }
}

__global__ void k_histogram(const int* __restrict__ topk, int64_t nk, int* __restrict__ scores) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < nk; j += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&scores[topk[j]], 1);
}

// Histogram of the first k ids of every row of lists [n][kmax] (S_k(u) is the first k
// entries of S_kmax(u) in order).  An id outside [0, m) flags an internal error.
__global__ void k_histogram_prefix(const int* __restrict__ lists, int64_t n, int kmax, int k, int64_t m,
                                   int* __restrict__ scores, DevStatus* st) {
    const int64_t total = n * k;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < total; j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = j / k;
        const int id = lists[u * kmax + (j - u * k)];
        if (id >= 0 && id < m) atomicAdd(&scores[id], 1);
        else st->internal_error = 1u;
    }
}

}  // namespace

void launch_histogram_prefix(const int* lists, int64_t n, int kmax, int k, int64_t m, int* scores, DevStatus* st,
                             cudaStream_t s) {
    if (n <= 0 || k <= 0) return;
    int64_t blocks = (n * k + 255) / 256;
    if (blocks > 65536) blocks = 65536;
    note_launch();
    k_histogram_prefix<<<(int)blocks, 256, 0, s>>>(lists, n, kmax, k, m, scores, st);
}

// Users per warp of K3: 32 fill the lanes of the FP64 sums; fewer when that would leave less
// than about two rounds of the 32 warps that an SM holds.
static int users_per_warp(int64_t n, int num_sms) {
    int per = 32;
    while (per > 1 && n < (int64_t)per * num_sms * 64) per >>= 1;
    return per;
}

static int exact_blocks(int64_t n, int per) {
    const int64_t blocks = (n + (int64_t)per * EX_WARPS - 1) / ((int64_t)per * EX_WARPS);
    return (int)(blocks > 65536 ? 65536 : blocks);
}

void launch_exact_tau(const ExactData& x, const Cand* cand, const int* cand_cnt, const unsigned* lfin_key,
                      int cap, int nseg, const int* item_perm, int64_t n, int k, double* tau, int* tid, int* topk,
                      DevStatus* st, int num_sms, cudaStream_t s, const int* uperm) {
    if (n <= 0) return;
    const int per = users_per_warp(n, num_sms);
    note_launch();
    k_exact_tau<<<exact_blocks(n, per), 32 * EX_WARPS, 0, s>>>(
        x, CandLists{cand, cand_cnt, lfin_key, cap, nseg, item_perm}, n, k, per, tau, tid, topk, st, uperm);
}

void launch_band_rescore(const ExactData& x, const int2* band, unsigned band_cap, const int* item_perm,
                         const double* tau, const int* tid, bool new_items, int* counts,
                         DevStatus* st, int num_sms, cudaStream_t s) {
    note_launch();
    k_band_rescore<<<8 * num_sms, 32 * BAND_WARPS, 0, s>>>(x, band, band_cap, item_perm, tau, tid, new_items, counts, st);
}

void launch_exact_tau_multi(const BatchJob* jobs, int count, int64_t total_users, int num_sms, cudaStream_t s) {
    if (total_users <= 0) return;
    const int per = users_per_warp(total_users, num_sms);
    note_launch();
    k_exact_tau_multi<<<exact_blocks(total_users, per), 32 * EX_WARPS, 0, s>>>(jobs, count, total_users, per);
}

void launch_band_multi(const BatchJob* jobs, int count, cudaStream_t s) {
    note_launch();
    k_band_rescore_multi<<<dim3(128, (unsigned)count), 32 * BAND_WARPS, 0, s>>>(jobs);
}

void launch_batch_reset(const BatchJob* jobs, int count, int64_t max_m, cudaStream_t s) {
    int64_t bx = (max_m + 255) / 256;
    if (bx > 64) bx = 64;
    if (bx < 1) bx = 1;
    note_launch();
    k_batch_reset<<<dim3((unsigned)bx, (unsigned)count), 256, 0, s>>>(jobs);
}

void launch_histogram(const int* topk, int64_t nk, int* scores, cudaStream_t s) {
    if (nk <= 0) return;
    int64_t blocks = (nk + 255) / 256;
    if (blocks > 65536) blocks = 65536;
    note_launch();
    k_histogram<<<(int)blocks, 256, 0, s>>>(topk, nk, scores);
}

}  // namespace rkm
