// FP32 CUDA-core product kernels: the plain exact path of the threshold pass (K2)
// and the counting pass (K5).  Each 128-user x 128-item tile is computed with
// sequential FP32 FMAs (so |v - u.p| <= gamma_d * ||u|| ||p||, Higham, "Accuracy and
// Stability of Numerical Algorithms", 2nd ed., Section 3.1), staged through shared
// memory and handed row by row to the per-user epilogues of epilogue.cuh.
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "count_units.cuh"
#include "epilogue.cuh"
#include "kernels.h"

namespace rkm {

namespace {

constexpr int KC = 32;          // k-chunk of the product loop
constexpr int ASTR = 132;       // row stride (floats) of the transposed operand chunks
constexpr int CSTR = 132;       // row stride of the staged score tile
constexpr int SIMT_THREADS = 256;

// The staged scores take the place of the operand chunks, which the product has finished with, so
// that two CTAs fit an SM: one's product then runs beside the other's epilogue (counting phase at
// 20,000 users x 5,000 items, d = 64: 416 -> 360 us).
union SimtSmem {
    struct {
        float As[KC * ASTR];    // users chunk, [k][user]
        float Bs[KC * ASTR];    // items chunk, [k][item]
    };
    float Cs[BU * CSTR];        // scores, [user][item]
};
constexpr int SIMT_CTAS = 2;             // per SM
constexpr int SIMT_PARTS = 4;            // most parts of the item tiles (simt_segments)
constexpr int SIMT_HALF = BI_SIMT / 2;   // columns of a tile that one thread of the epilogue reads
static_assert(SIMT_THREADS == 2 * BU && BU == 128, "two threads of the epilogue per user");

// Load a 128-row x 32-k chunk of a packed operand (row stride dp) transposed into S[k][row].
__device__ __forceinline__ void load_chunk_t(const float* __restrict__ X, int64_t row0, int dp, int k0,
                                             float* S) {
    const int t = threadIdx.x;
    const int r = t & 127;
    const int kq0 = t >> 7;  // 0 or 1
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int kq = kq0 + 2 * i;  // float4 index within the chunk, 0..7
        const float4 x = *reinterpret_cast<const float4*>(X + (row0 + r) * (int64_t)dp + k0 + kq * 4);
        S[(kq * 4 + 0) * ASTR + r] = x.x;
        S[(kq * 4 + 1) * ASTR + r] = x.y;
        S[(kq * 4 + 2) * ASTR + r] = x.z;
        S[(kq * 4 + 3) * ASTR + r] = x.w;
    }
}

// Cs = A[row0a .. +128) . B[row0b .. +128)^T over the padded depth dp (multiple of 32).
__device__ void simt_tile(const float* __restrict__ A, int64_t row0a, const float* __restrict__ B,
                          int64_t row0b, int dp, SimtSmem& sm) {
    const int t = threadIdx.x;
    const int tx = t & 15, ty = t >> 4;
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
    for (int k0 = 0; k0 < dp; k0 += KC) {
        load_chunk_t(A, row0a, dp, k0, sm.As);
        load_chunk_t(B, row0b, dp, k0, sm.Bs);
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < KC; ++kk) {
            const float4 a0 = *reinterpret_cast<const float4*>(&sm.As[kk * ASTR + ty * 4]);
            const float4 a1 = *reinterpret_cast<const float4*>(&sm.As[kk * ASTR + 64 + ty * 4]);
            const float4 b0 = *reinterpret_cast<const float4*>(&sm.Bs[kk * ASTR + tx * 4]);
            const float4 b1 = *reinterpret_cast<const float4*>(&sm.Bs[kk * ASTR + 64 + tx * 4]);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int row = (i < 4) ? (ty * 4 + i) : (64 + ty * 4 + i - 4);
        *reinterpret_cast<float4*>(&sm.Cs[row * CSTR + tx * 4]) =
            make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        *reinterpret_cast<float4*>(&sm.Cs[row * CSTR + 64 + tx * 4]) =
            make_float4(acc[i][4], acc[i][5], acc[i][6], acc[i][7]);
    }
    __syncthreads();
}

__device__ __forceinline__ void load_row_chunk(const SimtSmem& sm, int row, int c0, float (&v)[32]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float4 x = *reinterpret_cast<const float4*>(&sm.Cs[row * CSTR + c0 + q * 4]);
        v[q * 4 + 0] = x.x;
        v[q * 4 + 1] = x.y;
        v[q * 4 + 2] = x.z;
        v[q * 4 + 3] = x.w;
    }
}

// K2: one CTA per user tile and part p of the item tiles (p, p + parts, ...), part after part.  A
// thread of the epilogue selects among half the columns of its user's row, into a list segment and
// a heap of its own; the 2 * parts threads of a user share their bounds through lfin_key.
// Bound by FP32 issue and by the epilogue of half a CTA's warps, which the other half and the
// other CTA of the SM now fill: 20,000 users x 5,000 items, d = 64, k = 25, where 157 user tiles took
// two rounds of one CTA per SM: 862 -> 502 us (two CTAs per SM alone: 735).
__global__ void __launch_bounds__(SIMT_THREADS, SIMT_CTAS) k_threshold_simt(ThresholdArgs a, int parts) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SimtSmem& sm = *reinterpret_cast<SimtSmem*>(smem_raw);
    const float* A = static_cast<const float*>(a.A);
    const float* B = static_cast<const float*>(a.B);
    const int t = threadIdx.x, r = t & (BU - 1), half = t >> 7;
    float* heap = reinterpret_cast<float*>(smem_raw + sizeof(SimtSmem)) + (size_t)half * a.k * BU;  // [2][k][BU]
    const int64_t user_tiles = (a.n + BU - 1) / BU;
    const int64_t item_tiles = (a.m + BI_SIMT - 1) / BI_SIMT;
    const int64_t ut = blockIdx.x % user_tiles;
    const int part = (int)(blockIdx.x / user_tiles);
    const int64_t u = ut * BU + r;
    const bool active = u < a.n;
    const int seg = part * 2 + half;
    SelState s;
    s.L = -INFINITY;
    s.hn = 0;
    s.Lw = -INFINITY;
    s.Lx = -INFINITY;
    s.thr = -INFINITY;
    s.cnt = 0;
    s.pub = nullptr;
    s.tag = 0u;
    s.mark = 0;
    s.Em = 0.f;
    for (int j = 0; j < a.k; ++j) heap[j * BU + r] = -INFINITY;
    const float un = active ? a.unrm[u] : 0.f;
    const float unh = active ? a.unhat[u] : 0.f;
    const float ud = active ? a.udel[u] : 0.f;
    Cand* mycand = a.cand + ((active ? u : 0) * a.nseg + seg) * (int64_t)a.cap;
    bool warm = false;
    int since = 0;               // tiles since candidates were offered to the heap
    float published = -INFINITY;
    int64_t items = 0;
    for (int64_t it = part; it < item_tiles; it += parts) {
        // Any bound the other threads of this user have published bounds tau_u from below.
        const unsigned lk = active ? __ldcg(&a.lfin_key[u]) : 0u;
        simt_tile(A, ut * BU, B, it * BI_SIMT, a.dp, sm);
        s.Lx = key_float(lk);
        const float E = err_bound(a.cacc, a.eabs, un, unh, ud, a.thmax[it], a.tdel[it]);
        const int pos0 = (int)(it * BI_SIMT) + half * SIMT_HALF;
        if (!warm) {
            // A lower bound before any candidate is recorded (see warm_bound): the k-th largest of
            // 32 maxima of 2 columns, -inf for k > 32.
            auto load = [&](int c0, float (&v)[32]) { load_row_chunk(sm, r, half * SIMT_HALF + c0, v); };
            const float lw = warm_bound<32, SIMT_HALF>(load, pos0, a.m, a.k, E);
            s.Lw = active ? lw : -INFINITY;
            warm = true;
        }
        s.thr = __fsub_rd(sel_bound(s), E);
#pragma unroll 1
        for (int c0 = 0; c0 < SIMT_HALF; c0 += 32) {
            float v[32];
            load_row_chunk(sm, r, half * SIMT_HALF + c0, v);
            sel_chunk(v, active, pos0 + c0, a.m, E, s, mycand, a.cap, a.st);
        }
        s.Em = fmaxf(s.Em, E);
        if (++since == MERGE_TILES || __any_sync(0xffffffffu, active && s.mark >= 0 && s.cnt - s.mark >= MERGE_HITS)) {
            sel_merge(s, mycand, heap, r, a.k, active);
            since = 0;
        }
        const float own = fmaxf(s.L, s.Lw);
        if (active && own > published) {
            published = own;
            atomicMax(&a.lfin_key[u], float_key(own));
        }
        items += a.m - it * BI_SIMT < BI_SIMT ? a.m - it * BI_SIMT : BI_SIMT;
        // Algorithm 1's stop by Cauchy-Schwarz: items come in descending order of their norms'
        // buckets, so once ||u|| times the end of the next tile's bucket (rounded up) is below a
        // lower bound of tau_u, no later item can reach tau_u or tie it.
        const bool need_next =
            active && it + parts < item_tiles && !(__fmul_ru(un, bucket_end(a.tmax[it + parts])) < sel_bound(s));
        if (!__syncthreads_or(need_next)) break;
    }
    if (t == 0) {
        const int64_t rows = (a.n - ut * BU < BU) ? a.n - ut * BU : BU;
        atomicAdd(&a.st->thr_pairs, (unsigned long long)(rows * items));
    }
    if (active) a.cand_cnt[u * a.nseg + seg] = s.cnt;
}

// K5: persistent over work units (item tile, group of user tiles) taken from a ticket.
__global__ void __launch_bounds__(SIMT_THREADS, SIMT_CTAS) k_count_simt(CountArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SimtSmem& sm = *reinterpret_cast<SimtSmem*>(smem_raw);
    int* cnt_s = reinterpret_cast<int*>(smem_raw + sizeof(SimtSmem));  // [BI_SIMT]
    BandStage stage{reinterpret_cast<int2*>(cnt_s + BI_SIMT) + (threadIdx.x >> 5) * BAND_STAGE, 0};
    __shared__ unsigned s_unit;
    const float* A = static_cast<const float*>(a.A);
    const float* B = static_cast<const float*>(a.B);
    const int t = threadIdx.x;
    const unsigned total = a.st->units_total;
    while (true) {
        if (t == 0) s_unit = atomicAdd(&a.st->ticket, 1u);
        __syncthreads();
        const unsigned w = s_unit;
        __syncthreads();
        if (w >= total) {
            band_flush(stage, a.band, a.band_cap, a.st);
            break;
        }
        int T;
        int64_t ut0, ut1;
        decode_count_unit(a, w, T, ut0, ut1);
        if (t < BI_SIMT) cnt_s[t] = 0;
        __syncthreads();
        const float pnh = a.thmax[T], pd = a.tdel[T];
        const int pos0 = T * BI_SIMT;
        for (int64_t ut = ut0; ut < ut1; ++ut) {
            simt_tile(A, ut * BU, B, (int64_t)T * BI_SIMT, a.dp, sm);
            const int r = t & (BU - 1), h0 = (t >> 7) * SIMT_HALF;
            const int64_t us = ut * BU + r;
            const bool active = us < a.n;
            float hi_t = 0.f, lo_t = 0.f;
            int u_orig = 0;
            if (active) {
                const UserMeta um = a.meta[us];
                const float E = err_bound(a.cacc, a.eabs, um.un, um.unh, um.ud, pnh, pd);
                hi_t = __fadd_ru(um.tau_hi, E);
                lo_t = __fsub_rd(um.tau_lo, E);
                u_orig = um.uorig;
            }
#pragma unroll 1
            for (int c0 = h0; c0 < h0 + SIMT_HALF; c0 += 32) {
                float v[32];
                load_row_chunk(sm, r, c0, v);
                count_chunk(v, active, c0, pos0 + c0, a.m, hi_t, lo_t, cnt_s, u_orig, stage, a.band, a.band_cap,
                            a.st);
            }
            if (stage.n > BAND_STAGE / 2) band_flush(stage, a.band, a.band_cap, a.st);
            __syncthreads();
        }
        if (t == 0 && ut1 > ut0) {
            unsigned long long users = (unsigned long long)((ut1 * BU < a.n ? ut1 * BU : a.n) - ut0 * BU);
            atomicAdd(&a.st->pairs_evaluated, users * (unsigned long long)BI_SIMT);
        }
        if (t < BI_SIMT && cnt_s[t] != 0 && pos0 + t < a.m) atomicAdd(&a.counts[pos0 + t], cnt_s[t]);
        __syncthreads();
    }
}

}  // namespace

// Parts of the item tiles: as many as give each CTA slot of the SMs about four units, at most
// SIMT_PARTS.  Each part selects on its own, so more parts record more candidates: at 20,000 users x
// 5,000 items, k = 25, threshold and exact phase take 735 + 35 us with one part (and one thread per
// row), 608 + 68 with two, 502 + 102 with four, 471 + 248 with eight.
int simt_segments(int64_t n, int64_t m, int num_sms) {
    const int64_t user_tiles = (n + BU - 1) / BU, item_tiles = (m + BI_SIMT - 1) / BI_SIMT;
    const int64_t want = ((int64_t)4 * SIMT_CTAS * num_sms + user_tiles - 1) / std::max<int64_t>(user_tiles, 1);
    return 2 * (int)std::max<int64_t>(1, std::min<int64_t>({want, SIMT_PARTS, item_tiles}));
}

void launch_threshold_simt(const ThresholdArgs& a, cudaStream_t s) {
    const size_t smem = sizeof(SimtSmem) + (size_t)2 * a.k * BU * sizeof(float);
    cudaFuncSetAttribute(k_threshold_simt, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(sizeof(SimtSmem) + (size_t)2 * KMAX * BU * sizeof(float)));
    const int parts = a.nseg / 2;
    const int64_t units = (a.n + BU - 1) / BU * parts;
    if (units < 1) return;
    note_launch();
    k_threshold_simt<<<(unsigned)units, SIMT_THREADS, smem, s>>>(a, parts);
}

void launch_count_simt(const CountArgs& a, cudaStream_t s) {
    const size_t smem = sizeof(SimtSmem) + BI_SIMT * sizeof(int) + (SIMT_THREADS / 32) * BAND_STAGE * sizeof(int2);
    cudaFuncSetAttribute(k_count_simt, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    note_launch();
    k_count_simt<<<a.num_sms * SIMT_CTAS, SIMT_THREADS, smem, s>>>(a);
}

}  // namespace rkm
