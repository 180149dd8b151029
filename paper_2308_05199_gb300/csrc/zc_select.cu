// zc_select.cu -- the per-chunk codec selector: chunk statistics, the
// 16-64-64-4 MLP (forward, loss gradient, momentum SGD) and the selection of
// block size or raw storage, written into a batched-compression plan.
//
// The statistics, the network and the cost model are defined in the header
// comment of zc.h (zc_batch_chunk_stats .. zc_batch_select).  Everything runs
// on the device; nothing is read back, so a whole select-then-compress
// sequence can be captured in one CUDA graph.
#include <cooperative_groups.h>
#include <cstddef>
#include <cstring>

#include "zc_launch.h"

namespace zc {

constexpr int N_STATS = ZC_STATS;
constexpr unsigned FULL_MASK_ALL = 0xffffffffu;
constexpr int ST_SPANS = 16;
constexpr int ST_SPAN = 128;

constexpr int NI = ZC_MLP_IN, NH = ZC_MLP_HIDDEN, NO = ZC_MLP_OUT;
constexpr int NPARAM = ZC_MLP_PARAMS;
constexpr int OFF_B1 = NH * NI, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH;
constexpr int OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NO * NH;
static_assert(OFF_B3 + NO == NPARAM, "parameter layout");
constexpr int NPAD = 5512;  // per-CTA partial gradient stride (NPARAM + loss, rounded)
constexpr int TB = 64;      // samples per CTA
constexpr int MT = 256;     // threads per MLP CTA

__device__ __forceinline__ int bitlen_u(unsigned v) { return 32 - __clz(v); }

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v)
{
#pragma unroll
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
    return v;
}

// ---- chunk statistics: one warp per item ----------------------------------------
// Lane l holds elements 4l .. 4l + 3 of a 128-element span (one 16-byte load
// of FP32, one 8-byte load of BF16, when the chunk is aligned for it), so
// three of every four differences are taken within the lane and a block of
// L elements is L / 4 consecutive lanes: its largest |delta| is one segmented
// warp reduction.  Per-lane sums stay 32-bit (64 sampled elements per lane at
// most: |q| < 2^23, |d| < 2^24, |d2| < 2^25) and are widened for the warp sum.
struct StatAcc {
    unsigned b16 = 0, b32 = 0, b64 = 0, b128 = 0;  // codec block bits per L (block-first lanes)
    unsigned sum_ad = 0, sum_aq = 0, sum_ad2 = 0;
    unsigned max_ad = 0, nz_d = 0, nz_q = 0, n_sc = 0, head_bits = 0;
    int qmin = 0x7fffffff, qmax = -0x7fffffff - 1;
    int bad = 0;
};

// The four elements of this lane in span [s0, s0 + cnt) (zero beyond cnt).
__device__ __forceinline__ void load_span4(const Item& it, bool vec, unsigned long long s0, int cnt,
                                           float v[4])
{
    const int lane = threadIdx.x & 31;
    const int i0 = 4 * lane;
    if (it.x_dtype == ZC_F32) {
        const float* p = (const float*)it.x + s0 + i0;
        if (vec && i0 + 4 <= cnt) {
            const float4 w = ld_dep((const float4*)p);
            v[0] = w.x; v[1] = w.y; v[2] = w.z; v[3] = w.w;
        } else {
#pragma unroll
            for (int m = 0; m < 4; ++m) v[m] = i0 + m < cnt ? ld_dep(p + m) : 0.0f;
        }
    } else {
        const unsigned short* p = (const unsigned short*)it.x + s0 + i0;
        if (vec && i0 + 4 <= cnt) {
            const uint2 w = ld_dep((const uint2*)p);
            v[0] = __uint_as_float(w.x << 16);
            v[1] = __uint_as_float(w.x & 0xffff0000u);
            v[2] = __uint_as_float(w.y << 16);
            v[3] = __uint_as_float(w.y & 0xffff0000u);
        } else {
#pragma unroll
            for (int m = 0; m < 4; ++m) v[m] = i0 + m < cnt ? bf16_to_f32(ld_dep(p + m)) : 0.0f;
        }
    }
}

// One span of cnt elements (v: this lane's four); returns the span's L = 32
// block bits (the same in every lane).  FULL: cnt == 128.  Branch-free:
// elements outside the span, and the differences that do not exist at the
// span's start, are masked out.
template <bool FULL>
__device__ __forceinline__ unsigned stat_span(const float v[4], int cnt, const Item& it,
                                              StatAcc& A)
{
    const int lane = threadIdx.x & 31;
    const int i0 = 4 * lane;
    int q[4];
    bool ok[4];
    // the exact quantizer: fast rounding for all four, the exact slow path
    // only when some lane's fast result may be off (one vote)
    bool slow = false;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        ok[m] = FULL || i0 + m < cnt;
        slow |= !quantize_fast(ok[m] ? v[m] : 0.0f, it.inv, q[m]);
    }
    if (__any_sync(FULL_MASK_ALL, slow)) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            int qq = 0;
            if (ok[m] && quantize(v[m], it.eb, it.two_eb, it.inv, qq) != 0) {
                A.bad = 1;
                qq = 0;
            }
            q[m] = qq;
        }
    }
    // first differences d (element i >= 1) and the previous one pd (i >= 2)
    int d[4], pd[4];
    d[0] = q[0] - __shfl_up_sync(FULL_MASK_ALL, q[3], 1);
#pragma unroll
    for (int m = 1; m < 4; ++m) d[m] = q[m] - q[m - 1];
    pd[0] = __shfl_up_sync(FULL_MASK_ALL, d[3], 1);
#pragma unroll
    for (int m = 1; m < 4; ++m) pd[m] = d[m - 1];
    unsigned rest = 0;  // largest |d| of elements 1..3 of the lane
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const bool v0 = ok[m];
        const bool v1 = v0 && (m > 0 || lane > 0);   // element i >= 1
        const bool v2 = v0 && (m > 1 || lane > 0);   // element i >= 2
        const unsigned aq = v0 ? (unsigned)abs(q[m]) : 0u;
        const unsigned ad = v1 ? (unsigned)abs(d[m]) : 0u;
        const unsigned ad2 = v2 ? (unsigned)abs(d[m] - pd[m]) : 0u;
        A.nz_q += (v0 && q[m] == 0) ? 1u : 0u;
        A.sum_aq += aq;
        A.qmin = min(A.qmin, v0 ? q[m] : 0x7fffffff);
        A.qmax = max(A.qmax, v0 ? q[m] : -0x7fffffff - 1);
        A.sum_ad += ad;
        A.max_ad = max(A.max_ad, ad);
        A.nz_d += (v1 && d[m] == 0) ? 1u : 0u;
        if (m > 0) rest = max(rest, ad);
        A.sum_ad2 += ad2;
        const bool sc = (d[m] ^ pd[m]) < 0 && d[m] != 0 && pd[m] != 0;
        A.n_sc += (v2 && sc) ? 1u : 0u;
    }
    const unsigned e0q = ok[0] ? (unsigned)abs(q[0]) : 0u;
    const unsigned e0d = (ok[0] && i0 >= 1) ? (unsigned)abs(d[0]) : 0u;
    // Largest block |delta| at blocks of 4, 8, 16 and 32 lanes, right in each
    // block's first lane: the block's first element counts as |q| (the head is
    // predicted from 0), every other lane's first element as |d|.  A block of
    // twice the size takes both halves and the second half's first |d|: five
    // shuffles for the four sizes (ten when each size reduced by itself).
    unsigned a = max(rest, (lane & 3) ? e0d : 0u);
    a = max(a, __shfl_xor_sync(FULL_MASK_ALL, a, 1));
    a = max(a, __shfl_xor_sync(FULL_MASK_ALL, a, 2));
    const unsigned m16 = max(a, e0q);
    if ((lane & 7) == 4) a = max(a, e0d);
    a = max(a, __shfl_xor_sync(FULL_MASK_ALL, a, 4));
    const unsigned m32 = max(a, e0q);
    if ((lane & 15) == 8) a = max(a, e0d);
    a = max(a, __shfl_xor_sync(FULL_MASK_ALL, a, 8));
    const unsigned m64 = max(a, e0q);
    if (lane == 16) a = max(a, e0d);
    a = max(a, __shfl_xor_sync(FULL_MASK_ALL, a, 16));
    const unsigned m128 = max(a, e0q);
    const unsigned b32 = ((lane & 7) == 0 && m32) ? (bitlen_u(m32) + 1) * 32 : 0u;
    A.b16 += ((lane & 3) == 0 && m16) ? (bitlen_u(m16) + 1) * 16 : 0u;
    A.b64 += ((lane & 15) == 0 && m64) ? (bitlen_u(m64) + 1) * 64 : 0u;
    A.b128 += (lane == 0 && m128) ? (bitlen_u(m128) + 1) * 128 : 0u;
    A.b32 += b32;
    A.head_bits += ((lane & 7) == 0 && ok[0]) ? bitlen_u(e0q) : 0u;
    return __reduce_add_sync(FULL_MASK_ALL, b32);
}

__global__ void __launch_bounds__(256, 4) k_chunk_stats(const Item* items, unsigned n_items,
                                                     float* feat)
{
    grid_dep_wait();
    grid_dep_launch();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned idx = blockIdx.x * 8 + warp;
    if (idx >= n_items) return;  // warp-uniform; only warp-level sync below
    const Item it = items[idx];
    float* out = feat + (size_t)idx * N_STATS;
    const unsigned long long n = it.n;
    if (n == 0 || it.x == nullptr || !(it.two_eb > 0.0f)) {
        if (lane < N_STATS) out[lane] = __int_as_float(0x7fc00000);  // NaN row
        return;
    }
    const unsigned long long m = n / ST_SPAN;
    const int S = m == 0 ? 1 : (int)(m < ST_SPANS ? m : ST_SPANS);
    const int cnt = m == 0 ? (int)n : ST_SPAN;  // elements of every sampled span
    // spans start at multiples of 128 elements: aligned loads when the chunk is
    const bool vec = ((uintptr_t)it.x & (it.x_dtype == ZC_F32 ? 15u : 7u)) == 0u;
    // span j starts at 128 floor(j (m - 1) / (S - 1)): stepped without a
    // division per span (quotient and remainder of (m - 1) / (S - 1) once)
    const unsigned long long den = S > 1 ? (unsigned long long)(S - 1) : 1ull;
    const unsigned long long num = m > 0 ? m - 1 : 0ull;
    const unsigned long long qa = num / den, ra = num % den;
    unsigned long long sq = 0ull, sr = 0ull;  // floor(j num / den) and its remainder, next span
    auto next_span0 = [&]() -> unsigned long long {
        const unsigned long long v = (unsigned long long)ST_SPAN * sq;
        sq += qa;
        sr += ra;
        if (sr >= den) {
            sr -= den;
            sq += 1ull;
        }
        return v;
    };
    StatAcc A;
    // sum over the spans of their L = 32 bits, and of its squares (warp-uniform;
    // a span holds at most 128 x 25 bits, so both fit 32 bits over 16 spans)
    unsigned span_b1 = 0u, span_b2 = 0u;
    auto add_span = [&](unsigned b) {
        span_b1 += b;
        span_b2 += b * b;
    };
    if (cnt == ST_SPAN) {
        // full spans: two loaded ahead of the one being summarised
        float xa[4], xb[4], xc[4];
        load_span4(it, vec, next_span0(), cnt, xa);
        if (S > 1) load_span4(it, vec, next_span0(), cnt, xb);
#pragma unroll 1
        for (int j = 0; j < S; ++j) {
            if (j + 2 < S) load_span4(it, vec, next_span0(), cnt, xc);
            add_span(stat_span<true>(xa, cnt, it, A));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                xa[k] = xb[k];
                xb[k] = xc[k];
            }
        }
    } else {
        float xa[4];
        load_span4(it, vec, 0ull, cnt, xa);
        add_span(stat_span<false>(xa, cnt, it, A));
    }
    const unsigned long long B16 = warp_sum_u64(A.b16), B32 = warp_sum_u64(A.b32);
    const unsigned long long B64 = warp_sum_u64(A.b64), B128 = warp_sum_u64(A.b128);
    const unsigned long long SAD = warp_sum_u64(A.sum_ad), SAQ = warp_sum_u64(A.sum_aq);
    const unsigned long long SAD2 = warp_sum_u64(A.sum_ad2);
    const unsigned long long NZD = __reduce_add_sync(FULL, A.nz_d);
    const unsigned long long NZQ = __reduce_add_sync(FULL, A.nz_q);
    const unsigned long long NSC = __reduce_add_sync(FULL, A.n_sc);
    const unsigned long long HB = __reduce_add_sync(FULL, A.head_bits);
    const unsigned MAD = __reduce_max_sync(FULL, A.max_ad);
    const int QMN = __reduce_min_sync(FULL, A.qmin), QMX = __reduce_max_sync(FULL, A.qmax);
    const int BAD = __any_sync(FULL, A.bad);
    if (lane != 0) return;
    if (BAD) {
        for (int k = 0; k < N_STATS; ++k) out[k] = __int_as_float(0x7fc00000);
        return;
    }
    const unsigned long long bits[4] = {B16, B32, B64, B128};
    // The features in FP32 (this GPU's FP64 rate is a small fraction of its
    // FP32 rate): counts are exact integers below 2^24, each quotient is one
    // correctly rounded division, each logarithm CUDA's log2f.
    const float tot = (float)(S * cnt), fn = (float)n;
    const float nd = (float)(S * (cnt - 1));
    const float nd2 = cnt >= 2 ? (float)(S * (cnt - 2)) : 0.0f;
    const float nheads = (float)(S * ((cnt + 31) / 32));
    const float hdr = __fdiv_rn(256.0f, fn);
    float f[N_STATS];
    f[0] = __fadd_rn(__fadd_rn(__fdiv_rn((float)bits[0], tot), 0.5f), hdr);
    f[1] = __fadd_rn(__fadd_rn(__fdiv_rn((float)bits[1], tot), 0.25f), hdr);
    f[2] = __fadd_rn(__fadd_rn(__fdiv_rn((float)bits[2], tot), 0.125f), hdr);
    f[3] = __fadd_rn(__fadd_rn(__fdiv_rn((float)bits[3], tot), 0.0625f), hdr);
    f[4] = log2f(1.0f + (float)((long long)QMX - (long long)QMN));
    f[5] = nd > 0.0f ? log2f(1.0f + __fdiv_rn((float)SAD, nd)) : 0.0f;
    f[6] = nd > 0.0f ? log2f(1.0f + (float)MAD) : 0.0f;
    f[7] = nd > 0.0f ? __fdiv_rn((float)NZD, nd) : 0.0f;
    f[8] = __fdiv_rn((float)NZQ, tot);
    f[9] = log2f(1.0f + __fdiv_rn((float)SAQ, tot));
    f[10] = nd2 > 0.0f ? log2f(1.0f + __fdiv_rn((float)SAD2, nd2)) : 0.0f;
    f[11] = nd2 > 0.0f ? __fdiv_rn((float)NSC, nd2) : 0.0f;
    f[12] = __fdiv_rn(__fdiv_rn((float)HB, nheads), 24.0f);
    // population spread of the spans' bits per element b_j / cnt, from exact
    // integer moments: S^2 cnt^2 var = S sum b_j^2 - (sum b_j)^2
    const long long dvar = (long long)S * (long long)span_b2 - (long long)span_b1 * (long long)span_b1;
    const float sc2 = (float)S * (float)cnt;
    f[13] = sqrtf(__fdiv_rn((float)dvar, __fmul_rn(sc2, sc2)));
    f[14] = it.x_dtype == ZC_F32 ? 1.0f : 0.5f;
    f[15] = __fdiv_rn(log2f(fn), 16.0f);
#pragma unroll
    for (int k = 0; k < N_STATS; ++k) out[k] = f[k];
}

// ---- MLP ------------------------------------------------------------------------------
// Shared memory of an MLP CTA (floats): the parameters with padded row
// strides (no bank conflicts), the normalised inputs, both layers'
// activations (after the ReLU), one 64 x 64 gradient buffer and the outputs.
// Rows that the forward pass reads four at a time (W2, W3, X, A1, A2) have
// strides of a multiple of 4 floats: 16-byte loads, and at stride 68 the 8
// rows of a quarter warp fall in distinct bank groups.
constexpr int NHP = NH + 4, NIP = NI + 4;
struct MlpSmem {
    float W1[NH][NI + 1], b1[NH];
    alignas(16) float W2[NH][NHP];
    float b2[NH];
    alignas(16) float W3[NO][NHP];
    float b3[NO];
    alignas(16) float X[TB][NIP];
    alignas(16) float A1[TB][NHP];
    alignas(16) float A2[TB][NHP];  // later: dA1
    float D[TB][NH + 1];            // dA2
    float Y[TB][NO];                // outputs, later dY
    float red[MT / 32];
};
static_assert(offsetof(MlpSmem, W2) % 16 == 0 && offsetof(MlpSmem, W3) % 16 == 0 &&
                  offsetof(MlpSmem, X) % 16 == 0 && offsetof(MlpSmem, A1) % 16 == 0 &&
                  offsetof(MlpSmem, A2) % 16 == 0,
              "16-byte rows");

__device__ __forceinline__ float relu(float v) { return v > 0.0f ? v : 0.0f; }

// Loads the parameters into shared memory (no barrier).
__device__ __forceinline__ void mlp_load_params(MlpSmem& sm, const float* P)
{
    const int t = threadIdx.x;
    for (int p = t; p < NH * NI; p += MT) sm.W1[p / NI][p % NI] = P[p];
    for (int p = t; p < NH * NH; p += MT) sm.W2[p / NH][p % NH] = P[OFF_W2 + p];
    for (int p = t; p < NO * NH; p += MT) sm.W3[p / NH][p % NH] = P[OFF_W3 + p];
    if (t < NH) {
        sm.b1[t] = P[OFF_B1 + t];
        sm.b2[t] = P[OFF_B2 + t];
    }
    if (t < NO) sm.b3[t] = P[OFF_B3 + t];
}

// Loads the tile's rows (normalised) into shared memory; rows past B are
// zero (no barrier).
__device__ __forceinline__ void mlp_load_rows(MlpSmem& sm, const float* norm, const float* X,
                                              const int* idx, int B, int row0)
{
    const int t = threadIdx.x;
    for (int p = t; p < TB * NI; p += MT) {
        const int s = p / NI, k = p % NI, r = row0 + s;
        float v = 0.0f;
        if (r < B) {
            const long long row = idx != nullptr ? (long long)idx[r] : (long long)r;
            v = __fmul_rn(__fsub_rn(X[row * NI + k], norm[k]), norm[NI + k]);
        }
        sm.X[s][k] = v;
    }
}

// Loads the parameters and the tile's rows.
__device__ __forceinline__ void mlp_load(MlpSmem& sm, const float* P, const float* norm,
                                         const float* X, const int* idx, int B, int row0)
{
    mlp_load_params(sm, P);
    mlp_load_rows(sm, norm, X, idx, B, row0);
    __syncthreads();
}

// H1 = relu(X W1^T + b1), H2 = relu(H1 W2^T + b2), Y = H2 W3^T + b3, each
// sum accumulated by FMAs in input order.  sm.A1 and sm.A2 hold the
// activations after the ReLU: the gradient's ReLU derivative only asks
// whether the pre-activation was positive, which H > 0 answers alike.
__device__ __forceinline__ void mlp_forward_tile(MlpSmem& sm)
{
    const int t = threadIdx.x, j = t & (NH - 1), g = t >> 6;
    {
        float w[NI];
#pragma unroll
        for (int k = 0; k < NI; ++k) w[k] = sm.W1[j][k];
        for (int i = 0; i < TB / 4; ++i) {
            const int s = g * (TB / 4) + i;
            float a = sm.b1[j];
#pragma unroll
            for (int k = 0; k < NI; k += 4) {
                const float4 x = *reinterpret_cast<const float4*>(&sm.X[s][k]);
                a = __fmaf_rn(w[k], x.x, a);
                a = __fmaf_rn(w[k + 1], x.y, a);
                a = __fmaf_rn(w[k + 2], x.z, a);
                a = __fmaf_rn(w[k + 3], x.w, a);
            }
            sm.A1[s][j] = relu(a);
        }
    }
    __syncthreads();
    {
        float acc[TB / 4];
#pragma unroll
        for (int i = 0; i < TB / 4; ++i) acc[i] = sm.b2[j];
#pragma unroll 2
        for (int k = 0; k < NH; k += 4) {
            const float4 w = *reinterpret_cast<const float4*>(&sm.W2[j][k]);
#pragma unroll
            for (int i = 0; i < TB / 4; ++i) {
                const float4 a = *reinterpret_cast<const float4*>(&sm.A1[g * (TB / 4) + i][k]);
                acc[i] = __fmaf_rn(w.x, a.x, acc[i]);
                acc[i] = __fmaf_rn(w.y, a.y, acc[i]);
                acc[i] = __fmaf_rn(w.z, a.z, acc[i]);
                acc[i] = __fmaf_rn(w.w, a.w, acc[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < TB / 4; ++i) sm.A2[g * (TB / 4) + i][j] = relu(acc[i]);
    }
    __syncthreads();
    {
        const int s = t >> 2, o = t & 3;
        float y = sm.b3[o];
#pragma unroll 4
        for (int k = 0; k < NH; k += 4) {
            const float4 w = *reinterpret_cast<const float4*>(&sm.W3[o][k]);
            const float4 a = *reinterpret_cast<const float4*>(&sm.A2[s][k]);
            y = __fmaf_rn(w.x, a.x, y);
            y = __fmaf_rn(w.y, a.y, y);
            y = __fmaf_rn(w.z, a.z, y);
            y = __fmaf_rn(w.w, a.w, y);
        }
        sm.Y[s][o] = y;
    }
    __syncthreads();
}

// Persistent over row tiles: the parameters are loaded once per CTA, then
// the CTA takes tiles blockIdx.x, blockIdx.x + gridDim.x, ... (every row's
// arithmetic is the same as with one tile per CTA).
__global__ void __launch_bounds__(MT) k_mlp_forward(const float* P, const float* norm,
                                                    const float* X, int B, float* Yout)
{
    grid_dep_wait();
    grid_dep_launch();
    extern __shared__ __align__(16) uint8_t raw[];
    MlpSmem& sm = *reinterpret_cast<MlpSmem*>(raw);
    const int ntiles = (B + TB - 1) / TB;
    mlp_load_params(sm, P);
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int row0 = tile * TB;
        mlp_load_rows(sm, norm, X, nullptr, B, row0);
        __syncthreads();
        mlp_forward_tile(sm);  // ends with a barrier: sm.Y is complete
        const int t = threadIdx.x, s = t >> 2, o = t & 3;
        if (row0 + s < B) Yout[(long long)(row0 + s) * NO + o] = sm.Y[s][o];
    }
}

// Per-CTA partial gradient of sum((Y - T)^2) / (B * NO) over its rows, and
// the partial sum of squared residuals, at partial + blockIdx.x * NPAD.
__global__ void __launch_bounds__(MT) k_mlp_grad(const float* P, const float* norm,
                                                 const float* X, const float* T, const int* idx,
                                                 int B, float* partial)
{
    extern __shared__ __align__(16) uint8_t raw[];
    MlpSmem& sm = *reinterpret_cast<MlpSmem*>(raw);
    const int row0 = blockIdx.x * TB;
    mlp_load(sm, P, norm, X, idx, B, row0);
    mlp_forward_tile(sm);
    const int t = threadIdx.x, j = t & (NH - 1), g = t >> 6;
    float* G = partial + (size_t)blockIdx.x * NPAD;
    const float scale = 2.0f / (float)(B * NO);
    // dY and the squared residuals
    {
        const int s = t >> 2, o = t & 3, r = row0 + s;
        float sq = 0.0f, dy = 0.0f;
        if (r < B) {
            const long long row = idx != nullptr ? (long long)idx[r] : (long long)r;
            const float res = __fsub_rn(sm.Y[s][o], T[row * NO + o]);
            sq = __fmul_rn(res, res);
            dy = __fmul_rn(scale, res);
        }
        __syncthreads();  // every Y read before it becomes dY
        sm.Y[s][o] = dy;
#pragma unroll
        for (int off = 16; off; off >>= 1) sq = __fadd_rn(sq, __shfl_xor_sync(FULL, sq, off));
        if ((t & 31) == 0) sm.red[t >> 5] = sq;
    }
    __syncthreads();
    if (t == 0) {
        float l = 0.0f;
        for (int w = 0; w < MT / 32; ++w) l = __fadd_rn(l, sm.red[w]);
        G[NPARAM] = l;
    }
    // dW3[o][k] = sum_s dY[s][o] H2[s][k]; db3
    {
        const int o = t >> 6, k = t & 63;
        float acc = 0.0f;
        for (int s = 0; s < TB; ++s) acc = __fadd_rn(acc, __fmul_rn(sm.Y[s][o], sm.A2[s][k]));
        G[OFF_W3 + o * NH + k] = acc;
        if (t < NO) {
            float b = 0.0f;
            for (int s = 0; s < TB; ++s) b = __fadd_rn(b, sm.Y[s][t]);
            G[OFF_B3 + t] = b;
        }
    }
    // dA2[s][j] = (sum_o dY[s][o] W3[o][j]) [H2 > 0]
    for (int i = 0; i < TB / 4; ++i) {
        const int s = g * (TB / 4) + i;
        float a = 0.0f;
#pragma unroll
        for (int o = 0; o < NO; ++o) a = __fadd_rn(a, __fmul_rn(sm.Y[s][o], sm.W3[o][j]));
        sm.D[s][j] = sm.A2[s][j] > 0.0f ? a : 0.0f;
    }
    __syncthreads();
    // dW2[j][k] = sum_s dA2[s][j] H1[s][k] for k in this thread's 16; db2
    {
        float acc[NH / 4];
#pragma unroll
        for (int kk = 0; kk < NH / 4; ++kk) acc[kk] = 0.0f;
        float b = 0.0f;
        for (int s = 0; s < TB; ++s) {
            const float a = sm.D[s][j];
            b = __fadd_rn(b, a);
#pragma unroll
            for (int kk = 0; kk < NH / 4; ++kk)
                acc[kk] = __fadd_rn(acc[kk], __fmul_rn(a, sm.A1[s][g * (NH / 4) + kk]));
        }
#pragma unroll
        for (int kk = 0; kk < NH / 4; ++kk) G[OFF_W2 + j * NH + g * (NH / 4) + kk] = acc[kk];
        if (g == 0) G[OFF_B2 + j] = b;
    }
    // dA1[s][k] = (sum_j dA2[s][j] W2[j][k]) [H1 > 0], into A2's storage (k = this thread's j)
    {
        float acc[TB / 4];
#pragma unroll
        for (int i = 0; i < TB / 4; ++i) acc[i] = 0.0f;
        for (int jj = 0; jj < NH; ++jj) {
            const float w = sm.W2[jj][j];
#pragma unroll
            for (int i = 0; i < TB / 4; ++i)
                acc[i] = __fadd_rn(acc[i], __fmul_rn(sm.D[g * (TB / 4) + i][jj], w));
        }
        __syncthreads();  // A2 (read above for dA2) is dead from here on
#pragma unroll
        for (int i = 0; i < TB / 4; ++i) {
            const int s = g * (TB / 4) + i;
            sm.A2[s][j] = sm.A1[s][j] > 0.0f ? acc[i] : 0.0f;
        }
    }
    __syncthreads();
    // dW1[j][k] = sum_s dA1[s][j] X[s][k] for k in this thread's 4; db1
    {
        float acc[NI / 4];
#pragma unroll
        for (int kk = 0; kk < NI / 4; ++kk) acc[kk] = 0.0f;
        float b = 0.0f;
        for (int s = 0; s < TB; ++s) {
            const float a = sm.A2[s][j];
            b = __fadd_rn(b, a);
#pragma unroll
            for (int kk = 0; kk < NI / 4; ++kk)
                acc[kk] = __fadd_rn(acc[kk], __fmul_rn(a, sm.X[s][g * (NI / 4) + kk]));
        }
#pragma unroll
        for (int kk = 0; kk < NI / 4; ++kk) G[j * NI + g * (NI / 4) + kk] = acc[kk];
        if (g == 0) G[OFF_B1 + j] = b;
    }
}

// Sums the CTAs' partial gradients in CTA order (deterministic).
__global__ void k_mlp_reduce(const float* partial, int nct, int B, float* grad, float* loss)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > NPARAM) return;
    float acc = 0.0f;
    for (int c = 0; c < nct; ++c) acc = __fadd_rn(acc, partial[(size_t)c * NPAD + p]);
    if (p < NPARAM) grad[p] = acc;
    else if (loss != nullptr) *loss = acc / (float)(B * NO);
}

// v <- momentum v + g; p <- p - lr v.
__global__ void k_mlp_sgd(float* P, float* V, const float* G, float lr, float momentum)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= NPARAM) return;
    const float v = __fadd_rn(__fmul_rn(momentum, V[p]), G[p]);
    V[p] = v;
    P[p] = __fsub_rn(P[p], __fmul_rn(lr, v));
}

// ---- a training epoch in one launch ------------------------------------------------
// A minibatch is a chain of three small launches (gradient of one CTA per 64
// rows, reduction, update), each of which loads the parameters anew; at 256
// rows it keeps 4 SMs busy, and an epoch of 10000 rows took 1545 us.  Here one
// cluster of FC CTAs trains for the whole epoch with the parameters in the
// shared memory of every CTA (359 us; with the permutation and the
// host's part of the epoch 573 us).  It does the very same
// arithmetic in the same order, so an epoch's results are those of the chain,
// bit for bit: a ReLU whose input is a rounding away from 0 would otherwise
// take the other side in one of the two.
//
// A turn takes 4 tiles of TB rows (the chain's CTAs).  Tile g is worked on by
// the CTAs 4 g .. 4 g + 3 ("quarters"):
//   rows: each quarter runs 16 of the tile's rows forward and backward and
//     writes their activations and deltas to the quarters that need them
//     (distributed shared memory);
//   sums: each quarter sums its share of the tile's gradient over all 64 rows
//     in order: the neurons j of both hidden layers with j / 16 = quarter, and
//     output o = quarter;
//   totals: a quarter's four CTAs (one per tile) add a quarter of its share
//     each over the tiles, in order; after the minibatch's last turn they
//     update velocity and parameters and write these into every CTA's copy.
// A cluster barrier closes every phase.
// What bounds it is the instructions of a warp's share, a serial chain of
// phases (256 threads per CTA: 3500 instructions per warp and minibatch of 256,
// 15.5 us; the sums over rows cannot be split further without another order).
constexpr int FC = 16, FT = 4;       // CTAs, tiles per turn
constexpr int FM = 512;              // threads per CTA
constexpr int FQ = FC / FT;          // quarters of a tile
constexpr int FR = TB / FQ;          // rows of a quarter
constexpr int FJ = NH / FQ;          // neurons of a quarter
// Larger minibatches keep more SMs busy in the chain than one cluster has:
// measured
// per epoch, cluster / chain: 10000 rows by 64 1349 / 5153 us, by 256 359 / 1318, by
// 1000 302 / 343; 16384 rows by 2048 460 / 267.
constexpr int FIT_MAX_BATCH = 1024;
// Shared-memory rows are padded so that 16-byte accesses of consecutive rows
// fall in distinct banks.
struct FitNet {
    alignas(16) float W1[NH][NIP];
    alignas(16) float W2[NH][NHP];
    alignas(16) float W3[NO][NHP];
    float b1[NH], b2[NH], b3[NO];
};
// A quarter's share of a tile's gradient, FSHARE floats: W2 rows, W1 rows, the
// W3 row, then the biases b2, b1, b3 and the sum of squares (quarter 0's).
constexpr int QS_W1 = FJ * NH, QS_W3 = QS_W1 + FJ * NI, QS_B2 = QS_W3 + NH, QS_B1 = QS_B2 + FJ,
              QS_B3 = QS_B1 + FJ, QS_LOSS = QS_B3 + 1, FSHARE = QS_LOSS + 1;
constexpr int FOWN = (FSHARE + FT - 1) / FT;  // of it, per CTA of the quarter
static_assert(FOWN <= FM && FQ == NO && NH % FQ == 0, "one entry per thread");
struct FitSmem {
    FitNet net;
    alignas(16) float X[2][TB][NIP];
    float T[2][FR][NO];
    alignas(16) float A1[TB][NHP];   // activations of the tile's rows
    alignas(16) float A2[TB][NHP];
    float D2q[TB][FJ + 1];           // dA2 and dA1 of the quarter's neurons
    float D1q[TB][FJ + 1];
    float Yq[TB];                    // dY of the quarter's output
    alignas(16) float D2[FR][NHP];   // dA2 of this CTA's rows
    float Y[FR][NO];                 // their dY
    float red[2 * FQ];               // squares of eight rows each (in quarter 0)
    alignas(16) float G[FSHARE];
};

// Parameter of entry e of quarter q's share (NPARAM: the loss, -1: none).
__device__ __forceinline__ int fit_param(int q, int e)
{
    if (e < QS_W1) return OFF_W2 + q * FJ * NH + e;
    if (e < QS_W3) return q * FJ * NI + (e - QS_W1);
    if (e < QS_B2) return OFF_W3 + q * NH + (e - QS_W3);
    if (e < QS_B1) return OFF_B2 + q * FJ + (e - QS_B2);
    if (e < QS_B3) return OFF_B1 + q * FJ + (e - QS_B1);
    if (e < QS_LOSS) return OFF_B3 + q;
    return e == QS_LOSS && q == 0 ? NPARAM : -1;
}
__device__ __forceinline__ float* fit_slot(FitNet& n, int p)
{
    if (p < OFF_B1) return &n.W1[p / NI][p % NI];
    if (p < OFF_W2) return &n.b1[p - OFF_B1];
    if (p < OFF_B2) return &n.W2[(p - OFF_W2) / NH][(p - OFF_W2) % NH];
    if (p < OFF_W3) return &n.b2[p - OFF_B2];
    if (p < OFF_B3) return &n.W3[(p - OFF_W3) / NH][(p - OFF_W3) % NH];
    return &n.b3[p - OFF_B3];
}

// Shared-memory address `a` in CTA `rank` of the cluster, and access to it.
__device__ __forceinline__ unsigned peer_addr(const void* a, unsigned rank)
{
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(a)), "r"(rank));
    return r;
}
__device__ __forceinline__ void peer_store(unsigned a, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ float peer_load(unsigned a)
{
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}

// This CTA's rows (`rows` of them real) of the tile in sm.X[buf]; quarter q of
// the tile is CTA rank0 + q.
__device__ __forceinline__ void fit_rows(FitSmem& sm, unsigned rank0, int quarter, int buf, int rows,
                                         float scale)
{
    const int t = threadIdx.x, j = t & (NH - 1);
    constexpr int RT = FR / (FM / NH);         // rows per thread
    const int s0 = (t / NH) * RT, r0 = quarter * FR;  // first row here, first row in the tile
    FitNet& n = sm.net;
    {
        float acc[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) acc[i] = n.b1[j];
#pragma unroll
        for (int k = 0; k < NI; k += 4) {
            const float4 w = *reinterpret_cast<const float4*>(&n.W1[j][k]);
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const float4 x = *reinterpret_cast<const float4*>(&sm.X[buf][r0 + s0 + i][k]);
                acc[i] = __fmaf_rn(w.x, x.x, acc[i]);
                acc[i] = __fmaf_rn(w.y, x.y, acc[i]);
                acc[i] = __fmaf_rn(w.z, x.z, acc[i]);
                acc[i] = __fmaf_rn(w.w, x.w, acc[i]);
            }
        }
#pragma unroll
        for (int q = 0; q < FQ; ++q) {
            const unsigned a = peer_addr(&sm.A1[r0 + s0][j], rank0 + q);
#pragma unroll
            for (int i = 0; i < RT; ++i) peer_store(a + i * (int)sizeof(sm.A1[0]), relu(acc[i]));
        }
    }
    __syncthreads();
    {
        float acc[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) acc[i] = n.b2[j];
#pragma unroll 4
        for (int k = 0; k < NH; k += 4) {
            const float4 w = *reinterpret_cast<const float4*>(&n.W2[j][k]);
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const float4 a = *reinterpret_cast<const float4*>(&sm.A1[r0 + s0 + i][k]);
                acc[i] = __fmaf_rn(w.x, a.x, acc[i]);
                acc[i] = __fmaf_rn(w.y, a.y, acc[i]);
                acc[i] = __fmaf_rn(w.z, a.z, acc[i]);
                acc[i] = __fmaf_rn(w.w, a.w, acc[i]);
            }
        }
#pragma unroll
        for (int q = 0; q < FQ; ++q) {
            const unsigned a = peer_addr(&sm.A2[r0 + s0][j], rank0 + q);
#pragma unroll
            for (int i = 0; i < RT; ++i) peer_store(a + i * (int)sizeof(sm.A2[0]), relu(acc[i]));
        }
    }
    __syncthreads();
    if (t < FR * NO) {  // outputs, their deltas and the squares of eight rows per warp
        const int s = t / NO, o = t % NO;
        float y = n.b3[o];
#pragma unroll 4
        for (int k = 0; k < NH; k += 4) {
            const float4 w = *reinterpret_cast<const float4*>(&n.W3[o][k]);
            const float4 a = *reinterpret_cast<const float4*>(&sm.A2[r0 + s][k]);
            y = __fmaf_rn(w.x, a.x, y);
            y = __fmaf_rn(w.y, a.y, y);
            y = __fmaf_rn(w.z, a.z, y);
            y = __fmaf_rn(w.w, a.w, y);
        }
        float sq = 0.0f, dy = 0.0f;
        if (s < rows) {
            const float res = __fsub_rn(y, sm.T[buf][s][o]);
            sq = __fmul_rn(res, res);
            dy = __fmul_rn(scale, res);
        }
        sm.Y[s][o] = dy;
        peer_store(peer_addr(&sm.Yq[r0 + s], rank0 + o), dy);
#pragma unroll
        for (int off = 16; off; off >>= 1) sq = __fadd_rn(sq, __shfl_xor_sync(FULL, sq, off));
        if ((t & 31) == 0) peer_store(peer_addr(&sm.red[2 * quarter + (t >> 5)], rank0), sq);
    }
    __syncthreads();
    const unsigned d2 = peer_addr(&sm.D2q[r0 + s0][j % FJ], rank0 + j / FJ);
#pragma unroll
    for (int i = 0; i < RT; ++i) {  // dA2[s][j] = (sum_o dY[s][o] W3[o][j]) [H2 > 0]
        const int s = s0 + i;
        float a = 0.0f;
#pragma unroll
        for (int o = 0; o < NO; ++o) a = __fadd_rn(a, __fmul_rn(sm.Y[s][o], n.W3[o][j]));
        const float d = sm.A2[r0 + s][j] > 0.0f ? a : 0.0f;
        sm.D2[s][j] = d;
        peer_store(d2 + i * (int)sizeof(sm.D2q[0]), d);
    }
    __syncthreads();
    {  // dA1[s][k] = (sum_j dA2[s][j] W2[j][k]) [H1 > 0] (k = this thread's j)
        float acc[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) acc[i] = 0.0f;
#pragma unroll 4
        for (int jj = 0; jj < NH; jj += 4) {
            const float w0 = n.W2[jj][j], w1 = n.W2[jj + 1][j], w2 = n.W2[jj + 2][j], w3 = n.W2[jj + 3][j];
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const float4 d = *reinterpret_cast<const float4*>(&sm.D2[s0 + i][jj]);
                acc[i] = __fadd_rn(acc[i], __fmul_rn(d.x, w0));
                acc[i] = __fadd_rn(acc[i], __fmul_rn(d.y, w1));
                acc[i] = __fadd_rn(acc[i], __fmul_rn(d.z, w2));
                acc[i] = __fadd_rn(acc[i], __fmul_rn(d.w, w3));
            }
        }
        const unsigned d1 = peer_addr(&sm.D1q[r0 + s0][j % FJ], rank0 + j / FJ);
#pragma unroll
        for (int i = 0; i < RT; ++i)
            peer_store(d1 + i * (int)sizeof(sm.D1q[0]), sm.A1[r0 + s0 + i][j] > 0.0f ? acc[i] : 0.0f);
    }
}

// This quarter's share of the tile's gradient, rows in order.
__device__ __forceinline__ void fit_sums(FitSmem& sm, int quarter, int buf)
{
    const int t = threadIdx.x;
    constexpr int HT = FM / 2;
    const int u = t % HT, j = u >> 4, k = u & 15;
    static_assert(HT == FJ * 16 && NI == 16 && NH == 64, "thread mapping");
    if (t < HT) {  // W2: neuron j, inputs 4 k .. 4 k + 3
        float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f, a3 = 0.0f;
#pragma unroll 8
        for (int s = 0; s < TB; ++s) {
            const float d2 = sm.D2q[s][j];
            const float4 a = *reinterpret_cast<const float4*>(&sm.A1[s][4 * k]);
            a0 = __fadd_rn(a0, __fmul_rn(d2, a.x));
            a1 = __fadd_rn(a1, __fmul_rn(d2, a.y));
            a2 = __fadd_rn(a2, __fmul_rn(d2, a.z));
            a3 = __fadd_rn(a3, __fmul_rn(d2, a.w));
        }
        *reinterpret_cast<float4*>(&sm.G[j * NH + 4 * k]) = make_float4(a0, a1, a2, a3);
        return;
    }
    // W1: neuron j, input k; some threads one more sum: the W3 row, then the
    // biases b2, b1, b3 (which follow one another in the share)
    float w1 = 0.0f, e = 0.0f;
#pragma unroll 8
    for (int s = 0; s < TB; ++s) w1 = __fadd_rn(w1, __fmul_rn(sm.D1q[s][j], sm.X[buf][s][k]));
    sm.G[QS_W1 + j * NI + k] = w1;
    if (u < NH) {
#pragma unroll 8
        for (int s = 0; s < TB; ++s) e = __fadd_rn(e, __fmul_rn(sm.Yq[s], sm.A2[s][u]));
    } else if (u < NH + 2 * FJ + 1) {
        const int b = u - NH;  // a column of D2q, of D1q, or Yq
        const float* const src = b < FJ ? &sm.D2q[0][b] : b < 2 * FJ ? &sm.D1q[0][b - FJ] : sm.Yq;
        const int stride = b < 2 * FJ ? FJ + 1 : 1;
#pragma unroll 8
        for (int s = 0; s < TB; ++s) e = __fadd_rn(e, src[s * stride]);
    } else if (u == HT - 1 && quarter == 0) {
#pragma unroll
        for (int w = 0; w < 2 * FQ; ++w) e = __fadd_rn(e, sm.red[w]);
    }
    if (u < NH + 2 * FJ + 1) sm.G[QS_W3 + u] = e;
    else if (u == HT - 1) sm.G[QS_LOSS] = e;
}

__global__ void __launch_bounds__(FM, 1) k_mlp_fit(float* P, float* V, float* grad, const float* norm,
                                                const float* X, const float* T, const int* idx,
                                                int N, int batch, float lr, float momentum,
                                                float* losses)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) uint8_t raw[];
    FitSmem& sm = *reinterpret_cast<FitSmem*>(raw);
    const int t = threadIdx.x, c = (int)cluster.block_rank();
    const int tile = c / FQ, quarter = c % FQ;
    for (int p = t; p < NPARAM; p += FM) *fit_slot(sm.net, p) = P[p];
    // this thread's entry of the quarter's share, its parameter and its place
    const int ent = t < FOWN && tile * FOWN + t < FSHARE ? tile * FOWN + t : -1;
    const int par = ent >= 0 ? fit_param(quarter, ent) : -1;
    const bool trained = par >= 0 && par < NPARAM;
    float pv = trained ? P[par] : 0.0f, vv = trained ? V[par] : 0.0f;
    const float* const slot = trained ? fit_slot(sm.net, par) : nullptr;
    const int k = t % NI, xr = t / NI;  // input of this thread, its rows xr + 16 i of the tile
    constexpr int XI = TB * NI / FM;
    static_assert(FM % NI == 0 && NO * FR <= FM, "input elements per thread");
    const int ts = t / NO, to = t % NO;  // target of the threads below FR * NO
    const bool has_t = t < FR * NO;
    const float nm = norm[k], ni = norm[NI + k];
    const int steps = (N + batch - 1) / batch;
    // Row r of this CTA's tile in turn q of minibatch m: its place in idx, or -1.
    auto place = [&](int m, int q, int r) {
        if (m >= steps) return -1;
        const int b = (q * FT + tile) * TB + r;
        return b < min(batch, N - m * batch) ? m * batch + b : -1;
    };
    auto next = [&](int& m, int& q) {
        if (m < steps && ++q * FT * TB >= min(batch, N - m * batch)) {
            q = 0;
            ++m;
        }
    };
    // Inputs are fetched a turn ahead, their row numbers two turns ahead.
    int rx[XI], rt;
    auto fetch_rows = [&](int m, int q) {
#pragma unroll
        for (int i = 0; i < XI; ++i) {
            const int at = place(m, q, xr + (FM / NI) * i);
            rx[i] = at >= 0 ? idx[at] : -1;
        }
        const int at = has_t ? place(m, q, quarter * FR + ts) : -1;
        rt = at >= 0 ? idx[at] : -1;
    };
    float xv[XI], tv;
    auto fetch = [&] {
#pragma unroll
        for (int i = 0; i < XI; ++i)
            xv[i] = rx[i] >= 0 ? X[(long long)rx[i] * NI + k] : nm;  // (normalises to 0)
        tv = rt >= 0 ? T[(long long)rt * NO + to] : 0.0f;
    };
    auto put = [&](int buf) {
#pragma unroll
        for (int i = 0; i < XI; ++i)  // normalised here, when the loads have long arrived
            sm.X[buf][xr + (FM / NI) * i][k] = __fmul_rn(__fsub_rn(xv[i], nm), ni);
        if (has_t) sm.T[buf][ts][to] = tv;
    };
    int m2 = 0, q2 = 0;  // the turn whose row numbers are fetched next
    fetch_rows(m2, q2);
    next(m2, q2);
    fetch();
    put(0);
    fetch_rows(m2, q2);
    next(m2, q2);
    int buf = 0;
    cluster.sync();
    for (int m = 0; m < steps; ++m) {
        const int B = min(batch, N - m * batch);
        const float scale = 2.0f / (float)(B * NO);
        float acc = 0.0f;
        for (int b0 = 0; b0 < B; b0 += FT * TB, buf ^= 1) {
            fetch();
            fetch_rows(m2, q2);
            next(m2, q2);
            const int tiles = min(FT, (B - b0 + TB - 1) / TB);  // of this turn
            if (tile < tiles)
                fit_rows(sm, tile * FQ, quarter, buf, min(FR, max(0, B - b0 - tile * TB - quarter * FR)), scale);
            put(buf ^ 1);
            cluster.sync();  // the tiles' rows are complete
            if (tile < tiles) fit_sums(sm, quarter, buf);
            cluster.sync();  // the tiles' sums are complete, nobody reads the parameters
            if (ent >= 0) {
                float g[FT];
#pragma unroll
                for (int r = 0; r < FT; ++r)
                    if (r < tiles) g[r] = peer_load(peer_addr(&sm.G[ent], r * FQ + quarter));
#pragma unroll
                for (int r = 0; r < FT; ++r)
                    if (r < tiles) acc = __fadd_rn(acc, g[r]);
            }
        }
        if (trained) {
            vv = __fadd_rn(__fmul_rn(momentum, vv), acc);
            pv = __fsub_rn(pv, __fmul_rn(lr, vv));
#pragma unroll
            for (int r = 0; r < FC; ++r) peer_store(peer_addr(slot, r), pv);
            if (m + 1 == steps) {
                P[par] = pv;
                V[par] = vv;
                grad[par] = acc;
            }
        } else if (par == NPARAM) {
            losses[m] = acc / (float)(B * NO);
        }
        cluster.sync();
    }
}

// ---- selection: one thread per item -------------------------------------------------
struct SelectArgs {
    float link, c[4], c_raw, judge, judge_time;
};

// With `pred_time`, a message's coded cost at L_k takes its own predicted ns
// per input byte, 2^pred_time[k], where that prediction is finite and within
// judge_time (log2) of the batch-wide rate c[k]; elsewhere c[k] stays.
__global__ void k_select(Item* items, unsigned n_items, const float* feat, const float* pred,
                         const float* pred_time, SelectArgs a, int* choice, unsigned* counts)
{
    grid_dep_wait();
    grid_dep_launch();
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_items) return;
    Item& it = items[i];
    const float nf = (float)it.n;
    const float bytes_in = nf * (it.x_dtype == ZC_F32 ? 4.0f : 2.0f);
    const float* f = feat + (size_t)i * N_STATS;
    const float cost_raw = __fadd_rn(__fmul_rn(bytes_in, a.c_raw), __fdiv_rn(__fadd_rn(32.0f, bytes_in), a.link));
    // the heuristic: L = 32 unless the sampled estimate says coding does not pay
    int h = 0;
    if (isfinite(f[1])) {
        const float c32 = __fadd_rn(__fmul_rn(bytes_in, a.c[1]),
                                    __fdiv_rn(__fdiv_rn(__fmul_rn(nf, f[1]), 8.0f), a.link));
        h = c32 < cost_raw ? 32 : 0;
    }
    int c = h;
    bool fell_back = false;
    if (pred != nullptr) {
        const float* y = pred + (size_t)i * NO;
        bool ok = true;
        for (int k = 0; k < 4; ++k) ok = ok && isfinite(y[k]) && isfinite(f[k]);
        if (ok) {
            int kb = 0;
            float best = 0.0f;
            for (int k = 0; k < 4; ++k) {
                const float bits = exp2f(y[k]);
                float rate = a.c[k];
                if (pred_time != nullptr) {
                    const float t = pred_time[(size_t)i * NO + k];
                    if (isfinite(t) && fabsf(__fsub_rn(t, log2f(a.c[k]))) <= a.judge_time)
                        rate = exp2f(t);
                }
                const float ck = __fadd_rn(__fmul_rn(bytes_in, rate),
                                           __fdiv_rn(__fdiv_rn(__fmul_rn(nf, bits), 8.0f), a.link));
                if (k == 0 || ck < best) {
                    best = ck;
                    kb = k;
                }
            }
            if (fabsf(__fsub_rn(y[kb], log2f(f[kb]))) > a.judge) fell_back = true;
            else c = best < cost_raw ? (16 << kb) : 0;
        } else {
            fell_back = true;
        }
    }
    if (!(it.two_eb > 0.0f)) c = 0;  // planned without a bound: raw only
    it.log2L = c == 16 ? 4 : c == 32 ? 5 : c == 64 ? 6 : c == 128 ? 7 : -1;
    if (choice != nullptr) choice[i] = c;
    if (counts != nullptr) {
        if (fell_back) atomicAdd(counts, 1u);
        if (c == 0) atomicAdd(counts + 1, 1u);
    }
}

}  // namespace zc

using namespace zc;

extern "C" {

int zc_batch_chunk_stats(const zc_batch* plan, float* d_feat, zc_stream_t s)
{
    if (plan == nullptr || plan->d_table == nullptr || plan->n_msgs < 1 || plan->decompress != 0 ||
        d_feat == nullptr || (reinterpret_cast<uintptr_t>(d_feat) & 3) != 0)
        return ZC_ERR_ARG;
    const unsigned n = (unsigned)plan->n_msgs;
    return launch_after(k_chunk_stats, (n + 7) / 8, 256, 0, (cudaStream_t)s, (const Item*)plan->d_table, n,
                        d_feat) == cudaSuccess
               ? ZC_OK
               : ZC_ERR_CUDA;
}

static cudaError_t mlp_prepare()
{
    const cudaError_t e1 = smem_limit<k_mlp_forward>((int)sizeof(MlpSmem));
    const cudaError_t e2 = smem_limit<k_mlp_grad>((int)sizeof(MlpSmem));
    return e1 != cudaSuccess ? e1 : e2;
}

int zc_mlp_forward(const float* d_params, const float* d_norm, const float* d_x, int B,
                   float* d_y, zc_stream_t s)
{
    if (d_params == nullptr || d_norm == nullptr || B < 0 || (B > 0 && (d_x == nullptr || d_y == nullptr)))
        return ZC_ERR_ARG;
    if (B == 0) return ZC_OK;
    if (mlp_prepare() != cudaSuccess) return ZC_ERR_CUDA;
    // two CTAs per SM fit (shared memory), each looping over row tiles
    int dev = 0, n_sm = 152;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return ZC_ERR_CUDA;
    const int ntiles = (B + TB - 1) / TB;
    const int grid = ntiles < 2 * n_sm ? ntiles : 2 * n_sm;
    return launch_after(k_mlp_forward, (unsigned)grid, MT, (int)sizeof(MlpSmem), (cudaStream_t)s, d_params,
                        d_norm, d_x, B, d_y) == cudaSuccess
               ? ZC_OK
               : ZC_ERR_CUDA;
}

size_t zc_mlp_scratch_bytes(int B)
{
    if (B < 1) return 0;
    return (size_t)((B + TB - 1) / TB) * NPAD * sizeof(float);
}

int zc_mlp_grad(const float* d_params, const float* d_norm, const float* d_x, const float* d_t,
                const int* d_idx, int B, float* d_grad, float* d_loss, void* d_scratch,
                size_t scratch_bytes, zc_stream_t s)
{
    if (d_params == nullptr || d_norm == nullptr || d_x == nullptr || d_t == nullptr || B < 1 ||
        d_grad == nullptr || d_scratch == nullptr || scratch_bytes < zc_mlp_scratch_bytes(B) ||
        (reinterpret_cast<uintptr_t>(d_scratch) & 3) != 0)
        return ZC_ERR_ARG;
    if (mlp_prepare() != cudaSuccess) return ZC_ERR_CUDA;
    const int nct = (B + TB - 1) / TB;
    k_mlp_grad<<<nct, MT, sizeof(MlpSmem), (cudaStream_t)s>>>(d_params, d_norm, d_x, d_t, d_idx, B,
                                                             (float*)d_scratch);
    if (cudaGetLastError() != cudaSuccess) return ZC_ERR_CUDA;
    k_mlp_reduce<<<(NPARAM + 1 + 255) / 256, 256, 0, (cudaStream_t)s>>>((const float*)d_scratch, nct,
                                                                       B, d_grad, d_loss);
    return cudaGetLastError() == cudaSuccess ? ZC_OK : ZC_ERR_CUDA;
}

int zc_mlp_sgd(float* d_params, float* d_vel, const float* d_grad, float lr, float momentum,
               zc_stream_t s)
{
    if (d_params == nullptr || d_vel == nullptr || d_grad == nullptr) return ZC_ERR_ARG;
    k_mlp_sgd<<<(NPARAM + 255) / 256, 256, 0, (cudaStream_t)s>>>(d_params, d_vel, d_grad, lr,
                                                                 momentum);
    return cudaGetLastError() == cudaSuccess ? ZC_OK : ZC_ERR_CUDA;
}

// Whether the current device runs a cluster of this launch (a partition of a GPU
// may have no room for one of this size); asked once per device.
static bool fit_cluster(const cudaLaunchConfig_t& cfg)
{
    static std::atomic<int> known[64];  // 0: not asked, 1: yes, 2: no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    std::atomic<int>* const k = dev >= 0 && dev < 64 ? &known[dev] : nullptr;
    if (k != nullptr && k->load(std::memory_order_acquire) != 0) return k->load(std::memory_order_acquire) == 1;
    int clusters = 0;
    const bool ok = smem_limit<k_mlp_fit>((int)sizeof(FitSmem)) == cudaSuccess &&
                    cudaFuncSetAttribute(k_mlp_fit, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&clusters, k_mlp_fit, &cfg) == cudaSuccess && clusters > 0;
    if (!ok) cudaGetLastError();
    if (k != nullptr) k->store(ok ? 1 : 2, std::memory_order_release);
    return ok;
}

int zc_mlp_fit_epoch(float* d_params, float* d_vel, float* d_grad, const float* d_norm,
                     const float* d_x, const float* d_t, const int* d_idx, int N, int batch,
                     double lr, double momentum, float* d_losses, void* d_scratch,
                     size_t scratch_bytes, zc_stream_t s)
{
    if (N < 0 || batch < 1) return ZC_ERR_ARG;
    if (N == 0) return ZC_OK;
    if (d_params == nullptr || d_vel == nullptr || d_grad == nullptr || d_norm == nullptr ||
        d_x == nullptr || d_t == nullptr || d_idx == nullptr || d_losses == nullptr)
        return ZC_ERR_ARG;
    if (batch > N) batch = N;
    // (whichever way the epoch runs: what is valid does not depend on the device)
    if (d_scratch == nullptr || scratch_bytes < zc_mlp_scratch_bytes(batch) ||
        (reinterpret_cast<uintptr_t>(d_scratch) & 3) != 0)
        return ZC_ERR_ARG;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(FC);
    cfg.blockDim = dim3(FM);
    cfg.dynamicSmemBytes = sizeof(FitSmem);
    cfg.stream = (cudaStream_t)s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = FC;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (batch > FIT_MAX_BATCH || !fit_cluster(cfg)) {
        for (int m = 0; (long long)m * batch < N; ++m) {
            const int B = N - m * batch < batch ? N - m * batch : batch;
            int st = zc_mlp_grad(d_params, d_norm, d_x, d_t, d_idx + (size_t)m * batch, B, d_grad,
                                 d_losses + m, d_scratch, scratch_bytes, s);
            if (st == ZC_OK) st = zc_mlp_sgd(d_params, d_vel, d_grad, (float)lr, (float)momentum, s);
            if (st != ZC_OK) return st;
        }
        return ZC_OK;
    }
    return cudaLaunchKernelEx(&cfg, k_mlp_fit, d_params, d_vel, d_grad, d_norm, d_x, d_t, d_idx, N,
                              batch, (float)lr, (float)momentum, d_losses) == cudaSuccess
               ? ZC_OK
               : ZC_ERR_CUDA;
}

int zc_batch_select_timed(const zc_batch* plan, const float* d_feat, const float* d_pred,
                          const float* d_pred_time, const zc_select_cfg* cfg, int* d_choice,
                          unsigned* d_counts, zc_stream_t s)
{
    if (plan == nullptr || plan->d_table == nullptr || plan->n_msgs < 1 || plan->decompress != 0 ||
        d_feat == nullptr || cfg == nullptr || !(cfg->link_gbs > 0.0f) || !(cfg->judge_log2 >= 0.0f))
        return ZC_ERR_ARG;
    if (d_pred_time != nullptr && (d_pred == nullptr || !(cfg->judge_time_log2 >= 0.0f)))
        return ZC_ERR_ARG;
    SelectArgs a;
    a.link = cfg->link_gbs;
    for (int k = 0; k < 4; ++k) a.c[k] = cfg->ns_per_byte[k];
    a.c_raw = cfg->raw_ns_per_byte;
    a.judge = cfg->judge_log2;
    a.judge_time = d_pred_time != nullptr ? cfg->judge_time_log2 : 0.0f;
    if (d_counts != nullptr &&
        cudaMemsetAsync(d_counts, 0, 2 * sizeof(unsigned), (cudaStream_t)s) != cudaSuccess)
        return ZC_ERR_CUDA;
    const unsigned n = (unsigned)plan->n_msgs;
    return launch_after(k_select, (n + 255) / 256, 256, 0, (cudaStream_t)s, (Item*)plan->d_table, n, d_feat,
                        d_pred, d_pred_time, a, d_choice, d_counts) == cudaSuccess
               ? ZC_OK
               : ZC_ERR_CUDA;
}

int zc_batch_select(const zc_batch* plan, const float* d_feat, const float* d_pred,
                    const zc_select_cfg* cfg, int* d_choice, unsigned* d_counts, zc_stream_t s)
{
    return zc_batch_select_timed(plan, d_feat, d_pred, nullptr, cfg, d_choice, d_counts, s);
}

}  // extern "C"
