// zc_rows.cuh -- the codec's arithmetic, one row of 32 elements per lane.
//
// A warp works on a group of 32 rows of 32 elements (1024 elements): lane r
// owns row r, so a block of L = 32 elements is one lane, L = 64 and 128 are 2
// and 4 neighbouring lanes, and L = 16 is half a lane's row.  Deltas, bit
// planes, widths and prefix sums then need no shuffles at all (L = 64 and
// 128: one to three per row for what crosses lanes), where a lane per element
// needs five shuffles per transpose and five per prefix sum of every row.
// What bounds the codec kernels is instruction issue, and this is the layout
// with the fewest instructions per element:
//   - quantization on pairs (fma/add.f32x2) with a residual test, 2.5 per
//     element; the test's largest values by three-operand maxima;
//   - deltas on packed pairs: t_j + 2^16 t_(j+16) differ by d_j + 2^16
//     d_(j+16), one subtraction for two elements;
//   - planes by 8 x 8 bit transposes inside eight words (48 instructions per
//     32 elements and byte of width), the sign and magnitude split on whole
//     planes (two instructions per plane instead of two per element).
// Measured against one element per lane (512^3 FP32 field, REL 1e-3, L = 32):
// decompression 162 -> 120 us, range pass and compression 314 -> 267.
//
// Values reach the lanes through a group buffer in shared memory: 32 rows of
// 128 bytes (FP32) whose 16-byte chunks are permuted by the row number (chunk
// c of row r at c ^ (r & 7)), so that the coalesced side (consecutive chunks
// by consecutive lanes) and the row side (the same chunk of 8 rows by 8
// lanes) are both free of bank conflicts.  BF16 rows are 64 bytes, chunk c of
// row r at c ^ ((r >> 1) & 3).
#pragma once

#include "zc_device.cuh"

namespace zc {

constexpr int GROWS = 32;             // rows of a group, one per lane
constexpr int GELEMS = GROWS * 32;    // elements of a group
constexpr int GBUF = GROWS * 128;     // bytes of a group buffer (FP32 rows)
// Largest payload of a group (25 planes everywhere) behind at most 15 carried
// bytes: it is staged in the buffer that held the group's values.
static_assert(15 + GROWS * 100 + 16 <= GBUF, "payload fits the group buffer");

// ---- packed FP32 and shared-memory access -----------------------------------

using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pk2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void up2(f32x2 v, float& a, float& b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// Largest magnitude of three; the second form keeps a NaN.
__device__ __forceinline__ float max3_abs(float a, float b, float c)
{
    float r;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float max3_abs_nan(float a, float b, float c)
{
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

__device__ __forceinline__ uint4 lds128(unsigned a)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(a)
                 : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds32(unsigned a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds16(unsigned a)
{
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts128(unsigned a, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w)
                 : "memory");
}
__device__ __forceinline__ void sts64(unsigned a, uint32_t x, uint32_t y)
{
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void sts32(unsigned a, uint32_t x)
{
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}
__device__ __forceinline__ void sts16(unsigned a, uint32_t x)
{
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((unsigned short)x) : "memory");
}
__device__ __forceinline__ void sts8(unsigned a, uint32_t x)
{
    asm volatile("{\n\t.reg .b16 h;\n\tcvt.u16.u32 h, %1;\n\tst.shared.u8 [%0], h;\n\t}" ::"r"(a), "r"(x)
                 : "memory");
}

// ---- asynchronous copies into a group buffer ----------------------------------

__device__ __forceinline__ void cp_async16(unsigned dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst),
                 "l"(__cvta_generic_to_global(src))
                 : "memory");
}
// The same for data that is read once: its lines are the first to leave L2.
// An encoder's input goes past the staged payloads that wait in L2 for their
// place; without the hint it displaces them (compression of the 512^3 field,
// REL 1e-3, L = 32: 176 us without, 153 us with it, nothing else changed).
__device__ __forceinline__ void cp_async16_once(unsigned dst, const void* src)
{
    asm volatile(
        "{\n\t.reg .b64 pol;\n\t"
        "createpolicy.fractional.L2::evict_first.b64 pol, 1.0;\n\t"
        "cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, pol;\n\t}" ::"r"(dst),
        "l"(__cvta_generic_to_global(src))
        : "memory");
}
__device__ __forceinline__ void cp_async4_once(unsigned dst, const void* src)
{
    asm volatile(
        "{\n\t.reg .b64 pol;\n\t"
        "createpolicy.fractional.L2::evict_first.b64 pol, 1.0;\n\t"
        "cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 4, pol;\n\t}" ::"r"(dst),
        "l"(__cvta_generic_to_global(src))
        : "memory");
}
template <int W>
__device__ __forceinline__ void cp_async_ca(unsigned dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst),
                 "l"(__cvta_generic_to_global(src)), "n"(W)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Shared-memory address of element e of the group in buffer `buf`.
template <typename T>
__device__ __forceinline__ unsigned elem_addr(unsigned buf, int e)
{
    const int r = e >> 5, i = e & 31;
    if (sizeof(T) == 4) return buf + r * 128 + (((i >> 2) ^ (r & 7)) << 4) + (i & 3) * 4;
    return buf + r * 64 + (((i >> 3) ^ ((r >> 1) & 3)) << 4) + (i & 7) * 2;
}

// The same of 4-byte word 32 k + lane (one FP32 or two BF16 elements): with k
// known at compile time, one XOR per eight (four) words and an immediate.
template <typename T>
__device__ __forceinline__ unsigned word_addr(unsigned buf, int k)
{
    const unsigned lane = threadIdx.x & 31;
    return ((buf + 4 * lane) ^ ((unsigned)(k & (sizeof(T) == 4 ? 7 : 3)) << 4)) + k * 128;
}

// Brings the group's elements into `buf` (one commit group): p[0 .. nrem), nrem
// what is left of the warp's unit; elements past nrem repeat the last one: their
// deltas are then zero, as the format's padding asks.  vec: p is 16-byte aligned;
// first: nothing of the input lies before p.  A whole aligned group takes 16-byte
// copies, a whole group at a multiple of 4 bytes 4-byte copies.  A whole BF16 group
// at an odd element loads aligned words and joins their halves, where the unit goes
// on behind it and the input has an element before it (the words reach one element
// beyond either end): all but the last group of a unit, the only one of 32-row
// units.  That one, the input's first and ragged groups go element by element.  (A
// relative-bound scatter pack of 200 MB in 8 segments that start anywhere took 194
// us with clamped single-element copies of every group and the range pass reading
// by elements, and takes 101.)
template <typename T>
__device__ __forceinline__ void stage_in(const T* p, int nrem, bool vec, unsigned buf, bool first)
{
    const int lane = threadIdx.x & 31;
    constexpr int WPL = GELEMS * sizeof(T) / 128;  // words per lane
    if (vec && nrem >= GELEMS) {
        constexpr int CPR = 32 * sizeof(T) / 16;  // chunks per row
        constexpr int RPI = 32 / CPR;             // rows per instruction
        const int c = lane & (CPR - 1), r0 = lane / CPR;
        const uint8_t* src = (const uint8_t*)p + lane * 16;
#pragma unroll
        for (int k = 0; k < CPR; ++k) {
            const int r = k * RPI + r0;
            const unsigned sw = sizeof(T) == 4 ? (unsigned)(r & 7) : (unsigned)((r >> 1) & 3);
            cp_async16_once(buf + r * (int)(32 * sizeof(T)) + ((c ^ sw) << 4), src + k * 512);
        }
    } else if (nrem >= GELEMS && ((uintptr_t)p & 3u) == 0) {
        const uint8_t* const src = (const uint8_t*)p + lane * 4;
#pragma unroll
        for (int k = 0; k < WPL; ++k) cp_async4_once(word_addr<T>(buf, k), src + k * 128);
    } else if (sizeof(T) == 2 && nrem > GELEMS && !first) {
        const unsigned* const src = (const unsigned*)((const uint8_t*)p - 2) + lane;
#pragma unroll 1
        for (int k0 = 0; k0 < WPL; k0 += 4) {
            uint32_t a[4], b[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                a[k] = ld_dep_once(src + 32 * (k0 + k));
                b[k] = ld_dep_once(src + 32 * (k0 + k) + 1);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) sts32(word_addr<T>(buf, k0 + k), __funnelshift_r(a[k], b[k], 16));
        }
    } else if (sizeof(T) == 4) {
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
            const int e = k * 32 + lane;
            cp_async_ca<4>(elem_addr<T>(buf, e), p + min(e, nrem - 1));
        }
    } else {
#pragma unroll 1
        for (int k0 = 0; k0 < 32; k0 += 8) {
            uint32_t v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                v[k] = ld_dep((const unsigned short*)p + min((k0 + k) * 32 + lane, nrem - 1));
#pragma unroll
            for (int k = 0; k < 8; ++k) sts16(elem_addr<T>(buf, (k0 + k) * 32 + lane), v[k]);
        }
    }
    cp_commit();
}

// Stores the group's elements buf[0 .. nrem) to p (coalesced); vec: p is
// 16-byte aligned.  Whole groups at other places go by 4-byte words, or by
// single BF16 elements at an odd one.
template <typename T>
__device__ __forceinline__ void stage_out(T* p, int nrem, bool vec, unsigned buf)
{
    const int lane = threadIdx.x & 31;
    if (vec && nrem >= GELEMS) {
        constexpr int CPR = 32 * sizeof(T) / 16;
        constexpr int RPI = 32 / CPR;
        const int c = lane & (CPR - 1), r0 = lane / CPR;
#pragma unroll
        for (int k = 0; k < CPR; ++k) {
            const int r = k * RPI + r0;
            const unsigned sw = sizeof(T) == 4 ? (unsigned)(r & 7) : (unsigned)((r >> 1) & 3);
            const uint4 v = lds128(buf + r * (int)(32 * sizeof(T)) + ((c ^ sw) << 4));
            *(uint4*)((uint8_t*)p + k * 512 + lane * 16) = v;
        }
    } else if (nrem >= GELEMS && ((uintptr_t)p & 3u) == 0) {
#pragma unroll 8
        for (int k = 0; k < (int)(GELEMS * sizeof(T) / 128); ++k)
            *((uint32_t*)((uint8_t*)p + k * 128) + lane) = lds32(word_addr<T>(buf, k));
    } else {
#pragma unroll 4
        for (int k = 0; k < 32; ++k) {
            const int e = k * 32 + lane;
            if (e < nrem) {
                if (sizeof(T) == 4) *((uint32_t*)p + e) = lds32(elem_addr<T>(buf, e));
                else *((unsigned short*)p + e) = (unsigned short)lds16(elem_addr<T>(buf, e));
            }
        }
    }
}

// ---- bit transposes -----------------------------------------------------------
// Eight words, four bytes each: bit p of byte b of word k <-> bit k of byte b
// of word p (its own inverse).  Word k holds in byte b a byte of element
// 8 b + k, so that plane word p has element e at bit e.
__device__ __forceinline__ void t8(uint32_t w[8])
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t a = w[k], b = w[k + 4];
        w[k] = (a & 0x0f0f0f0fu) | ((b << 4) & 0xf0f0f0f0u);
        w[k + 4] = ((a >> 4) & 0x0f0f0f0fu) | (b & 0xf0f0f0f0u);
    }
#pragma unroll
    for (int h = 0; h < 8; h += 4)
#pragma unroll
        for (int k = h; k < h + 2; ++k) {
            const uint32_t a = w[k], b = w[k + 2];
            w[k] = (a & 0x33333333u) | ((b << 2) & 0xccccccccu);
            w[k + 2] = ((a >> 2) & 0x33333333u) | (b & 0xccccccccu);
        }
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
        const uint32_t a = w[k], b = w[k + 1];
        w[k] = (a & 0x55555555u) | ((b << 1) & 0xaaaaaaaau);
        w[k + 1] = ((a >> 1) & 0x55555555u) | (b & 0xaaaaaaaau);
    }
}
// One plane of two's complement with sign plane s and running carry c (c = s
// before the lowest plane) -> the magnitude plane.  The same step turns
// magnitude planes into two's complement.
__device__ __forceinline__ uint32_t neg_plane(uint32_t d, uint32_t s, uint32_t& c)
{
    const uint32_t m = d ^ s ^ c;
    c = (d ^ s) & c;
    return m;
}

// ---- encoding -------------------------------------------------------------------

// What a lane's row needs of its neighbours and of the stream.
struct EncArgs {
    unsigned buf;       // the group buffer (values in, payload out)
    int nrem;           // valid elements of the group (1 .. 1024)
    float eb, two_eb, inv;
    int r0;             // bytes carried from the group before (0 .. 15)
    uint32_t carry;     // lanes 0 .. 3: those bytes, as words
    unsigned wb;        // width bytes of the group (shared memory)
    uint8_t* hout;      // heads apart: the group's head fields
};

// Rows per block and the block size in bytes per plane.
template <int LOG2L>
struct Blk {
    static constexpr int L = 1 << LOG2L;
    static constexpr int RPB = L >= 32 ? L / 32 : 1;
};

// Payload places of the group's rows: np planes of the lane's row (np2: the
// second block of the row at L = 16), raised to the block's.  Writes the width bytes and the carried bytes,
// returns the group's payload size; `at`: the lane's byte offset in the
// buffer of its block's plane 0 (its own word of it at L = 64, 128).
template <int LOG2L>
__device__ __forceinline__ int place_rows(const EncArgs& A, int& np, int np2, unsigned& at)
{
    constexpr int L = Blk<LOG2L>::L, RPB = Blk<LOG2L>::RPB;
    const int lane = threadIdx.x & 31;
    if (L >= 64) np = max(np, __shfl_xor_sync(FULL, np, 1));
    if (L >= 128) np = max(np, __shfl_xor_sync(FULL, np, 2));
    const int sz = L == 16 ? 2 * (np + np2) : 4 * np;
    const int s = scan_incl<32>(sz);
    const int tot = __shfl_sync(FULL, s, 31);
    const int sub = lane & (RPB - 1);
    at = A.buf + A.r0 + (s - sz) - sub * sz + 4 * sub;
    // width bytes (0 for no planes, else planes - 1)
    const uint32_t w = (uint32_t)max(np - 1, 0);
    if (L == 16) sts16(A.wb + 2 * lane, w | ((uint32_t)max(np2 - 1, 0) << 8));
    else if (sub == 0) sts8(A.wb + lane / RPB, w);
    return tot;
}

// Before the payload is written over the values: every lane has read its row;
// the carried bytes go first (at L = 16 their last word is shared with the
// first plane).
__device__ __forceinline__ void open_payload(const EncArgs& A)
{
    __syncwarp();
    if ((threadIdx.x & 31) < 4) sts32(A.buf + 4 * (threadIdx.x & 31), A.carry);
    __syncwarp();
}

// Plane k of the lane's block(s).
template <int LOG2L>
__device__ __forceinline__ void put_plane(unsigned at, int k, uint32_t v, int np, int np2)
{
    constexpr int L = Blk<LOG2L>::L, RPB = Blk<LOG2L>::RPB;
    if (L == 16) {
        if (k < np) sts16(at + 2 * k, v & 0xffffu);
        if (k < np2) sts16(at + 2 * np + 2 * k, v >> 16);
    } else {
        if (k < np) sts32(at + 4 * RPB * k, v);
    }
}

// Planes of the lane's block(s) from its sign plane and NM magnitude planes.
template <int LOG2L, int NM>
__device__ __forceinline__ int put_planes(const EncArgs& A, uint32_t S, const uint32_t (&m)[NM])
{
    constexpr int L = Blk<LOG2L>::L, RPB = Blk<LOG2L>::RPB;
    const int lane = threadIdx.x & 31;
    int np = 0, np2 = 0;
#pragma unroll
    for (int k = 0; k < NM; ++k) {
        if (L == 16) {
            if (m[k] & 0xffffu) np = k + 2;
            if (m[k] >> 16) np2 = k + 2;
        } else {
            if (m[k]) np = k + 2;
        }
    }
    // a block that starts past the end has no planes (its values repeat the last element)
    if ((lane & ~(RPB - 1)) * 32 >= A.nrem) np = 0;
    if (L == 16 && lane * 32 + 16 >= A.nrem) np2 = 0;
    unsigned at;
    const int tot = place_rows<LOG2L>(A, np, np2, at);
    open_payload(A);
    put_plane<LOG2L>(at, 0, S, np, np2);
#pragma unroll
    for (int k = 0; k < NM; ++k) put_plane<LOG2L>(at, k + 1, m[k], np, np2);
    return tot;
}

// Heads apart: the 24-bit head fields of the lane's block(s).
template <int LOG2L>
__device__ __forceinline__ void put_heads(const EncArgs& A, int t0, int t16)
{
    constexpr int L = Blk<LOG2L>::L, RPB = Blk<LOG2L>::RPB;
    const int lane = threadIdx.x & 31;
    if ((lane & (RPB - 1)) != 0) return;
#pragma unroll
    for (int h = 0; h < (L == 16 ? 2 : 1); ++h) {
        const int b = L == 16 ? 2 * lane + h : lane / RPB;
        if (b * L < A.nrem) {
            const int head = (h ? t16 : t0) - QBIAS;
            A.hout[3 * b] = (uint8_t)head;
            A.hout[3 * b + 1] = (uint8_t)(head >> 8);
            A.hout[3 * b + 2] = (uint8_t)(head >> 16);
        }
    }
}

// BF16 rows of a group buffer -> FP32 rows of the same buffer.
__device__ __forceinline__ void expand_bf16(unsigned buf)
{
    const int lane = threadIdx.x & 31;
    uint4 v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = lds128(buf + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4));
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const unsigned row = buf + lane * 128;
        sts128(row + (((2 * c) ^ (lane & 7)) << 4), v[c].x << 16, v[c].x & 0xffff0000u, v[c].y << 16,
               v[c].y & 0xffff0000u);
        sts128(row + (((2 * c + 1) ^ (lane & 7)) << 4), v[c].z << 16, v[c].z & 0xffff0000u,
               v[c].w << 16, v[c].w & 0xffff0000u);
    }
    __syncwarp();
}

// The general path of a group: any width, any rounding, errors.  `bad`: rows
// that hold a value whose fast rounding is not proven (near a tie, or beyond
// 2^20: `far`).  Bad rows are settled a lane per element: q next to x inv is at
// most one off, and the residual e = x - q 2eb decides (exact where |e| is near
// eb: there it is a multiple of ulp(eb), see quantize).  Their values are replaced
// by q 2eb, whose fast rounding is q again (|q| < 2^20, heads apart 2^21: x' and inv
// are off by at most 2^-24 relatively, so x' inv is within 1/4 of q).  With `far`
// set every row is quantized by quantize(), errors and all, and the buffer then holds
// the rounding results themselves.  Then 32-bit deltas, byte by byte.  Not
// inlined: a few groups in a hundred come here (near-tie values, |q| >=
// 16000), and the fast path keeps its registers.  Where every row is bad (bytes at
// 2eb = 2: each odd one is a tie; 2^24 of them, L = 32) compression takes 42 us,
// where quantize() for bad rows too took 61.
template <int LOG2L, bool HEADS, bool BF>
__device__ __noinline__ int encode_rows_general(const EncArgs A, unsigned bad, bool far, int* err)
{
    constexpr int L = Blk<LOG2L>::L, RPB = Blk<LOG2L>::RPB;
    const int lane = threadIdx.x & 31;
    if (BF) expand_bf16(A.buf);
    // q 2eb of a value near FLT_MAX may overflow (x = FLT_MAX, 2eb = 1.5 2^126: q =
    // 3); |q| < 2^21 keeps it finite for a 2eb below 2^107
    if (bad != 0u && A.two_eb >= 0x1p107f) far = true;
    if (far) {
#pragma unroll 1
        for (int r = 0; r < GROWS; ++r) {
            const unsigned p = elem_addr<float>(A.buf, r * 32 + lane);
            int q;
            *err |= quantize(__uint_as_float(lds32(p)), A.eb, A.two_eb, A.inv, q);
            sts32(p, (uint32_t)(q + QBIAS));
        }
    } else {
        while (bad) {  // warp-uniform
            const unsigned p = elem_addr<float>(A.buf, (__ffs(bad) - 1) * 32 + lane);
            bad &= bad - 1;
            const float x = __uint_as_float(lds32(p));
            const float t = __fmaf_rn(x, A.inv, 12582912.0f);
            float q = __fsub_rn(t, 12582912.0f);
            const int e = __float_as_int(__fmaf_rn(-q, A.two_eb, x));
            // |e| > eb, or = eb at an odd q (positive floats order like their bits)
            if ((e & 0x7fffffff) + (__float_as_int(t) & 1) > __float_as_int(A.eb)) q += e < 0 ? -1.0f : 1.0f;
            sts32(p, __float_as_uint(__fmul_rn(q, A.two_eb)));
        }
    }
    __syncwarp();
    int d[32];
    const unsigned row = A.buf + lane * 128 + ((lane & 7) << 4);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const uint4 v = lds128(row ^ (c << 4));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
            d[4 * c + i] = far ? (int)w[i]
                               : __float_as_int(__fmaf_rn(__uint_as_float(w[i]), A.inv, 12582912.0f));
    }
    const int t0 = d[0], t16 = d[16];
    int fill = HEADS ? t0 : QBIAS;
    if (L >= 64) {
        const int up = __shfl_up_sync(FULL, d[31], 1);
        if ((lane & (RPB - 1)) != 0) fill = up;
    }
#pragma unroll
    for (int i = 31; i > 0; --i) {
        if (L == 16 && i == 16) d[i] = HEADS ? 0 : d[i] - QBIAS;
        else d[i] -= d[i - 1];
    }
    d[0] -= fill;
    if (HEADS) put_heads<LOG2L>(A, t0, t16);
    // widths: the bit length of the block's largest |d|
    uint32_t S = 0, o1 = 0, o2 = 0;
#pragma unroll
    for (int i = 31; i >= 0; --i) {
        S = __funnelshift_l((uint32_t)d[i], S, 1);
        const uint32_t a = (uint32_t)(d[i] < 0 ? -d[i] : d[i]);
        if (L == 16 && i >= 16) o2 |= a;
        else o1 |= a;
    }
    // (levels lie within 2^22, so deltas fit; a row's place is for no more planes)
    int np = o1 ? min(33 - __clz(o1), ZC_MAX_WIDTH + 1) : 0;
    int np2 = L == 16 && o2 ? min(33 - __clz(o2), ZC_MAX_WIDTH + 1) : 0;
    if ((lane & ~(RPB - 1)) * 32 >= A.nrem) np = 0;
    if (L == 16 && lane * 32 + 16 >= A.nrem) np2 = 0;
    const int npmax = __reduce_max_sync(FULL, max(np, np2));
    unsigned at;
    const int tot = place_rows<LOG2L>(A, np, np2, at);
    open_payload(A);
    put_plane<LOG2L>(at, 0, S, np, np2);
    uint32_t c = S;
#pragma unroll
    for (int lev = 0; lev < 3; ++lev) {
        if (lev * 8 + 1 >= npmax) break;  // warp-uniform
        const uint32_t s2 = 0x40u + 0x11u * lev;
        uint32_t w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            w[k] = __byte_perm(__byte_perm((uint32_t)d[k], (uint32_t)d[k + 8], s2),
                               __byte_perm((uint32_t)d[k + 16], (uint32_t)d[k + 24], s2), 0x5410);
        t8(w);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            put_plane<LOG2L>(at, 8 * lev + k + 1, neg_plane(w[k], S, c), np, np2);
    }
    return tot;
}

// The four rounding results of v (the bits of x inv + 1.5 2^23), the largest
// residual |x - q 2eb| and the largest |q - ref|.
template <bool REF>
__device__ __forceinline__ void quant4(const float v[4], f32x2 inv2, f32x2 nte2, f32x2 nref2,
                                       int t[4], float& me, float& mr)
{
    const f32x2 mag = pk2(12582912.0f, 12582912.0f), nmag = pk2(-12582912.0f, -12582912.0f);
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
        const f32x2 x = pk2(v[i], v[i + 1]);
        const f32x2 tt = fma2(x, inv2, mag);
        const f32x2 r = add2(tt, nmag);
        float a, b;
        up2(fma2(r, nte2, x), a, b);
        me = max3_abs(me, a, b);
        up2(REF ? add2(r, nref2) : r, a, b);
        mr = max3_abs_nan(mr, a, b);
        up2(tt, a, b);
        t[i] = __float_as_int(a);
        t[i + 1] = __float_as_int(b);
    }
}

// Encodes the group in A.buf (values of type T, FP32 or BF16 rows) into the
// same buffer: its payload behind the A.r0 carried bytes; returns the
// payload's size.
//
// Rounding.  t = x inv + 1.5 2^23, rounded once, holds the integer q next to
// x inv in its low bits.  The residual e = x - q 2eb, rounded once, proves q:
// rounding is monotone, so |e| < eb says |x - q 2eb| < eb, and q is the one
// nearest integer.  Anything else (ties, an x inv that was off by its own
// rounding, NaN) goes to the general path; so do |q| >= 16000, where deltas
// may need more than 16 bits.
//
// Deltas.  U_j = t_j + 2^16 t_(j+16) mod 2^32; U_j - U_(j-1) = d_j + 2^16
// d_(j+16) exactly, and adding 0x8080 to both halves keeps them apart (|d| <=
// 32000).  A half's high byte is then 0x80 iff d fits 8 bits, and its low
// byte is d with the top bit flipped.
template <int LOG2L, typename T, bool HEADS>
__device__ __forceinline__ int encode_rows(const EncArgs& A, int& err)
{
    constexpr int L = Blk<LOG2L>::L, RPB = Blk<LOG2L>::RPB;
    constexpr float QLIM = HEADS ? 8000.0f : 16000.0f;
    const int lane = threadIdx.x & 31;
    const f32x2 inv2 = pk2(A.inv, A.inv), nte2 = pk2(-A.two_eb, -A.two_eb);
    f32x2 nref2 = 0ull;
    float ref = 0.0f;
    if (HEADS) {  // differences to the row's first value stay small where the values do not
        const unsigned p = elem_addr<T>(A.buf, lane * 32);
        const float x0 = sizeof(T) == 4 ? __uint_as_float(lds32(p)) : __uint_as_float(lds16(p) << 16);
        ref = __fsub_rn(__fmaf_rn(x0, A.inv, 12582912.0f), 12582912.0f);
        nref2 = pk2(-ref, -ref);
    }
    uint32_t C[16];  // U_j, then the biased deltas of elements j and j + 16
    float me = 0.0f, mr = 0.0f;
    bool jump = false;  // heads apart: more than 16 bits between this row and the one before
    int t0 = 0, t16 = 0, t31 = 0;
    uint32_t u0 = 0, up = 0;
    if (sizeof(T) == 4) {
        const unsigned row = A.buf + lane * 128 + ((lane & 7) << 4);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint4 va = lds128(row ^ (c << 4)), vb = lds128(row ^ ((c + 4) << 4));
            const float a[4] = {__uint_as_float(va.x), __uint_as_float(va.y), __uint_as_float(va.z),
                                __uint_as_float(va.w)};
            const float b[4] = {__uint_as_float(vb.x), __uint_as_float(vb.y), __uint_as_float(vb.z),
                                __uint_as_float(vb.w)};
            int ta[4], tb[4];
            quant4<HEADS>(a, inv2, nte2, nref2, ta, me, mr);
            quant4<HEADS>(b, inv2, nte2, nref2, tb, me, mr);
            if (c == 0) {
                t0 = ta[0];
                t16 = tb[0];
            }
            if (c == 3) t31 = tb[3];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t u = (uint32_t)ta[i] + ((uint32_t)tb[i] << 16);
                if (c == 0 && i == 0) u0 = u;
                else C[4 * c + i] = u - up + 0x80808080u;
                up = u;
            }
        }
    } else {
        const unsigned row = A.buf + lane * 64 + (((lane >> 1) & 3) << 4);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const uint4 va = lds128(row ^ (c << 4)), vb = lds128(row ^ ((c + 2) << 4));
            const uint32_t wa[4] = {va.x, va.y, va.z, va.w}, wb[4] = {vb.x, vb.y, vb.z, vb.w};
#pragma unroll
            for (int h = 0; h < 4; h += 2) {
                float a[4], b[4];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    a[2 * i] = __uint_as_float(wa[h + i] << 16);
                    a[2 * i + 1] = __uint_as_float(wa[h + i] & 0xffff0000u);
                    b[2 * i] = __uint_as_float(wb[h + i] << 16);
                    b[2 * i + 1] = __uint_as_float(wb[h + i] & 0xffff0000u);
                }
                int ta[4], tb[4];
                quant4<HEADS>(a, inv2, nte2, nref2, ta, me, mr);
                quant4<HEADS>(b, inv2, nte2, nref2, tb, me, mr);
                if (c == 0 && h == 0) {
                    t0 = ta[0];
                    t16 = tb[0];
                }
                if (c == 1 && h == 2) t31 = tb[3];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t u = (uint32_t)ta[i] + ((uint32_t)tb[i] << 16);
                    if (c == 0 && h == 0 && i == 0) u0 = u;
                    else C[8 * c + 2 * h + i] = u - up + 0x80808080u;
                    up = u;
                }
            }
        }
    }
    // the row's first elements: predicted from 0 (from themselves when heads
    // are apart), or from the block's row before; element 16 from element 15
    {
        int fill = HEADS ? t0 : QBIAS;
        if (L >= 64) {
            const int prev = __shfl_up_sync(FULL, t31, 1);
            if ((lane & (RPB - 1)) != 0) {
                fill = prev;
                // heads apart: only differences within a row are bounded so far.
                // (A flag of its own: mr tells apart what the row itself holds.)
                if (HEADS) jump = (uint32_t)t0 - (uint32_t)prev + 15999u > 31998u;
            }
        }
        uint32_t um;
        if (L == 16) um = HEADS ? u0 : (uint32_t)QBIAS + ((uint32_t)QBIAS << 16);
        else um = (uint32_t)fill + (up << 16);
        C[0] = u0 - um + 0x80808080u;
    }
    const bool far = !(mr < 1048576.0f) || (HEADS && !(fabsf(ref) < 1048576.0f));
    const bool bad = !(me < A.eb) || far;
    if (__any_sync(FULL, bad || jump || !(mr < QLIM)))
        return encode_rows_general<LOG2L, HEADS, sizeof(T) == 2>(A, __ballot_sync(FULL, bad),
                                                                 __any_sync(FULL, far), &err);
    if (HEADS) put_heads<LOG2L>(A, t0, t16);
    uint32_t hb = 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) hb |= C[j] ^ 0x80008000u;
    if (!__any_sync(FULL, (hb & 0xff00ff00u) != 0u)) {
        uint32_t w[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) w[k] = __byte_perm(C[k], C[k + 8], 0x6240);
        t8(w);
        const uint32_t S = ~w[7];
        uint32_t c = S, m[8];
#pragma unroll
        for (int k = 0; k < 7; ++k) m[k] = neg_plane(w[k], S, c);
        m[7] = c;  // d = -128
        return put_planes<LOG2L, 8>(A, S, m);
    }
    uint32_t w[8], h[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint32_t a = C[k] - 0x00800080u, b = C[k + 8] - 0x00800080u;  // d + 0x8000
        w[k] = __byte_perm(a, b, 0x6240);
        h[k] = __byte_perm(a, b, 0x7351);
    }
    t8(w);
    t8(h);
    const uint32_t S = ~h[7];
    uint32_t c = S, m[15];
#pragma unroll
    for (int k = 0; k < 8; ++k) m[k] = neg_plane(w[k], S, c);
#pragma unroll
    for (int k = 0; k < 7; ++k) m[8 + k] = neg_plane(h[k], S, c);
    return put_planes<LOG2L, 15>(A, S, m);
}

// ---- decoding -------------------------------------------------------------------

// Where a lane's planes lie: in shared memory (SMEM) or in the stream.
template <bool SMEM>
struct PlaneSrc {
    unsigned sp;        // shared-memory address of the lane's first word
    const uint8_t* gp;  // or its place in the stream
    __device__ __forceinline__ uint32_t u32(int off) const
    {
        if (SMEM) return lds32(sp + off);
        return ld_dep((const unsigned*)(gp + off));
    }
    __device__ __forceinline__ uint32_t u16(int off) const
    {
        if (SMEM) return lds16(sp + off);
        return ld_dep((const unsigned short*)(gp + off));
    }
};

// Plane k of the lane's block(s), 0 beyond its planes.
template <int LOG2L, bool SMEM>
__device__ __forceinline__ uint32_t get_plane(const PlaneSrc<SMEM>& P, int k, int np, int np2)
{
    constexpr int L = Blk<LOG2L>::L, RPB = Blk<LOG2L>::RPB;
    if (L == 16) {
        uint32_t lo = 0, hi = 0;
        if (k < np) lo = P.u16(2 * k);
        if (k < np2) hi = P.u16(2 * np + 2 * k);
        return lo | (hi << 16);
    }
    return k < np ? P.u32(4 * RPB * k) : 0u;
}

// Exclusive sum of `tot` over the block's rows before this lane's.
template <int RPB>
__device__ __forceinline__ int rows_before(int tot)
{
    const int lane = threadIdx.x & 31;
    int s = tot;
#pragma unroll
    for (int off = 1; off < RPB; off <<= 1) {
        const int o = __shfl_up_sync(FULL, s, off);
        if ((lane & (RPB - 1)) >= off) s += o;
    }
    return s - tot;
}

// Four consecutive values x^ = q 2eb from the bits of q + 1.5 2^23 (|q| <= 2^22).
template <typename Emit>
__device__ __forceinline__ void emit_bits(int c, const int b[4], f32x2 te2, const Emit& emit)
{
    const f32x2 nmag = pk2(-12582912.0f, -12582912.0f);
    float v[4];
    up2(mul2(add2(pk2(__int_as_float(b[0]), __int_as_float(b[1])), nmag), te2), v[0], v[1]);
    up2(mul2(add2(pk2(__int_as_float(b[2]), __int_as_float(b[3])), nmag), te2), v[2], v[3]);
    emit(c, v);
}

// The same from any q: a stream's heads and wide deltas can sum to levels beyond
// 2^22, which no encoder writes but which have a value all the same.
template <typename Emit>
__device__ __forceinline__ void emit_ints(int c, const int q[4], f32x2 te2, const Emit& emit)
{
    float v[4];
    up2(mul2(pk2(__int2float_rn(q[0]), __int2float_rn(q[1])), te2), v[0], v[1]);
    up2(mul2(pk2(__int2float_rn(q[2]), __int2float_rn(q[3])), te2), v[2], v[3]);
    emit(c, v);
}

// More than 16 planes somewhere in the group.
template <int LOG2L, bool SMEM, bool HEADS, typename Sync, typename Emit>
__device__ __forceinline__ void decode_rows_wide(const PlaneSrc<SMEM>& P, int np, int np2, int h0,
                                                 int h16, float two_eb, const Sync& sync,
                                                 const Emit& emit)
{
    constexpr int L = Blk<LOG2L>::L, RPB = Blk<LOG2L>::RPB;
    const uint32_t S = get_plane<LOG2L, SMEM>(P, 0, np, np2);
    uint32_t w[3][8];
#pragma unroll
    for (int lev = 0; lev < 3; ++lev) {
#pragma unroll
        for (int k = 0; k < 8; ++k) w[lev][k] = get_plane<LOG2L, SMEM>(P, 8 * lev + k + 1, np, np2);
        t8(w[lev]);
    }
    sync();  // every lane has its planes
    int tot = 0;
    auto delta = [&](int i) {  // sign and magnitude of element i = 8 b + k
        const int k = i & 7, b = i >> 3;
        const uint32_t m = __byte_perm(__byte_perm(w[0][k], w[1][k], 0x0040 + 0x11 * b),
                                       w[2][k], 0x0410 + 0x100 * b) &
                           0xffffffu;
        const int s = (int)(S << (31 - i)) >> 31;
        return ((int)m ^ s) - s;
    };
    if (L >= 64) {
#pragma unroll
        for (int i = 0; i < 32; ++i) tot += delta(i);
    }
    // (a head reaches its block's later rows through the sums)
    int q = (HEADS ? h0 : 0) + (L >= 64 ? rows_before<RPB>(tot + (HEADS ? h0 : 0)) : 0);
    const f32x2 te2 = pk2(two_eb, two_eb);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        if (L == 16 && c == 4) q = HEADS ? h16 : 0;
        int b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) b[i] = q += delta(4 * c + i);
        emit_ints(c, b, te2, emit);
    }
}

// Decodes the lane's row: np planes (np2: the row's second block at L = 16),
// block heads h0 / h16 when stored apart (0 in lanes that hold none).
// sync() runs once all planes are in registers; emit(c, v) takes the values
// of elements 4 c .. 4 c + 3, x^ = q 2eb, rounded once.
//   At most 8 planes everywhere (|d| <= 127): one transpose gives the bytes d
//   + 128, and the prefix sums run on pairs (elements j and j + 16 in halves
//   of one word, q + 2^15 each: |q| <= 128 * 127 < 2^15).
//   At most 16 planes: two transposes, prefix sums per element.
template <int LOG2L, bool SMEM, bool HEADS, typename Sync, typename Emit>
__device__ __forceinline__ void decode_rows(const PlaneSrc<SMEM>& P, int np, int np2, int h0,
                                            int h16, float two_eb, const Sync& sync,
                                            const Emit& emit)
{
    constexpr int L = Blk<LOG2L>::L, RPB = Blk<LOG2L>::RPB;
    const int npm = max(np, np2);
    if (__any_sync(FULL, npm > 16)) {
        decode_rows_wide<LOG2L, SMEM, HEADS>(P, np, np2, h0, h16, two_eb, sync, emit);
        return;
    }
    const bool wide8 = __any_sync(FULL, npm > 8);
    const uint32_t S = get_plane<LOG2L, SMEM>(P, 0, np, np2);
    uint32_t w[8], c = S;
#pragma unroll
    for (int k = 0; k < 7; ++k) w[k] = neg_plane(get_plane<LOG2L, SMEM>(P, k + 1, np, np2), S, c);
    const f32x2 te2 = pk2(two_eb, two_eb);
    if (!wide8) {
        sync();
        w[7] = ~(S ^ c);  // the sign bit (0 for a zero), flipped: bytes d + 128
        t8(w);
        if constexpr (!HEADS) {
            uint32_t s = 0x80008000u;
            if (L >= 32) {
                unsigned t = 0;
#pragma unroll
                for (int k = 0; k < 8; ++k) t = __dp4a(w[k], 0x00000101u, t);
                const int half = (int)t - 16 * 128;  // sum of the first 16 deltas
                int off = 0;
                if (L >= 64) {
                    unsigned t2 = 0;
#pragma unroll
                    for (int k = 0; k < 8; ++k) t2 = __dp4a(w[k], 0x01010000u, t2);
                    off = rows_before<RPB>(half + (int)t2 - 16 * 128);
                }
                s += (uint32_t)off + ((uint32_t)(off + half) << 16);
            }
            const f32x2 nb2 = pk2(-8421376.0f, -8421376.0f);  // 2^23 + 2^15
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4) {
                float lo[4], hi[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int j = 4 * q4 + i;
                    s += __byte_perm(w[j & 7], 0u, j < 8 ? 0x4240 : 0x4341) - 0x00800080u;
                    lo[i] = __uint_as_float(__byte_perm(s, 0x4b00u, 0x5410));
                    hi[i] = __uint_as_float(__byte_perm(s, 0x4b00u, 0x5432));
                }
                float v[4];
                up2(mul2(add2(pk2(lo[0], lo[1]), nb2), te2), v[0], v[1]);
                up2(mul2(add2(pk2(lo[2], lo[3]), nb2), te2), v[2], v[3]);
                emit(q4, v);
                up2(mul2(add2(pk2(hi[0], hi[1]), nb2), te2), v[0], v[1]);
                up2(mul2(add2(pk2(hi[2], hi[3]), nb2), te2), v[2], v[3]);
                emit(q4 + 4, v);
            }
            return;
        } else {
            int tot = 0;
            if (L >= 64) {
                unsigned t = 0;
#pragma unroll
                for (int k = 0; k < 8; ++k) t = __dp4a(w[k], 0x01010101u, t);
                tot = (int)t - 32 * 128;
            }
            int q = h0 + (L >= 64 ? rows_before<RPB>(tot + h0) : 0);
#pragma unroll
            for (int cc = 0; cc < 8; ++cc) {
                if (L == 16 && cc == 4) q = h16;
                int b[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int e = 4 * cc + i;
                    b[i] = q += (int)__byte_perm(w[e & 7], 0u, 0x4440 + (e >> 3)) - 128;
                }
                emit_ints(cc, b, te2, emit);
            }
            return;
        }
    }
    uint32_t h[8];
    w[7] = neg_plane(get_plane<LOG2L, SMEM>(P, 8, np, np2), S, c);
#pragma unroll
    for (int k = 0; k < 7; ++k) h[k] = neg_plane(get_plane<LOG2L, SMEM>(P, k + 9, np, np2), S, c);
    h[7] = S ^ c;  // the sign bit
    sync();
    t8(w);
    t8(h);
    // halves: elements k and k + 16, then k + 8 and k + 24, as signed 16 bits
    uint32_t a[16];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        a[k] = __byte_perm(w[k], h[k], 0x6240);
        a[k + 8] = __byte_perm(w[k], h[k], 0x7351);
    }
    // (without heads |q| <= 128 (2^15 - 1) < 2^22)
    int q = HEADS ? h0 : QBIAS;
    if (L >= 64) {
        int tot = HEADS ? h0 : 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) tot = __dp2a_lo((int)a[k], 0x0101, tot);
        q += rows_before<RPB>(tot);
    }
#pragma unroll
    for (int cc = 0; cc < 8; ++cc) {
        if (L == 16 && cc == 4) q = HEADS ? h16 : QBIAS;
        int b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)  // one element of the pair added per dot product
            b[i] = q = __dp2a_lo((int)a[(4 * cc + i) & 15], cc < 4 ? 0x0001 : 0x0100, q);
        if (HEADS) emit_ints(cc, b, te2, emit);
        else emit_bits(cc, b, te2, emit);
    }
}

// A lane's planes and its block's place within a group, from its width byte(s)
// wv (L = 16: two bytes): `at` the byte offset of its first word from the
// group's payload start.  Returns the group's payload size; `bad` reports a
// width beyond the format's (taken as none).
template <int LOG2L>
__device__ __forceinline__ int rows_meta(uint32_t wv, int& np, int& np2, int& at, bool& bad)
{
    constexpr int L = Blk<LOG2L>::L, RPB = Blk<LOG2L>::RPB;
    const int lane = threadIdx.x & 31;
    auto planes = [&](uint32_t w) {
        if (w > ZC_MAX_WIDTH) {
            bad = true;
            return 0;
        }
        return w ? (int)w + 1 : 0;
    };
    np = planes(wv & 0xffu);
    np2 = L == 16 ? planes((wv >> 8) & 0xffu) : 0;
    const int sz = L == 16 ? 2 * (np + np2) : 4 * np;
    const int s = scan_incl<32>(sz);
    const int tot = __shfl_sync(FULL, s, 31);
    const int sub = lane & (RPB - 1);
    at = (s - sz) - sub * sz + 4 * sub;
    return tot;
}

}  // namespace zc
