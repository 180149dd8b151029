// zc_codec.cuh -- the tile kernels: compress, decompress, the fused ring step
// (decompress -> add -> recompress) and the scatter pack.
//
// Geometry.  A warp unit is U rows of 32 elements (U = 32, 64 or 128), worked
// on 32 rows at a time, one row per lane (zc_rows.cuh); an encoder tile is 8
// consecutive units, one per encoder warp of a CTA, a decode tile 8 units of
// DEC_U rows.  Blocks never straddle groups of 32 rows.
//
// Encoder offsets.  Every encoder warp appends its blocks' planes to its own
// ring segment (the running offset is warp-uniform: no scan), so nothing waits
// until the whole tile is encoded.  The tile's position in the stream comes
// from a decoupled look-back over the tiles' sizes, run by a resolver warp;
// then every warp copies its segment to its place.  The first tile of a stream
// also counts the 32-byte header and the padded width bytes; the last one
// rounds the stream up to 16 bytes; in packed mode (the scatter pack) one
// chain runs through all streams.
//
// Decoder offsets.  k_wscan reads only the width bytes of a stream and
// writes the payload offset of every warp unit (a chain over chunks of WSCAN
// units); decoding then needs no look-back and no barrier.
#pragma once

#include "zc_rows.cuh"

namespace zc {

constexpr int WSCAN = NTHREADS;        // warp units per width-scan chunk
// Rows per warp unit of the decompressor.  A unit starts with a chain of three
// round trips (header, width bytes and offset, payload), about a third of a
// 64-row unit's time; large launches take 128-row units, small ones keep enough
// CTAs with 64 (measured at 64 / 128: 2^27
// elements of the field 126.5 / 124 us, 2^25 47.5 / 49.8, 2^26 BF16 gradients 75.3 / 73.2,
// a batch of 250 messages 380 / 359).
constexpr int DEC_U = 64;
constexpr int DEC_U_LARGE = 128;
// Batched decompression: items of at most this many decode tiles get no
// width-scan chunks; their decoder CTAs find the unit offsets themselves.
constexpr unsigned DEC_LOCAL_TILES = 4;
// In launches of at most this many tiles (about two per resident CTA) that
// holds for larger items too: up to DEC_LOCAL_FEW_TILES decode tiles, and in
// the fused step up to RED_LOCAL_BLOCKS blocks (width bytes).  Few CTAs then
// each read at most 128 KiB of width bytes, from L2, where the scan would be a
// launch in front of a short one (the five-rank recursive doubling of 1M
// elements: 139 us with four scans, 118 us without).
constexpr unsigned LOCAL_LAUNCH_TILES = 1024;
constexpr unsigned DEC_LOCAL_FEW_TILES = 128;
constexpr unsigned RED_LOCAL_BLOCKS = 1u << 16;
// Decompression of one stream: up to this many decode tiles (16384 elements
// each) every CTA sums the width bytes before its tile itself, 16 bytes per
// thread and load, and there is no width scan: the scan costs a launch and
// some seven dependent round trips, the sums of a last tile here at most
// 256 KiB / 4 KiB = 64 loads per thread, four in flight.  Measured with / without
// the scan: 2^21 elements 10.8 / 7.5 us at L = 32, 12.6 / 9.2 at L = 16; 2^22 elements
// 13.7 / 10.5 and 15.8 / 13.5; 2^23 elements 17.4 / 20.5 and 20.3 / 29.0.
constexpr unsigned DEC_LOCAL_SINGLE_TILES = 256;

// Rows per warp unit of an encoder tile of `chunks` 2048-element chunks.
__host__ __device__ constexpr int unit_rows(int chunks) { return chunks * 8; }
// Largest payload of one warp unit of U rows: 32 U elements x 25 planes / 8.
__host__ __device__ constexpr int seg_bytes(int U) { return U * 100; }

struct Item {
    const void* x;            // raw input (compress) or local chunk (ring step), or null
    const uint8_t* cin;       // received stream, or null
    uint8_t* out;             // output stream (non-packed) / packed buffer base, or null
    void* raw_out;            // decoded values / FP32 sum, or null
    unsigned long long* out_bytes;
    unsigned long long n, cin_cap, out_cap;
    float eb, two_eb, inv;    // encoding bound
    unsigned tile_begin, ntiles;    // tiles of this launch's geometry
    unsigned chunk_begin, nchunks;  // width-scan chunks
    int x_dtype, out_dtype;
    int log2L;                // batched compression: block size, or -1 for a raw stream
};

struct Launch {
    Ctl* ctl;
    Chain chB;                        // encoder tiles
    Chain chC;                        // width-scan chunks
    unsigned long long* offs;         // payload offset of every decode tile (global slot)
    ulonglong2* seg_rec;              // packed mode: stream start published per item
    unsigned long long* seg_off;      // packed mode: P + 1 stream offsets (caller's)
    const Item* items;                // device items, or null for `one`
    Item one;
    unsigned n_items, total_tiles;    // total_tiles: tiles (or chunks for k_wscan)
    int urows;                        // rows per warp unit (decode slot = tile * NWARPS + warp)
    int eb_from_ctl;                  // relative bound resolved into ctl
    int packed;
    WaitCfg wc;
    // batched decompression: item i's stream sits at in_base + in_off[i] (in_off
    // written by an earlier launch; in_cap bytes at in_base)
    const uint8_t* in_base;
    const unsigned long long* in_off;
    unsigned long long in_cap;
    // item of every tile (written by k_tile_map before the launch), or null:
    // then the item is found by a binary search over tile_begin
    const unsigned* tile_map;
    // encoder launches: the CTAs' tile rings (ring_cta_bytes each, in CTA order)
    uint8_t* ring;
    unsigned long long ring_bytes;
    unsigned long long ws_cap;  // entries of every workspace array (bounds-checked builds)
    // grouped batch (packed mode): the streams lie in ticket order, not item
    // order, so seg_off[i] is only item i's start and seg_off[n_items] the
    // packed total; a decoder bounds a stream by seg_off[n_items]
    int grouped;
};

struct Smem {
    LbSmem lb;
    unsigned ticket, item, E;
    int abort;
};

// Encoder CTAs: NWARPS encoder warps plus one resolver warp, enc_slots(U)
// tiles in flight.  Every tile slot has, per encoder warp, a payload segment
// of seg_bytes(U) in the CTA's ring (global memory) and U * 2 width bytes in
// shared memory.  Three slots give the resolver two tiles' time; the largest
// tiles take two, which keeps the rings of all CTAs inside L2.
__host__ __device__ constexpr int enc_slots(int U) { return U >= 128 ? 2 : 3; }
constexpr int ENC_SLOTS_MAX = 3;
constexpr int ENC_THREADS = NTHREADS + 32;
constexpr int ENC_CTAS_PER_SM = 3;            // resident encoder CTAs per SM (registers)
constexpr unsigned BAR_ENCW = 1;              // named barrier: the encoder warps
constexpr unsigned BAR_ENC = 2;               // + slot: tile encoded (resolver waits)
constexpr unsigned BAR_RES = BAR_ENC + ENC_SLOTS_MAX;  // + slot: tile resolved (encoders wait)
static_assert(BAR_RES + ENC_SLOTS_MAX <= 16, "named barriers per CTA");
__host__ __device__ constexpr unsigned long long ring_cta_bytes(int U)
{
    return (unsigned long long)enc_slots(U) * NWARPS * seg_bytes(U);
}
// Dynamic shared memory of an encoder CTA: every encoder warp's two group
// buffers, then the width bytes of every slot and warp.
__host__ __device__ constexpr int enc_wb_bytes(int U) { return enc_slots(U) * NWARPS * U * 2; }
__host__ __device__ constexpr int enc_smem_bytes(int U) { return NWARPS * 2 * GBUF + enc_wb_bytes(U); }
// Of a decoder CTA: two group buffers per warp.
constexpr int DEC_SMEM_BYTES = NWARPS * 2 * GBUF;
constexpr int DEC_CTAS_PER_SM = 3;

__device__ __forceinline__ void store_raw(void* p, int dtype, unsigned long long i, float v)
{
    if (dtype == ZC_F32) ((float*)p)[i] = v;
    else ((uint16_t*)p)[i] = f32_to_bf16(v);
}

__device__ __forceinline__ int warp_excl_scan(int v, int lane, int& total)
{
    int s = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(FULL, s, off);
        if (lane >= off) s += o;
    }
    total = __shfl_sync(FULL, s, 31);
    return s - v;
}

// Reads and checks an input stream header for `it`; returns its log2 L (plus
// 8 when its block heads are stored apart), -1 for a format error (reported
// when `report`), -2 / -3 for a raw FP32 / BF16 stream.  A caller that names
// the block size it expects (the fused ring step) takes plain streams only.
// WHOLE: the stream was complete before the kernel started (the scanned decoder:
// the width scan before it has waited for it), so the loads may be non-coherent.
template <bool WHOLE = false>
__device__ __forceinline__ int check_header(const Item& it, Ctl* ctl, unsigned item_idx,
                                            int expect_log2L, float& eb_in, bool report)
{
    const uint8_t* s = it.cin;
    auto ld = [](const auto* p) { return WHOLE ? __ldg(p) : ld_dep(p); };
    if (it.cin_cap < 32) {
        if (report) fail(ctl, ZC_ERR_FORMAT, item_idx);
        return -1;
    }
    const uint32_t w0 = ld((const unsigned*)s);
    const uint32_t w1 = ld((const unsigned*)s + 1);
    const unsigned long long n = ld((const unsigned long long*)s + 1);
    eb_in = __uint_as_float(ld((const unsigned*)s + 4));
    const uint32_t nb = ld((const unsigned*)s + 5);
    const unsigned long long payload = ld((const unsigned long long*)s + 3);
    const int dtype = w1 & 0xff, lg = (w1 >> 8) & 0xff, flags = (w1 >> 16) & 0xff;
    bool ok = w0 == 0x3176435au && (w1 >> 24) == 0u && (dtype == 0 || dtype == 1) &&
              (flags & ~3) == 0 && flags != 3 && n == it.n;
    int ret = lg;
    if (ok && (flags & 1)) {
        const unsigned long long es = dtype == 0 ? 4ull : 2ull;
        ok = nb == 0u && payload == n * es && 32ull + ceil16(payload) <= it.cin_cap &&
             expect_log2L < 0;
        ret = -2 - dtype;
    } else if (ok) {
        const bool heads = (flags & 2) != 0;
        ok = lg >= 4 && lg <= 7 && (expect_log2L < 0 || (lg == expect_log2L && !heads)) &&
             (unsigned long long)nb == ((n + (1ull << lg) - 1) >> lg) &&
             32ull + ceil16(nb) + (heads ? ceil16(3ull * nb) : 0ull) + ceil16(payload) <=
                 it.cin_cap;
        if (ok && nb > 0) ok = is_normal(eb_in) && eb_in > 0.0f && isfinite(eb_in + eb_in);
        if (heads) ret = lg + 8;
    }
    if (!ok) {
        if (report) fail(ctl, ZC_ERR_FORMAT, item_idx);
        return -1;
    }
    return ret;
}

__device__ __forceinline__ int planes_of(int w) { return w ? w + 1 : 0; }


// ---- stream access ------------------------------------------------------------
// Block head of the heads-apart format: 24-bit two's complement, little-endian.
__device__ __forceinline__ int load_head(const uint8_t* p)
{
    const unsigned v = (unsigned)ld_dep(p) | ((unsigned)ld_dep(p + 1) << 8) |
                       ((unsigned)ld_dep(p + 2) << 16);
    return (int)v - ((v & 0x800000u) ? (1 << 24) : 0);
}

// Width byte(s) of this lane's row of the group whose first block is bg (a
// multiple of 8; L = 16: the two bytes of the row's blocks).  The width bytes
// are zero padded to 16, blocks beyond them have none.
template <int LOG2L>
__device__ __forceinline__ uint32_t load_widths(const uint8_t* cin, unsigned long long nb,
                                                unsigned long long bg)
{
    const int lane = threadIdx.x & 31;
    const unsigned long long b =
        bg + (LOG2L == 4 ? 2u * lane : LOG2L == 5 ? lane : LOG2L == 6 ? lane / 2 : lane / 4);
    if (b >= ceil16(nb)) return 0u;
    return LOG2L == 4 ? (uint32_t)ld_dep((const unsigned short*)(cin + 32 + b))
                      : (uint32_t)ld_dep(cin + 32 + b);
}

// Whether 16 bytes can all be widths.
__device__ __forceinline__ bool widths_fit(const uint4& v)
{
    const unsigned up = 0x01010101u * (127 - ZC_MAX_WIDTH);  // bit 7 of a byte: above the largest
    return ((v.x | (v.x + up) | v.y | (v.y + up) | v.z | (v.z + up) | v.w | (v.w + up)) & 0x80808080u) == 0u;
}

// Planes of 16 width bytes at byte b of a stream's width array: the sum of
// w + 1 over the nonzero widths, four bytes at a time (a width above the
// format's counts as none and is reported when `ctl` is set).
__device__ __forceinline__ int planes16(const uint4& v, Ctl* ctl, unsigned long long b)
{
    const unsigned w[4] = {v.x, v.y, v.z, v.w};
    unsigned sum = 0u, bad = 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        sum = __dp4a(w[q], 0x01010101u, sum);
        sum += __popc((w[q] + 0x7f7f7f7fu) & 0x80808080u);          // bytes that are not 0
        bad |= w[q] | (w[q] + 0x01010101u * (127 - ZC_MAX_WIDTH));  // bit 7: above the largest
    }
    if ((bad & 0x80808080u) == 0u) return (int)sum;
    sum = 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        for (int k = 0; k < 4; ++k) {
            const int x = (w[q] >> (8 * k)) & 0xff;
            if (x <= ZC_MAX_WIDTH) sum += planes_of(x);
            else if (ctl != nullptr) fail(ctl, ZC_ERR_FORMAT, b + 4 * q + k);
        }
    return (int)sum;
}

// ---- encoder tiles -------------------------------------------------------------
// An encoder CTA runs two kinds of warps.  Its NWARPS encoder warps take tiles
// in ticket order and encode each of the tile's warp units into the CTA's ring
// (global memory, enc_slots(U) tiles deep) and its width bytes into shared
// memory.  Its resolver warp takes every encoded tile, sums the units' sizes,
// runs the tile's look-back (and, for packed streams, the stream-start wait)
// and hands the tile's place in the output back.  enc_slots(U) - 1 tiles later
// the encoder warps copy the tile from the ring to the stream.  So the encoder
// warps never stop for a look-back: the wait for the tiles before this one
// overlaps the encoding of the tiles after it.

// Copies `len` bytes (a multiple of UNIT) from the ring (16-byte aligned) to
// `dst` (UNIT-aligned) with one warp, through `buf`, a free group buffer of
// the warp: asynchronous copies bring the bytes into shared memory displaced
// by dst's distance from a 16-byte boundary (to the word; the odd half word of
// 2-byte units is shifted on the way out), all of them in flight at once, and
// 16-byte stores take them out.  (Copied through registers, four 4-byte loads
// at a time, a 4 KiB segment took eight round trips to L2.)  The staged bytes
// are dead afterwards: the L2 lines of 128 bytes that lie wholly in the segment
// (of SEG bytes; all of them when the workspace starts on such a line, as it need
// not) are dropped without a write-back, so the ring costs no DRAM traffic as long
// as a tile's lines stay in L2 until it is stored.
template <int UNIT, int SEG>
__device__ __forceinline__ void ring_copy(uint8_t* dst, const uint8_t* src, int len, unsigned buf)
{
    constexpr int W = UNIT == 2 ? 4 : UNIT;  // bytes per asynchronous copy
    constexpr int PIECE = GBUF - 32;         // bytes per round (a multiple of 16), with room to displace
    const int lane = threadIdx.x & 31;
    for (int p = 0; p < len; p += PIECE) {
        const int n = min(len - p, PIECE);
        uint8_t* const d = dst + p;
        const int sh = (int)((uintptr_t)d & 15);
        const uint8_t* s = src + p + W * lane;
        unsigned a = buf + (sh & ~(W - 1)) + W * lane;
#pragma unroll 8
        for (int o = W * lane; o < n; o += 32 * W, s += 32 * W, a += 32 * W) cp_async_ca<W>(a, s);
        cp_commit();
        cp_wait<0>();
        __syncwarp();
        uint8_t* const d0 = d - sh;  // 16-byte aligned
        const int end = sh + n;
        const bool half = UNIT == 2 && (sh & 2) != 0;
        for (int c = 16 * lane; c < end; c += 512) {
            uint4 v = lds128(buf + c);
            if (half) {
                const uint32_t b = c ? lds32(buf + c - 4) : 0u;
                v = make_uint4(__byte_perm(b, v.x, 0x5432), __byte_perm(v.x, v.y, 0x5432),
                               __byte_perm(v.y, v.z, 0x5432), __byte_perm(v.z, v.w, 0x5432));
            }
            if (c >= sh && c + 16 <= end) {
                __stcs((uint4*)(d0 + c), v);
            } else {  // the first and the last chunk
                const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int h = 0; h < 8; ++h) {
                    const int q = c + 2 * h;
                    if (q >= sh && q < end) *(uint16_t*)(d0 + q) = (uint16_t)(w[h >> 1] >> (16 * (h & 1)));
                }
            }
        }
        __syncwarp();  // the buffer is free
    }
    const int skew = (int)(0u - (unsigned)(uintptr_t)src) & 127;  // to the first whole line
    for (int l = skew + 128 * lane; l < len && l + 128 <= SEG; l += 128 * 32)
        asm volatile("discard.global.L2 [%0], 128;" ::"l"(__cvta_generic_to_global(src + l)) : "memory");
}

// Packed mode (one chain through many streams): the first tile of a stream
// publishes where the stream starts (its exclusive value ex), the stream's
// other tiles wait for that.  Outside packed mode a stream starts at 0.
// Returns false (status set) when the wait runs out.  Run by one warp.
__device__ __forceinline__ bool packed_start_warp(const Launch& P, bool first, unsigned item_idx,
                                                  unsigned long long ex, unsigned g, unsigned E,
                                                  unsigned long long& start)
{
    const int lane = threadIdx.x & 31;
    start = 0ull;
    if (!P.packed) return true;
    if (first) {
        start = ex;
        if (lane == 0) {
            P.seg_off[item_idx] = ex;
            rec_store(P.seg_rec + item_idx, E, ST_PREFIX, false, ex);
        }
        return true;
    }
    int ok = 1;
    unsigned long long v = 0ull;
    if (lane == 0) {
        ok = wait_rec(P.seg_rec + item_idx, E, P.wc.limit_ns, v);
        if (!ok) fail(P.ctl, ZC_ERR_TIMEOUT, g);
    }
    ok = __shfl_sync(FULL, ok, 0);
    start = __shfl_sync(FULL, v, 0);
    return ok != 0;
}

// One tile in flight.  The encoder warps fill it (thread 0 the scalars, lane
// 0 of every warp its unit's size), the resolver warp adds ex, start and ok.
struct TileSlot {
    unsigned g, item, tile;       // ticket, item, tile within the item
    int valid;                    // g is a tile of this launch
    int pub;                      // the tile takes part in the chain
    int first, last;              // first / last tile of its stream
    unsigned long long head;      // bytes of the tile besides its units' payload
    int segsz[NWARPS];            // payload bytes of every warp unit
    unsigned long long ex, start; // place in the chain, start of its stream
    int ok;                       // ex and start are usable: store the tile
    int nfin;                     // encoder warps done with the tile
};

struct EncShared {
    unsigned E;    // launch generation
    int abort;     // 1: unusable workspace (the CTA does nothing), 2: no usable bound
    int hdr_bad;   // fused ring step: the tile's input stream failed its check
    float eb_in;   // its bound
    unsigned pre[NWARPS], own[NWARPS];  // planes before the tile and of its units (items without a width scan)
};

// Payload offset of this warp's unit of a received stream without a width
// scan: the encoder warps of the CTA sum the width bytes before the tile and
// of its units (16 bytes per thread and load).  The item's last tile checks
// the total against the header's payload size, as the scan does, and the last
// width bytes, whose padding may lie beyond the last group of rows (blocks of 128).
template <int LOG2L, int U>
__device__ __forceinline__ unsigned long long tile_unit_offset(const Item& it, unsigned t, Ctl* ctl,
                                                               unsigned item_idx, EncShared& es)
{
    constexpr unsigned BPU = U * 32 >> LOG2L;  // blocks per unit: 8, or a multiple of 16
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned wbytes = (unsigned)ceil16((it.n + (1ull << LOG2L) - 1) >> LOG2L);
    const uint8_t* const w = it.cin + 32;
    const unsigned t0 = min(t * NWARPS * BPU, wbytes);  // a multiple of 16
    unsigned pre = 0u, own = 0u;
#pragma unroll 4
    for (unsigned o = 16 * tid; o < t0; o += 16 * NTHREADS) pre += planes16(ld_dep((const uint4*)(w + o)), nullptr, 0ull);
    const unsigned u0 = (t * NWARPS + warp) * BPU;
    if (BPU == 8) {
        if (lane == 0 && u0 < wbytes) {
            const uint2 v = ld_dep((const uint2*)(w + u0));
            own = planes16(make_uint4(v.x, v.y, 0u, 0u), nullptr, 0ull);
        }
    } else {
        const unsigned o = u0 + 16 * lane;
        if (lane < (int)(BPU / 16) && o < wbytes) own = planes16(ld_dep((const uint4*)(w + o)), nullptr, 0ull);
    }
    pre = __reduce_add_sync(FULL, pre);
    own = __reduce_add_sync(FULL, own);
    if (lane == 0) {
        es.pre[warp] = pre;
        es.own[warp] = own;
    }
    bar_sync_n(BAR_ENCW, NTHREADS);
    unsigned off = 0u, total = 0u;
#pragma unroll
    for (int v = 0; v < NWARPS; ++v) {
        off += es.pre[v] + (v < warp ? es.own[v] : 0u);
        total += es.pre[v] + es.own[v];
    }
    constexpr unsigned long long PB = (1ull << LOG2L) / 8;
    if (t + 1 == it.ntiles && tid == 0 &&
        (total * PB != ld_dep((const unsigned long long*)it.cin + 3) ||
         (LOG2L == 7 && wbytes != 0u && !widths_fit(ld_dep((const uint4*)(w + wbytes - 16))))))
        fail(ctl, ZC_ERR_FORMAT, item_idx);
    return off * PB;
}

// Encoder warp `warp`'s unit of one tile: quantize, delta-code and bit-plane
// pack its U rows, 32 rows at a time (zc_rows.cuh), into its ring segment
// `seg`, and its width bytes into `wb`; returns the segment's size.  `bufs`
// (shared memory) are the warp's two group buffers: the next group's values
// arrive in one while the other is encoded and its payload, built over the
// values, copied to the ring.  HAS_CIN: decode `it.cin` first (same block
// size, unit offsets from k_wscan) and add the local chunk; the FP32 sum then
// goes to `it.raw_out` when that is set.  Null pointers switch a step off.
// HEADS (block heads stored apart, single unpacked streams) writes the heads
// straight to their fixed place in the output.  Thread 0 fills the slot's
// scalars.
template <int LOG2L, int U, bool HAS_CIN, typename TX, bool HEADS = false>
__device__ __forceinline__ int enc_tile(const Launch& P, const Item& it, unsigned item_idx,
                                        unsigned tile_in_item, uint8_t* seg, uint8_t* wb,
                                        unsigned bufs, TileSlot& S, EncShared& es)
{
    static_assert(!HEADS || !HAS_CIN, "heads apart: compression only");
    static_assert(U % GROWS == 0, "whole groups");
    constexpr int L = 1 << LOG2L;
    constexpr int BPG = GELEMS / L;  // blocks per group
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    Ctl* ctl = P.ctl;
    const unsigned long long n = it.n;
    const unsigned long long ue0 = (unsigned long long)tile_in_item * (NWARPS * U * 32) +
                                   (unsigned long long)warp * U * 32;
    const unsigned long long nb = (n + L - 1) >> LOG2L;
    const unsigned long long wbytes = ceil16(nb);
    const bool first = tile_in_item == 0;
    const bool do_cin = HAS_CIN && it.cin != nullptr;
    const bool do_enc = it.out != nullptr;
    if (tid == 0) {
        S.first = first;
        S.last = tile_in_item + 1 == it.ntiles;
        S.head = first ? 32ull + wbytes + (HEADS ? ceil16(3ull * nb) : 0ull) : 0ull;
        S.pub = do_enc;
    }
    const int un = ue0 < n ? (int)min(n - ue0, (unsigned long long)(U * 32)) : 0;  // unit elements
    const TX* const xp = (const TX*)it.x + ue0;
    const bool vec = ((uintptr_t)xp & 15u) == 0;
    // (requesting the whole unit into L2 here cost 5 of 152 us on the 512^3
    // field: it displaces ring lines)
    if (un > 0) stage_in<TX>(xp, un, vec, bufs, ue0 == 0);
    float two_eb_in = 0.0f;
    if (do_cin) {
        if (tid == 0) {
            float eb_in;
            const int lg = check_header(it, ctl, item_idx, LOG2L, eb_in, first);
            es.hdr_bad = lg != LOG2L;
            es.eb_in = eb_in;
            if (es.hdr_bad) S.pub = 0;
        }
        bar_sync_n(BAR_ENCW, NTHREADS);
        if (es.hdr_bad) {
            cp_wait<0>();
            return 0;
        }
        two_eb_in = __fadd_rn(es.eb_in, es.eb_in);
    }
    if (un == 0 && !(do_cin && it.nchunks == 0)) return 0;
    EncArgs A;
    A.eb = it.eb;
    A.two_eb = it.two_eb;
    A.inv = it.inv;
    if (P.eb_from_ctl) {
        A.eb = ctl->eb;
        A.two_eb = ctl->two_eb;
        A.inv = ctl->inv;
    }
    A.r0 = 0;
    A.carry = 0u;
    unsigned long long pos = 0ull;  // received stream: payload position of the group
    uint32_t wv = 0u;               // and its width byte(s) of this lane's row
    if (do_cin) {
        if (it.nchunks == 0) {
            pos = 32ull + wbytes + tile_unit_offset<LOG2L, U>(it, tile_in_item, ctl, item_idx, es);
        } else {
            const unsigned slot = S.g * NWARPS + warp;
            pos = 32ull + wbytes + (dcheck(ctl, slot < P.ws_cap, slot) ? P.offs[slot] : 0ull);
        }
        if (un == 0) return 0;  // (its warp took part in the tile's sums)
        wv = load_widths<LOG2L>(it.cin, nb, ue0 >> LOG2L);
    }
    int err = 0;
    int sbase = 0;  // ring bytes written; the payload so far is sbase + A.r0
#pragma unroll 1
    for (int g = 0; g * GELEMS < un; ++g) {
        const int e0 = g * GELEMS;
        A.nrem = min(un - e0, GELEMS);
        A.buf = bufs + (g & 1) * GBUF;
        const bool more = e0 + GELEMS < un;
        if (more) {
            stage_in<TX>(xp + e0 + GELEMS, un - e0 - GELEMS, vec, bufs + ((g + 1) & 1) * GBUF, false);
            cp_wait<1>();
        } else {
            cp_wait<0>();
        }
        __syncwarp();
        if constexpr (HAS_CIN) {
            if (do_cin) {
                int np, np2, at;
                bool bad = false;
                const int tot = rows_meta<LOG2L>(wv, np, np2, at, bad);
                if (bad) fail(ctl, ZC_ERR_FORMAT, ue0 + e0);
                const bool ok = pos + (unsigned long long)tot <= it.cin_cap;
                if (!ok) {
                    if (lane == 0) fail(ctl, ZC_ERR_FORMAT, S.g * NWARPS + warp);
                    np = np2 = 0;
                }
                const PlaneSrc<false> ps{0u, it.cin + pos + at};
                if (more) wv = load_widths<LOG2L>(it.cin, nb, (ue0 + e0 + GELEMS) >> LOG2L);
                pos += (unsigned long long)tot;
                const unsigned row = A.buf + lane * 128 + ((lane & 7) << 4);
                decode_rows<LOG2L, false, false>(
                    ps, np, np2, 0, 0, two_eb_in, [] {},
                    [&](int c, const float v[4]) {
                        const uint4 x = lds128(row ^ (c << 4));
                        sts128(row ^ (c << 4), __float_as_uint(__fadd_rn(v[0], __uint_as_float(x.x))),
                               __float_as_uint(__fadd_rn(v[1], __uint_as_float(x.y))),
                               __float_as_uint(__fadd_rn(v[2], __uint_as_float(x.z))),
                               __float_as_uint(__fadd_rn(v[3], __uint_as_float(x.w))));
                    });
                __syncwarp();
                if (A.nrem < GELEMS) {  // the padding repeats the last sum
                    const uint32_t v = lds32(elem_addr<float>(A.buf, A.nrem - 1));
                    __syncwarp();
                    for (int e = A.nrem + lane; e < GELEMS; e += 32) sts32(elem_addr<float>(A.buf, e), v);
                    __syncwarp();
                }
                if (!do_enc) {  // the quantizer does not see these sums
                    float m = 0.0f;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const uint4 x = lds128(row ^ (c << 4));
                        m = max3_abs_nan(m, __uint_as_float(x.x), __uint_as_float(x.y));
                        m = max3_abs_nan(m, __uint_as_float(x.z), __uint_as_float(x.w));
                    }
                    if (!isfinite(m)) err |= ZC_ERR_NONFINITE;
                }
            }
            if (it.raw_out != nullptr) {
                float* const op = (float*)it.raw_out + ue0 + e0;
                stage_out<float>(op, A.nrem, ((uintptr_t)op & 15u) == 0, A.buf);
            }
        }
        if (do_enc) {
            const unsigned long long bg = (ue0 + e0) >> LOG2L;  // first block of the group
            if (HEADS) {
                A.hout = it.out + 32 + wbytes + 3ull * bg;
                if (DEBUG_BUILD)
                    dcheck(ctl, 32 + wbytes + 3ull * min(bg + BPG, nb) <= it.out_cap, ue0);
            }
            A.wb = (unsigned)__cvta_generic_to_shared(wb) + g * BPG;
            const int end = A.r0 + encode_rows<LOG2L, TX, HEADS>(A, err);
            __syncwarp();
            // the payload to the ring, in 16-byte chunks; the partial last
            // one is written now and again, complete, with the next group
            int n16 = (end + 15) >> 4;
            if (!dcheck(ctl, end <= GBUF && sbase + 16 * n16 <= seg_bytes(U), ue0)) n16 = 0;
            for (int i = lane; i < n16; i += 32)
                ((uint4*)(seg + sbase))[i] = lds128(A.buf + 16 * i);
            if (lane < 4) A.carry = lds32(A.buf + (end & ~15) + 4 * lane);
            sbase += end & ~15;
            A.r0 = end & 15;
        }
        __syncwarp();  // the buffer is free
    }
    {
        const unsigned bad = __ballot_sync(FULL, err != 0);
        if (bad && lane == __ffs(bad) - 1) fail(ctl, (unsigned)err, ue0);
    }
    return do_enc ? sbase + A.r0 : 0;
}

// Stores of one encoded tile once its place is known: every encoder warp
// copies its unit's segment from the ring and its width bytes; the last tile
// of a stream zero-pads the width array (and the heads) and the payload and
// writes the header.
template <int LOG2L, int U, bool HAS_CIN, bool HEADS = false>
__device__ __forceinline__ void fin_tile(const Launch& P, const Item& it, unsigned item_idx,
                                         unsigned tile_in_item, unsigned g, const TileSlot& S,
                                         const uint8_t* seg, const uint8_t* wb, unsigned buf)
{
    constexpr int L = 1 << LOG2L;
    constexpr int PB = L / 8;
    constexpr int BU = U * 32 / L;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned long long n = it.n;
    const unsigned long long ue0 = (unsigned long long)tile_in_item * (NWARPS * U * 32) +
                                   (unsigned long long)warp * U * 32;
    const unsigned long long nb = (n + L - 1) >> LOG2L;
    const unsigned long long wbytes = ceil16(nb);
    const unsigned long long hbytes = HEADS ? ceil16(3ull * nb) : 0ull;
    int segoff = 0, payload_i = 0;
#pragma unroll
    for (int w = 0; w < NWARPS; ++w) {
        if (w < warp) segoff += S.segsz[w];
        payload_i += S.segsz[w];
    }
    const unsigned long long payload = (unsigned long long)payload_i;
    const unsigned long long ex = S.ex, start = S.start;
    const unsigned long long base = ex + S.head;
    const unsigned long long cap = it.out_cap;
    uint8_t* const out = it.out;
    const unsigned long long end = base + payload;  // unpadded end of this tile's payload
    if (base + payload <= cap) {
        if (dcheck(P.ctl, S.segsz[warp] <= seg_bytes(U), g))
            ring_copy<PB, seg_bytes(U)>(out + base + segoff, seg, S.segsz[warp], buf);
    } else if (tid == 0) {
        fail(P.ctl, ZC_ERR_CAPACITY, g);
    }
    {
        const unsigned long long b0 = ue0 >> LOG2L;
        const unsigned long long pos0 = start + 32 + b0;  // 16-byte aligned when BU is
        if (BU % 16 == 0 && b0 + BU <= nb && pos0 + BU <= cap) {
            if (lane < BU / 16) ((uint4*)(out + pos0))[lane] = ((const uint4*)wb)[lane];
        } else {
            for (int i = lane; i < BU; i += 32) {
                const unsigned long long b = b0 + i;
                const unsigned long long pos = pos0 + i;
                if (b < nb && pos < cap) out[pos] = wb[i];
            }
        }
    }
    if (S.last) {
        const unsigned long long total = ceil16(end);
        const unsigned long long pl = end - start - 32 - wbytes - hbytes;
        for (unsigned long long p = start + 32 + nb + tid; p < start + 32 + wbytes; p += NTHREADS)
            if (p < cap) out[p] = 0;
        if (HEADS)
            for (unsigned long long p = start + 32 + wbytes + 3 * nb + tid;
                 p < start + 32 + wbytes + hbytes; p += NTHREADS)
                if (p < cap) out[p] = 0;
        for (unsigned long long p = end + tid; p < total; p += NTHREADS)
            if (p < cap) out[p] = 0;
        if (tid < 8 && start + 32 <= cap) {
            uint32_t v = 0;
            const int xdt = HAS_CIN ? ZC_F32 : it.x_dtype;
            switch (tid) {
            case 0: v = 0x3176435au; break;  // "ZCv1"
            case 1: v = (uint32_t)xdt | ((uint32_t)LOG2L << 8) | (HEADS ? (2u << 16) : 0u); break;
            case 2: v = (uint32_t)n; break;
            case 3: v = (uint32_t)(n >> 32); break;
            case 4: v = __float_as_uint(P.eb_from_ctl ? P.ctl->eb : it.eb); break;
            case 5: v = (uint32_t)nb; break;
            case 6: v = (uint32_t)pl; break;
            default: v = (uint32_t)(pl >> 32); break;
            }
            ((uint32_t*)(out + start))[tid] = v;
        }
        if (tid == 0) {
            if (it.out_bytes) *it.out_bytes = total - start;
            if (P.packed && !P.grouped) P.seg_off[item_idx + 1] = total;
            else if (P.packed && g + 1 == P.total_tiles) P.seg_off[P.n_items] = total;
        }
    }
}

// One tile of a raw (verbatim) stream: the item's elements of this tile go
// unchanged after the 32-byte header (flag bit 0 set, no width bytes).  Same
// tile geometry, look-back and stream-start protocol as an encoded tile, so
// raw and encoded streams mix in one packed launch.  Nothing is staged: the
// tile's size is known from its element count.
template <int U>
__device__ __forceinline__ int enc_raw(const Item& it, unsigned tile_in_item, TileSlot& S)
{
    if (threadIdx.x == 0) {
        constexpr unsigned long long TE = (unsigned long long)NWARPS * U * 32;
        const unsigned long long es = it.x_dtype == ZC_F32 ? 4ull : 2ull;
        const unsigned long long te0 = (unsigned long long)tile_in_item * TE;
        const unsigned long long cnt = te0 < it.n ? min(it.n - te0, TE) : 0ull;
        S.first = tile_in_item == 0;
        S.last = tile_in_item + 1 == it.ntiles;
        S.head = cnt * es + (tile_in_item == 0 ? 32ull : 0ull);
        S.pub = it.out != nullptr;
    }
    return 0;
}

// Copies `len` bytes (even) from `src` (2-byte aligned) to `dst` (16-byte aligned)
// with one warp: asynchronously through `buf`, both group buffers of the warp, then
// out by 16-byte stores.  Up to 8 KiB are in flight without a register for them:
// several loads in registers made the batch kernel's coded tiles spill (250 messages
// in 4-chunk tiles: 1488 us as here, 1606 with eight).
__device__ __forceinline__ void raw_copy(uint8_t* dst, const uint8_t* src, int len, unsigned buf)
{
    const int lane = threadIdx.x & 31;
    int done = 0;
    if (((uintptr_t)src & 3u) == 0) {
        const bool vec = ((uintptr_t)src & 15u) == 0;
        for (const int whole = len & ~15; done < whole;) {
            const int n = min(whole - done, 2 * GBUF);
            if (vec) {
                for (int o = 16 * lane; o < n; o += 512) cp_async16(buf + o, src + done + o);
            } else {
                for (int o = 4 * lane; o < n; o += 128) cp_async_ca<4>(buf + o, src + done + o);
            }
            cp_commit();
            cp_wait<0>();
            __syncwarp();
            for (int o = 16 * lane; o < n; o += 512) *(uint4*)(dst + done + o) = lds128(buf + o);
            __syncwarp();  // the buffers are free
            done += n;
        }
    }
    for (int o = done + 2 * lane; o < len; o += 256) {
        uint16_t v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = o + 64 * k < len ? ld_dep((const uint16_t*)(src + o + 64 * k)) : (uint16_t)0;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (o + 64 * k < len) *(uint16_t*)(dst + o + 64 * k) = v[k];
    }
}

template <int U>
__device__ __forceinline__ void fin_raw(const Launch& P, const Item& it, unsigned item_idx,
                                        unsigned tile_in_item, unsigned g, const TileSlot& S,
                                        unsigned buf)
{
    constexpr unsigned long long TE = (unsigned long long)NWARPS * U * 32;
    const int tid = threadIdx.x;
    const unsigned long long n = it.n;
    const unsigned long long es = it.x_dtype == ZC_F32 ? 4ull : 2ull;
    const unsigned long long te0 = (unsigned long long)tile_in_item * TE;
    const unsigned long long cnt = te0 < n ? min(n - te0, TE) : 0ull;
    const unsigned long long bytes = cnt * es;
    const unsigned long long ex = S.ex, start = S.start;
    const unsigned long long base = ex + (S.first ? 32ull : 0ull);  // 16-byte aligned
    const unsigned long long cap = it.out_cap;
    uint8_t* const out = it.out;
    if (base + bytes <= cap) {
        const unsigned long long unit = U * 32 * es, w0 = (tid >> 5) * unit;  // this warp's share
        if (w0 < bytes)
            raw_copy(out + base + w0, (const uint8_t*)it.x + te0 * es + w0, (int)min(unit, bytes - w0), buf);
    } else if (tid == 0) {
        fail(P.ctl, ZC_ERR_CAPACITY, g);
    }
    if (S.last) {
        const unsigned long long end = ex + S.head;
        const unsigned long long total = ceil16(end);
        const unsigned long long pl = n * es;
        for (unsigned long long p = end + tid; p < total; p += NTHREADS)
            if (p < cap) out[p] = 0;
        if (tid < 8 && start + 32 <= cap) {
            uint32_t v = 0;
            switch (tid) {
            case 0: v = 0x3176435au; break;  // "ZCv1"
            case 1: v = (uint32_t)it.x_dtype | (5u << 8) | (1u << 16); break;  // raw flag
            case 2: v = (uint32_t)n; break;
            case 3: v = (uint32_t)(n >> 32); break;
            case 4: v = 0u; break;  // eb: none
            case 5: v = 0u; break;  // no blocks
            case 6: v = (uint32_t)pl; break;
            default: v = (uint32_t)(pl >> 32); break;
            }
            ((uint32_t*)(out + start))[tid] = v;
        }
        if (tid == 0) {
            if (it.out_bytes) *it.out_bytes = total - start;
            if (P.packed && !P.grouped) P.seg_off[item_idx + 1] = total;
            else if (P.packed && g + 1 == P.total_tiles) P.seg_off[P.n_items] = total;
        }
    }
}

// ---- item sources ------------------------------------------------------------

struct ItemsSrc {
    const Launch& P;
    __device__ unsigned find(unsigned g) const
    {
        if (P.items == nullptr) return 0u;
        if (P.tile_map != nullptr) return P.tile_map[g];
        unsigned lo = 0, hi = P.n_items;
        while (hi - lo > 1) {
            const unsigned mid = (lo + hi) >> 1;
            if (P.items[mid].tile_begin <= g) lo = mid;
            else hi = mid;
        }
        return lo;
    }
    __device__ Item get(unsigned i) const { return P.items != nullptr ? P.items[i] : P.one; }
};

// Scatter pack: segments of one input, described by value in the kernel
// parameters (so a call needs no descriptor upload).
constexpr int SCATTER_MAX = 1024;
struct ScatterParams {
    unsigned tile_begin[SCATTER_MAX + 1];
    unsigned long long displ[SCATTER_MAX];
    unsigned long long count[SCATTER_MAX];
};
struct ScatterSrc {
    const Launch& P;
    const ScatterParams& S;
    __device__ unsigned find(unsigned g) const
    {
        unsigned lo = 0, hi = P.n_items;
        while (hi - lo > 1) {
            const unsigned mid = (lo + hi) >> 1;
            if (S.tile_begin[mid] <= g) lo = mid;
            else hi = mid;
        }
        return lo;
    }
    __device__ Item get(unsigned i) const
    {
        Item it = P.one;  // shared fields: out, out_cap, eb, dtype
        const unsigned long long es = it.x_dtype == ZC_F32 ? 4ull : 2ull;
        it.x = (const uint8_t*)P.one.x + S.displ[i] * es;
        it.n = S.count[i];
        it.tile_begin = S.tile_begin[i];
        it.ntiles = S.tile_begin[i + 1] - S.tile_begin[i];
        it.out_bytes = nullptr;
        return it;
    }
};

// Published by the last encoder warp to finish a tile: the tile's aggregate
// (its byte count), so that the look-backs of the tiles after it need not wait
// until this CTA's resolver warp reaches it (the resolver handles its tiles in
// order, and a tile it is still waiting on would hold back this one's
// aggregate).  The resolver then publishes the tile's inclusive prefix.  A
// chain's first tile publishes its prefix at once (resolver), and a withheld
// tile (test hook) publishes nothing.
__device__ __forceinline__ void publish_aggregate(const Launch& P, const TileSlot& S, unsigned E)
{
    if (!S.valid || !S.pub) return;
    const unsigned g0 = P.packed ? 0u : S.g - S.tile;
    if (S.g == g0 || (long long)S.g == P.wc.withhold || S.g >= P.ws_cap) return;
    unsigned long long agg = S.head;
#pragma unroll
    for (int w = 0; w < NWARPS; ++w) agg += (unsigned long long)S.segsz[w];
    rec_store(P.chB.rec + S.g, E, ST_AGG, S.last != 0, agg);
}

// Resolver warp: the tile's place in the chain (look-back over the tiles
// before it) and, in packed mode, its stream's start.
__device__ __forceinline__ void resolve_slot(const Launch& P, TileSlot& S, unsigned E)
{
    int ok = 0;
    unsigned long long ex = 0ull, start = 0ull;
    if (S.pub && dcheck(P.ctl, S.g < P.ws_cap && S.item < max(P.n_items, 1u), S.g)) {
        unsigned long long agg = S.head;
#pragma unroll
        for (int w = 0; w < NWARPS; ++w) agg += (unsigned long long)S.segsz[w];
        const unsigned g0 = P.packed ? 0u : S.g - S.tile;
        bool expired = false;
        // the encoder warps published the aggregate already (publish_aggregate)
        ex = lookback_warp(P.chB, S.g, g0, agg, S.last != 0, E, P.wc, P.ctl, expired, true);
        ok = !expired && packed_start_warp(P, S.first != 0, S.item, ex, S.g, E, start);
    }
    if ((threadIdx.x & 31) == 0) {
        S.ex = ex;
        S.start = start;
        S.ok = ok;
    }
}

// The encoder CTA.  Tickets are taken in order, so a tile only ever waits for
// tiles taken earlier by CTAs that are running or done; every resolver
// publishes its tiles in ticket order, so the chain always advances.  The
// last CTA to finish advances the launch generation.
//   enc(item, index, tile in item, segment, width bytes, stage, slot, shared) -> unit size
//   fin(item, index, tile in item, ticket, slot, segment, width bytes, free group buffer)
// Barrier protocol per tile in slot s: the encoder warps arrive on BAR_ENC + s
// after encoding it, the resolver waits there, resolves it and arrives on
// BAR_RES + s, where the encoder warps wait NS - 1 tiles later before
// storing it.  A slot's barriers are used again only after both sides have
// passed them, and every path through the loops meets every barrier.
template <int U, typename Src, typename Enc, typename Fin>
__device__ __forceinline__ void enc_pipeline(const Launch& P, const Src& src, Enc enc, Fin fin)
{
    constexpr int NS = enc_slots(U);  // tiles in flight
    constexpr int D = NS - 1;         // tiles between a tile's encoding and its stores
    __shared__ TileSlot slots[NS];
    __shared__ EncShared es;
    extern __shared__ __align__(128) uint8_t dsm[];  // group buffers, width bytes [slot][warp][2U]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // every thread: what the kernels before wrote (a relative bound, offsets,
    // the tile map) is read below and in every tile
    grid_dep_wait();
    grid_dep_launch();
    const unsigned modulus = P.total_tiles + gridDim.x - 1u;
    const bool rings = (unsigned long long)gridDim.x * ring_cta_bytes(U) <= P.ring_bytes;
    unsigned g0 = 0u;  // thread 0: the first ticket, taken with the control block's words
    if (tid == 0) {
        if (rings) g0 = atomicInc(&P.ctl->ticket, modulus);
        es.E = ld_volatile_u32(&P.ctl->epoch) + 1u;
        int a = ld_volatile_u32(&P.ctl->magic) != WS_MAGIC;
        if (a) {
            fail(P.ctl, ZC_ERR_WORKSPACE, 0);
        } else if (!rings) {
            a = 1;  // more CTAs than rings: the whole launch does nothing
            if (blockIdx.x == 0) fail(P.ctl, ZC_ERR_WORKSPACE, 1);
        } else if (P.eb_from_ctl && ld_volatile_u32(&P.ctl->eb_ok) != 1u) {
            a = 2;
        }
        es.abort = a;
    }
    __syncthreads();
    if (es.abort == 1) return;
    const bool no_eb = es.abort == 2;
    const unsigned E = es.E;
    uint8_t* const ring = P.ring + (unsigned long long)blockIdx.x * ring_cta_bytes(U);
    if (warp < NWARPS) {
        auto seg_of = [&](int s) { return ring + (unsigned long long)(s * NWARPS + warp) * seg_bytes(U); };
        auto wb_of = [&](int s) { return dsm + NWARPS * 2 * GBUF + (s * NWARPS + warp) * (U * 2); };
        const unsigned bufs = (unsigned)__cvta_generic_to_shared(dsm) + warp * (2 * GBUF);
        auto store = [&](int q) {
            bar_sync_n(BAR_RES + q, ENC_THREADS);
            const TileSlot& Q = slots[q];
            if (Q.ok) {
                const Item it = src.get(Q.item);
                fin(it, Q.item, Q.tile, Q.g, Q, seg_of(q), wb_of(q), bufs);
            }
        };
        int s = 0;
        for (int i = 0;; ++i) {
            bar_sync_n(BAR_ENCW, NTHREADS);  // slot s's previous tile is stored
            if (tid == 0) {
                TileSlot& S = slots[s];
                const unsigned g = i == 0 ? g0 : atomicInc(&P.ctl->ticket, modulus);
                S.g = g;
                S.valid = g < P.total_tiles;
                S.item = g < P.total_tiles ? src.find(g) : 0u;
                S.pub = 0;
                S.nfin = 0;
            }
            bar_sync_n(BAR_ENCW, NTHREADS);
            TileSlot& S = slots[s];
            const bool valid = S.valid != 0;
            int lo = 0;
            if (valid && !no_eb) {
                const Item it = src.get(S.item);
                const unsigned t = S.g - it.tile_begin;
                if (tid == 0) S.tile = t;
                lo = enc(it, S.item, t, seg_of(s), wb_of(s), bufs, S, es);
            }
            if (lane == 0) {
                S.segsz[warp] = lo;
                __threadfence_block();
                if (atomicAdd(&S.nfin, 1) == NWARPS - 1) {  // the tile's last encoder warp
                    __threadfence_block();
                    publish_aggregate(P, S, E);
                }
            }
            bar_arrive_n(BAR_ENC + s, ENC_THREADS);
            if (!valid) {
                // the tiles still waiting for their stores, oldest first
                for (int k = (i < D ? i : D) - 1; k >= 0; --k) store((s + NS - 1 - k) % NS);
                break;
            }
            if (i >= D) store((s + 1) % NS);
            s = s + 1 == NS ? 0 : s + 1;
        }
    } else {
        int s = 0;
        while (true) {
            bar_sync_n(BAR_ENC + s, ENC_THREADS);
            TileSlot& S = slots[s];
            if (!S.valid) break;
            resolve_slot(P, S, E);
            __syncwarp();
            bar_arrive_n(BAR_RES + s, ENC_THREADS);
            s = s + 1 == NS ? 0 : s + 1;
        }
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        if (atomicInc(&P.ctl->done, gridDim.x - 1u) == gridDim.x - 1u) {
            P.ctl->epoch = E;
            __threadfence();
        }
    }
}

template <int LOG2L, int U, typename TX, bool HEADS = false>
__global__ void __launch_bounds__(ENC_THREADS, ENC_CTAS_PER_SM) k_compress(const Launch P)
{
    enc_pipeline<U>(
        P, ItemsSrc{P},
        [&](const Item& it, unsigned idx, unsigned t, uint8_t* seg, uint8_t* wb, unsigned bufs,
            TileSlot& S, EncShared& es) {
            return enc_tile<LOG2L, U, false, TX, HEADS>(P, it, idx, t, seg, wb, bufs, S, es);
        },
        [&](const Item& it, unsigned idx, unsigned t, unsigned g, const TileSlot& S,
            const uint8_t* seg, const uint8_t* wb, unsigned buf) { fin_tile<LOG2L, U, false, HEADS>(P, it, idx, t, g, S, seg, wb, buf); });
}

template <int LOG2L, int U, typename TX>
__global__ void __launch_bounds__(ENC_THREADS, ENC_CTAS_PER_SM) k_scatter(const Launch P,
                                                                          const ScatterParams SP)
{
    enc_pipeline<U>(
        P, ScatterSrc{P, SP},
        [&](const Item& it, unsigned idx, unsigned t, uint8_t* seg, uint8_t* wb, unsigned bufs,
            TileSlot& S, EncShared& es) {
            return enc_tile<LOG2L, U, false, TX>(P, it, idx, t, seg, wb, bufs, S, es);
        },
        [&](const Item& it, unsigned idx, unsigned t, unsigned g, const TileSlot& S,
            const uint8_t* seg, const uint8_t* wb, unsigned buf) { fin_tile<LOG2L, U, false>(P, it, idx, t, g, S, seg, wb, buf); });
}

template <int LOG2L, int U>
__global__ void __launch_bounds__(ENC_THREADS, ENC_CTAS_PER_SM) k_reduce(const Launch P)
{
    enc_pipeline<U>(
        P, ItemsSrc{P},
        [&](const Item& it, unsigned idx, unsigned t, uint8_t* seg, uint8_t* wb, unsigned bufs,
            TileSlot& S, EncShared& es) {
            return enc_tile<LOG2L, U, true, float>(P, it, idx, t, seg, wb, bufs, S, es);
        },
        [&](const Item& it, unsigned idx, unsigned t, unsigned g, const TileSlot& S,
            const uint8_t* seg, const uint8_t* wb, unsigned buf) { fin_tile<LOG2L, U, true>(P, it, idx, t, g, S, seg, wb, buf); });
}

// ---- batched compression -----------------------------------------------------
// Every item is a stream of its own block size and input type (or raw), all
// packed back to back by one chain; the CTAs take tiles of all items from one
// ticket counter, so one launch of a few CTAs per SM covers any mix of
// message sizes.
template <int U>
__global__ void __launch_bounds__(ENC_THREADS, ENC_CTAS_PER_SM) k_batch(const Launch P)
{
    enc_pipeline<U>(
        P, ItemsSrc{P},
        [&](const Item& it, unsigned idx, unsigned t, uint8_t* seg, uint8_t* wb, unsigned bufs,
            TileSlot& S, EncShared& es) -> int {
            const bool f32 = it.x_dtype == ZC_F32;
            switch (it.log2L) {
            case 4:
                return f32 ? enc_tile<4, U, false, float>(P, it, idx, t, seg, wb, bufs, S, es)
                           : enc_tile<4, U, false, uint16_t>(P, it, idx, t, seg, wb, bufs, S, es);
            case 5:
                return f32 ? enc_tile<5, U, false, float>(P, it, idx, t, seg, wb, bufs, S, es)
                           : enc_tile<5, U, false, uint16_t>(P, it, idx, t, seg, wb, bufs, S, es);
            case 6:
                return f32 ? enc_tile<6, U, false, float>(P, it, idx, t, seg, wb, bufs, S, es)
                           : enc_tile<6, U, false, uint16_t>(P, it, idx, t, seg, wb, bufs, S, es);
            case 7:
                return f32 ? enc_tile<7, U, false, float>(P, it, idx, t, seg, wb, bufs, S, es)
                           : enc_tile<7, U, false, uint16_t>(P, it, idx, t, seg, wb, bufs, S, es);
            default: return enc_raw<U>(it, t, S);
            }
        },
        [&](const Item& it, unsigned idx, unsigned t, unsigned g, const TileSlot& S,
            const uint8_t* seg, const uint8_t* wb, unsigned buf) {
            switch (it.log2L) {
            case 4: fin_tile<4, U, false>(P, it, idx, t, g, S, seg, wb, buf); break;
            case 5: fin_tile<5, U, false>(P, it, idx, t, g, S, seg, wb, buf); break;
            case 6: fin_tile<6, U, false>(P, it, idx, t, g, S, seg, wb, buf); break;
            case 7: fin_tile<7, U, false>(P, it, idx, t, g, S, seg, wb, buf); break;
            default: fin_raw<U>(P, it, idx, t, g, S, buf); break;
            }
        });
}

// Batched decompression: item idx's stream, from a packed buffer written by an
// earlier launch.  A start or an end outside the buffer, or a start that is
// not 16-byte aligned, leaves a stream too short for its header (reported as
// a format error by the decoder).
__device__ __forceinline__ void resolve_packed(const Launch& P, Item& it, unsigned idx)
{
    if (P.in_off == nullptr) return;
    const unsigned long long a = P.in_off[idx];
    const unsigned long long b = P.in_off[P.grouped ? P.n_items : idx + 1];
    const bool ok = (a & 15ull) == 0 && a <= b && b <= P.in_cap;
    it.cin = P.in_base + (ok ? a : 0ull);
    it.cin_cap = ok ? b - a : 0ull;
}

#ifdef ZC_DECODE_KERNELS  // defined by the one translation unit that launches them

// Item of every encoder tile (by_chunk: of every width-scan chunk) of a
// multi-item launch, so that a CTA finds its ticket's item with one load
// instead of a binary search of dependent loads.
// Launched dependent on a width scan (the fused ring step), the map is
// built while the scan runs; the kernel then waits for the scan, so that it
// never completes before it (the step launched dependent on the map reads
// the scan's offsets too).  Thread 0 always reaches the wait.
__global__ void __launch_bounds__(NTHREADS) k_tile_map(const Item* items, unsigned n_items,
                                                      unsigned total_tiles, unsigned* map,
                                                      int by_chunk)
{
    grid_dep_launch();
    const unsigned g = blockIdx.x * NTHREADS + threadIdx.x;
    if (g >= total_tiles) return;
    unsigned lo = 0, hi = n_items;
    while (hi - lo > 1) {
        const unsigned mid = (lo + hi) >> 1;
        const unsigned b = by_chunk ? ld_dep(&items[mid].chunk_begin) : ld_dep(&items[mid].tile_begin);
        if (b <= g) lo = mid;
        else hi = mid;
    }
    map[g] = lo;
    grid_dep_wait();
}

// ---- grouped batches ------------------------------------------------------------
// The tiles of all messages of one block size (classes: raw, 16, 32, 64, 128)
// take consecutive tickets, so the CTAs running at any time mostly run one
// encoder variant.  Within a class, messages keep their order.  Three small
// launches over GROUP_T messages per CTA: per-CTA tile sums of every class;
// one CTA turns them into every CTA's first ticket per class; each CTA then
// gives its messages their first tickets and fills the ticket -> item map.
constexpr int GROUP_T = 256;
constexpr int GROUP_CLASSES = 5;
__device__ __forceinline__ int group_class(int log2L) { return log2L < 4 ? 0 : log2L - 3; }

__global__ void __launch_bounds__(GROUP_T) k_group_count(const Item* items, unsigned n_items,
                                                         unsigned* part)
{
    grid_dep_wait();
    grid_dep_launch();
    __shared__ unsigned red[GROUP_CLASSES][GROUP_T / 32];
    const unsigned i = blockIdx.x * GROUP_T + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int c = -1;
    unsigned t = 0;
    if (i < n_items) {
        c = group_class(ld_dep(&items[i].log2L));
        t = ld_dep(&items[i].ntiles);
    }
#pragma unroll
    for (int k = 0; k < GROUP_CLASSES; ++k) {
        const unsigned v = __reduce_add_sync(FULL, c == k ? t : 0u);
        if (lane == 0) red[k][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < GROUP_CLASSES) {
        unsigned v = 0;
        for (int w = 0; w < GROUP_T / 32; ++w) v += red[threadIdx.x][w];
        part[(size_t)blockIdx.x * GROUP_CLASSES + threadIdx.x] = v;
    }
}

// One CTA of 1024 threads: part[b][c] (tiles of class c in CTA b's messages)
// becomes the first ticket of class c in CTA b: the class's base (the tiles
// of all smaller classes) plus the class's tiles in CTAs before b.
__global__ void __launch_bounds__(1024) k_group_scan(unsigned* part, unsigned nblk)
{
    grid_dep_wait();
    grid_dep_launch();
    __shared__ unsigned wsum[32];
    __shared__ unsigned carry[GROUP_CLASSES];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < GROUP_CLASSES) carry[tid] = 0;
    __syncthreads();
    // pass over the classes: exclusive scans within each class
    for (int c = 0; c < GROUP_CLASSES; ++c) {
        for (unsigned b0 = 0; b0 < nblk; b0 += 1024) {
            const unsigned b = b0 + tid;
            const unsigned v = b < nblk ? part[(size_t)b * GROUP_CLASSES + c] : 0u;
            unsigned s = v;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned o = __shfl_up_sync(FULL, s, off);
                if (lane >= off) s += o;
            }
            if (lane == 31) wsum[warp] = s;
            __syncthreads();
            if (warp == 0) {
                unsigned w = wsum[lane];
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const unsigned o = __shfl_up_sync(FULL, w, off);
                    if (lane >= off) w += o;
                }
                wsum[lane] = w;  // inclusive over warps
            }
            __syncthreads();
            const unsigned excl = carry[c] + (warp ? wsum[warp - 1] : 0u) + s - v;
            if (b < nblk) part[(size_t)b * GROUP_CLASSES + c] = excl;
            __syncthreads();
            if (tid == 0) carry[c] += wsum[31];
            __syncthreads();
        }
    }
    // class bases: the tiles of the smaller classes
    unsigned base = 0;
    for (int c = 0; c < GROUP_CLASSES; ++c) {
        const unsigned tot = carry[c];
        for (unsigned b = tid; b < nblk; b += 1024) part[(size_t)b * GROUP_CLASSES + c] += base;
        base += tot;
    }
}

__global__ void __launch_bounds__(GROUP_T) k_group_place(Item* items, unsigned n_items,
                                                         const unsigned* part, unsigned* map)
{
    grid_dep_wait();
    grid_dep_launch();
    __shared__ unsigned wsum[GROUP_CLASSES][GROUP_T / 32];
    const unsigned i = blockIdx.x * GROUP_T + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int c = -1;
    unsigned t = 0;
    if (i < n_items) {
        c = group_class(items[i].log2L);
        t = items[i].ntiles;
    }
    unsigned mine = 0;  // exclusive sum of this class's tiles before message i within the warp
#pragma unroll
    for (int k = 0; k < GROUP_CLASSES; ++k) {
        const unsigned v = c == k ? t : 0u;
        unsigned s = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned o = __shfl_up_sync(FULL, s, off);
            if (lane >= off) s += o;
        }
        if (lane == 31) wsum[k][warp] = s;
        if (c == k) mine = s - v;
    }
    __syncthreads();
    if (i >= n_items) return;
    unsigned first = part[(size_t)blockIdx.x * GROUP_CLASSES + c] + mine;
    for (int w = 0; w < warp; ++w) first += wsum[c][w];
    items[i].tile_begin = first;
    for (unsigned k = 0; k < t; ++k) map[first + k] = i;
}

// ---- width scan: payload offset of every decode tile --------------------------
// One CTA per chunk of WSCAN warp units of one item; thread i sums the plane
// bytes of unit i from its width bytes, four 16-byte loads in flight (the first
// one of a line brings the others' bytes to L1); a CTA scan and a look-back over the
// item's chunks give every unit's payload offset (global decode slot = item
// tile slot * NWARPS + unit in tile).  A multi-item launch finds a chunk's
// item in P.tile_map, here the chunk -> item map (k_tile_map by chunk).
__global__ void __launch_bounds__(NTHREADS) k_wscan(const Launch P)
{
    __shared__ Smem sm;
    __shared__ int wsum[NWARPS];
    grid_dep_wait();
    grid_dep_launch();  // the decoder after it may be launched now (it waits for the offsets)
    const unsigned modulus = P.total_tiles + gridDim.x - 1u;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the first ticket is taken with the control block's words: one round trip
    unsigned first = 0u;
    if (tid == 0) {
        first = atomicInc(&P.ctl->ticket, modulus);
        sm.E = ld_volatile_u32(&P.ctl->epoch) + 1u;
        sm.abort = ld_volatile_u32(&P.ctl->magic) != WS_MAGIC;
        if (sm.abort) fail(P.ctl, ZC_ERR_WORKSPACE, 0);
    }
    for (bool again = false;; again = true) {
        __syncthreads();
        if (warp == 0) {
            const unsigned g = __shfl_sync(FULL, again && lane == 0 ? atomicInc(&P.ctl->ticket, modulus) : first, 0);
            unsigned it = 0;
            if (P.items != nullptr && g < P.total_tiles) {
                if (P.tile_map != nullptr) {
                    it = P.tile_map[g];  // the chunk map of this launch
                } else {  // the last item that begins at or before g, 32 candidates per round trip
                    for (unsigned i0 = 0; i0 < P.n_items; i0 += 32) {
                        const bool le = i0 + lane < P.n_items && P.items[i0 + lane].chunk_begin <= g;
                        const unsigned m = __ballot_sync(FULL, le);
                        if (m) it = i0 + 31 - __clz(m);
                        if (m != FULL) break;
                    }
                }
            }
            if (lane == 0) {
                sm.ticket = g;
                sm.item = it;
            }
        }
        __syncthreads();
        if (sm.abort) return;
        const unsigned c = sm.ticket;
        if (c >= P.total_tiles) break;
        Item it = P.items != nullptr ? P.items[sm.item] : P.one;
        resolve_packed(P, it, sm.item);
        if (it.cin == nullptr) continue;  // nothing received: no offsets needed
        const unsigned chunk = c - it.chunk_begin;
        float eb_in;
        const int lg = check_header(it, P.ctl, sm.item, -1, eb_in, false);
        if (lg < 4) continue;  // raw or malformed: the decoder reports it
        const int lgb = lg & 7;  // block size (heads apart or not: same widths)
        const unsigned long long L = 1ull << lgb;
        const unsigned long long nb = (it.n + L - 1) >> lgb;
        const int PB = (int)(L / 8);
        const unsigned long long ntile = (unsigned long long)it.ntiles * NWARPS;  // units
        const unsigned long long k = (unsigned long long)chunk * WSCAN + tid;    // unit in item
        const int bpt = (P.urows * 32) >> lgb;                                   // blocks per unit
        // bpt is 8 (32-row units at L = 128) or a power of two from 16 on
        const unsigned long long b0 = k * bpt, wend = ceil16(nb);
        int sum = 0;
        if (k < ntile && b0 < wend) {
            const uint8_t* const w = it.cin + 32 + b0;
            if (bpt == 8) {
                const uint2 v = ld_dep((const uint2*)w);
                sum = planes16(make_uint4(v.x, v.y, 0u, 0u), P.ctl, b0);
            } else {
                const int nv = (int)min((unsigned long long)bpt, wend - b0) / 16;
                for (int i = 0; i < nv; i += 4) {
                    uint4 v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        v[q] = i + q < nv ? ld_dep((const uint4*)w + i + q) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                    for (int q = 0; q < 4; ++q) sum += planes16(v[q], P.ctl, b0 + 16 * (i + q));
                }
            }
            sum *= PB;
        }
        int tot;
        const int ex = warp_excl_scan(sum, lane, tot);
        if (lane == 0) wsum[warp] = tot;
        __syncthreads();
        unsigned long long wbase = 0, cagg = 0;
        for (int w = 0; w < NWARPS; ++w) {
            if (w < warp) wbase += wsum[w];
            cagg += wsum[w];
        }
        bool to = false;
        if (DEBUG_BUILD && tid == 0) dcheck(P.ctl, c < P.ws_cap, c);
        const unsigned long long cex =
            lookback_cta(P.chC, c, it.chunk_begin, cagg, false, sm.E, P.wc, P.ctl, to, sm.lb);
        if (to) continue;
        const unsigned long long oslot = (unsigned long long)it.tile_begin * NWARPS + k;
        if (k < ntile && dcheck(P.ctl, oslot < P.ws_cap, oslot)) P.offs[oslot] = cex + wbase + ex;
        if (chunk + 1 == it.nchunks && tid == 0) {
            const unsigned long long payload = ld_dep((const unsigned long long*)it.cin + 3);
            if (cex + cagg != payload) fail(P.ctl, ZC_ERR_FORMAT, sm.item);
        }
    }
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicInc(&P.ctl->done, gridDim.x - 1u) == gridDim.x - 1u) {
            P.ctl->epoch = sm.E;
            __threadfence();
        }
    }
}

// ---- decompression -------------------------------------------------------------

// Raw streams: copy (and convert) the elements of this warp unit.
template <int DU>
__device__ __forceinline__ void unit_raw_copy(const Item& it, int src_dtype, unsigned long long ue0)
{
    const uint8_t* src = it.cin + 32;
    const int lane = threadIdx.x & 31;
    for (int r = 0; r < DU; r += 4) {  // four loads in flight
        const unsigned long long e = ue0 + (unsigned long long)r * 32 + lane;
        float v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned long long ek = e + 32 * k;
            v[k] = ek >= it.n ? 0.0f
                   : src_dtype == ZC_F32 ? ld_dep((const float*)src + ek)
                                         : bf16_to_f32(ld_dep((const unsigned short*)src + ek));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (e + 32 * k < it.n) store_raw(it.raw_out, it.out_dtype, e + 32 * k, v[k]);
    }
}

// One warp unit of a coded stream (zc_rows.cuh), 32 rows at a time.  `bufs`:
// the warp's two group buffers; a group's payload arrives in its buffer while the
// group before it is decoded, and the decoded rows take its place before they are
// stored, 16 bytes a lane.
// off_local >= 0: the unit's payload offset found by the caller (a small
// item's decoder CTA), in place of the width scan's P.offs[slot].
template <int LOG2L, typename TO, int DU, bool HEADS = false>
__device__ __forceinline__ void unit_decode(const Launch& P, const Item& it, unsigned slot,
                                            unsigned long long ue0, float two_eb, unsigned bufs,
                                            long long off_local)
{
    static_assert(DU % GROWS == 0, "whole groups");
    constexpr int L = 1 << LOG2L;
    constexpr int RPB = Blk<LOG2L>::RPB;
    const int lane = threadIdx.x & 31;
    const unsigned long long nb = (it.n + L - 1) >> LOG2L;
    const unsigned long long b0 = ue0 >> LOG2L;
    const int un = (int)min(it.n - ue0, (unsigned long long)(DU * 32));
    uint32_t wn = load_widths<LOG2L>(it.cin, nb, b0 + GELEMS / L);
    const uint32_t wv = load_widths<LOG2L>(it.cin, nb, b0);
    const bool slot_ok = off_local >= 0 || dcheck(P.ctl, slot < P.ws_cap, slot);
    unsigned long long pos = 32ull + ceil16(nb) + (HEADS ? ceil16(3ull * nb) : 0ull) +
                             (off_local >= 0 ? (unsigned long long)off_local
                                             : (slot_ok ? P.offs[slot] : 0ull));
    struct Group {
        int np, np2;
        unsigned sp;  // the lane's first plane word in the group buffer
    };
    // Requests the payload of a group (at `pos`) into its buffer.  The 16-byte
    // chunks it touches lie inside the stream (16-byte aligned and padded).
    auto fetch = [&](uint32_t wv, unsigned buf) {
        Group G;
        int at;
        bool bad = false;
        const int tot = rows_meta<LOG2L>(wv, G.np, G.np2, at, bad);
        if (bad) fail(P.ctl, ZC_ERR_FORMAT, b0);
        const unsigned long long c0 = pos & ~15ull, c1 = ceil16(pos + (unsigned long long)tot);
        if (slot_ok && c1 <= it.cin_cap) {
            const uint8_t* const src = it.cin + c0;
            const int n16 = (int)((c1 - c0) >> 4);
            for (int i = lane; i < n16; i += 32) cp_async16(buf + 16 * i, src + 16 * i);
        } else {
            if (lane == 0) fail(P.ctl, ZC_ERR_FORMAT, slot);
            G.np = G.np2 = 0;
        }
        cp_commit();
        G.sp = buf + (unsigned)(pos & 15ull) + at;
        pos += (unsigned long long)tot;
        return G;
    };
    // Two groups: both copies before the first is decoded.  More: each group's
    // copy while the one before it is decoded (two copies in flight throughout
    // took more registers: 377 us for a batch that takes 359).
    constexpr bool PAIR = DU == 2 * GROWS;
    Group G = fetch(wv, bufs), G1 = G;
    if (PAIR) G1 = fetch(wn, bufs + GBUF);
#pragma unroll 1
    for (int g = 0; g * GELEMS < un; ++g) {
        const int nrem = min(un - g * GELEMS, GELEMS);
        const unsigned buf = bufs + (g & 1) * GBUF;
        if (!PAIR && (g + 1) * GELEMS < un) {
            G1 = fetch(wn, bufs + ((g + 1) & 1) * GBUF);
            if ((g + 2) * GELEMS < un)
                wn = load_widths<LOG2L>(it.cin, nb, b0 + (unsigned)((g + 2) * (GELEMS / L)));
        } else if (!PAIR) {
            cp_commit();
        }
        int h0 = 0, h16 = 0;
        if (HEADS) {  // the heads of this lane's blocks
            const unsigned long long b = b0 + (unsigned)(g * (GELEMS / L)) +
                                         (L == 16 ? 2 * lane : lane / RPB);
            const uint8_t* const hp = it.cin + 32 + ceil16(nb) + 3ull * b;
            if ((lane & (RPB - 1)) == 0 && b < nb) h0 = load_head(hp);
            if (L == 16 && b + 1 < nb) h16 = load_head(hp + 3);
        }
        if (!PAIR || g == 0) cp_wait<1>();
        else cp_wait<0>();
        __syncwarp();
        const PlaneSrc<true> ps{G.sp, nullptr};
        const unsigned row = sizeof(TO) == 4 ? buf + lane * 128 + ((lane & 7) << 4)
                                             : buf + lane * 64 + (((lane >> 1) & 3) << 4);
        decode_rows<LOG2L, true, HEADS>(
            ps, G.np, G.np2, h0, h16, two_eb, [] { __syncwarp(); },
            [&](int c, const float v[4]) {
                if (sizeof(TO) == 4) {
                    sts128(row ^ (c << 4), __float_as_uint(v[0]), __float_as_uint(v[1]),
                           __float_as_uint(v[2]), __float_as_uint(v[3]));
                } else {
                    sts64((row ^ ((c >> 1) << 4)) + (c & 1) * 8, f32_to_bf16x2(v[0], v[1]),
                          f32_to_bf16x2(v[2], v[3]));
                }
            });
        __syncwarp();
        TO* const op = (TO*)it.raw_out + ue0 + g * GELEMS;
        stage_out<TO>(op, nrem, ((uintptr_t)op & 15u) == 0, buf);
        if (!PAIR) __syncwarp();  // the buffer is free
        G = G1;
    }
    cp_wait<0>();
}

// Items planned with no width-scan chunks (small ones): the decoder CTA of tile
// t sums the plane bytes of the item's blocks before its tile itself and its
// warps' units (one value per warp), which gives every warp its unit's payload
// offset; the item's last tile checks the total against the header's payload
// size, as the width scan does, and every tile reports its own bytes that no
// width can have, padding included.  Called by every thread of the CTA (coded
// streams only: lg >= 4).
template <bool BATCH, int DU>
__device__ __forceinline__ unsigned long long local_unit_offset(const Item& it, int lg, unsigned t,
                                                                Ctl* ctl, unsigned item_idx)
{
    __shared__ unsigned s_pre[NWARPS], s_own[NWARPS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int lgb = lg & 7;
    const unsigned long long PB = (1ull << lgb) / 8;
    const unsigned long long nb = (it.n + (1ull << lgb) - 1) >> lgb;
    const unsigned bpu = (unsigned)(DU * 32) >> lgb;  // blocks per unit: 16 to 256
    // width bytes, 16 at a time (the array is zero padded to 16; a unit and a
    // tile start at multiples of 16)
    const uint4* const w = (const uint4*)(it.cin + 32);
    const unsigned v_end = (unsigned)(ceil16(nb) / 16);
    const unsigned v_pre = min(t * NWARPS * bpu / 16, v_end);
    unsigned pre = 0u;  // planes: at most 25 per block
#pragma unroll 4
    for (unsigned v = tid; v < v_pre; v += NTHREADS) pre += planes16(ld_dep(w + v), nullptr, 0ull);
    const unsigned v_lo = (t * NWARPS + warp) * (bpu / 16) + lane;
    unsigned own = 0u;
    if (lane < (int)(bpu / 16) && v_lo < v_end) own = planes16(ld_dep(w + v_lo), ctl, 16ull * v_lo);
    pre = __reduce_add_sync(FULL, pre);
    own = __reduce_add_sync(FULL, own);
    if (lane == 0) {
        s_pre[warp] = pre;
        s_own[warp] = own;
    }
    __syncthreads();
    unsigned off = 0u, total = 0u;
#pragma unroll
    for (int v = 0; v < NWARPS; ++v) {
        off += s_pre[v] + (v < warp ? s_own[v] : 0u);
        total += s_pre[v] + s_own[v];
    }
    if (t + 1 == it.ntiles && tid == 0) {
        const unsigned long long payload = ld_dep((const unsigned long long*)it.cin + 3);
        if (total * PB != payload) {
            // a batch's small items may have widths in their padding, as long as
            // what these stand for lies inside the stream's room
            unsigned pad = 0u;
            if (BATCH && it.ntiles <= DEC_LOCAL_TILES &&
                32ull + ceil16(nb) + (lg >= 8 ? ceil16(3ull * nb) : 0ull) + total * PB <= it.cin_cap)
                for (unsigned long long b = nb; b < ceil16(nb); ++b) pad += planes_of(ld_dep(it.cin + 32 + b));
            if ((total - pad) * PB != payload) fail(ctl, ZC_ERR_FORMAT, item_idx);
        }
    }
    return off * PB;
}

// NWARPS warp units per CTA, one per warp, independent of each other; the
// block size comes from the stream's header.
// BATCH: a multi-item launch; LOCAL: (some) items find their own unit offsets.
// The decoder of a single scanned stream is compiled without that path, which
// would cost it registers.
template <bool BATCH, bool LOCAL, int DU>
__device__ __forceinline__ void decompress_tile(const Launch& P)
{
    extern __shared__ __align__(128) uint8_t dsm[];
    if (BATCH || LOCAL) grid_dep_wait();
    grid_dep_launch();
    const unsigned tile = blockIdx.x;
    unsigned idx = 0;
    if (P.tile_map != nullptr) {
        idx = P.tile_map[tile];
    } else if (P.items != nullptr) {
        unsigned lo = 0, hi = P.n_items;
        while (hi - lo > 1) {
            const unsigned mid = (lo + hi) >> 1;
            if (P.items[mid].tile_begin <= tile) lo = mid;
            else hi = mid;
        }
        idx = lo;
    }
    Item it = P.items != nullptr ? P.items[idx] : P.one;
    resolve_packed(P, it, idx);
    // a workspace that is not initialised is refused (by the width scan where
    // there is one; batched items of a few tiles never had one)
    if (LOCAL && it.nchunks == 0 && (!BATCH || it.ntiles > DEC_LOCAL_TILES) &&
        ld_volatile_u32(&P.ctl->magic) != WS_MAGIC) {
        if (threadIdx.x == 0) fail(P.ctl, ZC_ERR_WORKSPACE, 0);
        return;
    }
    const unsigned t = tile - it.tile_begin;
    const int warp = threadIdx.x >> 5;
    const unsigned long long ue0 = ((unsigned long long)t * NWARPS + warp) * (DU * 32);
    const unsigned slot = tile * NWARPS + warp;
    const unsigned bufs = (unsigned)__cvta_generic_to_shared(dsm) + warp * (2 * GBUF);
    float eb_in;
    const int lg = check_header<!BATCH && !LOCAL>(it, P.ctl, idx, -1, eb_in, threadIdx.x == 0 && t == 0);
    long long loff = -1;  // the unit's payload offset, when this CTA finds it
    if (LOCAL && it.nchunks == 0 && lg >= 4)  // uniform in the CTA
        loff = (long long)local_unit_offset<BATCH, DU>(it, lg, t, P.ctl, idx);
    // the width scan's offsets are read from here on: a single-stream decoder
    // launched dependent on the scan has looked up its tile and checked the
    // header while the scan ran, and waits for it now.  Every thread passes
    // this wait, so the decoder never completes before the scan (later
    // launches on the stream find the scan finished).
    if (!BATCH && !LOCAL) grid_dep_wait();
    if (ue0 >= it.n) return;
    const float two = __fadd_rn(eb_in, eb_in);
    if (it.out_dtype == ZC_F32) {
        switch (lg) {
        case 4: unit_decode<4, float, DU>(P, it, slot, ue0, two, bufs, loff); return;
        case 5: unit_decode<5, float, DU>(P, it, slot, ue0, two, bufs, loff); return;
        case 6: unit_decode<6, float, DU>(P, it, slot, ue0, two, bufs, loff); return;
        case 7: unit_decode<7, float, DU>(P, it, slot, ue0, two, bufs, loff); return;
        case 12: unit_decode<4, float, DU, true>(P, it, slot, ue0, two, bufs, loff); return;
        case 13: unit_decode<5, float, DU, true>(P, it, slot, ue0, two, bufs, loff); return;
        case 14: unit_decode<6, float, DU, true>(P, it, slot, ue0, two, bufs, loff); return;
        case 15: unit_decode<7, float, DU, true>(P, it, slot, ue0, two, bufs, loff); return;
        default: break;
        }
    } else {
        switch (lg) {
        case 4: unit_decode<4, uint16_t, DU>(P, it, slot, ue0, two, bufs, loff); return;
        case 5: unit_decode<5, uint16_t, DU>(P, it, slot, ue0, two, bufs, loff); return;
        case 6: unit_decode<6, uint16_t, DU>(P, it, slot, ue0, two, bufs, loff); return;
        case 7: unit_decode<7, uint16_t, DU>(P, it, slot, ue0, two, bufs, loff); return;
        case 12: unit_decode<4, uint16_t, DU, true>(P, it, slot, ue0, two, bufs, loff); return;
        case 13: unit_decode<5, uint16_t, DU, true>(P, it, slot, ue0, two, bufs, loff); return;
        case 14: unit_decode<6, uint16_t, DU, true>(P, it, slot, ue0, two, bufs, loff); return;
        case 15: unit_decode<7, uint16_t, DU, true>(P, it, slot, ue0, two, bufs, loff); return;
        default: break;
        }
    }
    if (lg == -2) unit_raw_copy<DU>(it, ZC_F32, ue0);
    else if (lg == -3) unit_raw_copy<DU>(it, ZC_BF16, ue0);
}

template <bool BATCH, bool LOCAL, int DU>
__global__ void __launch_bounds__(NTHREADS, DEC_CTAS_PER_SM) k_decompress(const Launch P)
{
    decompress_tile<BATCH, LOCAL, DU>(P);
}

#endif  // ZC_DECODE_KERNELS

}  // namespace zc
