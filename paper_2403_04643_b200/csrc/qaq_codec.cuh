// The one copy of the codec arithmetic and of the tile layout, used by the quantize, re-quantize,
// export and decode kernels (not part of the ABI).
//
// Codes (Section 4.1 of the paper: the range [min,max] of a token's non-outlier entries is cut into 2^B equal
// segments): step = (max-min) * 2^-B, code = min(2^B-1, floor((x-min) * (1/step))) in binary32 with separately
// rounded operations; an outlier's code slot holds 0.
//
// Tile layout in the code pool.  A tile (QAQ_TILE consecutive tokens of one (b,h) and tensor) holds its tokens sorted by
// width, widest first (ties in token order); the position of a token in that order is its slot, kept with its width in
// the token's metadata.  Everything of one width is one section, and a section is a list of rows:
//   keys:    a row is one token.
//   values:  a row is a group of four consecutive slots, at the width of the widest of them (empty slots are zero).
// All sections of a tile are cut into the same units, which are what a lane of the decode kernels loads at a time: the
// registers it hands to the integer tensor-core instruction are one or two instructions away from the loaded words.
// Nibble words: 32 codes of up to 4 bits are four words v0..v3, eight codes a word, code A(b) of byte b in its low and
// B(b) in its high nibble, so that (v & mask) and (v & mask << 4) are operand registers (four codes, one per byte).
// A unit stores them in as many words x as the codes have bits:
//   4 bits: x_u = v_u     2 bits: x0 = v0 | v1 << 2, x1 = v2 | v3 << 2     1 bit: x0 = v0 | v1 << 1 | v2 << 2 | v3 << 3
//   3 bits: x_u = v_u (u < 3) plus one bit of every nibble of v3 in the free bit of theirs: bit i of a nibble of v3 is
//           bit 3 of the same nibble of x_i
// and codes of 5..8 bits are two units, the low 4 bits (the main part) and the rest (the high part).  The main parts of
// all rows of 4 bits and more are one list, so the main part of a tile is at most four lists and its high part four more.
//   keys:    unit p of a row (p < head_dim/32) = the token's channels 32p .. 32p+31; in v_u, byte b is A = channel
//            32p + 8u + b and B = channel 32p + 8u + 4 + b.
//   values:  unit 4p + b of a row = byte b of those words for its four tokens: byte i of v_u belongs to slot 4G + i, A and
//            B as above.  Rows of a list are interleaved by fours (the last m rows of a list by m): unit e of row
//            4k + t lies at index 16k * head_dim/32 + e * m + t, which makes the loads of a warp contiguous.
// Storage: a header of QAQ_TILE_HDR bytes (number of rows of every width, byte offsets of the zones below, the largest magnitude
// among the ranges and the outliers of the tile as a binary16 pattern), then
// the parts of the sections ordered by unit size so that every load is aligned: zone 4 (main parts of widths 8 .. 4,
// 16-byte units; then the high part of width 8), zone 2 (high part of width 6, then width 2; 8-byte units), zone 13 (high
// part of width 7, width 3, high part of width 5, width 1; 12- and 4-byte units).  A tile of keys takes the header plus
// sum_t head_dim*B_t/8 bytes; a tile of values that plus what the widest tokens of mixed groups cost the others.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "qaq.h"

namespace qaqc {

// ------------------------------------------------------------------------------------------ small helpers
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}
// binary32 (x - c) with x a binary16 value: one rounding, same as widening x exactly and subtracting
__device__ __forceinline__ float sub_f32_f16(unsigned short x, float c) {
    float d;
    asm("sub.rn.f32.f16 %0, %1, %2;" : "=f"(d) : "h"(x), "f"(c));
    return d;
}

// B = min{b in [bmin,bmax] : v <= c * 2^b}, bmax if none (the bit count of Section 4.1 without a logarithm;
// c * 2^b is an exact power-of-two scaling).  For positive normal v and c the answer is read off the exponents:
// with v = mv * 2^ev, c = mc * 2^ec (mv, mc in [1,2)) the smallest b is ev - ec if mv <= mc, else ev - ec + 1.
__device__ __forceinline__ int ladder(float v, float c, int bmin, int bmax) {
    if (!(c > 0.f)) return bmax;
    if (v <= __fmul_rn(c, (float)(1 << bmin))) return bmin;
    const int vb = __float_as_int(v), cb = __float_as_int(c);
    if (cb < 0x00800000 || vb < 0x00800000) {  // subnormal operand: plain ladder
        for (int b = bmin; b <= bmax; ++b)
            if (v <= __fmul_rn(c, (float)(1 << b))) return b;
        return bmax;
    }
    const int b = (vb >> 23) - (cb >> 23) + (((vb & 0x7FFFFF) > (cb & 0x7FFFFF)) ? 1 : 0);
    return b < bmin ? bmin : (b > bmax ? bmax : b);
}

// step of a token from its stored range and width (exact scaling)
__device__ __forceinline__ float step_of(float mn, float mx, int B) {
    return __fmul_rn(__fsub_rn(mx, mn), __int_as_float((127 - B) << 23));
}

// Codes of 32 channels held as 16 binary16 pairs (v[k] = channels 2k, 2k+1; outliers already replaced by -inf,
// which yields code 0): creg[j] = codes of channels 4j..4j+3, one per byte.
__device__ __forceinline__ void codes32(const uint32_t (&v)[16], float mn, float mx, int B, uint32_t (&creg)[8]) {
    const float step = step_of(mn, mx, B);
    const float inv = step > 0.f ? __fdiv_rn(1.0f, step) : 0.f;
    // zero step (constant token): every code is 0, and -inf * 0 = NaN must not clamp to the top code
    const float topf = step > 0.f ? (float)((1 << B) - 1) : 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        uint32_t f[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t pair = v[2 * j + (i >> 1)];
            const unsigned short h = (i & 1) ? (unsigned short)(pair >> 16) : (unsigned short)(pair & 0xFFFF);
            float t = __fmul_rn(sub_f32_f16(h, mn), inv);   // -inf for an outlier
            t = fminf(t, topf);
            f[i] = __float_as_uint(__fadd_rd(t, 8388608.0f));   // 2^23 + floor(t): the code is the low byte (0 for -inf)
        }
        creg[j] = prmt(prmt(f[0], f[1], 0x0040u), prmt(f[2], f[3], 0x0040u), 0x5410u);
    }
}

// outliers (entries outside [lo2, hi2], NaN included) of 16 binary16 pairs replaced by -inf
__device__ __forceinline__ void mask_outliers32(uint32_t (&v)[16], __half2 lo2, __half2 hi2) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const __half2 x = *reinterpret_cast<const __half2*>(&v[k]);
        const uint32_t m = __hge2_mask(x, lo2) & __hle2_mask(x, hi2);
        v[k] = (v[k] & m) | (0xFC00FC00u & ~m);
    }
}

template <int NW>          // aligned to the widest access taken: 16 bytes for multiples of four words, 8 for two, else 4
__device__ __forceinline__ void load_words(const uint8_t* p, uint32_t* w) {
    if (NW % 4 == 0) {
#pragma unroll
        for (int i = 0; i < NW; i += 4) {
            const uint4 v = *reinterpret_cast<const uint4*>(p + 4 * i);
            w[i] = v.x; w[i + 1] = v.y; w[i + 2] = v.z; w[i + 3] = v.w;
        }
    } else if (NW == 2) {
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        w[0] = v.x; w[1] = v.y;
    } else {
#pragma unroll
        for (int i = 0; i < NW; ++i) w[i] = reinterpret_cast<const uint32_t*>(p)[i];
    }
}

// ------------------------------------------------------------------------------------------ tile layout
constexpr int QAQ_TILE_HDR = 16;

// largest tile: the header and 64 tokens at 8 bits
__host__ __device__ constexpr int tile_bytes_max(int D) { return QAQ_TILE_HDR + QAQ_TILE_TOKENS * D; }
// units per row: keys head_dim/32, values four times that
template <int D, bool IS_V> constexpr int UNITS = IS_V ? D / 8 : D / 32;

constexpr uint32_t NIB = 0x0F0F0F0Fu;
// (a & m) | (b & ~m)
__device__ __forceinline__ uint32_t bitsel(uint32_t a, uint32_t b, uint32_t m) { return (a & m) | (b & ~m); }

// The w-bit words of a unit, from its nibble words (bits beyond the w lowest of a nibble are zero).
__device__ __forceinline__ void store_nibbles(uint8_t* dst, int w, const uint32_t (&v)[4]) {
    if (w == 4) {
        *reinterpret_cast<uint4*>(dst) = make_uint4(v[0], v[1], v[2], v[3]);
    } else if (w == 3) {
        uint32_t* x = reinterpret_cast<uint32_t*>(dst);
        x[0] = v[0] | ((v[3] & 0x11111111u) << 3);
        x[1] = v[1] | ((v[3] & 0x22222222u) << 2);
        x[2] = v[2] | ((v[3] & 0x44444444u) << 1);
    } else if (w == 2) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(v[0] | (v[1] << 2), v[2] | (v[3] << 2));
    } else {
        *reinterpret_cast<uint32_t*>(dst) = v[0] | (v[1] << 1) | (v[2] << 2) | (v[3] << 3);
    }
}
// The nibble words of codes one per byte: bits shift .. shift+3 of them.
__device__ __forceinline__ void nibbles_of(const uint32_t (&creg)[8], int shift, uint32_t (&v)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const uint32_t a = shift ? creg[2 * u] >> 4 : creg[2 * u], b = shift ? creg[2 * u + 1] : creg[2 * u + 1] << 4;
        v[u] = bitsel(a, b, NIB);
    }
}
// The nibble words of a unit of w-bit words.  Bits of a nibble beyond the w lowest are undefined.
template <int W>
__device__ __forceinline__ void nibble_words(const uint32_t* x, uint32_t (&v)[4]) {
    if (W == 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = x[u];
    } else if (W == 3) {
        v[0] = x[0]; v[1] = x[1]; v[2] = x[2];
        v[3] = ((x[0] >> 3) & 0x11111111u) | ((x[1] >> 2) & 0x22222222u) | ((x[2] >> 1) & 0x44444444u);
    } else if (W == 2) {
        v[0] = x[0]; v[1] = x[0] >> 2; v[2] = x[1]; v[3] = x[1] >> 2;
    } else {
        v[0] = x[0]; v[1] = x[0] >> 1; v[2] = x[0] >> 2; v[3] = x[0] >> 3;
    }
}
// ------------------------------------------------------------------------------------------ a tile by two warps
// What the kernels that give a tile 64 threads, one per token, find out about it.  Counts by width are kept a byte each, widths
// 1..4 in one word and 5..8 in the other, and sums over widths are taken in the bytes (they stay below 256).
constexpr uint32_t ONES = 0x01010101u;
__device__ __forceinline__ uint32_t byte_of(uint32_t lo, uint32_t hi, int w) { return prmt(lo, hi, (uint32_t)(w - 1)) & 0xFFu; }

// The lanes of this warp whose token has the same width (0: no token), and for the other warp how many have which.
__device__ __forceinline__ uint32_t count_half(int b, int lane, uint32_t (&count)[2]) {
    const uint32_t b0 = __ballot_sync(0xFFFFFFFFu, (b - 1) & 1), b1 = __ballot_sync(0xFFFFFFFFu, (b - 1) & 2), b2 = __ballot_sync(0xFFFFFFFFu, (b - 1) & 4);
    const uint32_t there = __ballot_sync(0xFFFFFFFFu, b != 0);
    auto tokens_of = [&](int k) { return (k & 1 ? b0 : ~b0) & (k & 2 ? b1 : ~b1) & (k & 4 ? b2 : ~b2) & there; };
    if (lane < 8) reinterpret_cast<uint8_t*>(count)[lane] = (uint8_t)__popc(tokens_of(lane));
    return tokens_of(b - 1);
}

// Rows of a tile by width: how many, and the first one.
struct TileRows { uint32_t nlo, nhi, slo, shi; };
// from the stored counts of rows
__device__ __forceinline__ TileRows rows_of_header(uint32_t nlo, uint32_t nhi) {
    const uint32_t ulo = nlo * ONES, uhi = nhi * ONES + (ulo >> 24) * ONES, all = (uhi >> 24) * ONES;      // rows of a width or less
    return {nlo, nhi, all - ulo, all - uhi};
}
// from the tokens of the halves of the tile; slot: this thread's token's place in the order
template <bool IS_V>
__device__ __forceinline__ TileRows rows_of_counts(const uint32_t (&count)[2][2], int b, uint32_t alike, int warp, int lane, int& slot) {
    const uint32_t clo = count[0][0] + count[1][0], chi = count[0][1] + count[1][1];
    const uint32_t ulo = clo * ONES, uhi = chi * ONES + (ulo >> 24) * ONES, n = uhi >> 24;
    slot = (int)(n - byte_of(ulo, uhi, b) + (warp ? byte_of(count[0][0], count[0][1], b) : 0u)) + __popc(alike & ((1u << lane) - 1u));
    if (!IS_V) return {clo, chi, n * ONES - ulo, n * ONES - uhi};
    // groups of four slots; a section has those whose first slot is in it
    TileRows r;
    r.slo = (((n + 3) * ONES - ulo) >> 2) & 0x3F3F3F3Fu;
    r.shi = (((n + 3) * ONES - uhi) >> 2) & 0x3F3F3F3Fu;
    r.nlo = ((r.slo << 8) | ((n + 3) >> 2)) - r.slo;
    r.nhi = __funnelshift_l(r.slo, r.shi, 8) - r.shi;
    return r;
}
// width of a row: one more than the widths that begin behind it
__device__ __forceinline__ int width_of_row(const TileRows& r, int row) {
    const uint32_t y = (uint32_t)row * ONES | 0x80808080u;
    return 9 - __popc((y - r.slo) & 0x80808080u) - __popc((y - r.shi) & 0x80808080u);
}
// Offsets of the parts (in the order of the storage, above), in words per unit: dot products of the rows of every width.
template <int D, bool IS_V>
__device__ __forceinline__ uint32_t at_words(const TileRows& r, uint32_t wlo, uint32_t whi) {
    return (uint32_t)QAQ_TILE_HDR + (uint32_t)(4 * UNITS<D, IS_V>) * __dp4a(r.nlo, wlo, __dp4a(r.nhi, whi, 0u));
}
template <int D, bool IS_V> __device__ __forceinline__ uint32_t at_h8(const TileRows& r) { return at_words<D, IS_V>(r, 0x04000000u, 0x04040404u); }
template <int D, bool IS_V> __device__ __forceinline__ uint32_t at_z2(const TileRows& r) { return at_words<D, IS_V>(r, 0x04000000u, 0x08040404u); }
template <int D, bool IS_V> __device__ __forceinline__ uint32_t at_z13(const TileRows& r) { return at_words<D, IS_V>(r, 0x04000200u, 0x08040604u); }
template <int D, bool IS_V> __device__ __forceinline__ uint32_t tile_total(const TileRows& r) { return at_words<D, IS_V>(r, 0x04030201u, 0x08070605u); }
template <int D, bool IS_V>
__device__ __forceinline__ uint4 header_of(const TileRows& r, uint32_t top) {
    return make_uint4(r.nlo, r.nhi, at_h8<D, IS_V>(r) | (at_z2<D, IS_V>(r) << 16), at_z13<D, IS_V>(r) | (top << 16));
}
// the largest magnitude a range (min | max << 16, binary16) has
__device__ __forceinline__ uint32_t top_of(uint32_t range) { return max(range & 0x7FFFu, (range >> 16) & 0x7FFFu); }
// Where a row of width w lies: byte offsets of its main and high part, and for values how far apart its units are (in units).
struct RowPlace { uint32_t main, high, mm, mh; };
template <int D, bool IS_V>
__device__ __forceinline__ RowPlace place_row(const TileRows& r, int row, int w) {
    constexpr int P = D / 32;
    const uint32_t m3 = at_words<D, IS_V>(r, 0x04000200u, 0x08070604u), m2 = at_words<D, IS_V>(r, 0x04000000u, 0x08040604u);
    const uint32_t m1 = at_words<D, IS_V>(r, 0x04030200u, 0x08070605u), h5 = at_words<D, IS_V>(r, 0x04030200u, 0x08070604u);
    const int wm = min(w, 4), wh = max(w - 4, 0), start = (int)byte_of(r.slo, r.shi, w), n = (int)byte_of(r.nlo, r.nhi, w);
    const int rm = w >= 4 ? row : row - start, rh = row - start;
    RowPlace o;
    o.main = w >= 4 ? (uint32_t)QAQ_TILE_HDR : w == 3 ? m3 : w == 2 ? m2 : m1;
    o.high = w == 8 ? at_h8<D, IS_V>(r) : w == 7 ? at_z13<D, IS_V>(r) : w == 6 ? at_z2<D, IS_V>(r) : h5;
    o.mm = o.mh = 0;
    if (!IS_V) {
        o.main += rm * P * 4 * wm;
        o.high += rh * P * 4 * wh;
    } else {                           // unit e of the row lies at e * m units from here; main parts of 4 bits and more are one list
        const int rows = w >= 4 ? (int)((r.slo >> 16) & 0xFFu) : n;
        o.mm = min(4, rows - (rm & ~3)); o.mh = min(4, n - (rh & ~3));
        o.main += ((rm & ~3) * (D / 8) + (rm & 3)) * 4 * wm;
        o.high += ((rh & ~3) * (D / 8) + (rh & 3)) * 4 * wh;
    }
    return o;
}
// The largest of the first nv (at most W) of W scores, `stride` apart.  Rows a token has no score in are left out of the maximum,
// not of the loads (the ring is allocated in full): those of a batch depend on nothing and go out together.  What is left after
// whole batches is read eight at a time, the last row again where there are fewer.  (One at a time, 128 tokens with 255 rows
// behind 32 (b,h) x 4096 took 29.2 us, so 17.4; 4096 tokens of 256 (b,h) with 16 rows 244 and 189.)  SEEN: rows from the 33rd on are read only as far as some token of the warp has a
// score in them (re-selection of 32 (b,h) x 4096 with one score each in 255 rows: every row read 24.6 us, so 4.5; a vote in front
// of every batch, 128 x 2048 with 32 rows take 7.4 instead of 6.6 us).  By whole warps.
template <int BATCH, bool SEEN = false>
__device__ __forceinline__ float window_max(const float* r, int W, long stride, int nv) {
    float m = __int_as_float(0xff800000);
    int i = 0;
    auto batch = [&]() {
        float v[BATCH];
#pragma unroll
        for (int u = 0; u < BATCH; ++u) v[u] = r[u * stride];
        if (__all_sync(0xFFFFFFFFu, i + BATCH <= nv)) {
#pragma unroll
            for (int u = 0; u < BATCH; ++u) m = fmaxf(m, v[u]);
        } else {
#pragma unroll
            for (int u = 0; u < BATCH; ++u) if (i + u < nv) m = fmaxf(m, v[u]);
        }
        i += BATCH;
        r += BATCH * stride;
    };
    const int first = SEEN ? min(W, 32) : W;
#pragma unroll 1
    while (i + BATCH <= first) batch();
    if (SEEN && W > 32) {
        W = max(32, __reduce_max_sync(0xFFFFFFFFu, nv));
#pragma unroll 1
        while (i + BATCH <= W) batch();
    }
#pragma unroll 1
    for (; i < W; i += 8, r += 8 * stride) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = r[min(u, W - 1 - i) * stride];
#pragma unroll
        for (int u = 0; u < 8; ++u) if (i + u < nv) m = fmaxf(m, v[u]);
    }
    return m;
}
// The same by one loop, whose last batch reads the last row again where it is short of rows: less code to fetch, which a one-token
// append waits for (with the loops above it takes 1 us more); whole tiles have the address arithmetic to pay (256 (b,h) x 4096: 3 us).
template <int BATCH>
__device__ __forceinline__ float window_max_one_loop(const float* r, int W, long stride, int nv) {
    float m = __int_as_float(0xff800000);
#pragma unroll 1
    for (int i = 0; i < W; i += BATCH) {
        const int rows = W - i;
        float v[BATCH];
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            v[u] = *r;
            if (u + 1 < rows) r += stride;
        }
#pragma unroll
        for (int u = 0; u < BATCH; ++u) if (i + u < nv) m = fmaxf(m, v[u]);
    }
    return m;
}
// The nibble words of one part (w bits, 1..4) of a lane's 32 channels of one token.  Keys: the unit at `at`; values: byte i of
// units 4p .. 4p+3, which lie m units apart from `at` on.
template <int W, bool IS_V>
__device__ __forceinline__ void take_words(const uint8_t* at, uint32_t m, int i, uint32_t (&v)[4]) {
    uint32_t x[W];
    if (!IS_V) {
        load_words<W>(at, x);
    } else {
        uint32_t u[4][W];
#pragma unroll
        for (int b = 0; b < 4; ++b) load_words<W>(at + b * m * 4 * W, u[b]);
        const uint32_t sel = 0x0040u + 0x0011u * (uint32_t)i;          // byte i of both operands
#pragma unroll
        for (int c = 0; c < W; ++c) x[c] = prmt(prmt(u[0][c], u[1][c], sel), prmt(u[2][c], u[3][c], sel), 0x5410u);
    }
    nibble_words<W>(x, v);
    constexpr uint32_t mask = 0x11111111u * ((1u << W) - 1u);
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] &= mask;
}
template <bool IS_V>
__device__ __forceinline__ void take_nibbles(const uint8_t* at, int w, uint32_t m, int i, uint32_t (&v)[4]) {
    if (w == 4) take_words<4, IS_V>(at, m, i, v);
    else if (w == 3) take_words<3, IS_V>(at, m, i, v);
    else if (w == 2) take_words<2, IS_V>(at, m, i, v);
    else take_words<1, IS_V>(at, m, i, v);
}
// Both parts of a stored token out of a tile in shared memory (`bytes` long): lo, hi are the nibble words of bits 0..3 and
// 4..7 of its codes.  main, high: byte offsets of its row, ow: the row's width, mm, mh: distances of the units of values,
// i: the slot's place in its group.  Whatever the metadata say, nothing beyond the buffer is read.
template <int D, bool IS_V>
__device__ __forceinline__ void take_token(const uint8_t* tile, uint32_t bytes, uint32_t main, uint32_t high, int ow, uint32_t mm, uint32_t mh, int i, int p,
                                           uint32_t (&lo)[4], uint32_t (&hi)[4]) {
    const int wm = min(ow, 4), wh = ow - 4;
    const uint32_t m_at = main + (IS_V ? 4 * p * mm : (uint32_t)p) * 4 * wm;
    if (m_at + (IS_V ? 3 * mm * 4 * wm : 0u) + 16 <= bytes) take_nibbles<IS_V>(tile + m_at, wm, mm, i, lo);
    if (wh > 0) {
        const uint32_t h_at = high + (IS_V ? 4 * p * mh : (uint32_t)p) * 4 * wh;
        if (h_at + (IS_V ? 3 * mh * 4 * wh : 0u) + 16 <= bytes) take_nibbles<IS_V>(tile + h_at, wh, mh, i, hi);
    }
}
// 4 x 4 bytes of every word, transposed over the four lanes that are S and 2S apart: lane i of them gets byte i of all four
template <int S>
__device__ __forceinline__ void transpose4(uint32_t (&v)[4], int i) {
#pragma unroll
    for (int step = 0; step < 2; ++step) {
        const bool up = step ? (i & 1) : (i >> 1);
        // the halves of a word (step 0) or its odd and even bytes (step 1): one stays, the other goes
        const uint32_t away = step ? (up ? 0x6420u : 0x7531u) : (up ? 0x5410u : 0x7632u);
        const uint32_t join0 = step ? (up ? 0x3514u : 0x5240u) : (up ? 0x3254u : 0x5410u);
        const uint32_t join1 = step ? (up ? 0x3716u : 0x7260u) : (up ? 0x3276u : 0x7610u);
#pragma unroll
        for (int k = 0; k < 4; k += 2) {
            const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, prmt(v[k], v[k + 1], away), step ? S : 2 * S);
            v[k] = prmt(v[k], o, join0);
            v[k + 1] = prmt(v[k + 1], o, join1);
        }
    }
}

}  // namespace qaqc
