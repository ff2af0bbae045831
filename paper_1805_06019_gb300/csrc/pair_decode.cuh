// Block decode and colour by one thread, two values to a 32-bit word, shared by
// the full decode, the binned decode and the renderer's on-demand decode; and
// the writer of output rows of any alignment.
#pragma once

#include "rlfc_device.cuh"

namespace rlfc {

// Reconstructions and residuals are held as 16-bit values plus a bias of
// 2^14, two to a word: then parent + residual is one 32-bit add for two
// values (no carry crosses a half while every value stays in
// [-2^14, 2^14)), and the inverse YCoCg-R runs on two pixels per
// instruction.
constexpr uint32_t kB2 = 0x40004000u;     // the bias in both halves (a zero pair)
constexpr uint32_t kHalfB2 = 0x20002000u;

// Decoder tables, built at compile time: the 28 modes (payload bits | b << 8
// | kind << 12, four unused entries), and the digits of t in base 3 (t <
// 256, five digits) and in base 5 (t < 128, three digits), three bits per
// digit.
struct DecodeTables {
    uint32_t mode[32];
    uint16_t dig[256 + 128];
};

constexpr DecodeTables make_tables()
{
    DecodeTables t{};
    constexpr uint32_t modes[kNumModes] = RLFC_MODE_TABLE_INIT;
    for (int k = 0; k < 32; k++)
        t.mode[k] = k < kNumModes ? modes[k] : 0u;
    for (uint32_t i = 0; i < 256 + 128; i++) {
        const uint32_t base = i < 256 ? 3u : 5u, n = i < 256 ? 5u : 3u;
        uint32_t x = i < 256 ? i : i - 256, e = 0;
        for (uint32_t k = 0; k < n; k++) {
            e |= (x % base) << (3 * k);
            x /= base;
        }
        t.dig[i] = (uint16_t)e;
    }
    return t;
}

static __device__ const DecodeTables g_tables = make_tables();

// ---- one BISE block, any mode, by one thread ---------------------------------
//
// The 16 values come out dequantised and biased, two to a word (value 2j in
// the low half of out[j], 2j + 1 in the high half), and are built two at a
// time: a pair stands for low half + 2^16 * high half modulo 2^32, and every
// term of (digit << b | low part) << shift + (min << shift) + 2^14 enters it
// as first + 2^16 * second, the possibly negative min included.  The terms of
// a half may leave its 16 bits (a minimum far below the values that the block
// holds); their sums do not (the loader bounds the values), so the result is
// exact, with one 32-bit multiply-add per term.
// Digits (trit and quint blocks) come first in the payload: the groups are
// split by the base-3 / base-5 tables (digit v at bits 3v of a 64-bit word).
// The low parts of block row rr (values 4rr .. 4rr + 3, 4b <= 40 bits) sit
// in one 64-bit window of the payload read from three record words.
__device__ __forceinline__ void decode_block_pairs(const uint32_t *rec, uint32_t pos, uint32_t hdr, uint32_t q,
                                                   const uint32_t *s_mode, const uint16_t *s_dig, uint32_t out[8])
{
    const uint32_t mp = s_mode[hdr & 31u];
    const uint32_t b = mode_b(mp), kind = mode_kind(mp);
    const uint32_t scale = 1u << (q + ((hdr >> 5) & 3u));
    const int32_t mn = ((int32_t)(hdr << 14)) >> 21;   // header bits 7..17, sign-extended
    const uint32_t base = (uint32_t)mn * scale + 0x4000u;
    const uint32_t base2 = base + (base << 16);
    const uint32_t m2 = ((1u << b) - 1u) * 0x10001u;   // the low-part mask in both halves
    const uint32_t sb = scale << b;
    uint64_t dw = 0;   // digit v at bits 3v
    uint32_t D = 0;    // digit bits in front of the low parts
    if (kind != 0) {
        const uint32_t *w = rec + (pos >> 5);
        const uint32_t x0 = w[0], x1 = w[1], x2 = w[2];
        const uint32_t A0 = __funnelshift_r(x0, x1, pos), A1 = __funnelshift_r(x1, x2, pos);
        if (kind == 1) {
            // trits: three 8-bit digit groups and a 2-bit one (value 15), low parts from bit 26
            uint32_t t3 = (A0 >> 24) & 3u;
            t3 = t3 == 3u ? 0u : t3;
            dw = (uint64_t)s_dig[A0 & 0xFFu] | ((uint64_t)s_dig[(A0 >> 8) & 0xFFu] << 15) |
                 ((uint64_t)s_dig[(A0 >> 16) & 0xFFu] << 30) | ((uint64_t)t3 << 45);
            D = 26;
        } else {
            // quints: five 7-bit digit groups and a 3-bit one (value 15), low parts from bit 38
            uint32_t t5 = (A1 >> 3) & 7u;
            t5 = t5 >= 5u ? t5 - 5u : t5;
            dw = (uint64_t)s_dig[256u + (A0 & 0x7Fu)] | ((uint64_t)s_dig[256u + ((A0 >> 7) & 0x7Fu)] << 9) |
                 ((uint64_t)s_dig[256u + ((A0 >> 14) & 0x7Fu)] << 18) |
                 ((uint64_t)s_dig[256u + ((A0 >> 21) & 0x7Fu)] << 27) |
                 ((uint64_t)s_dig[256u + (__funnelshift_r(A0, A1, 28) & 0x7Fu)] << 36) | ((uint64_t)t5 << 45);
            D = 38;
        }
    }
#pragma unroll
    for (uint32_t rr = 0; rr < 4; rr++) {
        const uint32_t lp = pos + D + 4u * rr * b;   // the row's first low part
        const uint32_t *w = rec + (lp >> 5);
        const uint32_t y0 = w[0], y1 = w[1], y2 = w[2];
        const uint32_t lo = __funnelshift_r(y0, y1, lp), hi = __funnelshift_r(y1, y2, lp);
        // low parts of values (0, 1) and (2, 3) of the row, one per half (shifts <= 3b <= 30)
        const uint32_t l01 = __byte_perm(lo, __funnelshift_r(lo, hi, b), 0x5410) & m2;
        const uint32_t l23 = __byte_perm(__funnelshift_r(lo, hi, 2 * b), __funnelshift_r(lo, hi, 3 * b), 0x5410) & m2;
        // digits of the row: 12 bits; d * (1 + 2^13) puts digit 1 at bit 16
        const uint32_t dr = (uint32_t)(dw >> (12 * rr)) & 0xFFFu;
        const uint32_t d01 = (dr * 0x2001u) & 0x70007u, d23 = ((dr >> 6) * 0x2001u) & 0x70007u;
        out[2 * rr] = d01 * sb + l01 * scale + base2;
        out[2 * rr + 1] = d23 * sb + l23 * scale + base2;
    }
}

// Reads the 18-bit headers of a record one after the other through a 64-bit
// window, a word at a time.
struct HeaderReader {
    const uint32_t *next;
    uint64_t win;
    uint32_t have;
    __device__ __forceinline__ HeaderReader(const uint32_t *rec, uint32_t MW)
    {
        next = rec + MW;
        win = *next++;
        have = 32;
    }
    __device__ __forceinline__ uint32_t take()
    {
        if (have < (uint32_t)kHdrBits) {
            win |= (uint64_t)*next++ << have;
            have += 32;
        }
        const uint32_t h = (uint32_t)win & 0x3FFFFu;
        win >>= kHdrBits;
        have -= kHdrBits;
        return h;
    }
};

__device__ __forceinline__ uint32_t clamp_biased_u8(uint32_t x)
{
    // each biased half into [2^14, 2^14 + 255]: its low byte is then the value
    uint32_t r;
    asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(0x40004000u));
    asm("min.u16x2 %0, %0, %1;" : "+r"(r) : "r"(0x40FF40FFu));
    return r;
}

// Inverse YCoCg-R (Section 4) of two pixels held as biased halves; returns
// R, G and B clamped to 8 bits in the low byte of each half.
__device__ __forceinline__ void ycocg_pair_to_rgb(uint32_t y, uint32_t co, uint32_t cg, uint32_t &r, uint32_t &g,
                                                  uint32_t &b)
{
    // (v + 2^14) >> 1 = floor(v / 2) + 2^13 in each half
    const uint32_t hcg = (cg >> 1) & 0x7FFF7FFFu, hco = (co >> 1) & 0x7FFF7FFFu;
    const uint32_t t = y - hcg + kHalfB2;   // y - floor(cg / 2)
    g = clamp_biased_u8(cg + t - kB2);
    const uint32_t bb = t - hco + kHalfB2;  // t - floor(co / 2)
    r = clamp_biased_u8(bb + co - kB2);
    b = clamp_biased_u8(bb);
}

// One block row (four pixels) from its biased Y, Co, Cg pairs: 12 RGB bytes
// in w[0..2] (R0 G0 B0 R1 | G1 B1 R2 G2 | B2 R3 G3 B3) or four packed words.
template <bool kPacked>
__device__ __forceinline__ void row_to_rgb(const uint2 y, const uint2 co, const uint2 cg, uint32_t w[4])
{
    uint32_t r01, g01, b01, r23, g23, b23;
    ycocg_pair_to_rgb(y.x, co.x, cg.x, r01, g01, b01);
    ycocg_pair_to_rgb(y.y, co.y, cg.y, r23, g23, b23);
    const uint32_t t01 = __byte_perm(r01, g01, 0x6240);   // R0 G0 R1 G1
    const uint32_t t23 = __byte_perm(r23, g23, 0x6240);   // R2 G2 R3 G3
    if (kPacked) {
        w[0] = __byte_perm(t01, b01, 0x0410) & 0xFFFFFFu;
        w[1] = __byte_perm(t01, b01, 0x0632) & 0xFFFFFFu;
        w[2] = __byte_perm(t23, b23, 0x0410) & 0xFFFFFFu;
        w[3] = __byte_perm(t23, b23, 0x0632) & 0xFFFFFFu;
    } else {
        w[0] = __byte_perm(t01, b01, 0x2410);
        w[1] = __byte_perm(__byte_perm(t01, b01, 0x0063), t23, 0x5410);
        w[2] = __byte_perm(b23, t23, 0x2760);
        w[3] = 0;
    }
}

// Bytes [0, len) of a strip row (`src`, word-aligned shared memory with a
// chunk of readable padding on each side) to `row`, whatever its alignment:
// the caller's lanes take its 16-byte aligned chunks ch = 0, 1, ... (len + 30) / 16 - 1,
// which begins at source byte 16 ch - (row & 15); five words funnel-shifted to
// four make it, and only the first and last chunk of the row, shared with the
// neighbouring strips, go out in smaller pieces.
//
// What bounds it: instruction issue (about 25 instructions for up to 512
// bytes; the edges another 30).  The 15 x 15 x 625 x 434 decode (31 MB stream)
// takes 0.246 ms with it; with single bytes or 4-byte words, each placed by
// divisions by the row length, it took 0.706 ms; with the edges as single
// bytes, 0.255.
__device__ __forceinline__ void store_row_unaligned(uint8_t *row, const uint32_t *src, uint32_t len, uint32_t ch)
{
    const int b0 = (int)(16u * ch) - (int)((uintptr_t)row & 15u);
    const int lo = max(0, -b0), hi = min(16, (int)len - b0);   // this chunk's bytes
    if (hi <= lo)
        return;
    const uint32_t *w = src + (b0 >> 2);
    const uint32_t sh = 8u * ((uint32_t)b0 & 3u);
    const uint32_t x0 = w[0], x1 = w[1], x2 = w[2], x3 = w[3], x4 = w[4];
    const uint32_t y0 = __funnelshift_r(x0, x1, sh), y1 = __funnelshift_r(x1, x2, sh);
    const uint32_t y2 = __funnelshift_r(x2, x3, sh), y3 = __funnelshift_r(x3, x4, sh);
    uint8_t *p = row + b0;
    if (hi - lo == 16) {
        *reinterpret_cast<uint4 *>(p) = make_uint4(y0, y1, y2, y3);
        return;
    }
    uint32_t *p4 = reinterpret_cast<uint32_t *>(p);
    if (lo <= 0 && hi >= 4)
        p4[0] = y0;
    if (lo <= 4 && hi >= 8)
        p4[1] = y1;
    if (lo <= 8 && hi >= 12)
        p4[2] = y2;
    if (lo <= 12 && hi >= 16)
        p4[3] = y3;
    // the boundary words: up to 3 bytes in front of a word boundary, up to 3
    // behind one, in pieces of their own alignment; bytes [lo, hi) of one word
    // where the row is that short
    if ((lo >> 2) == (hi >> 2)) {
        const uint8_t *sb = reinterpret_cast<const uint8_t *>(src) + b0;
        for (int j = lo; j < hi; j++)
            p[j] = sb[j];
        return;
    }
    if (lo & 3) {
        const uint32_t a = lo < 8 ? (lo < 4 ? y0 : y1) : (lo < 12 ? y2 : y3);
        if (lo & 1)
            p[lo] = (uint8_t)(a >> (8 * (lo & 3)));
        if ((lo & 3) != 3)
            *reinterpret_cast<uint16_t *>(p + (lo & ~3) + 2) = (uint16_t)(a >> 16);
    }
    if (hi & 3) {
        const uint32_t a = hi < 8 ? (hi < 4 ? y0 : y1) : (hi < 12 ? y2 : y3);
        const int w = hi & ~3;
        if (hi & 2)
            *reinterpret_cast<uint16_t *>(p + w) = (uint16_t)a;
        if (hi & 1)
            p[hi - 1] = (uint8_t)(a >> (8 * ((hi - 1) & 3)));
    }
}

}  // namespace rlfc
