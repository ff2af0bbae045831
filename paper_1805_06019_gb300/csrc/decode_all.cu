// Full light-field decode: Algorithm 2 for every (view, block location).
//
// One CTA owns a strip of kNL consecutive block locations of one block row.
// Its 3 * kNL records (location-major, then Y / Co / Cg) are contiguous in the
// stream; they are copied into shared memory when they fit the CTA's staging
// budget and read from the stream otherwise.  Phases:
//  1. parse (a warp per record): each record's presence mask, the
//     stored-block count in front of each mask word, and the payload bit
//     offset of every stored block (closed-form lengths of the 18-bit
//     headers, warp scan), in one compact table for the strip;
//  2. internal nodes (levels >= 1, first in BFS order), level by level from
//     the top, a thread per (location, node, channel): the reconstruction is
//     the parent reconstruction (or top RKV) plus the decoded residual where
//     a block is stored; then a thread per (location, parent, block row)
//     converts the view parents' rows to RGB.  Barriers separate these steps.
//     The last warp also prefetches into L2 the records and top-RKV blocks
//     of the strip a CTA of the next wave will take; then
//  3. the views, one unit of kUnit (8) BFS positions at a time per warp
//     (each warp takes the next unit from a shared counter and never waits
//     for the others).  The unit's output rows (8 views x 4 block rows x
//     the strip's 96 bytes) are assembled in the warp's shared-memory
//     buffer and written once:
//     a. the buffer starts as every view's parent rows (RGB), the exact
//        result for every block without a stored residual (most of them);
//     b. the unit's items (a view's block with at least one stored channel)
//        and slots (a stored channel block): lane = (view, quarter of the
//        strip) reads the three channel masks of its two locations, and one
//        warp scan of the per-lane counts places every item and slot; lanes
//        whose slots do not fit the warp's kWSlots decode slots go in a
//        further run.  Every slot is decoded by one lane (a mode-generic
//        BISE decoder that builds two values per multiply-add, see
//        decode_block_pairs); then four lanes per item, one block row each,
//        add the residual rows to the parent rows, apply the inverse
//        YCoCg-R two pixels per instruction and overwrite the item's bytes
//        in the buffer;
//     c. the buffer is written as whole 16-byte chunks, consecutive lanes
//        on consecutive chunks of one view row (one large L2 write per view
//        row instead of one per block row).  Rows that do not start on a
//        16-byte boundary go out as the destination's aligned chunks, shifted
//        into place (store_row_unaligned).
// Reconstructions are 16-bit values plus a bias of 2^14, two to a word (the
// loader refuses streams whose values could leave that range).  Every stored
// block of the strip is decoded once.
//
// A second instantiation writes one packed RGB word per pixel (r | g << 8 |
// b << 16) and decodes only the views a per-view mask asks for, into the
// output slots a table gives; the renderer uses it to decode, from the
// compressed stream, just the views a batch of new cameras samples.
#include <cuda_runtime.h>

#include <algorithm>

#include "pair_decode.cuh"
#include "warp_decode.cuh"

namespace rlfc {
namespace {

constexpr int kNL = (int)kDecodeStrip;          // block locations per CTA
constexpr int kRecs = 3 * kNL;
constexpr int kWarps = 12;                       // warps per CTA at most
constexpr int kThreads = 32 * kWarps;
constexpr int kUnit = 8;                         // BFS positions per unit of view work (a quarter mask word)
constexpr int kWSlots = 32;                      // decode slots per warp
constexpr int kZeroSlot = kWSlots;               // a slot of zero residuals, for channels without a stored block
constexpr int kWItems = kNL * kUnit;             // items per warp at most (every block of a unit)
constexpr uint32_t kSmemBudget = 200 * 1024 + 16 * 2 * kWarps + 4 * kWItems * kWarps;   // larger trees are refused
constexpr size_t kSmSmem = 228 * 1024;           // shared memory of an SM, and what a CTA takes of it besides its dynamic part
constexpr size_t kCtaOwn = 1024 + 1536;
constexpr uint32_t kNodeSmemMax = 4096;          // node tables up to this size are cached per CTA

static_assert(kNL == 8, "the location and group splits below assume eight locations per strip");
static_assert(3 * kNL <= 32 && (kNL & (kNL - 1)) == 0, "the strip's records fit one warp's lanes; locations are a power of two");
static_assert(kUnit == 8, "a unit is a quarter of a 32-bit mask word");
static_assert(kNL == 8 && kUnit * 4 == 32, "the list builder's lanes are (view of the unit, quarter of the strip)");
static_assert(kWSlots >= 6, "one lane's slots (two locations, three channels) must fit a run");

// Shared-memory layout of a CTA: 32-bit word offsets, computed once on the host.
struct Layout {
    uint32_t slots;   // [warp][kWSlots + 1][8]  decoded blocks, biased pairs; slot kZeroSlot is zero
    uint32_t top;     // [n_top][kNL][24]  biased pairs
    uint32_t inter;   // [n_int][kNL][24]  internal reconstructions, biased pairs
    uint32_t mask;    // [kRecs][MW]
    uint32_t mpre;    // [kRecs][MW]  stored blocks in front of each mask word
    uint32_t need;    // [MW]  views to decode (bit per BFS position)
    uint32_t node;    // [S]  node table (when cached)
    uint32_t sent;    // [warp][kWSlots]  record | rank << 8
    uint32_t items;   // [warp][kWItems] uint2: parent's block and the item's place in the buffer; its channels' slots
    uint32_t obuf;    // [warp][kUnit][4][kNL * 4 * bytes per pixel]  the unit's output rows
    uint32_t prgb;    // [n_par][4][kNL][row_words]  parent rows converted to RGB
    uint32_t off;     // [pmax]  payload bit offset of each stored block (OffT), record after record
    uint32_t stage;   // [stage_words]  the strip's records, from a 16-byte boundary
};

struct Args {
    const uint32_t *records;
    const uint32_t *offsets;
    const int16_t *top;
    const uint32_t *node_info;
    uint8_t *out;            // RGB bytes, or packed RGB words (packed instantiation)
    const uint8_t *needed;   // packed instantiation: per-view mask (nonzero = decode), may be null
    const uint32_t *slot_of; // packed instantiation with a mask: output slot of each needed view
    uint32_t S, n_int, n_top, L, q, MW;
    uint32_t par_base;       // BFS position (or top index) of the first parent of a view
    uint32_t n_par;          // parents of views
    uint32_t nlx, nloc, W, H;
    uint32_t pitch;          // pixels from one output row to the next: W, or the packed views' padded row (packed_pitch)
    uint32_t vec16;          // every view row of a strip starts on a 16-byte boundary (16-byte aligned output; RGB: W % 16 == 0; packed: always)
    uint32_t pmax;           // largest number of stored blocks in the records of one strip
    uint32_t n_units;        // ceil(S / kUnit)
    uint32_t node_smem;      // the node table is cached in shared memory
    uint32_t stage_words;    // shared-memory words for the strip's records (0: read them from the stream)
    uint32_t lvl_begin[kMaxLevels];  // first BFS position of each internal level, top level first; [L-2] = n_int
    uint32_t *dbg;           // debug builds: the stream's flag word
    uint32_t n_out;          // output views (or slots of the packed instantiation)
    Layout at;               // where the shared-memory arrays start
    uint32_t warps;          // warps per CTA
    uint32_t ahead;          // CTAs resident at once: the strip this many ahead is prefetched into L2
};

template <bool kPacked>
__host__ __device__ constexpr uint32_t row_words() { return kPacked ? 4u : 3u; }
// one warp's output buffer, in 16-byte chunks: kUnit views x 4 rows x kNL
// locations x row_words, between one chunk of padding on each side (the
// unaligned row writer reads up to 16 bytes around a row)
template <bool kPacked>
__host__ __device__ constexpr uint32_t obuf_words() { return kUnit * 4 * kNL * row_words<kPacked>() / 4 + 2; }

extern __shared__ __align__(16) uint32_t g_smem[];

// Fills the layout; returns its size in bytes.
template <bool kPacked>
size_t layout(Args &a, size_t off_size)
{
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t p = at;
        at += (bytes + 15) & ~size_t(15);
        return (uint32_t)(p / 4);
    };
    a.at.slots = take(32ull * (kWSlots + 1) * a.warps);
    a.at.top = take(96ull * a.n_top * kNL);
    a.at.inter = take(96ull * a.n_int * kNL);
    a.at.mask = take(4ull * kRecs * a.MW);
    a.at.mpre = take(4ull * kRecs * a.MW);
    a.at.need = take(4ull * a.MW);
    a.at.node = take(a.node_smem ? 4ull * a.S : 0);
    a.at.sent = take(4ull * kWSlots * a.warps);
    a.at.items = take(8ull * kWItems * a.warps);
    a.at.obuf = take(16ull * obuf_words<kPacked>() * a.warps);
    a.at.prgb = take(16ull * row_words<kPacked>() * a.n_par * kNL);
    a.at.off = take(off_size * a.pmax);
    a.at.stage = take(4ull * a.stage_words);
    return at;
}

template <bool kPacked, typename OffT>
__global__ void __launch_bounds__(kThreads, 2) decode_all_kernel(const Args a)
{
    __shared__ uint32_t s_mode[32];
    __shared__ uint16_t s_dig[256 + 128];
    __shared__ uint32_t s_roff[kRecs];
    __shared__ uint32_t s_np[kRecs];      // stored blocks of each record of the strip
    __shared__ uint32_t s_obase[kRecs];   // where each record's payload offsets start in m_off
#ifdef RLFC_DEBUG
    __shared__ uint32_t s_rbits[kRecs];   // length of each record in bits
#endif
    __shared__ uint32_t s_unit;   // next unit of view work
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t threads = blockDim.x, warps = a.warps;
    const uint32_t bx0 = blockIdx.x * kNL, by = blockIdx.y;
    const uint32_t nl = min((uint32_t)kNL, a.nlx - bx0);
    const uint32_t b0 = by * a.nlx + bx0;
    struct {
        uint32_t *slots, *top, *inter, *mask, *mpre, *need, *node, *sent, *obuf, *prgb, *stage;
        uint2 *items;
    } m;
    m.slots = g_smem + a.at.slots;
    m.top = g_smem + a.at.top;
    m.inter = g_smem + a.at.inter;
    m.mask = g_smem + a.at.mask;
    m.mpre = g_smem + a.at.mpre;
    m.need = g_smem + a.at.need;
    m.node = g_smem + a.at.node;
    m.sent = g_smem + a.at.sent;
    m.items = reinterpret_cast<uint2 *>(g_smem + a.at.items);
    m.obuf = g_smem + a.at.obuf;
    m.prgb = g_smem + a.at.prgb;
    m.stage = g_smem + a.at.stage;
    OffT *m_off = reinterpret_cast<OffT *>(g_smem + a.at.off);
    constexpr uint32_t RW = row_words<kPacked>();
    const uint32_t *nodes = a.node_smem ? m.node : a.node_info;

    // ---- set-up: tables, the strip's records and top-RKV blocks, zero reconstructions
    if (tid < 32)
        s_mode[tid] = g_tables.mode[tid];
    for (uint32_t i = tid; i < (256 + 128) / 2; i += threads)
        reinterpret_cast<uint32_t *>(s_dig)[i] = reinterpret_cast<const uint32_t *>(g_tables.dig)[i];
    if (tid == 0)
        s_unit = 0;
    // the strip's records are contiguous in the stream: stage them (from a
    // 16-byte boundary, plus the eight words the decoder may read past a
    // payload; the stream ends in zero padding) when they fit
    const uint32_t w_lo = __ldg(a.offsets + 3 * b0) & ~3u;
    const uint32_t n4 = (__ldg(a.offsets + 3 * (b0 + nl)) + 8 - w_lo + 3) / 4;
    const bool staged = 4 * n4 <= a.stage_words;
    if (staged) {
        const uint4 *src = reinterpret_cast<const uint4 *>(a.records + w_lo);
        uint4 *dst = reinterpret_cast<uint4 *>(m.stage);
        for (uint32_t i = tid; i < n4; i += threads)
            dst[i] = __ldg(src + i);
    }
    const uint32_t *rb = staged ? m.stage : a.records;   // records base: smem copy or stream
    if (tid < kRecs)
        s_roff[tid] = tid < 3 * (int)nl ? __ldg(a.offsets + 3 * b0 + tid) - (staged ? w_lo : 0u) : 0u;
    // the records of the strip a CTA of the next wave will take: the last
    // warp loads their range now and prefetches them into L2 once the parse
    // is done, so that CTA's staging reads hit L2 instead of DRAM
    uint32_t pf_lo = 0, pf_hi = 0, pf_top = 0xFFFFFFFFu, pf_nl = 0;   // pf_top, pf_nl: the strip's first location and count
    {
        const uint32_t strip2 = blockIdx.y * gridDim.x + blockIdx.x + a.ahead;
        if (warp == (int)warps - 1 && a.ahead && strip2 < gridDim.x * gridDim.y) {
            const uint32_t bx2 = (strip2 % gridDim.x) * kNL, b02 = (strip2 / gridDim.x) * a.nlx + bx2;
            const uint32_t nl2 = min((uint32_t)kNL, a.nlx - bx2);
            pf_lo = __ldg(a.offsets + 3 * b02) & ~31u;
            pf_hi = __ldg(a.offsets + 3 * (b02 + nl2));
            pf_top = b02;
            pf_nl = nl2;
        }
    }
#ifdef RLFC_DEBUG
    if (tid < kRecs)
        s_rbits[tid] = tid < 3 * (int)nl ? 32u * (__ldg(a.offsets + 3 * b0 + tid + 1) - __ldg(a.offsets + 3 * b0 + tid)) : 0u;
#endif
    {
        const uint32_t *tg = reinterpret_cast<const uint32_t *>(a.top);
        for (uint32_t i = tid; i < a.n_top * kNL * 24; i += threads) {
            const uint32_t t = i / (kNL * 24), rest = i - t * (kNL * 24), loc = rest / 24, wi = rest - loc * 24;
            m.top[i] = loc < nl ? (__ldg(tg + ((size_t)t * a.nloc + b0 + loc) * 24 + wi) ^ 0x80008000u) - kB2 : kB2;
        }
    }
    uint32_t *wslots = m.slots + warp * (8 * (kWSlots + 1));   // this warp's slots
    uint32_t *wsent = m.sent + warp * kWSlots;
    uint2 *witems = m.items + warp * kWItems;
    if (lane < 8)
        wslots[kZeroSlot * 8 + lane] = kB2;   // the warp's zero slot
    if (a.node_smem)
        for (uint32_t i = tid; i < a.S; i += threads)
            m.node[i] = __ldg(a.node_info + i);
    __syncthreads();
    // the views to decode, one bit per BFS position (internal positions 0)
    for (uint32_t w0 = warp * 32; w0 < a.MW * 32; w0 += warps * 32) {
        const uint32_t p = w0 + lane;
        bool need = p >= a.n_int && p < a.S;
        if (need && kPacked && a.needed)
            need = __ldg(a.needed + node_view(nodes[p])) != 0;
        const unsigned bal = __ballot_sync(kFullMask, need);
        if (lane == 0)
            m.need[w0 >> 5] = bal;
    }

    // ---- phases 1 and 2, spread over all warps: parse the strip's records
    // (a warp per record), reconstruct the internal nodes level by level (a
    // thread per (location, node, channel)), convert the view parents' rows
    // to RGB (a thread per (location, parent, block row))
    const uint32_t hdr0 = 32 * a.MW;
    // 1a. per record: mask words and the stored blocks in front of each
    // (nothing stored past the end of the row), and where the records' payload
    // offsets start in m_off, record after record.  Masks of up to four words:
    // one warp, a lane per record (a warp per record spends most of its lanes
    // on nothing: 9 x 9 x 512^2, three words, 75 against 79 us); longer ones:
    // a warp per record (eight words: 161 against 168 us).
    const bool short_masks = a.MW <= 4;
    uint32_t np_l = 0;
    if (short_masks && warp == 0 && lane < kRecs) {
        const bool live = (uint32_t)lane < 3 * nl;
        const uint32_t *rec = rb + s_roff[lane];
        for (uint32_t i = 0; i < a.MW; i++) {
            const uint32_t word = live ? rec[i] : 0u;
            m.mask[lane * a.MW + i] = word;
            m.mpre[lane * a.MW + i] = np_l;
            np_l += (uint32_t)__popc(word);
        }
        s_np[lane] = np_l;
    }
    if (!short_masks) {
        for (uint32_t r = warp; r < (uint32_t)kRecs; r += warps) {
            const bool live = r < 3 * nl;
            uint32_t *mk = m.mask + r * a.MW;
            uint32_t *mp = m.mpre + r * a.MW;
            const uint32_t *rec = rb + s_roff[r];
            uint32_t P = 0;
            for (uint32_t w0 = 0; w0 < a.MW; w0 += 32) {
                const uint32_t word = (live && w0 + lane < a.MW) ? rec[w0 + lane] : 0u;
                const uint32_t cnt = (uint32_t)__popc(word);
                const uint32_t incl = warp_inclusive_scan(cnt, lane);
                if (w0 + lane < a.MW) {
                    mk[w0 + lane] = word;
                    mp[w0 + lane] = P + incl - cnt;
                }
                P += __shfl_sync(kFullMask, incl, 31);
            }
            if (lane == 0)
                s_np[r] = P;
        }
        __syncthreads();
        np_l = lane < kRecs ? s_np[lane] : 0u;
    }
    if (warp == 0) {
        const uint32_t base = warp_inclusive_scan(np_l, lane) - np_l;
        if (lane < kRecs)
            s_obase[lane] = base;
    }
    __syncthreads();
    // 1b. per record: payload offset of every stored block (closed-form
    // lengths of the 18-bit headers, warp scan)
    for (uint32_t r = warp; r < 3 * nl; r += warps) {
        const uint32_t *rec = rb + s_roff[r];
        const uint32_t P = s_np[r];
        OffT *o = m_off + s_obase[r];
        uint32_t run = hdr0 + kHdrBits * P;
        for (uint32_t h0 = 0; h0 < P; h0 += 32) {
            const uint32_t h = h0 + lane;
            uint32_t len = 0;
            if (h < P) {
                const uint32_t bp = hdr0 + kHdrBits * h;
                len = mode_bits(s_mode[__funnelshift_r(rec[bp >> 5], rec[(bp >> 5) + 1], bp) & 31u]);
            }
            const uint32_t incl = warp_inclusive_scan(len, lane);
            if (h < P)
                o[h] = (OffT)(run + incl - len);
            run += __shfl_sync(kFullMask, incl, 31);
        }
    }
    __syncthreads();
    // 2. internal nodes, level by level from the top: reconstruction =
    // parent reconstruction (top RKV or a node of the level above) + the
    // decoded residual where a block is stored
    for (uint32_t lv = 0; lv + 2 < a.L; lv++) {
        const uint32_t g0 = a.lvl_begin[lv], g1 = a.lvl_begin[lv + 1];
        const uint32_t *src = lv == 0 ? m.top : m.inter;
        for (uint32_t t = tid; t < (g1 - g0) * 3 * kNL; t += threads) {
            const uint32_t l = t & (kNL - 1), q = t / kNL;
            if (l >= nl)
                continue;
            const uint32_t p = g0 + q / 3, c = q - 3 * (q / 3), r = 3 * l + c;
            const uint32_t word = m.mask[r * a.MW + (p >> 5)];
            uint32_t v[8];
            if ((word >> (p & 31u)) & 1u) {
                const uint32_t rank = m.mpre[r * a.MW + (p >> 5)] + __popc(word & ((1u << (p & 31u)) - 1u));
                const uint32_t *rec = rb + s_roff[r];
                const uint32_t bp = hdr0 + kHdrBits * rank;
                const uint32_t hdr = __funnelshift_r(rec[bp >> 5], rec[(bp >> 5) + 1], bp) & 0x3FFFFu;
                const uint32_t pos = m_off[s_obase[r] + rank];
#ifdef RLFC_DEBUG
                if (RLFC_DBG_BLOCK_OK(a.dbg, hdr & 31u, bp + kHdrBits, hdr0 + kHdrBits * s_np[r], pos,
                                      (hdr & 31u) < (uint32_t)kNumModes ? mode_bits(s_mode[hdr & 31u]) : 0u,
                                      s_rbits[r]))
                    decode_block_pairs(rec, pos, hdr, a.q, s_mode, s_dig, v);
                else
                    for (int j = 0; j < 8; j++)
                        v[j] = kB2;
#else
                decode_block_pairs(rec, pos, hdr, a.q, s_mode, s_dig, v);
#endif
            } else {
#pragma unroll
                for (int j = 0; j < 8; j++)
                    v[j] = kB2;
            }
            const uint4 *ps = reinterpret_cast<const uint4 *>(src + (node_parent(nodes[p]) * kNL + l) * 24 + c * 8);
            uint4 *pd = reinterpret_cast<uint4 *>(m.inter + (p * kNL + l) * 24 + c * 8);
            const uint4 s0 = ps[0], s1 = ps[1];
            pd[0] = make_uint4(s0.x + v[0] - kB2, s0.y + v[1] - kB2, s0.z + v[2] - kB2, s0.w + v[3] - kB2);
            pd[1] = make_uint4(s1.x + v[4] - kB2, s1.y + v[5] - kB2, s1.z + v[6] - kB2, s1.w + v[7] - kB2);
        }
        __syncthreads();
    }
    // 3. the block rows of every parent of a view, as RGB
    {
        const uint32_t *src = a.L == 2 ? m.top : m.inter;
        for (uint32_t t = tid; t < a.n_par * 4 * kNL; t += threads) {
            const uint32_t l = t & (kNL - 1), q = t / kNL, n = q >> 2, rr = q & 3u;
            if (l >= nl)
                continue;
            const uint32_t *sl = src + ((a.par_base + n) * kNL + l) * 24 + rr * 2;
            uint32_t w[4];
            row_to_rgb<kPacked>(*reinterpret_cast<const uint2 *>(sl), *reinterpret_cast<const uint2 *>(sl + 8),
                                *reinterpret_cast<const uint2 *>(sl + 16), w);
            uint32_t *d = m.prgb + ((n * 4 + rr) * kNL + l) * RW;
#pragma unroll
            for (uint32_t k = 0; k < RW; k++)
                d[k] = w[k];
        }
    }
    __syncthreads();
    if (warp == (int)warps - 1) {
        for (uint32_t i = pf_lo + 32u * lane; i < pf_hi; i += 32u * 32u)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(__cvta_generic_to_global(a.records + i)));
        // the strip's top-RKV blocks: 96 bytes per location, per top RKV
        if (pf_top != 0xFFFFFFFFu && lane < (int)a.n_top * 6 && (lane % 6) * 64 < pf_nl * 48)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(__cvta_generic_to_global(
                a.top + ((size_t)(lane / 6) * a.nloc + pf_top) * 48 + (lane % 6) * 64)));
    }

    // ---- phase 3: the views, one unit of kUnit positions at a time per warp.
    // The unit's output rows (kUnit views x 4 rows x the strip's kNL
    // locations) are assembled in the warp's buffer, then written once, each
    // view row as whole 16-byte chunks by consecutive lanes: few, large L2
    // writes instead of one per block row.
    const uint32_t *par_slab = a.L == 2 ? m.top : m.inter;
    const uint32_t u_first = a.n_int / kUnit;
    const uint32_t nrows = min(4u, a.H - by * 4);
    constexpr uint32_t BPP = kPacked ? 4u : 3u;     // output bytes per pixel
    constexpr uint32_t CH = kNL * 4 * BPP / 16;     // 16-byte chunks per view row of the strip
    uint4 *wbuf = reinterpret_cast<uint4 *>(m.obuf) + warp * obuf_words<kPacked>() + 1;
    // a strip row written as whole chunks: 16-byte aligned rows with room for
    // the whole strip (a packed row is padded to whole strips)
    const bool whole = a.vec16 && bx0 * 4 + kNL * 4 <= a.pitch;
    // otherwise the strip row's bytes (the image may end inside the strip)
    const uint32_t piece = min(nl * 4u, a.W - bx0 * 4u) * BPP;
    // this lane's piece of a view's strip: its 16-byte chunk, or, for the
    // unaligned writer, its row
    const size_t view_bytes = (size_t)a.pitch * a.H * BPP;
    uint8_t *out_lane = a.out + ((size_t)(by * 4 + (whole ? (uint32_t)lane / CH : (uint32_t)lane >> 3)) * a.pitch + bx0 * 4) * BPP +
                        (whole ? 16u * ((uint32_t)lane % CH) : 0u);
    for (;;) {
        uint32_t u = 0;
        if (lane == 0)
            u = atomicAdd(&s_unit, 1u);
        u = __shfl_sync(kFullMask, u, 0) + u_first;
        if (u >= a.n_units)
            break;
        const uint32_t w = u >> 2, ub = kUnit * (u & 3u);   // the unit is bits [ub, ub + 8) of mask word w
        const uint32_t P0 = max(u * kUnit, a.n_int), P1 = min(u * kUnit + kUnit, a.S);
        const uint32_t lo = P0 - w * 32, hi = P1 - w * 32;
        const uint32_t sel = (hi >= 32 ? 0xFFFFFFFFu : ((1u << hi) - 1u)) & ~((1u << lo) - 1u) & m.need[w];
        // per view of the unit (lane v < kUnit): its parent's rows and blocks,
        // and its output rows
        uint32_t par_v = 0, ov_v = 0;
        bool bad = false;
        if ((uint32_t)lane < (uint32_t)kUnit && ((sel >> (ub + lane)) & 1u)) {
            const uint32_t info = nodes[w * 32 + ub + lane];
            par_v = node_parent(info);
            ov_v = a.slot_of ? __ldg(a.slot_of + node_view(info)) : node_view(info);
            bad = !RLFC_DBG_INDEX_OK(a.dbg, ov_v, a.n_out);
        }
        // the unit's views, and those of them that go out
        const uint32_t selv = (sel >> ub) & 0xFFu, goes = selv & ~__ballot_sync(kFullMask, bad);
        // (a) the buffer starts as every view's parent rows (RGB), the exact
        // result for every block without a stored residual; lane = (row,
        // chunk of the view row)
        const uint32_t f_rr = (uint32_t)lane / CH;
        const uint32_t fill = (uint32_t)lane < 4 * CH ? selv : 0u;
        const uint4 *prgb4 = reinterpret_cast<const uint4 *>(m.prgb) + lane;
#pragma unroll
        for (uint32_t vv = 0; vv < (uint32_t)kUnit; vv++) {
            const uint32_t pv = (__shfl_sync(kFullMask, par_v, vv) - a.par_base) * 4 * CH;
            if (fill & (1u << vv))
                wbuf[vv * 4 * CH + lane] = prgb4[pv];
        }
        // (b) items and slots.  Lane = (view ub + v, quarter qd of the strip):
        // the stored channels of its two locations 2qd, 2qd + 1
        const uint32_t v = (uint32_t)lane & 7u, qd = (uint32_t)lane >> 3, bit = ub + v;
        const uint32_t lt = (1u << bit) - 1u;   // positions in front of this view in mask word w
        const bool vsel = (selv >> v) & 1u;
        // this lane's first block of its view's parent, and its place in the buffer
        const uint32_t place = (__shfl_sync(kFullMask, par_v, v) * kNL + 2 * qd) * 24 | ((v * 4 * kNL + 2 * qd) * RW) << 16;
        uint32_t f[2][3];   // channel masks (word w) of the lane's locations
        uint32_t st = 0;    // stored channels of location 2qd + j at bits 3j .. 3j + 2
        uint32_t ni = 0, ns = 0;
#pragma unroll
        for (uint32_t j = 0; j < 2; j++) {
            const uint32_t l = 2u * qd + j;
#pragma unroll
            for (uint32_t c = 0; c < 3; c++)
                f[j][c] = m.mask[(3 * l + c) * a.MW + w];
            const uint32_t s3 = vsel ? (((f[j][0] >> bit) & 1u) | (((f[j][1] >> bit) & 1u) << 1) |
                                        (((f[j][2] >> bit) & 1u) << 2))
                                     : 0u;
            st |= s3 << (3 * j);
            ni += s3 != 0;
            ns += (uint32_t)__popc(s3);
        }
        const uint32_t cnt = ni | (ns << 16);
        const uint32_t incl = warp_inclusive_scan(cnt, lane);
        const uint32_t excl = incl - cnt;
        __syncwarp();
        // runs of lanes whose slots fit the warp's kWSlots (one lane has at most 6)
        for (uint32_t L0 = 0; L0 < 32;) {
            const uint32_t rb_i = __shfl_sync(kFullMask, excl & 0xFFFFu, L0);
            const uint32_t rb_s = __shfl_sync(kFullMask, excl >> 16, L0);
            const unsigned fit = __ballot_sync(kFullMask, (uint32_t)lane >= L0 && (incl >> 16) - rb_s <= (uint32_t)kWSlots);
            const uint32_t L1 = 32u - (uint32_t)__clz(fit);
            const uint32_t tot = __shfl_sync(kFullMask, incl, L1 - 1);
            const uint32_t n_items = (tot & 0xFFFFu) - rb_i, n_slots = (tot >> 16) - rb_s;
            if ((uint32_t)lane >= L0 && (uint32_t)lane < L1 && st) {
                uint32_t item = (excl & 0xFFFFu) - rb_i, slot = (excl >> 16) - rb_s;
#pragma unroll
                for (uint32_t j = 0; j < 2; j++) {
                    const uint32_t s3 = (st >> (3 * j)) & 7u, l = 2u * qd + j;
                    if (s3) {
                        // slots of the channels, times 32: the stored ones in
                        // order, the zero slot for the others
                        const uint32_t zy = (s3 & 1u) ? slot : (uint32_t)kZeroSlot;
                        const uint32_t zo = (s3 & 2u) ? slot + (s3 & 1u) : (uint32_t)kZeroSlot;
                        const uint32_t zg = (s3 & 4u) ? slot + __popc(s3 & 3u) : (uint32_t)kZeroSlot;
                        witems[item++] = make_uint2(place + j * (24u | RW << 16), zy << 5 | zo << 13 | zg << 21);
#pragma unroll
                        for (uint32_t c = 0; c < 3; c++)
                            if ((s3 >> c) & 1u) {
                                const uint32_t r = 3 * l + c;
                                wsent[slot++] = r | ((m.mpre[r * a.MW + w] + __popc(f[j][c] & lt)) << 8);
                            }
                    }
                }
            }
            __syncwarp();
            // decode every slot of the run, one lane each
            for (uint32_t t = lane; t < n_slots; t += 32) {
                const uint32_t e = wsent[t];
                const uint32_t r = e & 255u, rank = e >> 8;
                const uint32_t *rec = rb + s_roff[r];
                const uint32_t bp = hdr0 + kHdrBits * rank;
                const uint32_t hdr = __funnelshift_r(rec[bp >> 5], rec[(bp >> 5) + 1], bp) & 0x3FFFFu;
                uint32_t dv[8];
#ifdef RLFC_DEBUG
                const uint32_t pos = m_off[s_obase[r] + rank];
                if (RLFC_DBG_BLOCK_OK(a.dbg, hdr & 31u, bp + kHdrBits, hdr0 + kHdrBits * s_np[r], pos,
                                      (hdr & 31u) < (uint32_t)kNumModes ? mode_bits(s_mode[hdr & 31u]) : 0u,
                                      s_rbits[r]))
                    decode_block_pairs(rec, pos, hdr, a.q, s_mode, s_dig, dv);
                else
                    for (int j = 0; j < 8; j++)
                        dv[j] = kB2;
#else
                decode_block_pairs(rec, m_off[s_obase[r] + rank], hdr, a.q, s_mode, s_dig, dv);
#endif
                uint4 *d = reinterpret_cast<uint4 *>(wslots + t * 8);
                d[0] = make_uint4(dv[0], dv[1], dv[2], dv[3]);
                d[1] = make_uint4(dv[4], dv[5], dv[6], dv[7]);
            }
            __syncwarp();
            // items: parent + residual -> RGB into the buffer, four lanes per item, one block row each
            for (uint32_t t = lane; t < 4 * n_items; t += 32) {
                const uint2 it = witems[t >> 2];
                const uint32_t rr = t & 3u;
                const uint32_t *ps = par_slab + (it.x & 0xFFFFu) + 2 * rr;
                const unsigned char *rs = reinterpret_cast<const unsigned char *>(wslots) + 8 * rr;
                const unsigned char *ry = rs + (it.y & 0x1FE0u), *rco = rs + ((it.y >> 8) & 0x1FE0u), *rcg = rs + ((it.y >> 16) & 0x1FE0u);
                const uint2 py = *reinterpret_cast<const uint2 *>(ps);
                const uint2 pco = *reinterpret_cast<const uint2 *>(ps + 8);
                const uint2 pcg = *reinterpret_cast<const uint2 *>(ps + 16);
                const uint2 vy = *reinterpret_cast<const uint2 *>(ry);
                const uint2 vco = *reinterpret_cast<const uint2 *>(rco);
                const uint2 vcg = *reinterpret_cast<const uint2 *>(rcg);
                uint32_t wv[4];
                row_to_rgb<kPacked>(make_uint2(py.x + vy.x - kB2, py.y + vy.y - kB2),
                                    make_uint2(pco.x + vco.x - kB2, pco.y + vco.y - kB2),
                                    make_uint2(pcg.x + vcg.x - kB2, pcg.y + vcg.y - kB2), wv);
                uint32_t *d = reinterpret_cast<uint32_t *>(wbuf) + (it.x >> 16) + rr * (kNL * RW);
#pragma unroll
                for (uint32_t k = 0; k < RW; k++)
                    d[k] = wv[k];
            }
            __syncwarp();
            L0 = L1;
        }
        // (c) write the unit's rows: consecutive lanes, consecutive chunks of one view row
        if (whole) {
            const uint32_t put = f_rr < nrows && (uint32_t)lane < 4 * CH ? goes : 0u;
#pragma unroll
            for (uint32_t vv = 0; vv < (uint32_t)kUnit; vv++) {
                const uint32_t ov = __shfl_sync(kFullMask, ov_v, vv);
                if (put & (1u << vv))
                    *reinterpret_cast<uint4 *>(out_lane + ov * view_bytes) = wbuf[vv * 4 * CH + lane];
            }
        } else if (!kPacked) {
            // rows not 16-byte aligned, or the right edge of the image: lane =
            // (row, 16-byte chunk of the destination)
            const uint32_t rr = (uint32_t)lane >> 3, ch = (uint32_t)lane & 7u;
            const uint32_t put = rr < nrows ? goes : 0u;
#pragma unroll 2
            for (uint32_t vv = 0; vv < (uint32_t)kUnit; vv++) {
                const uint32_t ov = __shfl_sync(kFullMask, ov_v, vv);
                if (put & (1u << vv))
                    store_row_unaligned(out_lane + ov * view_bytes, reinterpret_cast<const uint32_t *>(wbuf + (vv * 4 + rr) * CH),
                                        piece, ch);
            }
        }
        __syncwarp();
    }
}

template <bool kPacked>
int launch_decode(const rlfc_stream *s, uint8_t *d_out, const uint8_t *needed, const uint32_t *slot_of, uint32_t n_out,
                  cudaStream_t st)
{
    const Tables &t = s->tab;
    Args a;
    a.records = s->d_records;
    a.offsets = s->d_offsets;
    a.top = s->d_top;
    a.node_info = s->d_node_info;
    a.out = d_out;
    a.needed = needed;
    a.slot_of = slot_of;
    a.S = t.S;
    a.n_int = t.n_int;
    a.n_top = t.n_top;
    a.L = t.L;
    a.q = s->info.q;
    a.MW = s->MW;
    a.nlx = s->info.nloc_x;
    a.nloc = s->info.nloc_x * s->info.nloc_y;
    a.W = s->info.W;
    a.H = s->info.H;
    // parents of views: the level-1 nodes (the last internal positions) or the tops
    if (t.L == 2) {
        a.par_base = 0;
        a.n_par = t.n_top;
    } else {
        uint32_t n1 = 0;
        for (uint32_t p = 0; p < t.n_int; p++)
            n1 += node_level(t.node_info[p]) == 1;
        a.par_base = t.n_int - n1;
        a.n_par = n1;
    }
    a.pitch = kPacked ? packed_pitch(a.W) : a.W;
    a.vec16 = ((uintptr_t)d_out & 15u) == 0 && (kPacked || (a.W & 15u) == 0);
    a.pmax = std::max<uint32_t>(s->max_strip_present, 1);
    a.n_units = (t.S + kUnit - 1) / kUnit;
    a.node_smem = t.S <= kNodeSmemMax;
    a.dbg = s->d_debug;
    a.n_out = n_out;
    a.ahead = 0;
    // internal levels in BFS order: L-2 first, down to 1
    for (uint32_t k = 0; k < (uint32_t)kMaxLevels; k++)
        a.lvl_begin[k] = t.n_int;
    for (uint32_t lv = 0; lv + 2 < t.L; lv++) {
        const uint32_t level = t.L - 2 - lv;
        uint32_t p = 0;
        while (p < t.n_int && node_level(t.node_info[p]) != level)
            p++;
        a.lvl_begin[lv] = p;
    }
    // payload offsets are bit positions inside one record: 16 bits suffice
    // unless a record reaches 2^16 bits
    const bool off16 = (uint64_t)s->max_record_words * 32 < 65536;
    const size_t off_size = off16 ? 2 : 4;
    // three CTAs of eight warps per SM where a strip's tables and the records
    // of most strips fit a third of its shared memory, else two of twelve:
    // set-up, parse and internal nodes wait on memory and barriers, and more
    // CTAs overlap them with the view work of the others.  Measured, three
    // against two: 9 x 9 x 512^2 (12 MB stream) 75 / 83 us, 32 of its views
    // packed 64 / 70, 5 x 5 x 64^2 16.8 / 17.4; 17 x 17 x 1024^2 (133 MB
    // stream), whose records then read from the stream, 706 / 693.  Strips
    // whose records do not fit what is left read them from the stream.
    const uint32_t strips = (a.nlx + kNL - 1) / kNL * s->info.nloc_y;
    const size_t longest = 4ull * ((s->max_strip_words + 8 + 3 + 3) & ~3u);
    const size_t most = std::min<size_t>(longest, 4ull * (s->record_words / strips) * 3 / 2 + 64);
    size_t base = 0, room = 0;
    for (uint32_t ctas = 3; ctas >= 2; ctas--) {
        a.warps = 24 / ctas;
        a.stage_words = 0;
        base = layout<kPacked>(a, off_size);
        const size_t have = kSmSmem / ctas - kCtaOwn;
        room = base < have ? (have - base) & ~size_t(15) : 0;
        if (room >= most)
            break;
    }
    a.stage_words = (uint32_t)(std::min(room, longest) / 4);
    const size_t smem = layout<kPacked>(a, off_size);
    if (smem > kSmemBudget || a.S >= 16384) {
        set_error("tree too large for the decode-all kernel's shared memory");
        return RLFC_E_UNSUPPORTED;
    }
    auto kern = off16 ? decode_all_kernel<kPacked, uint16_t> : decode_all_kernel<kPacked, uint32_t>;
    // (the same limit for every call: the attribute belongs to the kernel, and
    // a smaller one set for another thread's light field would refuse this launch)
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget);
    if (e != cudaSuccess)
        return cuda_fail(e, "decode_all: shared memory attribute");
    dim3 grid((a.nlx + kNL - 1) / kNL, s->info.nloc_y);
    {
        int sms = 0, per_sm = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, s->device) == cudaSuccess &&
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, (int)(32 * a.warps), smem) == cudaSuccess)
            a.ahead = (uint32_t)(std::max(sms, 0) * std::max(per_sm, 0));
    }
    { rlfc::TraceScope trace_((kPacked ? "decode_all_kernel<packed>" : "decode_all_kernel"), st); kern<<<grid, 32 * a.warps, smem, st>>>(a); }
    e = cudaGetLastError();
    if (e != cudaSuccess)
        return cuda_fail(e, "decode_all launch");
    return RLFC_OK;
}

}  // namespace

int launch_decode_all(const rlfc_stream *s, uint8_t *d_out, cudaStream_t st)
{
    return launch_decode<false>(s, d_out, nullptr, nullptr, s->tab.n_views, st);
}

int launch_decode_packed(const rlfc_stream *s, uint32_t *d_out, const uint8_t *needed, const uint32_t *slot_of,
                         uint32_t n_slots, cudaStream_t st)
{
    return launch_decode<true>(s, reinterpret_cast<uint8_t *>(d_out), needed, slot_of, n_slots, st);
}

}  // namespace rlfc
