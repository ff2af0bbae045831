// Batched random-access block decode: Algorithm 2's DecompressLFIBlock for
// many (view, location) requests in one call, with the progressive stop level
// of Section 3.6.
//
// The requests are grouped by block location with a counting sort (count,
// scan, scatter), then a persistent kernel serves the locations.  Its warps
// take locations from an atomic work queue (no waits: a warp that finds the
// queue empty exits).  For each location a warp
//   1. optionally copies the location's three channel records (they are
//      contiguous in the stream) into its shared-memory slice, or has them
//      copied there ahead of time (cp.async) while it serves the previous
//      location;
//   2. parses the three records once, side by side: presence-mask popcount
//      prefixes, then the closed-form payload length of every stored block
//      from its 5-bit mode, turned into payload bit offsets by a warp scan;
//   3. for up to sixteen requests at a time: seeds accumulators (biased 16-bit
//      pairs, pair_decode.cuh) with the top-RKV block, lists the stored
//      ancestor blocks (request, channel, level) with a ballot compaction,
//      decodes them one thread per block with the pair decoder and adds them
//      into the accumulators (a packed add is exact modulo 2^32, so the order
//      does not matter), then a thread per block row converts to RGB and the
//      48 bytes of a request go out as three 16-byte stores.
// The record gather (mask, headers, offsets) is paid once per location and
// shared by every request there, which is the point of batching.
//
// What bounds it: the chain of dependent loads per location and instruction
// issue (57 % of the slots, 27 of 32 lanes active); 10^6 requests on the 17 x
// 17 x 1024^2 light field take 0.198 ms (133 MB stream) or 0.183 (99 MB, L2
// flushed; timed one by one 0.155 here, 0.045 the binning).  With 32-bit
// accumulators, an atomic per value, the sequential bit reader, eight requests
// a round and one record parsed after the other: 0.338 ms (133 MB).
#include <cuda_runtime.h>

#include <cuda_pipeline.h>

#include <algorithm>
#include <new>

#include "pair_decode.cuh"
#include "rlfc_internal.h"

namespace rlfc {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr uint32_t kSlots = 16, kSlotsTight = 12;   // requests of one location per round; fewer where shared memory is short
constexpr uint32_t kStaticLimit = 112;  // static shared memory that the limits of create and set_config count
constexpr uint32_t kStageCap = 1024;    // words of records staged per warp at most
constexpr uint32_t kBadRank = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t scan_incl(uint32_t x, int lane)
{
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, x, d);
        if (lane >= d)
            x += y;
    }
    return x;
}

struct BinArgs {
    const uint32_t *view;
    const uint32_t *loc;
    uint8_t *out;
    uint8_t *status;
    uint32_t *cnt;      // [nloc + 2]: counts, then bin starts; [nloc + 1] is the queue head,
                        // followed by the scan's per-chunk counts
    uint32_t *rank;     // [n]: position of the request inside its bin
    uint2 *sorted;      // [n]: requests grouped by location: index, view
    uint32_t n, n_views, nloc, aligned;
};

// Validate, count per location, remember the position inside the bin.
__global__ void bin_count_kernel(const BinArgs a)
{
    const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= a.n)
        return;
    const uint32_t view = a.view[r], loc = a.loc[r];
    const uint32_t bad = view >= a.n_views ? (uint32_t)RLFC_REQ_BAD_VIEW
                                           : (loc >= a.nloc ? (uint32_t)RLFC_REQ_BAD_LOCATION : 0u);
    if (a.status)
        a.status[r] = (uint8_t)bad;
    if (bad) {
        uint8_t *dst = a.out + (size_t)r * 48;
        if (a.aligned) {
            for (int w = 0; w < 12; w++)
                reinterpret_cast<uint32_t *>(dst)[w] = 0u;
        } else {
            for (int b = 0; b < 48; b++)
                dst[b] = 0;
        }
        a.rank[r] = kBadRank;
        return;
    }
    a.rank[r] = atomicAdd(&a.cnt[loc], 1u);
}

constexpr uint32_t kScanChunk = 4096;   // locations per CTA of the scan (1024 threads x 4)

__device__ __forceinline__ uint32_t block_sum(uint32_t x, uint32_t *s_warp)
{
    const int lane = (int)(threadIdx.x & 31u);
    x = __reduce_add_sync(kFull, x);
    if (lane == 0)
        s_warp[threadIdx.x >> 5] = x;
    __syncthreads();
    const uint32_t r = __reduce_add_sync(kFull, lane < (int)(blockDim.x >> 5) ? s_warp[lane] : 0u);
    __syncthreads();
    return r;
}

// Scan, pass 1: the request count of every chunk of kScanChunk locations.
__global__ void __launch_bounds__(1024) bin_reduce_kernel(const uint32_t *cnt, uint32_t nloc, uint32_t *part)
{
    __shared__ uint32_t s_warp[32];
    const uint32_t base = blockIdx.x * kScanChunk;
    uint32_t x = 0;
#pragma unroll
    for (uint32_t k = 0; k < 4; k++) {
        const uint32_t i = base + k * 1024 + threadIdx.x;
        x += i < nloc ? cnt[i] : 0u;
    }
    x = block_sum(x, s_warp);
    if (threadIdx.x == 0)
        part[blockIdx.x] = x;
}

// Scan, pass 2: exclusive scan of cnt[0..nloc) in place, chunk by chunk in
// parallel (each chunk starts at the sum of the chunks before it);
// cnt[nloc] = total.
__global__ void __launch_bounds__(1024) bin_scan_kernel(uint32_t *cnt, uint32_t nloc, const uint32_t *part)
{
    __shared__ uint32_t s_warp[32];
    const int lane = (int)(threadIdx.x & 31u);
    const uint32_t warp = threadIdx.x >> 5;
    uint32_t before = 0;
    for (uint32_t c = threadIdx.x; c < blockIdx.x; c += 1024)
        before += part[c];
    before = block_sum(before, s_warp);
    // four consecutive locations per thread
    const uint32_t i0 = blockIdx.x * kScanChunk + 4 * threadIdx.x;
    uint32_t v[4];
#pragma unroll
    for (uint32_t k = 0; k < 4; k++)
        v[k] = i0 + k < nloc ? cnt[i0 + k] : 0u;
    const uint32_t sum = v[0] + v[1] + v[2] + v[3];
    const uint32_t incl = scan_incl(sum, lane);
    if (lane == 31)
        s_warp[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const uint32_t x = s_warp[lane];
        s_warp[lane] = scan_incl(x, lane) - x;
    }
    __syncthreads();
    uint32_t run = before + s_warp[warp] + incl - sum;
#pragma unroll
    for (uint32_t k = 0; k < 4; k++) {
        if (i0 + k < nloc)
            cnt[i0 + k] = run;
        run += v[k];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 1023)
        cnt[nloc] = run;
}

__global__ void bin_scatter_kernel(const BinArgs a)
{
    const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= a.n)
        return;
    const uint32_t rk = a.rank[r];
    if (rk != kBadRank) {
        // (one random 8-byte store per request: index and view side by side)
        a.sorted[a.cnt[a.loc[r]] + rk] = make_uint2(r, a.view[r]);
    }
}

struct DecArgs {
    const uint32_t *records;
    const uint32_t *offsets;
    const int16_t *top;       // [n_top][nloc][48]
    const uint32_t *view_anc; // [n_views][kMaxLevels]
    const uint32_t *start;    // [nloc + 1] bin starts
    const uint2 *sorted;
    uint8_t *out;
    uint32_t *queue;
    uint32_t nloc, L, q, MW, level, pmax, locs_per_pop, stage, stage_words, warp_words;
    uint32_t slots;           // requests per round
    uint32_t aligned;         // output alignment: 16, 4 or 1 bytes
    uint32_t anc_views;       // views whose ancestors are cached in shared memory, 16 bits each (0: read them from global)
    uint32_t *dbg;            // debug builds: the stream's flag word
};

// Per-warp shared-memory words for a configuration (the CTA adds the cached
// ancestor table after its warps' slices).
// stage: 0 none, 1 one buffer, 2 two buffers (prefetch); each buffer holds
// stage_words + 4 words.  What a configuration may need (create and
// set_config refuse larger ones) is at least what it uses with kSlotsTight.
__host__ __device__ inline uint32_t warp_words_limit(uint32_t MW, uint32_t pmax, uint32_t L, uint32_t stage,
                                                     uint32_t stage_words)
{
    const uint32_t w = 6 * MW + 3 * pmax + 528 + 24 * (L - 1) + stage * (stage_words + 4);
    return (w + 3u) & ~3u;
}
// masks and their prefixes, payload offsets, accumulators (8 pairs of each of
// 3 channels per slot, at an odd pitch), request index and view, task list
__host__ __device__ inline uint32_t warp_words_for(uint32_t MW, uint32_t pmax, uint32_t L, uint32_t stage, uint32_t stage_words,
                                                   uint32_t off_bytes, uint32_t n)
{
    const uint32_t w = 6 * MW + (3 * pmax * off_bytes + 3) / 4 + 8 * (3 * n + 1) + 2 * n + 3 * n * (L - 1) +
                       stage * (stage_words + 4);
    return (w + 3u) & ~3u;
}

template <typename OffT>
__global__ void __launch_bounds__(512, 2) decode_binned_kernel(const DecArgs a)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ uint32_t s_mode[32];
    __shared__ uint16_t s_dig[256 + 128];
    if (threadIdx.x < 32)
        s_mode[threadIdx.x] = g_tables.mode[threadIdx.x];
    for (uint32_t i = threadIdx.x; i < (256 + 128) / 2; i += blockDim.x)
        reinterpret_cast<uint32_t *>(s_dig)[i] = reinterpret_cast<const uint32_t *>(g_tables.dig)[i];
    // the ancestor table, shared by the CTA's warps when it is small
    uint16_t *s_anc = reinterpret_cast<uint16_t *>(smem + (blockDim.x >> 5) * a.warp_words);
    for (uint32_t i = threadIdx.x; i < a.anc_views * kMaxLevels; i += blockDim.x)
        s_anc[i] = (uint16_t)a.view_anc[i];
    __syncthreads();
    const auto ancestor = [&](uint32_t view, uint32_t l) -> uint32_t {
        return a.anc_views ? s_anc[view * kMaxLevels + l] : a.view_anc[view * kMaxLevels + l];
    };
    const int lane = (int)(threadIdx.x & 31u);
    const uint32_t pitch = 3 * a.slots + 1;
    uint32_t *s_mask = smem + (threadIdx.x >> 5) * a.warp_words;   // [3][MW]
    uint32_t *s_mpre = s_mask + 3 * a.MW;                           // [3][MW] stored blocks in front of each word, records one after the other
    uint32_t *s_acc = s_mpre + 3 * a.MW;                            // [8][pitch] pair j of (slot, channel)
    uint32_t *s_list = s_acc + 8 * pitch;                           // [slots * 3 * (L-1)]
    uint32_t *s_req = s_list + 3 * a.slots * (a.L - 1), *s_view = s_req + a.slots;
    OffT *s_off = reinterpret_cast<OffT *>(s_view + a.slots);       // [3 pmax] payload bit offsets, records one after the other
    uint32_t *s_stage = s_view + a.slots + (3 * a.pmax * (uint32_t)sizeof(OffT) + 3) / 4;
    const uint32_t nl = a.L - 1 - a.level;   // SRV levels added to the top RKV
    const uint32_t hdr0 = 32 * a.MW;
    // (division of task numbers below 2^10 by 3 nl and nl)
    const uint32_t inv3 = nl ? (65536u + 3 * nl - 1) / (3 * nl) : 0u, inv1 = nl ? (65536u + nl - 1) / nl : 0u;

    // One location: parse its three records (from `staged` when they were
    // copied to shared memory, else from the stream) and serve its requests.
    auto serve = [&](uint32_t loc, const uint32_t *staged) {
        const uint32_t r0 = a.start[loc], r1 = a.start[loc + 1];
        if (r0 == r1)
            return;
        const uint32_t o0 = a.offsets[3 * loc];
        const uint32_t d1 = a.offsets[3 * loc + 1] - o0, d2 = a.offsets[3 * loc + 2] - o0;
        const uint32_t span = a.offsets[3 * loc + 3] - o0;
        const uint32_t *base = staged ? staged : a.records + o0;
        if (!staged && a.stage == 1 && span <= a.stage_words) {
            // the bit reader may touch two words past a record: copy them too
            // (the stream carries zero padding after its last record)
            for (uint32_t i = lane; i < span + 2; i += 32)
                s_stage[i] = base[i];
            __syncwarp();
            base = s_stage;
        }
        const auto rec_of = [&](uint32_t c) { return base + (c == 0 ? 0u : (c == 1 ? d1 : d2)); };
        // masks: a lane per (channel, word)
        uint32_t total = 0, p1 = 0, p2 = 0;   // stored blocks; those in front of records 1 and 2
        for (uint32_t w0 = 0; w0 < 3 * a.MW; w0 += 32) {
            const uint32_t i = w0 + lane;
            const uint32_t c = (i >= a.MW) + (i >= 2 * a.MW);
            const uint32_t word = i < 3 * a.MW ? rec_of(c)[i - c * a.MW] : 0u;
            const uint32_t cnt = __popc(word);
            const uint32_t excl = total + scan_incl(cnt, lane) - cnt;
            if (i < 3 * a.MW) {
                s_mask[i] = word;
                s_mpre[i] = excl;
            }
            if (a.MW - w0 < 32)
                p1 = __shfl_sync(kFull, excl, a.MW - w0);
            if (2 * a.MW - w0 < 32)
                p2 = __shfl_sync(kFull, excl, 2 * a.MW - w0);
            total = __shfl_sync(kFull, excl + cnt, 31);
        }
        // headers, record after record: payload offset of every stored block
        // inside its record
        const uint32_t pay0[3] = {hdr0 + kHdrBits * p1, hdr0 + kHdrBits * (p2 - p1), hdr0 + kHdrBits * (total - p2)};
        uint32_t run = 0, g1 = 0, g2 = 0;     // payload bits so far; in front of records 1 and 2
#pragma unroll 2
        for (uint32_t h0 = 0; h0 < total; h0 += 32) {
            const uint32_t i = h0 + lane;
            const uint32_t c = (i >= p1) + (i >= p2), h = i - (c == 0 ? 0u : (c == 1 ? p1 : p2));
            const uint32_t len = i < total ? mode_bits(s_mode[get_bits(rec_of(c), hdr0 + kHdrBits * h, 5)]) : 0u;
            const uint32_t incl = scan_incl(len, lane), excl = run + incl - len;
            if (p1 - h0 < 32)
                g1 = __shfl_sync(kFull, excl, p1 - h0);
            if (p2 - h0 < 32)
                g2 = __shfl_sync(kFull, excl, p2 - h0);
            if (i < total)
                s_off[i] = (OffT)(pay0[0] * (c == 0) + (pay0[1] - g1) * (c == 1) + (pay0[2] - g2) * (c == 2) + excl);
            run += __shfl_sync(kFull, incl, 31);
        }
        __syncwarp();
        for (uint32_t j0 = r0; j0 < r1; j0 += a.slots) {
            const uint32_t ns = min(a.slots, r1 - j0);
            if ((uint32_t)lane < ns) {
                const uint2 rq = a.sorted[j0 + lane];
                s_req[lane] = rq.x;
                s_view[lane] = rq.y;
            }
            __syncwarp();
            // ReadBlock(RKV^n, BlkIdx): the accumulators start at the top RKV
            // (96 bytes per slot, as six 16-byte loads)
            for (uint32_t i = lane; i < ns * 6; i += 32) {
                const uint32_t slot = (i * 10923u) >> 16, k = i - slot * 6;
                const uint32_t top = ancestor(s_view[slot], a.L - 1);
                const uint4 v = __ldg(reinterpret_cast<const uint4 *>(a.top + ((size_t)top * a.nloc + loc) * 48) + k);
                uint32_t *d = s_acc + 4 * (k & 1) * pitch + slot * 3 + (k >> 1);
                d[0] = (v.x ^ 0x80008000u) - kB2;
                d[pitch] = (v.y ^ 0x80008000u) - kB2;
                d[2 * pitch] = (v.z ^ 0x80008000u) - kB2;
                d[3 * pitch] = (v.w ^ 0x80008000u) - kB2;
            }
            // stored ancestor blocks of these requests, compacted
            const uint32_t ntask = ns * 3 * nl;
            uint32_t cnt = 0;
            for (uint32_t t0 = 0; t0 < ntask; t0 += 32) {
                const uint32_t t = t0 + lane;
                uint32_t code = 0;
                bool pres = false;
                if (t < ntask) {
                    const uint32_t slot = (t * inv3) >> 16, rem = t - slot * 3 * nl;
                    const uint32_t c = (rem * inv1) >> 16, l = a.level + (rem - c * nl);
                    const uint32_t node = ancestor(s_view[slot], l);
                    const uint32_t wi = c * a.MW + (node >> 5), bit = node & 31u;
                    const uint32_t word = s_mask[wi];
                    pres = (word >> bit) & 1u;
                    code = (s_mpre[wi] + __popc(word & ((1u << bit) - 1u))) | (c << 16) | (slot << 18);
                }
                const uint32_t bal = __ballot_sync(kFull, pres);
                if (pres)
                    s_list[cnt + __popc(bal & ((1u << lane) - 1u))] = code;
                cnt += __popc(bal);
            }
            __syncwarp();
            // BISEDecode + CombineBlocks, one thread per stored block
            for (uint32_t i = lane; i < cnt; i += 32) {
                const uint32_t code = s_list[i];
                const uint32_t at = code & 0xFFFFu, c = (code >> 16) & 3u, slot = code >> 18;   // at: among the three records' blocks
                const uint32_t rank = at - (c == 0 ? 0u : (c == 1 ? p1 : p2));
                const uint32_t *rc = rec_of(c);
                const uint32_t hdr = get_bits(rc, hdr0 + kHdrBits * rank, kHdrBits), pos = s_off[at];
#ifdef RLFC_DEBUG
                {
                    const uint32_t mode = hdr & 31u;
                    const uint32_t rec_words = c == 0 ? d1 : (c == 1 ? d2 - d1 : span - d2);
                    const uint32_t P = c == 0 ? p1 : (c == 1 ? p2 - p1 : total - p2);
                    if (!RLFC_DBG_BLOCK_OK(a.dbg, mode, hdr0 + kHdrBits * (rank + 1), hdr0 + kHdrBits * P, pos,
                                           mode < (uint32_t)kNumModes ? mode_bits(s_mode[mode]) : 0u, 32u * rec_words))
                        continue;
                }
#endif
                uint32_t v[8];
                decode_block_pairs(rc, pos, hdr, a.q, s_mode, s_dig, v);
                uint32_t *dst = s_acc + slot * 3 + c;
#pragma unroll
                for (int j = 0; j < 8; j++)
                    atomicAdd(dst + j * pitch, v[j] - kB2);
            }
            __syncwarp();
            // a lane per block row
            for (uint32_t t0 = 0; t0 < 4 * ns; t0 += 32) {
                const uint32_t t = t0 + lane, slot = min(t >> 2, ns - 1), rr = t & 3u;
                const uint32_t *p = s_acc + 2 * rr * pitch + slot * 3;
                uint32_t w[4];
                row_to_rgb<false>(make_uint2(p[0], p[pitch]), make_uint2(p[1], p[pitch + 1]), make_uint2(p[2], p[pitch + 2]), w);
                uint8_t *o = a.out + (size_t)s_req[slot] * 48;
                if (a.aligned == 16) {
                    // rows of 12 bytes to three 16-byte pieces: row rr gives its
                    // piece rr the words it holds of it, row rr + 1 the rest
                    const uint32_t n0 = __shfl_down_sync(kFull, w[0], 1), n1 = __shfl_down_sync(kFull, w[1], 1),
                                   n2 = __shfl_down_sync(kFull, w[2], 1);
                    const uint4 v = rr == 0 ? make_uint4(w[0], w[1], w[2], n0)
                                            : (rr == 1 ? make_uint4(w[1], w[2], n0, n1) : make_uint4(w[2], n0, n1, n2));
                    if (t < 4 * ns && rr < 3)
                        reinterpret_cast<uint4 *>(o)[rr] = v;
                } else if (t < 4 * ns) {
                    if (a.aligned == 4) {
#pragma unroll
                        for (int k = 0; k < 3; k++)
                            reinterpret_cast<uint32_t *>(o)[3 * rr + k] = w[k];
                    } else {
#pragma unroll
                        for (int k = 0; k < 12; k++)
                            o[12 * rr + k] = (uint8_t)(w[k >> 2] >> (8 * (k & 3)));
                    }
                }
            }
            __syncwarp();
        }
    };

    if (a.stage == 2) {
        // prefetching: while a location is served, the records of the next
        // one are copied into the warp's other buffer (cp.async)
        uint32_t *const buf0 = s_stage, *const buf1 = s_stage + a.stage_words + 4;
        auto pop = [&]() {
            uint32_t v = 0;
            if (lane == 0)
                v = atomicAdd(a.queue, 1u);
            return __shfl_sync(kFull, v, 0);
        };
        auto prefetch = [&](uint32_t loc, uint32_t *dst) {
            if (loc >= a.nloc)
                return false;
            const uint32_t o0 = a.offsets[3 * loc], span = a.offsets[3 * loc + 3] - o0;
            if (span > a.stage_words)
                return false;
            for (uint32_t i = lane; i < span + 2; i += 32)
                __pipeline_memcpy_async(dst + i, a.records + o0 + i, 4);
            return true;
        };
        uint32_t cur = pop();
        bool cur_in = prefetch(cur, buf0);
        __pipeline_commit();
        uint32_t parity = 0;
        while (cur < a.nloc) {
            const uint32_t nxt = pop();
            const bool nxt_in = prefetch(nxt, parity ? buf0 : buf1);
            __pipeline_commit();
            __pipeline_wait_prior(1);   // this lane's copies of `cur` are done
            __syncwarp();               // and every lane's
            serve(cur, cur_in ? (parity ? buf1 : buf0) : nullptr);
            __syncwarp();               // the buffer is free for the prefetch after next
            cur = nxt;
            cur_in = nxt_in;
            parity ^= 1u;
        }
        __pipeline_wait_prior(0);
        return;
    }
    for (;;) {
        uint32_t first = 0;
        if (lane == 0)
            first = atomicAdd(a.queue, a.locs_per_pop);
        first = __shfl_sync(kFull, first, 0);
        if (first >= a.nloc)
            break;
        const uint32_t last = min(first + a.locs_per_pop, a.nloc);
        for (uint32_t loc = first; loc < last; loc++)
            serve(loc, nullptr);
    }
}

bool valid_config(const rlfc_batch_config &c)
{
    return (c.warps_per_cta == 4 || c.warps_per_cta == 8 || c.warps_per_cta == 16) && c.locs_per_pop >= 1 &&
           c.locs_per_pop <= 64 && c.stage <= 2 && c.graph <= 1;
}

}  // namespace
}  // namespace rlfc

struct rlfc_batch {
    const rlfc_stream *s = nullptr;
    int device = 0;
    size_t max_n = 0;
    uint32_t nloc = 0, pmax = 1, stage_words = 0, smem_optin = 0, smem_dyn = 0, sms = 0;   // smem_dyn: what the kernel has besides its static part
    uint32_t *d_cnt = nullptr;      // nloc + 2 words, then one per scan chunk
    uint32_t *d_rank = nullptr;     // max_n
    uint2 *d_sorted = nullptr;      // max_n
    uint32_t anc_views = 0;         // views whose ancestors are cached per CTA (0 = none)
    uint32_t off_bytes = 4;         // bytes of a payload offset: 2 while every record is shorter than 2^16 bits
    rlfc_batch_config cfg{8, 1, 0, 1};
    cudaStream_t cap = nullptr;     // private stream, only ever capturing
    cudaGraphExec_t exec = nullptr;
    struct Key {
        const void *view, *loc, *out, *status;
        size_t n;
        uint32_t level;
        bool operator==(const Key &o) const
        {
            return view == o.view && loc == o.loc && out == o.out && status == o.status && n == o.n &&
                   level == o.level;
        }
    } key{};
};

namespace rlfc {
namespace {

uint32_t warp_words(const rlfc_batch *b, const rlfc_batch_config &c, uint32_t slots)
{
    return warp_words_for(b->s->MW, b->pmax, b->s->tab.L, c.stage, b->stage_words, b->off_bytes, slots);
}
uint32_t smem_bytes(const rlfc_batch *b, const rlfc_batch_config &c, uint32_t slots)
{
    return c.warps_per_cta * 4u * warp_words(b, c, slots) + 2u * kMaxLevels * b->anc_views;
}
uint32_t slots_for(const rlfc_batch *b, const rlfc_batch_config &c)
{
    return smem_bytes(b, c, kSlots) <= b->smem_dyn ? kSlots : kSlotsTight;
}

bool fits(const rlfc_batch *b, const rlfc_batch_config &c)
{
    return c.warps_per_cta * 4u * warp_words_limit(b->s->MW, b->pmax, b->s->tab.L, c.stage, b->stage_words) +
               4u * kMaxLevels * b->anc_views <= b->smem_optin - kStaticLimit;
}

using BinnedKernel = void (*)(const DecArgs);
BinnedKernel binned_kernel(uint32_t off_bytes)
{
    return off_bytes == 2 ? decode_binned_kernel<uint16_t> : decode_binned_kernel<uint32_t>;
}

int enqueue(rlfc_batch *b, const rlfc_batch_config &cfg, const uint32_t *view, const uint32_t *loc, uint32_t n,
            uint32_t level, uint8_t *out, uint8_t *status, cudaStream_t st)
{
    const rlfc_stream *s = b->s;
    cudaError_t e = cudaMemsetAsync(b->d_cnt, 0, (size_t)(b->nloc + 2) * 4, st);
    if (e != cudaSuccess)
        return cuda_fail(e, "batch scratch clear");
    BinArgs ba;
    ba.view = view;
    ba.loc = loc;
    ba.out = out;
    ba.status = status;
    ba.cnt = b->d_cnt;
    ba.rank = b->d_rank;
    ba.sorted = b->d_sorted;
    ba.n = n;
    ba.n_views = s->tab.n_views;
    ba.nloc = b->nloc;
    ba.aligned = ((uintptr_t)out & 3u) == 0;
    const uint32_t g = (n + 255) / 256;
    { TraceScope trace_("bin_count_kernel", st); bin_count_kernel<<<g, 256, 0, st>>>(ba); }
    const uint32_t chunks = (b->nloc + kScanChunk - 1) / kScanChunk;
    uint32_t *part = b->d_cnt + b->nloc + 2;
    { TraceScope trace_("bin_reduce_kernel", st); bin_reduce_kernel<<<chunks, 1024, 0, st>>>(b->d_cnt, b->nloc, part); }
    { TraceScope trace_("bin_scan_kernel", st); bin_scan_kernel<<<chunks, 1024, 0, st>>>(b->d_cnt, b->nloc, part); }
    { TraceScope trace_("bin_scatter_kernel", st); bin_scatter_kernel<<<g, 256, 0, st>>>(ba); }

    DecArgs da;
    da.dbg = s->d_debug;
    da.records = s->d_records;
    da.offsets = s->d_offsets;
    da.top = s->d_top;
    da.view_anc = s->d_view_anc;
    da.start = b->d_cnt;
    da.sorted = b->d_sorted;
    da.anc_views = b->anc_views;
    da.slots = slots_for(b, cfg);
    da.out = out;
    da.queue = b->d_cnt + b->nloc + 1;
    da.nloc = b->nloc;
    da.L = s->tab.L;
    da.q = s->info.q;
    da.MW = s->MW;
    da.level = level;
    da.pmax = b->pmax;
    da.locs_per_pop = cfg.locs_per_pop;
    da.stage = cfg.stage;
    da.stage_words = b->stage_words;
    da.warp_words = warp_words(b, cfg, da.slots);
    da.aligned = ((uintptr_t)out & 15u) == 0 ? 16u : (ba.aligned ? 4u : 1u);
    const uint32_t threads = cfg.warps_per_cta * 32, smem = smem_bytes(b, cfg, da.slots);
    int per_sm = 0;
    const BinnedKernel kern = binned_kernel(b->off_bytes);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, (int)threads, smem);
    if (e != cudaSuccess)
        return cuda_fail(e, "batch occupancy");
    const uint32_t grid = b->sms * (uint32_t)std::max(per_sm, 1);
    { TraceScope trace_("decode_binned_kernel", st); kern<<<grid, threads, smem, st>>>(da); }
    e = cudaGetLastError();
    if (e != cudaSuccess)
        return cuda_fail(e, "batch decode launch");
    return RLFC_OK;
}

void drop_graph(rlfc_batch *b)
{
    if (b->exec)
        cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
}

int check_args(const rlfc_batch *b, const uint32_t *view, const uint32_t *loc, size_t n, uint32_t level,
               const uint8_t *out)
{
    if (!b || (n && (!view || !loc || !out))) {
        set_error("rlfc_batch: null argument");
        return RLFC_E_INVALID_ARG;
    }
    if (level > b->s->tab.L - 1) {
        set_error("rlfc_batch_decode: level must be at most L-1");
        return RLFC_E_INVALID_ARG;
    }
    if (n > b->max_n) {
        set_error("rlfc_batch_decode: more requests than the batch object was created for");
        return RLFC_E_RANGE;
    }
    return RLFC_OK;
}

}  // namespace
}  // namespace rlfc

extern "C" {

RLFC_API int rlfc_batch_create(const rlfc_stream *s, size_t max_requests, rlfc_batch **out)
{
    using namespace rlfc;
    if (!s || !out) {
        set_error("rlfc_batch_create: null argument");
        return RLFC_E_INVALID_ARG;
    }
    *out = nullptr;
    if (max_requests >= (1ull << 31)) {
        set_error("rlfc_batch_create: max_requests must be below 2^31");
        return RLFC_E_RANGE;
    }
    DeviceGuard g(s->device);
    rlfc_batch *b = new (std::nothrow) rlfc_batch;
    if (!b) {
        set_error("rlfc_batch_create: out of host memory");
        return RLFC_E_OOM;
    }
    b->s = s;
    b->device = s->device;
    b->max_n = std::max<size_t>(max_requests, 1);
    b->nloc = s->info.nloc_x * s->info.nloc_y;
    b->pmax = std::max<uint32_t>(s->max_present, 1u);
    b->stage_words = std::min<uint32_t>(3u * s->max_record_words, kStageCap);
    // the ancestor table is cached per CTA up to 1024 views
    b->anc_views = s->tab.n_views <= 1024u ? s->tab.n_views : 0u;
    b->off_bytes = s->max_record_words < 2048u ? 2u : 4u;
    int v = 0;
    cudaError_t e = cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, s->device);
    b->smem_optin = e == cudaSuccess ? (uint32_t)v : 48u * 1024u;
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, s->device);
    b->sms = (uint32_t)v;
    cudaFuncAttributes fa{};
    if (e == cudaSuccess)
        e = cudaFuncGetAttributes(&fa, binned_kernel(b->off_bytes));
    if (e == cudaSuccess) {
        // the opt-in limit covers static and dynamic shared memory together
        b->smem_dyn = b->smem_optin - std::min<uint32_t>(b->smem_optin, (uint32_t)fa.sharedSizeBytes);
        e = cudaFuncSetAttribute(binned_kernel(b->off_bytes), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)b->smem_dyn);
    }
    if (e != cudaSuccess) {
        delete b;
        return cuda_fail(e, "rlfc_batch_create");
    }
    rlfc_batch_config c{4, 1, 0, 1};
    if (!fits(b, c)) {
        set_error("rlfc_batch_create: the records' parse state does not fit in shared memory");
        delete b;
        return RLFC_E_UNSUPPORTED;
    }
    if (!fits(b, b->cfg))
        b->cfg = c;
    const size_t chunks = (b->nloc + kScanChunk - 1) / kScanChunk;
    if ((e = cudaMalloc(&b->d_cnt, (size_t)(b->nloc + 2 + chunks) * 4)) != cudaSuccess ||
        (e = cudaMalloc(&b->d_rank, b->max_n * 4)) != cudaSuccess ||
        (e = cudaMalloc(&b->d_sorted, b->max_n * 8)) != cudaSuccess ||
        (e = cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking)) != cudaSuccess) {
        const int rc = e == cudaErrorMemoryAllocation ? RLFC_E_OOM : RLFC_E_CUDA;
        cuda_fail(e, "rlfc_batch_create");
        cudaGetLastError();
        rlfc_batch_free(b);
        return rc;
    }
    *out = b;
    return RLFC_OK;
}

RLFC_API int rlfc_batch_set_config(rlfc_batch *b, const rlfc_batch_config *cfg)
{
    using namespace rlfc;
    if (!b || !cfg || !valid_config(*cfg)) {
        set_error("rlfc_batch_set_config: invalid configuration");
        return RLFC_E_INVALID_ARG;
    }
    if (!fits(b, *cfg)) {
        set_error("rlfc_batch_set_config: configuration needs more shared memory than a CTA has");
        return RLFC_E_UNSUPPORTED;
    }
    DeviceGuard g(b->device);
    drop_graph(b);
    b->cfg = *cfg;
    return RLFC_OK;
}

RLFC_API int rlfc_batch_get_config(const rlfc_batch *b, rlfc_batch_config *cfg)
{
    if (!b || !cfg) {
        rlfc::set_error("rlfc_batch_get_config: null argument");
        return RLFC_E_INVALID_ARG;
    }
    *cfg = b->cfg;
    return RLFC_OK;
}

RLFC_API int rlfc_batch_decode(rlfc_batch *b, const uint32_t *d_view, const uint32_t *d_loc, size_t n,
                               uint32_t level, uint8_t *d_out, uint8_t *d_status, void *cuda_stream)
{
    using namespace rlfc;
    int rc = check_args(b, d_view, d_loc, n, level, d_out);
    if (rc != RLFC_OK || n == 0)
        return rc;
    DeviceGuard g(b->device);
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (!b->cfg.graph)
        return enqueue(b, b->cfg, d_view, d_loc, (uint32_t)n, level, d_out, d_status, st);
    const rlfc_batch::Key k{d_view, d_loc, d_out, d_status, n, level};
    if (!b->exec || !(k == b->key)) {
        drop_graph(b);
        cudaError_t e = cudaStreamBeginCapture(b->cap, cudaStreamCaptureModeRelaxed);
        if (e != cudaSuccess)
            return cuda_fail(e, "batch graph capture");
        rc = enqueue(b, b->cfg, d_view, d_loc, (uint32_t)n, level, d_out, d_status, b->cap);
        cudaGraph_t graph = nullptr;
        e = cudaStreamEndCapture(b->cap, &graph);
        if (rc != RLFC_OK) {
            if (graph)
                cudaGraphDestroy(graph);
            return rc;
        }
        if (e != cudaSuccess)
            return cuda_fail(e, "batch graph capture");
        e = cudaGraphInstantiate(&b->exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            b->exec = nullptr;
            return cuda_fail(e, "batch graph instantiate");
        }
        b->key = k;
    }
    cudaError_t e;
    {
        TraceScope trace_("batch_graph", st);
        e = cudaGraphLaunch(b->exec, st);
    }
    if (e != cudaSuccess)
        return cuda_fail(e, "batch graph launch");
    return RLFC_OK;
}

RLFC_API int rlfc_batch_autotune(rlfc_batch *b, const uint32_t *d_view, const uint32_t *d_loc, size_t n,
                                 uint8_t *d_out, uint8_t *d_status, void *cuda_stream,
                                 rlfc_batch_config *chosen)
{
    using namespace rlfc;
    int rc = check_args(b, d_view, d_loc, n, 0, d_out);
    if (rc != RLFC_OK)
        return rc;
    DeviceGuard g(b->device);
    cudaStream_t st = (cudaStream_t)cuda_stream;
    rlfc_batch_config best = b->cfg;
    if (n > 0) {
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        cudaError_t e = cudaEventCreate(&e0);
        if (e == cudaSuccess)
            e = cudaEventCreate(&e1);
        float best_ms = 1e30f;
        const uint32_t warps[3] = {4, 8, 16}, pops[2] = {1, 4};
        for (uint32_t wi = 0; wi < 3 && e == cudaSuccess && rc == RLFC_OK; wi++)
            for (uint32_t pi = 0; pi < 2 && e == cudaSuccess && rc == RLFC_OK; pi++)
                for (uint32_t stg = 0; stg < 3 && e == cudaSuccess && rc == RLFC_OK; stg++) {
                    if (stg == 2 && pi != 0)
                        continue;   // prefetching takes one location at a time
                    const rlfc_batch_config c{warps[wi], pops[pi], stg, b->cfg.graph};
                    if (!fits(b, c))
                        continue;
                    rc = enqueue(b, c, d_view, d_loc, (uint32_t)n, 0, d_out, d_status, st);   // warm-up
                    if (rc != RLFC_OK)
                        break;
                    e = cudaEventRecord(e0, st);
                    for (int rep = 0; rep < 3 && rc == RLFC_OK; rep++)
                        rc = enqueue(b, c, d_view, d_loc, (uint32_t)n, 0, d_out, d_status, st);
                    if (e == cudaSuccess)
                        e = cudaEventRecord(e1, st);
                    if (e == cudaSuccess)
                        e = cudaEventSynchronize(e1);
                    float ms = 0.f;
                    if (e == cudaSuccess)
                        e = cudaEventElapsedTime(&ms, e0, e1);
                    if (e == cudaSuccess && rc == RLFC_OK && ms < best_ms) {
                        best_ms = ms;
                        best = c;
                    }
                }
        if (e0)
            cudaEventDestroy(e0);
        if (e1)
            cudaEventDestroy(e1);
        if (rc != RLFC_OK)
            return rc;
        if (e != cudaSuccess)
            return cuda_fail(e, "batch autotune");
    }
    drop_graph(b);
    b->cfg = best;
    if (chosen)
        *chosen = best;
    return RLFC_OK;
}

RLFC_API void rlfc_batch_free(rlfc_batch *b)
{
    if (!b)
        return;
    rlfc::DeviceGuard g(b->device);
    // a decode still in flight may use the batch's buffers: let the device finish first
    cudaDeviceSynchronize();
    rlfc::drop_graph(b);
    if (b->cap)
        cudaStreamDestroy(b->cap);
    cudaFree(b->d_cnt);
    cudaFree(b->d_rank);
    cudaFree(b->d_sorted);
    delete b;
}

}  // extern "C"
