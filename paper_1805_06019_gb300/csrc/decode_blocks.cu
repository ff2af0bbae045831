// Random-access block decode, Algorithm 2 DecompressLFIBlock(ImgIdx, BlkIdx),
// for a batch of independent requests.  Few requests: one warp each, using the
// warp-cooperative block decoder (the shortest chain of loads).  Many: one
// thread per (request, channel), which walks its record alone (a sixth of the
// instructions).  Out-of-range requests get a status byte and a zeroed block;
// nothing traps.
#include <cuda_runtime.h>

#include "pair_decode.cuh"
#include "warp_decode.cuh"

namespace rlfc {
namespace {

constexpr int kWarpsPerCta = 8;
// The thread-per-channel form pays from this many requests on (fewer leave its
// long walks with too little to overlap), more for records of many nodes.
// Measured, a warp per request / a thread per channel, us of queued calls (of
// the 10.4 at 4096 requests the kernel takes 9.2): 9 x 9 views (three
// mask words) 10.4 / 14.8 at 4096, 14.6 / 14.6 at 8192, 98 / 33 at 10^5; 17 x
// 17 views (ten words) 16.7 / 24.7 at 8192, 24.8 / 24.8 at 16384, 103 / 55 at
// 10^5; 5 x 5 views 10.0 / 9.2 at 4096, 103 / 21 at 10^5.
constexpr uint32_t kWalkFrom = 8192, kWalkFromLong = 16384, kWalkShortMask = 4;
constexpr uint32_t kReqs = 64;   // requests per CTA of the thread-per-channel form: two warps per channel

__constant__ uint32_t c_modes[kNumModes] = RLFC_MODE_TABLE_INIT;

struct Args {
    StreamView sv;
    const uint32_t *req_view;
    const uint32_t *req_loc;
    uint8_t *out;
    uint8_t *status;
    uint32_t n;
    uint32_t aligned;   // output 4-byte aligned: store whole words
};

__global__ void __launch_bounds__(kWarpsPerCta * 32) decode_blocks_kernel(const Args a)
{
    __shared__ uint32_t s_mode[kNumModes];
    if (threadIdx.x < kNumModes)
        s_mode[threadIdx.x] = c_modes[threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const uint32_t r = blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5);
    if (r >= a.n)
        return;
    const uint32_t view = a.req_view[r], loc = a.req_loc[r];
    uint8_t *dst = a.out + (size_t)r * 48;
    const uint32_t bad = view >= a.sv.n_views ? (uint32_t)RLFC_REQ_BAD_VIEW
                                              : (loc >= a.sv.nloc ? (uint32_t)RLFC_REQ_BAD_LOCATION : 0u);
    if (a.status && lane == 0)
        a.status[r] = (uint8_t)bad;
    if (bad) {
        if (a.aligned) {
            if (lane < 12)
                reinterpret_cast<uint32_t *>(dst)[lane] = 0u;
        } else {
            for (int b = lane; b < 48; b += 32)
                dst[b] = 0;
        }
        return;
    }
    const uint32_t rgb = warp_decode_block(a.sv, s_mode, view, loc, lane);
    if (a.aligned) {
        // 48 bytes as 12 words: word w holds bytes 4w..4w+3, which start at
        // byte (4w) % 3 of pixel (4w) / 3 and end inside the next pixel
        const uint32_t p0 = (uint32_t)(lane * 4) / 3;
        const uint32_t lo = __shfl_sync(kFullMask, rgb, min(p0, 31u));
        const uint32_t hi = __shfl_sync(kFullMask, rgb, min(p0 + 1, 31u));
        if (lane < 12) {
            const uint32_t sh = (uint32_t)(lane * 4) % 3;   // first byte of the word inside pixel p0
            reinterpret_cast<uint32_t *>(dst)[lane] =
                __byte_perm(lo, hi, sh == 0 ? 0x4210u : (sh == 1 ? 0x5421u : 0x6542u));
        }
    } else if (lane < 16) {
        dst[3 * lane] = (uint8_t)rgb;
        dst[3 * lane + 1] = (uint8_t)(rgb >> 8);
        dst[3 * lane + 2] = (uint8_t)(rgb >> 16);
    }
}

// Warp w of a CTA takes channel w / 2 of 32 requests, a lane each: it walks the
// record's headers up to the view's ancestors (in BFS order: coarse levels
// first) and adds their blocks to the top RKV with the pair decoder; then a
// thread per (request, block row) converts and stores.
// What bounds it: instruction issue and the walks' dependent loads; 10^5
// requests on 9 x 9 x 512^2 take 33 us (98 with a warp per request).
__global__ void __launch_bounds__(kReqs * 3) decode_blocks_walk_kernel(const Args a)
{
    __shared__ uint32_t s_mode[32];
    __shared__ uint16_t s_dig[256 + 128];
    __shared__ uint32_t s_acc[8][kReqs * 3 + 1];   // pair j of (channel, request)
    __shared__ uint8_t s_bad[kReqs];
    const uint32_t tid = threadIdx.x;
    if (tid < 32)
        s_mode[tid] = g_tables.mode[tid];
    for (uint32_t i = tid; i < (256 + 128) / 2; i += kReqs * 3)
        reinterpret_cast<uint32_t *>(s_dig)[i] = reinterpret_cast<const uint32_t *>(g_tables.dig)[i];
    __syncthreads();
    const uint32_t c = tid / kReqs, q = tid - c * kReqs, r = blockIdx.x * kReqs + q;
    const uint32_t L1 = a.sv.L - 1;
    uint32_t bad = 0, view = 0, loc = 0;
    if (r < a.n) {
        view = a.req_view[r];
        loc = a.req_loc[r];
        bad = view >= a.sv.n_views ? (uint32_t)RLFC_REQ_BAD_VIEW : (loc >= a.sv.nloc ? (uint32_t)RLFC_REQ_BAD_LOCATION : 0u);
        if (c == 0) {
            s_bad[q] = (uint8_t)bad;
            if (a.status)
                a.status[r] = (uint8_t)bad;
        }
    }
    if (r < a.n && !bad) {
        const uint32_t *anc = a.sv.view_anc + view * kMaxLevels;
        const uint4 *tp = reinterpret_cast<const uint4 *>(a.sv.top + ((size_t)anc[L1] * a.sv.nloc + loc) * 48 + c * 16);
        const uint4 t0 = __ldg(tp), t1 = __ldg(tp + 1);
        uint32_t v[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
#pragma unroll
        for (int j = 0; j < 8; j++)
            v[j] = (v[j] ^ 0x80008000u) - kB2;
        const uint32_t *rec = a.sv.records + a.sv.offsets[3 * loc + c];
        uint32_t P = 0;
        for (uint32_t m = 0; m < a.sv.MW; m++)
            P += __popc(rec[m]);
        const uint32_t hdr0 = 32 * a.sv.MW;
        uint32_t off = hdr0 + kHdrBits * P, rank = 0, at = 0, word = rec[0], before = 0;   // before: blocks in front of word `at`
        HeaderReader hr(rec, a.sv.MW);
        for (uint32_t l = L1; l-- > 0;) {
            const uint32_t p = anc[l], bit = 1u << (p & 31u);
            while (at < (p >> 5)) {
                before += __popc(word);
                word = rec[++at];
            }
            if (!(word & bit))
                continue;
            const uint32_t target = before + __popc(word & (bit - 1u));
            for (; rank < target; rank++)
                off += mode_bits(s_mode[hr.take() & 31u]);
            const uint32_t hdr = hr.take();
            rank++;
            const uint32_t pay = mode_bits(s_mode[hdr & 31u]);
#ifdef RLFC_DEBUG
            const uint32_t rec_bits = 32u * (a.sv.offsets[3 * loc + c + 1] - a.sv.offsets[3 * loc + c]);
            if (RLFC_DBG_BLOCK_OK(a.sv.dbg, hdr & 31u, hdr0 + kHdrBits * rank, hdr0 + kHdrBits * P, off, pay, rec_bits))
#endif
            {
                uint32_t d[8];
                decode_block_pairs(rec, off, hdr, a.sv.q, s_mode, s_dig, d);
#pragma unroll
                for (int j = 0; j < 8; j++)
                    v[j] += d[j] - kB2;
            }
            off += pay;
        }
#pragma unroll
        for (int j = 0; j < 8; j++)
            s_acc[j][c * kReqs + q] = v[j];
    }
    __syncthreads();
    const uint32_t here = min(kReqs, a.n - blockIdx.x * kReqs);
    for (uint32_t t = tid; t < 4 * here; t += kReqs * 3) {
        const uint32_t e = t >> 2, rr = t & 3u;
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (!s_bad[e])
            row_to_rgb<false>(make_uint2(s_acc[2 * rr][e], s_acc[2 * rr + 1][e]),
                              make_uint2(s_acc[2 * rr][kReqs + e], s_acc[2 * rr + 1][kReqs + e]),
                              make_uint2(s_acc[2 * rr][2 * kReqs + e], s_acc[2 * rr + 1][2 * kReqs + e]), w);
        uint8_t *o = a.out + ((size_t)blockIdx.x * kReqs + e) * 48 + 12 * rr;
        if (a.aligned) {
#pragma unroll
            for (int k = 0; k < 3; k++)
                reinterpret_cast<uint32_t *>(o)[k] = w[k];
        } else {
#pragma unroll
            for (int k = 0; k < 12; k++)
                o[k] = (uint8_t)(w[k >> 2] >> (8 * (k & 3)));
        }
    }
}

// One thread per record: every stored block decoded, the largest
// |(min + u) * 2^(q + shift)| over the record, reduced per warp into *out.
__global__ void __launch_bounds__(256) block_magnitude_kernel(const uint32_t *records, const uint32_t *offsets,
                                                              uint32_t n_rec, uint32_t MW, uint32_t q,
                                                              uint32_t *out)
{
    const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t mx = 0;
    if (r < n_rec) {
        const uint32_t *rec = records + offsets[r];
        uint32_t P = 0;
        for (uint32_t w = 0; w < MW; w++)
            P += __popc(rec[w]);
        const uint32_t hdr0 = 32 * MW;
        uint32_t pos = hdr0 + kHdrBits * P;
        for (uint32_t h = 0; h < P; h++) {
            const BlockHeader hd = unpack_header(get_bits(rec, hdr0 + kHdrBits * h, kHdrBits));
            const uint32_t mode = c_modes[hd.mode];
            int32_t u[kVals];
            bise_decode16(rec, pos, mode, u);
            int32_t lo = u[0], hi = u[0];
#pragma unroll
            for (int v = 1; v < kVals; v++) {
                lo = min(lo, u[v]);
                hi = max(hi, u[v]);
            }
            const int32_t a = hd.min + lo, b = hd.min + hi;
            mx = max(mx, (uint32_t)max(abs(a), abs(b)) << (q + hd.shift));
            pos += mode_bits(mode);
        }
    }
    mx = __reduce_max_sync(kFullMask, mx);
    if ((threadIdx.x & 31) == 0)
        atomicMax(out, mx);
}

}  // namespace

int block_magnitude(const rlfc_stream *s, cudaStream_t st, uint32_t *mag)
{
    const uint32_t n_rec = 3 * s->info.nloc_x * s->info.nloc_y;
    uint32_t *d = nullptr;
    cudaError_t e = cudaMallocAsync(&d, 4, st);
    if (e != cudaSuccess)
        return cuda_fail(e, "block magnitude: allocation");
    if ((e = cudaMemsetAsync(d, 0, 4, st)) == cudaSuccess) {
        { rlfc::TraceScope trace_("block_magnitude_kernel", st); block_magnitude_kernel<<<(n_rec + 255) / 256, 256, 0, st>>>(s->d_records, s->d_offsets, n_rec, s->MW, s->info.q, d); }
        if ((e = cudaGetLastError()) == cudaSuccess && (e = cudaMemcpyAsync(mag, d, 4, cudaMemcpyDeviceToHost, st)) == cudaSuccess)
            e = cudaStreamSynchronize(st);
    }
    cudaFreeAsync(d, st);
    if (e != cudaSuccess)
        return cuda_fail(e, "block magnitude");
    return RLFC_OK;
}

int launch_decode_blocks(const rlfc_stream *s, const uint32_t *d_view, const uint32_t *d_loc, uint32_t n,
                         uint8_t *d_out, uint8_t *d_status, cudaStream_t st)
{
    Args a;
    a.sv.records = s->d_records;
    a.sv.offsets = s->d_offsets;
    a.sv.top = s->d_top;
    a.sv.view_anc = s->d_view_anc;
    a.sv.n_views = s->tab.n_views;
    a.sv.nloc = s->info.nloc_x * s->info.nloc_y;
    a.sv.nlx = s->info.nloc_x;
    a.sv.L = s->tab.L;
    a.sv.q = s->info.q;
    a.sv.MW = s->MW;
    a.sv.dbg = s->d_debug;
    a.req_view = d_view;
    a.req_loc = d_loc;
    a.out = d_out;
    a.status = d_status;
    a.n = n;
    a.aligned = ((uintptr_t)d_out & 3u) == 0;
    if (n >= (s->MW <= kWalkShortMask ? kWalkFrom : kWalkFromLong)) {
        { rlfc::TraceScope trace_("decode_blocks_walk_kernel", st); decode_blocks_walk_kernel<<<(n + kReqs - 1) / kReqs, kReqs * 3, 0, st>>>(a); }
        const cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? RLFC_OK : cuda_fail(e, "decode_blocks launch");
    }
    const uint32_t grid = (n + kWarpsPerCta - 1) / kWarpsPerCta;
    { rlfc::TraceScope trace_("decode_blocks_kernel", st); decode_blocks_kernel<<<grid, kWarpsPerCta * 32, 0, st>>>(a); }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return cuda_fail(e, "decode_blocks launch");
    return RLFC_OK;
}

}  // namespace rlfc
