// GPU encoder, Algorithm 1 (CompressLFI):
//   RKV^0 <- YCoCg-R of the (edge-padded) views                 [ycocg_pad_kernel]
//   ComputeRKVTree: binomial-weighted cluster filter per level   [filter_kernel]
//   ComputeSRVTree: closed-loop residuals, pixel / block-energy
//                   thresholds, quantisation, reconstruction     [srv_kernel]
//   per (location, channel): BFS-ordered blocks -> mode, header,
//                   BISE payload                                 [record_size_kernel, record_pack_kernel]
//   stream = header : top RKVs (raw int16) : offsets : records   [host]
// Every rule is integer arithmetic (the filter is the binomial approximation
// of the Gaussian weighting, normalised by a power of two), so the stream is
// byte-identical to any other encoder that follows the same rules.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "rlfc_device.cuh"
#include "rlfc_internal.h"

namespace rlfc {
namespace {

// ranges of the 28 modes, ascending
__constant__ uint32_t c_rangeN[kNumModes] = {1,  2,  3,  4,   5,   6,   8,   10,  12,  16,  20,  24,  32,  40,
                                             48, 64, 80, 96, 128, 160, 192, 256, 320, 384, 512, 640, 768, 1024};
__constant__ uint32_t c_modes[kNumModes] = RLFC_MODE_TABLE_INIT;

#include "ks_device.cuh"

// Four pixels of a padded row per thread; blockIdx.y = view.  What bounds it:
// DRAM (3 B read and 6 B written per pixel): 81 views of 512 x 512
// take 39 us (80 with a pixel per thread and 64-bit index divisions).
__global__ void __launch_bounds__(256) ycocg_pad_kernel(const uint8_t *rgb, int16_t *x0, uint32_t W, uint32_t H, uint32_t Wp,
                                                        uint32_t Hp, uint32_t words)
{
    const uint32_t quads = Wp / 4, i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= quads * Hp)
        return;
    const uint32_t view = blockIdx.y, y = i / quads, x = 4 * (i - y * quads);
    const size_t plane = (size_t)Wp * Hp;
    const uint8_t *row = rgb + ((size_t)view * H + min(y, H - 1)) * W * 3;
    uint8_t px[12];
    if (words && x + 4 <= W) {
        // the row starts on a 4-byte boundary (words), so x does too
        const uint32_t *p = reinterpret_cast<const uint32_t *>(row + 3 * x);
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const uint32_t v = __ldg(p + k);
#pragma unroll
            for (int b = 0; b < 4; b++)
                px[4 * k + b] = (uint8_t)(v >> (8 * b));
        }
    } else {
#pragma unroll
        for (uint32_t k = 0; k < 4; k++) {
            const uint8_t *p = row + 3 * min(x + k, W - 1);
            px[3 * k] = p[0];
            px[3 * k + 1] = p[1];
            px[3 * k + 2] = p[2];
        }
    }
    int16_t v[3][4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int R = px[3 * k], G = px[3 * k + 1], B = px[3 * k + 2];
        const int co = R - B;
        const int t = B + (co >> 1);
        const int cg = G - t;
        v[0][k] = (int16_t)(t + (cg >> 1));
        v[1][k] = (int16_t)co;
        v[2][k] = (int16_t)cg;
    }
    int16_t *dst = x0 + (size_t)view * 3 * plane + (size_t)y * Wp + x;
#pragma unroll
    for (int c = 0; c < 3; c++)
        *reinterpret_cast<short4 *>(dst + c * plane) = make_short4(v[c][0], v[c][1], v[c][2], v[c][3]);
}

// One parent node per blockIdx.y: floor((sum w X + 2^(s-1)) / 2^s) over its
// members, with members/weights/shift given per parent; four values per
// thread.  The sums are 32-bit while 2^s times the largest value fits (Acc).
// What bounds it: DRAM, every child read once.
template <typename Acc>
__global__ void __launch_bounds__(256) filter_kernel(const int16_t *child, int16_t *parent, const uint32_t *member_start,
                                                     const uint32_t *member_idx, const int64_t *member_w, const uint32_t *shift,
                                                     size_t npix)
{
    const uint32_t p = blockIdx.y;
    const uint32_t m0 = member_start[p], m1 = member_start[p + 1];
    const uint32_t s = shift[p];
    const Acc half = s > 0 ? (Acc)1 << (s - 1) : 0;
    for (size_t i = 4 * (blockIdx.x * (size_t)blockDim.x + threadIdx.x); i < npix; i += 4 * (size_t)gridDim.x * blockDim.x) {
        Acc acc[4] = {half, half, half, half};
#pragma unroll 4
        for (uint32_t m = m0; m < m1; m++) {
            const short4 v = __ldg(reinterpret_cast<const short4 *>(child + (size_t)member_idx[m] * npix + i));
            const Acc w = (Acc)member_w[m];
            acc[0] += w * v.x;
            acc[1] += w * v.y;
            acc[2] += w * v.z;
            acc[3] += w * v.w;
        }
        *reinterpret_cast<short4 *>(parent + (size_t)p * npix + i) =
            make_short4((short)(acc[0] >> s), (short)(acc[1] >> s), (short)(acc[2] >> s), (short)(acc[3] >> s));
    }
}

constexpr uint8_t kAbsent = 0xFF;

// The smallest mode whose range holds `span` values (the last one when none
// does): the ranges above 4 are 5, 6 and 8 times 2^(e - 2) for each power of
// two 2^e.
__device__ __forceinline__ uint32_t smallest_mode(int span)
{
    const int x = span - 1;
    if (x < 3)
        return (uint32_t)x;
    const int e = 31 - __clz(x);
    const int k = e < 2 ? 3 * e : (x < (5 << (e - 2)) ? 3 * e - 2 : (x < (6 << (e - 2)) ? 3 * e - 1 : 3 * e));
    return (uint32_t)min(k, kNumModes - 1);
}

struct SrvArgs {
    int16_t *child;           // RKVs of level l-1; replaced by the quantised SRV
    const int16_t *rec_par;   // reconstruction of level l
    int16_t *rec_child;       // reconstruction of level l-1 (null for level 0)
    const uint32_t *parent;   // parent index of each child node
    uint8_t *kmode;           // [child node][3][nloc]: k | s << 5 of a stored block, kAbsent where none is stored
    const uint8_t *leaf_modes;   // level 0 only, may be null: given k | s << 5, 0xFF = search
    int16_t *leaf_resid;      // level 0 only, may be null: residuals after the pixel threshold
    uint8_t *leaf_label;      // level 0 only, may be null: search result, 0xFF = not kept
    int *error;
    uint32_t nlx, nloc, Wp, Hp;
    int32_t tau_p, tau_b;
    uint32_t q;
    uint32_t mode_space, lam_q8;
    int32_t tau_err;
};

// (shift, mode) search: ks_device.cuh, included above with these tables in scope

// Eq. 3 with the thresholds and quantisation of Section 3.2, one thread per
// block; blockIdx.y = (child node, channel).  Block rows are 8-byte accesses,
// neighbouring threads on neighbouring blocks.  What bounds it: DRAM (the
// children read and their quantised residuals written).  kAid: with the (shift,
// mode) search or its labels, which need twice the registers.
template <bool kAid>
__global__ void __launch_bounds__(256) srv_kernel(const SrvArgs a)
{
    const size_t plane = (size_t)a.Wp * a.Hp;
    const uint32_t node = blockIdx.y / 3, c = blockIdx.y - 3 * node;
    const uint32_t par = a.parent[node];
    for (uint32_t loc = blockIdx.x * blockDim.x + threadIdx.x; loc < a.nloc; loc += gridDim.x * blockDim.x) {
        const uint32_t by = loc / a.nlx, bx = loc - by * a.nlx;
        const size_t at = (size_t)by * 4 * a.Wp + 4 * bx;
        int16_t *xc = a.child + ((size_t)node * 3 + c) * plane + at;
        const int16_t *xp = a.rec_par + ((size_t)par * 3 + c) * plane + at;
        int r[kVals], p[kVals];
        int energy = 0;
#pragma unroll
        for (int y = 0; y < 4; y++) {
            const short4 vc = *reinterpret_cast<const short4 *>(xc + (size_t)y * a.Wp);
            const short4 vp = *reinterpret_cast<const short4 *>(xp + (size_t)y * a.Wp);
            const int cc[4] = {vc.x, vc.y, vc.z, vc.w}, pp[4] = {vp.x, vp.y, vp.z, vp.w};
#pragma unroll
            for (int x = 0; x < 4; x++) {
                int v = cc[x] - pp[x];
                if (abs(v) < a.tau_p)
                    v = 0;
                r[4 * y + x] = v;
                p[4 * y + x] = pp[x];
                energy += abs(v);
            }
        }
        bool keep = energy > 0 && energy >= a.tau_b;
        const size_t bi = ((size_t)node * 3 + c) * a.nloc + loc;
        if (a.leaf_resid) {
#pragma unroll
            for (int k = 0; k < kVals; k++)
                a.leaf_resid[bi * kVals + k] = (int16_t)r[k];
        }
        if (kAid && a.leaf_label) {
            uint32_t lk = 0, ls = 0;
            a.leaf_label[bi] = keep && ks_search(r, a.q, a.tau_err, a.lam_q8, lk, ls) ? (uint8_t)(lk | ls << 5)
                                                                                     : (uint8_t)0xFF;
        }
        uint32_t ks_k = 0, ks_s = 0;
        if (kAid && keep && a.mode_space) {
            bool have = false;
            if (a.leaf_modes && a.leaf_modes[bi] != 0xFF) {
                // a given mode is used when it is a candidate
                const uint32_t gk = a.leaf_modes[bi] & 31u, gs = a.leaf_modes[bi] >> 5;
                long long cost;
                if (ks_cost(r, a.q, gs, gk, a.tau_err, a.lam_q8, cost)) {
                    ks_k = gk;
                    ks_s = gs;
                    have = true;
                }
            }
            if (!have && !ks_search(r, a.q, a.tau_err, a.lam_q8, ks_k, ks_s))
                atomicExch(a.error, 3);
        }
        const uint32_t t = a.q + ks_s;
        const int half = t > 0 ? 1 << (t - 1) : 0;
        bool nonzero = false;
        int mn = 0, mx = 0;
#pragma unroll
        for (int k = 0; k < kVals; k++) {
            const int qm = (abs(r[k]) + half) >> t;
            r[k] = keep ? (r[k] < 0 ? -qm : qm) : 0;
            nonzero |= r[k] != 0;
            mn = k == 0 ? r[k] : min(mn, r[k]);
            mx = k == 0 ? r[k] : max(mx, r[k]);
        }
        keep = keep && nonzero;
        if (keep && (!kAid || !a.mode_space)) {
            // the plain method: the smallest range that holds the span
            ks_k = smallest_mode(mx - mn + 1);
        }
        if (keep && ((int)c_rangeN[ks_k] < mx - mn + 1 || mn < -1024 || mn > 1023))
            atomicExch(a.error, 1);
        a.kmode[bi] = keep ? (uint8_t)(ks_k | ks_s << 5) : kAbsent;
        int16_t *rc = a.rec_child ? a.rec_child + ((size_t)node * 3 + c) * plane + at : nullptr;
#pragma unroll
        for (int y = 0; y < 4; y++) {
            short q[4], o[4];
#pragma unroll
            for (int x = 0; x < 4; x++) {
                const int qv = keep ? r[4 * y + x] : 0;
                q[x] = (short)qv;
                o[x] = (short)(p[4 * y + x] + qv * (1 << t));
            }
            if (rc)
                *reinterpret_cast<short4 *>(rc + (size_t)y * a.Wp) = make_short4(o[0], o[1], o[2], o[3]);
            *reinterpret_cast<short4 *>(xc + (size_t)y * a.Wp) = make_short4(q[0], q[1], q[2], q[3]);
        }
    }
}

struct RecArgs {
    const int16_t *const *srv;   // per level < L-1: quantised SRV images
    const uint8_t *const *kmode;  // per level < L-1: k | s << 5 of each stored block, kAbsent for the others
    const uint32_t *bfs_level;   // [S]
    const uint32_t *bfs_node;    // [S]
    uint32_t S, MW, nlx, nloc, Wp, Hp;
    uint32_t *words;             // record_size: per-record word count; record_pack: the records, zeroed
    const uint32_t *offsets;     // record_pack only
    int *error;
};

// Word count of every record; a thread per record, neighbouring threads on
// neighbouring locations of one channel (blockIdx.y).
__global__ void __launch_bounds__(128) record_size_kernel(const RecArgs a)
{
    const uint32_t loc = blockIdx.x * blockDim.x + threadIdx.x, c = blockIdx.y;
    if (loc >= a.nloc)
        return;
    uint32_t bits = 32 * a.MW;
#pragma unroll 8
    for (uint32_t pos = 0; pos < a.S; pos++) {
        const uint32_t km = a.kmode[a.bfs_level[pos]][((size_t)a.bfs_node[pos] * 3 + c) * a.nloc + loc];
        bits += km == kAbsent ? 0u : kHdrBits + mode_bits(c_modes[km & 31u]);
    }
    a.words[3 * (size_t)loc + c] = (bits + 31) / 32;
}

// ORs the low `width` (up to 32) bits of v into the bit string at `pos`; the
// words are shared with other lanes.
__device__ __forceinline__ void or_bits(uint32_t *w, uint32_t pos, uint32_t v, uint32_t width)
{
    const uint32_t sh = pos & 31u;
    atomicOr(w + (pos >> 5), v << sh);
    if (sh + width > 32)
        atomicOr(w + (pos >> 5) + 1, v >> (32 - sh));
}

// Writes a payload from bit `pos`: words that it fills are stored, the first
// and last, shared with its neighbours, ORed.
struct BitWriter {
    uint32_t *out;
    uint64_t acc;
    uint32_t n;
    bool shared;
    __device__ __forceinline__ BitWriter(uint32_t *w, uint32_t pos)
        : out(w + (pos >> 5)), acc(0), n(pos & 31u), shared((pos & 31u) != 0)
    {
    }
    __device__ __forceinline__ void put(uint32_t v, uint32_t width)
    {
        acc |= (uint64_t)v << n;
        n += width;
        if (n >= 32) {
            if (shared)
                atomicOr(out, (uint32_t)acc);
            else
                *out = (uint32_t)acc;
            shared = false;
            out++;
            acc >>= 32;
            n -= 32;
        }
    }
    __device__ __forceinline__ void flush()
    {
        if (n > 0 && (uint32_t)acc != 0)
            atomicOr(out, (uint32_t)acc);
    }
};

constexpr int kPackWarps = 8;

// A warp per record.  The nodes are taken 32 at a time: a ballot makes the mask
// word, a scan of the closed-form lengths every payload's offset; the stored
// blocks are listed densely and written one lane each, 32 at a time.
// What bounds it: instruction issue (the 2-byte accesses and the bit writer of
// the form it replaces, one thread per record over two passes, took 0.29 ms
// for 9 x 9 views of 512 x 512; this takes 0.085).
__global__ void __launch_bounds__(32 * kPackWarps) record_pack_kernel(const RecArgs a)
{
    __shared__ uint2 s_list[kPackWarps][64];   // node | k, s << 16; payload offset
    const int lane = threadIdx.x & 31;
    uint2 *list = s_list[threadIdx.x >> 5];
    const uint32_t rec_i = blockIdx.x * kPackWarps + (threadIdx.x >> 5);
    if (rec_i >= 3 * a.nloc)
        return;
    const uint32_t loc = rec_i / 3, c = rec_i - 3 * loc;
    uint32_t *rec = a.words + a.offsets[rec_i];
    const uint32_t nwords = a.offsets[rec_i + 1] - a.offsets[rec_i];
    const size_t plane = (size_t)a.Wp * a.Hp;
    const uint32_t by = loc / a.nlx, bx = loc - by * a.nlx;
    const size_t at = c * plane + (size_t)by * 4 * a.Wp + 4 * bx;
    const auto mode_of = [&](uint32_t pos) -> uint32_t {
        return pos < a.S ? a.kmode[a.bfs_level[pos]][((size_t)a.bfs_node[pos] * 3 + c) * a.nloc + loc] : (uint32_t)kAbsent;
    };
    // mask words, and the number of stored blocks
    uint32_t P = 0;
    for (uint32_t m = 0; m < a.MW; m++) {
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, mode_of(32 * m + lane) != kAbsent);
        if (lane == 0)
            rec[m] = bal;
        P += __popc(bal);
    }
    const uint32_t hdr0 = 32 * a.MW;
    uint32_t run = hdr0 + kHdrBits * P, rank0 = 0, have = 0;
    // the first n listed blocks, a lane each: header and payload
    const auto write = [&](uint32_t n) {
        __syncwarp();
        if ((uint32_t)lane < n) {
            const uint2 e = list[lane];
            const uint32_t pos = e.x & 0xFFFFu, km = e.x >> 16;
            const int16_t *img = a.srv[a.bfs_level[pos]] + (size_t)a.bfs_node[pos] * 3 * plane + at;
            int v[kVals];
#pragma unroll
            for (int y = 0; y < 4; y++) {
                const short4 q = __ldg(reinterpret_cast<const short4 *>(img + (size_t)y * a.Wp));
                v[4 * y] = q.x;
                v[4 * y + 1] = q.y;
                v[4 * y + 2] = q.z;
                v[4 * y + 3] = q.w;
            }
            int mn = v[0];
#pragma unroll
            for (int k = 1; k < kVals; k++)
                mn = min(mn, v[k]);
            // header: mode 5 | shift 2 | min 11
            or_bits(rec, hdr0 + kHdrBits * (rank0 + lane), (km & 127u) | (((uint32_t)mn & 0x7FFu) << 7), kHdrBits);
            // payload: digit words, then the low bits
            const uint32_t m = c_modes[km & 31u];
            const uint32_t b = mode_b(m), kind = mode_kind(m);
            uint32_t u[kVals];
#pragma unroll
            for (int k = 0; k < kVals; k++)
                u[k] = (uint32_t)(v[k] - mn);
            BitWriter bw(rec, e.y);
            if (kind == 1) {
#pragma unroll
                for (int g = 0; g < 4; g++) {
                    uint32_t word = 0, scale = 1;
#pragma unroll
                    for (int d = 0; d < 5; d++) {
                        const int k = 5 * g + d;
                        if (k < kVals) {
                            word += (u[k] >> b) * scale;
                            scale *= 3;
                        }
                    }
                    bw.put(word, g < 3 ? 8u : 2u);
                }
            } else if (kind == 2) {
#pragma unroll
                for (int g = 0; g < 6; g++) {
                    uint32_t word = 0, scale = 1;
#pragma unroll
                    for (int d = 0; d < 3; d++) {
                        const int k = 3 * g + d;
                        if (k < kVals) {
                            word += (u[k] >> b) * scale;
                            scale *= 5;
                        }
                    }
                    bw.put(word, g < 5 ? 7u : 3u);
                }
            }
            if (b != 0) {
                // two low parts at a time (20 bits at most)
#pragma unroll
                for (int k = 0; k < kVals; k += 2)
                    bw.put((u[k] & ((1u << b) - 1u)) | ((u[k + 1] & ((1u << b) - 1u)) << b), 2 * b);
            }
            bw.flush();
        }
        __syncwarp();
        rank0 += n;
    };
    for (uint32_t p0 = 0; p0 < a.S; p0 += 32) {
        const uint32_t km = mode_of(p0 + lane);
        const bool stored = km != kAbsent;
        const unsigned bal = __ballot_sync(0xFFFFFFFFu, stored);
        const uint32_t len = stored ? mode_bits(c_modes[km & 31u]) : 0u;
        uint32_t incl = len;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
            if (lane >= d)
                incl += y;
        }
        if (stored)
            list[have + __popc(bal & ((1u << lane) - 1u))] = make_uint2((p0 + lane) | (km << 16), run + incl - len);
        have += __popc(bal);
        run += __shfl_sync(0xFFFFFFFFu, incl, 31);
        if (have >= 32) {
            write(32);
            have -= 32;
            const uint2 e = list[32 + lane];
            __syncwarp();
            list[lane] = e;
            __syncwarp();
        }
    }
    write(have);
    if (lane == 0 && (run + 31) / 32 != nwords)
        atomicExch(a.error, 2);
}

int tile_count(uint32_t G, uint32_t c) { return (int)((G + c - 1) / c); }

struct DevBuf {
    std::vector<void *> ptrs;
    uint8_t *arena = nullptr;   // when set, buffers are carved from this caller-provided block
    size_t arena_size = 0, arena_used = 0;
    ~DevBuf()
    {
        for (void *p : ptrs)
            cudaFree(p);
    }
    template <typename T>
    cudaError_t alloc(T **p, size_t count)
    {
        if (arena) {
            const size_t at = (arena_used + 255) & ~size_t(255);
            const size_t bytes = count * sizeof(T) + 16;
            if (at + bytes > arena_size)
                return cudaErrorMemoryAllocation;
            *p = reinterpret_cast<T *>(arena + at);
            arena_used = at + bytes;
            return cudaSuccess;
        }
        return alloc_own(p, count);
    }
    // a buffer of its own
    template <typename T>
    cudaError_t alloc_own(T **p, size_t count)
    {
        cudaError_t e = cudaMalloc((void **)p, count * sizeof(T) + 16);
        if (e == cudaSuccess)
            ptrs.push_back((void *)*p);
        return e;
    }
};

void put32(std::vector<uint8_t> &b, size_t at, uint32_t v)
{
    b[at] = (uint8_t)v;
    b[at + 1] = (uint8_t)(v >> 8);
    b[at + 2] = (uint8_t)(v >> 16);
    b[at + 3] = (uint8_t)(v >> 24);
}

size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

}  // namespace

namespace {

// Upper bounds of the device scratch that encode_gpu carves for these
// parameters (every buffer rounded up to 256 bytes): everything but the
// records, and the records at their largest possible size; false when the
// parameters are invalid.
bool scratch_bounds(const rlfc_enc_params *p, uint64_t &fixed, uint64_t &records)
{
    if (!p || p->B != 4 || p->U < 1 || p->V < 1 || (uint64_t)p->U * p->V > 16383 || p->W < 1 || p->H < 1 ||
        p->W > 65536 || p->H > 65536 || p->L < 2 || p->L > (uint32_t)kMaxLevels)
        return false;
    const uint32_t L = p->L;
    std::vector<uint64_t> cnt(L);
    uint64_t Gu = p->U, Gv = p->V;
    cnt[0] = Gu * Gv;
    for (uint32_t l = 1; l < L; l++) {
        if (p->c[l] < 1)
            return false;
        Gu = (Gu + p->c[l] - 1) / p->c[l];
        Gv = (Gv + p->c[l] - 1) / p->c[l];
        cnt[l] = Gu * Gv;
    }
    const uint64_t Wp = (p->W + 3) / 4 * 4, Hp = (p->H + 3) / 4 * 4, nloc = (Wp / 4) * (Hp / 4);
    const uint64_t npix = 3 * Wp * Hp;
    uint64_t S = 0;
    for (uint32_t l = 0; l + 1 < L; l++)
        S += cnt[l];
    uint64_t total = 0;
    auto add = [&](uint64_t bytes) { total += ((bytes + 16) + 255) / 256 * 256; };
    for (uint32_t l = 0; l < L; l++) {
        add(2 * npix * cnt[l]);
        if (l >= 1 && l + 1 < L)
            add(2 * npix * cnt[l]);
        if (l + 1 < L)
            add(cnt[l] * 3 * nloc);
    }
    add(sizeof(int));
    for (uint32_t l = 1; l < L; l++) {
        add(4 * (cnt[l] + 1));
        add(4 * cnt[l - 1]);
        add(4 * cnt[l]);
        add(8 * cnt[l - 1]);
        add(4 * cnt[l - 1]);
    }
    add(4 * S);
    add(4 * S);
    add(4 * 3 * nloc);
    add(4 * (3 * nloc + 1));
    add(sizeof(void *) * L);
    add(sizeof(void *) * L);
    const uint64_t MW = (S + 31) / 32;
    fixed = total;
    total = 0;
    add(4 * (3 * nloc * (MW + (S * (kHdrBits + 160) + 31) / 32) + 1));
    records = total;
    return true;
}

}  // namespace

size_t encode_scratch_bound(const rlfc_enc_params *p)
{
    uint64_t fixed = 0, records = 0;
    return scratch_bounds(p, fixed, records) ? (size_t)(fixed + records) : 0;
}

int encode_gpu(const rlfc_enc_params *p, const uint8_t *d_rgb, cudaStream_t st, std::vector<uint8_t> &out,
               uint8_t *arena, size_t arena_size, const uint8_t *d_leaf_modes, int16_t *d_leaf_resid,
               uint8_t *d_leaf_label)
{
    if (p->B != 4) {
        set_error("the GPU encoder writes 4x4 blocks only");
        return RLFC_E_UNSUPPORTED;
    }
    if (p->U < 1 || p->V < 1 || (uint64_t)p->U * p->V > 16383 || p->W < 1 || p->H < 1 || p->W > 65536 ||
        p->H > 65536 || p->L < 2 || p->L > (uint32_t)kMaxLevels || p->tau_p < 0 || p->tau_b < 0 || p->q > 7 ||
        p->mode_space > 1 || p->tau_err < 0) {
        set_error("encoder parameters out of range");
        return RLFC_E_INVALID_ARG;
    }
    const uint32_t L = p->L;
    for (uint32_t l = 1; l < L; l++)
        if (p->c[l] < 1) {
            set_error("cluster side must be >= 1");
            return RLFC_E_INVALID_ARG;
        }
    // tree shape (Eq. 1 reading): uniform tiling per level
    std::vector<uint32_t> Gu(L), Gv(L), cnt(L);
    Gu[0] = p->U;
    Gv[0] = p->V;
    for (uint32_t l = 1; l < L; l++) {
        Gu[l] = tile_count(Gu[l - 1], p->c[l]);
        Gv[l] = tile_count(Gv[l - 1], p->c[l]);
    }
    for (uint32_t l = 0; l < L; l++)
        cnt[l] = Gu[l] * Gv[l];
    std::vector<std::vector<uint32_t>> parent(L);
    // tile a of k covering G nodes: [floor(aG/k), floor((a+1)G/k))
    auto tile_of = [](uint32_t x, uint32_t G, uint32_t k) {
        uint32_t a = 0;
        while (!((uint64_t)(a + 1) * G / k > x))
            a++;
        return a;
    };
    for (uint32_t l = 0; l + 1 < L; l++) {
        parent[l].resize(cnt[l]);
        for (uint32_t y = 0; y < Gv[l]; y++)
            for (uint32_t x = 0; x < Gu[l]; x++)
                parent[l][y * Gu[l] + x] = tile_of(y, Gv[l], Gv[l + 1]) * Gu[l + 1] + tile_of(x, Gu[l], Gu[l + 1]);
    }
    Tables tab;
    if (build_tables(L, cnt, parent, tab) != 0 || tab.S >= 16384) {
        set_error("tree too large");
        return RLFC_E_RANGE;
    }
    const uint32_t W = p->W, H = p->H, Wp = (W + 3) / 4 * 4, Hp = (H + 3) / 4 * 4;
    const uint32_t nlx = Wp / 4, nly = Hp / 4, nloc = nlx * nly;
    const size_t plane = (size_t)Wp * Hp, npix = 3 * plane;

    DevBuf buf;
    buf.arena = arena;
    buf.arena_size = arena_size;
    cudaError_t e;
    if (!arena) {
        // one allocation for everything but the records (a dozen of them, and
        // as many frees, took 0.25 ms)
        uint64_t fixed = 0, records = 0;
        scratch_bounds(p, fixed, records);
        if ((e = buf.alloc_own(&buf.arena, fixed)) != cudaSuccess)
            return cuda_fail(e, "encoder allocation");
        buf.arena_size = fixed;
    }
    std::vector<int16_t *> img(L, nullptr), rec(L, nullptr);
    std::vector<uint8_t *> kmode(L, nullptr);
    for (uint32_t l = 0; l < L; l++) {
        if ((e = buf.alloc(&img[l], npix * cnt[l])) != cudaSuccess)
            return cuda_fail(e, "encoder allocation");
        if (l >= 1 && l + 1 < L && (e = buf.alloc(&rec[l], npix * cnt[l])) != cudaSuccess)
            return cuda_fail(e, "encoder allocation");
        if (l + 1 < L && (e = buf.alloc(&kmode[l], (size_t)cnt[l] * 3 * nloc)) != cudaSuccess)
            return cuda_fail(e, "encoder allocation");
    }
    int *d_err;
    if ((e = buf.alloc(&d_err, 1)) != cudaSuccess)
        return cuda_fail(e, "encoder allocation");
    cudaMemsetAsync(d_err, 0, sizeof(int), st);
    rec[L - 1] = img[L - 1];
    const int threads = 256;
    const unsigned quad_blocks = (unsigned)((plane / 4 + threads - 1) / threads);
    const uint32_t words_in = ((uintptr_t)d_rgb & 3u) == 0 && W % 4 == 0;

    { rlfc::TraceScope trace_("ycocg_pad_kernel", st); ycocg_pad_kernel<<<dim3(quad_blocks, cnt[0]), threads, 0, st>>>(d_rgb, img[0], W, H, Wp, Hp, words_in); }

    // bottom-up filter
    for (uint32_t l = 1; l < L; l++) {
        std::vector<uint32_t> mstart(1, 0), midx, shift;
        std::vector<int64_t> mw;
        const uint32_t ku = Gu[l], kv = Gv[l];
        for (uint32_t b = 0; b < kv; b++)
            for (uint32_t a2 = 0; a2 < ku; a2++) {
                const uint32_t x0 = (uint64_t)a2 * Gu[l - 1] / ku, x1 = (uint64_t)(a2 + 1) * Gu[l - 1] / ku;
                const uint32_t y0 = (uint64_t)b * Gv[l - 1] / kv, y1 = (uint64_t)(b + 1) * Gv[l - 1] / kv;
                const uint32_t mu = x1 - x0, mv = y1 - y0;
                // Pascal's triangle rows mu-1 and mv-1
                std::vector<int64_t> ru(mu, 1), rv(mv, 1);
                for (uint32_t i = 1; i + 1 < mu; i++)
                    ru[i] = ru[i - 1] * (mu - i) / i;
                for (uint32_t i = 1; i + 1 < mv; i++)
                    rv[i] = rv[i - 1] * (mv - i) / i;
                for (uint32_t y = y0; y < y1; y++)
                    for (uint32_t x = x0; x < x1; x++) {
                        midx.push_back(y * Gu[l - 1] + x);
                        mw.push_back(ru[x - x0] * rv[y - y0]);
                    }
                mstart.push_back((uint32_t)midx.size());
                shift.push_back((mu - 1) + (mv - 1));
                if ((mu - 1) + (mv - 1) > 40) {
                    set_error("cluster too large");
                    return RLFC_E_RANGE;
                }
            }
        uint32_t *d_ms, *d_mi, *d_sh;
        int64_t *d_mw;
        if ((e = buf.alloc(&d_ms, mstart.size())) != cudaSuccess || (e = buf.alloc(&d_mi, midx.size())) != cudaSuccess ||
            (e = buf.alloc(&d_sh, shift.size())) != cudaSuccess || (e = buf.alloc(&d_mw, mw.size())) != cudaSuccess)
            return cuda_fail(e, "encoder allocation");
        cudaMemcpyAsync(d_ms, mstart.data(), 4 * mstart.size(), cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(d_mi, midx.data(), 4 * midx.size(), cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(d_sh, shift.data(), 4 * shift.size(), cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(d_mw, mw.data(), 8 * mw.size(), cudaMemcpyHostToDevice, st);
        dim3 grid((unsigned)std::min<size_t>((npix / 4 + threads - 1) / threads, 4096), cnt[l]);
        // values stay below 2^10, so 32-bit sums hold weights up to 2^20
        const bool narrow = *std::max_element(shift.begin(), shift.end()) <= 20;
        auto filter = narrow ? filter_kernel<int32_t> : filter_kernel<int64_t>;
        { rlfc::TraceScope trace_("filter_kernel", st); filter<<<grid, threads, 0, st>>>(img[l - 1], img[l], d_ms, d_mi, d_mw, d_sh, npix); }
        // keep the host vectors alive until the copies are done
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess)
            return cuda_fail(e, "encoder filter");
    }

    // top-down residuals (closed loop)
    for (uint32_t l = L - 1; l >= 1; l--) {
        uint32_t *d_par;
        if ((e = buf.alloc(&d_par, cnt[l - 1])) != cudaSuccess)
            return cuda_fail(e, "encoder allocation");
        cudaMemcpyAsync(d_par, parent[l - 1].data(), 4ull * cnt[l - 1], cudaMemcpyHostToDevice, st);
        SrvArgs s;
        s.child = img[l - 1];
        s.rec_par = rec[l];
        s.rec_child = (l - 1 >= 1) ? rec[l - 1] : nullptr;
        s.parent = d_par;
        s.kmode = kmode[l - 1];
        s.leaf_modes = l == 1 ? d_leaf_modes : nullptr;
        s.leaf_resid = l == 1 ? d_leaf_resid : nullptr;
        s.leaf_label = l == 1 ? d_leaf_label : nullptr;
        s.error = d_err;
        s.mode_space = p->mode_space;
        s.lam_q8 = p->lam_q8;
        s.tau_err = p->tau_err;
        s.nlx = nlx;
        s.nloc = nloc;
        s.Wp = Wp;
        s.Hp = Hp;
        s.tau_p = p->tau_p;
        s.tau_b = p->tau_b;
        s.q = p->q;
        auto srv = s.mode_space || s.leaf_label ? srv_kernel<true> : srv_kernel<false>;
        { rlfc::TraceScope trace_("srv_kernel", st); srv<<<dim3(std::min<unsigned>((nloc + threads - 1) / threads, 4096), 3 * cnt[l - 1]), threads, 0, st>>>(s); }
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess)
            return cuda_fail(e, "encoder residuals");
    }

    // BFS tables for the record kernels
    std::vector<uint32_t> bfs_level(tab.S), bfs_node(tab.S);
    for (uint32_t pos = 0; pos < tab.S; pos++)
        bfs_level[pos] = node_level(tab.node_info[pos]);
    // node index of every BFS position: every node is an ancestor of some view
    for (uint32_t v = 0; v < cnt[0]; v++) {
        uint32_t a2 = v;
        for (uint32_t l = 0; l + 1 < L; l++) {
            bfs_node[tab.view_anc[(size_t)v * kMaxLevels + l]] = a2;
            a2 = parent[l][a2];
        }
    }
    const uint32_t S = tab.S, MW = (S + 31) / 32;
    uint32_t *d_bl, *d_bn, *d_words_n, *d_off, *d_rec;
    const int16_t **d_srv;
    const uint8_t **d_km;
    if ((e = buf.alloc(&d_bl, S)) != cudaSuccess || (e = buf.alloc(&d_bn, S)) != cudaSuccess ||
        (e = buf.alloc(&d_words_n, 3ull * nloc)) != cudaSuccess || (e = buf.alloc(&d_off, 3ull * nloc + 1)) != cudaSuccess ||
        (e = buf.alloc(&d_srv, L)) != cudaSuccess || (e = buf.alloc(&d_km, L)) != cudaSuccess)
        return cuda_fail(e, "encoder allocation");
    std::vector<const int16_t *> srv_ptrs(img.begin(), img.end());
    std::vector<const uint8_t *> km_ptrs(kmode.begin(), kmode.end());
    cudaMemcpyAsync(d_bl, bfs_level.data(), 4ull * S, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(d_bn, bfs_node.data(), 4ull * S, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(d_srv, srv_ptrs.data(), sizeof(void *) * L, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(d_km, km_ptrs.data(), sizeof(void *) * L, cudaMemcpyHostToDevice, st);
    RecArgs ra;
    ra.srv = d_srv;
    ra.kmode = d_km;
    ra.bfs_level = d_bl;
    ra.bfs_node = d_bn;
    ra.S = S;
    ra.MW = MW;
    ra.nlx = nlx;
    ra.nloc = nloc;
    ra.Wp = Wp;
    ra.Hp = Hp;
    ra.words = d_words_n;
    ra.offsets = nullptr;
    ra.error = d_err;
    { rlfc::TraceScope trace_("record_size_kernel", st); record_size_kernel<<<dim3((nloc + 127) / 128, 3), 128, 0, st>>>(ra); }
    std::vector<uint32_t> words(3ull * nloc), offsets(3ull * nloc + 1);
    int h_err = 0;
    cudaMemcpyAsync(words.data(), d_words_n, 4ull * 3 * nloc, cudaMemcpyDeviceToHost, st);
    cudaMemcpyAsync(&h_err, d_err, sizeof(int), cudaMemcpyDeviceToHost, st);
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess)
        return cuda_fail(e, "encoder record sizes");
    if (h_err) {
        set_error(h_err == 3 ? "a residual block has no (mode, shift) candidate"
                             : "a residual block's range does not fit the 28 BISE modes");
        return RLFC_E_RANGE;
    }
    uint64_t total = 0;
    for (size_t i = 0; i < words.size(); i++) {
        offsets[i] = (uint32_t)total;
        total += words[i];
    }
    offsets.back() = (uint32_t)total;
    if (total >= (1ull << 32) - 16) {
        set_error("stream larger than 16 GiB");
        return RLFC_E_RANGE;
    }
    if ((e = arena ? buf.alloc(&d_rec, total + 1) : buf.alloc_own(&d_rec, total + 1)) != cudaSuccess)
        return cuda_fail(e, "encoder allocation");
    cudaMemcpyAsync(d_off, offsets.data(), 4ull * offsets.size(), cudaMemcpyHostToDevice, st);
    cudaMemsetAsync(d_rec, 0, 4ull * total, st);   // shared words are ORed
    ra.words = d_rec;
    ra.offsets = d_off;
    { rlfc::TraceScope trace_("record_pack_kernel", st); record_pack_kernel<<<(3 * nloc + kPackWarps - 1) / kPackWarps, 32 * kPackWarps, 0, st>>>(ra); }

    // assemble the stream
    const size_t hdr_end = 64 + 8ull * L + 4ull * S;
    const size_t off_top = align16(hdr_end);
    const size_t top_bytes = 2ull * cnt[L - 1] * npix;
    const size_t off_offsets = align16(off_top + top_bytes);
    const size_t off_records = align16(off_offsets + 4ull * offsets.size());
    out.assign(off_records + 4ull * total, 0);
    const uint32_t hdr[15] = {0x43464C52u, 1u, p->U, p->V, W, H, 4u, L, p->q, cnt[L - 1], S,
                              (uint32_t)off_top, (uint32_t)off_offsets, (uint32_t)off_records, (uint32_t)total};
    for (int i = 0; i < 15; i++)
        put32(out, 4 * i, hdr[i]);
    size_t at = 64;
    for (uint32_t l = 0; l < L; l++, at += 8) {
        put32(out, at, Gu[l]);
        put32(out, at + 4, Gv[l]);
    }
    for (uint32_t l = 0; l + 1 < L; l++)
        for (uint32_t i = 0; i < cnt[l]; i++, at += 4)
            put32(out, at, parent[l][i]);
    cudaMemcpyAsync(out.data() + off_top, img[L - 1], top_bytes, cudaMemcpyDeviceToHost, st);
    for (size_t i = 0; i < offsets.size(); i++)
        put32(out, off_offsets + 4 * i, offsets[i]);
    cudaMemcpyAsync(out.data() + off_records, d_rec, 4ull * total, cudaMemcpyDeviceToHost, st);
    cudaMemcpyAsync(&h_err, d_err, sizeof(int), cudaMemcpyDeviceToHost, st);
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess)
        return cuda_fail(e, "encoder packing");
    if (h_err) {
        set_error("record packing disagreed with the sizing pass");
        return RLFC_E_CUDA;
    }
    return RLFC_OK;
}

}  // namespace rlfc
