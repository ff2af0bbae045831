// New-view rendering with on-demand decode (Section 3.6), for a few cameras at
// any output size: one CTA renders one tile of one camera and decodes, from
// the compressed stream, the blocks of the four neighbour views under it.
//
//  1. camera and footprints: s and t are monotone in x and y, so the tile's
//     samples in neighbour k fall in the block rectangle of its corner rays;
//  2. a thread per (block location, channel) of the rectangles' union walks
//     the location's record once, in BFS order, and tables the payload offset
//     and header of every node the neighbours need (their leaves and
//     ancestors); neighbours whose rectangles lie too far apart for one table
//     are walked one after the other;
//  3. a thread per (neighbour, block, channel) adds the top RKV block and the
//     ancestors' residuals (pair decoder), then a thread per (neighbour,
//     block, row) converts to RGB;
//  4. every thread blends its pixels' 16 samples.
// At the views' own size the stencil of a neighbour is the same for every
// pixel; the arithmetic is then that of render_windows.cu, so a view does not
// depend on the path that rendered it.
//
// What bounds it: the latency of its phases (a view has fewer tiles than the
// GPU has room for CTAs, so all run at once), hence small tiles, short walks and
// as many threads per phase as there are independent blocks.  One 512 x 512
// view of a 9 x 9 light field takes 26 us (the call 27 to 33, by the light
// field); with 64 x 16 tiles, a cell list made first and a sequential bit
// reader per block, 63 to 73 us (the call 67 to 78).
#include <cuda_runtime.h>

#include <algorithm>

#include "pair_decode.cuh"
#include "render_camera.cuh"
#include "warp_decode.cuh"

namespace rlfc {
namespace {

constexpr int kThreads = 256;
constexpr uint32_t kSmemMost = 200 * 1024;
constexpr uint32_t kSmemFourCtas = 54 * 1024;

struct Args {
    StreamView sv;
    const float *uv, *disp;
    float *out;
    uint8_t *out8;      // when set, 8-bit RGB goes here instead of out
    Grid grid;
    uint32_t out_w, out_h, tiles_x;
    int tx_log2, tx, ty;   // tile size (tx a power of two)
    uint32_t fp_blocks; // blocks of one neighbour's footprint at most
    uint32_t un_blocks; // blocks of the union that the node table holds
};

__device__ __forceinline__ float chan(uint32_t rgb, int c) { return (float)((rgb >> (8 * c)) & 255u); }

struct Rect {
    int x0, y0, nx, ny;   // in blocks; nx = 0: not used
};

extern __shared__ __align__(16) uint32_t g_smem[];

template <bool kNative>
__global__ void __launch_bounds__(kThreads, 4) render_demand_kernel(const Args a)
{
    __shared__ uint32_t s_mode[32];
    __shared__ uint16_t s_dig[256 + 128];
    __shared__ Rect s_rect[4], s_union;
    __shared__ uint32_t s_view[4], s_top[4];
    __shared__ float s_w[4];
    __shared__ Stencil s_st[4];
    __shared__ uint32_t s_need[4 * kMaxLevels];
    __shared__ int s_slot[4][kMaxLevels];
    __shared__ int s_nn;
    __shared__ uint32_t s_together;   // the union of the rectangles fits the node table
    const uint32_t L1 = a.sv.L - 1, ent_stride = 4 * L1;
    uint4 *s_rec = reinterpret_cast<uint4 *>(g_smem);                    // [4][fp_blocks][3][2] biased pairs
    // the node table, and, once every block is reconstructed, the RGB rows
    uint2 *s_ent = reinterpret_cast<uint2 *>(s_rec + 4 * a.fp_blocks * 6);   // [un_blocks][3][4 (L - 1)]
    uint4 *s_px = s_rec + 4 * a.fp_blocks * 6;                               // [4][fp_blocks][4] packed RGB rows
    const int tid = threadIdx.x, lane = tid & 31;
    const int W = (int)a.grid.W, H = (int)a.grid.H;
    const uint32_t n = blockIdx.y;
    const uint32_t x0 = (blockIdx.x % a.tiles_x) * a.tx, y0 = (blockIdx.x / a.tiles_x) * a.ty;
    const uint32_t x1 = min(x0 + a.tx, a.out_w) - 1, y1 = min(y0 + a.ty, a.out_h) - 1;
    if (tid < 32) {
        s_mode[tid] = g_tables.mode[tid];
        // ---- 1. lane k < 4: neighbour k
        CameraCell c;
        camera_cell(a.grid, a.uv, n, c);
        float w[4];
        Stencil st[4];
        camera_stencils(a.grid, c, a.disp[n], w, st);
        Rect r{0, 0, 0, 0};
#pragma unroll
        for (int k = 0; k < 4; k++)
            if (lane == k && w[k] != 0.0f) {   // a zero weight contributes nothing
                int ax, bx, ay, by;
                if (kNative) {
                    ax = min(max((int)x0 + st[k].ox, 0), W - 1);
                    bx = min(max((int)x1 + st[k].ox + 1, 0), W - 1);
                    ay = min(max((int)y0 + st[k].oy, 0), H - 1);
                    by = min(max((int)y1 + st[k].oy + 1, 0), H - 1);
                } else {
                    float f;
                    int t;
                    taps(ray_s(x0, a.grid.W, a.out_w) + st[k].sx, a.grid.W, ax, t, f);
                    taps(ray_s(x1, a.grid.W, a.out_w) + st[k].sx, a.grid.W, t, bx, f);
                    taps(ray_s(y0, a.grid.H, a.out_h) + st[k].sy, a.grid.H, ay, t, f);
                    taps(ray_s(y1, a.grid.H, a.out_h) + st[k].sy, a.grid.H, t, by, f);
                }
                r = Rect{ax / kBlock, ay / kBlock, bx / kBlock - ax / kBlock + 1, by / kBlock - ay / kBlock + 1};
            }
        const bool used = r.nx != 0;
        const int ux0 = __reduce_min_sync(kFullMask, used ? r.x0 : INT_MAX), uy0 = __reduce_min_sync(kFullMask, used ? r.y0 : INT_MAX);
        const int ux1 = __reduce_max_sync(kFullMask, used ? r.x0 + r.nx : 0), uy1 = __reduce_max_sync(kFullMask, used ? r.y0 + r.ny : 0);
        if (lane < 4) {
            s_rect[lane] = r;
            const uint32_t v = neighbour_view(a.grid, c.ci, c.cj, lane);
            s_view[lane] = v;
            s_top[lane] = a.sv.view_anc[v * kMaxLevels + L1];
#pragma unroll
            for (int k = 0; k < 4; k++)
                if (lane == k) {
                    s_w[k] = w[k];
                    s_st[k] = st[k];
                }
        }
        if (lane == 0) {
            s_union = Rect{ux0, uy0, ux1 - ux0, uy1 - uy0};
            s_together = (uint64_t)(ux1 - ux0) * (uint64_t)(uy1 - uy0) <= a.un_blocks;
        }
    } else {
        for (int i = tid - 32; i < (256 + 128) / 2; i += kThreads - 32)
            reinterpret_cast<uint32_t *>(s_dig)[i] = reinterpret_cast<const uint32_t *>(g_tables.dig)[i];
    }
    __syncthreads();
    const bool together = s_together;
    const uint32_t hdr0 = 32 * a.sv.MW;
    // the four neighbours in one pass, or one after the other
    for (int pass = 0; pass < (together ? 1 : 4); pass++) {
        const Rect un = together ? s_union : s_rect[pass];
        if (un.nx == 0)
            continue;
        if (tid < 32) {
            // the distinct nodes the pass needs, ascending: lane = (neighbour, level)
            const int k = lane / (int)L1, l = lane - k * (int)L1;
            const bool mine = k < 4 && (together || k == pass) && s_rect[k & 3].nx != 0;
            const uint32_t p = mine ? a.sv.view_anc[s_view[k] * kMaxLevels + l] : 0xFFFFFFFFu;
            const unsigned same = __match_any_sync(kFullMask, p);
            const bool first = mine && (same & ((1u << lane) - 1u)) == 0;
            int e = 0, total = 0;
            for (int j = 0; j < 32; j++) {
                const uint32_t q = __shfl_sync(kFullMask, p, j);
                const bool f = __shfl_sync(kFullMask, (int)first, j) != 0;
                e += f && q < p;
                total += f;
            }
            if (first)
                s_need[e] = p;
            if (mine)
                s_slot[k][l] = e;
            if (lane == 0)
                s_nn = total;
        }
        __syncthreads();
        const int nn = s_nn;
        // ---- 2. table entry of needed node e at union block li, channel c:
        // x = payload offset | present << 31, y = header
        for (int task = tid; task < un.nx * un.ny * 3; task += kThreads) {
            const int li = task / 3, c = task - 3 * li;
            const int ry = li / un.nx, rx = li - ry * un.nx;
            const uint32_t loc = (uint32_t)(un.y0 + ry) * a.sv.nlx + (uint32_t)(un.x0 + rx);
            const uint32_t *rec = a.sv.records + a.sv.offsets[3 * loc + c];
            uint2 *my = s_ent + (size_t)task * ent_stride;
            uint32_t P = 0;
            for (uint32_t m = 0; m < a.sv.MW; m++)
                P += __popc(rec[m]);
            uint32_t off = hdr0 + kHdrBits * P, rank = 0, m_at = 0, word = rec[0], before = 0;   // before: blocks in front of word m_at
            HeaderReader hr(rec, a.sv.MW);
            for (int e = 0; e < nn; e++) {
                const uint32_t p = s_need[e];
                while (m_at < (p >> 5)) {
                    before += __popc(word);
                    word = rec[++m_at];
                }
                const uint32_t bit = 1u << (p & 31u), target = before + __popc(word & (bit - 1u));
                for (; rank < target; rank++)
                    off += mode_bits(s_mode[hr.take() & 31u]);
                uint2 v = make_uint2(0u, 0u);
                if (word & bit) {
                    const uint32_t hdr = hr.take();
                    rank++;
#ifdef RLFC_DEBUG
                    const uint32_t mode = hdr & 31u, pay = mode < (uint32_t)kNumModes ? mode_bits(s_mode[mode]) : 0u;
                    const uint32_t rec_bits = 32u * (a.sv.offsets[3 * loc + c + 1] - a.sv.offsets[3 * loc + c]);
                    // a block that fails the checks of a debug build is left out
                    if (RLFC_DBG_BLOCK_OK(a.sv.dbg, mode, hdr0 + kHdrBits * rank, hdr0 + kHdrBits * P, off, pay, rec_bits))
#else
                    const uint32_t pay = mode_bits(s_mode[hdr & 31u]);
#endif
                        v = make_uint2(off | 0x80000000u, hdr);
                    off += pay;
                }
                my[e] = v;
            }
        }
        __syncthreads();
        // ---- 3. reconstructions of every neighbour's blocks
        const int k0 = together ? 0 : pass, k1 = together ? 4 : pass + 1;
        for (int k = k0; k < k1; k++) {
            const Rect r = s_rect[k];
            const uint32_t top = s_top[k];
            for (int task = tid; task < r.nx * r.ny * 3; task += kThreads) {
                const int li = task / 3, c = task - 3 * li;
                const int ry = li / r.nx, rx = li - ry * r.nx;
                const int bx = r.x0 + rx, by = r.y0 + ry;
                const uint32_t loc = (uint32_t)by * a.sv.nlx + (uint32_t)bx;
                const uint4 *tp = reinterpret_cast<const uint4 *>(a.sv.top + ((size_t)top * a.sv.nloc + loc) * 48 + c * 16);
                uint4 v0 = __ldg(tp), v1 = __ldg(tp + 1);
                // two's complement halves to biased ones: flip the sign (a bias of
                // 2^15), then take 2^14 off; both halves at once, no borrow crosses
                uint32_t v[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
                for (int j = 0; j < 8; j++)
                    v[j] = (v[j] ^ 0x80008000u) - kB2;
                const uint2 *ent = s_ent + (size_t)(((by - un.y0) * un.nx + bx - un.x0) * 3 + c) * ent_stride;
                const uint32_t *rec = a.sv.records + a.sv.offsets[3 * loc + c];
                for (uint32_t l = 0; l < L1; l++) {
                    const uint2 e = ent[s_slot[k][l]];
                    if (!(e.x >> 31))
                        continue;
                    uint32_t d[8];
                    decode_block_pairs(rec, e.x & 0x7FFFFFFFu, e.y, a.sv.q, s_mode, s_dig, d);
#pragma unroll
                    for (int j = 0; j < 8; j++)
                        v[j] += d[j] - kB2;
                }
                uint4 *o = s_rec + ((size_t)k * a.fp_blocks + li) * 6 + c * 2;
                o[0] = make_uint4(v[0], v[1], v[2], v[3]);
                o[1] = make_uint4(v[4], v[5], v[6], v[7]);
            }
        }
        __syncthreads();
    }
    for (int k = 0; k < 4; k++) {
        const Rect r = s_rect[k];
        for (int task = tid; task < r.nx * r.ny * 4; task += kThreads) {
            const uint2 *p = reinterpret_cast<const uint2 *>(s_rec + ((size_t)k * a.fp_blocks + (task >> 2)) * 6) + (task & 3);
            uint32_t w[4];
            row_to_rgb<true>(p[0], p[4], p[8], w);
            s_px[(size_t)k * a.fp_blocks * 4 + task] = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
    __syncthreads();
    // ---- 4. blend
    const uint32_t *px_all = reinterpret_cast<const uint32_t *>(s_px);
    for (int i = tid; i < a.tx * a.ty; i += kThreads) {
        const uint32_t x = x0 + (uint32_t)(i & (a.tx - 1)), y = y0 + (uint32_t)(i >> a.tx_log2);
        if (x > x1 || y > y1)
            continue;
        float acc[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const Rect r = s_rect[k];
            if (r.nx == 0)
                continue;
            const uint32_t *fp = px_all + (size_t)k * a.fp_blocks * 16;
            auto px = [&](int xx, int yy) -> uint32_t {
                const int blk = (yy / kBlock - r.y0) * r.nx + (xx / kBlock - r.x0);
                return fp[blk * 16 + (yy % kBlock) * kBlock + (xx % kBlock)];
            };
            if (kNative) {
                const Stencil st = s_st[k];
                const float wk = s_w[k] * (1.0f / 255.0f);
                const float w00 = wk * (1.0f - st.fx) * (1.0f - st.fy), w10 = wk * st.fx * (1.0f - st.fy);
                const float w01 = wk * (1.0f - st.fx) * st.fy, w11 = wk * st.fx * st.fy;
                const int xa = min(max((int)x + st.ox, 0), W - 1), xb = min(max((int)x + st.ox + 1, 0), W - 1);
                const int ya = min(max((int)y + st.oy, 0), H - 1), yb = min(max((int)y + st.oy + 1, 0), H - 1);
                const uint32_t p00 = px(xa, ya), p10 = px(xb, ya), p01 = px(xa, yb), p11 = px(xb, yb);
#pragma unroll
                for (int c = 0; c < 3; c++)
                    acc[c] = fmaf(w11, chan(p11, c), fmaf(w01, chan(p01, c), fmaf(w10, chan(p10, c), fmaf(w00, chan(p00, c), acc[c]))));
            } else {
                int xa, xb, ya, yb;
                float fx, fy;
                taps(ray_s(x, a.grid.W, a.out_w) + s_st[k].sx, a.grid.W, xa, xb, fx);
                taps(ray_s(y, a.grid.H, a.out_h) + s_st[k].sy, a.grid.H, ya, yb, fy);
                sample_add(s_w[k], fx, fy, px(xa, ya), px(xb, ya), px(xa, yb), px(xb, yb), acc);
            }
        }
        store_rgb(a.out, a.out8, ((size_t)n * a.out_h + y) * a.out_w + x, acc[0], acc[1], acc[2]);
    }
}

// Blocks that `px` output pixels at `src` / `out` source pixels each span: the
// samples, the bilinear neighbour, and whole blocks around them (one more for
// the float rounding of the corner rays).
uint64_t span_blocks(uint32_t px, uint32_t src, uint32_t out, uint32_t most)
{
    const double s = (px - 1) * (double)src / out + 2.0;
    return std::min<uint64_t>((uint64_t)(s / kBlock) + (src == out ? 2 : 3), most);
}

}  // namespace

// n views decoded on demand; RLFC_E_UNSUPPORTED when a tile's footprint does
// not fit shared memory (heavy downscaling: the caller has another path).
int launch_render_demand(const rlfc_stream *s, const float *d_uv, const float *d_disp, uint32_t out_w, uint32_t out_h,
                         uint32_t n, float *d_out, cudaStream_t st, uint8_t *d_out8)
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
    a.uv = d_uv;
    a.disp = d_disp;
    a.out = d_out;
    a.out8 = d_out8;
    a.grid = make_grid(s->info.U, s->info.V, s->info.W, s->info.H);
    a.out_w = out_w;
    a.out_h = out_h;
    const bool native = out_w == s->info.W && out_h == s->info.H;
    // the largest tile that leaves room for four CTAs per SM and, where the
    // views are small, still makes two CTAs per SM; a footprint too large for
    // that takes the smallest tile
    static const int tiles[][2] = {{32, 16}, {32, 8}, {16, 8}, {8, 8}};
    int sms = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, s->device);
    if (e != cudaSuccess)
        return cuda_fail(e, "render_demand: SM count");
    uint32_t smem = 0;
    for (const auto &t : tiles) {
        a.tx = t[0];
        a.ty = t[1];
        a.tx_log2 = t[0] == 32 ? 5 : (t[0] == 16 ? 4 : 3);
        const uint64_t bx = span_blocks(t[0], s->info.W, out_w, s->info.nloc_x), by = span_blocks(t[1], s->info.H, out_h, s->info.nloc_y);
        // the union of the four footprints: two blocks more on each axis cover
        // disparities up to five pixels per view; larger ones are walked apart
        const uint64_t un = std::min<uint64_t>(bx + 2, s->info.nloc_x) * std::min<uint64_t>(by + 2, s->info.nloc_y);
        const uint64_t need = 4 * bx * by * 96 + std::max<uint64_t>(4 * bx * by * 64, un * 3 * 4 * (s->tab.L - 1) * 8);
        a.fp_blocks = (uint32_t)std::min<uint64_t>(bx * by, UINT32_MAX);
        a.un_blocks = (uint32_t)std::min<uint64_t>(un, UINT32_MAX);
        smem = (uint32_t)std::min<uint64_t>(need, UINT32_MAX);
        a.tiles_x = (out_w + t[0] - 1) / t[0];
        const uint64_t ctas = (uint64_t)a.tiles_x * ((out_h + t[1] - 1) / t[1]) * n;
        if (smem <= kSmemFourCtas && ctas >= 2 * (uint64_t)sms)
            break;
    }
    const uint64_t n_tiles = (uint64_t)a.tiles_x * ((out_h + a.ty - 1) / a.ty);
    if (smem > kSmemMost || n_tiles >= (1ull << 31))
        return RLFC_E_UNSUPPORTED;
    auto kern = native ? render_demand_kernel<true> : render_demand_kernel<false>;
    // (the same limit for every call: the attribute belongs to the kernel, and
    // a smaller one set for another thread's light field would refuse this launch)
    if (smem > 40u * 1024u && (e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMost)) != cudaSuccess)
        return cuda_fail(e, "render_demand: shared memory attribute");
    { TraceScope trace_("render_demand_kernel", st); kern<<<dim3((uint32_t)n_tiles, n), kThreads, smem, st>>>(a); }
    if ((e = cudaGetLastError()) != cudaSuccess)
        return cuda_fail(e, "render_demand launch");
    return RLFC_OK;
}

}  // namespace rlfc
