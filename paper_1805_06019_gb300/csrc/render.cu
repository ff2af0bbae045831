// New-view rendering (Section 3.6): quadrilinear interpolation of the light
// field, decoding the needed blocks on demand from the compressed stream.
//
// Ray geometry (the dynamically reparameterised focal plane the paper cites):
// the camera sits at continuous (u, v) on the grid, clamped to it; output
// pixel (x, y) follows s = (x + 0.5) W / out_w - 0.5, t = (y + 0.5) H / out_h
// - 0.5; in neighbour view (i, j) it lands at (s + d (i - u), t + d (j - v)),
// sampled bilinearly with clamp-to-edge; the neighbours i0 = min(floor(u),
// U - 2), i1 = i0 + 1 are blended with weights 1 - fu, fu, and the same in v.
//
// This file routes a call to the renderers of render_windows.cu and
// render_demand.cu, and holds the renderer of thumbnails (outputs much smaller
// than the views): each thread decodes the pixels that it samples, one by one.
#include <cuda_runtime.h>

#include <algorithm>

#include "render_camera.cuh"
#include "warp_decode.cuh"

namespace rlfc {
namespace {

// Calls of at least this many cameras over at least this many source pixels
// decode the neighbour views they need first (one pass over every record,
// then a cheap blend per camera); smaller ones decode tile by tile on demand,
// which costs more per camera but touches only what a camera sees.  Measured at
// the views' own size, on demand / decoded first, us of queued calls: 9 x 9 x
// 512^2 27 / 58 (one camera), 47 / 65 (two), 70 / 68 (three), 90 / 73 (four);
// 17 x 17 x 1024^2 126 / 374, 205 / 393, 370 / 421, 492 / 441; 15 x 15 x 625 x
// 434 36 / 109, 58 / 117, 100 / 126, 134 / 134; 5 x 5 x 256^2 23 / 33 (three),
// 27 / 35 (four), 45 / 39 (eight).  So the line lies between three and four
// cameras; three on the larger fields are up to a quarter slower for it.
constexpr uint32_t kDecodeFirstViews = 3;
constexpr uint64_t kDecodeFirstPixels = 400000;
// A call under stream capture that allocates makes memory nodes, and a graph
// with those can be neither a child graph nor instantiated twice.  Only native
// calls of this many cameras may: the others are captured on demand or pixel
// by pixel, which need no scratch.
constexpr uint32_t kCapturedScratchViews = 4;

__constant__ uint32_t c_modes[kNumModes] = RLFC_MODE_TABLE_INIT;

struct Args {
    StreamView sv;
    const float *uv;
    const float *disp;
    float *out;
    uint8_t *out8;      // when set, 8-bit RGB goes here instead of out
    Grid grid;
    uint32_t out_w, out_h;
};

// One pixel of one view, decoded by a single thread: walk the record of each
// channel to the view's ancestors and extract the one value needed.
__device__ uint32_t thread_decode_pixel(const StreamView &sv, const uint32_t *s_mode, uint32_t view,
                                        uint32_t x, uint32_t y)
{
    const uint32_t loc = (y / kBlock) * sv.nlx + x / kBlock;
    const uint32_t v = (y % kBlock) * kBlock + x % kBlock;
    const uint32_t *anc = sv.view_anc + view * kMaxLevels;
    int32_t ycc[3];
    for (int c = 0; c < 3; c++) {
        const uint32_t *rec = sv.records + sv.offsets[3 * loc + c];
        int32_t acc = sv.top[((size_t)anc[sv.L - 1] * sv.nloc + loc) * 48 + c * 16 + v];
        uint32_t P = 0;
        for (uint32_t m = 0; m < sv.MW; m++)
            P += __popc(rec[m]);
        const uint32_t hdr0 = 32 * sv.MW;
        for (uint32_t l = 0; l + 1 < sv.L; l++) {
            const uint32_t p = anc[l];
            if (!((rec[p >> 5] >> (p & 31u)) & 1u))
                continue;
            uint32_t rank = 0;
            for (uint32_t m = 0; m < (p >> 5); m++)
                rank += __popc(rec[m]);
            rank += __popc(rec[p >> 5] & ((1u << (p & 31u)) - 1u));
            uint32_t off = hdr0 + kHdrBits * P;
            for (uint32_t h = 0; h < rank; h++)
                off += mode_bits(s_mode[get_bits(rec, hdr0 + kHdrBits * h, 5)]);
            const BlockHeader hd = unpack_header(get_bits(rec, hdr0 + kHdrBits * rank, kHdrBits));
            const uint32_t u = bise_value(rec, off, s_mode[hd.mode], v);
            acc += (hd.min + (int32_t)u) * (1 << (sv.q + hd.shift));
        }
        ycc[c] = acc;
    }
    return ycocg_to_rgb24(ycc[0], ycc[1], ycc[2]);
}

__global__ void __launch_bounds__(256) render_direct_kernel(const Args a)
{
    __shared__ uint32_t s_mode[kNumModes];
    if (threadIdx.x < kNumModes)
        s_mode[threadIdx.x] = c_modes[threadIdx.x];
    __syncthreads();
    const uint32_t n = blockIdx.y;
    const uint32_t pix = blockIdx.x * blockDim.x + threadIdx.x;
    if (pix >= a.out_w * a.out_h)
        return;
    const uint32_t x = pix % a.out_w, y = pix / a.out_w;
    CameraCell cell;
    camera_cell(a.grid, a.uv, n, cell);
    Stencil st[4];
    float w[4];
    camera_stencils(a.grid, cell, a.disp[n], w, st);
    const float s = ray_s(x, a.grid.W, a.out_w), t = ray_s(y, a.grid.H, a.out_h);
    float acc[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll 1
    for (int k = 0; k < 4; k++) {
        if (w[k] == 0.0f)
            continue;
        int xa, xb, ya, yb;
        float fx, fy;
        taps(s + st[k].sx, a.grid.W, xa, xb, fx);
        taps(t + st[k].sy, a.grid.H, ya, yb, fy);
        const uint32_t vw = neighbour_view(a.grid, cell.ci, cell.cj, k);
        const uint32_t p00 = thread_decode_pixel(a.sv, s_mode, vw, xa, ya);
        const uint32_t p10 = thread_decode_pixel(a.sv, s_mode, vw, xb, ya);
        const uint32_t p01 = thread_decode_pixel(a.sv, s_mode, vw, xa, yb);
        const uint32_t p11 = thread_decode_pixel(a.sv, s_mode, vw, xb, yb);
        sample_add(w[k], fx, fy, p00, p10, p01, p11, acc);
    }
    store_rgb(a.out, a.out8, ((size_t)n * a.out_h + y) * a.out_w + x, acc[0], acc[1], acc[2]);
}

// Times of a call at another size than the views' by the three paths, in us,
// fitted to 500 calls (5 x 5 x 256^2 to 17 x 17 x 2048^2 and 5 x 5 x 4096^2, 1
// to 1000 cameras, outputs of a half to a 128th of the views' width; median
// errors 4 % decoded, 16 % direct).  A thumbnail samples a few pixels of many
// blocks: pixel by pixel it costs its header walks, while the other paths
// decode every block in view.  Measured, one camera, direct / decoded first:
// 9 x 9 x 2048^2 at 128 x 128 163 / 485; 17 x 17 x 2048^2 at 64 x 64 274 / 1122;
// 5 x 5 x 4096^2 at 256 x 256 134 / 1405, at 682 x 682 435 / 751 (on demand);
// and where it does not pay: 17 x 17 x 1024^2 at 128 x 128 377 / 136 (on
// demand), 9 x 9 x 512^2 at 32 x 32 170 / 54, 1000 cameras of 9 x 9 x 1024^2 at
// 32 x 32 3171 / 334.
struct Estimate {
    double n, nodes;                   // cameras, tree nodes
    double src, stream, needed, px;    // megapixels of a view, megabytes of records, megapixels of the needed views and of the output
    Estimate(const rlfc_stream &s, uint32_t out_w, uint32_t out_h, uint32_t cams)
        : n(cams), nodes(s.tab.S), src(1e-6 * s.info.W * s.info.H), stream(4e-6 * s.record_words),
          needed(src * std::min<double>(s.tab.n_views, 4.0 * n)), px(1e-6 * out_w * out_h * n)
    {
    }
    double decoded() const { return 25 + src * (49 + 0.41 * nodes) + 1.35 * stream + 1.13 * needed + 25 * px; }
    double demand() const { return 20 + n * src * (36 + 0.22 * nodes); }
    double direct() const { return 90 + nodes * (n < 3 ? 0.7 : 1.5) + px * (700 + 12 * nodes); }
};

bool capturing(cudaStream_t st)
{
    cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &c) != cudaSuccess) {
        cudaGetLastError();   // the legacy stream beside another one's capture: not captured itself
        return false;
    }
    return c != cudaStreamCaptureStatusNone;
}

}  // namespace

int launch_render(const rlfc_stream *s, const float *d_uv, const float *d_disp, uint32_t out_w,
                  uint32_t out_h, uint32_t n, float *d_out, cudaStream_t st, uint8_t *d_out8)
{
    const bool native = out_w == s->info.W && out_h == s->info.H;
    const bool scratch = (native && n >= kCapturedScratchViews) || !capturing(st);
    const bool first = scratch && n >= kDecodeFirstViews && (uint64_t)n * s->info.W * s->info.H >= kDecodeFirstPixels;
    const Estimate cost(*s, out_w, out_h, n);
    for (int turn = 0; turn < 2; turn++) {
        // the other path where the first cannot run: no scratch to decode
        // into, or a tile's footprint too large for shared memory
        const bool decode = (turn == 0) == first;
        if (decode && !scratch)
            continue;
        if (!native && cost.direct() < 0.95 * (decode ? cost.decoded() : cost.demand()))
            break;
        const int rc = decode ? launch_render_decoded(s, d_uv, d_disp, out_w, out_h, n, d_out, st, d_out8)
                              : launch_render_demand(s, d_uv, d_disp, out_w, out_h, n, d_out, st, d_out8);
        if (rc != RLFC_E_UNSUPPORTED)
            return rc;
    }
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
    const uint64_t pix = (uint64_t)out_w * out_h;
    if (pix >= (1ull << 31)) {
        set_error("output view too large");
        return RLFC_E_RANGE;
    }
    { rlfc::TraceScope trace_("render_direct_kernel", st); render_direct_kernel<<<dim3((uint32_t)((pix + 255) / 256), n), 256, 0, st>>>(a); }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return cuda_fail(e, "render launch");
    return RLFC_OK;
}

}  // namespace rlfc
