// New-view rendering for batches of cameras (Section 3.6): the neighbour views
// the batch needs are decoded once, then every camera is blended from them: at
// the views' own resolution from shared windows, at others sample by sample.
//
// Every new camera (u, v) inside grid cell (i0, j0) blends the same four
// neighbour views (i0, j0), (i0+1, j0), (i0, j0+1), (i0+1, j0+1), and at
// native size the ray of output pixel x lands at x + d (i - u) in neighbour
// i: a shift that is constant over the view, so each neighbour contributes a
// fixed 2 x 2 stencil with four fixed weights.
//
//  1. render_plan_kernel (one CTA): sorts the cameras by cell, computes each
//     camera's stencils once, cuts every cell's cameras into groups whose
//     shifted windows fit shared memory, marks the views needed and numbers
//     their slots;
//  2. the needed views are decoded into packed RGB slots (decode_all.cu);
//  3. render_native_kernel: persistent CTAs take (group, 64 x 16 tile) items
//     from a queue, fill one window of the tile per neighbour, and blend the
//     group's cameras from the windows.
#include <cuda_runtime.h>

#include <algorithm>

#include "pair_decode.cuh"
#include "render_camera.cuh"

namespace rlfc {
namespace {

constexpr int kTW = 64, kTH = 16;          // output tile
constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kRows = 4;                   // rows of the pixel pair that a thread blends
constexpr int kGroup = 32;                 // cameras per group at most (a warp plans one)
constexpr int kPitch = 18;                 // quads of a window row: a compile-time pitch for shift spreads up to 4 at least
// shared memory for a group's windows: three CTAs per SM with the group's
// cameras and the staged output rows (fewer bytes for 8-bit output)
constexpr uint32_t kWinBytes = 46 * 1024, kWinBytesU8 = 64 * 1024;
constexpr int kPlanThreads = 1024;
constexpr uint32_t kPlanViews = 32 * kPlanThreads;   // views at most: a mask word per thread
constexpr uint32_t plan_bytes(uint32_t n_cells, uint32_t n_views) { return 4u * (n_cells + 1 + 2 * ((n_views + 31) / 32)) + 2u * n_cells; }
// (one limit for every call: the attribute that sets it belongs to the kernel,
// not to the call; a grid has no more cells than views)
constexpr uint32_t kPlanSmemMost = plan_bytes(kPlanViews, kPlanViews);

// One camera: the four neighbours' stencil weights (blend weight / 255 times
// the bilinear weights) and integer shifts.
struct __align__(16) Cam {
    float w[4][4];     // [k][00, 10, 01, 11]
    int ox[4], oy[4];
    uint32_t r;        // view index of the call
    uint32_t used;     // bit k: neighbour k has a non-zero weight
    uint32_t pad[2];
};

// Cameras [first, first + count) of the sorted list, all of one cell, whose
// windows fit shared memory together: the extent of their shifts.
struct __align__(16) Group {
    uint32_t first, count, cell, used;
    int oxmin[4], oxmax[4], oymin[4], oymax[4];
};

struct Plan {
    const float *uv, *disp;
    Cam *cams;             // [n] sorted by cell
    Group *groups;         // [n] at most
    uint32_t *rank;        // [n] position of a camera in its cell
    uint32_t *counts;      // [0] groups, [1] queue head
    uint8_t *needed;       // [n_views]
    uint32_t *slot_of;     // [n_views]
    Grid grid;
    uint32_t n, n_views;
    uint32_t win_bytes;    // shared memory for the windows of a group
    uint32_t group_cap;    // cameras per group at most
};

// A window starts at a multiple of four source pixels (16-byte loads of the
// packed rows) and holds whole quads.
__host__ __device__ __forceinline__ int window_quads(int oxmin, int oxmax)
{
    return ((oxmin & 3) + (oxmax - oxmin) + kTW + 1 + 3) >> 2;
}
__host__ __device__ __forceinline__ int window_rows(int oymin, int oymax) { return kTH + 1 + oymax - oymin; }

// One CTA.  What bounds it: its own latency (a few passes over the cameras and
// the grid); it replaces four small launches and the camera scan that every
// tile's CTA did, and takes 16 us for 1000 cameras on a 9 x 9 grid, 9 for 24.
__global__ void __launch_bounds__(kPlanThreads) render_plan_kernel(const Plan a)
{
    extern __shared__ uint32_t sm[];
    const uint32_t n_cells = a.grid.cells_u * a.grid.cells_v;
    const uint32_t need_words = (a.n_views + 31) / 32;
    uint32_t *cell_at = sm;                  // counts, then the start of each cell's cameras
    uint32_t *need = sm + n_cells + 1;       // bit per view
    uint32_t *need_at = need + need_words;   // needed views in front of each word
    uint16_t *live = reinterpret_cast<uint16_t *>(need_at + need_words);   // the cells that hold cameras
    __shared__ uint32_t s_warp[kPlanThreads / 32];
    __shared__ uint32_t s_groups, s_live;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (uint32_t i = tid; i < n_cells + 1 + need_words; i += kPlanThreads)
        sm[i] = 0u;
    if (tid == 0)
        s_groups = s_live = 0u;
    __syncthreads();
    for (uint32_t r = tid; r < a.n; r += kPlanThreads) {
        CameraCell c;
        camera_cell(a.grid, a.uv, r, c);
        a.rank[r] = atomicAdd(&cell_at[c.cj * a.grid.cells_u + c.ci], 1u);
    }
    __syncthreads();
    // exclusive scan of the counts, a run of cells per thread
    const auto block_scan = [&](uint32_t x) {
        uint32_t incl = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
            if (lane >= d)
                incl += y;
        }
        if (lane == 31)
            s_warp[warp] = incl;
        __syncthreads();
        uint32_t before = 0;
        if (warp == 0) {
            uint32_t w = s_warp[lane];
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, w, d);
                if (lane >= d)
                    w += y;
            }
            s_warp[lane] = w;
        }
        __syncthreads();
        before = warp ? s_warp[warp - 1] : 0u;
        __syncthreads();
        return before + incl - x;
    };
    {
        const uint32_t per = (n_cells + kPlanThreads - 1) / kPlanThreads;
        const uint32_t c0 = min(n_cells, tid * per), c1 = min(n_cells, c0 + per);
        uint32_t sum = 0;
        for (uint32_t c = c0; c < c1; c++)
            sum += cell_at[c];
        uint32_t at = block_scan(sum);
        for (uint32_t c = c0; c < c1; c++) {
            const uint32_t k = cell_at[c];
            cell_at[c] = at;
            at += k;
            if (k)
                live[atomicAdd(&s_live, 1u)] = (uint16_t)c;
        }
        if (tid == 0)
            cell_at[n_cells] = a.n;
    }
    __syncthreads();
    for (uint32_t r = tid; r < a.n; r += kPlanThreads) {
        CameraCell cc;
        camera_cell(a.grid, a.uv, r, cc);
        Stencil st[4];
        float w[4];
        camera_stencils(a.grid, cc, a.disp[r], w, st);
        Cam c;
        c.r = r;
        c.used = 0u;
        c.pad[0] = c.pad[1] = 0u;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const float wk = w[k] * (1.0f / 255.0f);
            c.w[k][0] = wk * (1.0f - st[k].fx) * (1.0f - st[k].fy);
            c.w[k][1] = wk * st[k].fx * (1.0f - st[k].fy);
            c.w[k][2] = wk * (1.0f - st[k].fx) * st[k].fy;
            c.w[k][3] = wk * st[k].fx * st[k].fy;
            c.ox[k] = st[k].ox;
            c.oy[k] = st[k].oy;
            if (w[k] != 0.0f) {
                c.used |= 1u << k;
                const uint32_t v = neighbour_view(a.grid, cc.ci, cc.cj, k);
                atomicOr(&need[v >> 5], 1u << (v & 31u));
            }
        }
        a.cams[cell_at[cc.cj * a.grid.cells_u + cc.ci] + a.rank[r]] = c;
    }
    __syncthreads();
    // groups: a warp takes a cell's cameras 32 at a time, and the longest
    // prefix of them whose windows fit
    {
        for (uint32_t i = warp; i < s_live; i += kPlanThreads / 32) {
            const uint32_t cell = live[i];
            const uint32_t end = cell_at[cell + 1];
            for (uint32_t first = cell_at[cell]; first < end;) {
                uint32_t count = min(a.group_cap, end - first);
                const Cam &c = a.cams[first + min((uint32_t)lane, count - 1)];
                int ox[4], oy[4];
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    ox[k] = c.ox[k];
                    oy[k] = c.oy[k];
                }
                const uint32_t cu = c.used;
                Group g;
                for (;;) {   // ends at count = 1, which always fits
                    int rows = 0, pitch = kPitch;
                    bool wide = false;   // (spreads this wide never fit, and their products could wrap)
                    const bool in = (uint32_t)lane < count;
                    g.used = __reduce_or_sync(0xFFFFFFFFu, in ? cu : 0u);
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        g.oxmin[k] = __reduce_min_sync(0xFFFFFFFFu, in ? ox[k] : INT_MAX);
                        g.oxmax[k] = __reduce_max_sync(0xFFFFFFFFu, in ? ox[k] : INT_MIN);
                        g.oymin[k] = __reduce_min_sync(0xFFFFFFFFu, in ? oy[k] : INT_MAX);
                        g.oymax[k] = __reduce_max_sync(0xFFFFFFFFu, in ? oy[k] : INT_MIN);
                        if ((g.used >> k) & 1u) {
                            wide |= (long long)g.oxmax[k] - g.oxmin[k] > 2048 || (long long)g.oymax[k] - g.oymin[k] > 2048;
                            rows += window_rows(g.oymin[k], g.oymax[k]);
                            pitch = max(pitch, window_quads(g.oxmin[k], g.oxmax[k]));
                        }
                    }
                    if (count == 1 || (!wide && 32u * (uint32_t)pitch * (uint32_t)rows <= a.win_bytes))
                        break;
                    count = (count + 1) / 2;
                }
                g.first = first;
                g.count = count;
                g.cell = cell;
                if (lane == 0)
                    a.groups[atomicAdd(&s_groups, 1u)] = g;
                first += count;
            }
        }
    }
    __syncthreads();
    // slots of the needed views, in view order (a mask word per thread)
    {
        const uint32_t at = block_scan((uint32_t)tid < need_words ? (uint32_t)__popc(need[tid]) : 0u);
        if ((uint32_t)tid < need_words)
            need_at[tid] = at;
    }
    __syncthreads();
    for (uint32_t v = tid; v < a.n_views; v += kPlanThreads) {
        const uint32_t word = need[v >> 5], bit = 1u << (v & 31u);
        a.needed[v] = (word & bit) != 0u;
        a.slot_of[v] = need_at[v >> 5] + (uint32_t)__popc(word & (bit - 1u));
    }
    if (tid == 0) {
        a.counts[0] = s_groups;
        a.counts[1] = 0u;
    }
}

struct Args {
    const Cam *cams;
    const Group *groups;
    uint32_t *counts;
    const uint32_t *decoded;   // packed RGB views [slot][H][pitch]
    const uint32_t *slot_of;
    float *out;
    uint8_t *out8;
    Grid grid;
    uint32_t pitch, tiles_x, n_tiles;
    uint32_t bulk;             // every row of a tile starts and ends on a 16-byte boundary
};

// A window pixel: R and G as bf16 halves of one word, B as a float; 8-bit
// values are exact in both, and each unpacks with one shift or mask, or none.
// byte -> float through the exponent of 2^23, on the FMA pipe (the integer
// conversion runs at a quarter of its rate)
__device__ __forceinline__ uint2 window_pixel(uint32_t rgb24)
{
    const float r = __uint_as_float(__byte_perm(rgb24, 0x4B000000u, 0x7440)) - 8388608.0f;
    const float g = __uint_as_float(__byte_perm(rgb24, 0x4B000000u, 0x7441)) - 8388608.0f;
    const float b = __uint_as_float(__byte_perm(rgb24, 0x4B000000u, 0x7442)) - 8388608.0f;
    return make_uint2(__byte_perm(__float_as_uint(r), __float_as_uint(g), 0x7632), __float_as_uint(b));
}
extern __shared__ __align__(16) uint2 g_win[];
__device__ __forceinline__ float3 win_rgb(uint32_t at)
{
    const uint2 p = *reinterpret_cast<const uint2 *>(reinterpret_cast<const char *>(g_win) + at);
    return make_float3(__uint_as_float(p.x << 16), __uint_as_float(p.x & 0xFFFF0000u), __uint_as_float(p.y));
}

// w00 a + w10 b + w01 c + w11 d added to acc, in that order; R and G as a pair
// (a paired FMA runs no faster than two, but takes one issue slot)
__device__ __forceinline__ float2 twice(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 rg(const float3 &a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ void blend_pixel(float4 w, const float3 &a, const float3 &b, const float3 &c, const float3 &d, float3 &acc)
{
    const float2 p = __ffma2_rn(twice(w.w), rg(d), __ffma2_rn(twice(w.z), rg(c), __ffma2_rn(twice(w.y), rg(b), __ffma2_rn(twice(w.x), rg(a), rg(acc)))));
    acc.x = p.x;
    acc.y = p.y;
    acc.z = fmaf(w.w, d.z, fmaf(w.z, c.z, fmaf(w.y, b.z, fmaf(w.x, a.z, acc.z))));
}

struct Window {
    uint32_t row0;     // rows of the windows in front of this one
    int nq;            // quads filled per row
    int sx0, sy0;      // source pixel of the window's first pixel
    uint32_t slot;
    uint32_t tasks;    // quads of the windows up to and including this one
    uint32_t inv;      // ceil(2^20 / nq)
};

struct __align__(16) CamS {
    float w[4][4];
    uint2 at[4];       // byte offset of window pixel x (x + 2 follows it) and of x + 1, for lane 0, row 0
    uint8_t *out;      // the camera's first output byte of the tile
    uint32_t used;
    uint32_t pad;
};

// The pixel pair (2 lane, 2 lane + 1) of kRows rows from r0 of one camera.
// kQ: quads per window row, or 0 for the pitch given.
template <int kQ>
__device__ __forceinline__ void blend_rows(const CamS &c, int pitch_quads, int r0, int lane, float3 acc[kRows][2])
{
    const uint32_t pitch = 32u * (uint32_t)(kQ ? kQ : pitch_quads);   // bytes
    const uint32_t used = c.used, off = (uint32_t)r0 * pitch + 8u * (uint32_t)lane;
#pragma unroll
    for (int rr = 0; rr < kRows; rr++)
        acc[rr][0] = acc[rr][1] = make_float3(0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int k = 0; k < 4; k++) {
        if (!((used >> k) & 1u))
            continue;
        const float4 w = *reinterpret_cast<const float4 *>(c.w[k]);
        const uint2 at = c.at[k];
        const uint32_t fa = at.x + off, fb = at.y + off;
        float3 u0 = win_rgb(fa), u1 = win_rgb(fb), u2 = win_rgb(fa + 8);
#pragma unroll
        for (int rr = 0; rr < kRows; rr++) {
            const uint32_t o = (uint32_t)(rr + 1) * pitch;
            const float3 x0 = win_rgb(fa + o), x1 = win_rgb(fb + o), x2 = win_rgb(fa + o + 8);
            blend_pixel(w, u0, u1, x0, x1, acc[rr][0]);
            blend_pixel(w, u1, u2, x1, x2, acc[rr][1]);
            u0 = x0;
            u1 = x1;
            u2 = x2;
        }
    }
}

// What bounds it: instruction issue and the shared-memory pipe (64 % and 71 %
// busy).  A thread blends two neighbouring pixels of four rows, so that a
// row of the pair's stencil is three window pixels instead of four; windows
// hold even and odd columns apart, so that the lanes' pairs are consecutive
// words whatever the shift; window rows have a compile-time pitch wherever
// the shifts allow.  Finished rows go through shared memory and out as bulk
// copies of 768 bytes: stores from the lanes, 8 bytes at a stride of 24, cost
// 0.75 ms for the 3.1 GB of 1000 views of 512 x 512 on their own, the bulk
// copies 0.56 ms.  Those views take 0.81 ms (3.9 TB/s); with one pixel column
// per thread, direct stores and the cameras' parameters computed by every
// tile, 1.15 ms.
template <bool kU8>
__global__ void __launch_bounds__(kThreads, 3) render_native_kernel(const Args a)
{
    constexpr int kPix = kU8 ? 3 : 12, kRowWords = kTW * kPix / 4;   // output bytes per pixel, staged words per row
    __shared__ Window s_win[4];
    __shared__ CamS s_cam[kGroup];
    __shared__ uint32_t s_item[2];
    __shared__ Group s_group[2];       // this item's group and the next one's
    __shared__ uint32_t s_slot[2][4];  // and the slots of their neighbours
    __shared__ int s_pitch;   // quads per window row
    // a warp's rows, with a chunk of padding on each side (store_row_unaligned)
    __shared__ __align__(16) uint32_t s_rows[kWarps][kRows * kRowWords + 8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t n_items = a.counts[0] * a.n_tiles;
    const int W = (int)a.grid.W, H = (int)a.grid.H;

    uint64_t policy;   // evict-first: the outputs stream through L2 without pushing out the decoded views
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    // one warp fetches an item, its group and its neighbours' slots one item
    // ahead: three dependent loads that the windows would wait for (24 8-bit
    // views of 625 x 434, mostly windows: 97 instead of 108 us)
    const auto fetch = [&](uint32_t turn) {
        uint32_t item = 0;
        if (lane == 0)
            item = atomicAdd(&a.counts[1], 1u);
        item = __shfl_sync(0xFFFFFFFFu, item, 0);
        if (lane == 0)
            s_item[turn] = item;
        if (item < n_items) {
            const Group *g = a.groups + item / a.n_tiles;
            if (lane < (int)(sizeof(Group) / 4))
                reinterpret_cast<uint32_t *>(&s_group[turn])[lane] = reinterpret_cast<const uint32_t *>(g)[lane];
            if (lane < 4 && ((g->used >> lane) & 1u))
                s_slot[turn][lane] = a.slot_of[neighbour_view(a.grid, g->cell % a.grid.cells_u, g->cell / a.grid.cells_u, lane)];
        }
    };
    if (warp == 0)
        fetch(0);
    __syncthreads();
    for (uint32_t turn = 0;; turn ^= 1u) {
        const uint32_t item = s_item[turn];
        if (item >= n_items)
            break;
        const Group &g = s_group[turn];
        const uint32_t tile = item % a.n_tiles;
        const int tx0 = (int)(tile % a.tiles_x) * kTW, ty0 = (int)(tile / a.tiles_x) * kTH;
        const uint32_t count = g.count;
        const int ng = min(kTH / kRows, (H - ty0 + kRows - 1) / kRows);   // row groups inside the image
        const int th = kRows * ng;
        // ---- the windows, and the cameras' positions in them
        if (tid < 32) {
            const int k = tid & 3;
            const bool used = (g.used >> k) & 1u;
            const int oxmin = g.oxmin[k], oymin = g.oymin[k];
            const int nq = used ? window_quads(oxmin, g.oxmax[k]) : 0;
            const int rows = used ? th + 1 + g.oymax[k] - oymin : 0;
            const uint32_t tasks = (uint32_t)(nq * rows);
            uint32_t before = 0, row0 = 0;
            int widest = max(nq, kPitch);
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const uint32_t t = __shfl_sync(0xFFFFFFFFu, tasks, j), r = __shfl_sync(0xFFFFFFFFu, (uint32_t)rows, j);
                before += j < k ? t : 0u;
                row0 += j < k ? r : 0u;
                widest = max(widest, __shfl_sync(0xFFFFFFFFu, nq, j));
            }
            if (tid == 0)
                s_pitch = widest;
            if (tid < 4) {
                Window wn;
                wn.row0 = row0;
                wn.nq = nq;
                wn.sx0 = tx0 + oxmin - (oxmin & 3);
                wn.sy0 = ty0 + oymin;
                wn.slot = used ? s_slot[turn][k] : 0u;
                wn.tasks = before + tasks;
                wn.inv = nq ? ((1u << 20) + (uint32_t)nq - 1u) / (uint32_t)nq : 0u;
                s_win[k] = wn;
            }
        }
        __syncthreads();
        const int pitch_q = s_pitch;
        if (tid < 4 * (int)count) {
            const int k = tid & 3;
            const Cam &c = a.cams[g.first + (tid >> 2)];
            CamS &d = s_cam[tid >> 2];
            *reinterpret_cast<float4 *>(d.w[k]) = *reinterpret_cast<const float4 *>(c.w[k]);
            // even columns of a window row first, then the odd ones (two per quad of each)
            const int x = c.ox[k] + tx0 - s_win[k].sx0, row = ((int)s_win[k].row0 + c.oy[k] + ty0 - s_win[k].sy0) * 4 * pitch_q;
            d.at[k] = make_uint2(8u * (uint32_t)(row + (x & 1) * 2 * pitch_q + (x >> 1)),
                                 8u * (uint32_t)(row + ((x & 1) ^ 1) * 2 * pitch_q + ((x + 1) >> 1)));
            if (k == 0) {
                d.out = (kU8 ? a.out8 : reinterpret_cast<uint8_t *>(a.out)) +
                        (((size_t)c.r * (uint32_t)H + (uint32_t)ty0) * (uint32_t)W + (uint32_t)tx0) * kPix;
                d.used = c.used;
            }
        }
        {
            // four source pixels at a time: 16-byte loads inside the image,
            // clamped single pixels at its edge
            const uint32_t n0 = s_win[0].tasks, n1 = s_win[1].tasks, n2 = s_win[2].tasks, total = s_win[3].tasks;
#pragma unroll 2
            for (uint32_t t = tid; t < total; t += kThreads) {
                const int k = (t >= n0) + (t >= n1) + (t >= n2);
                const Window &wn = s_win[k];
                const uint32_t i = t - (k ? s_win[k - 1].tasks : 0u);
                const uint32_t row = (i * wn.inv) >> 20, q = i - row * (uint32_t)wn.nq;
                const int x = wn.sx0 + 4 * (int)q, y = min(max(wn.sy0 + (int)row, 0), H - 1);
                const uint32_t *src = a.decoded + ((size_t)wn.slot * (uint32_t)H + (uint32_t)y) * a.pitch;
                uint4 v;
                if (x >= 0 && x + 3 < W) {
                    v = __ldg(reinterpret_cast<const uint4 *>(src + x));
                } else {
                    v.x = __ldg(src + min(max(x, 0), W - 1));
                    v.y = __ldg(src + min(max(x + 1, 0), W - 1));
                    v.z = __ldg(src + min(max(x + 2, 0), W - 1));
                    v.w = __ldg(src + min(max(x + 3, 0), W - 1));
                }
                const uint2 p0 = window_pixel(v.x), p1 = window_pixel(v.y), p2 = window_pixel(v.z), p3 = window_pixel(v.w);
                uint2 *d = g_win + (wn.row0 + row) * 4u * (uint32_t)pitch_q + 2u * q;
                *reinterpret_cast<uint4 *>(d) = make_uint4(p0.x, p0.y, p2.x, p2.y);
                *reinterpret_cast<uint4 *>(d + 2 * pitch_q) = make_uint4(p1.x, p1.y, p3.x, p3.y);
            }
        }
        if (warp == kWarps - 1)
            fetch(turn ^ 1u);
        __syncthreads();
        // ---- blend: a warp takes (camera, four rows of the tile)
        uint32_t *stage = s_rows[warp] + 4;
        const uint32_t len = (uint32_t)(kPix * min(kTW, W - tx0)), pitch = (uint32_t)(kPix * W);   // bytes
        for (uint32_t it = warp; it < count * (uint32_t)ng; it += kWarps) {
            const uint32_t ci = ng == kTH / kRows ? it / (kTH / kRows) : it / (uint32_t)ng;
            const int r0 = kRows * (int)(it - ci * (uint32_t)ng);
            const CamS &c = s_cam[ci];
            float3 acc[kRows][2];
            if (pitch_q == kPitch)
                blend_rows<kPitch>(c, pitch_q, r0, lane, acc);
            else
                blend_rows<0>(c, pitch_q, r0, lane, acc);
            // the rows through the warp's buffer, then out whole
            if (a.bulk && lane < kRows)
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
#pragma unroll
            for (int rr = 0; rr < kRows; rr++) {
                const float3 p = acc[rr][0], q = acc[rr][1];
                if (kU8) {
                    uint16_t *s = reinterpret_cast<uint16_t *>(stage + rr * kRowWords) + 3 * lane;
                    s[0] = (uint16_t)__byte_perm(u8_value(p.x), u8_value(p.y), 0x0040);
                    s[1] = (uint16_t)__byte_perm(u8_value(p.z), u8_value(q.x), 0x0040);
                    s[2] = (uint16_t)__byte_perm(u8_value(q.y), u8_value(q.z), 0x0040);
                } else {
                    float2 *s = reinterpret_cast<float2 *>(stage + rr * kRowWords) + 3 * lane;
                    s[0] = make_float2(p.x, p.y);
                    s[1] = make_float2(p.z, q.x);
                    s[2] = make_float2(q.y, q.z);
                }
            }
            const int rows = min(kRows, H - ty0 - r0);
            uint8_t *o = c.out + (size_t)(uint32_t)r0 * pitch;
            if (a.bulk) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane < rows) {
                    asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;" ::"l"(
                                     __cvta_generic_to_global(o + (size_t)lane * pitch)),
                                 "r"((uint32_t)__cvta_generic_to_shared(stage + lane * kRowWords)), "r"(len), "l"(policy)
                                 : "memory");
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
            } else {
                __syncwarp();
                constexpr int kLanes = kU8 ? 16 : 32;   // lanes per row: an 8-bit row spans at most 13 chunks
                for (int rr = lane / kLanes; rr < rows; rr += 32 / kLanes)
                    for (uint32_t ch = (uint32_t)(lane % kLanes); ch < (len + 30) / 16; ch += kLanes)
                        store_row_unaligned(o + (size_t)rr * pitch, stage + rr * kRowWords, len, ch);
            }
        }
        __syncthreads();   // the next item reuses the windows
    }
    if (a.bulk)
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the staged rows are read before the CTA ends
}

// Any output size: a thread per output pixel samples the decoded views through
// the caches.  What bounds it: instruction issue (16 samples, their weights and
// coordinates per pixel); eight 800 x 600 views take 79 us, and with the
// decode of their neighbours 0.14 ms (1.0 with a warp per block of every tile).
constexpr int kSX = 32, kSY = 8;

__global__ void __launch_bounds__(kSX * kSY) render_sampled_kernel(const Args a, const float *uv, const float *disp, uint32_t out_w,
                                                                    uint32_t out_h, uint32_t tiles_x)
{
    const uint32_t n = blockIdx.y;
    const uint32_t x = (blockIdx.x % tiles_x) * kSX + threadIdx.x % kSX, y = (blockIdx.x / tiles_x) * kSY + threadIdx.x / kSX;
    if (x >= out_w || y >= out_h)
        return;
    CameraCell c;
    camera_cell(a.grid, uv, n, c);
    Stencil st[4];
    float w[4];
    camera_stencils(a.grid, c, disp[n], w, st);
    const float s = ray_s(x, a.grid.W, out_w), t = ray_s(y, a.grid.H, out_h);
    float acc[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < 4; k++) {
        if (w[k] == 0.0f)
            continue;
        int xa, xb, ya, yb;
        float fx, fy;
        taps(s + st[k].sx, a.grid.W, xa, xb, fx);
        taps(t + st[k].sy, a.grid.H, ya, yb, fy);
        const uint32_t *v = a.decoded + (size_t)a.slot_of[neighbour_view(a.grid, c.ci, c.cj, k)] * a.grid.H * a.pitch;
        const uint32_t *ra = v + (size_t)(uint32_t)ya * a.pitch, *rb = v + (size_t)(uint32_t)yb * a.pitch;
        sample_add(w[k], fx, fy, __ldg(ra + xa), __ldg(ra + xb), __ldg(rb + xa), __ldg(rb + xb), acc);
    }
    store_rgb(a.out, a.out8, ((size_t)n * out_h + y) * out_w + x, acc[0], acc[1], acc[2]);
}

}  // namespace

// Rendering of n views from views decoded for the call: planned, decoded into
// slots, then blended (at native size from windows, at others by samples).
// Returns RLFC_E_UNSUPPORTED when the scratch cannot be had (the caller
// decodes on demand instead).
int launch_render_decoded(const rlfc_stream *s, const float *d_uv, const float *d_disp, uint32_t out_w, uint32_t out_h, uint32_t n,
                          float *d_out, cudaStream_t st, uint8_t *d_out8)
{
    const bool native = out_w == s->info.W && out_h == s->info.H;
    Plan p;
    Args a;
    p.grid = a.grid = make_grid(s->info.U, s->info.V, s->info.W, s->info.H);
    const uint32_t n_views = s->tab.n_views, n_cells = p.grid.cells_u * p.grid.cells_v;
    a.pitch = packed_pitch(s->info.W);
    a.tiles_x = (s->info.W + kTW - 1) / kTW;
    a.n_tiles = a.tiles_x * ((s->info.H + kTH - 1) / kTH);
    const uint32_t stiles_x = (out_w + kSX - 1) / kSX;
    const uint64_t stiles = (uint64_t)stiles_x * ((out_h + kSY - 1) / kSY);
    if (n_views > kPlanViews || (uint64_t)a.n_tiles * n >= (1ull << 32) - (1u << 20) || stiles >= (1ull << 31))
        return RLFC_E_UNSUPPORTED;
    // one stream-ordered block: the plan, then a slot per needed view (a
    // camera needs at most four views, so min(views, 4n) slots suffice)
    const auto r256 = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t n_slots = std::min<size_t>(n_views, 4ull * n);
    const size_t at_cams = 256, at_groups = at_cams + r256(sizeof(Cam) * (size_t)n);
    const size_t at_rank = at_groups + r256(sizeof(Group) * (size_t)n), at_need = at_rank + r256(4ull * n);
    const size_t at_slot = at_need + r256(n_views), at_dec = at_slot + r256(4ull * n_views);
    uint8_t *scratch = nullptr;
    if (scratch_alloc(s, (void **)&scratch, at_dec + 4ull * a.pitch * s->info.H * n_slots, st) != cudaSuccess) {
        cudaGetLastError();
        return RLFC_E_UNSUPPORTED;
    }
    p.uv = d_uv;
    p.disp = d_disp;
    p.counts = a.counts = reinterpret_cast<uint32_t *>(scratch);
    p.cams = reinterpret_cast<Cam *>(scratch + at_cams);
    p.groups = reinterpret_cast<Group *>(scratch + at_groups);
    p.rank = reinterpret_cast<uint32_t *>(scratch + at_rank);
    p.needed = scratch + at_need;
    p.slot_of = reinterpret_cast<uint32_t *>(scratch + at_slot);
    p.n = n;
    p.n_views = n_views;
    a.cams = p.cams;
    a.groups = p.groups;
    a.slot_of = p.slot_of;
    a.decoded = reinterpret_cast<uint32_t *>(scratch + at_dec);
    a.out = d_out;
    a.out8 = d_out8;
    a.bulk = d_out8 ? ((uintptr_t)d_out8 & 15u) == 0 && s->info.W % 16 == 0 : ((uintptr_t)d_out & 15u) == 0 && s->info.W % 4 == 0;
    const uint32_t win_bytes = p.win_bytes = d_out8 ? kWinBytesU8 : kWinBytes;
    auto kern = d_out8 ? render_native_kernel<true> : render_native_kernel<false>;
    const uint32_t plan_smem = plan_bytes(n_cells, n_views);
    int sms = 0, per_sm = 0, rc = RLFC_OK;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)win_bytes)) != cudaSuccess ||
        (plan_smem > 40u * 1024u && (e = cudaFuncSetAttribute(render_plan_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                              (int)kPlanSmemMost)) != cudaSuccess) ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, s->device)) != cudaSuccess ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, win_bytes)) != cudaSuccess)
        rc = cuda_fail(e, "render: launch configuration");
    const uint32_t resident = (uint32_t)std::max(sms, 1) * (uint32_t)std::max(per_sm, 1);
    // groups small enough for about four items per resident CTA: with fewer,
    // a last round that few CTAs take doubles the time of a small call
    p.group_cap = (uint32_t)std::min<uint64_t>(kGroup, std::max<uint64_t>(1, (uint64_t)n * a.n_tiles / (4ull * resident)));
    if (rc == RLFC_OK) {
        { TraceScope trace_("render_plan_kernel", st); render_plan_kernel<<<1, kPlanThreads, plan_smem, st>>>(p); }
        rc = launch_decode_packed(s, reinterpret_cast<uint32_t *>(scratch + at_dec), p.needed, p.slot_of, (uint32_t)n_slots, st);
    }
    if (rc == RLFC_OK && !native) {
        { TraceScope trace_("render_sampled_kernel", st); render_sampled_kernel<<<dim3((uint32_t)stiles, n), kSX * kSY, 0, st>>>(a, d_uv, d_disp, out_w, out_h, stiles_x); }
        if ((e = cudaGetLastError()) != cudaSuccess)
            rc = cuda_fail(e, "render_sampled launch");
    } else if (rc == RLFC_OK) {
        const uint32_t grid = (uint32_t)std::min<uint64_t>(resident, (uint64_t)a.n_tiles * n);
        { TraceScope trace_("render_native_kernel", st); kern<<<grid, kThreads, win_bytes, st>>>(a); }
        if ((e = cudaGetLastError()) != cudaSuccess)
            rc = cuda_fail(e, "render_windows launch");
    }
    cudaFreeAsync(scratch, st);
    return rc;
}

}  // namespace rlfc
