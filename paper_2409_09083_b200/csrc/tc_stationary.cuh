// bf16 path, executed groups of one conv layer (with its pool): the filter gradient by a weight-stationary
// tensor-core kernel, the forward pass and the input delta by a banded tensor-core convolution (further down),
// and their helpers (dz planes, loss, window unroll and input entries for the first layer).
//
// Filter gradient.  In the fused tile-stack kernel every sub-tile adds its whole partial filter gradient (K*K*cout*cin fp32) to
// the block's partial set, because tensor memory cannot keep the accumulators of a wide layer across sub-tiles.
// For layers with hundreds of channels that flush costs several times the MMAs.  Here the roles are turned
// round: a block owns a slice of the FILTER GRADIENT (64 or 128 output channels x up to 48 input channels x all
// window positions; plus 16 columns for the bias gradient) and keeps
// it in tensor memory while bands of rows of the whole batch stream past it, so the gradient leaves the SM
// once.  The pixels are dealt out in `shares`; a share is one partial gradient set of Section 4.1, summed by
// the same cross-tile reduction as the sets of the fused kernels.
//
// A band is R rows (even) x Cw columns (a multiple of 8, at most 128 tile entries with the halo) of one image at the conv's
// resolution.  The delta in front of the activation (dz, bf16 planes, written by the input-delta kernel of the layer above or by
// delta_act_planes_kernel) arrives by one TMA copy as [plane][row][Cw entries], the layer's saved input by another as
// [row][plane][Cw + K - 1 entries] with its halo; what lies outside the map arrives as zeros.  Both operands are MN-major (8
// pixels x 8 channels per core matrix).  A K step of 16 pixels is 8 pixels of a row and the 8 below them, so that only a width that
// no multiple of 8 covers is padded (38 columns: 40 instead of the 48 of 16 pixels in a row).  Because the planes of a
// row of the input lie between it and the next row, the 8-channel groups (window row ky, plane p) of ONE window column stand at one
// stride: an MMA covers the three window rows of its column, K * ncols accumulator columns, and the window column moves the
// start by an entry.  With one MMA per window position instead (48 columns each, both operands from shared memory) an MMA took
// the 44 cycles in which shared memory delivers 5.5 KB, for 24 cycles of arithmetic, and dz was read nine times
// for a K step; 144 columns take 72 cycles and dz is read three times.  Now it waits for copies: no unit is near its limit (4 images of
// 38 x 38, 256 -> 512: tensor core 33 %, L2 26 %, shared memory 39 %), but of the two stages one is read while the other's 93 KB
// arrive, at about 20 bytes a cycle and SM.  us before and after: 256 -> 512, 16 x 38 x 38: 97 -> 66 (826 TFLOP/s); 128 -> 256, 76 x 76: 81 -> 60; 64 -> 128,
// 152 x 152: 91 -> 52; 32 -> 64, 304 x 304: 112 -> 76; 256 -> 512 on 8 x 13 x 13: 40 -> 26; 1x1 512 -> 256: 29 -> 21.
// Two stages (copies of the next band behind the MMAs of this one).
#pragma once

#include <algorithm>

#include "kernels_tc.cuh"

namespace ftp {

// Tensor maps of bf16 planes [N x C16/8][H][W][8] as the TMA engine sees them here: 3-dimensional, rows of 2 W
// eight-byte elements (a pixel's 8 channels = two elements), so that a box row is one contiguous run of Wp pixels
// instead of Wp separate 16-byte pieces; a box row holds at most 256 elements, i.e. Wp <= 128 pixels.
struct TcFilterGradArgs {
    alignas(64) unsigned char tmap_dz[128];   // dz as {columns, rows, planes, images}: box = Cw columns x R rows x dz_box planes
    alignas(64) unsigned char tmap_x[128];    // the layer's input as {columns, planes, rows, images}: box = (Cw + K - 1) x ncols / 8 x (R + K - 1)
    alignas(64) unsigned char tmap_left[128]; // first layer: the same without the map's last column, for the copies of window column 0
    float* partial;                           // partial sets of the group
    long long set_floats, tgp_off;            // floats per set, offset of this layer inside a set
    int* error;
    int hurry;                                // a short launch: see kHurryCycles in launch.cuh
    int K, H, W, cout16, cin16;
    int Ms, slices;                           // output channels per block (64 or 128) and number of such slices
    int ncols, nci;                           // input channels per block (multiple of 16) and number of such slices
    int narrow;                               // first layer: x is the plane of InputEntries (ncols 8 or 16, the bias gradient its channel 7)
    int units;                                // accumulator units: 3x3: K * ncols columns, one per window column; 1x1 and the first
                                              //   layer (9 * ncols columns): row pairs in turn
    int R, Cw, ncc;                           // rows per band, columns of a band and column chunks per row band
    int bands_img, bands, shares;             // bands per image / in the batch, pixel shares
    int dz_box, x_off, stage_bytes;           // dz planes a copy brings, offset of the input tile in a stage, bytes of a stage
};

struct DeltaActPlanesArgs {
    const void* dmap; int dmap_planes;        // delta at the layer's output: bf16 planes, or fp32 NCHW (dmap_planes = 0)
    const uint4* y; const unsigned long long* arg;   // saved output (planes) and, for a fused pool, its arg-max bytes
    uint4* dz;                                // out: planes at the conv's resolution
    int N, cout, cout16, out_H, out_W, pool;
    float slope;
};

// Entry of dz for 8 channels of pixel (y, x) of an H x W output map, plane `plane` of the batch; arg: their arg-max bytes where a
// pool follows (four entries at twice the resolution), else null.
__device__ __forceinline__ void store_dz(uint4* dz, const float (&v)[8], const unsigned long long* arg, size_t plane, int y, int x, int H, int W)
{
    if (!arg) { dz[(plane * H + y) * W + x] = tcd::pack8(v); return; }
    const unsigned long long am = *arg;
    const int W2 = 2 * W;
    uint4* o = dz + (plane * (2 * H) + 2 * y) * W2 + 2 * x;
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        float z[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) z[c] = (int)((am >> (c * 8)) & 3ull) == w ? v[c] : 0.f;
        o[(w >> 1) * W2 + (w & 1)] = tcd::pack8(z);
    }
}

// dz = delta * act'(y), routed through the arg-max of a fused pool (zeros at the three other positions of a
// window): the same arithmetic and roundings as the fused backward kernel applies when it fills its dz tile.
__global__ void delta_act_planes_kernel(const __grid_constant__ DeltaActPlanesArgs A)
{
    previous_launches();
    const int planes = A.cout16 / 8;
    const size_t total = (size_t)A.N * planes * A.out_H * A.out_W;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int x = (int)(e % A.out_W); size_t t = e / A.out_W;
        const int y = (int)(t % A.out_H); t /= A.out_H;
        const int pl = (int)(t % planes); const int n = (int)(t / planes);
        float v[8], yv[8];
        if (A.dmap_planes) {
            tcd::unpack8(__ldg(static_cast<const uint4*>(A.dmap) + e), v);
        } else {
            const float* d = static_cast<const float*>(A.dmap);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int ch = pl * 8 + c;
                v[c] = ch < A.cout ? __ldg(d + (((size_t)n * A.cout + ch) * A.out_H + y) * A.out_W + x) : 0.f;
            }
        }
        tcd::unpack8(__ldg(A.y + e), yv);
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] *= yv[c] > 0.f ? 1.f : A.slope;
        store_dz(A.dz, v, A.pool ? A.arg + e : nullptr, (size_t)n * planes + pl, y, x, A.out_H, A.out_W);
    }
}

// Mean-squared-error loss of a step whose last group is a one-conv group: from the saved output (planes) and the target straight to
// that group's dz planes, and per-block partial sums of (y - t)^2.  The values are those of planes_to_nchw_kernel,
// mse_delta_kernel and delta_act_planes_kernel one after another, which moved 24 bytes a value instead of 8.  Bound: DRAM.
// us, with the kernels overlapping: 256 channels on 16 x 38 x 38, 51 -> 16; 64 images, 215 -> 70; 4 x 52 x 52, 23 -> 8.
struct LossPlanesArgs {
    const uint4* y; const unsigned long long* arg;   // saved output (planes) and, for a fused pool, its arg-max bytes
    const float* target;                             // fp32 NCHW
    uint4* dz;                                       // out: planes at the conv's resolution
    float* block_sums;
    int N, C, C16, H, W, pool;                       // output map
    float slope;
};

__global__ void __launch_bounds__(256) loss_planes_kernel(const __grid_constant__ LossPlanesArgs A)
{
    next_launch();
    previous_launches();
    __shared__ float red[256];
    const int planes = A.C16 / 8;
    const size_t HW = (size_t)A.H * A.W, total = (size_t)A.N * planes * HW, M = (size_t)A.N * A.C * HW;
    const float scale = 2.0f / (float)M;
    float sum = 0.f;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const size_t px = e % HW, t = e / HW;
        const int pl = (int)(t % planes), n = (int)(t / planes);
        const float* tg = A.target + ((size_t)n * A.C + pl * 8) * HW + px;
        float v[8], yv[8], tv[8];
        const uint4 yq = __ldg(A.y + e);
#pragma unroll
        for (int c = 0; c < 8; ++c) tv[c] = pl * 8 + c < A.C ? __ldg(tg + c * HW) : 0.f;
        tcd::unpack8(yq, yv);
        float part = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float diff = pl * 8 + c < A.C ? yv[c] - tv[c] : 0.f;
            part += diff * diff;
            v[c] = scale * diff * (yv[c] > 0.f ? 1.f : A.slope);
        }
        sum += part;
        store_dz(A.dz, v, A.pool ? A.arg + e : nullptr, t, (int)(px / A.W), (int)(px % A.W), A.H, A.W);
    }
    red[threadIdx.x] = sum;
    __syncthreads();
    for (int k = 128; k >= 1; k >>= 1) {
        if ((int)threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) A.block_sums[blockIdx.x] = red[0];
}

// First layer: the fp32 network input [N][C][H][W] -> window-unrolled bf16 planes [N][C16'/8][H][W][8] with channel
// ci * 9 + ky * 3 + kx of pixel (y, x) = input(ci, y + ky - 1, x + kx - 1) (zero outside the map and beyond 9 C).
// One thread per pixel: it reads the 9 C values of its window once and writes its entry of every plane (the
// channel -> (ci, ky, kx) arithmetic is resolved at compile time).  On that copy the forward pass is a 1x1 conv.  (On the entries
// below it is a 3x3 conv without the copy, 99 us less for 16 x 608 x 608, but the sums of an MMA are then other ones, a few
// rounded outputs in a million with them, and through the ties of the pools whole deltas at the network input.)
// ent, if not null: the entries for the backward pass (see InputEntries), written in the same pass.
template <int C>
__global__ void unroll_windows_kernel(const float* __restrict__ x, uint4* __restrict__ col, uint4* __restrict__ ent, int N, int H, int W)
{
    previous_launches();
    constexpr int planes = (9 * C + 15) / 16 * 2;
    const size_t HW = (size_t)H * W, total = (size_t)N * HW;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int px = (int)(e % W); size_t t = e / W;
        const int py = (int)(t % H); const int n = (int)(t / H);
        float v[planes * 8];
        const float* ctr = x + (size_t)n * C * HW + (size_t)py * W + px;       // this pixel in channel 0
        if (py > 0 && py < H - 1 && px > 0 && px < W - 1) {                    // the whole window lies inside the map
#pragma unroll
            for (int j = 0; j < planes * 8; ++j) {
                const int ci = j / 9, tap = j - ci * 9, ky = tap / 3, kx = tap - ky * 3;
                v[j] = ci < C ? __ldg(ctr + (size_t)ci * HW + (ky - 1) * W + (kx - 1)) : 0.f;
            }
        } else {
#pragma unroll
            for (int j = 0; j < planes * 8; ++j) {
                const int ci = j / 9, tap = j - ci * 9, ky = tap / 3, kx = tap - ky * 3;
                const int yy = py + ky - 1, xx = px + kx - 1;
                v[j] = (ci < C && yy >= 0 && yy < H && xx >= 0 && xx < W) ? __ldg(ctr + (size_t)ci * HW + (ky - 1) * W + (kx - 1)) : 0.f;
            }
        }
#pragma unroll
        for (int pl = 0; pl < planes; ++pl) col[((size_t)n * planes + pl) * HW + (size_t)py * W + px] = tcd::pack8(v + 8 * pl);
        if (ent) {
            float c[8];
#pragma unroll
            for (int ci = 0; ci < 7; ++ci) c[ci] = ci < C ? v[ci < C ? ci * 9 + 4 : 0] : 0.f;
            c[7] = 1.f;
            ent[e] = tcd::pack8(c);
        }
    }
}

// for the channel counts the route takes (9 C <= 64)
inline void launch_unroll_windows(const float* x, uint4* col, uint4* ent, int N, int C, int H, int W, LaunchStream st)
{
    const int blocks = (int)std::min<size_t>(((size_t)N * H * W + 255) / 256, (size_t)kSmCount * 16);
    switch (C) {
        case 1: launch(unroll_windows_kernel<1>, blocks, 256, 0, st, x, col, ent, N, H, W); break;
        case 2: launch(unroll_windows_kernel<2>, blocks, 256, 0, st, x, col, ent, N, H, W); break;
        case 3: launch(unroll_windows_kernel<3>, blocks, 256, 0, st, x, col, ent, N, H, W); break;
        case 4: launch(unroll_windows_kernel<4>, blocks, 256, 0, st, x, col, ent, N, H, W); break;
        case 5: launch(unroll_windows_kernel<5>, blocks, 256, 0, st, x, col, ent, N, H, W); break;
        case 6: launch(unroll_windows_kernel<6>, blocks, 256, 0, st, x, col, ent, N, H, W); break;
        default: launch(unroll_windows_kernel<7>, blocks, 256, 0, st, x, col, ent, N, H, W); break;
    }
}

constexpr int kTcFgThreads = 256;

__global__ void __launch_bounds__(kTcFgThreads, 1) filter_grad_tc_rows_kernel(const __grid_constant__ TcFilterGradArgs A)
{
    using namespace tc;
    extern __shared__ __align__(1024) unsigned char fg_smem[];
    struct Hdr {
        unsigned long long full[2], empty[2], done;
        uint32_t tmem_base;
        volatile int failed;
        __align__(16) __nv_bfloat16 ones[64];
    };
    static_assert(sizeof(Hdr) <= kTcFgHeader, "header does not fit");
    Hdr* H = reinterpret_cast<Hdr*>(fg_smem);
    unsigned char* stages = fg_smem + kTcFgHeader;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int K = A.K, KK = K * K;

    // this block's slice of the gradient and share of the bands
    const int nroles = A.slices * A.nci;
    const int role = (int)blockIdx.x % nroles, share = (int)blockIdx.x / nroles;
    const int slice = role / A.nci, cs = role - slice * A.nci;
    const int ci0 = cs * A.ncols, cols = min(A.ncols, A.cin16 - ci0), wide = (A.narrow ? 9 : K) * A.ncols;
    const int b_lo = (int)((long long)share * A.bands / A.shares), b_hi = (int)((long long)(share + 1) * A.bands / A.shares);
    const int nb = b_hi - b_lo;
    // input tile: planes, entries of a plane's row, entries from row to row.  First layer: each row three times, shifted by the window
    // column, in the place of planes, so that all nine window positions of its few channels stand at one stride and share an
    // MMA (on the unrolled copy with K = 1 144 us a launch for 16 x 608 x 608, 3 -> 32; with three MMAs of 24 columns 142; now 101, 479 MB).
    const bool turns = K == 1 || A.narrow;
    const int np = A.ncols / 8, Wx = A.narrow ? A.Cw : A.Cw + K - 1, pitch = (A.narrow ? 3 : 1) * np * Wx;
    // Pixels that only fill up a K step have zero dz, and a zero times an infinite input is NaN: they must not meet pixels of the map.
    // Columns: the first layer's copies of window column 0 leave out the last column, which only the window columns 1 and 2 of
    // a pixel read (elsewhere a row of the tile serves all window columns, and such a value at the end of a row shows).
    // Rows: where the last row of an odd height stands alone, the second half of its K steps reads the input two rows on instead of one,
    // below the map for all window rows; at the last row of a band that is one row behind the copied tile, zeros from here on.
    const bool odd_h = K == 3 && (A.H & 1);

    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) { mbar_init(smem_u32(&H->full[s]), 1); mbar_init(smem_u32(&H->empty[s]), kTcIssuers); }
        mbar_init(smem_u32(&H->done), kTcIssuers);
        H->failed = 0;
        fence_mbar_init();
    }
    if (warp == 0) { __syncwarp(); tmem_alloc(smem_u32(&H->tmem_base), (uint32_t)kTcTmemCols); }
    for (int i = threadIdx.x; i < 64; i += blockDim.x) H->ones[i] = __float2bfloat16(1.0f);
    if (odd_h)
        for (int s = 0; s < 2; ++s) tcd::zero_bytes(stages + (size_t)s * A.stage_bytes + A.x_off + (size_t)(A.R + K - 1) * pitch * 16, (size_t)pitch * 16);
    fence_async_smem();
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    previous_launches();
    const uint32_t tmem = H->tmem_base;

    auto wait = [&](unsigned long long* bar, uint32_t parity, unsigned sleep_ns = 0) {
        if (H->failed) return false;
        if (mbar_wait(smem_u32(bar), parity, kWaitLimitCycles, sleep_ns)) return true;
        H->failed = 1;
        atomicExch(A.error, 1);
        return false;
    };
    if ((smem_u32(fg_smem) & 127u) != 0) {                  // tensor copies want 128-byte aligned destinations
        if (threadIdx.x == 0) { H->failed = 1; atomicExch(A.error, 1); }
        __syncthreads();
    }
    // image and origin of band b of the batch
    auto band_of = [&](int b, int& n, int& y0, int& x0) {
        n = b / A.bands_img;
        const int bi = b - n * A.bands_img, rb = bi / A.ncc;
        y0 = rb * A.R; x0 = (bi - rb * A.ncc) * A.Cw;
    };
    auto pairs_of = [&](int y0) { return (min(A.R, A.H - y0) + 1) >> 1; };       // row pairs with pixels

    if (warp == kTcIssuers && lane == 0) {
        // producer: the two tiles of a band, one tensor copy each
        int issued[2] = {0, 0};
        for (int i = 0; i < nb; ++i) {
            const int s = i & 1;
            if (!wait(&H->empty[s], ((uint32_t)(i >> 1) & 1u) ^ 1u)) break;
            int n, y0, x0;
            band_of(b_lo + i, n, y0, x0);
            const uint32_t dst = smem_u32(stages + (size_t)s * A.stage_bytes), bar = smem_u32(&H->full[s]);
            mbar_expect_tx(bar, (uint32_t)(A.dz_box * A.R * A.Cw + (A.R + K - 1) * pitch) * 16u);
            tma_load_4d(dst, A.tmap_dz, 2 * x0, y0, slice * (A.Ms / 8), n, bar);
            if (A.narrow)
                for (int r = 0; r < A.R + 2; ++r)
                    for (int kx = 0; kx < 3; ++kx)      // (a map of one column: window column 0 has none, a box in front of the map)
                        tma_load_4d(dst + (uint32_t)(A.x_off + (r * 3 + kx) * np * Wx * 16), kx ? A.tmap_x : A.tmap_left,
                                    2 * (A.W == 1 && kx == 0 ? -A.Cw : x0 + kx - 1), 0, y0 + r - 1, n, bar);
            else
                tma_load_4d(dst + (uint32_t)A.x_off, A.tmap_x, 2 * (x0 - K / 2), ci0 / 8, y0 - K / 2, n, bar);
            ++issued[s];
        }
        if (H->failed)       // gave up somewhere: let the copies already under way land before the block leaves
            for (int s = 0; s < 2; ++s)
                if (issued[s] > 0) mbar_wait(smem_u32(&H->full[s]), (uint32_t)(issued[s] - 1) & 1u, 200000000ll);
    } else if (warp < kTcIssuers && lane == 0) {
        // MMA issue: issuers 0 .. units - 1 an accumulator unit each, the last one the bias gradient (dz against ones).
        // A block takes the bias of every nci-th row pair, so that the blocks of a share, one per slice of the input channels,
        // have the same work; the reduction adds their parts.
        const bool is_bias = warp == kTcIssuers - 1;
        const uint32_t a_hi = desc_hi((uint32_t)(A.R * A.Cw) * 16u), x_hi = is_bias ? desc_hi(0) : desc_hi((uint32_t)Wx * 16u);
        const uint32_t idesc = make_idesc(A.Ms, is_bias ? 16 : wide, true, true);
        const uint32_t col = tmem + (uint32_t)((is_bias ? A.units : warp) * wide);
        const uint32_t a_pair = 2u * (uint32_t)A.Cw, x_pair = is_bias ? 0u : 2u * (uint32_t)pitch, x_step = is_bias ? 0u : 8u;
        const int every = is_bias ? A.nci : turns ? A.units : 1, first = is_bias ? cs : turns ? warp : 0;
        bool acc = false;
        int turn = first;                                    // row pairs until this issuer's next one
        for (int i = 0; i < nb; ++i) {
            const int s = i & 1;
            if (!wait(&H->full[s], (uint32_t)(i >> 1) & 1u)) break;
            fence_after_sync();
            if (is_bias ? !A.narrow : warp < A.units) {
                int n, y0, x0;
                band_of(b_lo + i, n, y0, x0);
                const uint32_t dst = smem_u32(stages + (size_t)s * A.stage_bytes);
                uint32_t ar = desc_lo(dst, (uint32_t)A.Cw * 16u);
                uint32_t xr = is_bias ? desc_lo(smem_u32(H->ones), 0)
                                      : desc_lo(dst + (uint32_t)A.x_off, (uint32_t)pitch * 16u) + (turns ? 0u : (uint32_t)warp);
                const int pairs = pairs_of(y0), groups = (min(A.Cw, A.W - x0) + 7) >> 3;
                const int alone = odd_h && !is_bias && A.H - y0 < A.R ? pairs - 1 : -1;       // the pair of a last row without a second
                for (int r = 0; r < pairs; ++r, ar += a_pair, xr += x_pair) {
                    if (turn > 0) { --turn; continue; }
                    turn = every - 1;
                    uint32_t a = ar, x = r == alone ? xr + ((uint32_t)pitch << 16) : xr;     // (desc_lo's stride: two rows)
#pragma unroll 4
                    for (int g = 0; g < groups; ++g, a += 8u, x += x_step) {
                        mma_bf16(col, desc64(a_hi, a), desc64(x_hi, x), idesc, acc);
                        acc = true;
                    }
                }
            }
            mma_commit(smem_u32(&H->empty[s]));
        }
        mma_commit(smem_u32(&H->done));
    }
    __syncwarp();
    const bool have = nb > 0 && wait(&H->done, 0, 256);        // (asleep between polls: the issuers share the schedulers)
    if (!have && nb > 0) mbar_wait(smem_u32(&H->done), 0, 200000000ll);   // gave up: the MMAs under way still end first
    fence_after_sync();

    if (A.hurry) next_launch();

    // what a block of few row pairs never touched: units and the bias beyond the number of its pairs
    int pairs = 0;
    for (int i = 0; i < nb && pairs <= max(A.units, cs); ++i) {
        int n, y0, x0;
        band_of(b_lo + i, n, y0, x0);
        pairs += pairs_of(y0);
    }
    const int used = !have ? 0 : turns ? min(A.units, pairs) : 1;

    // tensor memory -> this share's partial set; lane quarter q holds rows 32q.. (Ms = 128) or rows 16q.. in its
    // first 16 lanes (Ms = 64).  The slices of the blocks are disjoint: plain stores.
    const int q = warp & 3, half = warp >> 2;
    const int row = A.Ms == 128 ? q * 32 + lane : q * 16 + lane;
    const bool row_ok = (A.Ms == 128 || lane < 16) && slice * A.Ms + row < A.cout16;
    const int co = slice * A.Ms + row;
    const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
    float* gset = A.partial + (size_t)share * A.set_floats + A.tgp_off;
    for (int u = 0; u < KK; ++u) {
        const int ky = u / K, kx = u - ky * K;
        for (int c0 = half * 16; c0 < cols; c0 += 32) {
            float v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = 0.f;
            for (int w = 0; w < used; ++w) {
                float t[16];
                tmem_ld16(tq + (uint32_t)((turns ? w : kx) * wide + (A.narrow ? u : ky) * A.ncols + c0), t);
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = w ? v[j] + t[j] : t[j];
            }
            if (row_ok) {
                float* g = gset + ((size_t)u * A.cout16 + co) * A.cin16 + ci0 + c0;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (c0 + 4 * j < cols) *reinterpret_cast<float4*>(g + 4 * j) = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            }
        }
    }
    if (half == 0) {
        float v[16];
        v[0] = 0.f;
        if (A.narrow) {
            float sum = 0.f;
            for (int w = 0; w < used; ++w) { tmem_ld16(tq + (uint32_t)(w * wide + 4 * A.ncols), v); sum += v[7]; }
            v[0] = sum;
        }
        else if (have && pairs > cs) tmem_ld16(tq + (uint32_t)(A.units * wide), v);
        if (row_ok) gset[(size_t)KK * A.cout16 * A.cin16 + (size_t)cs * A.cout16 + co] = v[0];
    }
    fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, (uint32_t)kTcTmemCols);
}

// ---------------------------------------------------------------------------------------------
// Convolution of a one-conv group over bands of rows (forward pass, and the input delta as the convolution of dz
// with the rotated filters).  A work item is a band of R rows x Cw columns of one image x a slice of Ns output
// channels: up to 512 / Ns accumulator blocks of 128 consecutive tile entries (pitch Wp = Cw + K - 1, so the entries
// of a block are pixels of consecutive rows with K - 1 discarded positions between them) stay in tensor memory
// while the input channels stream past in chunks: per chunk one tile of `kpc` 8-channel planes of the band (with
// its K - 1 halo rows, TMA tensor copies) and the filters of those channels for the slice (one bulk copy),
// through a ring of stages.  Window position (ky, kx) moves the A operand by ky * Wp + kx entries.  Against the
// fused sub-tile kernel, whose sub-tiles follow the tile grid (64 pixels a tile on the deepest maps) and which
// streams all filters of the layer once per 128 pixels, the filters read per pixel shrink by the number of
// accumulator blocks and the pixels per block no longer depend on the grid.
//
// Persistent blocks (one per SM) walk over the items; the warps have fixed roles: warps 0-15 read the accumulators
// back (bias, leaky ReLU, bf16 planes; with a fused 2x2 pool the first maximum in window order, with the arg-max bytes the
// backward pass routes deltas by: from accumulator blocks of one row in registers, from blocks of 128 entries through a staging
// area, 16 channels or more at a time), lane 0 of warps 16-19 issues the MMAs (each for its own accumulator blocks), lane 0 of
// warp 20 issues the copies and runs ahead into the next item while the accumulators of the current one are read back.
// ---------------------------------------------------------------------------------------------
struct TcConvRowsArgs {
    alignas(64) unsigned char tmap_x[128];    // input planes (rows of 2 W eight-byte elements): box = Wp pixels x (R + K - 1) rows
    const __nv_bfloat16* w;                   // filters of the layer, [slice][chunk][window position][kpc][Ns][8]: the
                                              //   filters a block needs for one chunk are one contiguous run
    const float* bias;                        // cout floats, or null
    uint4* out;                               // output planes [N][cout16/8][OH][OW] (OH = H / 2 with the pool)
    unsigned long long* arg;                  // pool: arg-max bytes in the same arrangement
    int* error;
    int hurry;                                // a short launch: see kHurryCycles in launch.cuh
    int N, K, cin16, cout16, cout, H, W;
    float slope;
    int Ns, slices;                           // output channels per item, number of slices
    int R, Wp, bands_img, nblk;               // rows per band, tile pitch, bands per image, accumulator blocks of a full band
    int share;                                // stack: output rows of an issuer
    int ncc, Cw;                              // column chunks per row band and their width (even with the pool; Wp = Cw + K - 1)
    int kpc;                                  // 8-channel planes per chunk (3x3: 2, or 4 with narrow slices; 1x1: up to 8)
    int x_plane, stage_bytes, stages;
    int items;                                // N * bands_img * slices
    int pool_planes;                          // pool: 8-channel planes the staging area holds (even)
    // input delta only: when the layer below is a one-conv group too, the delta goes straight into ITS dz planes (`out`;
    // at twice the resolution if it ends with a pool): prev_y = that layer's saved output (= this conv's output shape),
    // prev_arg = its pool's arg-max bytes or null, prev_slope = its leaky slope.  prev_y null: plain delta planes.
    const uint4* prev_y; const unsigned long long* prev_arg; float prev_slope;
    float* out_f;                             // fp32 NCHW output in the place of planes (delta at the network input), else null
    // forms of the kernel: accumulator blocks of 128 consecutive entries (plain, pool), or one per row of the band: with a pool, or, 3x3 with
    // slices of 16 channels, with the window rows in one MMA (stack; see the issuers)
    int nbuf;                                 // accumulator buffers (2: items of at most 256 columns alternate between the halves
                                              //   of the tensor memory, so the MMAs of one run while the other is read back)
};

constexpr int kTcConvMaxStages = 4;
constexpr int kTcConvEpiWarps = 16;           // four per lane quarter of the tensor memory
constexpr int kTcConvEpiThreads = kTcConvEpiWarps * 32;
constexpr int kTcConvThreads = (kTcConvEpiWarps + kTcIssuers + 1) * 32;

// bias and leaky ReLU of 8 accumulators, rounded: both sides of the activation are formed and rounded, the sign of the sum picks, which a
// sum that rounds to zero keeps: with a slope above 1 a positive one must not become slope times itself (3 instructions a value instead of 5.5: pairs are added, multiplied, rounded and selected together; an epilogue warp is bound by
// instruction issue).
__device__ __forceinline__ uint4 act8(const float* v, const float* bias, float slope)
{
    const float2 s2 = make_float2(slope, slope);
    uint32_t o[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const float4 b = *reinterpret_cast<const float4*>(bias + 4 * h);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float2 z = __fadd2_rn(make_float2(v[4 * h + 2 * j], v[4 * h + 2 * j + 1]), j ? make_float2(b.z, b.w) : make_float2(b.x, b.y));
            const float2 n = __fmul2_rn(z, s2);
            const __nv_bfloat162 zb = __float22bfloat162_rn(z), nb = __float22bfloat162_rn(n);
            const uint32_t zw = *reinterpret_cast<const uint32_t*>(&zb);
            uint32_t m;
            asm("prmt.b32 %0, %1, 0, 0xBB99;" : "=r"(m) : "r"(zw));      // the halves' signs, spread over their bits
            o[2 * h + j] = (*reinterpret_cast<const uint32_t*>(&nb) & m) | (zw & ~m);
        }
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// 8 deltas times the derivative of the layer below (1 where its stored output y is positive, else its slope), rounded
__device__ __forceinline__ uint4 derive8(const uint4& d, const uint4& y, float slope)
{
    const uint32_t dw[4] = {d.x, d.y, d.z, d.w}, yw[4] = {y.x, y.y, y.z, y.w};
    const float2 s2 = make_float2(slope, slope);
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 n = __fmul2_rn(make_float2(__uint_as_float(dw[j] << 16), __uint_as_float(dw[j] & 0xffff0000u)), s2);
        const __nv_bfloat162 nb = __float22bfloat162_rn(n);
        const uint32_t m = __hgt2_mask(*reinterpret_cast<const __nv_bfloat162*>(&yw[j]), __nv_bfloat162(__ushort_as_bfloat16(0), __ushort_as_bfloat16(0)));
        o[j] = (dw[j] & m) | (*reinterpret_cast<const uint32_t*>(&nb) & ~m);
    }
    return make_uint4(o[0], o[1], o[2], o[3]);
}

// Two neighbouring entries, the first at an even index of a 256-byte aligned area.
__device__ __forceinline__ void store_pair(uint4* dst, const uint4& a, const uint4& b)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 :: "l"(dst), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w) : "memory");
}

// 2x2 maximum of 8 channels (bf16 pairs, compared as stored, two channels per instruction): the first maximum in window order,
// i.e. a later member wins only if it is greater; returns the members' numbers, a byte per channel.
__device__ __forceinline__ unsigned long long pool4(const uint4& m0, const uint4& m1, const uint4& m2, const uint4& m3, uint4& best)
{
    const uint32_t w[4][4] = {{m0.x, m1.x, m2.x, m3.x}, {m0.y, m1.y, m2.y, m3.y}, {m0.z, m1.z, m2.z, m3.z}, {m0.w, m1.w, m2.w, m3.w}};
    uint32_t val[4], code[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t m = w[j][0], a = 0u;
#pragma unroll
        for (int k = 1; k < 4; ++k) {
            const uint32_t gt = __hgt2_mask(*reinterpret_cast<const __nv_bfloat162*>(&w[j][k]), *reinterpret_cast<const __nv_bfloat162*>(&m));
            m = (w[j][k] & gt) | (m & ~gt);
            a = (((uint32_t)k * 0x00010001u) & gt) | (a & ~gt);
        }
        val[j] = m; code[j] = a;
    }
    best = make_uint4(val[0], val[1], val[2], val[3]);
    // channel 2j in the low half of code[j], channel 2j + 1 in the high half
    return (unsigned long long)__byte_perm(code[0], code[1], 0x6420) | ((unsigned long long)__byte_perm(code[2], code[3], 0x6420) << 32);
}

// One instance per form of the epilogue and the issue: a launch waits for its instructions too, and no instance spills (8 layers, 4
// images: a step 283 us as one kernel with all forms, 276 so; the fp32 output inside the plain form: 64 -> 1024 forward on 7 x 84 x 116 416 us,
// without 415).
enum { kConvPlain, kConvPool, kConvInput, kConvRowPool, kConvStack };      // (input, stack: the delta at the network input, out_f)

template <int FORM>
__global__ void __launch_bounds__(kTcConvThreads, 1) conv_tc_rows_kernel(const __grid_constant__ TcConvRowsArgs A)
{
    using namespace tc;
    extern __shared__ __align__(1024) unsigned char cv_smem[];
    struct Hdr {
        unsigned long long full[kTcConvMaxStages], empty[kTcConvMaxStages];
        unsigned long long done[2];     // the MMAs of an item have completed (one commit per issuer), per accumulator buffer
        unsigned long long tfree[2];    // its accumulators have been read back (one arrival per epilogue warp)
        unsigned long long drain;       // all MMAs of the block have completed
        uint32_t tmem_base;
        volatile int failed;
        volatile int epi_stop[2];       // the epilogue warps' common view of `failed` (they meet at named barriers), items in turn
        __align__(16) float bias[128];
    };
    static_assert(sizeof(Hdr) <= kTcFgHeader, "header does not fit");
    Hdr* H = reinterpret_cast<Hdr*>(cv_smem);
    unsigned char* stages = cv_smem + kTcFgHeader;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int K = A.K, KK = K * K;
    const int kplanes = A.cin16 / 8, nchunks = (kplanes + A.kpc - 1) / A.kpc;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kTcConvMaxStages; ++s) { mbar_init(smem_u32(&H->full[s]), 1); mbar_init(smem_u32(&H->empty[s]), kTcIssuers); }
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&H->done[i]), kTcIssuers); mbar_init(smem_u32(&H->tfree[i]), kTcConvEpiWarps); }
        mbar_init(smem_u32(&H->drain), kTcIssuers);
        H->failed = 0;
        fence_mbar_init();
    }
    if (warp == 0) { __syncwarp(); tmem_alloc(smem_u32(&H->tmem_base), (uint32_t)kTcTmemCols); }
    tcd::zero_bytes(stages, (size_t)A.stages * A.stage_bytes);       // what the copies never write is read as zeros
    fence_async_smem();
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    previous_launches();
    const uint32_t tmem = H->tmem_base;

    auto wait = [&](unsigned long long* bar, uint32_t parity, unsigned sleep_ns = 0) {
        if (H->failed) return false;
        if (mbar_wait(smem_u32(bar), parity, kWaitLimitCycles, sleep_ns)) return true;
        H->failed = 1;
        atomicExch(A.error, 1);
        return false;
    };
    if ((smem_u32(cv_smem) & 127u) != 0) {                  // tensor copies want 128-byte aligned destinations
        if (threadIdx.x == 0) { H->failed = 1; atomicExch(A.error, 1); }
        __syncthreads();
    }
    // item -> (slice, image, band origin); every role walks the same sequence of items
    struct Item { int slice, n, y0, x0, rows, cw, co0, cols, nblk; };
    auto item_of = [&](int it) {
        Item I;
        I.slice = it % A.slices;
        const int band = it / A.slices;
        I.n = band / A.bands_img;
        const int bi = band - I.n * A.bands_img;
        I.y0 = (bi / A.ncc) * A.R; I.x0 = (bi % A.ncc) * A.Cw;
        I.rows = min(A.R, A.H - I.y0); I.cw = min(A.Cw, A.W - I.x0);
        I.co0 = I.slice * A.Ns; I.cols = min(A.Ns, A.cout16 - I.co0);
        I.nblk = FORM >= kConvRowPool ? I.rows : (I.rows * A.Wp + 127) >> 7;
        return I;
    };
    const uint32_t w_tap = (uint32_t)A.kpc * (uint32_t)A.Ns * 16u;                      // filter bytes of one window position
    const uint32_t w_chunk = (uint32_t)KK * w_tap;

    if (warp == kTcConvEpiWarps + kTcIssuers) {
        if (lane == 0) {
            // producer
            int issued[kTcConvMaxStages] = {0, 0, 0, 0};
            uint32_t g = 0;                                                             // chunks issued so far
            for (int it = blockIdx.x; it < A.items && !H->failed; it += gridDim.x) {
                const Item I = item_of(it);
                for (int c = 0; c < nchunks; ++c, ++g) {
                    const int s = (int)(g % (uint32_t)A.stages);
                    if (!wait(&H->empty[s], ((g / (uint32_t)A.stages) & 1u) ^ 1u)) break;
                    const int kp0 = c * A.kpc, np = min(A.kpc, kplanes - kp0);
                    unsigned char* xs = stages + (size_t)s * A.stage_bytes;
                    unsigned char* ws = xs + (size_t)A.kpc * A.x_plane;
                    const uint32_t bar = smem_u32(&H->full[s]);
                    mbar_expect_tx(bar, (uint32_t)(np * (A.R + K - 1) * A.Wp) * 16u + w_chunk);
                    for (int pl = 0; pl < np; ++pl)
                        tma_load_3d(smem_u32(xs + (size_t)pl * A.x_plane), A.tmap_x, 2 * (I.x0 - K / 2), I.y0 - K / 2,
                                    I.n * kplanes + kp0 + pl, bar);
                    bulk_g2s(smem_u32(ws), A.w + ((size_t)I.slice * nchunks + c) * (w_chunk / 2), w_chunk, bar);
                    ++issued[s];
                }
            }
            if (H->failed)       // gave up somewhere: let the copies already under way land before the block leaves
                for (int s = 0; s < A.stages; ++s)
                    if (issued[s] > 0) mbar_wait(smem_u32(&H->full[s]), (uint32_t)(issued[s] - 1) & 1u, 200000000ll);
        }
    } else if (warp >= kTcConvEpiWarps) {
        if (lane == 0) {
            // MMA issue: every issuer takes every kTcIssuers-th accumulator block; K-major operands: 8 pixels (or 8
            // output channels) x 16 bytes per core matrix, the next 8 rows 128 bytes on, the next 8 channels one plane on
            const int iw = warp - kTcConvEpiWarps;
            const uint32_t a_hi = desc_hi(128), b_hi = desc_hi(128);
            const uint32_t xstep = 2u * ((uint32_t)A.x_plane >> 4), wstep = 2u * (uint32_t)A.Ns;   // one K step, 16-byte units
            const uint32_t w_tap16 = w_tap >> 4;
            uint32_t g = 0, k = 0;
            for (int it = blockIdx.x; it < A.items && !H->failed; it += gridDim.x, ++k) {
                const Item I = item_of(it);
                const uint32_t idesc = make_idesc(128, I.cols, false, false);
                const uint32_t buf = k % (uint32_t)A.nbuf, use = k / (uint32_t)A.nbuf;  // accumulator buffer and how often it was used
                if (use > 0 && !wait(&H->tfree[buf], (use - 1) & 1u)) break;            // its accumulators have been read back
                fence_after_sync();
                for (int c = 0; c < nchunks; ++c, ++g) {
                    const int s = (int)(g % (uint32_t)A.stages);
                    if (!wait(&H->full[s], (g / (uint32_t)A.stages) & 1u)) break;
                    fence_after_sync();
                    const int nks = min(A.kpc, kplanes - c * A.kpc) >> 1;
                    const uint32_t xaddr = smem_u32(stages + (size_t)s * A.stage_bytes), waddr = xaddr + (uint32_t)(A.kpc * A.x_plane);
                    const uint32_t b_lo0 = desc_lo(waddr, (uint32_t)A.Ns * 16u);
                    if constexpr (FORM == kConvStack) {
                        // An MMA reads 4 KB of A however narrow it is: with 16 columns it takes 36 cycles, with 48 44.  An input row
                        // belongs to the three output rows around it, whose accumulators are neighbouring columns, so it meets
                        // the filters of up to three window rows (packed bottom row first) in one MMA.  An issuer has up to four output
                        // rows of its own (A.share); a row's accumulators start with the input row above it.
                        const uint32_t wp = (uint32_t)A.Wp, kxw = (uint32_t)A.kpc * 48u;
                        const int s0 = iw * A.share, n = min(4, min(A.share, I.rows - s0));      // (a bound that the compiler sees: the rows unroll)
                        const uint32_t a0 = desc_lo(xaddr, (uint32_t)A.x_plane) + (uint32_t)s0 * wp, w0 = desc_lo(waddr, 768u);
                        const uint32_t d0 = tmem + buf * 256u + (uint32_t)s0 * 16u;
                        for (int kx = 0; kx < 3; ++kx)
                            for (int ks = 0; ks < nks; ++ks) {
                                const uint32_t w = w0 + (uint32_t)kx * kxw + (uint32_t)ks * 96u;
                                const bool fresh = (c | kx | ks) == 0;
                                uint32_t a = a0 + (uint32_t)kx + (uint32_t)ks * xstep;
                                for (int r = 0; n > 0 && r < n + 2; ++r, a += wp) {          // input row s0 + r - 1: output rows r - 2 .. r of the issuer
                                    const int lo = max(r - 2, 0), hi = min(r, n - 1);
                                    const bool first = fresh && r < n;                       // output row r begins
                                    const int joint = hi - lo + (first ? 0 : 1);
                                    const uint32_t wl = w + (uint32_t)(lo + 2 - r) * 16u;
                                    if (joint > 0) mma_bf16(d0 + (uint32_t)lo * 16u, desc64(a_hi, a), desc64(b_hi, wl), make_idesc(128, joint * 16, false, false), true);
                                    if (first) mma_bf16(d0 + (uint32_t)r * 16u, desc64(a_hi, a), desc64(b_hi, w + 32u), make_idesc(128, 16, false, false), false);
                                }
                            }
                    } else {
                    // (the thread that issues is the bottleneck of a narrow MMA: descriptors advance by adds only)
                    for (int b = iw; b < I.nblk; b += kTcIssuers) {
                        const uint32_t tcol = tmem + buf * 256u + (uint32_t)(b * A.Ns);
                        const uint32_t a0 = desc_lo(xaddr + (uint32_t)(b * (FORM >= kConvRowPool ? A.Wp : 128)) * 16u, (uint32_t)A.x_plane);
                        if (K == 3) {
                            // nine MMAs per K step, one per window position, written out: the issuing thread runs a few dozen
                            // instructions per MMA if it has to loop, and then it, not the tensor core, sets the pace
                            // (measured: an MMA every 100 cycles with the loops, every 40-64 with straight-line code)
                            const uint32_t wp = (uint32_t)A.Wp;
                            uint32_t a = a0, w0 = b_lo0;
                            for (int ks = 0; ks < nks; ++ks, a += xstep, w0 += wstep) {
                                mma_bf16(tcol, desc64(a_hi, a), desc64(b_hi, w0), idesc, (c | ks) != 0);
                                mma_bf16(tcol, desc64(a_hi, a + 1), desc64(b_hi, w0 + w_tap16), idesc, true);
                                mma_bf16(tcol, desc64(a_hi, a + 2), desc64(b_hi, w0 + 2 * w_tap16), idesc, true);
                                mma_bf16(tcol, desc64(a_hi, a + wp), desc64(b_hi, w0 + 3 * w_tap16), idesc, true);
                                mma_bf16(tcol, desc64(a_hi, a + wp + 1), desc64(b_hi, w0 + 4 * w_tap16), idesc, true);
                                mma_bf16(tcol, desc64(a_hi, a + wp + 2), desc64(b_hi, w0 + 5 * w_tap16), idesc, true);
                                mma_bf16(tcol, desc64(a_hi, a + 2 * wp), desc64(b_hi, w0 + 6 * w_tap16), idesc, true);
                                mma_bf16(tcol, desc64(a_hi, a + 2 * wp + 1), desc64(b_hi, w0 + 7 * w_tap16), idesc, true);
                                mma_bf16(tcol, desc64(a_hi, a + 2 * wp + 2), desc64(b_hi, w0 + 8 * w_tap16), idesc, true);
                            }
                        } else {
                            uint32_t a_lo = a0, b_lo = b_lo0;
                            bool acc = c > 0;
                            for (int ks = 0; ks < nks; ++ks) {
                                mma_bf16(tcol, desc64(a_hi, a_lo), desc64(b_hi, b_lo), idesc, acc);
                                acc = true; a_lo += xstep; b_lo += wstep;
                            }
                        }
                    }
                    }
                    mma_commit(smem_u32(&H->empty[s]));
                }
                mma_commit(smem_u32(&H->done[buf]));
            }
            mma_commit(smem_u32(&H->drain));
        }
    } else {
        // epilogue warps: lane quarter q = warp % 4 of every accumulator block
        const int q = warp & 3, part = warp >> 2;                  // the warps of a quarter share its (block, 16 columns) units
        constexpr int kParts = kTcConvEpiWarps / 4;
        const int oplanes = A.cout16 / 8;
        const float slope = A.slope;
        const int E = A.nblk * 128;                                   // entries per plane of the pooling layout
        uint4* S = reinterpret_cast<uint4*>(stages + (size_t)A.stages * A.stage_bytes);
        const int et = threadIdx.x;                                   // 0 .. kTcConvEpiThreads - 1
        uint32_t k = 0;
        // one slice of output channels: its bias is fetched once, and an item costs the epilogue warps one barrier (the
        // stop word of item k is written before that barrier and read behind it; its slot is written again two items
        // on, behind the barrier of the item between, at which every thread has read it)
        const bool one_slice = A.slices == 1;
        if (one_slice)
            for (int c = et; c < A.Ns; c += kTcConvEpiThreads) H->bias[c] = (A.bias && c < A.cout) ? __ldg(A.bias + c) : 0.f;
        for (int it = blockIdx.x; it < A.items; it += gridDim.x, ++k) {
            const Item I = item_of(it);
            if (!one_slice) {
                asm volatile("bar.sync 1, %0;" :: "n"(kTcConvEpiThreads) : "memory");        // every warp is through with the bias of the item before
                for (int c = et; c < A.Ns; c += kTcConvEpiThreads) H->bias[c] = (A.bias && I.co0 + c < A.cout) ? __ldg(A.bias + I.co0 + c) : 0.f;
            }
            if (et == 0) H->epi_stop[k & 1u] = H->failed;
            asm volatile("bar.sync 1, %0;" :: "n"(kTcConvEpiThreads) : "memory");
            if (H->epi_stop[k & 1u]) break;                           // the same answer for all epilogue threads: they leave together
            const uint32_t buf = k % (uint32_t)A.nbuf, use = k / (uint32_t)A.nbuf;
            const uint32_t tbuf = tmem + buf * 256u;
            wait(&H->done[buf], use & 1u, 128);                       // asleep between polls; (ran out: the item is written from
                                                                      // whatever is there; the error word is set)
            fence_after_sync();
            if constexpr (FORM == kConvPlain || FORM == kConvInput || FORM == kConvStack) {
                const int nc = I.cols >> 4, nunits = I.nblk * nc;
                const size_t gstep = (size_t)A.H * A.W;
                // where unit u (accumulator block b, channels c0 .. c0 + 15) of this thread lies in the output planes
                auto place = [&](int u, int& b, int& c0, size_t& g0, int& r, int& c) {
                    b = u / nc; c0 = (u - b * nc) << 4;
                    const int p = b * 128 + q * 32 + lane;
                    r = FORM == kConvStack ? b : p / A.Wp; c = FORM == kConvStack ? q * 32 + lane : p - r * A.Wp;
                    g0 = (((size_t)I.n * oplanes + ((I.co0 + c0) >> 3)) * A.H + I.y0 + r) * A.W + I.x0 + c;
                    return r < I.rows && c < I.cw;
                };
                for (int u = part; u < nunits; u += kParts) {
                    int b, c0, r, c; size_t g0;
                    const bool valid = place(u, b, c0, g0, r, c);
                    // what the fused dz step reads of the layer below is requested before the accumulators, so that the
                    // latencies overlap (requested a whole unit ahead, even for the launches through a pool only, the
                    // kernel was measured slower)
                    uint4 yq[2] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};
                    unsigned long long amq[2] = {0ull, 0ull};
                    if (FORM == kConvPlain && A.prev_y && valid) {
                        yq[0] = __ldg(A.prev_y + g0); yq[1] = __ldg(A.prev_y + g0 + gstep);
                        if (A.prev_arg) { amq[0] = __ldg(A.prev_arg + g0); amq[1] = __ldg(A.prev_arg + g0 + gstep); }
                    }
                    float v[16];
                    tmem_ld16(tbuf + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * A.Ns + c0), v);
                    if constexpr (FORM != kConvPlain) {       // (a delta: neither bias nor activation)
                        if (!valid) continue;
                        float* dst = A.out_f + (((size_t)I.n * A.cout + I.co0 + c0) * A.H + I.y0 + r) * A.W + I.x0 + c;
#pragma unroll
                        for (int j = 0; j < 16; ++j) if (I.co0 + c0 + j < A.cout) dst[j * gstep] = v[j];
                    } else if (valid && !A.prev_y) {
                        A.out[g0] = act8(v, H->bias + c0, slope);
                        A.out[g0 + gstep] = act8(v + 8, H->bias + c0 + 8, slope);
                    } else if (valid) {
                        // input delta straight into the dz planes of the layer below: rounded as a stored delta
                        // would be, times the derivative of that layer's activation, through its pool's arg-max
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint4 dq = derive8(tcd::pack8(v + 8 * h), yq[h], A.prev_slope);
                            if (!A.prev_arg) { A.out[g0 + h * gstep] = dq; continue; }
                            // the four members of every channel's pool window: the delta where the arg-max byte names the
                            // member, zero elsewhere (byte masks widened to the bf16 halves)
                            const uint32_t alo = (uint32_t)amq[h] & 0x03030303u, ahi = (uint32_t)(amq[h] >> 32) & 0x03030303u;
                            const int W2 = 2 * A.W;
                            uint4* o2 = A.out + (((size_t)I.n * oplanes + ((I.co0 + c0) >> 3) + h) * (2 * A.H) + 2 * (I.y0 + r)) * W2 + 2 * (I.x0 + c);
                            // (a 32-byte store covers a whole sector; as two of 16 bytes: us of the launch 177 -> 150, 64 -> 32 channels to
                            // 16 x 608 x 608; 96 -> 76, 128 -> 64 channels to 304 x 304)
                            auto member = [&](uint32_t w) {
                                const uint32_t ml = __vcmpeq4(alo, w * 0x01010101u), mh = __vcmpeq4(ahi, w * 0x01010101u);
                                return make_uint4(dq.x & __byte_perm(ml, 0u, 0x1100), dq.y & __byte_perm(ml, 0u, 0x3322),
                                                  dq.z & __byte_perm(mh, 0u, 0x1100), dq.w & __byte_perm(mh, 0u, 0x3322));
                            };
                            store_pair(o2, member(0), member(1));
                            store_pair(o2 + W2, member(2), member(3));
                        }
                    }
                }
            } else if constexpr (FORM == kConvRowPool) {
                // The rows of a window are the same lanes of two blocks and its columns two neighbouring lanes: no staging area and
                // no barriers.  The even lane takes the lower 8 channels of a unit, the odd lane the upper ones.
                // us, staged and so (with the cheaper activation and an instance of its own): 3 -> 32, 16 x 608 x 608 152 -> 130; 32 -> 64,
                // 304 x 304 123 -> 95.
                const int OH = A.H >> 1, OW = A.W >> 1, nc = I.cols >> 4, odd = lane & 1, col = q * 32 + lane;
                const bool valid = (col & ~1) < I.cw;
                for (int u = part; u < (I.rows >> 1) * nc; u += kParts) {
                    const int pr = u / nc, c0 = (u - pr * nc) << 4;
                    const uint32_t at = tbuf + ((uint32_t)(q * 32) << 16) + (uint32_t)(2 * pr * A.Ns + c0);
                    float v[2][16];
                    tmem_ld16x2(at, at + (uint32_t)A.Ns, v[0], v[1]);
                    uint4 own[2], got[2];
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const uint4 lo = act8(v[r], H->bias + c0, slope), hi = act8(v[r] + 8, H->bias + c0 + 8, slope);
                        own[r] = odd ? hi : lo;
                        const uint4 away = odd ? lo : hi;
                        got[r] = make_uint4(__shfl_xor_sync(0xffffffffu, away.x, 1), __shfl_xor_sync(0xffffffffu, away.y, 1),
                                            __shfl_xor_sync(0xffffffffu, away.z, 1), __shfl_xor_sync(0xffffffffu, away.w, 1));
                    }
                    uint4 best;
                    // (operands picked before the comparison: two calls behind a branch would both run)
                    auto pick = [&](const uint4& a, const uint4& b) { return make_uint4(odd ? b.x : a.x, odd ? b.y : a.y, odd ? b.z : a.z, odd ? b.w : a.w); };
                    const unsigned long long am = pool4(pick(own[0], got[0]), pick(got[0], own[0]), pick(own[1], got[1]), pick(got[1], own[1]), best);
                    const size_t gi = (((size_t)I.n * oplanes + ((I.co0 + c0) >> 3) + odd) * OH + (I.y0 >> 1) + pr) * OW + (I.x0 >> 1) + (col >> 1);
                    if (valid) { A.out[gi] = best; A.arg[gi] = am; }
                }
            } else {
                const int OH = A.H / 2, OW = A.W / 2, prs = I.rows / 2, pcs = I.cw / 2;
                for (int pl0 = 0; pl0 < (I.cols >> 3); pl0 += A.pool_planes) {
                    const int npl = min(A.pool_planes, (I.cols >> 3) - pl0);
                    // the band as it would be stored, planes pl0 .. pl0 + npl - 1
                    const int nc = npl >> 1;
                    for (int u = part; u < I.nblk * nc; u += kParts) {
                        const int b = u / nc, c0 = pl0 * 8 + ((u - b * nc) << 4);
                        const int p = b * 128 + q * 32 + lane;
                        {
                            float v[16];
                            tmem_ld16(tbuf + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * A.Ns + c0), v);
                            S[(size_t)((c0 >> 3) - pl0) * E + p] = act8(v, H->bias + c0, slope);
                            S[(size_t)((c0 >> 3) - pl0 + 1) * E + p] = act8(v + 8, H->bias + c0 + 8, slope);
                        }
                    }
                    asm volatile("bar.sync 1, %0;" :: "n"(kTcConvEpiThreads) : "memory");
                    // one thread per pooled pixel and plane
                    const int npix = prs * pcs, total = npl * npix;
                    for (int e = et; e < total; e += kTcConvEpiThreads) {
                        const int pl = e / npix, pix = e - pl * npix, pr = pix / pcs, pc = pix - pr * pcs;
                        const uint4* s4 = S + (size_t)pl * E + (size_t)(2 * pr) * A.Wp + 2 * pc;
                        const uint4 m0 = s4[0], m1 = s4[1], m2 = s4[A.Wp], m3 = s4[A.Wp + 1];
                        uint4 best;
                        const unsigned long long am = pool4(m0, m1, m2, m3, best);
                        const size_t gi = (((size_t)I.n * oplanes + (I.co0 >> 3) + pl0 + pl) * OH + (I.y0 >> 1) + pr) * OW + (I.x0 >> 1) + pc;
                        A.out[gi] = best;
                        A.arg[gi] = am;
                    }
                    asm volatile("bar.sync 1, %0;" :: "n"(kTcConvEpiThreads) : "memory");    // the staging area is free for the next planes
                }
            }
            fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&H->tfree[buf]));
        }
    }
    if (A.hurry) next_launch();
    __syncthreads();
    // every MMA of the block has completed before the tensor memory goes back (also when a wait gave up)
    if (warp == 0) {
        if (lane == 0) mbar_wait(smem_u32(&H->drain), 0, 200000000ll);
        __syncwarp();
        fence_after_sync();
        tmem_dealloc(tmem, (uint32_t)kTcTmemCols);
    }
}

}  // namespace ftp
