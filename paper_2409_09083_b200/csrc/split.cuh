// fp32 path, executed groups of one conv layer with enough channels: the contractions of the training step on the
// tensor cores without giving up fp32 accuracy.
//
// Operands.  Every fp32 value is kept as the sum of three bf16 values, a = a0 + a1 + a2: a0 = a rounded to 6 significant
// bits, a1 = bf16(a - a0), a2 = a - a0 - a1, which together hold the 24 bits of an fp32 exactly (the differences are exact in
// fp32; values below 2^-110, whose last part falls under the smallest bf16, lose bits there, and values next to the largest
// fp32 one bit, see split8).  A product is formed as
// the six products a0 b0, a0 b1, a1 b0, a0 b2, a1 b1, a2 b0, each exact in fp32; what is left out (a1 b2, a2 b1, a2 b2) has
// either sign and measures 2^-24 of |a b| in the 2-norm, the rounding of one fp32 multiply-add.
//
// Sums.  The tensor core adds to its fp32 accumulators by truncation (measured: an addend of 0.99 units in the last place
// vanishes).  A long chain of such sums loses a part of itself, always towards zero: with 9 large steps between two
// additions to fp32 registers a layer shrinks its map by 1.1e-7, which the 24 layer passes of a 16-layer step add up to
// 2.4e-6 of a filter gradient (the multiply-add chains of stationary.cuh: 3e-7, in no preferred direction).  Two measures
// take that away.  The large products a0 b0 have accumulators of their own (H), and with 6 + 6 significant bits they leave 12
// of the accumulator's 24 bits to the range of their sum, so that little is cut off; and a chain of them is 2 to 4 steps long
// before the epilogue warps add it to their registers, rounded to nearest.  The five small products go to a second set of
// accumulators (L): they measure 2^-7 of the sum and their signs have nothing to do with its sign, so their chains may last for
// an item (64 stages of the filter gradient).  What is left is 2e-9 to 1e-8 a layer.  Against fp64 sums maps, deltas and
// gradients are 1.7 to 7 times closer than those of stationary.cuh (table in tests/test_gpu_split.py).
//
// Maps travel between the layers in split form (split_args.hpp): 6 bytes a value instead of 4, split once by the epilogue
// that produces them, with the zero padding in memory so that any run of entries is a tile: one plain bulk copy per plane
// and row, no bounds logic, and blocks of 128 consecutive entries cover the batch without ragged tiles.
//
//   conv_split_kernel    forward pass, and the input delta as the convolution of dz with the rotated filters
//   fgrad_split_kernel   filter and bias gradient
#pragma once

#include "pack.cuh"
#include "split_args.hpp"
#include "split_parts.cuh"
#include "tc.cuh"

namespace ftp {
namespace sp {

using namespace tc;

// 32 lanes x 32 consecutive fp32 columns of tensor memory
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

constexpr int kMaxA = 3, kMaxB = 8;
constexpr int kConvThreads = 384;             // 8 epilogue warps; producer, MMA issuers of the large and (two) of the small products
constexpr int kEpiThreads = 256;

// ---------------------------------------------------------------------------------------------
// Convolution.  A work item is a tile of nblk x 128 output entries x a slice of Ns <= 128 output channels.  The input
// channels stream past in chunks: the tile with its halo (three parts; ring of a_stages), and the filters of the
// chunk part by part (ring of b_stages), so that a stage of filters serves the products a0 b0, a1 b0, a2 b0 | a0 b1, a1 b1 |
// a0 b2.  Of the 512 tensor-memory columns one half holds H and one L.  One thread issues the a0 b0 products of all
// blocks, a chain per window row and chunk; while the epilogue warps add a chain to their registers
// (256 entries x 128 channels of running sums) the tensor core works on the small products of two other threads, which
// are five sixths of the work and wait for nothing but the loads.
//
// Bound: tensor pipe for Ns = 128 (six products of 64 cycles per 128 entries, 16 channels and window position; the loads
// are 21 bytes a cycle and SM); narrower slices by the shared-memory reads of the A tile (48 cycles at 64 channels).
// ---------------------------------------------------------------------------------------------
template <int K, int NB>
__global__ void __launch_bounds__(kConvThreads, 1) conv_split_kernel(const __grid_constant__ SplitConvArgs A)
{
    constexpr int kChains = K;                  // chains of large products a chunk (one per window row)
    constexpr int UPB = 8 / NB;                 // 16-column units an epilogue warp holds per accumulator block (NB blocks a warp)
    extern __shared__ __align__(1024) unsigned char sp_smem[];
    struct Hdr {
        unsigned long long a_full[kMaxA], a_empty[kMaxA], b_full[kMaxB], b_empty[kMaxB];
        unsigned long long hdone[2], hfree[2], ldone[2], lfree[2], drain;     // [half]: blocks 0, 2, ... and 1, 3, ... of an item
        uint32_t tmem_base;
        volatile int failed;
        volatile int stop[2];
    };
    static_assert(sizeof(Hdr) <= kSplitHeader, "header does not fit");
    Hdr* H = reinterpret_cast<Hdr*>(sp_smem);
    unsigned char* a_ring = sp_smem + kSplitHeader;
    const int a_bytes = A.a_bytes;
    unsigned char* b_ring = a_ring + (size_t)A.a_stages * a_bytes;
    float* pool_s = reinterpret_cast<float*>(b_ring + (size_t)A.b_stages * A.b_stage);
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (the shuffle tells the compiler that it is the same for the warp)

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxA; ++s) { mbar_init(smem_u32(&H->a_full[s]), 1); mbar_init(smem_u32(&H->a_empty[s]), 3); }
        for (int s = 0; s < kMaxB; ++s) { mbar_init(smem_u32(&H->b_full[s]), 1); mbar_init(smem_u32(&H->b_empty[s]), 3); }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&H->hdone[s]), 1); mbar_init(smem_u32(&H->hfree[s]), 4);
            mbar_init(smem_u32(&H->ldone[s]), 1); mbar_init(smem_u32(&H->lfree[s]), 4);
        }
        mbar_init(smem_u32(&H->drain), 3);
        H->failed = 0;
        fence_mbar_init();
    }
    if (warp == 0) { __syncwarp(); tmem_alloc(smem_u32(&H->tmem_base), (uint32_t)kTcTmemCols); }
    previous_launches();
    // entries of the output map that no item covers
    if (A.out_s) {
        if (A.mode == kSplitPool) zero_margins(A.out_s, A.og, kSplitLead + A.og.wp, kSplitLead + A.og.rows * A.og.wp);
        else if (A.mode == kSplitTile || A.prev_arg) zero_margins(A.out_s, A.og, kSplitLead, kSplitLead + A.og.rows * A.og.wp);
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    const uint32_t tmem = H->tmem_base;

    auto wait = [&](unsigned long long* bar, uint32_t parity, unsigned sleep_ns = 0) {
        if (H->failed) return false;
        if (mbar_wait(smem_u32(bar), parity, kWaitLimitCycles, sleep_ns)) return true;
        H->failed = 1;
        atomicExch(A.error, 1);
        return false;
    };
    // item -> slice and tile; every role walks the same sequence
    struct Item { int slice, cols, nblk, e0, n, y0, row0, x0, rows, cw; };
    auto item_of = [&](int it) {
        Item I;
        I.slice = it % A.slices;
        const int t = it / A.slices;
        I.cols = min(A.Ns, A.cout16 - I.slice * A.Ns);
        I.nblk = A.nblk; I.e0 = 0; I.n = I.y0 = I.row0 = I.x0 = I.rows = I.cw = 0;
        if (A.mode == kSplitFlat) { I.e0 = t * A.nblk * 128; return I; }
        const int tx = t % A.tiles_x, ty = t / A.tiles_x;
        I.x0 = tx * A.Cw;
        if (A.mode == kSplitTile) {
            I.row0 = ty * A.R;
            I.rows = min(A.R, A.g.rows - I.row0); I.cw = min(A.Cw, A.g.wp - I.x0);
        } else {
            I.n = ty / A.tiles_y; I.y0 = (ty - I.n * A.tiles_y) * A.R;
            I.row0 = 1 + I.n * (A.g.H + 1) + I.y0;
            I.rows = min(A.R, A.g.H - I.y0); I.cw = min(A.Cw, A.g.W - I.x0);
        }
        I.nblk = (I.rows * A.pitch + 127) >> 7;
        return I;
    };

    if (warp < 8) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        // ---- epilogue: lane quarter q of the accumulator blocks half, half + 2, ... ----
        const int q = warp & 3, half = warp >> 2, et = threadIdx.x;
        const size_t opart = (size_t)A.og.planes * A.og.tp;
        uint32_t gh = 0, gl = 0, k = 0;                       // chains and items of this half so far
        for (int it = blockIdx.x; it < A.items; it += gridDim.x, ++k) {
            const Item I = item_of(it);
            const int co0 = I.slice * A.Ns;
            float bias[4];                                    // lane l: channels l, 32 + l, ... of the item
#pragma unroll
            for (int i = 0; i < 4; ++i) bias[i] = A.bias && co0 + i * 32 + lane < A.cout ? __ldg(A.bias + co0 + i * 32 + lane) : 0.f;
            float acc[128];
#pragma unroll
            for (int j = 0; j < 128; ++j) acc[j] = 0.f;
            auto plain = [](float a, float b) { return a + b; };
            auto add = [&](uint32_t col, auto sum) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int bl = half + 2 * (2 * i / UPB), c0 = (2 * i % UPB) * 16;      // two units at a time
                    if (bl < I.nblk && c0 < I.cols) {
                        float v[32];
                        tmem_ld32(tmem + col + ((uint32_t)(q * 32) << 16) + (uint32_t)(bl * A.Ns + c0), v);
#pragma unroll
                        for (int j = 0; j < 32; ++j) acc[i * 32 + j] = sum(acc[i * 32 + j], v[j]);
                    }
                }
                fence_before_sync();
                __syncwarp();
            };
            bool ok = true;
            if (half < I.nblk) {
                for (int c = 0; c < kChains * A.nchunks; ++c, ++gh) {
                    if (!wait(&H->hdone[half], gh & 1u, 32)) { ok = false; break; }
                    fence_after_sync();
                    add(0, plain);
                    if (lane == 0) mbar_arrive(smem_u32(&H->hfree[half]));
                }
                if (ok && wait(&H->ldone[half], gl & 1u, 32)) {
                    fence_after_sync();
                    add(256, add_small);
                    if (lane == 0) mbar_arrive(smem_u32(&H->lfree[half]));
                    ++gl;
                } else ok = false;
            }
            if (A.mode == kSplitPool) {
                if (et == 0) H->stop[k & 1u] = (H->failed || !ok) ? 1 : 0;
                asm volatile("bar.sync 1, %0;" :: "n"(kEpiThreads) : "memory");
                if (H->stop[k & 1u]) break;                 // the same answer for all: they leave together
            } else if (!ok) break;
            if (A.mode != kSplitPool) {
#pragma unroll
                for (int nb = 0; nb < NB; ++nb) {
                    const int bl = half + 2 * nb;
                    if (bl >= I.nblk) break;
                    const int p = bl * 128 + q * 32 + lane;
                    int e; bool in = true;
                    if (A.mode == kSplitFlat) { e = I.e0 + p; in = e < A.g.tp; }
                    else {
                        const int r = p / A.pitch, cc = p - r * A.pitch;
                        in = r < I.rows && cc < I.cw;
                        e = kSplitLead + (I.row0 + r) * A.g.wp + I.x0 + cc;
                    }
                    int n = 0, y = 0, x = 0;
                    const bool valid = in && pixel_of(A.g, e, n, y, x);
#pragma unroll
                    for (int u = 0; u < UPB; ++u) {
                        const int c0 = u * 16;
                        if (c0 >= I.cols) break;
                        float* v = acc + (nb * UPB + u) * 16;
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            float z = v[j] + __shfl_sync(0xffffffffu, bias[u / 2], (u & 1) * 16 + j);
                            if (A.act) z = z > 0.f ? z : A.slope * z;
                            v[j] = valid ? z : 0.f;
                        }
                        if (A.out_f && valid) {
                            float* dst = A.out_f + (((size_t)n * A.cout + co0 + c0) * A.g.H + y) * A.g.W + x;
                            const size_t step = (size_t)A.g.H * A.g.W;
#pragma unroll
                            for (int j = 0; j < 16; ++j) if (co0 + c0 + j < A.cout) dst[j * step] = v[j];
                        }
                        if (A.out_s && in) {
                            const int pl = (co0 + c0) >> 3;
                            if (A.prev_y) {
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    const uint4 yq = __ldg(A.prev_y + (size_t)(pl + h) * A.g.tp + e);
                                    const uint32_t* yw = &yq.x;
#pragma unroll
                                    for (int j = 0; j < 4; ++j) {               // the sign and the zero of a value are those of its first part
                                        const float lo = __uint_as_float(yw[j] << 16), hi = __uint_as_float(yw[j] & 0xffff0000u);
                                        v[h * 8 + 2 * j] *= lo > 0.f ? 1.f : A.prev_slope;
                                        v[h * 8 + 2 * j + 1] *= hi > 0.f ? 1.f : A.prev_slope;
                                    }
                                }
                            }
                            if (!A.prev_arg) {
                                store_split(A.out_s, opart, (size_t)pl * A.og.tp + e, v);
                                store_split(A.out_s, opart, (size_t)(pl + 1) * A.og.tp + e, v + 8);
                            }
                        }
                        if (A.prev_arg) {
                            // Through the arg-max of the pool below: the delta at one member of the window, zeros at the others; the
                            // zero entries of the low-resolution map stand for those of the high-resolution one.  Lane l writes the
                            // column l % 2 of the window of lane l / 2 (then 16 + l / 2), so that a store covers 512 contiguous bytes (one lane per
                            // pixel, with half a sector per lane and store: 112 against 35 thousand cycles for this phase of an item
                            // without the arg-max, 128 -> 64 channels on 152 x 152; a step of that net with 16 images 11.40 -> 11.02 ms,
                            // together with the bias in lanes, which took the 16 dependent loads per unit out of the phase).
                            const int row = (e - kSplitLead) / A.g.wp;
                            const bool wr = in && x <= A.g.W && y <= A.g.H && e >= kSplitLead && (valid || e < kSplitLead + A.g.rows * A.g.wp);
                            const int fl = (wr ? 1 : 0) | (wr && row > 0 && y < A.g.H ? 2 : 0) | (x < A.g.W ? 4 : 0);
                            const int e2 = kSplitLead + (row == 0 ? 0 : 1 + n * A.og.H + n + 2 * y) * A.og.wp + 2 * x;
                            const int pl = (co0 + c0) >> 3, wc = lane & 1;
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const unsigned long long am = valid ? __ldg(A.prev_arg + (size_t)(pl + h) * A.g.tp + e) : 0ull;
                                uint4 s[3];
                                split8<false>(v + h * 8, s[0], s[1], s[2]);
#pragma unroll
                                for (int k2 = 0; k2 < 2; ++k2) {
                                    const int src = 16 * k2 + (lane >> 1);
                                    const uint32_t alo = __shfl_sync(0xffffffffu, (uint32_t)am, src) & 0x03030303u;
                                    const uint32_t ahi = __shfl_sync(0xffffffffu, (uint32_t)(am >> 32), src) & 0x03030303u;
                                    const int f = __shfl_sync(0xffffffffu, fl, src), es = __shfl_sync(0xffffffffu, e2, src) + wc;
                                    uint4 z[3];
#pragma unroll
                                    for (int t = 0; t < 3; ++t)
                                        z[t] = make_uint4(__shfl_sync(0xffffffffu, s[t].x, src), __shfl_sync(0xffffffffu, s[t].y, src),
                                                          __shfl_sync(0xffffffffu, s[t].z, src), __shfl_sync(0xffffffffu, s[t].w, src));
#pragma unroll
                                    for (int wr2 = 0; wr2 < 2; ++wr2) {
                                        if (!(f & (1 + wr2)) || (wc && !(f & 4))) continue;
                                        const uint32_t w = (uint32_t)(2 * wr2 + wc) * 0x01010101u;
                                        const uint32_t ml = __vcmpeq4(alo, w), mh = __vcmpeq4(ahi, w);
                                        const uint32_t m0 = __byte_perm(ml, 0u, 0x1100), m1 = __byte_perm(ml, 0u, 0x3322);
                                        const uint32_t m2 = __byte_perm(mh, 0u, 0x1100), m3 = __byte_perm(mh, 0u, 0x3322);
#pragma unroll
                                        for (int t = 0; t < 3; ++t)
                                            A.out_s[t * opart + (size_t)(pl + h) * A.og.tp + (size_t)es + (size_t)wr2 * A.og.wp] =
                                                make_uint4(z[t].x & m0, z[t].y & m1, z[t].z & m2, z[t].w & m3);
                                    }
                                }
                            }
                        }
                    }
                }
            } else {
                // 2x2 maximum of the activated values, first one in window order, 16 channels at a time through shared memory
                const int E = A.nblk * 128, OH = A.g.H >> 1, OW = A.g.W >> 1;
                const int prs = I.rows >> 1, pcs = I.cw >> 1;
                const int er = prs + (I.y0 + I.rows == A.g.H ? 1 : 0), ec = pcs + (I.x0 + I.cw == A.g.W ? 1 : 0);   // with the zero entries behind
                const int npix = er * ec;
#pragma unroll
                for (int u = 0; u < UPB; ++u) {
                    const int c0 = u * 16;
                    if (c0 < I.cols) {
#pragma unroll
                        for (int nb = 0; nb < NB; ++nb) {
                            const int bl = half + 2 * nb;
                            if (bl < I.nblk) {
                                const int p = bl * 128 + q * 32 + lane;
#pragma unroll
                                for (int j = 0; j < 16; ++j) {
                                    float z = acc[(nb * UPB + u) * 16 + j] + __shfl_sync(0xffffffffu, bias[u / 2], (u & 1) * 16 + j);
                                    pool_s[j * E + p] = z > 0.f ? z : A.slope * z;
                                }
                            }
                        }
                        asm volatile("bar.sync 1, %0;" :: "n"(kEpiThreads) : "memory");
                        for (int i = et; i < 2 * npix; i += kEpiThreads) {
                            const int h = i / npix, pix = i - h * npix, pr = pix / ec, pc = pix - pr * ec;
                            const int yo = (I.y0 >> 1) + pr, xo = (I.x0 >> 1) + pc;
                            const bool real = pr < prs && pc < pcs;
                            float best[8];
                            unsigned long long am = 0ull;
                            const float* s = pool_s + h * 8 * E + 2 * pr * A.pitch + 2 * pc;
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                best[j] = 0.f;
                                if (real) {
                                    const float2 a = *reinterpret_cast<const float2*>(s + j * E), b = *reinterpret_cast<const float2*>(s + j * E + A.pitch);
                                    float m = a.x; unsigned long long w = 0;
                                    if (a.y > m) { m = a.y; w = 1; }
                                    if (b.x > m) { m = b.x; w = 2; }
                                    if (b.y > m) { m = b.y; w = 3; }
                                    best[j] = m; am |= w << (8 * j);
                                }
                            }
                            const int pl = ((co0 + c0) >> 3) + h;
                            const size_t eo = (size_t)kSplitLead + (size_t)(1 + I.n * (OH + 1) + yo) * A.og.wp + xo;
                            if (real) A.arg[(size_t)pl * A.og.tp + eo] = am;
                            if (A.out_s) store_split(A.out_s, opart, (size_t)pl * A.og.tp + eo, best);
                            if (A.out_f && real) {
                                float* dst = A.out_f + (((size_t)I.n * A.cout + pl * 8) * OH + yo) * OW + xo;
#pragma unroll
                                for (int j = 0; j < 8; ++j) if (pl * 8 + j < A.cout) dst[(size_t)j * OH * OW] = best[j];
                            }
                        }
                        asm volatile("bar.sync 1, %0;" :: "n"(kEpiThreads) : "memory");
                    }
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
        if (warp == 8) {
            // ---- producer: per chunk the tile, then the three parts of the filters ----
            uint32_t g = 0, gb = 0;
            bool ok = true;
            const int part_planes = A.g.planes;
            for (int it = blockIdx.x; it < A.items && ok; it += gridDim.x) {
                const Item I = item_of(it);
                const int e_first = I.e0 - (K / 2) * (A.g.wp + 1);        // flat run: one row and one column back
                const uint4* wsrc = A.w + (size_t)I.slice * A.nchunks * 3 * (A.b_stage / 16);
                for (int c = 0; c < A.nchunks && ok; ++c) {
                    const int s = (int)(g % (uint32_t)A.a_stages);
                    ok = __all_sync(0xffffffffu, wait(&H->a_empty[s], ((g / (uint32_t)A.a_stages) & 1u) ^ 1u));
                    if (!ok) break;
                    const int kp0 = c * A.kpc;
                    const uint32_t bar = smem_u32(&H->a_full[s]), dst0 = smem_u32(a_ring + (size_t)s * a_bytes);
                    if (A.mode != kSplitFlat) {            // one box: the tile with its halo, the planes of the chunk, three parts
                        if (lane == 0) {
                            mbar_expect_tx(bar, (uint32_t)(3 * A.kpc * A.a_plane));
                            tma_load_4d(dst0, A.tmap, 2 * (I.x0 - K / 2), I.row0 - K / 2, kp0, 0, bar);
                        }
                    } else if (K == 1) {                   // no halo: one box per block of 128 entries
                        if (lane == 0) {
                            mbar_expect_tx(bar, (uint32_t)a_bytes);
                            for (int b = 0; b < A.nblk; ++b) tma_load_3d(dst0 + (uint32_t)(b * A.a_block * 16), A.tmap, 2 * (I.e0 + b * 128), kp0, 0, bar);
                        }
                    } else {                               // a run per plane
                        const int np = min(A.kpc, part_planes - kp0), copies = 3 * np;
                        if (lane == 0) mbar_expect_tx(bar, (uint32_t)(copies * A.run_len) * 16u);
                        __syncwarp();
                        if (lane < copies) {
                            const int part = lane / np, pl = lane - part * np;
                            const long long src = ((long long)part * part_planes + kp0 + pl) * A.g.tp + e_first;
                            bulk_g2s(dst0 + (uint32_t)((part * A.kpc + pl) * A.a_plane), A.in + src, (uint32_t)A.run_len * 16u, bar);
                        }
                    }
                    __syncwarp();
                    ++g;
                    for (int j = 0; j < 3; ++j) {
                        const int sb = (int)(gb % (uint32_t)A.b_stages);
                        ok = __all_sync(0xffffffffu, wait(&H->b_empty[sb], ((gb / (uint32_t)A.b_stages) & 1u) ^ 1u));
                        if (!ok) break;
                        if (lane == 0) {
                            const uint32_t bb = smem_u32(&H->b_full[sb]);
                            mbar_expect_tx(bb, (uint32_t)A.b_stage);
                            bulk_g2s(smem_u32(b_ring + (size_t)sb * A.b_stage), wsrc + (size_t)(3 * c + j) * (A.b_stage / 16), (uint32_t)A.b_stage, bb);
                        }
                        __syncwarp();
                        ++gb;
                    }
                }
            }
            if (H->failed) {     // let the copies already under way land before the block leaves
                auto land = [&](unsigned long long* full, int stages, uint32_t count) {
                    for (int s = 0; s < stages; ++s) {
                        const uint32_t n = count > (uint32_t)s ? (count - 1 - (uint32_t)s) / (uint32_t)stages + 1 : 0;   // copies into stage s
                        if (n > 0) mbar_wait(smem_u32(&full[s]), (n - 1) & 1u, 200000000ll);
                    }
                };
                land(H->a_full, A.a_stages, g);
                land(H->b_full, A.b_stages, gb);
            }
        } else {
            // ---- MMA issue: warp 9 the large products of all blocks, warps 10 and 11 the small ones of the blocks 0, 2, ... and
            // 1, 3, ...; the whole warp runs the loops, so that the descriptors stay in uniform registers, and one lane issues.
            // Every issuer releases every stage, in order ----
            const int role = warp - 9;                    // 0: large; 1, 2: small
            const bool leader = lane == 0;
            const uint32_t hi = desc_hi(128);
            const uint32_t a_step = 2u * ((uint32_t)A.a_plane >> 4), b_step = 2u * (uint32_t)A.Ns;      // one K step of 16 channels
            const uint32_t a_part = (uint32_t)A.kpc * ((uint32_t)A.a_plane >> 4), b_tap = (uint32_t)(A.kpc * A.Ns);
            const uint32_t wp = (uint32_t)(A.mode == kSplitFlat ? A.g.wp : A.pitch);
            uint32_t ga = 0, gb = 0, gh[2] = {0, 0}, gl = 0;
            bool ok = true;
            for (int it = blockIdx.x; it < A.items && ok; it += gridDim.x) {
                const Item I = item_of(it);
                const uint32_t idesc = make_idesc(128, I.cols, false, false);
                const bool mine = role > 0 && role - 1 < I.nblk;              // this item has blocks of this issuer's small products
                if (mine) {
                    if (gl > 0) ok = __all_sync(0xffffffffu, wait(&H->lfree[role - 1], (gl - 1) & 1u));
                    fence_after_sync();
                    ++gl;
                }
                for (int c = 0; c < A.nchunks && ok; ++c, ++ga) {
                    const int sa = (int)(ga % (uint32_t)A.a_stages);
                    ok = __all_sync(0xffffffffu, wait(&H->a_full[sa], (ga / (uint32_t)A.a_stages) & 1u));
                    const int nks = min(A.kpc, A.g.planes - c * A.kpc) >> 1;
                    const uint32_t a0 = desc_lo(smem_u32(a_ring + (size_t)sa * a_bytes), (uint32_t)A.a_plane);
                    for (int j = 0; j < 3 && ok; ++j, ++gb) {
                        const int sb = (int)(gb % (uint32_t)A.b_stages);
                        ok = __all_sync(0xffffffffu, wait(&H->b_full[sb], (gb / (uint32_t)A.b_stages) & 1u));
                        if (!ok) break;
                        fence_after_sync();
                        const uint32_t b0 = desc_lo(smem_u32(b_ring + (size_t)sb * A.b_stage), (uint32_t)A.Ns * 16u);
                        if (role == 0) {
                            if (j == 0)
#pragma unroll
                                for (int ch = 0; ch < kChains; ++ch)
                                    for (int h = 0; h < 2; ++h) {
                                        if (h >= I.nblk) break;
                                        if (gh[h] > 0) ok = __all_sync(0xffffffffu, ok && wait(&H->hfree[h], (gh[h] - 1) & 1u));
                                        if (!ok) break;
                                        ++gh[h];
                                        fence_after_sync();
                                        for (int b = h; b < I.nblk; b += 2) {
                                            const uint32_t tcol = tmem + (uint32_t)(b * A.Ns);
                                            uint32_t a = a0 + (uint32_t)(b * A.a_block) + (uint32_t)ch * wp, w = b0 + (uint32_t)(ch * K) * b_tap;
                                            for (int ks = 0; ks < nks; ++ks, a += a_step, w += b_step) {
                                                if (leader) {
                                                    mma_bf16(tcol, desc64(hi, a), desc64(hi, w), idesc, ks > 0);
                                                    if (K == 3) {
                                                        mma_bf16(tcol, desc64(hi, a + 1), desc64(hi, w + b_tap), idesc, true);
                                                        mma_bf16(tcol, desc64(hi, a + 2), desc64(hi, w + 2 * b_tap), idesc, true);
                                                    }
                                                }
                                                __syncwarp();
                                            }
                                        }
                                        if (leader) mma_commit(smem_u32(&H->hdone[h]));
                                        __syncwarp();
                                    }
                        } else {
                            for (int pa = j == 0 ? 1 : 0; pa < 3 - j; ++pa)
                                for (int b = role - 1; b < I.nblk; b += 2) {
                                    const uint32_t tcol = tmem + 256u + (uint32_t)(b * A.Ns);
                                    uint32_t a = a0 + (uint32_t)pa * a_part + (uint32_t)(b * A.a_block), w = b0;
                                    for (int ks = 0; ks < nks; ++ks, a += a_step, w += b_step) {
                                        const bool acc = c > 0 || j > 0 || pa > 1 || ks > 0;
                                        if (leader) {
                                            mma_bf16(tcol, desc64(hi, a), desc64(hi, w), idesc, acc);
                                            if (K == 3) {
                                                mma_bf16(tcol, desc64(hi, a + 1), desc64(hi, w + b_tap), idesc, true);
                                                mma_bf16(tcol, desc64(hi, a + 2), desc64(hi, w + 2 * b_tap), idesc, true);
                                                mma_bf16(tcol, desc64(hi, a + wp), desc64(hi, w + 3 * b_tap), idesc, true);
                                                mma_bf16(tcol, desc64(hi, a + wp + 1), desc64(hi, w + 4 * b_tap), idesc, true);
                                                mma_bf16(tcol, desc64(hi, a + wp + 2), desc64(hi, w + 5 * b_tap), idesc, true);
                                                mma_bf16(tcol, desc64(hi, a + 2 * wp), desc64(hi, w + 6 * b_tap), idesc, true);
                                                mma_bf16(tcol, desc64(hi, a + 2 * wp + 1), desc64(hi, w + 7 * b_tap), idesc, true);
                                                mma_bf16(tcol, desc64(hi, a + 2 * wp + 2), desc64(hi, w + 8 * b_tap), idesc, true);
                                            }
                                        }
                                        __syncwarp();
                                    }
                                }
                        }
                        if (!ok) break;
                        if (leader) mma_commit(smem_u32(&H->b_empty[sb]));
                    }
                    if (!ok) break;
                    if (leader) mma_commit(smem_u32(&H->a_empty[sa]));
                    __syncwarp();
                }
                if (ok && mine && leader) mma_commit(smem_u32(&H->ldone[role - 1]));
                __syncwarp();
            }
            if (leader) mma_commit(smem_u32(&H->drain));
        }
        __syncwarp();
    }
    __syncthreads();
    if (warp == 0) {             // every MMA of the block has completed before the tensor memory goes back (also when a wait gave up)
        if (lane == 0) mbar_wait(smem_u32(&H->drain), 0, 200000000ll);
        __syncwarp();
        fence_after_sync();
        tmem_dealloc(tmem, (uint32_t)kTcTmemCols);
    }
}

// ---------------------------------------------------------------------------------------------
// Filter gradient: dW[co][ci][tap] = sum over entries e of dz[co][e] x[ci][e + shift(tap)].  The zero entries of the maps
// make the batch one flat run, cut into stages of E entries.  A block owns Ms output channels x up to three accumulator
// units of `ncols` columns and a share of the stages:
//   3x3: one row of the window; unit kx is the input shifted by kx (one tile of E + 2 entries serves all three);
//   3x3 with at most 32 input channels (`rows3`): the whole window; unit ky holds the three window columns side by side (an
//        input tile per window row; a block per window row would be bound by its loads: the layer 32 -> 64 at
//        304 x 304, 16 images, 554 us that way);
//   1x1: one or two slices of the input channels.
// Every unit has accumulators for its small products, which last for kFgFlush stages; the large products of the units take one or
// two further slots in turn (4 steps a chain), which 12 warps (four per unit) add to their registers while the tensor core
// works on small products.  The bias gradient is the same contraction with a tile of ones (blocks of the first
// input-channel slice and window row only).
//
// Bound: tensor pipe at 128 columns (64 cycles an MMA; loads 21 bytes a cycle and SM), shared-memory reads below.
// ---------------------------------------------------------------------------------------------
constexpr int kFgThreads = 512;
constexpr int kFgMaxStages = 4, kFgFlush = 64;

__global__ void __launch_bounds__(kFgThreads, 1) fgrad_split_kernel(const __grid_constant__ SplitFgArgs A)
{
    extern __shared__ __align__(1024) unsigned char sp_smem[];
    struct Hdr {
        unsigned long long full[kFgMaxStages], empty[kFgMaxStages];
        unsigned long long hdone[4], hfree[4];     // large products of unit 0, 1, 2; bias
        unsigned long long ldone[3], lfree[3], drain;
        uint32_t tmem_base;
        volatile int failed;
        __align__(16) __nv_bfloat16 ones[64];      // one core matrix of 1.0: operand of the bias gradient
    };
    static_assert(sizeof(Hdr) <= kSplitHeader, "header does not fit");
    Hdr* H = reinterpret_cast<Hdr*>(sp_smem);
    unsigned char* ring = sp_smem + kSplitHeader;
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (the shuffle tells the compiler that it is the same for the warp)
    const int K = A.K, KK = K * K, E = A.E;

    const int kr = A.rows3 ? 1 : K;                                   // window rows that are roles of their own
    const int nroles = A.slices * A.nci * kr;
    const int role = (int)blockIdx.x % nroles, share = (int)blockIdx.x / nroles;
    const int ky = role % kr, cs = (role / kr) % A.nci, slice = role / (kr * A.nci);
    const int mp = A.Ms / 8;
    const int ci0 = cs * A.ncols * (K == 1 ? A.units : 1);
    const int cspan = min(A.ncols * (K == 1 ? A.units : 1), A.cin16 - ci0);       // input channels of this block
    const int nu = K == 1 ? (cspan + A.ncols - 1) / A.ncols : A.units;             // units with work
    const bool with_bias = cs == 0 && ky == 0;
    const int s_lo = (int)((long long)share * A.stages_total / A.shares), s_hi = (int)((long long)(share + 1) * A.stages_total / A.shares);
    const int ns = s_hi - s_lo;
    // entries between the parts of the two tiles (planes beyond the layer's channels arrive as zeros, or are read from what
    // lies behind: they only reach accumulator rows and columns of no channel)
    const uint32_t dz_part = (uint32_t)(A.dz_box * E), x_part = (uint32_t)(A.x_box * A.x_entries);
    const uint32_t x_tile = 3u * x_part;                              // entries of an input tile (rows3: one per window row)
    auto unit_cols = [&](int u) { return K == 1 ? min(A.ncols, cspan - u * A.ncols) : cspan; };

    const int wide = (A.rows3 ? 3 : 1) * A.ncols;                     // columns of a unit's accumulators
    // Steps of a stage: the large products of every unit, then the bias.  Step g (over all stages) takes slot g % slots behind
    // the accumulators of the small products, and starts when step g - slots has been read.  Barriers by step of the
    // stage: their phases are the stages
    // (no more slots than steps: with two phases of one barrier under way a waiter could miss the older one)
    const uint32_t hcol = (uint32_t)(A.units * wide);
    const int steps = nu + (with_bias ? 1 : 0), slots = min(steps, min(2, (kTcTmemCols - A.units * wide) / wide));

    if (threadIdx.x == 0) {
        for (int s = 0; s < kFgMaxStages; ++s) { mbar_init(smem_u32(&H->full[s]), 1); mbar_init(smem_u32(&H->empty[s]), 3); }
        for (int s = 0; s < 4; ++s) { mbar_init(smem_u32(&H->hdone[s]), 1); mbar_init(smem_u32(&H->hfree[s]), 4); }
        for (int s = 0; s < 3; ++s) { mbar_init(smem_u32(&H->ldone[s]), A.rows3 ? 2 : 1); mbar_init(smem_u32(&H->lfree[s]), 4); }
        mbar_init(smem_u32(&H->drain), 3);
        H->failed = 0;
        fence_mbar_init();
    }
    if (threadIdx.x < 64) H->ones[threadIdx.x] = __float2bfloat16(1.0f);
    if (warp == 0) { __syncwarp(); tmem_alloc(smem_u32(&H->tmem_base), (uint32_t)kTcTmemCols); }
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

    if (warp < 12) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");
        const int u = warp >> 2, q = warp & 3;
        if (u < nu) {
            const int cols = unit_cols(u) * (A.rows3 ? 3 : 1);
            float acc[128];
#pragma unroll
            for (int j = 0; j < 128; ++j) acc[j] = 0.f;
            float bacc = 0.f;
            const bool bias = with_bias && u == 0;
            auto plain = [](float a, float b) { return a + b; };
            auto add = [&](uint32_t col, auto sum) {
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if (t * 16 < cols) {
                        float v[16];
                        tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + col + (uint32_t)(t * 16), v);
#pragma unroll
                        for (int j = 0; j < 16; ++j) acc[t * 16 + j] = sum(acc[t * 16 + j], v[j]);
                    }
                fence_before_sync();
                __syncwarp();
            };
            for (int i = 0; i < ns; ++i) {
                if (!wait(&H->hdone[u], (uint32_t)i & 1u, 32)) break;
                fence_after_sync();
                add(hcol + (uint32_t)((i * steps + u) % slots * wide), plain);
                if (lane == 0) mbar_arrive(smem_u32(&H->hfree[u]));
                if (bias) {
                    if (!wait(&H->hdone[3], (uint32_t)i & 1u, 32)) break;
                    fence_after_sync();
                    const uint32_t at = tmem + ((uint32_t)(q * 32) << 16) + hcol + (uint32_t)((i * steps + nu) % slots * wide);
                    uint32_t r, rs;
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(at) : "memory");
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(rs) : "r"(at + 16u) : "memory");
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    bacc = add_small(bacc + __uint_as_float(r), __uint_as_float(rs));
                    fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&H->hfree[3]));
                }
                if (i % kFgFlush == kFgFlush - 1 || i == ns - 1) {
                    if (!wait(&H->ldone[u], (uint32_t)(i / kFgFlush) & 1u, 32)) break;
                    fence_after_sync();
                    add((uint32_t)(u * wide), add_small);       // (the large products of the same stages are in)
                    if (lane == 0) mbar_arrive(smem_u32(&H->lfree[u]));
                }
            }
            // registers -> this share's partial set: lane quarter q holds rows 32 q .. (Ms = 128) or rows 16 q .. in its first 16 lanes
            const int row = A.Ms == 128 ? q * 32 + lane : q * 16 + lane;
            const int co = slice * A.Ms + row;
            if ((A.Ms == 128 || lane < 16) && co < A.cout16) {
                float* set = A.partial + (size_t)share * A.set_floats + A.tgp_off;
#pragma unroll
                for (int t = 0; t < 8; ++t)
                    if (t * 16 < cols) {
                        int tap, ci;
                        if (A.rows3) { const int kx = t * 16 / A.cin16; tap = u * 3 + kx; ci = t * 16 - kx * A.cin16; }
                        else if (K == 1) { tap = 0; ci = ci0 + u * A.ncols + t * 16; }
                        else { tap = ky * 3 + u; ci = ci0 + t * 16; }
                        float4* dst = reinterpret_cast<float4*>(set + ((size_t)tap * A.cout16 + co) * A.cin16 + ci);
#pragma unroll
                        for (int j = 0; j < 4; ++j) dst[j] = make_float4(acc[t * 16 + 4 * j], acc[t * 16 + 4 * j + 1], acc[t * 16 + 4 * j + 2], acc[t * 16 + 4 * j + 3]);
                    }
                if (bias) set[(size_t)KK * A.cout16 * A.cin16 + co] = bacc;
            }
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (warp == 12) {
            // ---- producer ----
            int issued = 0;
            for (int i = 0; i < ns; ++i) {
                const int s = i % A.nstages;
                bool ok = wait(&H->empty[s], ((uint32_t)(i / A.nstages) & 1u) ^ 1u);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (lane == 0) {
                    const int e = A.e_lo + (s_lo + i) * E;
                    const uint32_t bar = smem_u32(&H->full[s]), dst0 = smem_u32(ring + (size_t)s * A.stage_bytes);
                    const uint32_t xdst0 = dst0 + 3u * dz_part * 16u;
                    mbar_expect_tx(bar, (3u * dz_part + (A.rows3 ? 3u : 1u) * x_tile) * 16u);
                    tma_load_3d(dst0, A.tmap_dz, 2 * e, slice * mp, 0, bar);
                    if (A.rows3)
                        for (int r = 0; r < 3; ++r) tma_load_3d(xdst0 + (uint32_t)r * x_tile * 16u, A.tmap_x, 2 * (e + (r - 1) * A.g.wp - 1), 0, 0, bar);
                    else
                        tma_load_3d(xdst0, A.tmap_x, 2 * (e + (K == 3 ? (ky - 1) * A.g.wp - 1 : 0)), ci0 / 8, 0, bar);
                }
                __syncwarp();
                ++issued;
            }
            if (H->failed)
                for (int s = 0; s < A.nstages; ++s) {
                    const int n = issued > s ? (issued - 1 - s) / A.nstages + 1 : 0;
                    if (n > 0) mbar_wait(smem_u32(&H->full[s]), (uint32_t)(n - 1) & 1u, 200000000ll);
                }
        } else {
            // ---- MMA issue: one thread the large products and the bias, two the small ones (by unit; rows3, where an MMA of 32
            // columns takes half the time that a thread needs to issue it: by unit and window column) ----
            const int role = warp - 13;
            if (lane == 0) {
                const uint32_t a_hi = desc_hi((uint32_t)E * 16u), x_hi = desc_hi((uint32_t)A.x_entries * 16u);
                const uint64_t ones_d = make_desc(smem_u32(H->ones), 0, 0);
                const uint32_t idb = make_idesc(A.Ms, 16, true, true);
                const int nk = E >> 4;
                bool ok = true;
                // one product of one unit (rows3: of one window column): a chain over the entries of the stage
                auto chain = [&](uint32_t tcol, uint32_t a, uint32_t x, uint32_t idesc, bool acc) {
                    mma_bf16(tcol, desc64(a_hi, a), desc64(x_hi, x), idesc, acc);
                    mma_bf16(tcol, desc64(a_hi, a + 16), desc64(x_hi, x + 16), idesc, true);
                    if (nk == 4) {
                        mma_bf16(tcol, desc64(a_hi, a + 32), desc64(x_hi, x + 32), idesc, true);
                        mma_bf16(tcol, desc64(a_hi, a + 48), desc64(x_hi, x + 48), idesc, true);
                    }
                };
                for (int i = 0; i < ns && ok; ++i) {
                    const int s = i % A.nstages;
                    if (!wait(&H->full[s], (uint32_t)(i / A.nstages) & 1u)) break;
                    fence_after_sync();
                    const uint32_t dz0 = desc_lo(smem_u32(ring + (size_t)s * A.stage_bytes), 128);
                    const uint32_t x0 = desc_lo(smem_u32(ring + (size_t)s * A.stage_bytes) + 3u * dz_part * 16u, 128);
                    auto unit_x = [&](int u) { return x0 + (A.rows3 ? (uint32_t)u * x_tile : (uint32_t)(K == 1 ? u * (A.ncols / 8) * A.x_entries : u)); };
                    if (role == 0) {
                        for (int k = 0; k < steps; ++k) {
                            const int g = i * steps + k, gp = g - slots;                 // the step that used the slot before
                            if (gp >= 0) {
                                const int kp = gp % steps;
                                if (!wait(&H->hfree[kp == nu ? 3 : kp], (uint32_t)(gp / steps) & 1u)) { ok = false; break; }
                                fence_after_sync();
                            }
                            const uint32_t tcol = tmem + hcol + (uint32_t)(g % slots * wide);
                            if (k < nu) {
                                const uint32_t idesc = make_idesc(A.Ms, unit_cols(k), true, true), xu = unit_x(k);
                                for (int kx = 0; kx < (A.rows3 ? 3 : 1); ++kx)
                                    chain(tcol + (uint32_t)(kx * A.cin16), dz0, xu + (uint32_t)kx, idesc, false);
                            } else
                                for (int part = 2; part >= 0; --part)                    // bias: sums of dz, a contraction with ones; 16 columns for
                                    for (int ks = 0; ks < nk; ++ks)                      // the first part, 16 for the others (a slot has 32 at least)
                                        mma_bf16(tcol + (part ? 16u : 0u), desc64(a_hi, dz0 + (uint32_t)part * dz_part + 16u * (uint32_t)ks), ones_d, idb, part == 1 || ks > 0);
                            mma_commit(smem_u32(&H->hdone[k == nu ? 3 : k]));
                        }
                    } else {
                        const bool fresh = i % kFgFlush == 0, last = i % kFgFlush == kFgFlush - 1 || i == ns - 1;
                        for (int u = 0; u < nu && ok; ++u) {
                            if (!A.rows3 && (u & 1) != role - 1) continue;
                            if (fresh && i > 0) {
                                if (!wait(&H->lfree[u], (uint32_t)(i / kFgFlush - 1) & 1u)) { ok = false; break; }
                                fence_after_sync();
                            }
                            const uint32_t idesc = make_idesc(A.Ms, unit_cols(u), true, true), xu = unit_x(u);
                            for (int kx = 0; kx < (A.rows3 ? 3 : 1); ++kx) {
                                if (A.rows3 && ((u * 3 + kx) & 1) != role - 1) continue;
                                const uint32_t tcol = tmem + (uint32_t)(u * wide + kx * A.cin16);
#pragma unroll
                                for (int j = 0; j < 5; ++j) {           // (dz part, x part)
                                    constexpr int pd[5] = {0, 2, 1, 0, 1}, px[5] = {2, 0, 1, 1, 0};
                                    chain(tcol, dz0 + (uint32_t)pd[j] * dz_part, xu + (uint32_t)px[j] * x_part + (uint32_t)kx, idesc, !(fresh && j == 0));
                                }
                            }
                            if (last) mma_commit(smem_u32(&H->ldone[u]));
                        }
                    }
                    if (!ok) break;
                    mma_commit(smem_u32(&H->empty[s]));
                }
                mma_commit(smem_u32(&H->drain));
            }
        }
        __syncwarp();
    }
    __syncthreads();
    if (warp == 0) {
        if (lane == 0) mbar_wait(smem_u32(&H->drain), 0, 200000000ll);
        __syncwarp();
        fence_after_sync();
        tmem_dealloc(tmem, (uint32_t)kTcTmemCols);
    }
}

// fp32 NCHW map -> split map, zero entries included.  One thread per entry and 8-channel plane.
__global__ void split_planes_kernel(const float* __restrict__ src, uint4* __restrict__ dst, const __grid_constant__ SplitGeom g, int C)
{
    previous_launches();
    const long long total = (long long)g.planes * g.tp;
    const size_t HW = (size_t)g.H * g.W, part = (size_t)g.planes * g.tp;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int pl = (int)(i / g.tp), e = (int)(i - (long long)pl * g.tp);
        int n, y, x;
        float v[8];
        const bool ok = pixel_of(g, e, n, y, x);
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = (ok && pl * 8 + c < C) ? __ldg(src + ((size_t)n * C + pl * 8 + c) * HW + (size_t)y * g.W + x) : 0.f;
        store_split(dst, part, (size_t)i, v);
    }
}

// dz = delta * leaky'(y) at the conv's resolution as a split map, from an fp32 NCHW delta (the last layer, and below a
// group that does not run on these kernels).  One thread per entry of the layer's OUTPUT map and plane; through a pool it
// writes the four members of the window.
__global__ void split_delta_kernel(const __grid_constant__ SplitDeltaArgs A)
{
    previous_launches();
    const SplitGeom& g = A.low;
    const long long total = (long long)g.planes * g.tp;
    const size_t HW = (size_t)g.H * g.W, part = (size_t)A.g.planes * A.g.tp;
    if (A.pool) zero_margins(A.dz, A.g, kSplitLead, kSplitLead + A.g.rows * A.g.wp);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int pl = (int)(i / g.tp), e = (int)(i - (long long)pl * g.tp);
        int n, y, x;
        float v[8];
        const bool ok = pixel_of(g, e, n, y, x);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            v[c] = 0.f;
            if (ok && pl * 8 + c < A.C) {
                const size_t at = ((size_t)n * A.C + pl * 8 + c) * HW + (size_t)y * g.W + x;
                v[c] = __ldg(A.d + at) * (__ldg(A.y + at) > 0.f ? 1.f : A.slope);
            }
        }
        if (!A.pool) { store_split(A.dz, part, (size_t)i, v); continue; }
        if (e < kSplitLead || e >= kSplitLead + g.rows * g.wp) continue;
        const int row = (e - kSplitLead) / g.wp, row2 = row == 0 ? 0 : 1 + n * (A.g.H + 1) + 2 * y;
        const bool two_r = row > 0 && y < g.H, two_c = x < g.W;
        const size_t e2 = (size_t)pl * A.g.tp + kSplitLead + (size_t)row2 * A.g.wp + 2 * x;
        const unsigned long long am = ok ? __ldg(A.arg + i) : 0ull;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            if (((w >> 1) && !two_r) || ((w & 1) && !two_c)) continue;
            float z[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) z[c] = (int)((am >> (8 * c)) & 3ull) == w ? v[c] : 0.f;
            store_split(A.dz, part, e2 + (size_t)(w >> 1) * A.g.wp + (w & 1), z);
        }
    }
}

__global__ void __launch_bounds__(256) pack_split_kernel(const __grid_constant__ PackTilesArgs A, const float* __restrict__ params)
{
    previous_launches();
    __shared__ float s[kPackSmemFloats];
    pack_tiles<3>(A, params, s, [](const float* v, uint4* p) { split8<false>(v, p[0], p[1], p[2]); });
}

}  // namespace sp
}  // namespace ftp
