// Filters [cout][cin][k][k] -> the packed arrangements of the tensor-core kernels that take a layer's channels in slices and
// chunks (tc_stationary.cuh: one bf16 part; split.cuh: three parts whose sum is the fp32 value), per slice and chunk the
// parts one after another:
//   wf[slice][chunk][part][tap][kpc][Ns][8]   rows = output channels, contraction = input channels     (forward)
//   wd[slice][chunk][part][tap'][kpc][Ns][8]  rows = input channels, contraction = output channels, rotated (input delta)
// Rows and planes beyond the padded channel counts are not written: the kernels' MMAs do not read them.
//
// A block takes a tile of 32 x 32 channels through shared memory, so that both sides are coalesced: the filters of 32 input
// channels are one contiguous run of an output channel's row, and the entries of 32 rows leave as 512-byte runs.  (One thread per
// entry, gathering its 8 filters at a stride of 36 bytes or of a whole row, took 230 us for the 79 MB of a 23-layer
// stack, this 53 us.)
#pragma once

#include "split_args.hpp"

namespace ftp {

template <int KK, int PARTS, class Parts>
__device__ __forceinline__ void pack_tile(const PackTilesLayer L, int t, int dirs, const float* __restrict__ params, float* s, Parts parts)
{
    constexpr int pitch = 32 * KK + 1;                        // odd: rows (output channels) of a column fall into different banks
    const int tci = (L.cin16 + 31) / 32, co0 = t / tci * 32, ci0 = t % tci * 32;
    const int run = min(32, L.cin - ci0) * KK, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = warp + 8 * i;
        const float* src = params + L.p_off + ((long long)(co0 + r) * L.cin + ci0) * KK;
        const bool ok = co0 + r < L.cout;
#pragma unroll
        for (int j = lane; j < 32 * KK; j += 32) s[r * pitch + j] = (ok && j < run) ? __ldg(src + j) : 0.f;
    }
    __syncthreads();
    constexpr int total = 32 * 4 * KK;
    for (int i = ((dirs & 1) ? 0 : total) + (int)threadIdx.x; i < ((dirs & 2) ? 2 * total : total); i += 256) {
        const bool fwd = i < total;
        const int j = fwd ? i : i - total, r = j & 31, o = (j >> 5) & 3, tap = j >> 7;   // row of the operand, octet of contraction channels
        const int row = (fwd ? co0 : ci0) + r, k0 = (fwd ? ci0 : co0) + o * 8;
        if (row >= (fwd ? L.cout16 : L.cin16) || k0 >= (fwd ? L.cin16 : L.cout16)) continue;
        const int ns = fwd ? L.ns_f : L.ns_d, kpc = fwd ? L.kpc_f : L.kpc_d;
        const int nch = ((fwd ? L.cin16 : L.cout16) / 8 + kpc - 1) / kpc;
        float v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = fwd ? s[r * pitch + (o * 8 + c) * KK + tap] : s[(o * 8 + c) * pitch + r * KK + KK - 1 - tap];
        uint4 p[PARTS];
        parts(v, p);
        const int sl = row / ns, rr = row - sl * ns, kp = k0 / 8, ch = kp / kpc, kj = kp - ch * kpc;
        const size_t stage = (size_t)KK * kpc * ns;
        const size_t at = !fwd && L.stack_d ? (size_t)(tap % 3 * kpc + kj) * 3 + (2 - tap / 3) : (size_t)tap * kpc + kj;
        uint4* dst = (fwd ? L.wf : L.wd) + ((size_t)sl * nch + ch) * PARTS * stage + at * ns + rr;
#pragma unroll
        for (int q = 0; q < PARTS; ++q) dst[q * stage] = p[q];
    }
}

template <int PARTS, class Parts>
__device__ __forceinline__ void pack_tiles(const PackTilesArgs& A, const float* __restrict__ params, float* s, Parts parts)
{
    if (A.error && blockIdx.x == 0 && threadIdx.x == 0) *A.error = 0;
    int l = 0;
    while (l + 1 < A.n && (int)blockIdx.x >= A.l[l + 1].tile_begin) ++l;
    const PackTilesLayer L = A.l[l];                          // (a copy: through a reference every field is a memory load)
    const int t = (int)blockIdx.x - L.tile_begin, dirs = L.only ? A.dirs & L.only : A.dirs;
    if (!dirs) return;
    if (L.k == 3) pack_tile<9, PARTS>(L, t, dirs, params, s, parts);
    else pack_tile<1, PARTS>(L, t, dirs, params, s, parts);
}

constexpr int kPackSmemFloats = 32 * (32 * 9 + 1);

}  // namespace ftp
