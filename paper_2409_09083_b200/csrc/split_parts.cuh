// Split maps (split_args.hpp) as the kernels that write them see them: the three bf16 parts of a value, the places of the entries.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "split_args.hpp"

namespace ftp {
namespace sp {

// largest magnitude of three values, NaN if one of them is
__device__ __forceinline__ float max_abs(float a, float b, float c)
{
    float d;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Three bf16 parts of eight values: the value rounded to 6 significant bits (nearest, ties away from zero), the rest rounded to
// bf16, and the rest of that, which bf16 holds exactly.  Where one of the eight is within 2^-7 of the largest fp32, so that its first
// part would be an infinity, or is infinite or NaN, the first parts are cut to 6 bits instead (the three parts then hold
// 23 bits at least).  An infinity becomes (itself, NaN, NaN), a NaN NaNs: see add_small.
// (One comparison for the eight.  One per value: a step with 16 layers 0.8 % slower; a branch to code for the rare ones in the
// midst of the unrolled output phases of conv_split_kernel: 5 %.)
// kSign: a positive value has a positive first part, however small it is (below 2^-132 the smallest bf16, 2^-133; the second part
// makes up for it): the backward pass takes the sign of a saved value from there.
template <bool kSign>
__device__ __forceinline__ void split8(const float* v, uint4& p0, uint4& p1, uint4& p2)
{
    uint32_t* a = &p0.x; uint32_t* b = &p1.x; uint32_t* c = &p2.x;
    const float top = max_abs(max_abs(max_abs(v[0], v[1], v[2]), v[3], v[4]), max_abs(v[5], v[6], v[7]), 0.f);
    const uint32_t round = top < __int_as_float(0x7f7e0000) ? 0x20000u : 0u;
    auto first = [&](float x) {
        const uint32_t f = (__float_as_uint(x) + round) & 0xfffc0000u;
        return kSign && __float_as_int(x) > 0 ? max(f, 0x10000u) : f;
    };
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float x = v[2 * i], y = v[2 * i + 1];
        const uint32_t bx = first(x), by = first(y);
        a[i] = __byte_perm(bx, by, 0x7632);
        const float rx = x - __uint_as_float(bx), ry = y - __uint_as_float(by);
        const __nv_bfloat162 h1 = __floats2bfloat162_rn(rx, ry);
        const float2 f1 = __bfloat1622float2(h1);
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(rx - f1.x, ry - f1.y);
        b[i] = *reinterpret_cast<const uint32_t*>(&h1);
        c[i] = *reinterpret_cast<const uint32_t*>(&h2);
    }
}
__device__ __forceinline__ void store_split(uint4* base, size_t part_stride, size_t at, const float* v)
{
    uint4 p0, p1, p2;
    split8<true>(v, p0, p1, p2);
    base[at] = p0; base[at + part_stride] = p1; base[at + 2 * part_stride] = p2;
}

// Adds the products of the lower parts (small) to a sum that holds those of the first parts (large).  Where an operand is infinite or
// NaN, the products of the first parts alone have the sum that fp32 multiply-adds have; the others stay out.
__device__ __forceinline__ float add_small(float large, float small) { return fabsf(large) < __int_as_float(0x7f800000) ? large + small : large; }

// pixel of an entry (n, y, x); false: a zero entry of the map (edge column, row between images, lead or tail)
__device__ __forceinline__ bool pixel_of(const SplitGeom& g, int e, int& n, int& y, int& x)
{
    const int r = e - kSplitLead, row = r / g.wp;
    x = r - row * g.wp;
    const int t = row - 1;
    n = t / (g.H + 1); y = t - n * (g.H + 1);
    return r >= 0 && t >= 0 && row < g.rows && x < g.W && y < g.H;
}

// zeros to the entries of every plane of a split map in front of `lo` and from `hi` on (all threads of the grid)
__device__ __forceinline__ void zero_margins(uint4* out, const SplitGeom& g, int lo, int hi)
{
    const int per = lo + (g.tp - hi);
    const long long total = 3ll * g.planes * per;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int pl = (int)(i / per), j = (int)(i - (long long)pl * per);
        out[(size_t)pl * g.tp + (j < lo ? j : hi + j - lo)] = make_uint4(0, 0, 0, 0);
    }
}

// zeros to every entry of a split map that is not a pixel: lead, tail, the column behind every row, the rows between the images
// (all threads of the grid; for kernels that write the pixels only)
__device__ __forceinline__ void zero_frame(uint4* out, const SplitGeom& g)
{
    const int lead = kSplitLead, tail = g.tp - kSplitLead - g.rows * g.wp, edge = g.rows, between = (g.N + 1) * g.W;
    const int per = lead + tail + edge + between;
    const long long total = 3ll * g.planes * per;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const int pl = (int)(i / per);
        int j = (int)(i - (long long)pl * per), e;
        if (j < lead) e = j;
        else if ((j -= lead) < tail) e = kSplitLead + g.rows * g.wp + j;
        else if ((j -= tail) < edge) e = kSplitLead + j * g.wp + g.W;
        else { j -= edge; const int r = j / g.W; e = kSplitLead + r * (g.H + 1) * g.wp + (j - r * g.W); }
        out[(size_t)pl * g.tp + e] = make_uint4(0, 0, 0, 0);
    }
}

}  // namespace sp
}  // namespace ftp
