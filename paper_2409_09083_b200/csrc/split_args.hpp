// Arguments and host-side launchers of the split kernels (split.cuh): the fp32 path on the tensor cores.
#pragma once

#include <cstddef>
#include <cstdint>

#include <vector_types.h>

#include "launch_stream.hpp"
#include "plan.hpp"

namespace ftp {

// A "split map" holds an fp32 map as three bf16 maps whose sum is the map (see split.cuh): 16-byte entries (8 channels of
// a pixel) in planes [part][channel / 8][entry], every plane one flat run of `tp` entries over the whole batch:
//   entry(n, y, x) = kSplitLead + (1 + n (H + 1) + y) wp + x,   wp = W + 1
// i.e. rows of W pixels and one zero entry behind them, one zero row above every image and below the last one, so that
// the neighbours of a pixel at the edge of its image are zeros and a window position is a constant offset.
constexpr int kSplitLead = 8;
struct SplitGeom {
    int N, H, W, planes;        // planes = channels padded to 16, / 8
    int wp, rows, tp;           // entries per row, rows (N (H + 1) + 1), entries per plane
};
inline SplitGeom split_geom(int N, int C, int H, int W)
{
    SplitGeom g{N, H, W, (C + 15) / 16 * 2, W + 1, N * (H + 1) + 1, 0};
    g.tp = (kSplitLead + g.rows * g.wp + g.wp + 80 + 7) / 8 * 8;      // the tail stays zero too: a stage of the filter gradient may run over
    return g;
}
inline size_t split_bytes(const SplitGeom& g) { return (size_t)3 * g.planes * g.tp * 16; }
constexpr size_t kSplitSlack = 256 * 1024;     // workspace bytes in front of and behind a split map that a tile may read (values discarded)

struct SplitConvArgs {
    alignas(64) unsigned char tmap[128];   // tensor map of `in`: kSplitFlat, 1x1: {entries, planes, parts}; tiles: {columns, rows, planes, parts}
    const uint4* in;                // split map, the conv's input (forward) or dz (input delta)
    const uint4* w;                 // packed filters, see pack_split_kernel
    const float* bias;              // cout floats or null
    int* error;
    SplitGeom g;                    // of `in`
    int K, nchunks, kpc;            // window, chunks of kpc 8-channel planes
    int cout, cout16, Ns, slices, nblk;
    int mode;                       // kSplitFlat, kSplitTile, kSplitPool
    int R, Cw, tiles_x, tiles_y, pitch, run_len;
    int items;
    int a_plane, a_bytes, a_block, a_stages, b_stage, b_stages, pool_bytes;   // a_block: entries between the 128-entry blocks of a tile
    float slope; int act;           // act != 0: leaky ReLU after the bias
    uint4* out_s; SplitGeom og;     // output as a split map (the pooled map in mode kSplitPool; dz of the layer below with prev_y), or
    float* out_f;                   // output as fp32 NCHW
    unsigned long long* arg;        // kSplitPool: arg-max bytes, one word per 8-channel plane and entry of the pooled map
    // input delta into the dz map of the split layer below: its saved output (part 0 gives the sign), its slope, and where it
    // ends with a pool its arg-max words (out_s then has twice the resolution)
    const uint4* prev_y; const unsigned long long* prev_arg; float prev_slope;
};

struct SplitFgArgs {
    alignas(64) unsigned char tmap_dz[128];   // {entries, planes, parts}: one box is a stage's dz tile
    alignas(64) unsigned char tmap_x[128];    // one box is a stage's input tile (rows3: one part of one copy)
    const uint4* dz; const uint4* x;
    SplitGeom g;                    // geometry (planes: of dz); x has the same rows and tp
    int x_planes;
    float* partial; long long set_floats, tgp_off;
    int* error;
    int K, cout16, cin16;
    int Ms, slices, ncols, units, nci, rows3;
    int E, e_lo, stages_total, shares;
    int nstages, stage_bytes, x_entries, dz_box, x_box;   // boxes: planes per part
};

struct SplitDeltaArgs {             // fp32 NCHW delta -> dz split map
    const float* d;                 // delta at the layer's output
    const float* y;                 // the layer's output, fp32 NCHW
    const unsigned long long* arg;  // pool: arg-max words of the pooled map (entries of `low`)
    uint4* dz; SplitGeom g;         // at the conv's resolution
    SplitGeom low;                  // geometry of the output map (= g without a pool)
    int C; float slope; int pool;
};

bool split_prepare_device();
void split_launch_conv(const SplitConvArgs& a, int nb, int blocks, int smem, LaunchStream ls);
void split_launch_fgrad(const SplitFgArgs& a, int blocks, int smem, LaunchStream ls);
void split_launch_planes(const float* src, uint4* dst, const SplitGeom& g, int C, LaunchStream ls);
void split_launch_delta(const SplitDeltaArgs& a, LaunchStream ls);

// Packing launches (pack.cuh): 32 x 32 channel tiles [tile_begin, next layer's tile_begin) of a layer.
struct PackTilesLayer { long long p_off; uint4* wf; uint4* wd; int cin, cout, k, cin16, cout16, ns_f, kpc_f, ns_d, kpc_d, tile_begin;
                        int stack_d;      // the rotated arrangement by window column, its rows from the last to the first (the stacked form of conv_tc_rows_kernel)
                        int only; };      // 1 / 2: the forward arrangement / the rotated one only
constexpr int kPackTilesLayers = 32;
struct PackTilesArgs {
    int n, tiles;
    int dirs;                       // 1: forward arrangement, 2: input delta, 3: both
    int* error;                     // error word to clear, or null
    PackTilesLayer l[kPackTilesLayers];
};
void split_launch_pack(const PackTilesArgs& a, const float* params, LaunchStream ls);   // three parts

}  // namespace ftp
