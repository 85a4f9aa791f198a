// Interface of dc_conv_cluster.cu: one (tile, channel block) per cluster of CTAs, the reduction split over its CTAs.
#pragma once
#include <cuda.h>

#include "dc_common.cuh"

constexpr int kClusterStages = 8;

struct dc_cluster_args {
    const float* bias; __nv_bfloat16* out;
    const int32_t* tile_list; const int32_t* tile_count; const uint32_t* masks;
    int Ho, Wo, Co, Ci, kh, kw, sh, sw, ph, pw, relu, tiles_x, tiles_y;
    int BN, NB, BK, kchunks, stages, a_bytes, b_bytes, nb_off, CS;
    uint32_t idesc, sbo, layout_type, tmem_cols;
    int32_t* status;
    unsigned long long wait_ns;
    int skip_loads;
    int early;                               // tile list, count and bitmaps are older than the kernel before this one (dc_lists_settled)
    // element-wise add of a later layer done here: add_out = (this layer's output) + add_in (+ ReLU), or NULL
    const __nv_bfloat16* add_in; __nv_bfloat16* add_out; int add_relu;
};

size_t dc_cluster_smem(int stages, int a_bytes, int b_bytes, int BN);
// clusters of cs CTAs with that much shared memory that the device runs at the same time
int dc_cluster_wave(int device, int cs, size_t smem);
// tiles: length of the tile list (upper bound of the count on the device)
int dc_launch_cluster_kernel(dc_cache* c, const CUtensorMap& tmA, const CUtensorMap& tmB, const dc_cluster_args& a, int tiles);
