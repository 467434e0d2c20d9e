// Host side of the row-walking upsample + cross-entropy kernel (k_upsample_ce_rows.cuh): which instantiation a launch takes, and
// the tile maps of its inputs.
#include "k_upsample_ce_rows.cuh"

#include <string.h>

namespace st {

static RowsKernels rows_kernels(int C)
{
    RowsKernels (*const file[])(int) = {rows_kernels_0, rows_kernels_1, rows_kernels_2, rows_kernels_3, rows_kernels_4};
    int k = 0;
    while (C > kRowsLast[k]) ++k;
    return file[k](C);
}

bool upsample_ce_rows_supported(int C) { return C <= 32; }

int upsample_ce_rows_blocks(int h, int w) { return ((h + RN_Y - 1) / RN_Y) * ((w + RN_X - 1) / RN_X); }

cudaError_t prepare_upsample_ce_rows(int C) { return rows_kernels(C).prepare(); }

void launch_upsample_ce_rows(const UpsampleCeArgs& a, const CUtensorMap* z_map, cudaStream_t s, const CUtensorMap* x_map, const CUtensorMap* w_map)
{
    CUtensorMap none;
    memset(&none, 0, sizeof(none));
    UpsampleCeArgs b = a;
    if (b.fused && !(x_map && w_map && fused_forward_supported(b.C, b.h, b.w, b.kblocks * 64))) b.fused = 0;
    if (b.fused) { b.has_map = 0; rows_kernels(b.C).launch(b, none, *x_map, *w_map, s); return; }
    b.x_early = 0;
    if (!(b.has_map && z_map)) b.has_map = 0;
    rows_kernels(b.C).launch(b, b.has_map ? *z_map : none, none, none, s);
}

// The block multiplies its own logits when the classifier is a 1x1 layer over at most 256 channels (a multiple of 64)
// and the feature map is at least one tile large.
bool fused_forward_supported(int C, int h, int w, int c_in)
{
    return upsample_ce_rows_supported(C) && c_in >= 64 && c_in % 64 == 0 && c_in / 64 <= fused::kMaxKBlocks && w >= fused::kTileCols && h >= fused::kTileRows;
}

bool make_logit_tile_map(CUtensorMap* m, const float* z, int S, int C, int h, int w)
{
    if (!upsample_ce_rows_supported(C) || w % 4 != 0 || w < kTwLoad || h < TZ_H || ((uintptr_t)z & 15u)) return false;
    const uint64_t dims[3] = {(uint64_t)w, (uint64_t)h, (uint64_t)S * C};
    const uint64_t strides[2] = {(uint64_t)w * sizeof(float), (uint64_t)h * w * sizeof(float)};
    const uint32_t box[3] = {(uint32_t)kTwLoad, (uint32_t)TZ_H, (uint32_t)C};
    char err[128];
    return encode_tensor_map(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, CU_TENSOR_MAP_SWIZZLE_NONE, z, 3, dims, strides, box, err,
                             sizeof(err), "logit tile");
}

bool make_feature_tile_map(CUtensorMap* m, const bf16* x, int S, int c_in, int h, int w)
{
    if (c_in % 64 != 0 || w < kTwFused || h < TZ_H || ((uintptr_t)x & 15u)) return false;
    const uint64_t c = (uint64_t)c_in;
    const uint64_t dims[4] = {c, (uint64_t)w, (uint64_t)h, (uint64_t)S};
    const uint64_t strides[3] = {c * 2, (uint64_t)w * c * 2, (uint64_t)h * w * c * 2};
    const uint32_t box[4] = {64, (uint32_t)kTwFused, (uint32_t)TZ_H, 1};
    char err[128];
    return encode_tensor_map(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, CU_TENSOR_MAP_SWIZZLE_128B, x, 4, dims, strides, box, err,
                             sizeof(err), "feature tile");
}

}  // namespace st
