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

void launch_upsample_ce_rows(const UpsampleCeArgs& a, const CUtensorMap* z_map, cudaStream_t s)
{
    CUtensorMap none;
    memset(&none, 0, sizeof(none));
    UpsampleCeArgs b = a;
    b.x_early = 0;
    if (!z_map) b.has_map = 0;
    rows_kernels(b.C).launch(b, b.has_map ? *z_map : none, s);
}

bool make_logit_tile_map(CUtensorMap* m, const float* z, int S, int C, int h, int w)
{
    if (!upsample_ce_rows_supported(C) || w % 4 != 0 || w < TZ_W || h < TZ_H || ((uintptr_t)z & 15u)) return false;
    const uint64_t dims[3] = {(uint64_t)w, (uint64_t)h, (uint64_t)S * C};
    const uint64_t strides[2] = {(uint64_t)w * sizeof(float), (uint64_t)h * w * sizeof(float)};
    const uint32_t box[3] = {(uint32_t)TZ_W, (uint32_t)TZ_H, (uint32_t)C};
    char err[128];
    return encode_tensor_map(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, CU_TENSOR_MAP_SWIZZLE_NONE, z, 3, dims, strides, box, err,
                             sizeof(err), "logit tile");
}

}  // namespace st
