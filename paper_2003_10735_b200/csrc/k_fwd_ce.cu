// Host side of the upsample + cross-entropy kernel for at most 32 classes (k_fwd_ce.cuh): which shapes its own forward takes, which
// instantiation a launch uses, and the tile map of the features.
#include "k_fwd_ce.cuh"

namespace st {

static FwdCeKernels fwd_ce_kernels(int C)
{
    FwdCeKernels (*const file[])(int) = {fwd_ce_kernels_0, fwd_ce_kernels_1, fwd_ce_kernels_2, fwd_ce_kernels_3, fwd_ce_kernels_4};
    int k = 0;
    while (C > kFwdCeLast[k]) ++k;
    return file[k](C);
}

// A classifier over at most 256 channels (a multiple of 64) and a feature map of at least one tile
bool fused_forward_supported(int C, int h, int w, int c_in)
{
    return C <= kClassPad && c_in >= 64 && c_in % 64 == 0 && c_in / 64 <= fused::kMaxKBlocks && w >= F_COLS && h >= F_ROWS;
}

bool upsample_ce_few_supported(int C) { return C <= kClassPad; }

int upsample_ce_few_blocks(int h, int w) { return ((h + FN_Y - 1) / FN_Y) * ((w + FN_X - 1) / FN_X); }

cudaError_t prepare_fwd_ce(int C, bool own_forward, bool with_gradient, int tiles, int n_sms) { return fwd_ce_kernels(C).prepare(own_forward, with_gradient, tiles, n_sms); }

void launch_fwd_ce(const UpsampleCeArgs& a, const CUtensorMap& x_map, const CUtensorMap& w_map, const CUtensorMap& row_map, cudaStream_t s) { fwd_ce_kernels(a.C).launch[1](a, x_map, w_map, row_map, s); }

void launch_upsample_ce_few(const UpsampleCeArgs& a, cudaStream_t s)
{
    UpsampleCeArgs b = a;
    b.x_early = 0; b.w_part = nullptr;
    CUtensorMap none;
    memset(&none, 0, sizeof none);
    fwd_ce_kernels(b.C).launch[0](b, none, none, none, s);
}

// one box: `channels` channels of `rows` rows of a tile
static bool make_tile_map(CUtensorMap* m, const bf16* x, int S, int c_in, int h, int w, int rows, int channels)
{
    if (c_in % 64 != 0 || w < F_COLS || h < F_ROWS || ((uintptr_t)x & 15u)) return false;
    const uint64_t c = (uint64_t)c_in;
    const uint64_t dims[4] = {c, (uint64_t)w, (uint64_t)h, (uint64_t)S};
    const uint64_t strides[3] = {c * 2, (uint64_t)w * c * 2, (uint64_t)h * w * c * 2};
    const uint32_t box[4] = {(uint32_t)channels, (uint32_t)F_COLS, (uint32_t)rows, 1};
    char err[128];
    return encode_tensor_map(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, channels == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, x, 4, dims, strides, box, err,
                             sizeof(err), "feature tile");
}

bool make_feature_tile_map(CUtensorMap* m, const bf16* x, int S, int c_in, int h, int w) { return make_tile_map(m, x, S, c_in, h, w, F_ROWS, 64); }
bool make_feature_chunk_map(CUtensorMap* m, const bf16* x, int S, int c_in, int h, int w, bool two_groups)
{
    const bool half = half_rows(two_groups ? kTwoGroups : kOneGroup);
    return make_tile_map(m, x, S, c_in, h, w, half ? F_ROWS : 5, half ? 32 : 64);
}
bool make_feature_row_map(CUtensorMap* m, const bf16* x, int S, int c_in, int h, int w) { return make_tile_map(m, x, S, c_in, h, w, 1, 64); }

}  // namespace st
