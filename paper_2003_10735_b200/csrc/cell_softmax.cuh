// Softmax over the 16 frame pixels between four neighbouring feature-map nodes (a "cell" of the bilinear x4 upsample):
// the arithmetic shared by the two upsample + cross-entropy kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace st {

constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;
// Largest change of a class's logit between two corners of a cell (in log2 units) for which the cell stays on the
// fast path.  All 16 products of the progressions are exponentials of the cell's own pixels (at most 1 after the
// shift), the step factors stay below 2^20, and the relative error of a product grows with the size of the exponent
// arguments: about 5e-6 at this limit, below the tolerance of the logit gradient.
#ifndef ST_K3_FAST_RANGE
#define ST_K3_FAST_RANGE 40.0f
#endif
constexpr float kFastRange = ST_K3_FAST_RANGE;

__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Byte k: (row eighths) x (column eighths of pixel k toward the left node column: 7, 5, 3, 1; toward the right one:
// 1, 3, 5, 7) -- the integer adjoint weights (units of 1/64) of a row's four pixels for one corner node.
__host__ __device__ constexpr uint32_t corner_weights(int row_eighths, bool right)
{
    return right ? (uint32_t)(row_eighths * 1) | (uint32_t)(row_eighths * 3) << 8 | (uint32_t)(row_eighths * 5) << 16 | (uint32_t)(row_eighths * 7) << 24
                 : (uint32_t)(row_eighths * 7) | (uint32_t)(row_eighths * 5) << 8 | (uint32_t)(row_eighths * 3) << 16 | (uint32_t)(row_eighths * 1) << 24;
}

// One class inside the lane's cell, its logit u bilinear between the four corner nodes (a, b: the lane's own node column,
// upper and lower node row, raw logits; the right-hand column comes from the next lane).  With ly_r = (2r+1)/8 and
// fr_k = (2k+1)/8:  u(r,k) = A + B k + G r + D k r, so the 16 exponentials E(r,k) = exp2(u(r,k) log2 e - M) are geometric
// progressions along k and r, products of four quantities that cost four exp2:  x01 = (E(0,0), E(1,0)),
// x23 = (E(2,0), E(3,0)) and the per-row ratios between neighbouring pixels q01 = (q_0, q_1), q23 = (q_2, q_3),
// E(r,k) = E(r,0) q_r^k.  Returns the largest corner difference in the logits' own units (the caller leaves the fast path
// if a class changes by more than kFastRange log2-units across the cell: the progressions would lose their small terms).
__device__ __forceinline__ float cell_bases(float a, float b, float M, float2& x01, float2& x23, float2& q01, float2& q23)
{
    const float ar = __shfl_down_sync(0xffffffffu, a, 1), br = __shfl_down_sync(0xffffffffu, b, 1);
    const float p = b - a, qq = br - ar, e0 = ar - a;
    const float qp = qq - p;
    const float wv = fmaf(qp, 0.125f, e0);
    const float A = fmaf(wv, 0.125f, fmaf(p, 0.125f, a));
    const float E00 = ex2_approx(fmaf(A, kLog2e, -M)), QB = ex2_approx((0.25f * kLog2e) * wv),
                TG = ex2_approx(fmaf(qp, 0.03125f * kLog2e, (0.25f * kLog2e) * p)), SD = ex2_approx((0.0625f * kLog2e) * qp);
    // rows (0, 1) and (2, 3) ride in the two halves of packed fp32x2 registers: one multiply advances two rows
    const float TG2 = TG * TG, SD2 = SD * SD;
    q01 = make_float2(QB, QB * SD);
    q23 = __fmul2_rn(q01, make_float2(SD2, SD2));
    x01 = make_float2(E00, E00 * TG);
    x23 = __fmul2_rn(x01, make_float2(TG2, TG2));
    return fmaxf(fabsf(p), fmaxf(fabsf(qq), fabsf(e0)));
}

// All 16 of them: X01[k] = (E(0,k), E(1,k)), X23[k] = (E(2,k), E(3,k)), 6 more packed multiplications
__device__ __forceinline__ float cell_exponentials(float a, float b, float M, float2 (&X01)[4], float2 (&X23)[4])
{
    float2 q01, q23;
    const float change = cell_bases(a, b, M, X01[0], X23[0], q01, q23);
#pragma unroll
    for (int k = 1; k < 4; ++k) {
        X01[k] = __fmul2_rn(X01[k - 1], q01);
        X23[k] = __fmul2_rn(X23[k - 1], q23);
    }
    return change;
}

// A class's sums of E(r,k) times the pixel weights W of the four rows (packed by row pairs like the exponentials).  A row's
// sum is E(r,0) times a cubic in q_r with the weights as coefficients: Horner's rule, the progression itself is not
// formed again.
__device__ __forceinline__ void cell_row_sums(float2 x01, float2 x23, float2 q01, float2 q23, const float2 (&W01)[4], const float2 (&W23)[4],
                                              float2& s01, float2& s23)
{
    s01 = W01[3]; s23 = W23[3];
#pragma unroll
    for (int k = 2; k >= 0; --k) { s01 = __ffma2_rn(s01, q01, W01[k]); s23 = __ffma2_rn(s23, q23, W23[k]); }
    s01 = __fmul2_rn(s01, x01); s23 = __fmul2_rn(s23, x23);
}

}  // namespace st
