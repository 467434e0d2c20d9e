// bf16 tensor-core GEMMs of the head (gemm_precision 1): Forward and PartialBackward of Algorithm 1
// for the trainable back part (Section 4.2), as TMA-fed tcgen05 kernels with fp32 accumulators in
// tensor memory.  Operands are bf16 (cached features, bf16 copies of the weights, rounded
// gradients); every accumulation is fp32.
//
//   fwd 1x1   z[c][pix]       = b[c] + sum_k A[pix][k] W[c][k]                 A = features or hidden
//   fwd 3x3   Hd[pix][co]     = ReLU(b1[co] + sum_{tap,ci} X[pix+tap][ci] W1[tap][co][ci])
//   wgrad 1x1 dW[c][k]        = sum_pix dz[c][pix] A[pix][k]                   split over pixel ranges
//   dgrad     dHd[pix][k]     = [Hd[pix][k] > 0] sum_c dz[c][pix] W2[c][k]     (bf16 out; one kernel with wgrad 1x1)
//   wgrad 3x3 dW1[tap][co][ci]= sum_pix dHd[pix][co] X[pix+tap][ci]            split over pixel ranges
//
// Pixel-major activations [pix][channel] are K-major operands when the GEMM reduces over channels
// (forward) and MN-major operands when it reduces over pixels (weight gradients); both forms are
// read straight from the same TMA 128-byte-swizzled tiles, no transposing pass exists.
// The zero padding of the 3x3 convolution is TMA's out-of-bounds fill: boxes reach beyond the map of a [channel][x][y][stream]
// tensor map.
#include "st_internal.h"
#include "tc_common.cuh"
#include "train_ctl.cuh"

#include <cstdio>
#include <algorithm>
#include <cstring>

namespace st {

using namespace tc;

namespace {

constexpr int kThreadsTc = 128;          // 4 warps: TMEM lanes 32w .. 32w+31 belong to warp w
constexpr int kBlockK = 64;              // bf16 elements per 128-byte swizzled row
constexpr int kTileM = 128;              // UMMA M
constexpr int kChunkPix = 64;            // pixels per pipeline stage of the weight-gradient GEMMs
constexpr int kTileW = 8, kTileH = 16;   // 3x3 forward: 128 pixels = 16 rows x 8 columns
constexpr int kChunkW = 32, kChunkH = 4; // 3x3 wgrad: 128 pixels = 4 rows x 32 columns
constexpr int kSmemAlign = 1024;
constexpr int kMaxKBlocks = 16;
// Pipeline depth of the 1x1 weight gradient (20 KB per stage): three, which lets three blocks work on an SM, or five where every
// block has an SM of its own
constexpr int kWg1Stages = 3, kWg1Deep = 5;

__device__ __forceinline__ uint8_t* align_smem(uint8_t* p)
{
    return (uint8_t*)(((uintptr_t)p + kSmemAlign - 1) & ~(uintptr_t)(kSmemAlign - 1));
}

// ------------------------------------------------------------------------------------------------
// fwd 1x1: one 128-pixel tile per block; the whole K extent is loaded at once (one barrier per
// 64-channel block so that the MMAs start while later blocks are still in flight).
// ------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreadsTc)
tc_fwd1x1_kernel(const __grid_constant__ CUtensorMap tmA,   // {K, p, S}  box {64, 128, 1}
                 const __grid_constant__ CUtensorMap tmB,   // {K, 32, S} box {64, 32, 1}
                 const float* __restrict__ theta, int64_t n_params, int64_t b_off,
                 float* __restrict__ z, int C, int p, int kblocks, unsigned int* err, const int* __restrict__ skip, int64_t skip_stride,
                 int a_early, uint32_t spin_limit, uint32_t stall_bytes)
{
    // spin_limit / stall_bytes: kSpinLimit and 0 in normal use.  A test of the give-up path lowers the limit and makes
    // the first barrier expect stall_bytes more than its copies deliver, so that the wait on it runs out: every copy
    // that was issued still lands, the kernel records where it gave up, writes nothing, frees its tensor memory and
    // returns.
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_smem(smem_raw);
    const uint32_t a_base = smem_u32(smem);
    const uint32_t b_base = a_base + kblocks * (kTileM * 128);
    __shared__ __align__(8) uint64_t bars[kMaxKBlocks + 1];
    __shared__ uint32_t tmem_slot, gave_up;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int s = blockIdx.y, pix0 = blockIdx.x * kTileM;

    if (warp == 0) tmem_alloc(smem_u32(&tmem_slot), 32);
    if (tid == 0) {
        for (int i = 0; i <= kblocks; ++i) mbar_init(smem_u32(&bars[i]), 1);
        gave_up = 0;
        fence_barrier_init();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_slot;
    // a_early: the kernel before this one on the stream (the previous iteration's parameter update) writes the weights
    // but not the activations, and this kernel was launched to start while that one still runs: the activation tile
    // is fetched now, the weights after the wait.  Each barrier expects both parts.
    if (a_early && warp == 0 && elect_one()) {
        for (int kb = 0; kb < kblocks; ++kb) {
            const uint32_t bar = smem_u32(&bars[kb]);
            mbar_expect_tx(bar, kTileM * 128 + kClassPad * 128 + (kb == 0 ? stall_bytes : 0u));
            tma_load_3d(a_base + kb * (kTileM * 128), &tmA, bar, kb * kBlockK, pix0, s);
        }
    }
    pdl_wait();                  // the weights (and, without a_early, the activations) come from the previous kernel
    if (skip && skip[(int64_t)blockIdx.y * skip_stride]) {     // this stream's training loop has ended (block-uniform; the flag
        tc_fence_before_sync();                                 // comes from an earlier kernel, so it is read after the wait)
        __syncthreads();
        if (warp == 0) tmem_dealloc(tmem, 32);
        return;
    }
    const uint32_t done_bar = smem_u32(&bars[kblocks]);
    bool ok = true;

    if (warp == 0) {
        if (elect_one())
            for (int kb = 0; kb < kblocks; ++kb) {
                const uint32_t bar = smem_u32(&bars[kb]);
                if (!a_early) {
                    mbar_expect_tx(bar, kTileM * 128 + kClassPad * 128 + (kb == 0 ? stall_bytes : 0u));
                    tma_load_3d(a_base + kb * (kTileM * 128), &tmA, bar, kb * kBlockK, pix0, s);
                }
                tma_load_3d(b_base + kb * (kClassPad * 128), &tmB, bar, kb * kBlockK, 0, s);
            }
    } else if (warp == 1) {
        constexpr uint32_t idesc = instr_desc(kTileM, kClassPad, 0, 0);
        for (int kb = 0; kb < kblocks; ++kb) {
            ok = mbar_wait(smem_u32(&bars[kb]), 0, err, kWaitFull, spin_limit);
            if (!ok) { gave_up = 1; break; }
            tc_fence_after_sync();
            if (elect_one()) {
                const uint64_t da = smem_desc(a_base + kb * (kTileM * 128), 16, 1024), db = smem_desc(b_base + kb * (kClassPad * 128), 16, 1024);
#pragma unroll
                for (int k = 0; k < 4; ++k) umma(tmem, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
            }
            __syncwarp();
        }
        if (elect_one()) umma_commit(done_bar);
    }
    __syncwarp();
    ok = mbar_wait(done_bar, 0, err, kWaitDone);
    pdl_launch_dependents();     // only the epilogue is left
    tc_fence_after_sync();
    __syncthreads();
    if (gave_up) ok = false;     // the issuing thread ran out of patience: nothing was multiplied, nothing is written
    if (ok) {
        float v[32];
        tmem_ld_32x32(tmem + ((uint32_t)(warp * 32) << 16), v);
        const int pix = pix0 + tid;
        if (pix < p) {
            const float* bias = theta + (int64_t)s * n_params + b_off;
            float* dst = z + (int64_t)s * C * p + pix;
#pragma unroll
            for (int c = 0; c < kClassPad; ++c)
                if (c < C) dst[(int64_t)c * p] = v[c] + __ldg(bias + c);
        }
    } else {
        drain_after_error();
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 32);
}

// ------------------------------------------------------------------------------------------------
// wgrad 1x1: D[k][c] += sum over this block's pixel chunks of A[pix][k] * dz[c][pix].
// A (pixel-major activations) is the MN-major operand with M = channel; dz rows are K-major.
// ------------------------------------------------------------------------------------------------
template <int STAGES>
__global__ void __launch_bounds__(kThreadsTc)
tc_wgrad1x1_kernel(const __grid_constant__ CUtensorMap tmA,   // {K, p, S}      box {64, 64, 1}
                   const __grid_constant__ CUtensorMap tmB,   // {p, 32, S}     box {64, 32, 1}
                   float* __restrict__ partials,              // [S][n_split][32][K]
                   int K, int n_chunks, int chunks_per_block, int m_split, int tmem_cols, unsigned int* err,
                   const int* __restrict__ skip, int64_t skip_stride, int a_early, int has_ctl, const TrainCtl ctl)
{
    // Train: the block after the last one of the weight gradient assesses the prediction (metric, best so far, break)
    // while the others multiply; it takes no part in anything below
    // The streams from the last to the first, as the loss kernel walks them from the first to the last: what it has left in L2 is read
    // from there, and so is what this kernel leaves by the next loss kernel.  us of a call of eight steps, 256 channels 180 x 320, first to
    // last / last to first: 4 streams 960 / 931, 8 1849 / 1799, 16 3513 / 3521; 128 channels, 6 streams 1146 / 1124.
    const int s = (int)gridDim.y - 1 - (int)blockIdx.y;
    if (has_ctl && blockIdx.x == gridDim.x - 1) {
        const TrainHistory hist = train_history(ctl, s);
        pdl_wait();
        bool stop, better;
        train_decision(ctl, s, true, hist, nullptr, stop, better);
        pdl_launch_dependents();
        return;
    }
    const int n_blocks_x = (int)gridDim.x - (has_ctl ? 1 : 0);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_smem(smem_raw);
    // m_split blocks share a pixel range, each with its own 128-channel accumulators: with the channels divided the
    // pixel ranges are longer and fewer, and the update has that many fewer partial sums to add per weight
    const int m_all = (K + kTileM - 1) / kTileM;     // accumulators (128 channels each) of the whole layer
    const int m_tiles = m_all / m_split;             // ... of this block
    const int m0 = ((int)blockIdx.x % m_split) * m_tiles;
    const int a_blocks = m_tiles * 2;                // 64-channel blocks loaded per stage (absent ones are zero-filled)
    const uint32_t a_stage_bytes = a_blocks * (kChunkPix * 128);
    const uint32_t stage_bytes = a_stage_bytes + kClassPad * 128;
    const uint32_t base = smem_u32(smem);
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], done;
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int split = (int)blockIdx.x / m_split, n_split = n_blocks_x / m_split;
    const int c_begin = split * chunks_per_block;
    const int c_end = min(n_chunks, c_begin + chunks_per_block);

    if (warp == 0) tmem_alloc(smem_u32(&tmem_slot), tmem_cols);
    if (tid == 0) {
        for (int i = 0; i < STAGES; ++i) { mbar_init(smem_u32(&full[i]), 1); mbar_init(smem_u32(&empty[i]), 1); }
        mbar_init(smem_u32(&done), 1);
        fence_barrier_init();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_slot;
    // a_early: the activations are the frozen features, which no kernel of the loop writes, and this kernel may have been
    // launched while its predecessor (which produces the logit gradient) is still running: the activation part of the
    // first stages is fetched now, the gradient part after the wait.  Each barrier expects both parts.
    const int n_pre = a_early ? min(STAGES, c_end - c_begin) : 0;
    if (warp == 0 && elect_one())
        for (int it = 0; it < n_pre; ++it) {
            const uint32_t bar = smem_u32(&full[it]), sa = base + it * stage_bytes;
            mbar_expect_tx(bar, stage_bytes);
            for (int cb = 0; cb < a_blocks; ++cb)
                tma_load_3d(sa + cb * (kChunkPix * 128), &tmA, bar, (2 * m0 + cb) * kBlockK, (c_begin + it) * kChunkPix, s);
        }
    pdl_wait();                  // inputs come from the previous kernel of the step
    if (skip && skip[(int64_t)s * skip_stride]) {     // this stream's training loop has ended (block-uniform; the flag
        tc_fence_before_sync();                                 // comes from an earlier kernel, so it is read after the wait)
        __syncthreads();
        if (warp == 0) tmem_dealloc(tmem, tmem_cols);
        return;
    }
    bool ok = true;

    if (warp == 0) {
        for (int i = c_begin; i < c_end; ++i) {
            const int it = i - c_begin, st = it % STAGES;
            if (it >= STAGES) ok = mbar_wait(smem_u32(&empty[st]), ((it / STAGES) - 1) & 1, err, kWaitEmpty);
            if (!ok) break;
            if (elect_one()) {
                const uint32_t bar = smem_u32(&full[st]), sa = base + st * stage_bytes;
                if (it >= n_pre) {
                    mbar_expect_tx(bar, stage_bytes);
                    for (int cb = 0; cb < a_blocks; ++cb)
                        tma_load_3d(sa + cb * (kChunkPix * 128), &tmA, bar, (2 * m0 + cb) * kBlockK, i * kChunkPix, s);
                }
                tma_load_3d(sa + a_stage_bytes, &tmB, bar, i * kChunkPix, 0, s);
            }
            __syncwarp();
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = instr_desc(kTileM, kClassPad, 1, 0);
        for (int i = c_begin; i < c_end; ++i) {
            const int it = i - c_begin, st = it % STAGES;
            ok = mbar_wait(smem_u32(&full[st]), (it / STAGES) & 1, err, kWaitFull);
            if (!ok) break;
            tc_fence_after_sync();
            if (elect_one()) {
                const uint64_t da = smem_desc(base + st * stage_bytes, kChunkPix * 128, 1024), db = smem_desc(base + st * stage_bytes + a_stage_bytes, 16, 1024);
                for (int m = 0; m < m_tiles; ++m)
#pragma unroll
                    for (int j = 0; j < kChunkPix / 16; ++j)
                        umma(tmem + m * kClassPad, da + ((2 * m * (kChunkPix * 128) + j * (16 * 128)) >> 4), db + 2 * j, idesc, (it | j) != 0);
                umma_commit(smem_u32(&empty[st]));
            }
            __syncwarp();
        }
        if (elect_one()) umma_commit(smem_u32(&done));
    }
    __syncwarp();
    ok = mbar_wait(smem_u32(&done), 0, err, kWaitDone);
    pdl_launch_dependents();     // only the epilogue is left
    tc_fence_after_sync();
    if (ok) {
        float* dst = partials + ((int64_t)s * n_split + split) * kClassPad * K;
        const bool any = c_end > c_begin;
        for (int m = 0; m < m_tiles; ++m) {
            float v[32];
            tmem_ld_32x32(tmem + ((uint32_t)(warp * 32) << 16) + m * kClassPad, v);
            const int k = (m0 + m) * kTileM + tid;
            if (k < K)
#pragma unroll
                for (int c = 0; c < kClassPad; ++c) dst[(int64_t)c * K + k] = any ? v[c] : 0.f;
        }
    } else {
        drain_after_error();
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, tmem_cols);
}

// ------------------------------------------------------------------------------------------------
// fwd 3x3 (+bias, ReLU), persistent: one block per SM walks items of one or two tiles (HALVES; a tile is 16 rows x 8 columns of
// pixels) times N output channels.  All nine taps read one slab of pixels: for 64 channels the 18 rows x (8 HALVES + 2) columns
// around the item, one copy.  A tap's operand of 128 pixels is the slab from another start: eight pixels of a row are eight
// consecutive 128-byte rows of the slab (the swizzle follows the address, so they may begin anywhere) and the next image row
// begins one slab row further, which is the descriptor's stride between groups of eight.  Four roles: warp 0 feeds a ring of weight
// stages (one tap of 64 channels each) and the last warp two slabs, by TMA across item boundaries (the pipeline never drains), a
// thread of warp 1 issues the MMAs into one of two sets of tensor-memory accumulators, two groups of four warps drain the other set (bias, ReLU,
// bf16, ReLU bit mask) meanwhile: a tile each, or every other 64 channels where an item is one tile.
// ------------------------------------------------------------------------------------------------
constexpr int kFwd3Threads = 352;

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// ------------------------------------------------------------------------------------------------
// fwd 1x1, persistent: gridDim.x blocks per stream walk the stream's 128-pixel tiles.  Three roles as in the 3x3
// forward: one thread feeds a ring of shared-memory stages by TMA across tile boundaries (one 128-pixel x 64-channel
// block per stage, 128 KB in flight), one thread issues the MMAs into one of two tensor-memory accumulators, the
// epilogue warps drain the other one (bias, fp32 logits, planar) meanwhile.  The classifier weights are loaded once
// per block.
// ------------------------------------------------------------------------------------------------
#ifndef ST_F1_STAGES
#define ST_F1_STAGES 8
#endif
constexpr int kF1Threads = 192, kF1Stages = ST_F1_STAGES;
constexpr uint32_t kOutPieceBytes = 32 * 128;     // 3x3 tile walk: 32 pixels x 64 channels of an epilogue warp on their way out
constexpr int kWg3LeastChunks = 5;                // chunks in a range of a 3x3 weight gradient
constexpr int kMaxWStages = 16;                   // ... weight stages of its ring
__host__ __device__ constexpr int slab_cols(int halves) { return kTileW * halves + 2; }
__host__ __device__ constexpr uint32_t slab_bytes(int halves) { return ((uint32_t)slab_cols(halves) * (kTileH + 2) * 128 + 1023) / 1024 * 1024; }
constexpr uint32_t kF1StageBytes = kTileM * 128;

__global__ void __launch_bounds__(kF1Threads)
tc_fwd1x1p_kernel(const __grid_constant__ CUtensorMap tmA,   // {K, p, S}  box {64, 128, 1}
                  const __grid_constant__ CUtensorMap tmB,   // {K, 32, S} box {64, 32, 1}
                  const float* __restrict__ theta, int64_t n_params, int64_t b_off,
                  float* __restrict__ z, int C, int p, int kblocks, unsigned int* err,
                  const int* __restrict__ skip, int64_t skip_stride)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_smem(smem_raw);
    const uint32_t a_base = smem_u32(smem);
    const uint32_t b_base = a_base + kF1Stages * kF1StageBytes;
    __shared__ __align__(8) uint64_t full[kF1Stages], empty[kF1Stages], b_full, acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int s = blockIdx.y;
    const int n_items = (p + kTileM - 1) / kTileM;

    if (warp == 0) tmem_alloc(smem_u32(&tmem_slot), 2 * kClassPad);
    if (tid == 0) {
        for (int i = 0; i < kF1Stages; ++i) { mbar_init(smem_u32(&full[i]), 1); mbar_init(smem_u32(&empty[i]), 1); }
        mbar_init(smem_u32(&b_full), 1);
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&acc_full[i]), 1); mbar_init(smem_u32(&acc_empty[i]), 4); }
        fence_barrier_init();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_slot;
    pdl_wait();                  // inputs come from the previous kernel of the step
    if (skip && skip[(int64_t)blockIdx.y * skip_stride]) {     // this stream's training loop has ended (block-uniform; the flag
        tc_fence_before_sync();                                 // comes from an earlier kernel, so it is read after the wait)
        __syncthreads();
        if (warp == 0) tmem_dealloc(tmem, 2 * kClassPad);
        return;
    }
    bool ok = true;

    if (warp == 0) {
        // ---- producer (it and the issuer walk their loops as whole warps, one lane issues)
        if (elect_one()) {
            const uint32_t bb = smem_u32(&b_full);
            mbar_expect_tx(bb, (uint32_t)kblocks * kClassPad * 128);
            for (int kb = 0; kb < kblocks; ++kb) tma_load_3d(b_base + kb * (kClassPad * 128), &tmB, bb, kb * kBlockK, 0, s);
        }
        __syncwarp();
        int g = 0;
        for (int it = blockIdx.x; it < n_items && ok; it += gridDim.x) {
            for (int kb = 0; kb < kblocks; ++kb, ++g) {
                const int st = g % kF1Stages;
                if (g >= kF1Stages) ok = mbar_wait(smem_u32(&empty[st]), ((g / kF1Stages) - 1) & 1, err, kWaitEmpty);
                if (!ok) break;
                if (elect_one()) {
                    const uint32_t bar = smem_u32(&full[st]);
                    mbar_expect_tx(bar, kF1StageBytes);
                    tma_load_3d(a_base + st * kF1StageBytes, &tmA, bar, kb * kBlockK, it * kTileM, s);
                }
                __syncwarp();
            }
        }
        pdl_launch_dependents();     // every load is issued: the next kernel of the step may set itself up
    } else if (warp == 1) {
        // ---- MMA issuer
        constexpr uint32_t idesc = instr_desc(kTileM, kClassPad, 0, 0);
        ok = mbar_wait(smem_u32(&b_full), 0, err, kWaitFull);
        int g = 0, j = 0;
        for (int it = blockIdx.x; it < n_items && ok; it += gridDim.x, ++j) {
            const int buf = j & 1;
            if (j >= 2) ok = mbar_wait(smem_u32(&acc_empty[buf]), ((j >> 1) - 1) & 1, err, kWaitEmpty);
            if (!ok) break;
            tc_fence_after_sync();
            const uint32_t acc = tmem + buf * kClassPad;
            for (int kb = 0; kb < kblocks; ++kb, ++g) {
                const int st = g % kF1Stages;
                ok = mbar_wait(smem_u32(&full[st]), (g / kF1Stages) & 1, err, kWaitFull);
                if (!ok) break;
                tc_fence_after_sync();
                if (elect_one()) {
                    const uint64_t da = smem_desc(a_base + st * kF1StageBytes, 16, 1024), db = smem_desc(b_base + kb * (kClassPad * 128), 16, 1024);
#pragma unroll
                    for (int k = 0; k < 4; ++k) umma(acc, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
                    umma_commit(smem_u32(&empty[st]));
                }
                __syncwarp();
            }
            if (ok && elect_one()) umma_commit(smem_u32(&acc_full[buf]));
            __syncwarp();
        }
    } else if (warp >= 2) {
        // ---- epilogue warps: TMEM lanes 32*(warp % 4) .. +31 = pixels of the tile
        const int q = warp & 3;
        const float* bias = theta + (int64_t)s * n_params + b_off;
        int j = 0;
        for (int it = blockIdx.x; it < n_items && ok; it += gridDim.x, ++j) {
            const int buf = j & 1;
            ok = mbar_wait(smem_u32(&acc_full[buf]), (j >> 1) & 1, err, kWaitDone);
            if (!ok) break;
            tc_fence_after_sync();
            float v[32];
            tmem_ld_32x32(tmem + ((uint32_t)(q * 32) << 16) + buf * kClassPad, v);
            const int pix = it * kTileM + q * 32 + lane;
            if (pix < p) {
                float* dst = z + (int64_t)s * C * p + pix;
#pragma unroll
                for (int c = 0; c < kClassPad; ++c)
                    if (c < C) dst[(int64_t)c * p] = v[c] + __ldg(bias + c);
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[buf]));
        }
    }
    if (!ok) drain_after_error();
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 2 * kClassPad);
}

// MODE 0: the layer's forward (bias, ReLU, bf16 output, one ReLU bit per output value).
// MODE 1: the gradient passed back through the layer to the block before it: the same walk over the layer's output gradient with
//         the weights transposed and their taps mirrored (prepared by the update kernel); the epilogue applies the ReLU mask of
//         the receiving block, writes bf16 and emits per-tile channel sums of the unrounded values (the receiving block's bias
//         gradient).
// The K loop runs over (kblocks1 + kblocks2) channel blocks x 9 taps: the first kblocks1 come from tmA (the previous block's
// output, or the frozen part's), the others from tmA2 (the block's skip input): the concatenation of Section 5.2 is never
// materialised.
// Bound by the tensor pipe at 256 channels inside a tile (560 cycles per weight stage where its multiplications need 512, 58 bytes a
// cycle of weights from L2), by the issue of MMAs at 64 (450 to 540 per stage of eight, which read operands for 384), and by start
// and tile changes.  us a launch, 720p, with a copy of the shifted pixels for every tap, tiles of 4 rows x 32 columns and a warp that
// waits, votes and elects per stage / now: 128 + 64 -> 64 channels 29.5 / 25.2, 64 + 64 -> 64 26.4 / 19.2, gradient 64 -> 64 passed
// back 16.0 / 13.5, 256 -> 128 35.7 / 30.3; three of 101 x 187, 192 -> 128 29.0 / 25.0; 256 -> 256 50.0 / 50.2 (180 rows are 11.25
// tiles; fewer copies, more tiles), at 1080p 110 / 109.  The slab alone, without the issuing thread, changed nothing: eight MMAs with a
// wait between them took 780 cycles; the slabs' own warp 1 us at 1080p; small rings of pieces 52.4 -> 50.2.
template <int HALVES, int MODE>
__global__ void __launch_bounds__(kFwd3Threads)
tc_fwd3x3_kernel(const __grid_constant__ CUtensorMap tmA,   // {C1, w, h, S}     box {64, 8 HALVES + 2, 18, 1}
                 const __grid_constant__ CUtensorMap tmA2,  // {C2, w, h, S}     same box (unused if kblocks2 == 0)
                 int kblocks1, int kblocks2,
                 const __grid_constant__ CUtensorMap tmB,   // {C1+C2, 9*Ch, S}  box {64, Ch, 1}
                 const __grid_constant__ CUtensorMap tmBq,  // same tensor, box {64, 64, 1}: one block of 64 output channels
                 int w_stages,                               // weight stages of the ring
                 int n_full, int n_items, int tail_split,    // items: n_full whole ones, then the others cut into tail_split (1, 2 or
                                                             // 4) ranges of output channels
                 const float* __restrict__ theta, int64_t n_params, int64_t b_off,   // MODE 0: bias
                 const __grid_constant__ CUtensorMap tmO,   // output {Ch, w, h, S} box {64, 8, 4, 1}
                 uint32_t* __restrict__ relu_bits,           // [S][p][Ch/32]: bit k of word j = out[32j + k] > 0 (MODE 0: written;
                                                             //   MODE 1: the receiving block's bits, read)
                 float* __restrict__ b_partials,             // MODE 1: [S][tiles per stream][Ch] channel sums of each tile
                 int Ch, int h, int w, int acc_cols, unsigned int* err, const int* __restrict__ skip, int64_t skip_stride)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_smem(smem_raw);
    const uint32_t base = smem_u32(smem);
    constexpr int P = slab_cols(HALVES);
    constexpr uint32_t kSlab = slab_bytes(HALVES);
    const uint32_t w_base = base + 2 * kSlab, w_bytes = (uint32_t)Ch * 128;
    // The ring of weight stages, and the one it becomes for items that are a range of the output channels: smaller stages, more of
    // them (with four stages the copies' latency, not the tensor pipe, sets the pace of such items).
    const int p_stages = min(kMaxWStages, w_stages * tail_split);
    const uint32_t p_bytes = w_bytes / (uint32_t)tail_split;
    __shared__ __align__(8) uint64_t s_full[2], s_empty[2], full[2 * kMaxWStages], empty[2 * kMaxWStages], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ __align__(16) float part_of[8 * 256];            // per epilogue warp: MODE 0 the bias, MODE 1 channel sums of the tile
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int tiles_x = (w + kTileW - 1) / kTileW, tiles_y = (h + kTileH - 1) / kTileH;
    const int items_x = (tiles_x + HALVES - 1) / HALVES, items_per_stream = items_x * tiles_y;
    const int kblocks = kblocks1 + kblocks2;
    struct Item { int s, tx, ty, ch0, chn; };
    auto item_of = [&](int wi) {
        Item it;
        int k = wi;
        it.ch0 = 0; it.chn = Ch;
        if (wi >= n_full) { const int q = wi - n_full; k = n_full + q / tail_split; it.chn = Ch / tail_split; it.ch0 = (q % tail_split) * it.chn; }
        it.s = k / items_per_stream;
        const int r = k - it.s * items_per_stream;
        it.ty = r / items_x; it.tx = (r - it.ty * items_x) * HALVES;
        return it;
    };

    if (warp == 0) {
        if (elect_one()) { prefetch_map(&tmA); prefetch_map(&tmB); }
        __syncwarp();
        tmem_alloc(smem_u32(&tmem_slot), acc_cols);
    }
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&s_full[i]), 1); mbar_init(smem_u32(&s_empty[i]), 1);
            mbar_init(smem_u32(&acc_full[i]), 1); mbar_init(smem_u32(&acc_empty[i]), 8);
        }
        for (int i = 0; i < 2 * kMaxWStages; ++i) { mbar_init(smem_u32(&full[i]), 1); mbar_init(smem_u32(&empty[i]), 1); }
        fence_barrier_init();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_slot;
    pdl_wait();                  // inputs come from the previous kernel of the step
    bool ok = true;

    if (warp == 0) {
        // ---- weights (the whole warp walks the loop, its first lane issues)
        int st = 0, n_st = w_stages;
        uint32_t parity = 1;             // a barrier nobody has arrived at yet counts as one whose phase 1 has ended
        uint32_t f0 = smem_u32(&full[0]), e0 = smem_u32(&empty[0]);
        bool pieces = false;
        for (int wi = blockIdx.x; wi < n_items && ok; wi += gridDim.x) {
            const Item im = item_of(wi);
            if (skip && skip[(int64_t)im.s * skip_stride]) continue;     // all roles leave out the same items
            const uint32_t item_w = (uint32_t)im.chn * 128;
            if (!pieces && im.chn != Ch) {                               // the other ring begins when all of the first one has been read
                for (int i = 0; i < w_stages && ok; ++i) {
                    ok = mbar_wait(e0 + 8 * st, parity, err, kWaitEmpty);
                    if (++st == w_stages) { st = 0; parity ^= 1; }
                }
                pieces = true;
                st = 0; n_st = p_stages; parity = 1;
                f0 += 8 * kMaxWStages; e0 += 8 * kMaxWStages;
            }
            for (int kb = 0; kb < kblocks && ok; ++kb)
                for (int row = 0; row < 9 * Ch; row += Ch) {
                    ok = mbar_wait(e0 + 8 * st, parity, err, kWaitEmpty);
                    if (!ok) break;
                    if (elect_one()) {
                        const uint32_t bar = f0 + 8 * st, sw = w_base + st * item_w;
                        mbar_expect_tx(bar, item_w);
                        if (im.chn == Ch) tma_load_3d(sw, &tmB, bar, kb * kBlockK, row, im.s);
                        else
                            for (int j = 0; j < im.chn / 64; ++j)    // 64 weight rows per copy, laid out like the single copy
                                tma_load_3d(sw + j * (64 * 128), &tmBq, bar, kb * kBlockK, row + im.ch0 + j * 64, im.s);
                    }
                    __syncwarp();
                    if (++st == n_st) { st = 0; parity ^= 1; }
                }
        }
        pdl_launch_dependents();     // every load is issued: the next kernel of the step may set itself up
    } else if (warp == kFwd3Threads / 32 - 1) {
        // ---- slabs
        int sl = 0;
        uint32_t parity = 1;
        for (int wi = blockIdx.x; wi < n_items && ok; wi += gridDim.x) {
            const Item im = item_of(wi);
            if (skip && skip[(int64_t)im.s * skip_stride]) continue;
            const int x = im.tx * kTileW - 1, y = im.ty * kTileH - 1;
            for (int kb = 0; kb < kblocks; ++kb) {
                ok = mbar_wait(smem_u32(&s_empty[sl]), parity, err, kWaitEmpty);
                if (!ok) break;
                if (elect_one()) {
                    const uint32_t bar = smem_u32(&s_full[sl]);
                    mbar_expect_tx(bar, P * (kTileH + 2) * 128);
                    if (kb < kblocks1) tma_load_4d(base + sl * kSlab, &tmA, bar, kb * kBlockK, x, y, im.s);
                    else tma_load_4d(base + sl * kSlab, &tmA2, bar, (kb - kblocks1) * kBlockK, x, y, im.s);
                }
                __syncwarp();
                sl ^= 1; parity ^= sl == 0;
            }
        }
    } else if (warp == 1) {
        // ---- MMA issuer: one thread
        if (elect_one()) {
            int st = 0, sl = 0, j = 0;
            uint32_t parity = 0, sl_parity = 0;
            uint32_t f0 = smem_u32(&full[0]), e0 = smem_u32(&empty[0]), w_step = w_bytes >> 4;
            int n_st = w_stages;
            bool pieces = false;
            const uint64_t a0 = smem_desc(base, 16, P * 128), b0 = smem_desc(w_base, 16, 1024);
            bool ready = false;                                        // what the look at stage `st` has said
            for (int wi = blockIdx.x; wi < n_items && ok; wi += gridDim.x) {
                if (skip && skip[(int64_t)((wi < n_full ? wi : n_full + (wi - n_full) / tail_split) / items_per_stream) * skip_stride]) continue;
                const uint32_t idesc = instr_desc(kTileM, wi < n_full ? Ch : Ch / tail_split, 0, 0);
                if (!pieces && tail_split > 1 && wi >= n_full) {
                    pieces = true;
                    st = 0; n_st = p_stages; parity = 0; ready = false;
                    f0 += 8 * kMaxWStages; e0 += 8 * kMaxWStages; w_step = p_bytes >> 4;
                }
                const int buf = j & 1;
                if (j >= 2) ok = mbar_wait_from(false, smem_u32(&acc_empty[buf]), ((j >> 1) - 1) & 1, err, kWaitEmpty);
                const uint32_t acc = tmem + buf * HALVES * Ch;
                for (int kb = 0; kb < kblocks && ok; ++kb) {
                    ok = mbar_wait_from(false, smem_u32(&s_full[sl]), sl_parity, err, kWaitFull);
                    const uint64_t as = a0 + sl * (kSlab >> 4);
#pragma unroll
                    for (int tap = 0; tap < 9; ++tap) {
                        if (ok) ok = mbar_wait_from(ready, f0 + 8 * st, parity, err, kWaitFull);
                        const int now = st;
                        if (++st == n_st) { st = 0; parity ^= 1; }
                        ready = mbar_try_wait(f0 + 8 * st, parity);
                        if (ok) {
                            tc_fence_after_sync();
                            const uint64_t da = as + ((tap / 3 * P + tap % 3) * 128 >> 4), db = b0 + now * w_step;
#pragma unroll
                            for (int hf = 0; hf < HALVES; ++hf)
#pragma unroll
                                for (int k = 0; k < 4; ++k)
                                    umma(acc + hf * Ch, da + hf * (kTileW * 128 >> 4) + 2 * k, db + 2 * k, idesc, (kb | tap | k) != 0);
                            umma_commit(e0 + 8 * now);
                        }
                    }
                    if (ok) umma_commit(smem_u32(&s_empty[sl]));
                    sl ^= 1; sl_parity ^= sl == 0;
                }
                if (ok) umma_commit(smem_u32(&acc_full[buf]));
                ++j;                                                   // j counts the items this block works on
            }
        }
        ok = __all_sync(0xffffffffu, ok);
    } else if (warp >= 2) {
        // ---- epilogue warps: TMEM lanes 32*(warp % 4) .. +31 = four rows of eight pixels of a tile
        const int q = warp & 3, set = (warp - 2) >> 2;
        const uint32_t piece = w_base + w_stages * w_bytes + (warp - 2) * kOutPieceBytes, orow = piece + lane * 128;
        float* part = part_of + set * 4 * 256;
        int j = -1;
        for (int wi = blockIdx.x; wi < n_items && ok; wi += gridDim.x) {
            const Item im = item_of(wi);
            const int s = im.s;
            if (skip && skip[(int64_t)s * skip_stride]) continue;
            ++j;
            const int hf = HALVES == 1 ? 0 : set, first = HALVES == 1 ? set * 64 : 0;
            constexpr int kStep = HALVES == 1 ? 128 : 64;              // this group's channels: `first`, + kStep, ... 64 at a time
            const int buf = j & 1, y = im.ty * kTileH + q * 4 + (lane >> 3);
            if (MODE == 0) {
                const float* bias = theta + (int64_t)s * n_params + b_off + im.ch0;
                for (int c = lane; c < im.chn; c += 32) part[q * 256 + c] = __ldg(bias + c);
                __syncwarp();
            }
            ok = mbar_wait(smem_u32(&acc_full[buf]), (j >> 1) & 1, err, kWaitDone);
            if (MODE == 1) {                                           // the four epilogue warps stay together: they share `part`
                int all_ok;
                asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, %2, 128, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                             : "=r"(all_ok) : "r"((int)ok), "r"(1 + set) : "memory");
                ok = all_ok != 0;
            }
            if (!ok) break;
            tc_fence_after_sync();
            {
                const int x = (im.tx + hf) * kTileW + (lane & 7);
                const bool in = y < h && x < w;
                const int64_t pixel = (int64_t)s * h * w + (int64_t)y * w + x;
                for (int n0 = first; n0 < im.chn; n0 += kStep) {
                    uint32_t words[2] = {0, 0};                        // ReLU bits
                    if (MODE == 1 && in) {
                        const uint2 b = __ldg(reinterpret_cast<const uint2*>(relu_bits + pixel * (Ch / 32) + (im.ch0 + n0) / 32));
                        words[0] = b.x; words[1] = b.y;                // ... none where the tile reaches beyond the frame
                    }
#pragma unroll
                    for (int g = 0; g < 2; ++g) {
                        float v[32];
                        tmem_ld_32x32(tmem + ((uint32_t)(q * 32) << 16) + (buf * HALVES + hf) * Ch + n0 + g * 32, v);
                        uint32_t o[16];
                        if (MODE == 0) {
                            const float4* b4 = reinterpret_cast<const float4*>(part + q * 256 + n0 + g * 32);
#pragma unroll
                            for (int k = 0; k < 16; ++k) {
                                const float4 b = b4[k >> 1];
                                const float x0f = fmaxf(v[2 * k] + ((k & 1) ? b.z : b.x), 0.f), x1f = fmaxf(v[2 * k + 1] + ((k & 1) ? b.w : b.y), 0.f);
                                const __nv_bfloat162 two = __floats2bfloat162_rn(x0f, x1f);
                                o[k] = *reinterpret_cast<const uint32_t*>(&two);
                                // the mask is taken on the stored (rounded) activation, the value the next layer sees
                                words[g] |= (__low2float(two) > 0.f ? 1u : 0u) << (2 * k);
                                words[g] |= (__high2float(two) > 0.f ? 1u : 0u) << (2 * k + 1);
                            }
                        } else {
#pragma unroll
                            for (int k = 0; k < 16; ++k) {
                                if (!((words[g] >> (2 * k)) & 1u)) v[2 * k] = 0.f;
                                if (!((words[g] >> (2 * k + 1)) & 1u)) v[2 * k + 1] = 0.f;
                                const __nv_bfloat162 two = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
                                o[k] = *reinterpret_cast<const uint32_t*>(&two);
                            }
                        }
                        if (g == 0) {
                            if (lane == 0) tma_store_wait_read<0>();   // the piece that was here before has been read
                            __syncwarp();
                        }
#pragma unroll
                        for (int k = 0; k < 4; ++k)                    // 128-byte swizzle: 16-byte chunks ^ (row % 8)
                            st_shared_128(orow + (((g * 4 + k) ^ (lane & 7)) << 4), o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
                        if (MODE == 1) {
                            // sums over the warp's 32 pixels in a fixed order: a reduce-scatter over the lanes, after which lane c
                            // holds the sum of channel c of the group
#pragma unroll
                            for (int half = 16; half >= 1; half >>= 1) {
                                const bool up = (lane & half) != 0;
#pragma unroll
                                for (int k = 0; k < half; ++k) {
                                    const float keep = up ? v[k + half] : v[k];
                                    const float send = up ? v[k] : v[k + half];
                                    v[k] = keep + __shfl_xor_sync(0xffffffffu, send, half);
                                }
                            }
                            part[q * 256 + n0 + g * 32 + lane] = v[0];
                        }
                    }
                    if (MODE == 0 && in)
                        *reinterpret_cast<uint2*>(relu_bits + pixel * (Ch / 32) + (im.ch0 + n0) / 32) = make_uint2(words[0], words[1]);
                    fence_async_shared();
                    __syncwarp();
                    if (lane == 0 && in) { tma_store_4d(&tmO, piece, im.ch0 + n0, x, y, s); tma_store_commit(); }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&acc_empty[buf])); // this warp's quarter of the accumulator is free
                if (MODE == 1) {
                    asm volatile("barrier.cta.sync %0, 128;" ::"r"(1 + set) : "memory");
                    const int e = ((warp - 2) & 3) * 32 + lane;        // 0..127 over the group's four warps
                    if (im.tx + hf < tiles_x)
                        for (int k = e; k < im.chn; k += 128)
                            if (HALVES == 2 || ((k >> 6) & 1) == set) b_partials[((int64_t)s * tiles_x * tiles_y + im.ty * tiles_x + im.tx + hf) * Ch + im.ch0 + k] =
                                (part[k] + part[256 + k]) + (part[512 + k] + part[768 + k]);
                    asm volatile("barrier.cta.sync %0, 128;" ::"r"(1 + set) : "memory");
                }
            }
        }
        if (lane == 0) tma_store_wait();
    }
    if (!ok) drain_after_error();
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, acc_cols);
}

// ------------------------------------------------------------------------------------------------
// wgrad 3x3: D[tap][ci][co] = sum over pixels q of X[q][ci] * dHd[q - tap][co].  A block takes 128 input channels, up to 128 output
// channels (COB blocks of 64), one vertical shift and a range of pixel chunks, and forms the three horizontal taps at once: the
// gradient arrives with one column more on either side, and the B operand of 192 columns is its 64 channels three times, each block
// of 64 one pixel (128 bytes) behind the one before it, which is the descriptor's stride between blocks.  Both operands are
// MN-major (pixel-major tensors, reduction over pixels).
// Where the input ends on an odd 64 channels, those stand twice in the A operand, an image row apart (five rows of pixels, the
// descriptor's stride again), and a block forms two vertical taps of theirs; the third has an operand to itself, half of which nobody
// looks at.  With such an operand for each of the three / so, us: 192 -> 128 at 720p 24.0 / 22.0, 192 -> 64 14.7 / 13.6, three of
// 101 x 187, 192 -> 128 33.7 / 32.8 (longer ranges for the same number of blocks become more and shorter ones).
// Bound by the tensor pipe (96 cycles for 192 columns; a chunk of eight takes 810 to 850 with 64 output channels a block, whose copies
// come at 60 bytes a cycle, and 1610 with 128) and by the partial sums at its end: 3 us for 14 MB at 256 channels.  A block per tap and
// all input channels, N = the output channels, before / now, us at 720p: 192 -> 64 20.3 / 15.1, 64 -> 64 14.1 / 10.3, 192 -> 128 28.4 /
// 24.9, 256 -> 128 28.3 / 25.2, 256 -> 256 47.0 / 46.5 (under the power cap; fewer partial sums for the update: 13 / 11.7); three of
// 101 x 187, 192 -> 128 38.4 / 34.6.
// ------------------------------------------------------------------------------------------------
constexpr uint32_t kWg3ABytes = kChunkW * kChunkH * 128, kWg3BCols = kChunkW + 2, kWg3BBytes = kWg3BCols * kChunkH * 128;   // 64 channels of a chunk
static_assert(kWg3ABytes % 1024 == 0 && kWg3BBytes % 1024 == 0, "the operands begin where the swizzle pattern does");
constexpr uint32_t kWg3OddBytes = kChunkW * (kChunkH + 1) * 128;
static_assert(kWg3OddBytes <= 2 * kWg3ABytes, "five rows of 64 channels lie where four of 128 do");
// blocks of one pixel range and output-channel group: three vertical taps per 128 input channels, two of an odd 64 in one
__host__ __device__ constexpr int wg3_units(int c_in) { return 3 * (c_in / kTileM) + 2 * (c_in / kBlockK % 2); }
__host__ __device__ constexpr uint32_t wg3_stage_bytes(int cob) { return 2 * kWg3ABytes + cob * kWg3BBytes; }

template <int STAGES, int COB>
__global__ void __launch_bounds__(kThreadsTc)
tc_wgrad3x3_kernel(const __grid_constant__ CUtensorMap tmA,   // previous output {C1, w, h, S} box {64, 32, 4, 1}
                   const __grid_constant__ CUtensorMap tmA2,  // skip input      {C2, w, h, S} same box (unused if C2 == 0)
                   int blocks1,                                // C1 / 64: input-channel blocks that come from tmA
                   const __grid_constant__ CUtensorMap tmO,   // where Cin ends on an odd 64: the source of those channels, box {64, 32, 5, 1}
                   int odd_c0,                                 // ... and their place in it
                   const __grid_constant__ CUtensorMap tmB,   // dHd {Ch, w, h, S} box {64, 34, 4, 1}
                   float* __restrict__ partials,              // [S][n_split][9][Ch][Cin]
                   int Cin, int Ch, int chunks_x, int n_chunks, int chunks_per_block, int n_split, unsigned int* err,
                   const int* __restrict__ skip, int64_t skip_stride, int a_early)
{
    // Cin = C1 + C2: the layer's input is the concatenation (previous output, skip input), read from its two sources
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_smem(smem_raw);
    const uint32_t base = smem_u32(smem);
    constexpr uint32_t kStage = wg3_stage_bytes(COB), kCols = COB == 1 ? 256 : 512;
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], done;
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    // the blocks of one pixel range are neighbours: what they share comes from L2
    const int per_group = wg3_units(Cin), units = per_group * (Ch / kBlockK / COB);
    const int unit = blockIdx.x % units, split = blockIdx.x / units, s = blockIdx.y;
    const int cg = unit / per_group, u = unit % per_group, m = min(u / 3, Cin / kTileM);
    const int a_blocks = min(2, Cin / kBlockK - 2 * m);
    const bool paired = a_blocks == 1 && u == 3 * m;            // vertical taps 0 and 1 of the odd 64 channels
    const int ky = a_blocks == 1 ? 2 * (u - 3 * m) : u - 3 * m;
    // a chunk's first rows: of the gradient y0 + 1 - ky, or y0 where two taps share it and the input begins a row above
    const int dy_b = paired ? 0 : 1 - ky;
    const int c_begin = min(n_chunks, split * chunks_per_block), c_end = min(n_chunks, c_begin + chunks_per_block);

    if (warp == 0) {
        if (elect_one()) { prefetch_map(&tmA); prefetch_map(&tmB); }
        __syncwarp();
        tmem_alloc(smem_u32(&tmem_slot), kCols);
    }
    if (tid == 0) {
        for (int i = 0; i < STAGES; ++i) { mbar_init(smem_u32(&full[i]), 1); mbar_init(smem_u32(&empty[i]), 1); }
        mbar_init(smem_u32(&done), 1);
        fence_barrier_init();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_slot;
    bool ok = true;
    // The third vertical tap of an odd 64 channels: the operand's upper half is what lies in the stage; nobody looks at those rows.
    auto load_a = [&](int i, int st) {                        // (one thread)
        const int x0 = i % chunks_x * kChunkW, y0 = i / chunks_x * kChunkH;
        const uint32_t bar = smem_u32(&full[st]), sa = base + st * kStage;
        mbar_expect_tx(bar, (paired ? kWg3OddBytes : a_blocks * kWg3ABytes) + COB * kWg3BBytes);
        if (paired) { tma_load_4d(sa, &tmO, bar, odd_c0, x0, y0 - 1, s); return; }
        for (int j = 0; j < a_blocks; ++j) {
            const int cb = 2 * m + j;
            if (cb < blocks1) tma_load_4d(sa + j * kWg3ABytes, &tmA, bar, cb * kBlockK, x0, y0, s);
            else tma_load_4d(sa + j * kWg3ABytes, &tmA2, bar, (cb - blocks1) * kBlockK, x0, y0, s);
        }
    };
    // a_early: the layer's input is frozen, so no kernel of the step writes it: the first stages' part of it is fetched before the
    // wait for the kernel that produces the gradient
    const int n_pre = a_early ? min(STAGES, c_end - c_begin) : 0;
    if (warp == 0 && elect_one())
        for (int it = 0; it < n_pre; ++it) load_a(c_begin + it, it);
    pdl_wait();                  // inputs come from the previous kernel of the step
    if (skip && skip[(int64_t)blockIdx.y * skip_stride]) {     // this stream's training loop has ended (block-uniform; the flag
        tc_fence_before_sync();                                 // comes from an earlier kernel, so it is read after the wait)
        __syncthreads();
        if (warp == 0) tmem_dealloc(tmem, kCols);
        return;
    }

    if (warp == 0) {             // the producer walks its loop as a whole warp, one lane issues
        int st = 0;
        uint32_t parity = 1;
        for (int i = c_begin; i < c_end && ok; ++i) {
            if (i - c_begin >= STAGES) ok = mbar_wait(smem_u32(&empty[st]), parity, err, kWaitEmpty);
            if (!ok) break;
            if (elect_one()) {
                if (i - c_begin >= n_pre) load_a(i, st);
                const int x0 = i % chunks_x * kChunkW, y0 = i / chunks_x * kChunkH;
                for (int j = 0; j < COB; ++j)
                    tma_load_4d(base + st * kStage + 2 * kWg3ABytes + j * kWg3BBytes, &tmB, smem_u32(&full[st]), (cg * COB + j) * kBlockK, x0 - 1, y0 + dy_b, s);
            }
            __syncwarp();
            if (++st == STAGES) { st = 0; parity ^= 1; }
        }
    } else if (warp == 1) {      // one thread issues
        if (elect_one()) {
            constexpr uint32_t idesc = instr_desc(kTileM, 3 * kBlockK, 1, 1);
            const uint64_t a0 = smem_desc(base, paired ? kChunkW * 128 : kWg3ABytes, 1024), b0 = smem_desc(base + 2 * kWg3ABytes, 128, 1024);
            const uint32_t f0 = smem_u32(&full[0]);
            int st = 0;
            uint32_t parity = 0;
            bool ready = false;
            for (int i = c_begin; i < c_end && ok; ++i) {
                ok = mbar_wait_from(ready, f0 + 8 * st, parity, err, kWaitFull);
                if (!ok) break;
                const int now = st;
                if (++st == STAGES) { st = 0; parity ^= 1; }
                ready = mbar_try_wait(f0 + 8 * st, parity);
                tc_fence_after_sync();
                const uint64_t da = a0 + now * (kStage >> 4), db = b0 + now * (kStage >> 4);
#pragma unroll
                for (int j = 0; j < kChunkW * kChunkH / 16; ++j)     // 16 pixels at a time, two to a row of the chunk
#pragma unroll
                    for (int c = 0; c < COB; ++c)
                        umma(tmem + c * (3 * kBlockK), da + (j * (16 * 128) >> 4), db + ((c * kWg3BBytes + (j / 2 * kWg3BCols + j % 2 * 16) * 128) >> 4), idesc,
                             i != c_begin || j != 0);
                umma_commit(smem_u32(&empty[now]));
            }
            umma_commit(smem_u32(&done));
        }
        ok = __all_sync(0xffffffffu, ok);
    }
    __syncwarp();
    if (!mbar_wait(smem_u32(&done), 0, err, kWaitDone)) ok = false;
    pdl_launch_dependents();     // only the epilogue is left
    tc_fence_after_sync();
    ok = __syncthreads_and(ok);
    if (ok) {
        const int ci = m * kTileM + (paired ? tid % kBlockK : tid), tap = ky + (paired ? tid / kBlockK : 0);
        float* dst = partials + (((int64_t)s * n_split + split) * 9 + tap * 3) * Ch * Cin + (int64_t)cg * COB * kBlockK * Cin + ci;
        const bool any = c_end > c_begin;
        for (int c = 0; c < COB; ++c)
            for (int n0 = 0; n0 < 3 * kBlockK; n0 += 32) {
                float v[32];
                tmem_ld_32x32(tmem + ((uint32_t)(warp * 32) << 16) + c * (3 * kBlockK) + n0, v);
                // the gradient's column x - 1 + k stands under input column x in block k of 64: horizontal tap 2 - k
                float* row = dst + ((int64_t)(2 - n0 / kBlockK) * Ch + c * kBlockK + n0 % kBlockK) * Cin;
                if (ci < Cin)
#pragma unroll
                    for (int k = 0; k < 32; ++k) row[(int64_t)k * Cin] = any ? v[k] : 0.f;
            }
    } else {
        drain_after_error();
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kCols);
}

// ------------------------------------------------------------------------------------------------
// Both backward products of the 1x1 output layer behind a trained hidden layer, in one pass over the logit gradient and the
// hidden activation:
//   dHd[pix][k] = [Hd[pix][k] > 0] * sum_c dz[c][pix] * W2[c][k]        (bf16, and its unrounded sums over pixels: the bias
//                                                                         gradient of the 3x3 layer)
//   dW2[c][k]  += dz[c][pix] * Hd[pix][k]
// A block owns 128 hidden channels (an odd 64 at the end of the layer arrives zero-filled) and a range of 128-pixel tiles.  dz
// rows [c][pix] are the MN-major A operand of the first product and the K-major B operand of the second, from one copy;
// weight rows [c][k] and activation rows [pix][k] are MN-major.  A ring of stages (producer warp), one warp that issues both
// products, two sets of four warps that drain the two accumulators of the first in turn; the second accumulates over the
// whole range, which leaves one partial sum per block, like the bias gradient.
// Bound by L2: at 720p and 256 channels 29 MB of activations come in and as much gradient goes out, 12.9 us (5 TB/s); 16.8 us
// with 32-byte stores straight from the accumulator rows, which go out through shared memory and TMA instead.  As two kernels
// (gradient: a block per 128 pixels and half of the channels; weight gradient: a pass of its own) 18.8 + 9.7 us; at 1080p
// 33.3 + 15.1 us, now 28.1.  Bias sums kept in registers over the tiles cost the narrow layers 2 us and gained nothing.
// ------------------------------------------------------------------------------------------------
constexpr int kBackStages = 3, kBackThreads = 320, kBackCols = 128;
constexpr uint32_t kBackActBytes = kTileM * 128 * 2, kBackDzBytes = 2 * kClassPad * 128, kBackStageBytes = kBackActBytes + kBackDzBytes, kBackWBytes = 2 * kClassPad * 128,
                   kBackOutBytes = 8 * 32 * kBackCols * 2;   // a 32 x 128 piece of the gradient for each epilogue warp

__global__ void __launch_bounds__(kBackThreads, 1)
tc_back1x1_kernel(const __grid_constant__ CUtensorMap tmH,   // Hd {Ch, p, S}  box {64, 128, 1}
                  const __grid_constant__ CUtensorMap tmD,   // dz {p, 32, S}  box {64, 32, 1}
                  const __grid_constant__ CUtensorMap tmW,   // W2 {Ch, 32, S} box {64, 32, 1}
                  const __grid_constant__ CUtensorMap tmO,   // dHd {Ch, p, S} box {64, 32, 1}
                  const uint32_t* __restrict__ relu_bits,     // [S][p][Ch/32]
                  float* __restrict__ b_partials,             // [S][n_split][Ch]
                  float* __restrict__ w_partials,             // [S][n_split][32][Ch]
                  int Ch, int p, int n_tiles, int per, int n_groups, unsigned int* err, const int* __restrict__ skip, int64_t skip_stride,
                  int has_ctl, const TrainCtl ctl)
{
    const int s = blockIdx.y;
    if (has_ctl && blockIdx.x == gridDim.x - 1) {            // Train: one more block assesses the prediction meanwhile
        const TrainHistory hist = train_history(ctl, s);
        pdl_wait();
        bool stop, better;
        train_decision(ctl, s, true, hist, nullptr, stop, better);
        pdl_launch_dependents();
        return;
    }
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_smem(smem_raw);
    const uint32_t base = smem_u32(smem), w_base = base + kBackStages * kBackStageBytes;
    __shared__ __align__(8) uint64_t full[kBackStages], empty[kBackStages], w_full, acc_full[2], acc_empty[2], done;
    __shared__ uint32_t tmem_slot;
    __shared__ float part[8 * kBackCols];                        // per-warp channel sums
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int n_split = ((int)gridDim.x - (has_ctl ? 1 : 0)) / n_groups, split = (int)blockIdx.x / n_groups, ch0 = (int)blockIdx.x % n_groups * kBackCols;
    const int t_begin = split * per, t_end = min(n_tiles, t_begin + per), width = min(kBackCols, Ch - ch0);

    if (warp == 0) tmem_alloc(smem_u32(&tmem_slot), 512);
    if (tid == 0) {
        for (int i = 0; i < kBackStages; ++i) { mbar_init(smem_u32(&full[i]), 1); mbar_init(smem_u32(&empty[i]), 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&acc_full[i]), 1); mbar_init(smem_u32(&acc_empty[i]), 4); }
        mbar_init(smem_u32(&w_full), 1); mbar_init(smem_u32(&done), 1);
        fence_barrier_init();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = tmem_slot, acc_w = tmem + 2 * kBackCols;       // two accumulators of the first product, then the second's
    pdl_wait();                  // inputs come from the previous kernel of the step
    if (skip && skip[(int64_t)s * skip_stride]) {            // this stream's training loop has ended (block-uniform)
        tc_fence_before_sync();
        __syncthreads();
        if (warp == 0) tmem_dealloc(tmem, 512);
        return;
    }
    bool ok = true;
    if (warp == 0) {
        // ---- producer (the whole warp walks the loop, its first lane issues)
        if (elect_one()) {
            mbar_expect_tx(smem_u32(&w_full), kBackWBytes);
            tma_load_3d(w_base, &tmW, smem_u32(&w_full), ch0, 0, s);
            tma_load_3d(w_base + kClassPad * 128, &tmW, smem_u32(&w_full), ch0 + kBlockK, 0, s);
        }
        for (int i = t_begin; i < t_end; ++i) {
            const int it = i - t_begin, st = it % kBackStages;
            if (it >= kBackStages) ok = mbar_wait(smem_u32(&empty[st]), ((it / kBackStages) - 1) & 1, err, kWaitEmpty);
            if (!ok) break;
            if (elect_one()) {
                const uint32_t bar = smem_u32(&full[st]), sa = base + st * kBackStageBytes;
                mbar_expect_tx(bar, kBackStageBytes);
                tma_load_3d(sa + kBackActBytes, &tmD, bar, i * kTileM, 0, s);
                tma_load_3d(sa + kBackActBytes + kClassPad * 128, &tmD, bar, i * kTileM + 64, 0, s);
                tma_load_3d(sa, &tmH, bar, ch0, i * kTileM, s);
                tma_load_3d(sa + kTileM * 128, &tmH, bar, ch0 + kBlockK, i * kTileM, s);
            }
            __syncwarp();
        }
    } else if (warp == 1) {
        // ---- both products
        ok = mbar_wait(smem_u32(&w_full), 0, err, kWaitFull);
        const uint64_t w_mn = smem_desc(w_base, kClassPad * 128, 1024);
        const uint32_t id1 = instr_desc(kTileM, width, 1, 1);
        constexpr uint32_t id2 = instr_desc(kTileM, kClassPad, 1, 0);
        for (int i = t_begin; i < t_end && ok; ++i) {
            const int it = i - t_begin, st = it % kBackStages, buf = it & 1;
            ok = mbar_wait(smem_u32(&full[st]), (it / kBackStages) & 1, err, kWaitFull);
            if (ok && it >= 2) ok = mbar_wait(smem_u32(&acc_empty[buf]), ((it >> 1) - 1) & 1, err, kWaitEmpty);
            if (!ok) break;
            tc_fence_after_sync();
            if (elect_one()) {
                const uint32_t sa = base + st * kBackStageBytes, sd = sa + kBackActBytes;
                const uint64_t dz_mn = smem_desc(sd, kClassPad * 128, 1024), dz_k = smem_desc(sd, 16, 1024), h_mn = smem_desc(sa, kTileM * 128, 1024);
#pragma unroll
                for (int j = 0; j < kClassPad / 16; ++j)
                    umma(tmem + buf * kBackCols, dz_mn + j * ((16 * 128) >> 4), w_mn + j * ((16 * 128) >> 4), id1, j != 0);
                umma_commit(smem_u32(&acc_full[buf]));
#pragma unroll
                for (int j = 0; j < kTileM / 16; ++j)
                    umma(acc_w, h_mn + j * ((16 * 128) >> 4), dz_k + (j >> 2) * ((kClassPad * 128) >> 4) + (j & 3) * 2, id2, (it | j) != 0);
                umma_commit(smem_u32(&empty[st]));
            }
            __syncwarp();
        }
        if (elect_one()) umma_commit(smem_u32(&done));
    } else {
        // ---- epilogue: set e takes every other tile; TMEM lanes 32*(warp % 4) .. +31 = pixels
        const int e = (warp - 2) >> 2, q = warp & 3, groups = width / 32;
        const uint32_t out_base = w_base + kBackWBytes + (warp - 2) * (32 * kBackCols * 2);
        float sums[4] = {0.f, 0.f, 0.f, 0.f};                // lane c: sum over the warp's pixels so far of channel ch0 + 32 g + c
        for (int i = t_begin + e; i < t_end && ok; i += 2) {
            const int pix = i * kTileM + q * 32 + lane;
            const bool in = pix < p;
            uint32_t bits[4] = {0, 0, 0, 0};                 // ReLU mask of this thread's pixel, fetched while the products run
            if (in) {
                const uint32_t* mp = relu_bits + ((int64_t)s * p + pix) * (Ch / 32) + ch0 / 32;
#pragma unroll
                for (int g = 0; g < 4; ++g) if (g < groups) bits[g] = __ldg(mp + g);
            }
            ok = mbar_wait(smem_u32(&acc_full[e]), ((i - t_begin) >> 1) & 1, err, kWaitDone);
            if (!ok) break;
            tc_fence_after_sync();
            if (lane == 0) tma_store_wait_read<0>();         // this warp's piece of the tile before last has been read
            __syncwarp();
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                if (g >= groups) break;
                float v[32];
                tmem_ld_32x32(tmem + ((uint32_t)(q * 32) << 16) + e * kBackCols + g * 32, v);
                uint32_t o[16];
#pragma unroll
                for (int k = 0; k < 16; ++k) {               // the mask of a pixel outside the frame is empty
                    if (!((bits[g] >> (2 * k)) & 1u)) v[2 * k] = 0.f;
                    if (!((bits[g] >> (2 * k + 1)) & 1u)) v[2 * k + 1] = 0.f;
                    const __nv_bfloat162 two = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
                    o[k] = *reinterpret_cast<const uint32_t*>(&two);
                }
                const uint32_t orow = out_base + (g >> 1) * 4096 + lane * 128;      // 128-byte swizzle: 16-byte chunks ^ (row % 8)
#pragma unroll
                for (int k = 0; k < 4; ++k) st_shared_128(orow + ((((g & 1) * 4 + k) ^ (lane & 7)) << 4), o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
                if (g & 1) {                                  // widths are multiples of 64
                    fence_async_shared();
                    __syncwarp();
                    if (lane == 0 && pix < p) { tma_store_3d(&tmO, out_base + (g >> 1) * 4096, ch0 + (g >> 1) * 64, pix, s); tma_store_commit(); }
                }
                // sums over the warp's 32 pixels, fixed order: a reduce-scatter over the lanes (lanes whose bit is set keep the
                // upper half of the channels), after which lane c holds the sum of channel c of the group
#pragma unroll
                for (int half = 16; half >= 1; half >>= 1) {
                    const bool up = (lane & half) != 0;
#pragma unroll
                    for (int k = 0; k < half; ++k) {
                        const float keep = up ? v[k + half] : v[k];
                        const float send = up ? v[k] : v[k + half];
                        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, half);
                    }
                }
                sums[g] += v[0];
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&acc_empty[e]));
        }
        if (lane == 0) tma_store_wait();
#pragma unroll
        for (int g = 0; g < 4; ++g) part[(warp - 2) * kBackCols + g * 32 + lane] = sums[g];
    }
    __syncwarp();
    if (!mbar_wait(smem_u32(&done), 0, err, kWaitDone)) ok = false;
    pdl_launch_dependents();     // only the partial sums are left
    tc_fence_after_sync();
    ok = __syncthreads_and(ok);
    if (ok) {
        const int64_t row = (int64_t)s * n_split + split;
        if (warp >= 6) {                                     // the second product: lanes = channels, columns = classes
            const int k = (warp & 3) * 32 + lane;
            float v[32];
            tmem_ld_32x32(acc_w + ((uint32_t)((warp & 3) * 32) << 16), v);
            float* dst = w_partials + row * kClassPad * Ch + ch0 + k;
            if (k < width)
#pragma unroll
                for (int c = 0; c < kClassPad; ++c) dst[(int64_t)c * Ch] = v[c];
        } else if (tid < width) {
            float t = 0.f;
#pragma unroll
            for (int x = 0; x < 8; ++x) t += part[x * kBackCols + tid];
            b_partials[row * Ch + ch0 + tid] = t;
        }
    } else {
        drain_after_error();
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ---- host side -------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (fn) return fn;
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) != cudaSuccess || !ptr) return nullptr;
    fn = (EncodeTiledFn)ptr;
    return fn;
}

// bf16 tensor, innermost dimension first; strides (bytes) for dimensions 1..rank-1; 128-byte swizzle.
bool make_map(CUtensorMap* m, const void* base, int rank, const uint64_t* dims, const uint64_t* strides,
              const uint32_t* box, char* err, size_t err_len, const char* what)
{
    return encode_tensor_map(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, CU_TENSOR_MAP_SWIZZLE_128B, base, rank, dims, strides, box,
                             err, err_len, what);
}

int pow2_cols(int n) { int c = 32; while (c < n) c <<= 1; return c; }

void split_geometry(int n_chunks, int target_blocks, int* per, int* n_split)
{
    int pb = (n_chunks + target_blocks - 1) / target_blocks;
    if (pb < 1) pb = 1;
    *per = pb;
    *n_split = (n_chunks + pb - 1) / pb;
    if (*n_split < 1) *n_split = 1;
}

}  // namespace

bool encode_tensor_map(CUtensorMap* m, CUtensorMapDataType dtype, CUtensorMapSwizzle swizzle, const void* base, int rank,
                       const uint64_t* dims, const uint64_t* strides, const uint32_t* box, char* err, size_t err_len,
                       const char* what)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) { snprintf(err, err_len, "cuTensorMapEncodeTiled is not available"); return false; }
    cuuint64_t d[5], st[4];
    cuuint32_t b[5], es[5];
    for (int i = 0; i < rank; ++i) { d[i] = dims[i]; b[i] = box[i]; es[i] = 1; }
    for (int i = 0; i + 1 < rank; ++i) st[i] = strides[i];
    CUresult r = fn(m, dtype, (cuuint32_t)rank, const_cast<void*>(base), d, st, b, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) { snprintf(err, err_len, "tensor map for %s rejected (CUresult %d)", what, (int)r); return false; }
    return true;
}

// Weight stages of the 3x3 tile walk: what fits beside two slabs and the epilogue's pieces
static int fwd3_stages(int n_out, int halves)
{
    const int n = (int)((218 * 1024 - 2 * (int)slab_bytes(halves) - 8 * (int)kOutPieceBytes - kSmemAlign) / (n_out * 128));
    return n < kMaxWStages ? n : kMaxWStages;
}
static size_t fwd3_bytes(int n_out, int halves)
{
    return 2 * (size_t)slab_bytes(halves) + (size_t)fwd3_stages(n_out, halves) * n_out * 128 + 8 * kOutPieceBytes + kSmemAlign;
}
// How a launch walks the map: tiles per item, items, blocks, and into how many ranges of output channels (multiples of 64) the
// items of a partly filled last round are cut, where that lets every piece have its own block.
struct Fwd3Walk { int halves, n_full, n_items, tail_split, grid; };
static Fwd3Walk fwd3_walk(int h, int w, int S, int n_out, int n_sms)
{
    const int tiles_x = (w + kTileW - 1) / kTileW, tiles_y = (h + kTileH - 1) / kTileH;
    // Two tiles to an item share the weight stages.  What an item of 64 input channels costs, in cycles: its shared-memory bytes at
    // 128 a cycle (36 MMAs per tile read 4 KB of pixels and 32 bytes per output channel each; slab and weights are written
    // once), or its multiplications at N / 2 cycles an MMA.  The accumulators of two tiles fit twice up to 128 channels.
    auto cost = [&](int halves) {
        const int64_t items = (int64_t)((tiles_x + halves - 1) / halves) * tiles_y * S, rounds = (items + n_sms - 1) / n_sms;
        const int64_t bytes = (int64_t)halves * 36 * (4096 + n_out * 32) + slab_bytes(halves) + 9 * n_out * 128, math = (int64_t)halves * 36 * n_out / 2;
        return rounds * (bytes / 128 > math ? bytes / 128 : math);
    };
    Fwd3Walk q;
    q.halves = n_out <= 128 && cost(2) < cost(1) ? 2 : 1;
    const int items = (tiles_x + q.halves - 1) / q.halves * tiles_y * S;
    q.grid = items < n_sms ? items : n_sms;
    q.tail_split = 1;
    const int tail = items % q.grid;
    if (tail > 0) {
        if (n_out % 256 == 0 && tail * 4 <= q.grid) q.tail_split = 4;
        else if (n_out % 128 == 0 && tail * 2 <= q.grid) q.tail_split = 2;
    } else if (items < n_sms) {                          // a small map: every item is cut
        if (n_out % 256 == 0 && items * 4 <= n_sms) q.tail_split = 4;
        else if (n_out % 128 == 0 && items * 2 <= n_sms) q.tail_split = 2;
        q.grid = items * q.tail_split;
    }
    q.n_full = q.tail_split > 1 ? items / q.grid * q.grid : items;
    q.n_items = q.n_full + (items - q.n_full) * q.tail_split;
    return q;
}
template <int MODE>
static decltype(&tc_fwd3x3_kernel<1, MODE>) fwd3_kernel(const Fwd3Walk& q) { return q.halves == 2 ? tc_fwd3x3_kernel<2, MODE> : tc_fwd3x3_kernel<1, MODE>; }
// The 3x3 weight gradient: output-channel blocks of 64 per block, its launch's units (input-channel tiles x output-channel groups x
// vertical shifts), pixel chunks and ranges.  About one block per SM for one stream, no range shorter than five chunks (a block's
// start and its partial sums cost as much; us of a call, four streams of 60 x 100, 128 channels: 693 with ranges of two
// or three, 590 with five; 45 x 80, 282 and 276; one stream of 90 x 160, 320 and 324).  The number of streams has no part in it.
// Blocks of 128 output channels fetch a third less per multiplication and leave twice the partial sums: they pay where ranges are
// long (us of a call, 64 / 128: 256 channels, 85 chunks of a 1080p map a block 4301 / 4246; 38 chunks at 720p 1176 / 1191; 90 x 160
// 538 / 562; three of 101 x 187, 128 channels 540 / 593).
struct Wg3Shape { int cob, units, chunks_x, chunks, per, n_split; };
static Wg3Shape wg3_shape(int c_in, int c_out, int h, int w)
{
    Wg3Shape q;
    q.chunks_x = (w + kChunkW - 1) / kChunkW;
    q.chunks = q.chunks_x * ((h + kChunkH - 1) / kChunkH);
    for (q.cob = c_out % 128 == 0 ? 2 : 1;; q.cob = 1) {
        q.units = wg3_units(c_in) * (c_out / kBlockK / q.cob);
        const int ranges = std::min(148 / q.units, q.chunks / kWg3LeastChunks);
        split_geometry(q.chunks, std::max(ranges, 1), &q.per, &q.n_split);
        if (q.cob == 1 || q.per >= 64) return q;
    }
}
static size_t wg3_bytes(const Wg3Shape& q) { return (size_t)(q.cob == 2 ? 3 : 4) * wg3_stage_bytes(q.cob) + kSmemAlign; }
static decltype(&tc_wgrad3x3_kernel<3, 2>) wgrad3_kernel(const Wg3Shape& q) { return q.cob == 2 ? tc_wgrad3x3_kernel<3, 2> : tc_wgrad3x3_kernel<4, 1>; }

struct TcBlockPlan {
    CUtensorMap in_fwd, skip_fwd;    // the block's two inputs {C, w, h, S}, box {64, 8 halves + 2, 18, 1} (forward slabs)
    CUtensorMap in_wg, skip_wg;      // same tensors, box {64, 32, 4, 1} (weight-gradient chunks)
    CUtensorMap odd_wg;              // the one that the last 64 of an odd number of channel blocks come from, box {64, 32, 5, 1}
    CUtensorMap w_map, w_map_q;      // {c_tot, 9*c_out, S}, boxes {64, c_out, 1} and {64, 64, 1}
    CUtensorMap wt_map, wt_map_q;    // mirrored, transposed weights {c_out, 9*c_prev, S}, boxes {64, c_prev, 1} and {64, 64, 1}
    CUtensorMap dout_fwd;            // the block's output gradient {c_out, w, h, S}, the slab's box (A operand when passed back)
    CUtensorMap out_st, dprev_st;    // the block's output and its first input's gradient {C, w, h, S}, box {64, 8, 4, 1} (stores)
    CUtensorMap dout_wg;             // same tensor, box {64, 34, 4, 1} (B operand of the weight gradient)
    Wg3Shape wg;
    Fwd3Walk walk_fwd, walk_back;
    size_t smem_fwd, smem_back;
};

struct TcPlan {
    TcBuffers b;
    int p, p_pad, c_last;
    CUtensorMap act_fwd;     // last-layer input {c_last, p, S} box {64, 128, 1}
    CUtensorMap act_wg;      // same tensor, box {64, 64, 1}
    CUtensorMap w2_map;      // {c_last, 32, S} box {64, 32, 1}
    CUtensorMap dz_map;      // {p, 32, S} box {64, 32, 1}
    CUtensorMap dout_map;    // gradient of the last-layer input, where it is formed: {c_last, p, S} box {64, 32, 1}
    TcBlockPlan blk[kMaxBlocks];
    int split2, chunks2, per2, cols2, msplit2;
    int tiles_b, per_b, split_b, groups_b;   // backward of the 1x1 layer behind a trained block: pixel tiles, tiles per range, ranges, channel groups
    size_t smem_fwd1, smem_fwd1p, smem_wg1, smem_back1;
    bool fwd1_persistent, wg1_deep;
    int n_sms;
    bool test_stall;         // test of the give-up path (environment ST_TEST_STALL_FWD1X1=1 when the plan is made)
};

// blocks per pixel range of the 1x1 weight gradient: one per 128-channel accumulator
static int wgrad1x1_m_split(int c_last) { const int m = (c_last + kTileM - 1) / kTileM; return m < 1 ? 1 : m; }

int tc_wgrad1x1_splits(int c_last, int h, int w)
{
    int per, n;
    const int64_t p = (int64_t)h * w;
    split_geometry((int)((p + kChunkPix - 1) / kChunkPix), 148 / wgrad1x1_m_split(c_last), &per, &n);
    return n;
}
int tc_wgrad3x3_splits(int c_in, int c_out, int h, int w) { return wg3_shape(c_in, c_out, h, w).n_split; }

// pixel ranges of the 1x1 layer's backward behind a trained hidden layer: with the groups of 128 channels about one block per SM
int tc_back_splits(int c_last, int h, int w)
{
    int per, n;
    split_geometry((int)(((int64_t)h * w + kTileM - 1) / kTileM), 148 / ((c_last + kBackCols - 1) / kBackCols), &per, &n);
    return n;
}

int tc_tile3_count(int h, int w) { return ((w + kTileW - 1) / kTileW) * ((h + kTileH - 1) / kTileH); }

int tc_dz_pitch(int h, int w) { return (int)((((int64_t)h * w + 63) / 64) * 64); }

TcPlan* tc_plan_create(const TcBuffers& b, char* err, size_t err_len)
{
    TcPlan* P = new TcPlan();
    memset((void*)P, 0, sizeof *P);
    P->b = b;
    P->p = b.h * b.w; P->p_pad = tc_dz_pitch(b.h, b.w);
    {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&P->n_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || P->n_sms < 1) P->n_sms = 148;
    }
    const int nb = b.n_blocks;
    P->c_last = nb ? b.blk[nb - 1].c_out : b.c_in;
    const uint64_t S = (uint64_t)b.S, p = (uint64_t)P->p, cl = (uint64_t)P->c_last;
    const bf16* act = nb ? b.blk[nb - 1].out : b.x;
    bool ok = true;
    {
        uint64_t dims[3] = {cl, p, S}, str[2] = {cl * 2, p * cl * 2};
        uint32_t box_f[3] = {64, 128, 1}, box_w[3] = {64, 64, 1};
        ok = ok && make_map(&P->act_fwd, act, 3, dims, str, box_f, err, err_len, "last-layer input (forward)");
        ok = ok && make_map(&P->act_wg, act, 3, dims, str, box_w, err, err_len, "last-layer input (wgrad)");
        uint32_t box_o[3] = {64, 32, 1};
        if (nb && b.blk[nb - 1].trained)
            ok = ok && make_map(&P->dout_map, b.blk[nb - 1].dout, 3, dims, str, box_o, err, err_len, "last-layer input gradient");
    }
    if (ok) {
        uint64_t dims[3] = {cl, (uint64_t)kClassPad, S}, str[2] = {cl * 2, (uint64_t)kClassPad * cl * 2};
        uint32_t box[3] = {64, (uint32_t)kClassPad, 1};
        ok = make_map(&P->w2_map, b.w2, 3, dims, str, box, err, err_len, "1x1 weight");
    }
    if (ok) {
        uint64_t dims[3] = {p, (uint64_t)kClassPad, S}, str[2] = {(uint64_t)P->p_pad * 2, (uint64_t)kClassPad * P->p_pad * 2};
        uint32_t box[3] = {64, (uint32_t)kClassPad, 1};
        ok = make_map(&P->dz_map, b.dz_bf16, 3, dims, str, box, err, err_len, "logit gradient");
    }
    const size_t lim = 227 * 1024;
    for (int i = 0; ok && i < nb; ++i) {
        const TcBlock& k = b.blk[i];
        TcBlockPlan& q = P->blk[i];
        const uint64_t w = (uint64_t)b.w, h = (uint64_t)b.h, c1 = (uint64_t)k.c_prev, c2 = (uint64_t)k.c_skip, co = (uint64_t)k.c_out,
                       ct = c1 + c2;
        q.walk_fwd = fwd3_walk(b.h, b.w, b.S, k.c_out, P->n_sms);
        q.walk_back = fwd3_walk(b.h, b.w, b.S, k.c_prev, P->n_sms);
        auto act_maps = [&](const bf16* base, uint64_t c, int halves, CUtensorMap* fwd, CUtensorMap* wg, int wg_cols, const char* what) {
            const uint32_t bf[4] = {64, (uint32_t)slab_cols(halves), (uint32_t)kTileH + 2, 1}, bw[4] = {64, (uint32_t)wg_cols, (uint32_t)kChunkH, 1};
            uint64_t d[4] = {c, w, h, S}, st[3] = {c * 2, w * c * 2, h * w * c * 2};
            return make_map(fwd, base, 4, d, st, bf, err, err_len, what) && make_map(wg, base, 4, d, st, bw, err, err_len, what);
        };
        ok = ok && act_maps(k.in_prev, c1, q.walk_fwd.halves, &q.in_fwd, &q.in_wg, kChunkW, "block input");
        if (c2) ok = ok && act_maps(k.in_skip, c2, q.walk_fwd.halves, &q.skip_fwd, &q.skip_wg, kChunkW, "skip input");
        else { q.skip_fwd = q.in_fwd; q.skip_wg = q.in_wg; }
        {
            const uint64_t c = c2 ? c2 : c1, d[4] = {c, w, h, S}, st[3] = {c * 2, w * c * 2, h * w * c * 2};
            const uint32_t bo[4] = {64, (uint32_t)kChunkW, (uint32_t)kChunkH + 1, 1};
            ok = ok && make_map(&q.odd_wg, c2 ? k.in_skip : k.in_prev, 4, d, st, bo, err, err_len, "block input (odd 64 channels)");
        }
        ok = ok && act_maps(k.dout, co, q.walk_back.halves, &q.dout_fwd, &q.dout_wg, kWg3BCols, "block output gradient");
        {
            uint64_t dw[3] = {ct, 9 * co, S}, sw[2] = {ct * 2, 9 * co * ct * 2};
            uint32_t bwt[3] = {64, (uint32_t)co, 1}, bwq[3] = {64, 64, 1};
            ok = ok && make_map(&q.w_map, k.w, 3, dw, sw, bwt, err, err_len, "3x3 weight");
            ok = ok && make_map(&q.w_map_q, k.w, 3, dw, sw, bwq, err, err_len, "3x3 weight (64 rows)");
        }
        auto store_map = [&](const bf16* base, uint64_t c, CUtensorMap* m, const char* what) {
            uint64_t d[4] = {c, w, h, S}, st[3] = {c * 2, w * c * 2, h * w * c * 2};
            uint32_t bo[4] = {64, (uint32_t)kTileW, 4, 1};
            return make_map(m, base, 4, d, st, bo, err, err_len, what);
        };
        ok = ok && store_map(k.out, co, &q.out_st, "block output (stores)");
        if (ok && k.pass_back) {
            ok = store_map(b.blk[i - 1].dout, c1, &q.dprev_st, "previous block's output gradient (stores)");
            uint64_t dw[3] = {co, 9 * c1, S}, sw[2] = {co * 2, 9 * c1 * co * 2};
            uint32_t bwt[3] = {64, (uint32_t)c1, 1}, bwq[3] = {64, 64, 1};
            ok = ok && make_map(&q.wt_map, k.w_t, 3, dw, sw, bwt, err, err_len, "3x3 weight, transposed");
            ok = ok && make_map(&q.wt_map_q, k.w_t, 3, dw, sw, bwq, err, err_len, "3x3 weight, transposed (64 rows)");
        }
        q.wg = wg3_shape((int)ct, k.c_out, b.h, b.w);
        q.smem_fwd = fwd3_bytes(k.c_out, q.walk_fwd.halves);
        q.smem_back = fwd3_bytes(k.c_prev, q.walk_back.halves);
        if (ok && (q.smem_fwd > lim || wg3_bytes(q.wg) > lim || (k.pass_back && (q.smem_back > lim || k.c_prev > 256)))) {
            snprintf(err, err_len, "shared memory per block exceeds 227 KB for these channel counts");
            ok = false;
        }
    }
    if (!ok) { delete P; return nullptr; }

    const int m_last = (P->c_last + kTileM - 1) / kTileM;
    P->chunks2 = (P->p + kChunkPix - 1) / kChunkPix;
    P->msplit2 = wgrad1x1_m_split(P->c_last);
    split_geometry(P->chunks2, 148 / P->msplit2, &P->per2, &P->split2);
    P->cols2 = pow2_cols((m_last / P->msplit2) * kClassPad);
    P->smem_fwd1 = (size_t)(P->c_last / kBlockK) * (kTileM * 128 + kClassPad * 128) + kSmemAlign;
    P->smem_fwd1p = (size_t)kF1Stages * kF1StageBytes + (size_t)(P->c_last / kBlockK) * kClassPad * 128 + kSmemAlign;
    {
        // One tile per block, or persistent blocks?  us, one-tile / persistent:
        // from 192 channels on the one-tile blocks are large (three an SM at 192, two at 256 and 320, one from 384 on) and the
        // line is their first wave: 192 channels, 444 tiles 8.4 / 8.6, 508 tiles 9.6 / 8.6; 256, 254 tiles 6.5 / 6.5, 339 tiles
        // 10.2 / 8.6, 7200 tiles 110 / 90 (0.93 of the HBM copy bandwidth); 320, 296 tiles 5.4 / 5.6, 450 tiles 9.3 / 7.7; 512, 148
        // tiles 5.2 / 5.5, 226 tiles 8.7 / 6.7; 704, 148 tiles 5.7 / 6.1, 226 tiles 9.7 / 8.1.
        // At 128 channels five blocks an SM have more bytes in flight than the ring and it pays late: 704 tiles 6.1 / 7.2, 1350
        // tiles 10.2 / 10.7, 1808 tiles 13.2 / 13.1, 2112 tiles 15.5 / 14.9, 3600 tiles 32.0 / 29.7.  At 64 channels never: 1350
        // tiles 8.7 / 10.2, 7200 tiles 36.7 / 40.8.
        // ST_FWD1X1_PERSISTENT=0/1 forces a choice.
        const int64_t tiles = (int64_t)((P->p + kTileM - 1) / kTileM) * b.S;
        const int slices = P->c_last / kBlockK, per_sm = (int)((size_t)227 * 1024 / P->smem_fwd1);
        bool use = slices >= 3 ? tiles > (int64_t)148 * per_sm : slices == 2 && tiles >= (int64_t)148 * 13;
        if (const char* e = getenv("ST_FWD1X1_PERSISTENT")) { if (e[0] == '0') use = false; else if (e[0] == '1') use = true; }
        if (const char* e = getenv("ST_TEST_STALL_FWD1X1")) if (e[0] == '1') { P->test_stall = true; use = false; }
        // the one-tile form keeps the whole channel extent of its tile in shared memory: beyond 704 channels it no
        // longer fits, and the persistent form (a ring of eight stages, whatever the channel count) takes over
        if (P->smem_fwd1 > (size_t)227 * 1024) use = true;
        P->fwd1_persistent = use && P->smem_fwd1p <= (size_t)227 * 1024;
    }
    // Launched early behind a loss kernel that fills the GPU, the weight gradient's blocks start as SMs are left: one block per SM
    // then keeps them from piling up on the first ones, and the room goes into the ring.  Where that kernel leaves SMs free (its
    // tiles are fewer), they start there at once, in pairs, and all features of a block's three stages are there when the gradient
    // is.  (Train: one more block per stream assesses the prediction.)  us of a call of eight steps, three stages / one block per SM with three, five, seven, ten: 256 channels 180 x 320
    // 283.7 / 278.5, 275.6, 276.2, 279.7; 128 channels 270 x 480 470 / 453, 442, 455, 460; 90 x 160 (78 tiles) 156.9 / 160.8, 161.8.
    const int64_t wg1_blocks = (int64_t)P->split2 * P->msplit2 * b.S;
    P->wg1_deep = b.chain_early && wg1_blocks + b.S <= P->n_sms && (int64_t)upsample_ce_blocks(b.h, b.w, b.C) * b.S > P->n_sms;
    P->smem_wg1 = (P->wg1_deep ? kWg1Deep : kWg1Stages) * ((size_t)(m_last / P->msplit2) * 2 * kChunkPix * 128 + kClassPad * 128) + kSmemAlign;
    if (P->wg1_deep) P->smem_wg1 = one_per_sm(P->smem_wg1, wg1_blocks, P->n_sms);
    if (nb) {
        P->tiles_b = (P->p + kTileM - 1) / kTileM;
        P->groups_b = (P->c_last + kBackCols - 1) / kBackCols;
        split_geometry(P->tiles_b, 148 / P->groups_b, &P->per_b, &P->split_b);
        P->smem_back1 = (size_t)kBackStages * kBackStageBytes + kBackWBytes + kBackOutBytes + kSmemAlign;
    }
    if (P->c_last / kBlockK > kMaxKBlocks || (!P->fwd1_persistent && P->smem_fwd1 > lim) || P->smem_wg1 > lim) {
        snprintf(err, err_len, "shared memory per block exceeds 227 KB for these channel counts");
        delete P; return nullptr;
    }
    cudaError_t e = allow_shared_memory(P->fwd1_persistent ? (const void*)tc_fwd1x1p_kernel : (const void*)tc_fwd1x1_kernel);
    if (e == cudaSuccess) e = P->wg1_deep ? allow_shared_memory((const void*)tc_wgrad1x1_kernel<kWg1Deep>) : allow_shared_memory((const void*)tc_wgrad1x1_kernel<kWg1Stages>);
    for (int i = 0; i < nb; ++i) {
        if (e == cudaSuccess) e = allow_shared_memory((const void*)fwd3_kernel<0>(P->blk[i].walk_fwd));
        if (e == cudaSuccess && b.blk[i].pass_back) e = allow_shared_memory((const void*)fwd3_kernel<1>(P->blk[i].walk_back));
        if (e == cudaSuccess) e = allow_shared_memory((const void*)wgrad3_kernel(P->blk[i].wg));
    }
    if (nb && e == cudaSuccess) e = allow_shared_memory((const void*)tc_back1x1_kernel);
    if (e != cudaSuccess) { snprintf(err, err_len, "shared-memory attribute: %s", cudaGetErrorString(e)); delete P; return nullptr; }
    return P;
}

void tc_plan_destroy(TcPlan* P) { delete P; }

static bool fwd1_early_enabled()     // ST_FWD1_EARLY=0 switches the early activation fetch off
{
    static const bool on = [] { const char* e = getenv("ST_FWD1_EARLY"); return !(e && e[0] == '0'); }();
    return on;
}

static const char* const kFwd3Names[kMaxBlocks] = {"tc_fwd3x3", "tc_fwd3x3#2"};
static const char* const kWg3Names[kMaxBlocks] = {"tc_wgrad3x3", "tc_wgrad3x3#2"};

int tc_forward_blocks(const TcPlan* P, int first, int last, cudaStream_t s, StageTimer* t, const int* skip, int64_t skip_stride)
{
    const TcBuffers& b = P->b;
    int n = 0;
    for (int i = first; i < last; ++i) {
        const TcBlock& k = b.blk[i];
        const TcBlockPlan& q = P->blk[i];
        const Fwd3Walk& wk = q.walk_fwd;
        ST_REPEAT(t) launch_early(b.chain_early != 0, fwd3_kernel<0>(wk), dim3(wk.grid), dim3(kFwd3Threads), q.smem_fwd, s,
            q.in_fwd, q.skip_fwd, k.c_prev / kBlockK, k.c_skip / kBlockK, q.w_map, q.w_map_q, fwd3_stages(k.c_out, wk.halves), wk.n_full, wk.n_items,
            wk.tail_split, b.theta, b.n_params, k.b_off, q.out_st, k.relu_bits, (float*)nullptr, k.c_out, b.h, b.w, pow2_cols(2 * wk.halves * k.c_out),
            b.err, skip, skip_stride);
        if (t) t->mark(kFwd3Names[i], s, st_repeats(t));
        n += st_repeats(t);
    }
    return n;
}

int tc_forward(const TcPlan* P, cudaStream_t s, StageTimer* t, const int* skip, int64_t skip_stride, bool after_update, int first_block)
{
    const TcBuffers& b = P->b;
    int n = tc_forward_blocks(P, first_block, b.n_blocks, s, t, skip, skip_stride);
    const int tiles1 = (P->p + kTileM - 1) / kTileM;
    if (P->fwd1_persistent) {
        int gx = P->n_sms / b.S;
        if (gx < 1) gx = 1;
        if (gx > tiles1) gx = tiles1;
        ST_REPEAT(t) launch_early(b.chain_early != 0, tc_fwd1x1p_kernel, dim3(gx, b.S), dim3(kF1Threads), P->smem_fwd1p, s,
            P->act_fwd, P->w2_map, b.theta, b.n_params, b.b2_off, b.z, b.C, P->p, P->c_last / kBlockK, b.err, skip, skip_stride);
    } else {
        // one-layer head, no per-stream skip flags to wait for, not a timing run: the activations are the frozen
        // features, which no kernel of the loop writes
        const bool a_early = after_update && !b.n_blocks && !skip && !t && fwd1_early_enabled();
        ST_REPEAT(t) launch_early(a_early || b.chain_early, tc_fwd1x1_kernel, dim3(tiles1, b.S), dim3(kThreadsTc), P->smem_fwd1, s,
            P->act_fwd, P->w2_map, b.theta, b.n_params, b.b2_off, b.z, b.C, P->p, P->c_last / kBlockK, b.err, skip, skip_stride,
            a_early ? 1 : 0, P->test_stall ? (1u << 12) : kSpinLimit, P->test_stall ? 16u : 0u);
    }
    if (t) t->mark("tc_fwd1x1", s, st_repeats(t));
    return n + st_repeats(t);
}

int tc_backward(const TcPlan* P, cudaStream_t s, StageTimer* t, const int* skip, int64_t skip_stride, const TrainCtl* ctl)
{
    const TcBuffers& b = P->b;
    int n = 0;
    TrainCtl no_ctl;
    memset(&no_ctl, 0, sizeof no_ctl);
    const int nb = b.n_blocks;
    if (!nb || !b.blk[nb - 1].trained) {                  // nothing is passed back into a frozen block (Section 4.2)
        // one-layer head: the activations are the frozen features, which no kernel of the loop writes
        const int a_early = (!nb && !skip && !t && b.chain_early) ? 1 : 0;
        ST_REPEAT(t) launch_early(b.chain_early != 0, P->wg1_deep ? tc_wgrad1x1_kernel<kWg1Deep> : tc_wgrad1x1_kernel<kWg1Stages>,
            dim3(P->split2 * P->msplit2 + (ctl ? 1 : 0), b.S), dim3(kThreadsTc), P->smem_wg1, s, P->act_wg, P->dz_map, b.w2_partials, P->c_last, P->chunks2, P->per2, P->msplit2, P->cols2, b.err, skip, skip_stride,
            a_early, ctl ? 1 : 0, ctl ? *ctl : no_ctl);
        if (t) t->mark("tc_wgrad1x1", s, st_repeats(t));
        return n + st_repeats(t);
    }
    {
        const TcBlock& k = b.blk[nb - 1];
        ST_REPEAT(t) launch_early(b.chain_early != 0, tc_back1x1_kernel, dim3(P->split_b * P->groups_b + (ctl ? 1 : 0), b.S), dim3(kBackThreads),
            P->smem_back1, s, P->act_fwd, P->dz_map, P->w2_map, P->dout_map, k.relu_bits, k.b_partials, b.w2_partials, k.c_out, P->p, P->tiles_b,
            P->per_b, P->groups_b, b.err, skip, skip_stride, ctl ? 1 : 0, ctl ? *ctl : no_ctl);
        if (t) t->mark("tc_back1x1", s, st_repeats(t));
        n += st_repeats(t);
    }
    for (int i = nb - 1; i >= 0 && b.blk[i].trained; --i) {
        const TcBlock& k = b.blk[i];
        const TcBlockPlan& q = P->blk[i];
        ST_REPEAT(t) launch_early(b.chain_early != 0, wgrad3_kernel(q.wg), dim3(q.wg.units * q.wg.n_split, b.S), dim3(kThreadsTc),
            wg3_bytes(q.wg), s, q.in_wg, q.skip_wg, k.c_prev / kBlockK, q.odd_wg, (k.c_skip ? k.c_skip : k.c_prev) - kBlockK, q.dout_wg, k.w_partials, k.c_prev + k.c_skip, k.c_out, q.wg.chunks_x, q.wg.chunks,
            q.wg.per, q.wg.n_split, b.err, skip, skip_stride, i == 0 && !skip && !t && b.chain_early ? 1 : 0);
        if (t) t->mark(kWg3Names[i], s, st_repeats(t));
        n += st_repeats(t);
        if (k.pass_back) {
            // gradient with respect to the previous block's output: the tile walk of the forward over this block's
            // output gradient, with the mirrored and transposed weights; masked by the previous block's ReLU bits
            const TcBlock& r = b.blk[i - 1];
            const Fwd3Walk& wk = q.walk_back;
            ST_REPEAT(t) launch_early(b.chain_early != 0, fwd3_kernel<1>(wk), dim3(wk.grid), dim3(kFwd3Threads), q.smem_back, s,
                q.dout_fwd, q.dout_fwd, k.c_out / kBlockK, 0, q.wt_map, q.wt_map_q, fwd3_stages(k.c_prev, wk.halves), wk.n_full, wk.n_items, wk.tail_split,
                (const float*)nullptr, (int64_t)0, (int64_t)0, q.dprev_st, r.relu_bits, r.b_partials, k.c_prev, b.h, b.w,
                pow2_cols(2 * wk.halves * k.c_prev), b.err, skip, skip_stride);
            if (t) t->mark("tc_dgrad3x3", s, st_repeats(t));
            n += st_repeats(t);
        }
    }
    return n;
}

}  // namespace st
