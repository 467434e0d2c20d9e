// Mean IoU of a confusion matrix, shared by the kernels that finish an agreement measurement themselves.
#pragma once

#include <cuda_runtime.h>

namespace st {

// Mean IoU (Section 3.2): IoU_c = conf[c][c] / (row_c + col_c - conf[c][c]), averaged over the
// classes present in the label (row_c > 0).  Integer counts, double arithmetic, fixed order.
// Called by all threads of a block of any number of whole warps; the value is returned to thread 0 only.  `iou` and `present`
// are the block's shared arrays, written for classes below C only.  The counts are read past the L1
// cache: the caller may be the last block of a kernel whose other blocks have just added to them.  Matrices of up to kMiouStage classes
// are first copied to shared memory in one coalesced pass (one memory latency instead of one per row element).
constexpr int kMiouStage = 32, kMiouClasses = 256;
// The copy to shared memory in two halves, for a caller that has other loads to issue while these are on their way:
// miou_fetch starts the thread's share (blocks of kMiouFetchThreads threads, C <= kMiouStage), block_miou takes it over.
constexpr int kMiouFetchThreads = 256;
struct MiouFetch { unsigned long long v[kMiouStage * kMiouStage / kMiouFetchThreads]; };
__device__ __forceinline__ MiouFetch miou_fetch(const unsigned long long* conf_g, int C)
{
    MiouFetch f;
#pragma unroll
    for (int k = 0; k < kMiouStage * kMiouStage / kMiouFetchThreads; ++k) {
        const int e = threadIdx.x + kMiouFetchThreads * k;
        f.v[k] = e < C * C ? __ldcg(conf_g + e) : 0ull;
    }
    return f;
}
// Mean over the present classes, added in class order (thread 0; 0 elsewhere)
__device__ __forceinline__ double mean_iou(int C, const double (&iou)[kMiouClasses], const int (&present)[kMiouClasses])
{
    double m = 0.0;
    if (threadIdx.x == 0) {
        double sum = 0.0; int n = 0;
        for (int k0 = 0; k0 < C; k0 += 8) {                // eight reads in flight, added in class order
            double v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) { v[j] = k0 + j < C ? iou[k0 + j] : 0.0; n += k0 + j < C ? present[k0 + j] : 0; }
#pragma unroll
            for (int j = 0; j < 8; ++j) sum += v[j];
        }
        m = n ? sum / n : 0.0;
    }
    return m;
}

__device__ __forceinline__ double block_miou(const unsigned long long* conf_g, int C, double (&iou)[kMiouClasses], int (&present)[kMiouClasses],
                                           const MiouFetch* fetched = nullptr)
{
    __shared__ unsigned long long staged[kMiouStage * kMiouStage];
    const unsigned long long* conf = conf_g;
    if (C <= kMiouStage) {                                 // block-uniform
        if (fetched) {
#pragma unroll
            for (int k = 0; k < kMiouStage * kMiouStage / kMiouFetchThreads; ++k) {
                const int e = threadIdx.x + kMiouFetchThreads * k;
                if (e < C * C) staged[e] = fetched->v[k];
            }
        } else {
            for (int e = threadIdx.x; e < C * C; e += blockDim.x) staged[e] = __ldcg(conf_g + e);
        }
        __syncthreads();
        conf = staged;
    }
    if (conf == staged) {
        // eight lanes per class, four classes to a warp (one thread per class: 42 dependent reads in a row for 21 classes)
        const int lane = threadIdx.x & 31, part = lane & 7;
        for (int c0 = (threadIdx.x >> 5) * 4; c0 < C; c0 += (blockDim.x >> 5) * 4) {      // the same for all lanes of a warp
            const int c = c0 + (lane >> 3);
            unsigned long long row = 0, col = 0;
#pragma unroll
            for (int k = 0; k < kMiouStage / 8; ++k) {
                const int q = part + 8 * k;
                if (c < C && q < C) { row += conf[c * C + q]; col += conf[q * C + c]; }
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) { row += __shfl_xor_sync(0xffffffffu, row, o); col += __shfl_xor_sync(0xffffffffu, col, o); }
            if (part == 0 && c < C) {
                const unsigned long long inter = conf[c * C + c];
                iou[c] = row > 0 ? (double)inter / (double)(row + col - inter) : 0.0;
                present[c] = row > 0;
            }
        }
    } else {
        // larger matrices stay in global memory: a warp per class, its lanes along the row and the column (81 classes: 162
        // dependent-latency loads per thread otherwise)
        const int lane = threadIdx.x & 31;
        for (int c = threadIdx.x >> 5; c < C; c += blockDim.x >> 5) {
            unsigned long long row = 0, col = 0;
#pragma unroll 4
            for (int q = lane; q < C; q += 32) { row += __ldcg(conf + c * C + q); col += __ldcg(conf + q * C + c); }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) { row += __shfl_xor_sync(0xffffffffu, row, o); col += __shfl_xor_sync(0xffffffffu, col, o); }
            if (lane == 0) {
                const unsigned long long inter = __ldcg(conf + c * C + c);
                iou[c] = row > 0 ? (double)inter / (double)(row + col - inter) : 0.0;
                present[c] = row > 0;
            }
        }
    }
    __syncthreads();
    return mean_iou(C, iou, present);
}

// The end of a kernel that counts: its last block reads the finished matrix once, delivers it (out; not if null, and the counters then stay),
// leaves the counters at zero and returns the mean IoU to thread 0, like block_miou.  `stage` is shared memory for C * C counts, which stay
// below 2^32.  (block_miou and a second pass that delivers: one more round trip, and with 81 classes, whose sums it fetches row by row
// and whose counts the second pass fetched one by one, 22 us behind a mask of 12.7.)
template <int THREADS>
__device__ __forceinline__ double deliver_matrix(unsigned long long* conf, int C, unsigned long long* out, unsigned int* stage, double (&iou)[kMiouClasses],
                                                 int (&present)[kMiouClasses])
{
    const int n = C * C, tid = threadIdx.x;
    for (int e0 = tid; e0 < n; e0 += 8 * THREADS) {
        unsigned long long v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = e0 + j * THREADS < n ? __ldcg(conf + e0 + j * THREADS) : 0ull;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int e = e0 + j * THREADS;
            if (e >= n) break;
            stage[e] = (unsigned int)v[j];
            if (out) { out[e] = v[j]; conf[e] = 0; }
        }
    }
    __syncthreads();
    // eight lanes per class, four classes to a warp
    const int lane = tid & 31, part = lane & 7;
    for (int c0 = (tid >> 5) * 4; c0 < C; c0 += THREADS / 8) {
        const int c = c0 + (lane >> 3);
        unsigned int row = 0, col = 0;
        if (c < C) {
#pragma unroll 4
            for (int q = part; q < C; q += 8) { row += stage[c * C + q]; col += stage[q * C + c]; }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) { row += __shfl_xor_sync(0xffffffffu, row, o); col += __shfl_xor_sync(0xffffffffu, col, o); }
        if (part == 0 && c < C) {
            const unsigned int inter = stage[c * C + c];
            iou[c] = row > 0 ? (double)inter / (double)((unsigned long long)row + col - inter) : 0.0;
            present[c] = row > 0;
        }
    }
    __syncthreads();
    return mean_iou(C, iou, present);
}

}  // namespace st
