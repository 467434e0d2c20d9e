// Loss weighting against class imbalance (Section 5.2): pixels near and within non-background objects weigh more.
// Computed once per key frame (the labels do not change over the K steps): a pixel is "near" if a pixel within
// `radius` rows and columns of it (square window, cut at the frame border) carries a label other than the
// background class.  The result is the label map again with bit 7 set on the weighted pixels, which is what the fused
// loss kernel reads, so that the weighting costs the step no extra memory traffic.  Labels above 126 cannot be tagged
// and become 127.
//
// A block tags 64 columns x 32 rows.  A warp reads the 128 columns around a row as one line (a radius above 32 needs 32 more on
// each side) and packs them into bits, a thread per row widens them by shifts that double, a thread per row and 32 columns
// takes the OR over its rows.  Bound by latency (a 720p frame is 0.9 MB): at radius 8 the label call of a frame, arg-max
// included, takes 19.3 us; 33.5 us with two passes over bytes, which read each 2 radius + 1 times.
#include "st_internal.h"

namespace st {

namespace {

constexpr int kTagCols = 64, kTagRows = 32, kTagRadius = 64, kTagThreads = 256;

__global__ void __launch_bounds__(kTagThreads)
near_tag_kernel(const uint8_t* __restrict__ lab, int H, int W, uint32_t background, int radius, uint8_t* __restrict__ out)
{
    __shared__ uint32_t seen[kTagRows + 2 * kTagRadius][6];                  // columns x0 - 64 .. x0 + 127
    __shared__ uint32_t wide[kTagRows + 2 * kTagRadius][2];
    __shared__ uint32_t near[kTagRows][2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int x0 = blockIdx.x * kTagCols, y0 = blockIdx.y * kTagRows, rows = kTagRows + 2 * radius;
    pdl_wait();
    // 32 columns per 8 lanes -> one word in the first of them; the frame width is a multiple of 4
    auto pack = [&](int y, int x) -> uint32_t {
        uint32_t m = 0;
        if (y >= 0 && y < H && x >= 0 && x < W) {
            const uint32_t v = *reinterpret_cast<const uint32_t*>(lab + (int64_t)y * W + x);
            m = ((__vcmpne4(v, background * 0x01010101u) & 0x08040201u) * 0x01010101u) >> 24;
        }
        m <<= 4 * (lane & 7);
#pragma unroll
        for (int k = 1; k < 8; k <<= 1) m |= __shfl_xor_sync(0xffffffffu, m, k);
        return m;
    };
    for (int r = warp; r < rows; r += kTagThreads / 32) {
        const int y = y0 - radius + r;
        const uint32_t m = pack(y, x0 - 32 + 4 * lane);
        uint32_t far = 0;
        if (radius > 32) far = pack(lane < 16 ? y : -1, lane < 8 ? x0 - 64 + 4 * lane : x0 + 96 + 4 * (lane - 8));
        if ((lane & 7) == 0) seen[r][1 + (lane >> 3)] = m;
        if (lane == 0 || lane == 8) seen[r][lane ? 5 : 0] = far;
    }
    __syncthreads();
    if (tid < rows) {
        const uint32_t* w = seen[tid];
        uint64_t lo = w[0] | (uint64_t)w[1] << 32, hi = w[4] | (uint64_t)w[5] << 32;
        uint64_t up = w[2] | (uint64_t)w[3] << 32, down = up;
        for (int have = 1; have < radius + 1;) {             // up: columns x - have + 1 .. x, down: x .. x + have - 1
            const int k = min(min(have, 32), radius + 1 - have);
            up |= up << k | lo >> (64 - k); lo |= lo << k;
            down |= down >> k | hi << (64 - k); hi |= hi >> k;
            have += k;
        }
        up |= down;
        wide[tid][0] = (uint32_t)up; wide[tid][1] = (uint32_t)(up >> 32);
    }
    __syncthreads();
    if (tid < 2 * kTagRows) {
        uint32_t m = 0;
        for (int k = 0; k <= 2 * radius; ++k) m |= wide[(tid >> 1) + k][tid & 1];
        near[tid >> 1][tid & 1] = m;
    }
    __syncthreads();
#pragma unroll
    for (int i = tid; i < kTagRows * kTagCols / 4; i += kTagThreads) {
        const int r = i / (kTagCols / 4), c = 4 * (i % (kTagCols / 4));
        if (y0 + r >= H || x0 + c >= W) continue;
        const int64_t at = (int64_t)(y0 + r) * W + x0 + c;
        const uint32_t four = near[r][c >> 5] >> (c & 31) & 15u;
        const uint32_t tags = (four * 0x00204081u & 0x01010101u) << 7;       // bit k of the four into byte k
        *reinterpret_cast<uint32_t*>(out + at) = __vminu4(*reinterpret_cast<const uint32_t*>(lab + at), 0x7f7f7f7fu) | tags;
    }
    pdl_launch_dependents();
}

}  // namespace

void launch_object_weight_tags(const uint8_t* labels, int H, int W, int background, int radius, uint8_t* tagged, cudaStream_t s)
{
    launch_early(pdl_enabled(), near_tag_kernel, dim3((W + kTagCols - 1) / kTagCols, (H + kTagRows - 1) / kTagRows), dim3(kTagThreads), 0, s,
                 labels, H, W, (uint32_t)background, radius, tagged);
}

}  // namespace st
