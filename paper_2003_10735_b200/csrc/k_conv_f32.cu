// fp32 CUDA-core convolutions of the head (gemm_precision 0): forward, weight/bias gradients and
// the gradient passed from the 1x1 output layer to the hidden activation.  Planar [C][h][w].
// These state Algorithm 1's Forward / PartialBackward for the trainable back part in plain FMA
// arithmetic with fixed-order reductions (bit-reproducible run to run).  The bf16 tensor-core path
// replaces them when gemm_precision is 1.
//
// Every operand that a convolution reads lies in a padded plane (PadF32: zeros around the map, rows of whole 16-byte vectors
// at any width), so that tiles are copied 16 bytes at a time and without bounds checks, and the zero padding of the
// 3x3 layer needs no code.
//
// What bounds them: the fp32 pipes (a 3x3 layer 96 -> 48 on 90 x 160 nodes is 0.6 G multiply-adds, 16 us at the rate this
// GPU sustains) and the issue slots beside them.  Both kernels therefore keep a register tile per thread whose operands
// come from shared memory without bank conflicts at eight or more multiply-adds per load, multiply two output channels at
// a time (packed fp32x2: half the instructions), and bring the next stage in with asynchronous copies while the current
// one is multiplied.  The copies' places are worked out once and advanced by additions: divisions for every vector of every stage took as
// many instructions as a 1x1 layer's multiplications.  us before / now: that layer's forward 50.0 / 41.7, weight gradient 37.3 / 35.2; 1x1 forward, 21
// classes over 256 channels on 180 x 320 43.0 / 34.5, 81 over 48 on 90 x 160 12.7 / 10.6, 100 over 200 on 120 x 200 64.4 / 51.5.
#include "st_internal.h"

namespace st {

namespace {

constexpr int kTileX = 32;      // pixels per tile row: one lane per column
constexpr int kFwdRows = 4;     // forward: pixel rows of a tile, all four held by one lane
constexpr int kCiSplit = 4;     // forward: warps that share an output tile, each with a quarter of the input channels
constexpr int kFwdGroups = 3;   // forward: groups of output channels per block at most (12 warps, two blocks per SM)

// `BYTES` of global memory to shared memory, or zeros where `ok` is false.
template <int BYTES>
__device__ __forceinline__ void copy_async(float* dst, const float* src, bool ok)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(ok ? 4 : 0) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// A tile row in shared memory: the 32 columns, and for a 3x3 layer four more on either side (whole vectors; one is used)
template <int KS> __host__ __device__ constexpr int row_floats() { return KS == 3 ? kTileX + 8 : kTileX; }
template <int KS> __host__ __device__ constexpr int first_tap() { return KS == 3 ? kPadLeft - 1 : 0; }

// ------------------------------------------------------------------------------------------------
// Weights are in internal order, [tap][cout][cin] (for a 1x1 layer [cout][cin]).
// Forward, and the gradient passed back through the 1x1 output layer (the same sum with the weight transposed).
//   out[co][y][x] = b[co] + sum_{ci,ky,kx} W[co][ci][ky][kx] * in[ci][y+ky-r][x+kx-r]  (zero padding)
// A warp computes 32 x 4 pixels times CO output channels: lane = column, so every input value is read from shared
// memory without conflicts and serves all taps of its column, and the weights are broadcasts.  kCiSplit warps share
// the tile with a quarter of the input channels each (with 32 sums per lane there are too few warps otherwise: 690 on
// 592 schedulers for the layer above); their sums are added in order at the end, warp q finishing pixel row q.
// ------------------------------------------------------------------------------------------------
struct ConvF32 {
    const float* in; const float* Wt; const float* b; const float* mask; float* out;
    int Cin, Cout, h, w, relu, transposed;      // transposed: W is [ci][co] (1x1 only); mask: nullptr, or zero the output where it is <= 0
    int out_pitch; int64_t out_plane;           // of the output and the mask: a plain plane or a padded one
    int64_t in_stride, w_stride, b_stride, out_stride;
};
template <int KS> __host__ __device__ constexpr int fwd_stage_ci() { return KS == 3 ? 2 : 4; }       // input channels per warp and stage
template <int KS> __host__ __device__ constexpr int fwd_in_floats() { return kCiSplit * fwd_stage_ci<KS>() * (kFwdRows + KS - 1) * row_floats<KS>(); }
template <int KS, int CO>
size_t fwd_smem(int ng)
{
    const size_t stage = fwd_in_floats<KS>() + (size_t)kCiSplit * fwd_stage_ci<KS>() * KS * KS * CO * ng;
    const size_t red = (size_t)kCiSplit * ng * kFwdRows * CO * 32;
    return (2 * stage > red ? 2 * stage : red) * sizeof(float);
}

template <int KS, int CO>
__global__ void __launch_bounds__(128 * kFwdGroups, 2)
conv_fwd_f32_kernel(ConvF32 a, int tiles_x)
{
    constexpr int T = KS * KS, CIC = fwd_stage_ci<KS>(), NC = kCiSplit * CIC, TH = kFwdRows + KS - 1, TW = row_floats<KS>(), VEC = TW / 4;
    extern __shared__ __align__(16) float smem_f[];
    const int ng = blockDim.x / (32 * kCiSplit), COB = CO * ng;
    const int stage = fwd_in_floats<KS>() + NC * T * COB;
    const int s = blockIdx.z, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cs = warp % kCiSplit, g = warp / kCiSplit;
    const int x0 = (blockIdx.x % tiles_x) * kTileX, y0 = (blockIdx.x / tiles_x) * kFwdRows, co0 = blockIdx.y * COB;
    const PadF32 pad(a.h, a.w);
    pdl_wait();
    // first row and vector of the tile in the padded planes
    const float* in = a.in + s * a.in_stride + (int64_t)(y0 + (KS == 3 ? 0 : kPadTop)) * pad.pitch + x0 + (KS == 3 ? 0 : kPadLeft);
    const float* Wt = a.Wt + s * a.w_stride;

    // The places of a thread's weights are the same in every stage but for the channel offset (NC consecutive input
    // channels of one tap and output channel lie side by side).
    constexpr int kWPer = (NC * T * CO + 32 * kCiSplit - 1) / (32 * kCiSplit);
    const int wc = tid % NC;
    int w_src[kWPer];          // a layer has fewer than 2^31 weights
    int w_dst[kWPer];
#pragma unroll
    for (int i = 0; i < kWPer; ++i) {
        const int q = tid / NC + i * ((int)blockDim.x / NC), t = q / COB, co = q % COB;
        w_dst[i] = t < T ? (wc * T + t) * COB + co : -1;
        w_src[i] = co0 + co >= a.Cout ? -1 : a.transposed ? wc * a.Cout + co0 + co : (t * a.Cout + co0 + co) * a.Cin + wc;
    }
    const int w_step = a.transposed ? a.Cout : 1;
    // ... and so are those of its input vectors: counted in vectors from the stage's first channel, they fit 32 bits on any map
    constexpr int kIn = NC * TH * VEC, kInPer = (kIn + 32 * kCiSplit - 1) / (32 * kCiSplit);
    const uint32_t plane_v = (uint32_t)(pad.plane / 4), pitch_v = (uint32_t)(pad.pitch / 4);
    uint32_t in_src[kInPer];
#pragma unroll
    for (int i = 0; i < kInPer; ++i) {
        const int e = tid + i * (int)blockDim.x;
        in_src[i] = (uint32_t)(e / (TH * VEC)) * plane_v + (uint32_t)(e / VEC % TH) * pitch_v + (uint32_t)(e % VEC);
    }
    auto fetch = [&](int c0, float* dst) {
        const float4* from = reinterpret_cast<const float4*>(in + (int64_t)c0 * pad.plane);
        const uint32_t end = (uint32_t)min(a.Cin - c0, NC) * plane_v;      // a place lies inside its channel's plane
        float* to = dst + 4 * tid;
#pragma unroll
        for (int i = 0; i < kInPer; ++i, to += 4 * blockDim.x) {
            const bool ok = in_src[i] < end;
            if (tid + i * (int)blockDim.x < kIn) copy_async<16>(to, reinterpret_cast<const float*>(from + (ok ? in_src[i] : 0u)), ok);
        }
        float* wd = dst + fwd_in_floats<KS>();              // [ci][tap][co]
#pragma unroll
        for (int i = 0; i < kWPer; ++i)
            if (w_dst[i] >= 0) {
                const bool ok = w_src[i] >= 0 && c0 + wc < a.Cin;
                copy_async<4>(wd + w_dst[i], ok ? Wt + w_src[i] + c0 * w_step : Wt, ok);
            }
        copy_commit();
    };

    float2 acc[kFwdRows][CO / 2];                           // two output channels side by side
#pragma unroll
    for (int r = 0; r < kFwdRows; ++r)
#pragma unroll
        for (int k = 0; k < CO / 2; ++k) acc[r][k] = make_float2(0.f, 0.f);
    fetch(0, smem_f);
    int buf = 0;
    for (int c0 = 0; c0 < a.Cin; c0 += NC, buf ^= 1) {
        if (c0 + NC < a.Cin) { fetch(c0 + NC, smem_f + (buf ^ 1) * stage); copy_wait<1>(); }
        else copy_wait<0>();
        __syncthreads();
        const float* xs = smem_f + buf * stage + cs * CIC * TH * TW + lane + first_tap<KS>();
        const float* ws = smem_f + buf * stage + fwd_in_floats<KS>() + cs * CIC * T * COB + g * CO;
#pragma unroll
        for (int c = 0; c < CIC; ++c) {
#pragma unroll
            for (int kx = 0; kx < KS; ++kx) {
                float v[TH];
#pragma unroll
                for (int r = 0; r < TH; ++r) v[r] = xs[(c * TH + r) * TW + kx];
#pragma unroll
                for (int ky = 0; ky < KS; ++ky) {
                    float2 wv[CO / 2];
#pragma unroll
                    for (int k = 0; k < CO / 2; k += 2)
                        *reinterpret_cast<float4*>(wv + k) = *reinterpret_cast<const float4*>(ws + (c * T + ky * KS + kx) * COB + 2 * k);
#pragma unroll
                    for (int r = 0; r < kFwdRows; ++r)
#pragma unroll
                        for (int k = 0; k < CO / 2; ++k) acc[r][k] = __ffma2_rn(wv[k], make_float2(v[r + ky], v[r + ky]), acc[r][k]);
                }
            }
        }
        __syncthreads();
    }
    pdl_launch_dependents();     // late: blocks of the next kernel launched earlier crowd the SMs that finish first
    // the four quarters of the input channels, added in order: [quarter][group][row][channel][lane]
    float* red = smem_f;
#pragma unroll
    for (int r = 0; r < kFwdRows; ++r)
#pragma unroll
        for (int k = 0; k < CO / 2; ++k) {
            float* q = red + (((cs * ng + g) * kFwdRows + r) * CO + 2 * k) * 32 + lane;
            q[0] = acc[r][k].x; q[32] = acc[r][k].y;
        }
    __syncthreads();
    const int y = y0 + cs, x = x0 + lane;
    if (y >= a.h || x >= a.w) return;
#pragma unroll
    for (int k = 0; k < CO; ++k) {
        const int co = co0 + g * CO + k;
        if (co >= a.Cout) continue;
        float v = a.b ? __ldg(a.b + s * a.b_stride + co) : 0.f;
#pragma unroll
        for (int q = 0; q < kCiSplit; ++q) v += red[(((q * ng + g) * kFwdRows + cs) * CO + k) * 32 + lane];
        if (a.relu) v = fmaxf(v, 0.f);
        const int64_t i = s * a.out_stride + co * a.out_plane + (int64_t)y * a.out_pitch + x;
        a.out[i] = a.mask && !(a.mask[i] > 0.f) ? 0.f : v;
    }
}

template <int KS, int CO>
void launch_fwd(const ConvF32& a, int S, bool early, cudaStream_t s)
{
    const int tiles_x = (a.w + kTileX - 1) / kTileX, tiles_y = (a.h + kFwdRows - 1) / kFwdRows;
    const int tiles = tiles_x * tiles_y, groups = (a.Cout + CO - 1) / CO;
    // Channel groups per block: more of them share a tile's copy, fewer make finer blocks.  Taken: the number for which the
    // busiest SM has the least to do (48 channels on 90 x 160 nodes: 690 blocks of one group, five on the busiest SM,
    // against two of three groups).
    int ng = 1, ny = groups;
    int64_t least = INT64_MAX;
    for (int n = kFwdGroups; n >= 1; --n) {
        const int y = (groups + n - 1) / n;
        const int64_t busiest = ((int64_t)tiles * y * S + 147) / 148 * n;
        if (busiest < least) { least = busiest; ng = n; ny = y; }
    }
    launch_early(early, conv_fwd_f32_kernel<KS, CO>, dim3((unsigned)tiles, (unsigned)ny, (unsigned)S), dim3(32 * kCiSplit * ng), fwd_smem<KS, CO>(ng), s, a, tiles_x);
}

// ------------------------------------------------------------------------------------------------
// Weight gradients: dW[tap][co][ci] = sum_{y,x} dout[co][y][x] * in[ci][y+ky-r][x+kx-r].
// lane = input channel, a warp holds CO output channels x all taps: per four pixels one vector of inputs per tap row, and per
// pixel a broadcast of the CO gradients, feed CO * taps multiply-adds a pixel.  A block walks the chunks (32 x wg_rows pixels) of its
// range and leaves its sums as one partial result; the parameter update adds the partial results in order.  The rows of a
// chunk are divided among as many warps, whose sums are added in order at the end: one warp per channel group leaves the
// schedulers idle while it waits (1.5 warps each for the layer above).
// A 1x1 layer's warps hold CI = 1, 2 or 4 input channels per lane: a broadcast vector of gradients takes four cycles of the SM's
// path from shared memory, so with one channel four of them feed eight packed multiply-adds that need four cycles, and the
// path sets the time.  21 classes over 256 channels on 180 x 320 nodes, one channel / four: 78.4 / 40.6 us; 81 over 48 on
// 90 x 160, one / two: 20.8 / 14.7; 40 over 128, one / four: 53.6 / 33.1; 12 over 40, one / two: 17.1 / 13.8.  A 3x3 layer's
// inputs serve nine taps each already.  One barrier per chunk instead of two, and the bias sums divided among the rows' warps:
// 3x3 96 -> 48 39.3 -> 37.3 us, 128 -> 128 503 -> 478.
// ------------------------------------------------------------------------------------------------
template <int KS> __host__ __device__ constexpr int wg_rows() { return KS == 1 ? 4 : 2; }      // pixel rows of a chunk = warps per channel group
template <int KS> __host__ __device__ constexpr int wg_most_groups() { return KS == 1 ? 3 : 6; } // twelve warps per block at most
// A channel's pixels of a chunk: whole rows and four floats more, so that the pitch between channels is odd in vectors and the
// lanes (one channel each) read their vectors without conflicts.
template <int KS> __host__ __device__ constexpr int wg_ci_pitch() { return (wg_rows<KS>() + KS - 1) * row_floats<KS>() + 4; }
// Gradient tile [pixel][co]: the pitch is a multiple of four floats for the broadcasts, odd in fours
__host__ __device__ constexpr int wg_co_pitch(int COB) { return COB + (COB / 4 % 2 ? 0 : 4); }
template <int KS, int CO, int CI>
size_t wg_smem(int ng)
{
    const size_t stage = (size_t)32 * CI * wg_ci_pitch<KS>() + (size_t)wg_rows<KS>() * kTileX * wg_co_pitch(CO * ng);
    const size_t red = (size_t)(wg_rows<KS>() - 1) * ng * KS * KS * CO * 32 * CI + (size_t)wg_rows<KS>() * ng * CO;
    return (2 * stage > red ? 2 * stage : red) * sizeof(float);
}

struct WgradF32 {
    const float* in; const float* dout; float* partials; float* b_partials;
    int Cin, Cout, h, w, n_split;
    int64_t in_stride, dout_stride;
};

template <int KS, int CO, int CI>
__global__ void __launch_bounds__(384)
conv_wgrad_f32_kernel(WgradF32 a, int tiles_x, int n_chunks, int ci_tiles)
{
    constexpr int T = KS * KS, RW = wg_rows<KS>(), TH = RW + KS - 1, TW = row_floats<KS>(), VEC = TW / 4, CP = wg_ci_pitch<KS>();
    // 1x1 with one channel per lane: the next copy before the wait and the bias by one warp per channel group are the faster form
    // (21 classes over 32 channels on 180 x 320 nodes, three streams: 28.2 us, as the others 29.4)
    constexpr bool kShort = KS == 1 && CI == 1;
    extern __shared__ __align__(16) float smem_w[];
    const int ng = blockDim.x / (32 * RW), COB = CO * ng, pitch = wg_co_pitch(COB);
    const int stage = 32 * CI * CP + RW * kTileX * pitch;
    const int s = blockIdx.z, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_warps = (int)blockDim.x >> 5;
    const int g = warp / RW, rw = warp % RW;
    const int split = blockIdx.x, ci0 = (blockIdx.y % ci_tiles) * 32 * CI, co0 = (blockIdx.y / ci_tiles) * COB;
    const PadF32 pad(a.h, a.w);
    pdl_wait();
    const float* in = a.in + s * a.in_stride + (KS == 3 ? 0 : kPadTop * pad.pitch + kPadLeft);
    const float* dout = a.dout + s * a.dout_stride + kPadTop * pad.pitch + kPadLeft;
    const int c_begin = (int)((int64_t)n_chunks * split / a.n_split), c_end = (int)((int64_t)n_chunks * (split + 1) / a.n_split);

    // The copies of a chunk: a warp takes a channel's vectors, 32 and (3x3) the eight that are left, from places that are worked out once;
    // a chunk lies 32 columns behind the one before it, or at the beginning of the next rows.
    constexpr int kVecs = TH * VEC;
    static_assert(kVecs == 32 || kVecs == 40, "a channel's vectors");
    const int v_rest = 32 + (lane & 7);
    const int src0 = lane / VEC * pad.pitch + 4 * (lane % VEC), dst0 = lane / VEC * TW + 4 * (lane % VEC);
    const int src1 = v_rest / VEC * pad.pitch + 4 * (v_rest % VEC), dst1 = v_rest / VEC * TW + 4 * (v_rest % VEC);
    int at = c_begin / tiles_x * RW * pad.pitch + c_begin % tiles_x * kTileX, at_col = c_begin % tiles_x;
    auto fetch = [&](float* dst) {                          // the next chunk
        const float* from = in + (int64_t)(ci0 + warp) * pad.plane + at;
        const int64_t channels_on = (int64_t)n_warps * pad.plane;
        for (int c = warp; c < 32 * CI; c += n_warps, from += channels_on) {
            const bool ok = ci0 + c < a.Cin;
            copy_async<16>(dst + c * CP + dst0, ok ? from + src0 : in, ok);
            if (kVecs > 32 && lane < kVecs - 32) copy_async<16>(dst + c * CP + dst1, ok ? from + src1 : in, ok);
        }
        float* dd = dst + 32 * CI * CP;
        for (int row = warp; row < COB * RW; row += n_warps) {      // a warp copies one row of one channel at a time
            const int c = row / RW, r = row % RW;
            const bool ok = co0 + c < a.Cout;
            copy_async<4>(dd + (r * kTileX + lane) * pitch + c, ok ? dout + (co0 + c) * pad.plane + at + r * pad.pitch + lane : dout, ok);
        }
        copy_commit();
        at += kTileX;
        if (++at_col == tiles_x) { at_col = 0; at += RW * pad.pitch - tiles_x * kTileX; }
    };

    float2 acc[CI][CO / 2][T];                              // two output channels side by side
    float bias = 0.f;
#pragma unroll
    for (int j = 0; j < CI; ++j)
#pragma unroll
        for (int k = 0; k < CO / 2; ++k)
#pragma unroll
            for (int t = 0; t < T; ++t) acc[j][k][t] = make_float2(0.f, 0.f);
    if (c_begin < c_end) fetch(smem_w);
    int buf = 0;
    for (int chunk = c_begin; chunk < c_end; ++chunk, buf ^= 1) {
        if (kShort) {
            if (chunk + 1 < c_end) { fetch(smem_w + (buf ^ 1) * stage); copy_wait<1>(); }
            else copy_wait<0>();
            __syncthreads();
        } else {
            copy_wait<0>();
            __syncthreads();        // and every thread has done with the chunk before, whose place the next copy takes
            if (chunk + 1 < c_end) fetch(smem_w + (buf ^ 1) * stage);
        }
        const float4* xs = reinterpret_cast<const float4*>(smem_w + buf * stage + lane * CP);
        const float* ds = smem_w + buf * stage + 32 * CI * CP + g * CO;
        {
            const int r = rw;
            // four pixels at a time; a 3x3 layer's window is the last column of the vector before, the vector, the first column after
            float before[KS];
            float4 now[KS];
#pragma unroll
            for (int ky = 0; ky < KS; ++ky)
                if (KS == 3) { before[ky] = xs[(r + ky) * VEC].w; now[ky] = xs[(r + ky) * VEC + 1]; }
#pragma unroll 1
            for (int v = 0; v < kTileX / 4; ++v) {
                float win[CI][KS][KS + 3];
#pragma unroll
                for (int j = 0; j < CI; ++j)
#pragma unroll
                    for (int ky = 0; ky < KS; ++ky) {
                        if (KS == 3) {
                            const float4 next = xs[(r + ky) * VEC + v + 2];
                            win[j][ky][0] = before[ky];
                            win[j][ky][1] = now[ky].x; win[j][ky][KS / 2 + 1] = now[ky].y; win[j][ky][KS] = now[ky].z; win[j][ky][KS + 1] = now[ky].w;
                            win[j][ky][KS + 2] = next.x;
                            before[ky] = now[ky].w; now[ky] = next;
                        } else {
                            const float4 t = xs[j * 8 * CP + r * VEC + v];      // 32 channels on, in vectors
                            win[j][0][0] = t.x; win[j][0][1] = t.y; win[j][0][2] = t.z; win[j][0][3] = t.w;
                        }
                    }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float2 d[CO / 2];
#pragma unroll
                    for (int k = 0; k < CO / 2; k += 2) *reinterpret_cast<float4*>(d + k) = *reinterpret_cast<const float4*>(ds + (r * kTileX + 4 * v + i) * pitch + 2 * k);
#pragma unroll
                    for (int j = 0; j < CI; ++j)
#pragma unroll
                        for (int ky = 0; ky < KS; ++ky)
#pragma unroll
                            for (int kx = 0; kx < KS; ++kx) {
                                const float x = win[j][ky][i + kx];
#pragma unroll
                                for (int k = 0; k < CO / 2; ++k) acc[j][k][ky * KS + kx] = __ffma2_rn(d[k], make_float2(x, x), acc[j][k][ky * KS + kx]);
                            }
                }
            }
        }
        if (a.b_partials && ci0 == 0 && lane < CO && (!kShort || rw == 0))   // bias gradient: the sum of the gradients themselves
            for (int i = 0; i < (kShort ? RW : 1) * kTileX; ++i) bias += ds[((kShort ? 0 : rw * kTileX) + i) * pitch + lane];
        if (kShort) __syncthreads();
    }
    if (!kShort) __syncthreads();
    pdl_launch_dependents();
    const bool has_bias = a.b_partials && ci0 == 0 && rw == 0 && lane < CO && co0 + g * CO + lane < a.Cout;
    float* b_dst = a.b_partials + ((int64_t)s * a.n_split + split) * a.Cout + co0 + g * CO + lane;
    if (kShort && has_bias) *b_dst = bias;
    // the rows' sums, added in order: [row warp - 1][group][channel of the lane, channel pair, tap][lane]
    float2* red = reinterpret_cast<float2*>(smem_w) + g * (CI * CO / 2 * T) * 32 + lane;
    const int red_row = ng * (CI * CO / 2 * T) * 32;
    float* red_b = smem_w + 2 * (RW - 1) * red_row + g * CO + lane;     // [row warp][group][channel]
    if (!kShort && lane < CO) red_b[rw * COB] = bias;
    if (rw > 0)
#pragma unroll
        for (int j = 0; j < CI; ++j)
#pragma unroll
            for (int k = 0; k < CO / 2; ++k)
#pragma unroll
                for (int t = 0; t < T; ++t) red[(rw - 1) * red_row + ((j * (CO / 2) + k) * T + t) * 32] = acc[j][k][t];
    __syncthreads();
    if (rw > 0) return;
    if (!kShort && has_bias) {
        for (int q = 1; q < RW; ++q) bias += red_b[q * COB];
        *b_dst = bias;
    }
    // (added one by one while the results are stored, no load moves ahead of a store: 32 -> 16, 3x3, six streams 18.8 -> 21.2 us)
    if (kShort) {
#pragma unroll
        for (int k = 0; k < CO / 2; ++k)
            for (int q = 0; q < RW - 1; ++q) acc[0][k][0] = __fadd2_rn(acc[0][k][0], red[q * red_row + k * 32]);
    } else {
#pragma unroll 1
        for (int q = 0; q < RW - 1; ++q)
#pragma unroll
            for (int j = 0; j < CI; ++j)
#pragma unroll
                for (int k = 0; k < CO / 2; ++k)
#pragma unroll
                    for (int t = 0; t < T; ++t) acc[j][k][t] = __fadd2_rn(acc[j][k][t], red[q * red_row + ((j * (CO / 2) + k) * T + t) * 32]);
    }
    float* dst = a.partials + ((int64_t)s * a.n_split + split) * T * a.Cout * a.Cin + ci0 + lane;
#pragma unroll
    for (int j = 0; j < CI; ++j) {
        if (ci0 + 32 * j + lane >= a.Cin) break;
#pragma unroll
        for (int k = 0; k < CO; ++k) {
            const int co = co0 + g * CO + k;
            if (co >= a.Cout) continue;
#pragma unroll
            for (int t = 0; t < T; ++t) dst[((int64_t)t * a.Cout + co) * a.Cin + 32 * j] = k & 1 ? acc[j][k / 2][t].y : acc[j][k / 2][t].x;
        }
    }
}

// Thread groups per block, channel tiles and pixel ranges of a weight gradient: as many ranges as give every SM about
// eight warps of one stream (a warp has enough independent sums to keep its scheduler busy with two), each range at least one
// chunk.  The number of streams has no part in it: the ranges group a gradient's sums, and a stream's results must be the same
// whatever it shares the launch with.
struct WgradShape { int ng, ci_tiles, co_tiles, tiles_x, n_chunks, n_split; };
template <int KS, int CO, int CI>
WgradShape wgrad_shape(int Cin, int Cout, int h, int w)
{
    WgradShape q;
    constexpr int RW = wg_rows<KS>(), kMost = wg_most_groups<KS>();
    const int groups = (Cout + CO - 1) / CO;
    q.co_tiles = (groups + kMost - 1) / kMost;
    q.ng = (groups + q.co_tiles - 1) / q.co_tiles;
    q.co_tiles = (groups + q.ng - 1) / q.ng;
    q.ci_tiles = (Cin + 32 * CI - 1) / (32 * CI);
    q.tiles_x = (w + kTileX - 1) / kTileX;
    q.n_chunks = q.tiles_x * ((h + RW - 1) / RW);
    const int per_range = q.ci_tiles * q.co_tiles, warps = q.ng * RW;
    int n = 148 * (warps >= 5 ? 1 : 8 / warps) / per_range;
    if (n > 128) n = 128;                              // the update adds the ranges' results one by one
    const int per = n < 1 ? q.n_chunks : (q.n_chunks + n - 1) / n;      // chunks of the longest range: no more ranges than it takes
    q.n_split = (q.n_chunks + per - 1) / per;
    return q;
}
// 1x1 layers: 16 channels per warp keep the loads below the multiply-adds; a head with a handful of classes takes 4
bool narrow(int Cout) { return Cout <= 4; }
// Input channels per lane: as many as the layer fills.  With at most 16 output channels a block has one channel group, and two
// blocks per SM need both buffers of two channels per lane (88 KB); with four a block's 156 KB would leave one of four warps.
int wg_lane_channels(int Cin, int Cout) { return Cin <= 32 ? 1 : Cin <= 64 || Cout <= 16 ? 2 : 4; }
WgradShape wgrad_shape_of(int Cin, int Cout, int h, int w, int ks)
{
    if (ks == 3) return wgrad_shape<3, 8, 1>(Cin, Cout, h, w);
    if (narrow(Cout)) return wgrad_shape<1, 4, 1>(Cin, Cout, h, w);
    const int ci = wg_lane_channels(Cin, Cout);
    return ci == 1 ? wgrad_shape<1, 16, 1>(Cin, Cout, h, w) : ci == 2 ? wgrad_shape<1, 16, 2>(Cin, Cout, h, w) : wgrad_shape<1, 16, 4>(Cin, Cout, h, w);
}

template <int KS, int CO, int CI>
void launch_wgrad(const WgradF32& a, const WgradShape& q, int S, bool early, cudaStream_t s)
{
    const dim3 grid((unsigned)q.n_split, (unsigned)(q.ci_tiles * q.co_tiles), (unsigned)S);
    // (blocks in pairs on the SMs that the loss kernel left first: 1x1, 21 classes, 180 x 320 29 us back to back, spread 24)
    const size_t smem = one_per_sm(wg_smem<KS, CO, CI>(q.ng), (int64_t)q.n_split * q.ci_tiles * q.co_tiles * S, 148);
    launch_early(early, conv_wgrad_f32_kernel<KS, CO, CI>, grid, dim3(32 * wg_rows<KS>() * q.ng), smem, s, a, q.tiles_x, q.n_chunks, q.ci_tiles);
}

}  // namespace

cudaError_t prepare_conv_f32()
{
    cudaError_t e = allow_shared_memory((const void*)conv_fwd_f32_kernel<3, 8>);
    if (e == cudaSuccess) e = allow_shared_memory((const void*)conv_fwd_f32_kernel<1, 8>);
    if (e == cudaSuccess) e = allow_shared_memory((const void*)conv_fwd_f32_kernel<1, 4>);
    if (e == cudaSuccess) e = allow_shared_memory((const void*)conv_wgrad_f32_kernel<3, 8, 1>);
    if (e == cudaSuccess) e = allow_shared_memory((const void*)conv_wgrad_f32_kernel<1, 16, 1>);
    if (e == cudaSuccess) e = allow_shared_memory((const void*)conv_wgrad_f32_kernel<1, 16, 2>);
    if (e == cudaSuccess) e = allow_shared_memory((const void*)conv_wgrad_f32_kernel<1, 16, 4>);
    if (e == cudaSuccess) e = allow_shared_memory((const void*)conv_wgrad_f32_kernel<1, 4, 1>);
    return e;
}

static void launch_fwd_any(const ConvF32& a, int ks, int S, bool early, cudaStream_t s)
{
    if (ks == 3) launch_fwd<3, 8>(a, S, early, s);
    else if (narrow(a.Cout)) launch_fwd<1, 4>(a, S, early, s);
    else launch_fwd<1, 8>(a, S, early, s);
}

void launch_conv_fwd_f32(const float* in, int Cin, int h, int w, const float* Wt, const float* b, int Cout, int ks, bool relu,
                         float* out, bool out_padded, int S, int64_t w_stride, bool early, cudaStream_t s)
{
    const PadF32 pad(h, w);
    const ConvF32 a = {in, Wt, b, nullptr, out_padded ? out + pad.origin : out, Cin, Cout, h, w, relu ? 1 : 0, 0,
                       out_padded ? pad.pitch : w, out_padded ? pad.plane : (int64_t)h * w,
                       Cin * pad.plane, w_stride, w_stride, Cout * (out_padded ? pad.plane : (int64_t)h * w)};
    launch_fwd_any(a, ks, S, early, s);
}

void launch_conv1x1_dgrad_relu_f32(const float* W2, const float* dz, const float* Hact, int C, int Ch, int h, int w, float* dH, int S,
                                   int64_t w_stride, bool early, cudaStream_t s)
{
    const PadF32 pad(h, w);
    const ConvF32 a = {dz, W2, nullptr, Hact + pad.origin, dH + pad.origin, C, Ch, h, w, 0, 1, pad.pitch, pad.plane,
                       C * pad.plane, w_stride, 0, Ch * pad.plane};
    launch_fwd_any(a, 1, S, early, s);
}

int conv_wgrad_f32_splits(int Cin, int Cout, int h, int w, int ks) { return wgrad_shape_of(Cin, Cout, h, w, ks).n_split; }

void launch_conv_wgrad_f32(const float* in, const float* dout, int Cin, int Cout, int h, int w, int ks, float* partials,
                           float* b_partials, int S, bool early, cudaStream_t s)
{
    const WgradShape q = wgrad_shape_of(Cin, Cout, h, w, ks);
    const PadF32 pad(h, w);
    const WgradF32 a = {in, dout, partials, b_partials, Cin, Cout, h, w, q.n_split, Cin * pad.plane, Cout * pad.plane};
    const int ci = wg_lane_channels(Cin, Cout);
    if (ks == 3) launch_wgrad<3, 8, 1>(a, q, S, early, s);
    else if (narrow(Cout)) launch_wgrad<1, 4, 1>(a, q, S, early, s);
    else if (ci == 1) launch_wgrad<1, 16, 1>(a, q, S, early, s);
    else if (ci == 2) launch_wgrad<1, 16, 2>(a, q, S, early, s);
    else launch_wgrad<1, 16, 4>(a, q, S, early, s);
}

// between plain planes [C][h][w] and padded ones (interior only)
__global__ void __launch_bounds__(256)
pad_planes_kernel(const float* __restrict__ src, float* __restrict__ dst, int h, int w, int64_t src_plane, int src_pitch, int64_t dst_plane, int dst_pitch)
{
    pdl_wait();
    pdl_launch_dependents();
    const int x = blockIdx.x * 32 + (threadIdx.x & 31), c = blockIdx.z;
    for (int y = blockIdx.y * 32 + (threadIdx.x >> 5), n = 0; n < 4 && y < h; ++n, y += 8)
        if (x < w) dst[c * dst_plane + (int64_t)y * dst_pitch + x] = __ldg(src + c * src_plane + (int64_t)y * src_pitch + x);
}

void launch_pad_planes(const float* plain, float* padded, int C, int h, int w, cudaStream_t s)
{
    const PadF32 pad(h, w);
    launch_early(pdl_enabled(), pad_planes_kernel, dim3((unsigned)((w + 31) / 32), (unsigned)((h + 31) / 32), (unsigned)C), dim3(256), 0, s,
        plain, padded + pad.origin, h, w, (int64_t)h * w, w, pad.plane, pad.pitch);
}

void launch_unpad_planes(const float* padded, float* plain, int C, int h, int w, cudaStream_t s)
{
    const PadF32 pad(h, w);
    launch_early(pdl_enabled(), pad_planes_kernel, dim3((unsigned)((w + 31) / 32), (unsigned)((h + 31) / 32), (unsigned)C), dim3(256), 0, s,
        padded + pad.origin, plain, h, w, pad.plane, pad.pitch, (int64_t)h * w, w);
}

}  // namespace st
