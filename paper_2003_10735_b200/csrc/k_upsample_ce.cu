// K3 for more than 32 classes — ComputeLoss and the first half of PartialBackward (Algorithm 1; loss of Section 5.2),
// fused: bilinear x4 upsample of the head's low-resolution logits z to frame resolution, per-pixel softmax cross-entropy
// against the one-byte labels, and the gradient of the mean loss with respect to z (the transpose of the upsample applied
// to softmax - onehot), without ever writing a frame-resolution tensor.  Same geometry and arithmetic as the kernel for
// fewer classes (k_fwd_ce.cuh): warp = row of cells, lane = node column and the 4 x 4 frame pixels to its right,
// 16 exponentials of a class as products of four (cell_softmax.cuh), exact per-pixel maxima for cells whose logits are
// steep, integer sums for the one-hot part.
//
// What differs is where things are kept.  With up to 255 classes neither the logit tile nor the cells' pulls fit shared
// memory next to anything else, so the logits are read from global memory (coalesced rows, L1/L2 hits after the first
// sweep) and the pulls go through shared memory kChunk classes at a time.  The time of a warp is its walk over the
// classes, so the classes of a cell row are divided among two or three warps, which exchange their per-pixel
// sums once.  81 classes on 90 x 160 nodes: 95.5 us with a thread per cell and three sweeps of direct
// exponentials, 39 us now.
#include "st_internal.h"
#include "cell_softmax.cuh"

namespace st {

namespace {

constexpr int kOwnX = 30;          // node columns a block owns (lanes 1..30)
constexpr int kChunk = 8;          // classes per group whose pulls are in shared memory at a time

struct ManyShape { int own_y, groups; };
// Fifteen or sixteen warps per block, one block per SM.  4 node rows and three warps per cell row where that fills the SMs once
// at most; otherwise 7 rows and two warps, which computes fewer rows twice.  81 classes, us with 4 / with 7 rows: 96 x 160 nodes (144
// blocks of 4) 38 / 55, 100 x 160 (150) 68 / 55, 180 x 320 (495) 139 / 106; 40 classes 24 / 32, 44 / 32, 88 / 61.  The line follows the map
// alone, although a second round of 4-row blocks would do for one stream of 135 x 240 (72 / 103) and four streams of 61 x 90 would
// rather have 7 rows (71 / 55): the shape groups the sums, and a stream's results must not depend on what shares its launch.
ManyShape many_shape(int h, int w)
{
    const int blocks4 = ((h + 3) / 4) * ((w + kOwnX - 1) / kOwnX);
    return blocks4 <= 148 ? ManyShape{4, 3} : ManyShape{7, 2};
}
template <int NY, int G>
size_t many_smem(int C, bool conf)
{
    const size_t pulls = (size_t)G * (NY + 1) * kChunk * 32 * 2, sums = (size_t)G * (NY + 1) * 16 * 32;
    return ((pulls > sums ? pulls : sums) + (size_t)G * kChunk * (NY + 2) * 32 + (size_t)C * (NY + 1) + 1 +
            (conf ? (size_t)(G - 1) * (NY + 1) * 16 * 32 * 2 : 0)) * sizeof(float);
}

// One class of a steep cell, without progressions: the interpolated logit (log2 units) of the lane's pixel (r, k)
struct CellCorners { float a, b, ar, br; };
__device__ __forceinline__ CellCorners corners(const float* q, int dq)
{
    CellCorners c;
    c.a = q[0]; c.b = q[dq];
    c.ar = __shfl_down_sync(0xffffffffu, c.a, 1); c.br = __shfl_down_sync(0xffffffffu, c.b, 1);
    return c;
}
__device__ __forceinline__ float pixel_u(const CellCorners& c, int r, int k)
{
    const float ly = (2 * r + 1) * 0.125f, lx = (2 * k + 1) * 0.125f;
    const float l = fmaf(ly, c.b - c.a, c.a), rr = fmaf(ly, c.br - c.ar, c.ar);
    return fmaf(lx, rr - l, l) * kLog2e;
}

template <int NY, int G, bool CONF>
__global__ void __launch_bounds__((NY + 1) * G * 32, 1)
upsample_ce_many_kernel(UpsampleCeArgs a)
{
    constexpr int NR = NY + 1, NT = NR * G * 32, TZ_H = NY + 2;
    extern __shared__ __align__(16) float smem[];
    const int C = a.C, h = a.h, w = a.w, H = h * kUp, W = w * kUp;
    float2* pull = reinterpret_cast<float2*>(smem);              // [G][NR][kChunk][32]: a cell's pull on its upper / lower node row
    float* part = smem;                                          // [G][NR][16][32]: per-pixel sums of a group (before the pulls)
    constexpr int kPull = G * NR * kChunk * 32 * 2, kPart = G * NR * 16 * 32;
    int* corr = reinterpret_cast<int*>(smem + (kPull > kPart ? kPull : kPart));   // [G][kChunk][TZ_H][32]: -64 * (adjoint of onehot)
    float* bsum = reinterpret_cast<float*>(corr + G * kChunk * TZ_H * 32);        // [C][NR]: bias-gradient sums of the node rows
    float2* later = reinterpret_cast<float2*>(bsum + (C * NR + 1) / 2 * 2);       // CONF: [G-1][NR][16][32] largest value and its class, later groups
    __shared__ float red[NR * G], red_max[NR * G], red_change[NR * G];

    const int s = blockIdx.z, x0 = blockIdx.x * kOwnX, y0 = blockIdx.y * NY;
    const int blk = blockIdx.y * gridDim.x + blockIdx.x, n_blk = gridDim.x * gridDim.y;
    const int64_t p = (int64_t)h * w;
    const uint8_t* labels = a.labels + (int64_t)s * H * W;
    const int tid = threadIdx.x, l = tid & 31, warp = tid >> 5, wi = warp % NR, g = warp / NR;
    pdl_wait();
    if (a.skip && a.skip[(int64_t)s * a.skip_stride]) return;     // this stream's training loop has ended (block-uniform)

    const int i = y0 - 1 + wi, n = x0 - 1 + l;                    // cell row, node column
    const bool row_ok = i <= h - 1, cell_ok = row_ok && l <= 30 && n >= -1 && n <= w - 1;
    const int yt = min(max(i, 0), h - 1), yb = min(max(i + 1, 0), h - 1), xl = min(max(n, 0), w - 1), xr = min(max(n + 1, 0), w - 1);
    const bool own_cell = cell_ok && yb >= y0 && yb < y0 + NY && xr >= x0 && xr < x0 + kOwnX;
    const bool fold_l = n == -1, fold_r = n == w - 1;             // at the clamped borders the outer node column is the inner one
    const int c_lo = C * g / G, c_hi = C * (g + 1) / G;           // this warp's classes
    const float* q0 = a.z + ((int64_t)s * C + c_lo) * p + (int64_t)yt * w + xl;       // own node column, upper node row, first class
    const int dq = (yb - yt) * w;

    // labels of the lane's 16 pixels, 255 where there is none
    uint32_t lab[4];
    unsigned n_bad = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int Y = 4 * i + 2 + r;
        lab[r] = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int X = 4 * n + 2 + k;
            uint32_t v = 255;
            if (cell_ok && Y >= 0 && Y < H && X >= 0 && X < W) {
                v = __ldg(labels + (int64_t)Y * W + X);
                if (v >= (uint32_t)C) { if (own_cell && g == 0) ++n_bad; v = 255; }
            }
            lab[r] |= v << (8 * k);
        }
    }
    auto label_of = [&](int j) { return (lab[j >> 2] >> (8 * (j & 3))) & 0xffu; };

    // ---- shift of the exponentials: the largest logit of the block's nodes
    float m = -INFINITY;
#pragma unroll 8
    for (int c = c_lo; c < c_hi; ++c) { const float* q = q0 + (c - c_lo) * p; m = fmaxf(m, fmaxf(q[0], q[dq])); }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (l == 0) red_max[warp] = m;
    __syncthreads();
    m = red_max[0];
#pragma unroll
    for (int k = 1; k < NR * G; ++k) m = fmaxf(m, red_max[k]);
    const float M = m * kLog2e;

    // ---- first sweep: sums of the exponentials (and the arg-max, lowest class on ties), this group's classes
    float Z[16], best[CONF ? 16 : 1];
    uint32_t arg[CONF ? 16 : 1];
    float change = 0.f;
#pragma unroll
    for (int j = 0; j < 16; ++j) { Z[j] = 0.f; if (CONF) { best[j] = -1.f; arg[j] = 0; } }
    {
        float2 Z01[4], Z23[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) Z01[k] = Z23[k] = make_float2(0.f, 0.f);
#pragma unroll 3
        for (int c = c_lo; c < c_hi; ++c) {
            const float* q = q0 + (c - c_lo) * p;
            float2 X01[4], X23[4];
            change = fmaxf(change, cell_exponentials(q[0], q[dq], M, X01, X23));
#pragma unroll
            for (int k = 0; k < 4; ++k) { Z01[k] = __fadd2_rn(Z01[k], X01[k]); Z23[k] = __fadd2_rn(Z23[k], X23[k]); }
            if (CONF) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float e[4] = {X01[k].x, X01[k].y, X23[k].x, X23[k].y};
#pragma unroll
                    for (int r = 0; r < 4; ++r) if (e[r] > best[4 * r + k]) { best[4 * r + k] = e[r]; arg[4 * r + k] = c; }
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) { Z[k] = Z01[k].x; Z[4 + k] = Z01[k].y; Z[8 + k] = Z23[k].x; Z[12 + k] = Z23[k].y; }
    }
    if (!cell_ok) change = 0.f;                                   // lanes without a cell hold nothing that is used
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) change = fmaxf(change, __shfl_xor_sync(0xffffffffu, change, o));
    if (l == 0) red_change[warp] = change;
    // a row's groups exchange a value per pixel: the sum, or the largest, over all classes, in group order
    auto over_groups = [&](float (&v)[16], bool largest) {
        if (G == 1) return;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 16; ++j) part[((g * NR + wi) * 16 + j) * 32 + l] = v[j];
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            float t = part[(wi * 16 + j) * 32 + l];
            for (int k = 1; k < G; ++k) { const float u = part[((k * NR + wi) * 16 + j) * 32 + l]; t = largest ? fmaxf(t, u) : t + u; }
            v[j] = t;
        }
    };
    over_groups(Z, false);
    __syncthreads();
    bool bad = false;
#pragma unroll
    for (int k = 0; k < G; ++k) bad |= !(red_change[k * NR + wi] <= kFastRange / kLog2e);
#pragma unroll
    for (int j = 0; j < 16; ++j) bad |= label_of(j) != 255 && !(Z[j] > 1e-18f);
    const bool slow = __any_sync(0xffffffffu, bad) && row_ok;     // the same for all groups of a row
    float mx[16];                                                 // shift per pixel
#pragma unroll
    for (int j = 0; j < 16; ++j) mx[j] = M;
    const bool any_slow = __syncthreads_or(slow);
    if (any_slow) {
        if (slow) {
#pragma unroll
            for (int j = 0; j < 16; ++j) mx[j] = -INFINITY;
            for (int c = c_lo; c < c_hi; ++c) {
                const CellCorners k4 = corners(q0 + (c - c_lo) * p, dq);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float u = pixel_u(k4, j >> 2, j & 3);
                    if (u > mx[j]) { mx[j] = u; if (CONF) arg[j] = c; }
                }
            }
            if (CONF)
#pragma unroll
                for (int j = 0; j < 16; ++j) best[j] = mx[j];
        }
        over_groups(mx, true);
        if (slow) {
#pragma unroll
            for (int j = 0; j < 16; ++j) Z[j] = 0.f;
            for (int c = c_lo; c < c_hi; ++c) {
                const CellCorners k4 = corners(q0 + (c - c_lo) * p, dq);
#pragma unroll
                for (int j = 0; j < 16; ++j) Z[j] += ex2_approx(pixel_u(k4, j >> 2, j & 3) - mx[j]);
            }
        } else if (g > 0) {
#pragma unroll
            for (int j = 0; j < 16; ++j) Z[j] = 0.f;              // already complete: group 0 alone carries it through the exchange
        }
        over_groups(Z, false);
        __syncthreads();
    }
    if (CONF) {                                                   // student's class: the largest over the groups, the first one on ties
        if (G > 1) {
            if (g > 0)
#pragma unroll
                for (int j = 0; j < 16; ++j) later[(((g - 1) * NR + wi) * 16 + j) * 32 + l] = make_float2(best[j], __uint_as_float(arg[j]));
            __syncthreads();
            if (g == 0)
                for (int k = 0; k < G - 1; ++k)
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float2 o = later[((k * NR + wi) * 16 + j) * 32 + l];
                        if (o.x > best[j]) { best[j] = o.x; arg[j] = __float_as_uint(o.y); }
                    }
        }
        if (g == 0 && own_cell) {                                 // one count per distinct (label, class) pair of the cell
            unsigned long long* conf = a.conf + (int64_t)s * a.conf_stream_stride;
            uint32_t left = 0;
#pragma unroll
            for (int j = 0; j < 16; ++j) left |= label_of(j) != 255 ? 1u << j : 0u;
            while (left) {
                const int first = __ffs(left) - 1;
                uint32_t key = 0, same = 0;
#pragma unroll
                for (int j = 0; j < 16; ++j) if (j == first) key = label_of(j) * C + arg[j];
#pragma unroll
                for (int j = 0; j < 16; ++j) if (((left >> j) & 1u) && label_of(j) * C + arg[j] == key) same |= 1u << j;
                atomicAdd(conf + key, (unsigned long long)__popc(same));
                left &= ~same;
            }
        }
    }

    // ---- loss: log Z + shift - label's logit, once per pixel (the block that owns the cell, group 0); 1/Z as adjoint weights
    float loss = 0.f;
    float wl[16], wr[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const bool ok = label_of(j) != 255;
        if (ok && own_cell && g == 0) {
            const float* q = a.z + (int64_t)s * C * p + (int64_t)label_of(j) * p + (int64_t)yt * w;
            const float ly = (2 * (j >> 2) + 1) * 0.125f, lx = (2 * (j & 3) + 1) * 0.125f;
            const float vl = fmaf(ly, q[xl + dq] - q[xl], q[xl]), vr = fmaf(ly, q[xr + dq] - q[xr], q[xr]);
            loss += (__log2f(Z[j]) - (fmaf(lx, vr - vl, vl) * kLog2e - mx[j])) * kLn2;
        }
        const float rz = ok ? 1.0f / Z[j] : 0.f, fr = (2 * (j & 3) + 1) * 0.125f;
        wl[j] = (fold_l ? 0.f : (fold_r ? 1.0f : 1.0f - fr)) * rz;
        wr[j] = (fold_r ? 0.f : (fold_l ? 1.0f : fr)) * rz;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (l == 0) red[warp] = loss;
    if (n_bad) atomicAdd(a.bad, n_bad);

    // ---- second sweep, kChunk classes of every group at a time: the cells' pulls on their node rows, then the nodes' sums
    float tw[4], bw[4];                                           // row weights toward the upper / lower node row
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float ly = (2 * r + 1) * 0.125f;
        tw[r] = i == -1 ? 0.f : (i == h - 1 ? 1.0f : 1.0f - ly);
        bw[r] = i == h - 1 ? 0.f : (i == -1 ? 1.0f : ly);
    }
    float2 WL01[4], WL23[4], WR01[4], WR23[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        WL01[k] = make_float2(wl[k], wl[4 + k]); WL23[k] = make_float2(wl[8 + k], wl[12 + k]);
        WR01[k] = make_float2(wr[k], wr[4 + k]); WR23[k] = make_float2(wr[8 + k], wr[12 + k]);
    }
    const float2 tw01 = make_float2(tw[0], tw[1]), tw23 = make_float2(tw[2], tw[3]);
    const float2 bw01 = make_float2(bw[0], bw[1]), bw23 = make_float2(bw[2], bw[3]);
    const float invP = 1.0f / ((float)H * (float)W);
    const bool node_ok = wi >= 1 && i < h && l >= 1 && l <= kOwnX && n < w;
    const int n_chunks = ((C + G - 1) / G + kChunk - 1) / kChunk;  // of the group with most classes
    int* my_corr = corr + g * kChunk * TZ_H * 32;
    float2* my_pull = pull + (g * NR + wi) * kChunk * 32 + l;
    for (int e = tid; e < G * kChunk * TZ_H * 32; e += NT) corr[e] = 0;
    __syncthreads();                                              // `part` is dead, corr is clear
    for (int chunk = 0; chunk < n_chunks; ++chunk) {
        const int c0 = c_lo + chunk * kChunk, c1 = min(c0 + kChunk, c_hi);
        if (row_ok) {
#pragma unroll 2
            for (int c = c0; c < c1; ++c) {
                const float* q = q0 + (c - c_lo) * p;
                float2 L01, L23, R01, R23;
                if (!slow) {
                    float2 x01, x23, q01, q23;
                    cell_bases(q[0], q[dq], M, x01, x23, q01, q23);
                    cell_row_sums(x01, x23, q01, q23, WL01, WL23, L01, L23);
                    cell_row_sums(x01, x23, q01, q23, WR01, WR23, R01, R23);
                } else {
                    const CellCorners k4 = corners(q, dq);
                    float sl[4], sr[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        sl[r] = sr[r] = 0.f;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const float e = ex2_approx(pixel_u(k4, r, k) - mx[4 * r + k]);
                            sl[r] = fmaf(wl[4 * r + k], e, sl[r]); sr[r] = fmaf(wr[4 * r + k], e, sr[r]);
                        }
                    }
                    L01 = make_float2(sl[0], sl[1]); L23 = make_float2(sl[2], sl[3]);
                    R01 = make_float2(sr[0], sr[1]); R23 = make_float2(sr[2], sr[3]);
                }
                if (!cell_ok) R01 = R23 = L01 = L23 = make_float2(0.f, 0.f);
                const float2 h01 = __fadd2_rn(L01, make_float2(__shfl_up_sync(0xffffffffu, R01.x, 1), __shfl_up_sync(0xffffffffu, R01.y, 1)));
                const float2 h23 = __fadd2_rn(L23, make_float2(__shfl_up_sync(0xffffffffu, R23.x, 1), __shfl_up_sync(0xffffffffu, R23.y, 1)));
                const float2 t2 = __ffma2_rn(h23, tw23, __fmul2_rn(h01, tw01)), b2 = __ffma2_rn(h23, bw23, __fmul2_rn(h01, bw01));
                my_pull[(c - c0) * 32] = make_float2(t2.x + t2.y, b2.x + b2.y);
            }
            // the one-hot part of the pixels whose label is one of these classes, exact in units of 1/64: one round per
            // distinct label of the cell, its pixels' corner weights (row eighths x column eighths) by byte-wise dot products
            uint32_t rem[4];
#pragma unroll
            for (int r = 0; r < 4; ++r)
                rem[r] = __vcmpgeu4(lab[r], (uint32_t)c0 * 0x01010101u) & ~__vcmpgeu4(lab[r], (uint32_t)c1 * 0x01010101u) & 0x01010101u;
            while (rem[0] | rem[1] | rem[2] | rem[3]) {
                const uint32_t wsel = rem[0] ? lab[0] : rem[1] ? lab[1] : rem[2] ? lab[2] : lab[3];
                const uint32_t rsel = rem[0] ? rem[0] : rem[1] ? rem[1] : rem[2] ? rem[2] : rem[3];
                const uint32_t cur = (wsel >> (__ffs(rsel) - 1)) & 0xffu;
                uint32_t tl = 0, tr = 0, bl = 0, br = 0;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint32_t eq = __vcmpeq4(lab[r], cur * 0x01010101u) & rem[r];
                    rem[r] ^= eq;
                    tl = __dp4a(eq, corner_weights(7 - 2 * r, false), tl);
                    tr = __dp4a(eq, corner_weights(7 - 2 * r, true), tr);
                    bl = __dp4a(eq, corner_weights(2 * r + 1, false), bl);
                    br = __dp4a(eq, corner_weights(2 * r + 1, true), br);
                }
                int* cc = my_corr + ((int)cur - c0) * TZ_H * 32 - (y0 - 1) * 32 - (x0 - 1);
                atomicAdd(cc + yt * 32 + xl, -(int)tl);
                atomicAdd(cc + yt * 32 + xr, -(int)tr);
                atomicAdd(cc + yb * 32 + xl, -(int)bl);
                atomicAdd(cc + yb * 32 + xr, -(int)br);
            }
        }
        __syncthreads();
        if (wi >= 1) {                                            // node row i = y0 - 1 + wi: own upper part + lower part of the row above + one-hot part
            for (int c = c0; c < c1; ++c) {
                int* cr = my_corr + (c - c0) * TZ_H * 32 + wi * 32 + l;
                float v = 0.f;
                if (node_ok) {
                    v = (my_pull[(c - c0) * 32].x + my_pull[(c - c0 - kChunk) * 32].y + (float)*cr * (1.0f / 64.0f)) * invP;
                    a.dz[((int64_t)s * C + c) * a.dz_plane + (int64_t)i * a.dz_pitch + n] = v;
                }
                *cr = 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (l == 0) bsum[c * NR + wi] = v;
            }
        } else {                                                  // node rows outside the block's own: nobody reads them
            for (int c = c0; c < c1; ++c) {
                my_corr[(c - c0) * TZ_H * 32 + l] = 0;
                my_corr[(c - c0) * TZ_H * 32 + (TZ_H - 1) * 32 + l] = 0;
            }
        }
        __syncthreads();
    }
    pdl_launch_dependents();
    for (int c = tid; c < C; c += NT) {
        float t = 0.f;
        for (int k = 1; k < NR; ++k) t += bsum[c * NR + k];
        a.db_part[((int64_t)s * n_blk + blk) * C + c] = t;
    }
    if (tid == 0) {
        float t = 0.f;
        for (int k = 0; k < NR; ++k) t += red[k];                  // group 0's warps
        a.loss_part[(int64_t)s * n_blk + blk] = t;
    }
}

template <int NY, int G>
cudaError_t allow_many()
{
    const cudaError_t e = allow_shared_memory((const void*)upsample_ce_many_kernel<NY, G, false>);
    return e != cudaSuccess ? e : allow_shared_memory((const void*)upsample_ce_many_kernel<NY, G, true>);
}

template <int NY, int G>
void launch_many(const UpsampleCeArgs& a, cudaStream_t s)
{
    const dim3 grid((unsigned)((a.w + kOwnX - 1) / kOwnX), (unsigned)((a.h + NY - 1) / NY), (unsigned)a.S), block((NY + 1) * G * 32);
    const bool early = a.chain_early != 0;
    if (a.conf) launch_early(early, upsample_ce_many_kernel<NY, G, true>, grid, block, many_smem<NY, G>(a.C, true), s, a);
    else launch_early(early, upsample_ce_many_kernel<NY, G, false>, grid, block, many_smem<NY, G>(a.C, false), s, a);
}

}  // namespace

int upsample_ce_blocks(int h, int w, int C)
{
    if (upsample_ce_few_supported(C)) return upsample_ce_few_blocks(h, w);
    const int ny = many_shape(h, w).own_y;
    return ((h + ny - 1) / ny) * ((w + kOwnX - 1) / kOwnX);
}

cudaError_t prepare_upsample_ce(int C, bool own_forward, bool with_gradient, int tiles, int n_sms)
{
    if (upsample_ce_few_supported(C)) return prepare_fwd_ce(C, own_forward, with_gradient, tiles, n_sms);
    const cudaError_t e = allow_many<7, 2>();
    return e != cudaSuccess ? e : allow_many<4, 3>();
}

void launch_upsample_ce(const UpsampleCeArgs& a, cudaStream_t s)
{
    if (upsample_ce_few_supported(a.C)) { launch_upsample_ce_few(a, s); return; }
    if (many_shape(a.h, a.w).own_y == 7) launch_many<7, 2>(a, s);
    else launch_many<4, 3>(a, s);
}

}  // namespace st
