// K5 — OptimStep of Algorithm 1 ("most simply gradient descent", Section 4.1.4) with heavy-ball
// momentum:  v <- mu*v + g ;  theta <- theta - lr*v   (mu = 0: plain gradient descent),
// on the fp32 master parameters; the bf16 copies read by the tensor-core GEMMs are refreshed in
// the same pass.  The kernel also finishes the reductions the step left open, always in a fixed
// order so that results are bit-reproducible: split-K partial sums of the weight gradients,
// per-block partial sums of the bias gradients, and the per-block loss partials.
// K7 — UpdatedPart(student) (Algorithm 3): the packed fp32 buffer of all trainable tensors.
#include "st_internal.h"
#include "miou.cuh"
#include "train_ctl.cuh"

#include <cstdlib>

namespace st {

bool pdl_enabled()
{
    static const bool on = [] { const char* e = getenv("ST_PDL"); return !(e && e[0] == '0'); }();
    return on;
}

constexpr int kUpdThreads = 256;
// how a layer is streamed (LayerUpdate::streamed): 1 or 4 weights to a thread, or the sums of its partials in vectors by 8 to 64 lanes
constexpr int kVec8 = 8, kVec16 = 16, kVec32 = 32, kVec64 = 64;
static_assert(kUpdThreads == kMiouFetchThreads, "the update fetches the confusion matrix with all of its threads");

// bf16 copies of weight element e (internal order [tap][cout][cin]) of a layer: the one the forward and the weight
// gradient read, and, for a 3x3 layer whose gradient is passed back, the mirrored and transposed one
__device__ __forceinline__ void write_shadows(const LayerUpdate& ly, int s, int64_t e, float value)
{
    const bf16 v = __float2bfloat16_rn(value);
    if (ly.shadow) ly.shadow[(int64_t)s * ly.shadow_stream_stride + e] = v;
    if (ly.shadow_t) {
        const int ci = (int)(e % ly.cin);
        if (ci < ly.c_take) {
            const int64_t r = e / ly.cin;
            const int co = (int)(r % ly.cout), tap = (int)(r / ly.cout);
            ly.shadow_t[(int64_t)s * ly.shadow_t_stream_stride + ((int64_t)(ly.taps - 1 - tap) * ly.c_take + ci) * ly.cout + co] = v;
        }
    }
}

// Bias corrections of Adam's step t, t = steps taken before this call + position in the call: the learning rate over 1 - b1^t, and the
// reciprocal of 1 - b2^t.  The same for all parameters of a stream: one warp of a block works them out while the others' loads are on their
// way (two exponentials per thread and two of a parameter's three divisions in double: 2.9 of 126 us a step with 331776 weights).
struct AdamCorr { double lr1, r2; };
template <bool ADAM>
__device__ __forceinline__ void adam_corrections(const UpdateArgs& a, int s, AdamCorr& shared)
{
    if (ADAM && threadIdx.x < 32) {
        const double t = (double)(a.step_base[s] + a.loss_slot + 1);
        const double lr1 = (double)a.lr / (1.0 - exp(t * a.ln_b1)), r2 = 1.0 / (1.0 - exp(t * a.ln_b2));
        if (threadIdx.x == 0) { shared.lr1 = lr1; shared.r2 = r2; }
    }
}

// OptimStep on one parameter.  Gradient descent with momentum: v <- mu v + g; theta <- theta - lr v.
// Adam (each element in double, stored as fp32): m <- b1 m + (1 - b1) g; v <- b2 v + (1 - b2) g^2;
// theta <- theta - lr (m / c1) / (sqrt(v / c2) + eps).
// The state of one parameter (value, momentum or first moment, second moment), which the gradient kernels before the
// update never write: it can be fetched before their results are waited for.
struct ParamState { float theta, vel, vel2; };
template <bool ADAM>
__device__ __forceinline__ ParamState load_state(const UpdateArgs& a, int64_t gi)
{
    ParamState p;
    p.theta = a.theta[gi]; p.vel = a.vel[gi]; p.vel2 = ADAM ? a.vel2[gi] : 0.f;
    return p;
}

template <bool ADAM>
__device__ __forceinline__ float updated(const UpdateArgs& a, float g, const AdamCorr& k, const ParamState& p, float& vel, float& vel2)
{
    if (ADAM) {
        const double gd = (double)g;
        const double m = a.b1 * (double)p.vel + (1.0 - a.b1) * gd;
        const double v = a.b2 * (double)p.vel2 + (1.0 - a.b2) * gd * gd;
        vel = (float)m; vel2 = (float)v;
        return (float)((double)p.theta - k.lr1 * m / (sqrt(v * k.r2) + a.eps));
    }
    vel = fmaf(a.mu, p.vel, g); vel2 = 0.f;
    return fmaf(-a.lr, vel, p.theta);
}
template <bool ADAM>
__device__ __forceinline__ float apply_update(const UpdateArgs& a, int64_t gi, float g, const AdamCorr& k, const ParamState& p)
{
    float vel, vel2;
    const float t = updated<ADAM>(a, g, k, p, vel, vel2);
    a.grad[gi] = g; a.vel[gi] = vel; a.theta[gi] = t;
    if (ADAM) a.vel2[gi] = vel2;
    return t;
}
template <bool ADAM>
__device__ __forceinline__ float apply_update(const UpdateArgs& a, int64_t gi, float g, const AdamCorr& k)
{
    return apply_update<ADAM>(a, gi, g, k, load_state<ADAM>(a, gi));
}

// Train, for a block that streams: does this prediction go on to the step (skip), was it the best so far.  With DECIDES a warp of its own finds
// out; `verdict` holds the answer behind the block's next barrier.  false: the thread has nothing more to do.  (The grouped part's
// first block writes the history.)
template <bool DECIDES>
__device__ __forceinline__ bool stream_control(const UpdateArgs& a, int s, const TrainHistory& hist, int& verdict, bool& skip, bool& better)
{
    skip = a.skip && a.skip[(int64_t)s * a.skip_stride]; better = false;
    if (DECIDES) {
        if (hist.ended) return false;
        if (threadIdx.x >= kUpdThreads) {
            train_decision_warp(a.ctl, s, false, hist, skip, better);
            if ((threadIdx.x & 31) == 0) verdict = (skip ? 1 : 0) | (better ? 2 : 0);
            __syncthreads();
            return false;
        }
        return true;
    }
    if (a.has_ctl == 1) { const MiouFetch f = train_fetch(a.ctl, s, hist); train_decision(a.ctl, s, false, hist, &f, skip, better); }
    else if (a.has_ctl && hist.ended) skip = true;
    else if (a.has_ctl) train_outcome(a.ctl, s, skip, better);
    return !skip || better;
}

// A layer of fewer weights.  A block takes 4 LANES consecutive weights: its thread groups of LANES read every
// G-th partial sum as vectors, `B` of them in flight, the group sums are added in group order, and then a thread takes the step for one weight.
// A thread per weight and group with scalar loads (the grouped part below) read twelve streams of 23 times 36864 weights at 1 TB/s.
template <int LANES, int B, bool ADAM, bool DECIDES>
__device__ __forceinline__ void update_vectors(const UpdateArgs& a, const LayerUpdate& ly, int s, int block, const AdamCorr& corr, int& verdict, float4 (&part)[kUpdThreads])
{
    constexpr int G = kUpdThreads / LANES, W = 4 * LANES;
    const int64_t nw = (int64_t)ly.cout * ly.cin * ly.taps, e = (int64_t)block * W + threadIdx.x, gi = (int64_t)s * a.n_params + ly.w_off + e;
    const bool mine = threadIdx.x < W && e < nw;
    ParamState state{};
    if (mine) state = load_state<ADAM>(a, gi);
    const TrainHistory hist = a.has_ctl ? train_history(a.ctl, s) : TrainHistory{};
    pdl_wait();
    pdl_launch_dependents();
    bool skip, better;
    if (!stream_control<DECIDES>(a, s, hist, verdict, skip, better)) return;
    const int lane = threadIdx.x % LANES;
    const int64_t v = (int64_t)block * W + 4 * lane;
    const float* src = ly.w_partials + (int64_t)s * ly.w_stream_stride + v;
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k0 = threadIdx.x / LANES; k0 < ly.n_split; k0 += B * G) {
        float4 t[B];
#pragma unroll
        for (int j = 0; j < B; ++j)
            t[j] = k0 + j * G < ly.n_split && v < nw ? __ldg(reinterpret_cast<const float4*>(src + (int64_t)(k0 + j * G) * ly.w_split_stride)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < B; ++j) { sum.x += t[j].x; sum.y += t[j].y; sum.z += t[j].z; sum.w += t[j].w; }
    }
    part[threadIdx.x] = sum;
    __syncthreads();
    if (DECIDES) { skip = (verdict & 1) != 0; better = (verdict & 2) != 0; }
    if (!mine || (skip && !better)) return;
    const float* sums = reinterpret_cast<const float*>(part);
    float g = 0.f;
#pragma unroll
    for (int k = 0; k < G; ++k) g += sums[k * W + threadIdx.x];
    if (better) a.ctl.best_theta[gi] = state.theta;
    if (!skip) write_shadows(ly, s, e, apply_update<ADAM>(a, gi, g, corr, state));
}

// weights of a block that streams a layer, by LayerUpdate::streamed
__host__ __device__ constexpr int streamed_per_block(int code) { return code >= kVec8 ? 4 * code : kUpdThreads * code; }

// A large weight tensor with a moderate number of split-K partials (a 3x3 layer): a pure stream.  Each thread owns VEC
// consecutive weights and reads them from every partial with all loads in flight.
template <int VEC, bool ADAM, bool DECIDES>
__device__ __forceinline__ void update_stream(const UpdateArgs& a, const LayerUpdate& ly, int s, int block, const AdamCorr& corr, int& verdict)
{
    pdl_wait();
    pdl_launch_dependents();
    bool skip, better;
    if (!stream_control<DECIDES>(a, s, a.has_ctl ? train_history(a.ctl, s) : TrainHistory{}, verdict, skip, better)) return;
    const int64_t nw = (int64_t)ly.cout * ly.cin * ly.taps;
    const int64_t mine = ((int64_t)block * kUpdThreads + threadIdx.x) * VEC, e = mine < nw ? mine : 0;    // (behind the end: loads for nothing)
    const float* src = ly.w_partials + (int64_t)s * ly.w_stream_stride + e;
    const int64_t gi = (int64_t)s * a.n_params + ly.w_off + e;
    const bool vec = VEC == 4 && (gi & 3) == 0;                        // the parameters as whole vectors too
    ParamState state[VEC];
    if (vec) {
        const float4 t = *reinterpret_cast<const float4*>(a.theta + gi), v = *reinterpret_cast<const float4*>(a.vel + gi);
        const float4 v2 = ADAM ? *reinterpret_cast<const float4*>(a.vel2 + gi) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float tt[4] = {t.x, t.y, t.z, t.w}, vv[4] = {v.x, v.y, v.z, v.w}, ww[4] = {v2.x, v2.y, v2.z, v2.w};
#pragma unroll
        for (int j = 0; j < VEC; ++j) { state[j].theta = tt[j % 4]; state[j].vel = vv[j % 4]; state[j].vel2 = ww[j % 4]; }
    } else {
#pragma unroll
        for (int j = 0; j < VEC; ++j) state[j] = load_state<ADAM>(a, gi + j);
    }
    float g[VEC];
#pragma unroll
    for (int j = 0; j < VEC; ++j) g[j] = 0.f;
    for (int k0 = 0; k0 < ly.n_split; k0 += 8) {
        if (VEC == 4) {
            float4 t[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                t[j] = k0 + j < ly.n_split ? __ldg(reinterpret_cast<const float4*>(src + (int64_t)(k0 + j) * ly.w_split_stride))
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 8; ++j) { g[0] += t[j].x; g[1 % VEC] += t[j].y; g[2 % VEC] += t[j].z; g[3 % VEC] += t[j].w; }
        } else {
            float t[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) t[j] = k0 + j < ly.n_split ? __ldg(src + (int64_t)(k0 + j) * ly.w_split_stride) : 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) g[0] += t[j];
        }
    }
    if (ADAM || DECIDES) __syncthreads();                              // `corr` and `verdict` are there
    if (DECIDES) { skip = (verdict & 1) != 0; better = (verdict & 2) != 0; }
    if (mine >= nw || (skip && !better)) return;
    if (!vec || skip) {
#pragma unroll
        for (int j = 0; j < VEC; ++j) {
            if (better) a.ctl.best_theta[gi + j] = state[j].theta;
            if (!skip) write_shadows(ly, s, e + j, apply_update<ADAM>(a, gi + j, g[j], corr, state[j]));
        }
        return;
    }
    if (better) *reinterpret_cast<float4*>(a.ctl.best_theta + gi) = make_float4(state[0].theta, state[1 % VEC].theta, state[2 % VEC].theta, state[3 % VEC].theta);
    float t[4], v[4], v2[4];
#pragma unroll
    for (int j = 0; j < VEC; ++j) t[j % 4] = updated<ADAM>(a, g[j], corr, state[j], v[j % 4], v2[j % 4]);
    *reinterpret_cast<float4*>(a.theta + gi) = make_float4(t[0], t[1], t[2], t[3]);
    *reinterpret_cast<float4*>(a.vel + gi) = make_float4(v[0], v[1], v[2], v[3]);
    if (ADAM) *reinterpret_cast<float4*>(a.vel2 + gi) = make_float4(v2[0], v2[1], v2[2], v2[3]);
    *reinterpret_cast<float4*>(a.grad + gi) = make_float4(g[0], g[1 % VEC], g[2 % VEC], g[3 % VEC]);
    if (ly.shadow && !ly.shadow_t) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(t[0], t[1]), hi = __floats2bfloat162_rn(t[2], t[3]);
        *reinterpret_cast<uint2*>(ly.shadow + (int64_t)s * ly.shadow_stream_stride + e) =
            make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    } else {
#pragma unroll
        for (int j = 0; j < VEC; ++j) write_shadows(ly, s, e + j, t[j % 4]);
    }
}

// Parameter blocks: a block covers kUpdThreads / G consecutive parameters; the G thread groups of a
// block each sum every G-th split-K partial of "their" parameter (coalesced along the parameters),
// the group sums are added in group order through shared memory, and group 0 applies the update.
// `B` of its loads are in flight at a time.  With DECIDES (Train) a block has one warp more, which assesses the prediction meanwhile.
template <int G, int E, int B, bool ADAM, bool DECIDES, bool VECS>
__global__ void __launch_bounds__(kUpdThreads + (DECIDES ? 32 : 0))
sgd_update_kernel(UpdateArgs a, int n_param_blocks, int n_grouped)
{
    constexpr int kRow = kUpdThreads / G;      // consecutive parameters covered by one thread group
    constexpr int kPer = kRow * E;             // parameters per block
    __shared__ float part[G][kPer];
    __shared__ int verdict;
    __shared__ AdamCorr corr;
    const int s = blockIdx.y;
    const int64_t base = (int64_t)s * a.n_params;
    adam_corrections<ADAM>(a, s, corr);                  // (the step count was written by an earlier call's last kernel)
    if ((int)blockIdx.x >= n_grouped) {                  // the streamed layers' blocks lie behind the grouped ones
        int block = (int)blockIdx.x - n_grouped;
        for (int L = 0; L < a.n_layers; ++L) {
            const LayerUpdate& ly = a.layer[L];
            if (!ly.streamed) continue;
            const int per = streamed_per_block(ly.streamed);
            const int blocks = (int)(((int64_t)ly.cout * ly.cin * ly.taps + per - 1) / per);
            if (block >= blocks) { block -= blocks; continue; }
            if constexpr (VECS) {
                __shared__ float4 vec_part[kUpdThreads];
                if (ly.streamed == kVec8) update_vectors<8, 10, ADAM, DECIDES>(a, ly, s, block, corr, verdict, vec_part);
                else if (ly.streamed == kVec16) update_vectors<16, 10, ADAM, DECIDES>(a, ly, s, block, corr, verdict, vec_part);
                else if (ly.streamed == kVec32) update_vectors<32, 10, ADAM, DECIDES>(a, ly, s, block, corr, verdict, vec_part);
                else update_vectors<64, 8, ADAM, DECIDES>(a, ly, s, block, corr, verdict, vec_part);
            } else {
                if (ly.streamed == 4) update_stream<4, ADAM, DECIDES>(a, ly, s, block, corr, verdict);
                else update_stream<1, ADAM, DECIDES>(a, ly, s, block, corr, verdict);
            }
            return;
        }
        return;
    }
    const bool param_block = (int)blockIdx.x < n_param_blocks;
    const int col = threadIdx.x % kRow, g = threadIdx.x / kRow;
    int layer[E];
    int64_t param[E];                          // index in one stream's parameters
    ParamState state[E];
    // which parameters this thread looks after (weights of the layers that are not streamed, one layer behind the other), and
    // (first thread group) their current state: none of it comes from the kernels just before this one, so it is done before
    // their completion is waited for
    if (param_block) {
#pragma unroll
        for (int e = 0; e < E; ++e) {
            int64_t i = (int64_t)blockIdx.x * kPer + e * kRow + col;
            layer[e] = -1; param[e] = 0;
            state[e].theta = state[e].vel = state[e].vel2 = 0.f;
            for (int L = 0; L < a.n_layers && layer[e] < 0; ++L) {
                const LayerUpdate& ly = a.layer[L];
                if (ly.streamed) continue;
                const int64_t nw = (int64_t)ly.cout * ly.cin * ly.taps;
                if (i < nw) { layer[e] = L; param[e] = ly.w_off + i; }
                else i -= nw;
            }
            if (g == 0 && layer[e] >= 0) state[e] = load_state<ADAM>(a, base + param[e]);
        }
    }
    TrainHistory hist{};
    if (a.has_ctl) hist = train_history(a.ctl, s);
    pdl_wait();
    pdl_launch_dependents();
    if (DECIDES) {
        if (hist.ended && blockIdx.x != 0 && param_block) return;
        if (threadIdx.x >= kUpdThreads) {
            bool stop, best;
            train_decision_warp(a.ctl, s, blockIdx.x == 0, hist, stop, best);
            if ((threadIdx.x & 31) == 0) verdict = (stop ? 1 : 0) | (best ? 2 : 0);
            __syncthreads();
            return;
        }
    }
    bool skip = a.skip && a.skip[(int64_t)s * a.skip_stride];   // block-uniform
    bool better = false;                                         // Train: this prediction is the best so far
    MiouFetch fetched{};
    const bool decide_here = a.has_ctl == 1 && !DECIDES;                     // 2: the backward before this kernel has assessed the prediction
    if (decide_here) fetched = train_fetch(a.ctl, s, hist);      // on their way while the partial sums are fetched and added
    if (a.has_ctl == 2 && !hist.ended) train_outcome(a.ctl, s, skip, better);
    float* best_theta = a.has_ctl ? a.ctl.best_theta : nullptr;
    if (param_block) {
        if (a.has_ctl && hist.ended) {                  // nothing to assess, nothing to update: the history goes on
            if (DECIDES) __syncthreads();
            if (decide_here) train_decision(a.ctl, s, blockIdx.x == 0, hist, &fetched, skip, better);
            return;
        }
        if (skip && !decide_here && !DECIDES && !better) return;
        float sum[E];
        // E parameters per thread, all of their split-K loads issued before any is consumed
#pragma unroll
        for (int e = 0; e < E; ++e) {
            sum[e] = 0.f;
            if (layer[e] >= 0) {
                const LayerUpdate& ly = a.layer[layer[e]];
                const float* src = ly.w_partials + (int64_t)s * ly.w_stream_stride + (param[e] - ly.w_off);
                // batches of predicated loads: all in flight together, no one-at-a-time remainder loop
                float t = 0.f;
                for (int k0 = g; k0 < ly.n_split; k0 += B * G) {
                    float v[B];
#pragma unroll
                    for (int j = 0; j < B; ++j) {
                        const int k = k0 + j * G;
                        v[j] = k < ly.n_split ? __ldg(src + (int64_t)k * ly.w_split_stride) : 0.f;
                    }
#pragma unroll
                    for (int j = 0; j < B; ++j) t += v[j];
                }
                sum[e] = t;
            }
        }
#pragma unroll
        for (int e = 0; e < E; ++e) part[g][e * kRow + col] = sum[e];
        if (decide_here) train_decision(a.ctl, s, blockIdx.x == 0, hist, &fetched, skip, better);
        __syncthreads();
        if (DECIDES) { skip = (verdict & 1) != 0; better = (verdict & 2) != 0; }
        if (g != 0 || (skip && !better)) return;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            if (layer[e] < 0) continue;
            const int64_t i = param[e];
            const LayerUpdate& ly = a.layer[layer[e]];
            float gr = 0.f;
#pragma unroll
            for (int k = 0; k < G; ++k) gr += part[k][e * kRow + col];
            if (better) best_theta[base + i] = state[e].theta;
            if (!skip) write_shadows(ly, s, i - ly.w_off, apply_update<ADAM>(a, base + i, gr, corr, state[e]));
        }
        return;
    }
    // ---- reduction warps: one warp per bias element that has partial sums, plus one for the loss
    if (decide_here) train_decision(a.ctl, s, blockIdx.x == 0, hist, &fetched, skip, better);
    else if (a.has_ctl && hist.ended) skip = true;
    const int warp = ((int)blockIdx.x - n_param_blocks) * (kUpdThreads / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    int item = warp, of = -1;                            // of: the layer whose bias element `item` is
    for (int L = 0; L < a.n_layers && of < 0; ++L) {
        if (item < a.layer[L].cout) of = L;
        else item -= a.layer[L].cout;
    }
    float g_bias = 0.f;
    if (of >= 0) {
        const LayerUpdate& ly = a.layer[of];
        const float* src = ly.b_partials + (int64_t)s * ly.n_bpart * ly.cout + item;
        for (int k0 = lane; k0 < ly.n_bpart; k0 += 8 * 32) {
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int k = k0 + j * 32;
                v[j] = k < ly.n_bpart ? __ldg(src + (int64_t)k * ly.cout) : 0.f;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) g_bias += v[j];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) g_bias += __shfl_xor_sync(0xffffffffu, g_bias, o);
    }
    if (DECIDES || ADAM) __syncthreads();
    if (DECIDES) {
        skip = (verdict & 1) != 0; better = (verdict & 2) != 0;
    }
    if (of >= 0) {
        const int64_t at = base + a.layer[of].b_off + item;
        if (lane == 0) {
            if (better) best_theta[at] = a.theta[at];
            if (!skip) apply_update<ADAM>(a, at, g_bias, corr);
        }
        return;
    }
    if (item == 0 && a.loss_part) {
        double t = 0.0;
        for (int k0 = lane; k0 < a.n_loss_part; k0 += 8 * 32) {
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int k = k0 + j * 32;
                v[j] = k < a.n_loss_part ? __ldg(a.loss_part + (int64_t)s * a.n_loss_part + k) : 0.f;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) t += (double)v[j];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) {
            if (a.loss_slot >= 0 && a.loss_slot < kMaxSteps) {
                a.loss_buf[(int64_t)s * kMaxSteps + a.loss_slot] = (float)(t * a.inv_P);
            }
        }
    }
}

template <bool ADAM>
static int launch_sgd_update_t(const UpdateArgs& a, cudaStream_t s)
{
    // Large layers are streamed, everything else (small layers, biases, loss) goes through the grouped part.  One launch: the
    // grouped part is all latency and hides behind the stream (256 -> 256 channels, 3x3: 19.9 us as two launches, 14.3 us as one, launch gap included).
    // Heads of small layers only: the partial sums are read as vectors, shared among the thread groups of a block so that a thread's are one
    // batch of loads: by 32 groups of 8 lanes, 16 of 16, 8 of 32 or 4 of 64.  us a step, a thread per weight and group / so: 5376 weights and 286 partial
    // sums 26.1 / 25.1, sixteen streams 286.5 / 278.5; 36864 weights and 23 partial sums 35.8 / 29.9, 65 partial sums 48.2 / 43.1, twelve streams of 7 79.4 / 53.2;
    // 73728 and 23 33.7 / 32.5.  From 110592 weights on no gain over a thread's whole vectors, next to which the small layers hide.
    UpdateArgs g = a;
    int64_t stream_blocks = 0, n_rest = 0;
    auto vectors = [&](const LayerUpdate& ly) {
        return (int64_t)ly.cout * ly.cin * ly.taps % 4 == 0 && ly.w_split_stride % 4 == 0 && ly.w_stream_stride % 4 == 0 && ((uintptr_t)ly.w_partials % 16 == 0);
    };
    bool vecs = true;
    for (int L = 0; L < a.n_layers; ++L) vecs = vecs && vectors(a.layer[L]) && a.layer[L].n_split > 1 && (int64_t)a.layer[L].cout * a.layer[L].cin * a.layer[L].taps < 98304;
    for (int L = 0; L < a.n_layers; ++L) {
        const LayerUpdate& ly = a.layer[L];
        const int64_t nw = (int64_t)ly.cout * ly.cin * ly.taps;
        if (vecs) g.layer[L].streamed = ly.n_split > 160 ? kVec8 : ly.n_split > 80 || nw < 32768 ? kVec16 : ly.n_split > 32 ? kVec32 : kVec64;
        else if (nw >= 65536) g.layer[L].streamed = vectors(ly) ? 4 : 1;
        if (g.layer[L].streamed) {
            const int per = streamed_per_block(g.layer[L].streamed);
            stream_blocks += (nw + per - 1) / per;
        } else n_rest += nw;
    }
    int items = 1, max_split = 1;
    for (int L = 0; L < a.n_layers; ++L) {
        items += a.layer[L].cout;
        if (!g.layer[L].streamed && a.layer[L].n_split > max_split) max_split = a.layer[L].n_split;
    }
    const int n_red_blocks = (items + kUpdThreads / 32 - 1) / (kUpdThreads / 32);
    const bool big = n_rest > 65536;
    // many partial sums per parameter: 16 thread groups, so that a group's share fits one batch of loads
    const int G = max_split <= 1 ? 1 : (max_split > 64 && !big ? 16 : 8), E = big ? 4 : 1;
    const int per = kUpdThreads / G * E;
    const int n_param_blocks = (int)((n_rest + per - 1) / per);
    const int n_grouped = n_param_blocks + n_red_blocks;
    const dim3 grid((unsigned)(n_grouped + stream_blocks), (unsigned)a.S);
    const bool early = a.chain_early != 0, decides = a.has_ctl == 1 && a.ctl.C <= kWarpClasses && !big;
    auto launch = [&](auto kernel) { launch_early(early, kernel, grid, dim3(kUpdThreads + (decides ? 32 : 0)), 0, s, g, n_param_blocks, n_grouped); };
    // (a batch of loads is a round trip: 286 partial sums take one with twenty, three with eight)
    const bool many = G == 16 && max_split > 16 * 8;
    if (vecs) launch(decides ? sgd_update_kernel<1, 1, 8, ADAM, true, true> : sgd_update_kernel<1, 1, 8, ADAM, false, true>);
    else if (G == 1 && E == 4) launch(sgd_update_kernel<1, 4, 8, ADAM, false, false>);
    else if (E == 4) launch(sgd_update_kernel<8, 4, 8, ADAM, false, false>);
    else if (G == 1) launch(decides ? sgd_update_kernel<1, 1, 8, ADAM, true, false> : sgd_update_kernel<1, 1, 8, ADAM, false, false>);
    else if (G == 8) launch(decides ? sgd_update_kernel<8, 1, 8, ADAM, true, false> : sgd_update_kernel<8, 1, 8, ADAM, false, false>);
    else if (many) launch(decides ? sgd_update_kernel<16, 1, 20, ADAM, true, false> : sgd_update_kernel<16, 1, 20, ADAM, false, false>);
    else launch(decides ? sgd_update_kernel<16, 1, 8, ADAM, true, false> : sgd_update_kernel<16, 1, 8, ADAM, false, false>);
    return 1;
}

int launch_sgd_update(const UpdateArgs& a, cudaStream_t s)
{
    return a.adam ? launch_sgd_update_t<true>(a, s) : launch_sgd_update_t<false>(a, s);
}

__global__ void step_tick_kernel(long long* step_base, int S, int add)
{
    const int s = threadIdx.x;
    pdl_wait();
    pdl_launch_dependents();
    if (s < S) step_base[s] += add;
}

void launch_step_tick(long long* step_base, int S, int add, cudaStream_t s)
{
    for (int s0 = 0; s0 < S; s0 += 256)
        launch_early(pdl_enabled(), step_tick_kernel, dim3(1), dim3(256), 0, s, step_base + s0, S - s0 < 256 ? S - s0 : 256, add);
}

__global__ void __launch_bounds__(256) miou_kernel(const unsigned long long* __restrict__ conf, int C, double* out)
{
    __shared__ double iou[kMiouClasses];
    __shared__ int present[kMiouClasses];
    const double m = block_miou(conf, C, iou, present);
    if (threadIdx.x == 0) *out = m;
}

// End of Train (Algorithm 1): student <- best_student for the trained parameters, with the bf16 copies the GEMMs read; Adam's
// step count moves on by the steps taken.
__global__ void __launch_bounds__(256) train_commit_kernel(UpdateArgs a, const float* __restrict__ best_theta, const int* __restrict__ n_updates)
{
    pdl_wait();
    pdl_launch_dependents();
    const int s = blockIdx.y;
    const int64_t base = (int64_t)s * a.n_params;
    for (int64_t i = a.param_begin + (int64_t)blockIdx.x * 256 + threadIdx.x; i < a.n_params; i += (int64_t)gridDim.x * 256) {
        const float t = best_theta[base + i];
        a.theta[base + i] = t;
        for (int L = 0; L < a.n_layers; ++L) {
            const LayerUpdate& ly = a.layer[L];
            const int64_t e = i - ly.w_off;
            if (e >= 0 && e < (int64_t)ly.cout * ly.cin * ly.taps) write_shadows(ly, s, e, t);
        }
    }
    if (a.adam && blockIdx.x == 0 && threadIdx.x == 0) a.step_base[s] += n_updates[s];
}

void launch_miou(const unsigned long long* conf, int C, double* out, cudaStream_t s)
{
    miou_kernel<<<1, 256, 0, s>>>(conf, C, out);
}

static unsigned copy_blocks(int64_t n_params)
{
    const int64_t b = (n_params + 256 * 8 - 1) / (256 * 8);      // about 8 values per thread
    return (unsigned)(b < 1 ? 1 : (b > 592 ? 592 : b));
}

void launch_train_commit(const UpdateArgs& a, const float* best_theta, const int* n_updates, cudaStream_t s)
{
    launch_early(pdl_enabled(), train_commit_kernel, dim3(copy_blocks(a.n_params - a.param_begin), (unsigned)a.S), dim3(256), 0, s, a, best_theta, n_updates);
}

__global__ void __launch_bounds__(256) train_begin_kernel(unsigned long long* __restrict__ conf, int64_t n, double* threshold, double value)
{
    pdl_wait();
    pdl_launch_dependents();
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) conf[i] = 0ull;
    if (blockIdx.x == 0 && threadIdx.x == 0) *threshold = value;
}

void launch_train_begin(unsigned long long* conf, int64_t n, double* threshold, double value, cudaStream_t s)
{
    launch_early(pdl_enabled(), train_begin_kernel, dim3(copy_blocks(n)), dim3(256), 0, s, conf, n, threshold, value);
}

__global__ void train_results_kernel(TrainCtl t, const float* __restrict__ loss_buf, TrainResults out)
{
    pdl_wait();
    pdl_launch_dependents();
    const int s = blockIdx.x, i = threadIdx.x, n = t.max_updates + 1;
    if (i == 0 && out.n_updates) out.n_updates[s] = t.n_updates[s];
    if (i == 0 && out.best) out.best[s] = t.best[(int64_t)s * kCtlPitch + n];
    if (i < n && out.metric) out.metric[(int64_t)s * n + i] = t.metric[(int64_t)s * kCtlPitch + i];
    if (i < n && out.loss) out.loss[(int64_t)s * n + i] = loss_buf[(int64_t)s * kMaxSteps + i];
}

void launch_train_results(const TrainCtl& t, const float* loss_buf, const TrainResults& out, cudaStream_t s)
{
    launch_early(pdl_enabled(), train_results_kernel, dim3((unsigned)t.S), dim3(kMaxSteps), 0, s, t, loss_buf, out);
}

// ---- pack / unpack ---------------------------------------------------------------------------------
// A block moves 256 (output, input) channel pairs of a layer with all their taps: the packed side, [pair][tap], is one contiguous
// piece, the internal side one piece per tap; a 3x3 layer's values change places in shared memory.  (A thread per packed
// value reads or writes with a stride of a whole tap plane: 11 us for 2.4 MB at 256 -> 256 channels, 4 us this way.)  The last block
// of a buffer takes the biases.  Unpacking also writes the bf16 copies that the GEMMs read.
// The packed buffer may be pinned host memory: it is then read or written over the bus by the kernel itself.
constexpr int kPackPairs = 256;
template <bool TO_PACKED>
__global__ void __launch_bounds__(kPackPairs)
pack_kernel(const float* __restrict__ src, float* __restrict__ dst, PackLayout L, int first, int64_t begin, int64_t count, UpdateArgs u, int s0)
{
    __shared__ float sh[kPackPairs * 9];
    pdl_wait();
    pdl_launch_dependents();
    const int s = blockIdx.y, tid = threadIdx.x;
    const float* from = src + (int64_t)s * (TO_PACKED ? L.n_params : count);
    float* to = dst + (int64_t)s * (TO_PACKED ? count : L.n_params);
    int blk = blockIdx.x;
    for (int k = first; k < L.n_layers; ++k) {
        const int64_t pairs = (int64_t)L.cout[k] * L.cin[k];
        const int blocks = (int)((pairs + kPackPairs - 1) / kPackPairs), taps = L.taps[k];
        if (blk >= blocks) { blk -= blocks; continue; }
        const int64_t p0 = (int64_t)blk * kPackPairs, w = L.w_off[k], packed = w - begin + p0 * taps;
        const int n = (int)(pairs - p0 < kPackPairs ? pairs - p0 : kPackPairs);
        if (TO_PACKED) {
            if (tid < n)
                for (int t = 0; t < taps; ++t) sh[tid * taps + t] = from[w + t * pairs + p0 + tid];
            __syncthreads();
            for (int e = tid; e < n * taps; e += kPackPairs) to[packed + e] = sh[e];
        } else {
            for (int e = tid; e < n * taps; e += kPackPairs) sh[e] = from[packed + e];
            __syncthreads();
            if (tid < n)
                for (int t = 0; t < taps; ++t) {
                    const int64_t e = t * pairs + p0 + tid;
                    const float v = sh[tid * taps + t];
                    to[w + e] = v;
                    if (u.n_layers) write_shadows(u.layer[k - first], s0 + s, e, v);
                }
        }
        return;
    }
    for (int k = first; k < L.n_layers; ++k)
        for (int i = tid; i < L.cout[k]; i += kPackPairs) {
            const int64_t b = L.b_off[k] + i;
            if (TO_PACKED) to[b - begin] = from[b];
            else to[b] = from[b - begin];
        }
}

static dim3 pack_grid(const PackLayout& L, int first, int n_bufs)
{
    int64_t blocks = 1;
    for (int k = first; k < L.n_layers; ++k) blocks += ((int64_t)L.cout[k] * L.cin[k] + kPackPairs - 1) / kPackPairs;
    return dim3((unsigned)blocks, (unsigned)n_bufs);
}

void launch_pack(const float* internal, float* packed, const PackLayout& L, int first, int n_bufs, cudaStream_t s)
{
    const int64_t begin = L.w_off[first];
    UpdateArgs none;
    none.n_layers = 0;
    launch_early(pdl_enabled(), pack_kernel<true>, pack_grid(L, first, n_bufs), dim3(kPackPairs), 0, s, internal, packed, L, first, begin, L.n_params - begin, none, 0);
}

void launch_unpack(const float* packed, float* internal, const PackLayout& L, int first, int n_bufs, const UpdateArgs& u, int s0, cudaStream_t s)
{
    const int64_t begin = L.w_off[first];
    launch_early(pdl_enabled(), pack_kernel<false>, pack_grid(L, first, n_bufs), dim3(kPackPairs), 0, s, packed, internal, L, first, begin, L.n_params - begin, u, s0);
}

}  // namespace st
