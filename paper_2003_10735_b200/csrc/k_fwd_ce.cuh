// K3 for at most 32 classes — ComputeLoss and the first half of PartialBackward (Algorithm 1; loss of Section 5.2): bilinear x4
// upsample of the low-resolution logits, per-pixel softmax cross-entropy against the labels, gradient of the mean loss with
// respect to the logits.  With FORWARD the block multiplies its logits itself (1x1 classifier over at most 256 bf16 channels);
// without it they are read from memory.  Both forms do the same with them, bit for bit.  For more classes: k_upsample_ce.cu.
//
// Geometry.  With half-pixel centres and factor 4 the frame pixels 4n+2 .. 4n+5 lie between node columns n and n+1 ("cell" n)
// with weights 1/8, 3/8, 5/8, 7/8 toward n+1; rows alike.  Cells -1 and w-1 are the clamped borders (their outer node is the
// inner one).  A tile owns 7 rows x 30 columns of nodes.  A group of eight warps works on it: warp i owns cell row y0-1+i (the 4 x 4 frame
// pixels between two node rows), lane l owns node column x0-1+l and the 16 pixels of the cell to its right.  Warp 0, lane 0 and
// lane 31 are halo (recomputed by the neighbouring tile), so that a tile's nodes are finished in a fixed summation order,
// without floating-point atomics.
//
// With an own forward a block is persistent: a producer feeds a ring of chunks by TMA, and two issuers (a thread each) feed the tensor core.
// Where the weight gradient is formed too (one-layer heads), and with more than 24 classes, it has an SM to itself and two groups take its
// tiles in turn; otherwise it is one group, and two blocks fit an SM.  A launch that forms the gradient of at most one tile per SM is one
// group to a block too: half of the warps would have nothing to do, and its warps take their registers for more classes in flight.
//   Logits.  The features of the tile's 9 x 32 nodes arrive in chunks (nodes outside the map arrive
//   as zeros), and four multiplications per 16 channels leave node row i of the tile and node row i+1 of it in the same 32
//   tensor-memory lanes: the two rows that warp i's cells lie between.  A warp therefore takes its logits out of tensor memory
//   alone, without the other warps: bias added, shifted by the largest of them, in log2 units, clamped at the frame's border, both rows of
//   a class side by side in the warp's own slots of shared memory [class][lane] (upper, lower).  The second class sweep leaves the
//   cell's pull on the two node rows in the same slots.  A group's next tile is fetched and multiplied while it works on this one.
//   Weight gradient of a one-layer head (w_part).  The epilogue leaves the bf16 gradient of the tile's own nodes in shared memory as an operand, the
//   features come once more, from L2, and their product (reduction over the nodes) becomes one partial sum per tile, which the update adds in
//   order.  A kernel of its own read the map again instead, from HBM where it is more than L2 holds, behind one more kernel boundary.
// Without FORWARD a block is one group with one tile, and a warp reads its two node rows from memory (all classes' loads in flight
// together).
//
// Fast path (the usual case), class by class for all 16 pixels of a cell: inside a cell the interpolated logit is
// u(r,k) = A + B k + G r + D k r, so its 16 exponentials are geometric progressions (cell_softmax.cuh).  Sweep 1 sums them per
// pixel, sweep 2 forms their bases again (cheaper than keeping 16 x C registers) and reduces them to the pull on the nodes.
// Slow path (a class that changes by more than kFastRange log2-units inside a cell, or a sum that underflows): the warp walks
// its four frame rows one by one with exact per-pixel maxima.
// The onehot part of the gradient is exact in units of 1/64: integer counts, two classes to a 32-bit word of shared memory (a
// node receives at most 1024 times the largest pixel weight, 5), added by shared-memory atomics, one round per distinct label of
// a cell.  Pixels tagged for the loss weighting (bit 7 of the label byte) count with an integer weight in the loss, in 1/Z and
// in those counts.
// The epilogue adds, per node row, the warp's upper pulls, the lower pulls of the warp above and the counts, writes the
// gradient, and reduces the tile's share of the bias gradient.  With CONF the student's class of every pixel is taken from sweep
// 1 and counted against the label.
//
// Bound by latency and issue slots at 16 working warps an SM (half of the slots go to the sweeps), and at a launch's start by L2, from
// which every block fetches two tiles (47 MB for one 720p frame of 256 channels): the first group has its logits after 8000 cycles, the
// second after 12800.  us of a call of eight steps with two blocks of one group on an SM, a warp each to feed the tensor core and a kernel of its own for the
// weight gradient / now, 256 channels on 180 x 320, 21 classes: 275.8 / 267.6, 4 streams 963 / 856, 16 streams 3535 / 3248; 30 classes (weight
// gradient apart), 4 streams 1274 / 1137; 32 classes 351 / 330; 4 classes 201 / 184; 128 channels on 90 x 160 156.7 / 146.8.  Behind a 3x3 layer (no weight
// gradient) two groups lose, since the kernels around theirs find no room beside a block that fills an SM; us a launch, a warp each to feed the
// tensor core / two groups / one group as it is: three maps of 101 x 187, 128 channels 18.5 / 19.2 / 18.0, 720p, 64 channels 16.9 / 16.8 / 16.5,
// 1080p, 256 channels 43.8 / 45.7 / 43.9; the stack's step 127.9 / 128.7 / 127.6.
// Tried: one group whose warps divide the classes (sums and labels are then worked out twice: 222 -> 370 us for 16 streams); places of the
// ring over both groups' slots for a block's first tile (no change: L2 sets the pace); bias sums through shared memory (one more
// barrier: 3250 -> 3280).
#pragma once

#include "st_internal.h"
#include "tc_common.cuh"
#include "fused_tile.cuh"
#include "cell_softmax.cuh"

#include <string.h>
#include <utility>

namespace st {

namespace {

constexpr int F_ROWS = fused::kTileRows, F_COLS = fused::kTileCols;         // nodes of a tile, halo included
constexpr int FN_Y = fused::kOwnRows, FN_X = fused::kOwnCols;               // nodes a tile owns
constexpr int F_WARPS = FN_Y + 1, F_WORKERS = F_WARPS * 32;                 // of a group: the warps that work on one tile
// What a block is: one group that reads stored logits; one group with its own forward, two blocks to an SM; two groups with their own
// forward, which have an SM to themselves; one group alone on an SM, with the registers for more classes in flight
enum Form { kStored = 0, kOneGroup = 1, kTwoGroups = 2, kLoneGroup = 3 };
__host__ __device__ constexpr bool form_alone(int form) { return form == kTwoGroups || form == kLoneGroup; }
__host__ __device__ constexpr int form_groups(int form) { return form == kTwoGroups ? 2 : 1; }
__host__ __device__ constexpr int form_threads(int form) { return form_groups(form) * F_WORKERS + (form == kStored ? 0 : 128); }
constexpr int kNodes = F_ROWS * F_COLS;
constexpr int kSweep1 = 7;                                                  // classes per iteration of the first sweep, of the second
__host__ __device__ constexpr int sweep2(int form) { return form == kLoneGroup ? 7 : 3; }
constexpr uint32_t kWBytes = fused::kWeightBytes;
constexpr uint32_t kRowBytes = F_COLS * 128;                                // a node row of 64 channels
constexpr int kLogitCols = 4 * kClassPad, kGradCols = 2 * kClassPad;        // tensor memory of a group: upper and lower rows of warps 0-3 and
                                                                            // 4-7; the weight gradient of 256 channels
constexpr int kIssuers = 2;
__host__ __device__ constexpr int max_places(int form) { return form == kLoneGroup ? 8 : 7; }
// A place of the ring.  Two groups: five node rows of 64 channels, so that a tile's channels are two chunks, rows 0-4 and 4-8.  One group,
// whose shared memory holds one such place next to 21 classes: the tile's nine rows of 32 channels, of which there is room for two.  (Half rows
// read from HBM are slower: with them in two groups 16 streams take 3312 us a call, 3260 with whole ones; one frame's 272 either way.)
__host__ __device__ constexpr bool half_rows(int form) { return form == kOneGroup; }
__host__ __device__ constexpr uint32_t chunk_bytes(int form) { return half_rows(form) ? F_ROWS * kRowBytes / 2 : 5 * kRowBytes; }
// Registers with an own forward.  A scheduler's 16384 registers give 96 a thread at launch with five warps on it (two groups), 80 with six
// (two blocks of one); the warpgroup of the producer and the issuers (its fourth warp returns at once) gives back what the workers take.
constexpr int kFeederRegs = 32;
__host__ __device__ constexpr int form_launch_regs(int form) { return form == kTwoGroups ? 96 : form == kLoneGroup ? 168 : 80; }
__host__ __device__ constexpr int form_worker_regs(int form) { return form == kTwoGroups ? 112 : form == kLoneGroup ? 232 : 104; }
constexpr bool regs_add_up(int form) { return form_groups(form) * F_WORKERS * form_worker_regs(form) + 128 * kFeederRegs <= form_threads(form) * form_launch_regs(form); }
static_assert(regs_add_up(kOneGroup) && regs_add_up(kTwoGroups) && regs_add_up(kLoneGroup), "registers handed on are registers the block was launched with");

// Shared memory: the ring, then the groups' arrays.  The ring's places go on over the last group's slots, which are free until that
// group has its first logits (and for good where it has no tile).
template <int C, bool CONF, int FORM>
struct FwdCeSmem {
    static constexpr bool FORWARD = FORM != kStored;
    static constexpr uint32_t kChunkBytes = chunk_bytes(FORM);
    static constexpr size_t kSlots = (size_t)F_WARPS * C * 32 * sizeof(float2), kCounts = (size_t)((C + 1) / 2) * kNodes * sizeof(uint32_t),
                            kHist = CONF ? (size_t)C * C * sizeof(unsigned int) : 0, kWeights = FORWARD ? (size_t)fused::kMaxKBlocks * kWBytes : 0;
    static constexpr int kN = form_groups(FORM);
    static constexpr size_t kGrad = form_alone(FORM) && classifier_gradient_fits(C) ? (size_t)4 * kWBytes : 0;     // bf16 gradient of a tile's own nodes: [two node rows][32 classes][64 nodes]
    static constexpr size_t kFixed = kN * (kSlots + kCounts + kHist + kGrad) + kWeights;
    // less what the system keeps of a block's share, the alignment and the static arrays
    static constexpr size_t kStatic = kN * (F_WARPS * 256 + 64) + 512, kMost = (form_alone(FORM) ? 228 * 1024 : 114 * 1024) - 2048 - kStatic;
    // (a lone group's one tile lies there whole, as far as there is room: all of it is fetched before the wait)
    static constexpr int kMaxPlaces = max_places(FORM), kCap = FORM == kLoneGroup ? kMaxPlaces : 4;
    static constexpr int kSteady = !FORWARD ? 0 : kMost < kFixed ? 0 : (kMost - kFixed) / kChunkBytes > kCap ? kCap : (int)((kMost - kFixed) / kChunkBytes);
    static constexpr int kExtra = !FORWARD ? 0 : kSteady + (int)(kSlots / kChunkBytes) > kMaxPlaces ? kMaxPlaces - kSteady : (int)(kSlots / kChunkBytes);
    static constexpr bool kFits = !FORWARD || (kMost >= kFixed && kSteady >= 1);
    // the last group's slots lie behind the ring
    static constexpr size_t kSlotsAt = kSteady * (size_t)kChunkBytes, kWeightsAt = kSlotsAt + kN * kSlots, kGradAt = kWeightsAt + kWeights,
                            kCountsAt = kGradAt + kN * kGrad, kHistAt = kCountsAt + kN * kCounts, kBytes = kHistAt + kN * kHist + 1024;
};

__device__ __forceinline__ float lg2_approx(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void arrive(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory"); }
// the warps of a group
__device__ __forceinline__ void workers_sync(int grp) { asm volatile("barrier.cta.sync %0, %1;" ::"r"(1 + grp), "n"(F_WORKERS) : "memory"); }
__device__ __forceinline__ bool workers_all(int grp, bool ok)
{
    int r;
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbarrier.cta.red.and.pred q, %3, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(r) : "r"((int)ok), "n"(F_WORKERS), "r"(1 + grp) : "memory");
    return r != 0;
}

// cell_bases of cell_softmax.cuh for values that are shifted and in log2 units already: L, R = (upper, lower) node row of the
// left and the right node column
__device__ __forceinline__ float cell_bases_log2(float2 L, float2 R, float2& x01, float2& x23, float2& q01, float2& q23)
{
    const float p = L.y - L.x, qq = R.y - R.x, e0 = R.x - L.x, qp = qq - p;
    const float wv = fmaf(qp, 0.125f, e0), A = fmaf(wv, 0.125f, fmaf(p, 0.125f, L.x));
    const float E00 = ex2_approx(A), QB = ex2_approx(0.25f * wv), TG = ex2_approx(fmaf(qp, 0.03125f, 0.25f * p)), SD = ex2_approx(0.0625f * qp);
    const float TG2 = TG * TG, SD2 = SD * SD;
    q01 = make_float2(QB, QB * SD);
    q23 = __fmul2_rn(q01, make_float2(SD2, SD2));
    x01 = make_float2(E00, E00 * TG);
    x23 = __fmul2_rn(x01, make_float2(TG2, TG2));
    return fmaxf(fabsf(p), fmaxf(fabsf(qq), fabsf(e0)));
}

// Slow path: values of the lane's four pixels of one frame row for a class
__device__ __forceinline__ void row_values(float2 L, float2 R, float ly, float (&u)[4])
{
    const float vl = fmaf(ly, L.y - L.x, L.x), d = fmaf(ly, R.y - R.x, R.x) - vl;
#pragma unroll
    for (int k = 0; k < 4; ++k) u[k] = fmaf((2 * k + 1) * 0.125f, d, vl);
}

// f(first, N) for C classes in groups of G: a rolled loop over the whole groups, then what is left
template <int C, int G, class F>
__device__ __forceinline__ void static_for_groups(F f)
{
#pragma unroll 1
    for (int c = 0; c + G <= C; c += G) f(c, std::integral_constant<int, G>());
    if constexpr (C % G != 0) f(C - C % G, std::integral_constant<int, C % G>());
}

// counts of one class (two classes to a word)
__device__ __forceinline__ void add_counts(uint32_t* node, int cls, int right, int below, uint32_t tl, uint32_t tr, uint32_t bl, uint32_t br)
{
    uint32_t* w = node + (cls >> 1) * kNodes;
    const int sh = (cls & 1) * 16;
    atomicAdd(w, tl << sh);
    atomicAdd(w + right, tr << sh);
    atomicAdd(w + below, bl << sh);
    atomicAdd(w + below + right, br << sh);
}

template <int C, bool CONF, int FORM>
__global__ void __launch_bounds__(form_threads(FORM), form_alone(FORM) ? 1 : 2)
fwd_ce_kernel(UpsampleCeArgs a, int tiles_x, int tiles_y, const __grid_constant__ CUtensorMap x_map, const __grid_constant__ CUtensorMap w_map,
              const __grid_constant__ CUtensorMap row_map)
{
    using Smem = FwdCeSmem<C, CONF, FORM>;
    static_assert(Smem::kFits, "a block's shared memory");
    constexpr bool FORWARD = FORM != kStored, with_grad = Smem::kGrad != 0;        // (with_grad: the classifier's weight gradient as well)
    constexpr int kGroups = form_groups(FORM), kAllWarps = kGroups * F_WARPS;
    constexpr uint32_t kChunkBytes = Smem::kChunkBytes;
    constexpr int kMaxPlaces = Smem::kMaxPlaces;
    extern __shared__ __align__(128) uint8_t smem_f[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_f + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t bars[2 * kMaxPlaces + 1 + 5 * kGroups];
    __shared__ uint32_t tmem_slot;
    __shared__ volatile uint32_t gave_up;
    __shared__ float red[kGroups][2][F_WARPS], wsum[kAllWarps][32];
    __shared__ __align__(16) float bias[kAllWarps][32];
    // barriers: places of the ring filled / free, weights; per group: logits there / taken, gradient there, its product there / taken
    const uint32_t full_bar = tc::smem_u32(&bars[0]), free_bar = full_bar + 8 * kMaxPlaces, w_bar = full_bar + 16 * kMaxPlaces, done_bars = w_bar + 8,
                   taken_bars = done_bars + 8 * kGroups, dz_bars = taken_bars + 8 * kGroups, grad_bars = dz_bars + 8 * kGroups, grad_taken_bars = grad_bars + 8 * kGroups;
    const int h = a.h, w = a.w, H = h * kUp, W = w * kUp;
    const int64_t p = (int64_t)h * w;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), l = tid & 31;
    const int grp = FORWARD ? warp / F_WARPS : 0, wi = warp % F_WARPS, gtid = tid % F_WORKERS;       // (of the workers)
    float2* slots = (float2*)(smem + Smem::kSlotsAt + (grp + 1 < kGroups ? Smem::kSlots : 0));      // [F_WARPS][C][32]
    uint32_t* counts = (uint32_t*)(smem + Smem::kCountsAt + grp * Smem::kCounts);                    // [(C + 1) / 2][F_ROWS][F_COLS]
    unsigned int* hist = (unsigned int*)(smem + Smem::kHistAt + grp * Smem::kHist);                  // [C][C] (CONF)
    const int per_stream = tiles_x * tiles_y, n_tiles = per_stream * a.S;
    // Tiles at the frame's border do extra work: the last tile row of a stream comes first, then rows 0, 1, ...
    // A block walks its tiles by additions: a division takes the warp that feeds the tensor core 1500 cycles beside sixteen others.
    struct Tile { int t, s, row, col; };                   // t: index in the order of the walk
    const int d_s = (int)gridDim.x / per_stream, d_row = (int)gridDim.x % per_stream / tiles_x, d_col = (int)gridDim.x % per_stream % tiles_x;
    auto step = [&](Tile& k) {
        k.t += gridDim.x; k.s += d_s; k.row += d_row; k.col += d_col;
        if (k.col >= tiles_x) { k.col -= tiles_x; ++k.row; }
        if (k.row >= tiles_y) { k.row -= tiles_y; ++k.s; }
    };
    // ... on to a tile whose stream still trains (the flags come from an earlier kernel: after the wait only)
    auto settle = [&](Tile& k) { while (a.skip && k.t < n_tiles && a.skip[(int64_t)k.s * a.skip_stride]) step(k); };
    auto next = [&](Tile& k) { step(k); settle(k); };
    const Tile first{(int)blockIdx.x, (int)blockIdx.x / per_stream, (int)blockIdx.x % per_stream / tiles_x, (int)blockIdx.x % per_stream % tiles_x};
    auto tile_row = [&](const Tile& k) { return k.row == 0 ? tiles_y - 1 : k.row - 1; };
    auto node_x = [&](const Tile& k) { return k.col * FN_X; };             // the first node a tile owns
    auto node_y = [&](const Tile& k) { return tile_row(k) * FN_Y; };
    constexpr int tmem_cols = (with_grad ? 2 : 1) * kGroups * kLogitCols;  // (a power of two)

    if (FORWARD && warp == kAllWarps + 1) {
        if (tc::elect_one()) { tc::prefetch_map(&x_map); tc::prefetch_map(&w_map); if (with_grad) tc::prefetch_map(&row_map); }
        __syncwarp();
        tc::tmem_alloc(tc::smem_u32(&tmem_slot), tmem_cols);
    }
    if (FORWARD && tid == 0) {
        for (int k = 0; k < kMaxPlaces; ++k) { tc::mbar_init(full_bar + 8u * (uint32_t)k, 1); tc::mbar_init(free_bar + 8u * (uint32_t)k, kIssuers); }
        tc::mbar_init(w_bar, 1);
        for (int g = 0; g < kGroups; ++g) {
            tc::mbar_init(done_bars + 8 * g, kIssuers); tc::mbar_init(grad_bars + 8 * g, kIssuers);
            tc::mbar_init(taken_bars + 8 * g, F_WARPS); tc::mbar_init(dz_bars + 8 * g, F_WARPS); tc::mbar_init(grad_taken_bars + 8 * g, F_WARPS);
        }
        gave_up = 0;
        tc::fence_barrier_init();
    }
    if (!FORWARD || warp < kAllWarps) {
        for (int e = gtid; e < (int)(Smem::kCounts / 16); e += F_WORKERS) reinterpret_cast<uint4*>(counts)[e] = make_uint4(0, 0, 0, 0);
        if (CONF) for (int e = gtid; e < C * C; e += F_WORKERS) hist[e] = 0;
    }
    tc::tc_fence_before_sync();
    __syncthreads();
    tc::tc_fence_after_sync();
    const uint32_t tmem = FORWARD ? tmem_slot : 0;

    if (FORWARD && warp >= kAllWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFeederRegs));
        if (warp > kAllWarps + kIssuers) return;
        // ---------------------------------------------------------------- the producer and the issuer
        // Both walk the same list: for every tile F, its logits (per 64 channels two chunks, node rows 0-4 and 4-8), and kLag tiles later
        // G, its weight gradient (per 128 channels four chunks of two own node rows).  A chunk takes the ring's next place.  One thread
        // each: a whole warp's waits and elections between two chunks of eight multiplications take as long as the multiplications.
        const bool producer = warp == kAllWarps;
        const int me = warp - kAllWarps - 1;               // issuer: the first takes the upper node rows, the second the lower ones
        const uint32_t ring = tc::smem_u32(smem), w_base = ring + (uint32_t)Smem::kWeightsAt;
        const int kblocks = a.kblocks, mt = (kblocks + 1) / 2;
        bool ok = true;
        if (tc::elect_one()) {
            int place = 0, n_places = Smem::kSteady + Smem::kExtra;
            uint32_t used = 0, parity = 0;                 // per place: has been filled; parity of the wait that comes next
            auto wait = [&](uint32_t bar, uint32_t par, unsigned code) { ok = ok && tc::mbar_wait_from(tc::mbar_try_wait(bar, par), bar, par, a.err, code); };
            auto advance = [&]() { place = place + 1 == n_places ? 0 : place + 1; };
            // (the producer) the place that is filled next, once what lay there has been multiplied
            auto claim = [&](uint32_t bytes) {
                const uint32_t bit = 1u << place;
                if (used & bit) {
                    wait(free_bar + 8 * place, (parity & bit) != 0, tc::kWaitEmpty);
                    parity ^= bit;
                }
                used |= bit;
                if (ok) tc::mbar_expect_tx(full_bar + 8 * place, bytes);
                return ok;
            };
            auto load_rows = [&](const Tile& k, int e, uint32_t stall) {   // chunk e of F
                if (!claim(kChunkBytes + stall)) return;
                tc::tma_load_4d(ring + place * kChunkBytes, &x_map, full_bar + 8 * place, half_rows(FORM) ? e * 32 : (e >> 1) * 64, node_x(k) - 1,
                                node_y(k) - 1 + (half_rows(FORM) ? 0 : 4 * (e & 1)), k.s);
                advance();
            };
            // Inside the step loop the features are frozen: the first chunks are fetched while the previous update still runs
            int pre = a.x_early ? min(n_places, 2 * kblocks) : 0;
            if (producer) {
                for (int e = 0; e < pre && ok; ++e) load_rows(first, e, e == 0 && a.test_stall ? 16u : 0u);
            }
            pdl_wait();                                    // the weights come from the previous kernel of the stream
            Tile k = first;
            settle(k);
            if (pre && k.t != first.t) {                   // the tile that was begun with is not worked on
                if (producer) {
                    for (int e = 0; e < pre; ++e) wait(full_bar + 8 * e, 0, tc::kWaitFull);
                    used = 0;
                } else parity = (1u << pre) - 1;
                pre = 0; place = 0;
            }
            constexpr int kLag = kGroups + 1;              // (a group takes its next tile's logits before it waits for this one's gradient)
            Tile back = k;                                 // the tile whose weight gradient comes next
            int w_stream = -1, n_weights = 0, n_items = 0;
            for (int q = 0; ok && (k.t < n_tiles || (with_grad && back.t < n_tiles)); ++q) {
                if (q == kGroups && n_items == kGroups) { n_places = Smem::kSteady; place = 0; }
                if (k.t < n_tiles) {
                    const int g = q % kGroups, j = q / kGroups;
                    if (producer) {
                        for (int e = q == 0 ? pre : 0; e < 2 * kblocks && ok; ++e) load_rows(k, e, q == 0 && e == 0 && a.test_stall ? 16u : 0u);
                    } else {
                        constexpr uint32_t idesc = tc::instr_desc(128, kClassPad, 0, 0);
                        if (w_stream != k.s) {             // the weights of the stream before are read until the last tile's logits are there
                            if (q) wait(done_bars + 8 * ((q - 1) % kGroups), ((q - 1) / kGroups) & 1, tc::kWaitDone);
                            if (ok && me == 0) {
                                tc::mbar_expect_tx(w_bar, (uint32_t)kblocks * kWBytes);
                                for (int kb = 0; kb < kblocks; ++kb) tc::tma_load_3d(w_base + kb * kWBytes, &w_map, w_bar, kb * 64, 0, k.s);
                            }
                            w_stream = k.s;
                            wait(w_bar, n_weights++ & 1, tc::kWaitFull);
                        }
                        if (j) wait(taken_bars + 8 * g, (j - 1) & 1, tc::kWaitEmpty);
                        const uint32_t logits = tmem + g * kLogitCols + me * 2 * kClassPad;
                        uint64_t dw = tc::smem_desc(w_base, 16, 1024);
                        for (int e = 0; e < 2 * kblocks && ok; ++e) {
                            const uint32_t bit = 1u << place, bar = full_bar + 8 * place;
                            if (a.test_stall) {
                                ok = false;
                                for (int it = 0; it < (1 << 12) && !ok; ++it) ok = tc::mbar_try_wait(bar, (parity & bit) != 0);
                                if (!ok) atomicCAS(a.err, 0u, (unsigned)tc::kWaitFull | (blockIdx.x << 8));
                            } else wait(bar, (parity & bit) != 0, tc::kWaitFull);
                            parity ^= bit;
                            if (!ok) break;
                            tc::tc_fence_after_sync();
                            const uint32_t at = ring + place * kChunkBytes;
                            // (rows 0-3, 4-7 upper; 1-4, 5-8 lower)
                            if constexpr (half_rows(FORM)) {
                                const uint64_t dx = tc::smem_desc_64(at + me * (kRowBytes / 2), 512);
#pragma unroll
                                for (int u = 0; u < 4; ++u)
                                    tc::umma(logits + (u & 1) * kClassPad, dx + (u & 1) * (2 * kRowBytes >> 4) + (u & 2), dw + (u & 2), idesc, (e | u >> 1) != 0);
                                dw += e & 1 ? (kWBytes >> 4) - 4 : 4;  // two chunks to the weights' 64 channels
                            } else {
                                const uint64_t dx = tc::smem_desc(at + me * kRowBytes, 16, 1024);
#pragma unroll
                                for (int u = 0; u < 4; ++u) tc::umma(logits + (e & 1) * kClassPad, dx + 2 * u, dw + 2 * u, idesc, (e >> 1 | u) != 0);
                                if (e & 1) dw += kWBytes >> 4;
                            }
                            tc::umma_commit(free_bar + 8 * place);
                            advance();
                        }
                        if (ok) tc::umma_commit(done_bars + 8 * g);
                    }
                    ++n_items;
                    next(k);
                }
                if (with_grad && q >= kLag && back.t < n_tiles && ok) {
                    // dW[channel][class] = sum of X[node][channel] dz[node][class] over the tile's own nodes: the group has left the bf16
                    // gradient in shared memory (K-major, zeros at the halo), the features come again (MN-major)
                    const int g = (q - kLag) % kGroups, j = (q - kLag) / kGroups;
                    if (producer) {
                        for (int e = 0; e < 4 * mt && ok; ++e) {
                            const int m = e >> 2, r0 = 2 * (e & 3), rows = r0 == 6 ? 1 : 2;
                            if (!claim((uint32_t)(2 * rows) * kRowBytes)) break;
                            for (int b = 0; b < 2; ++b)
                                for (int r = 0; r < rows; ++r)
                                    tc::tma_load_4d(ring + place * kChunkBytes + (uint32_t)(b * rows + r) * kRowBytes, &row_map, full_bar + 8 * place, (2 * m + b) * 64, node_x(back) - 1, node_y(back) + r0 + r, back.s);
                            advance();
                        }
                    } else {
                        constexpr uint32_t idesc = tc::instr_desc(128, kClassPad, 1, 0);
                        wait(dz_bars + 8 * g, j & 1, tc::kWaitFull);
                        if (j) wait(grad_taken_bars + 8 * g, (j - 1) & 1, tc::kWaitEmpty);
                        const uint32_t to = tmem + kGroups * kLogitCols + g * kGradCols;
                        const uint64_t dz = tc::smem_desc(ring + (uint32_t)Smem::kGradAt + g * (uint32_t)Smem::kGrad, 16, 1024);
                        for (int e = 0; e < 4 * mt && ok; ++e) {
                            const uint32_t bit = 1u << place;
                            wait(full_bar + 8 * place, (parity & bit) != 0, tc::kWaitFull);
                            parity ^= bit;
                            if (!ok) break;
                            if ((e >> 2) != me) { arrive(free_bar + 8 * place); advance(); continue; }     // the other issuer's channels
                            tc::tc_fence_after_sync();
                            const uint64_t dg = dz + (e & 3) * (kWBytes >> 4);
                            const bool last = (e & 3) == 3;
                            const uint64_t dx = tc::smem_desc(ring + place * kChunkBytes, last ? kRowBytes : 2 * kRowBytes, 1024);
#pragma unroll
                            for (int u = 0; u < 4; ++u)            // sixteen nodes at a time
                                if (u < 2 || !last) tc::umma(to + (e >> 2) * kClassPad, dx + ((u * 16 * 128) >> 4), dg + 2 * u, idesc, ((e & 3) | u) != 0);
                            tc::umma_commit(free_bar + 8 * place);
                            advance();
                        }
                        if (ok) tc::umma_commit(grad_bars + 8 * g);
                    }
                    next(back);
                }
            }
            if (!producer) {
                for (int it = n_items > kGroups ? n_items - kGroups : 0; it < n_items && ok; ++it) {
                    wait(taken_bars + 8 * (it % kGroups), (it / kGroups) & 1, tc::kWaitEmpty);
                    if (with_grad) wait(grad_taken_bars + 8 * (it % kGroups), (it / kGroups) & 1, tc::kWaitEmpty);
                }
            }
            if (!ok) {                                     // nothing more is multiplied and nothing is written
                gave_up = 1;
                if (!producer) for (int g = 0; g < kGroups; ++g) { arrive(done_bars + 8 * g); arrive(grad_bars + 8 * g); }
                tc::drain_after_error();
            }
        }
        __syncwarp();
        if (me != 0) return;
        tc::tc_fence_after_sync();
        tc::tmem_dealloc(tmem, tmem_cols);
        return;
    }

    // -------------------------------------------------------------------- the workers
    if (FORWARD) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(form_worker_regs(FORM)));
    const uint32_t done_bar = done_bars + 8 * grp, taken_bar = taken_bars + 8 * grp, dz_bar = dz_bars + 8 * grp, grad_bar = grad_bars + 8 * grp,
                   grad_taken = grad_taken_bars + 8 * grp, logits_at = tmem + grp * kLogitCols, grads_at = tmem + kGroups * kLogitCols + grp * kGradCols;
    float2* my = slots + (size_t)wi * C * 32 + l;          // this lane's slot of class c: my[c * 32]
    const int hw1 = a.heavy_w - 1;                         // what a weighted pixel counts on top of 1
    const float invP = 1.0f / ((float)H * (float)W);
    int n_done = 0;
    bool waited = false;
    // (neighbouring tiles at the same time on neighbouring blocks: what they share comes from L2)
    // The weight gradient of the tile before this one, as the tensor core has left it -> its partial sum
    auto store_gradient = [&](const Tile& k) {
        const int m = wi >> 2, ch = m * 128 + (wi & 3) * 32 + l, K = a.kblocks * 64;
        tc::tc_fence_after_sync();
        if (2 * m < a.kblocks) {                           // warp-uniform
            float g[32];
            const uint32_t from = grads_at + ((uint32_t)((wi & 3) * 32) << 16) + m * kClassPad;
            if constexpr (C <= 16) tc::tmem_ld_32x16(from, reinterpret_cast<float(&)[16]>(g));
            else tc::tmem_ld_32x32(from, g);
            float* dst = a.w_part + ((int64_t)k.s * per_stream + tile_row(k) * tiles_x + k.col) * C * K + ch;
            if (ch < K)
#pragma unroll
                for (int c = 0; c < C; ++c) dst[c * K] = g[c];
        }
        tc::tc_fence_before_sync();
        __syncwarp();
        if (tc::elect_one()) arrive(grad_taken);
    };
    // the groups take the block's tiles in turn
    Tile k = first, before = first;
    if (grp) step(k);
    while (k.t < n_tiles) {
        const int x0 = node_x(k), y0 = node_y(k), s = k.s, blk = tile_row(k) * tiles_x + k.col;
        const int i = y0 - 1 + wi, n = x0 - 1 + l;         // cell row (frame rows 4i+2 .. 4i+5, node rows i, i+1), own node column
        const bool cell_row = i <= h - 1, cell_valid = l <= 30 && n <= w - 1, node_owned = l >= 1 && l <= FN_X && n < w;
        // the aligned 4-pixel words of the label rows: a cell's pixels are the upper half of its own column's word and the lower
        // half of the next one's
        uint32_t labw[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int Y = 4 * i + 2 + r;
            labw[r] = cell_row && Y >= 0 && Y < H && n >= 0 && n < w
                          ? __ldg(reinterpret_cast<const uint32_t*>(a.labels + (int64_t)s * H * W + (int64_t)Y * W + 4 * n)) : 0u;
        }
        if (!waited) {                                     // the parameters come from the previous kernel of the stream
            pdl_wait();
            waited = true;
            if (FORWARD && a.skip) {                       // ... and so does which tiles are worked on
                Tile f = first;
                settle(f);
                if (grp) next(f);
                if (f.t != k.t) { k = f; continue; }
            }
        }
        if (!FORWARD && a.skip && a.skip[(int64_t)s * a.skip_stride]) return;
        const Tile now = k;
        next(k);
        float bias_l = 0.f;
        bool ok = true;
        ++n_done;
        if constexpr (FORWARD) {
            if (l < C) bias_l = a.theta[(int64_t)s * a.n_params + a.b_off + l];
            ok = tc::mbar_wait(done_bar, (n_done - 1) & 1, a.err, tc::kWaitDone);
            tc::tc_fence_after_sync();
            if (gave_up) ok = false;
        }
        float loss = 0.f;
        unsigned n_bad = 0;
        // where the cell's left and right node columns lie relative to the own slot (clamped at the frame's left and right border)
        const int at_l = n == -1 ? 1 : 0, to_r = (l < 31 && n >= 0 && n < w - 1) ? 1 : 0;
        const bool fold_l = n == -1, fold_r = n == w - 1;
        const int t_row = min(i + 1, h - 1), t_col = min(n + 1, w - 1);    // the tile that owns this node counts the cell's loss
        const bool own_cell = cell_row && cell_valid && t_row >= y0 && t_row < y0 + FN_Y && t_col >= x0 && t_col < x0 + FN_X;
        if (cell_row && ok) {                              // warp-uniform
            {
                // ---- the warp's two node rows, upper and lower, clamped at the frame's border -> slots
                const bool in_cols = n >= 0 && n < w;
                float up[32], lo[32], m = -INFINITY;
                if constexpr (FORWARD) {
                    bias[warp][l] = bias_l;
                    __syncwarp();
                    const uint32_t lanes = logits_at + ((uint32_t)((wi & 3) * 32) << 16), upper = lanes + (wi >> 2) * kClassPad, lower = upper + 2 * kClassPad;
                    if constexpr (C <= 16) {
                        tc::tmem_ld_32x16(i == -1 ? lower : upper, reinterpret_cast<float(&)[16]>(up));
                        tc::tmem_ld_32x16(i == h - 1 ? upper : lower, reinterpret_cast<float(&)[16]>(lo));
                    } else {
                        tc::tmem_ld_32x32(i == -1 ? lower : upper, up);
                        tc::tmem_ld_32x32(i == h - 1 ? upper : lower, lo);
                    }
                    tc::tc_fence_before_sync();
                    __syncwarp();
                    if (tc::elect_one()) arrive(taken_bar);
#pragma unroll
                    for (int c4 = 0; c4 < C; c4 += 4) {
                        const float4 b4 = *reinterpret_cast<const float4*>(&bias[warp][c4]);
                        const float b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
                        for (int c = c4; c < c4 + 4 && c < C; ++c) { up[c] += b[c - c4]; lo[c] += b[c - c4]; }
                    }
                } else {
                    const float *zu = a.z + (int64_t)s * C * p + (int64_t)max(i, 0) * w + n, *zl = a.z + (int64_t)s * C * p + (int64_t)min(i + 1, h - 1) * w + n;
#pragma unroll
                    for (int c = 0; c < C; ++c) { up[c] = in_cols ? zu[(int64_t)c * p] : 0.f; lo[c] = in_cols ? zl[(int64_t)c * p] : 0.f; }
                }
#pragma unroll
                for (int c = 0; c < C; ++c) m = fmaxf(m, fmaxf(up[c], lo[c]));
                if (!in_cols) m = -INFINITY;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (FORWARD && a.z_out && wi >= 1 && node_owned) {    // the own nodes, where the caller wants the logits kept
                    float* zo = a.z_out + (int64_t)s * C * p + (int64_t)i * w + n;
#pragma unroll
                    for (int c = 0; c < C; ++c) zo[(int64_t)c * p] = up[c];
                }
                // nodes outside the frame hold the bare bias: nobody's pixels, but they must not disturb the warp's vote
                const float scale = in_cols ? kLog2e : 0.f, shift = in_cols ? -m * kLog2e : 0.f;
#pragma unroll
                for (int c = 0; c < C; ++c) my[c * 32] = make_float2(fmaf(up[c], scale, shift), fmaf(lo[c], scale, shift));
                __syncwarp();
            }
            const float2* ps = my + at_l;
            // ---- sweep 1: sums of the 16 pixels' exponentials
            float2 Z01[4], Z23[4];                         // Z01[k] = (Z(0,k), Z(1,k)), Z23[k] = (Z(2,k), Z(3,k))
#pragma unroll
            for (int q = 0; q < 4; ++q) Z01[q] = Z23[q] = make_float2(0.f, 0.f);
            float wmax = 0.f;
            // CONF: the exponentials are positive and monotone in the logits, so the largest one marks the arg-max; its bit
            // pattern with the low five bits replaced by 31 - c is compared as an integer (equal values: the lowest class
            // wins).  Dropping five bits can only swap classes whose logits differ by less than 3e-6 relative.
            uint32_t key[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) key[j] = 0;
#pragma unroll kSweep1
            for (int c = 0; c < C; ++c) {
                float2 X01[4], X23[4], q01, q23;
                wmax = fmaxf(wmax, cell_bases_log2(ps[c * 32], ps[c * 32 + to_r], X01[0], X23[0], q01, q23));
#pragma unroll
                for (int q = 1; q < 4; ++q) { X01[q] = __fmul2_rn(X01[q - 1], q01); X23[q] = __fmul2_rn(X23[q - 1], q23); }
#pragma unroll
                for (int q = 0; q < 4; ++q) { Z01[q] = __fadd2_rn(Z01[q], X01[q]); Z23[q] = __fadd2_rn(Z23[q], X23[q]); }
                if (CONF) {
                    const uint32_t tag = 31u - (uint32_t)c;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        key[q] = max(key[q], (__float_as_uint(X01[q].x) & ~31u) | tag);
                        key[4 + q] = max(key[4 + q], (__float_as_uint(X01[q].y) & ~31u) | tag);
                        key[8 + q] = max(key[8 + q], (__float_as_uint(X23[q].x) & ~31u) | tag);
                        key[12 + q] = max(key[12 + q], (__float_as_uint(X23[q].y) & ~31u) | tag);
                    }
                }
            }
            // ---- labels: the four rows' pixels of this cell, a byte each; 0x01 in the byte of a weighted pixel (hv), of a pixel
            // inside the frame (vb) and of one that counts (rem: inside the frame, label below C)
            uint32_t rem[4], hv[4], all = 0x01010101u;
            {
                const uint32_t cols = (cell_valid && n >= 0 ? 0x00000101u : 0u) | (cell_valid && n < w - 1 ? 0x01010000u : 0u);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int Y = 4 * i + 2 + r;
                    labw[r] = __byte_perm(labw[r], __shfl_down_sync(0xffffffffu, labw[r], 1), 0x5432);
                    const uint32_t vb = Y >= 0 && Y < H ? cols : 0u;
                    hv[r] = 0;
                    if (hw1 > 0) { hv[r] = (labw[r] >> 7) & 0x01010101u; labw[r] &= 0x7f7f7f7fu; }
                    const uint32_t t8 = ((labw[r] & 0x7f7f7f7fu) + (uint32_t)(128 - C) * 0x01010101u) | labw[r];   // bit 7: label >= C
                    rem[r] = (~t8 >> 7) & vb;
                    all &= rem[r];
                    if (own_cell) n_bad += __popc(rem[r] ^ vb);
                }
            }
            float zmin = fminf(fminf(Z01[0].x, Z01[0].y), fminf(Z23[0].x, Z23[0].y));
#pragma unroll
            for (int q = 1; q < 4; ++q) zmin = fminf(zmin, fminf(fminf(Z01[q].x, Z01[q].y), fminf(Z23[q].x, Z23[q].y)));
            bool off = !(wmax <= kFastRange) || (cell_valid && !(zmin > 1e-18f));
            // a sum that is not a number passes fminf: all 16 are looked at through their total
            {
                float2 tot = make_float2(0.f, 0.f);
#pragma unroll
                for (int q = 0; q < 4; ++q) tot = __fadd2_rn(tot, __fadd2_rn(Z01[q], Z23[q]));
                off |= cell_valid && !(tot.x + tot.y < INFINITY);
            }
            uint32_t* node = counts + (min(max(i, 0), h - 1) - (y0 - 1)) * F_COLS + (min(max(n, 0), w - 1) - (x0 - 1));
            const int right = min(max(n + 1, 0), w - 1) - min(max(n, 0), w - 1), below = (min(max(i + 1, 0), h - 1) - min(max(i, 0), h - 1)) * F_COLS;
            if (!__any_sync(0xffffffffu, off)) {
                float2 WL01[4], WL23[4], WR01[4], WR23[4];                 // a pixel's weight toward the left / right node column, over Z
                float lz = 0.f;
                if (__all_sync(0xffffffffu, hw1 == 0 && (all == 0x01010101u || !cell_valid))) {
                    // every cell of the warp counts whole (nobody reads the pulls of lanes without a cell)
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float2 r01 = make_float2(rcp_approx(Z01[q].x), rcp_approx(Z01[q].y)), r23 = make_float2(rcp_approx(Z23[q].x), rcp_approx(Z23[q].y));
                        const float fr = (2 * q + 1) * 0.125f;
                        const float2 f2 = make_float2(fr, fr), g2 = make_float2(1.0f - fr, 1.0f - fr);
                        WL01[q] = __fmul2_rn(r01, g2); WL23[q] = __fmul2_rn(r23, g2);
                        WR01[q] = __fmul2_rn(r01, f2); WR23[q] = __fmul2_rn(r23, f2);
                        // sums lie between 1e-18 and C: products of two stay normal
                        lz += lg2_approx(Z01[q].x * Z01[q].y) + lg2_approx(Z23[q].x * Z23[q].y);
                    }
                } else {
                    float wl[16], wr[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const int r = j >> 2, q = j & 3;
                        const float Z = r == 0 ? Z01[q].x : r == 1 ? Z01[q].y : r == 2 ? Z23[q].x : Z23[q].y;
                        const bool counts_j = (rem[r] >> (8 * q)) & 1u;
                        const float fr = (2 * q + 1) * 0.125f;
                        const float wj = ((hv[r] >> (8 * q)) & 1u) ? (float)a.heavy_w : 1.0f;
                        const float rz = counts_j ? rcp_approx(Z) * wj : 0.f;
                        lz += counts_j ? wj * lg2_approx(Z) : 0.f;
                        wl[j] = (fold_l ? 0.f : (fold_r ? 1.0f : 1.0f - fr)) * rz;
                        wr[j] = (fold_r ? 0.f : (fold_l ? 1.0f : fr)) * rz;
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        WL01[q] = make_float2(wl[q], wl[4 + q]); WL23[q] = make_float2(wl[8 + q], wl[12 + q]);
                        WR01[q] = make_float2(wr[q], wr[4 + q]); WR23[q] = make_float2(wr[8 + q], wr[12 + q]);
                    }
                }
                if (CONF) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (own_cell && ((rem[j >> 2] >> (8 * (j & 3))) & 1u))
                            atomicAdd(&hist[((labw[j >> 2] >> (8 * (j & 3))) & 0xffu) * C + (31u - (key[j] & 31u))], 1u);
                }
                // One round per distinct label of the cell (one round for most cells).  The pixels carrying the label pull
                // the four corner nodes with integer weights (row eighths x column eighths, summed by byte-wise dot products);
                // the same four sums weight the label's corner logits in the loss.
                float lsum = 0.f;
                while (rem[0] | rem[1] | rem[2] | rem[3]) {
                    const uint32_t wsel = rem[0] ? labw[0] : rem[1] ? labw[1] : rem[2] ? labw[2] : labw[3];
                    const uint32_t rsel = rem[0] ? rem[0] : rem[1] ? rem[1] : rem[2] ? rem[2] : rem[3];
                    const uint32_t cur = (wsel >> (__ffs(rsel) - 1)) & 0xffu;
                    const uint32_t cur4 = cur * 0x01010101u;
                    uint32_t tl = 0, tr = 0, bl = 0, br = 0;
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        const uint32_t eq = ((0x80808080u - ((labw[r] ^ cur4) & 0x7f7f7f7fu)) >> 7) & rem[r];
                        rem[r] ^= eq;
                        const uint32_t ew = eq + (eq & hv[r]) * (uint32_t)hw1;          // each byte: the pixel's weight (1..5) or 0
                        tl = __dp4a(ew, corner_weights(7 - 2 * r, false), tl);
                        tr = __dp4a(ew, corner_weights(7 - 2 * r, true), tr);
                        bl = __dp4a(ew, corner_weights(2 * r + 1, false), bl);
                        br = __dp4a(ew, corner_weights(2 * r + 1, true), br);
                    }
                    add_counts(node, (int)cur, right, below, tl, tr, bl, br);
                    const float2 L = ps[cur * 32], R = ps[cur * 32 + to_r];
                    lsum = fmaf((float)tl, L.x, fmaf((float)tr, R.x, fmaf((float)bl, L.y, fmaf((float)br, R.y, lsum))));
                }
                if (own_cell) loss = (lz - lsum * (1.0f / 64.0f)) * kLn2;
                // vertical weights of the rows toward the upper / lower node row (clamped borders fold into the inner row)
                float tw[4], bw[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float ly = (2 * r + 1) * 0.125f;
                    tw[r] = i == -1 ? 0.f : (i == h - 1 ? 1.0f : 1.0f - ly);
                    bw[r] = i == h - 1 ? 0.f : (i == -1 ? 1.0f : ly);
                }
                const float2 tw01 = make_float2(tw[0], tw[1]), tw23 = make_float2(tw[2], tw[3]);
                const float2 bw01 = make_float2(bw[0], bw[1]), bw23 = make_float2(bw[2], bw[3]);
                __syncwarp();
                // ---- sweep 2 (packed fp32x2: rows (0,1) and (2,3) side by side): the slots turn from logits into pulls.  The
                // shuffles stand between every lane's reads of a class and its neighbours' writes.
                auto pulls = [&](float2 L, float2 R) {
                    float2 x01, x23, q01, q23, aL01, aL23, aR01, aR23;
                    cell_bases_log2(L, R, x01, x23, q01, q23);
                    cell_row_sums(x01, x23, q01, q23, WL01, WL23, aL01, aL23);
                    cell_row_sums(x01, x23, q01, q23, WR01, WR23, aR01, aR23);
                    // own cell's left part + left cell's right part, per row
                    const float2 hs01 = __fadd2_rn(aL01, make_float2(__shfl_up_sync(0xffffffffu, aR01.x, 1), __shfl_up_sync(0xffffffffu, aR01.y, 1)));
                    const float2 hs23 = __fadd2_rn(aL23, make_float2(__shfl_up_sync(0xffffffffu, aR23.x, 1), __shfl_up_sync(0xffffffffu, aR23.y, 1)));
                    const float2 t2 = __ffma2_rn(hs23, tw23, __fmul2_rn(hs01, tw01));
                    const float2 b2 = __ffma2_rn(hs23, bw23, __fmul2_rn(hs01, bw01));
                    return make_float2(t2.x + t2.y, b2.x + b2.y);
                };
                constexpr int G = sweep2(FORM);                 // classes in flight: all their reads come before the first write
                static_for_groups<C, G>([&](int c0, auto count) {
                    constexpr int N = decltype(count)::value;
                    float2 L[N], R[N], o[N];
#pragma unroll
                    for (int g = 0; g < N; ++g) { L[g] = ps[(c0 + g) * 32]; R[g] = ps[(c0 + g) * 32 + to_r]; }
#pragma unroll
                    for (int g = 0; g < N; ++g) o[g] = pulls(L[g], R[g]);
#pragma unroll
                    for (int g = 0; g < N; ++g) my[(c0 + g) * 32] = o[g];
                });
            } else {
                // ---- slow path: row by row, exact per-pixel maxima; the pulls stay in registers until the slots' logits are done with
                float2 pull[C];
#pragma unroll
                for (int c = 0; c < C; ++c) pull[c] = make_float2(0.f, 0.f);
                for (int r = 0; r < 4; ++r) {
                    const int Y = 4 * i + 2 + r;
                    if (!(Y >= 0 && Y < H)) continue;                      // warp-uniform
                    const float ly = (2 * r + 1) * 0.125f;
                    const uint32_t lab4 = r == 0 ? labw[0] : r == 1 ? labw[1] : r == 2 ? labw[2] : labw[3];
                    const uint32_t rem4 = r == 0 ? rem[0] : r == 1 ? rem[1] : r == 2 ? rem[2] : rem[3];
                    const uint32_t hv4 = r == 0 ? hv[0] : r == 1 ? hv[1] : r == 2 ? hv[2] : hv[3];
                    float ex[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY}, Zs[4] = {0.f, 0.f, 0.f, 0.f};
                    uint32_t arg[4] = {0, 0, 0, 0};
#pragma unroll 3
                    for (int c = 0; c < C; ++c) {
                        float u[4];
                        row_values(ps[c * 32], ps[c * 32 + to_r], ly, u);
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (CONF) { if (u[q] > ex[q]) { ex[q] = u[q]; arg[q] = c; } }
                            else ex[q] = fmaxf(ex[q], u[q]);
                    }
#pragma unroll 3
                    for (int c = 0; c < C; ++c) {
                        float u[4];
                        row_values(ps[c * 32], ps[c * 32 + to_r], ly, u);
#pragma unroll
                        for (int q = 0; q < 4; ++q) Zs[q] += ex2_approx(u[q] - ex[q]);
                    }
                    float wl[4], wr[4];
                    const int wy1 = 2 * r + 1, wy0 = 8 - wy1;              // eighths toward node rows i+1 / i
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int lab = (lab4 >> (8 * q)) & 0xff;
                        float rz = 0.f;
                        if ((rem4 >> (8 * q)) & 1u) {
                            const int iw = ((hv4 >> (8 * q)) & 1u) ? a.heavy_w : 1;
                            rz = rcp_approx(Zs[q]) * (float)iw;
                            if (own_cell) {
                                float u[4];
                                row_values(ps[lab * 32], ps[lab * 32 + to_r], ly, u);
                                loss += (float)iw * (lg2_approx(Zs[q]) - (u[q] - ex[q])) * kLn2;
                                if (CONF) atomicAdd(&hist[lab * C + arg[q]], 1u);
                            }
                            const uint32_t wb = (2 * q + 1) * iw, wa = (7 - 2 * q) * iw;   // eighths toward node columns n+1 / n, times the weight
                            add_counts(node, lab, right, below, wy0 * wa, wy0 * wb, wy1 * wa, wy1 * wb);
                        }
                        const float fr = (2 * q + 1) * 0.125f;
                        wl[q] = (fold_l ? 0.f : (fold_r ? 1.0f : 1.0f - fr)) * rz;
                        wr[q] = (fold_r ? 0.f : (fold_l ? 1.0f : fr)) * rz;
                    }
                    const float twr = i == -1 ? 0.f : (i == h - 1 ? 1.0f : 1.0f - ly), bwr = i == h - 1 ? 0.f : (i == -1 ? 1.0f : ly);
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        float u[4], e[4];
                        row_values(ps[c * 32], ps[c * 32 + to_r], ly, u);
#pragma unroll
                        for (int q = 0; q < 4; ++q) e[q] = ex2_approx(u[q] - ex[q]);
                        const float aL = fmaf(wl[0], e[0], fmaf(wl[1], e[1], fmaf(wl[2], e[2], wl[3] * e[3])));
                        const float aR = fmaf(wr[0], e[0], fmaf(wr[1], e[1], fmaf(wr[2], e[2], wr[3] * e[3])));
                        const float hs = aL + __shfl_up_sync(0xffffffffu, aR, 1);
                        pull[c] = make_float2(fmaf(twr, hs, pull[c].x), fmaf(bwr, hs, pull[c].y));
                    }
                }
                __syncwarp();
#pragma unroll
                for (int c = 0; c < C; ++c) my[c * 32] = pull[c];
            }
        } else if (FORWARD && ok) {                        // a warp below the frame has nothing to take, but says so
            tc::tc_fence_before_sync();
            __syncwarp();
            if (tc::elect_one()) arrive(taken_bar);
        }
        // loss of the tile, fixed order
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
        if (l == 0) red[grp][n_done & 1][wi] = loss;       // (two of them: warps may be one tile ahead of the one that adds)
        if (n_bad) atomicAdd(a.bad, n_bad);
        if (FORWARD && with_grad && ok && n_done > 1) {    // the product of the group's tile before: its gradient has been read
            ok = tc::mbar_wait(grad_bar, n_done & 1, a.err, tc::kWaitDone);
            if (gave_up) ok = false;
        }
        if (!workers_all(grp, ok)) return;                 // uniform over the group: a wait ran out, nothing is written
        if (!FORWARD || k.t >= n_tiles) pdl_launch_dependents();      // the block's last tile: only the epilogue is left
        if (CONF) {                                        // one global update per non-empty counter of the tile
            for (int e = gtid; e < C * C; e += F_WORKERS) {
                const unsigned int v = hist[e];
                if (v) { atomicAdd(a.conf + (int64_t)s * a.conf_stream_stride + e, (unsigned long long)v); hist[e] = 0; }
            }
        }
        if (FORWARD && with_grad && n_done > 1) store_gradient(before);
        before = now;
        // ---- node row y0-1+wi (warps 1..FN_Y): own upper pulls + lower pulls of the warp above - counts
        const bool node_ok = wi >= 1 && i < h && node_owned;
        float v[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) v[c] = 0.f;
        if (node_ok) {
            const float2* above = my - C * 32;
            uint32_t* mine = counts + wi * F_COLS + l;
#pragma unroll
            for (int c = 0; c < C; c += 2) {
                const uint32_t ct = mine[(c >> 1) * kNodes];
                mine[(c >> 1) * kNodes] = 0;               // ready for the next tile (words outside the owned nodes are never read)
                v[c] = (my[c * 32].x + above[c * 32].y - (float)(ct & 0xffffu) * (1.0f / 64.0f)) * invP;
                if (c + 1 < C) v[c + 1] = (my[(c + 1) * 32].x + above[(c + 1) * 32].y - (float)(ct >> 16) * (1.0f / 64.0f)) * invP;
            }
            if (a.dz) {
                float* dzp = a.dz + (int64_t)s * C * a.dz_plane + (int64_t)i * a.dz_pitch + n;
#pragma unroll
                for (int c = 0; c < C; ++c) dzp[(int64_t)c * a.dz_plane] = v[c];
            }
            if (a.dz_bf16) {
                bf16* dzb = a.dz_bf16 + (int64_t)s * kClassPad * a.dz_bf16_pitch + (int64_t)i * w + n;
#pragma unroll
                for (int c = 0; c < C; ++c) dzb[(int64_t)c * a.dz_bf16_pitch] = __float2bfloat16_rn(v[c]);
            }
        }
        if (FORWARD && with_grad) {
            // bf16, K-major with the 128-byte swizzle: [two node rows][class][64 nodes]
            if (wi >= 1) {
                uint8_t* to = smem + Smem::kGradAt + grp * Smem::kGrad + ((wi - 1) >> 1) * kWBytes + (l & 7) * 2;
                const uint32_t chunk = (((wi - 1) & 1) * 4 + (l >> 3)) * 16;
#pragma unroll
                for (int c = 0; c < C; ++c) *reinterpret_cast<bf16*>(to + c * 128 + (chunk ^ ((c & 7) * 16))) = __float2bfloat16_rn(v[c]);
            }
            tc::fence_async_shared();                      // read by way of the async proxy
            __syncwarp();
            if (tc::elect_one()) arrive(dz_bar);
        }
        // bias-gradient partial of the tile.  Lane reduce-scatter inside each warp (31 exchanges: at distance o a lane keeps the
        // half of its values whose class has bit o equal to its own lane bit and adds the partner's), after which lane c holds
        // class c; then the warps' sums are added in warp order.  Fixed order throughout.
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const bool hi = l & o;
#pragma unroll
            for (int j = 0; j < o; ++j) {
                const float send = hi ? v[j] : v[j + o];
                const float keep = hi ? v[j + o] : v[j];
                v[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        wsum[warp][l] = v[0];
        workers_sync(grp);
        if (gtid < C) {
            float q = 0.f;
#pragma unroll
            for (int r = 1; r < F_WARPS; ++r) q += wsum[grp * F_WARPS + r][gtid];
            a.db_part[((int64_t)s * per_stream + blk) * C + gtid] = q;
        }
        if (gtid == 32) {
            float q = 0.f;
            for (int r = 0; r < F_WARPS; ++r) q += red[grp][n_done & 1][r];
            a.loss_part[(int64_t)s * per_stream + blk] = q;
        }
        if (kGroups > 1) next(k);                          // the other group's
    }
    if (FORWARD && with_grad && n_done > 0) {
        if (tc::mbar_wait(grad_bar, (n_done - 1) & 1, a.err, tc::kWaitDone) && !gave_up) store_gradient(before);
    }
}

// A block that was launched with fewer registers than its warps ask for would wait for them forever
template <int C, bool CONF, int FORM>
cudaError_t prepare_fwd_ce_form()
{
    const void* kernel = (const void*)fwd_ce_kernel<C, CONF, FORM>;
    cudaError_t e = allow_shared_memory(kernel);
    cudaFuncAttributes at;
    if (FORM != kStored && e == cudaSuccess) e = cudaFuncGetAttributes(&at, kernel);
    return e != cudaSuccess ? e : FORM != kStored && at.numRegs < form_launch_regs(FORM) ? cudaErrorInvalidConfiguration : cudaSuccess;
}

template <int C, int FORM>
cudaError_t prepare_fwd_ce_both()
{
    const cudaError_t e = prepare_fwd_ce_form<C, false, FORM>();
    return e != cudaSuccess ? e : prepare_fwd_ce_form<C, true, FORM>();
}
// The kernels that a context may launch: on stored logits, and its form with an own forward (each that is touched is loaded, 0.2 ms)
template <int C>
cudaError_t prepare_fwd_ce_as(bool own_forward, bool with_gradient, int tiles, int n_sms)
{
    const cudaError_t e = prepare_fwd_ce_both<C, kStored>();
    if (e != cudaSuccess || !own_forward) return e;
    if constexpr (classifier_gradient_fits(C)) {
        if (!with_gradient) return prepare_fwd_ce_both<C, kOneGroup>();
        if (tiles <= n_sms) return prepare_fwd_ce_both<C, kLoneGroup>();
    }
    return prepare_fwd_ce_both<C, kTwoGroups>();
}

template <int C, bool CONF, int FORM>
void launch_fwd_ce_as(const UpsampleCeArgs& a, const CUtensorMap& x_map, const CUtensorMap& w_map, const CUtensorMap& row_map, cudaStream_t s)
{
    using Smem = FwdCeSmem<C, CONF, FORM>;
    const int tx = (a.w + FN_X - 1) / FN_X, ty = (a.h + FN_Y - 1) / FN_Y, tiles = tx * ty * a.S, resident = FORM == kStored ? tiles : a.n_sms * (FORM == kOneGroup ? 2 : 1);
    const size_t smem = one_per_sm(Smem::kBytes, tiles, a.n_sms);
    launch_early(a.chain_early != 0 || a.x_early != 0, fwd_ce_kernel<C, CONF, FORM>, dim3(tiles < resident ? tiles : resident), dim3(form_threads(FORM)), smem, s, a, tx, ty, x_map, w_map, row_map);
}

template <int C, int FORM>
void launch_fwd_ce_form(const UpsampleCeArgs& a, const CUtensorMap& x_map, const CUtensorMap& w_map, const CUtensorMap& row_map, cudaStream_t s)
{
    if (a.conf) launch_fwd_ce_as<C, true, FORM>(a, x_map, w_map, row_map, s);
    else launch_fwd_ce_as<C, false, FORM>(a, x_map, w_map, row_map, s);
}

template <int C, bool FORWARD>
void launch_fwd_ce_of(const UpsampleCeArgs& a, const CUtensorMap& x_map, const CUtensorMap& w_map, const CUtensorMap& row_map, cudaStream_t s)
{
    if constexpr (!FORWARD) launch_fwd_ce_form<C, kStored>(a, x_map, w_map, row_map, s);
    else {
        if constexpr (!loss_kernel_two_groups(C, false)) if (!loss_kernel_two_groups(C, a.w_part != nullptr)) return launch_fwd_ce_form<C, kOneGroup>(a, x_map, w_map, row_map, s);
        // at most a tile per SM: us a step, two groups / a lone one, 128 channels on 90 x 160 (78 tiles) 14.8 / 14.6, 256 channels on 45 x 70
        // (21 tiles) 16.8 / 16.4, with 4 classes 12.2 / 11.5.  With more tiles an SM has work for two groups.
        if constexpr (classifier_gradient_fits(C))
            if (upsample_ce_few_blocks(a.h, a.w) * a.S <= a.n_sms) return launch_fwd_ce_form<C, kLoneGroup>(a, x_map, w_map, row_map, s);
        launch_fwd_ce_form<C, kTwoGroups>(a, x_map, w_map, row_map, s);
    }
}

}  // namespace

// The kernels of one class count
struct FwdCeKernels {
    cudaError_t (*prepare)(bool own_forward, bool with_gradient, int tiles, int n_sms);
    void (*launch[2])(const UpsampleCeArgs& a, const CUtensorMap& x_map, const CUtensorMap& w_map, const CUtensorMap& row_map, cudaStream_t s);   // stored logits, own forward
};

// ... of class count `n`, one of FIRST + I...
template <int FIRST, int... I>
static FwdCeKernels fwd_ce_kernels_of(int n, std::integer_sequence<int, I...>)
{
    static const FwdCeKernels all[] = {{prepare_fwd_ce_as<FIRST + I>, {launch_fwd_ce_of<FIRST + I, false>, launch_fwd_ce_of<FIRST + I, true>}}...};
    return all[n - FIRST];
}

// one file each, so that they compile side by side
constexpr int kFwdCeLast[] = {12, 18, 23, 28, 32};      // the last class count of each file; the first one begins at 2
FwdCeKernels fwd_ce_kernels_0(int n);
FwdCeKernels fwd_ce_kernels_1(int n);
FwdCeKernels fwd_ce_kernels_2(int n);
FwdCeKernels fwd_ce_kernels_3(int n);
FwdCeKernels fwd_ce_kernels_4(int n);

}  // namespace st
