// MLP quality head (Section 4.2) on the tensor cores, for bf16 heads: the first layer U[N,h] = X[N,d] x W1[h,d]^T is
// a dense contraction, so it runs as tcgen05 MMAs fed by TMA, and the rest of the head (bias, exact GELU, w2 dot
// product, sigmoid, bin, posterior look-up: Appendix A.4) is finished in the same kernel.
//
//   pack_rows_kernel      copies the N scored rows (one per rollout, anywhere in the hidden buffer) into a packed
//                         [N,d] block so that TMA can tile them; skipped when the rows are already evenly strided.
//                         (Fetching the rows in place from inside the contraction, four warps of 16-byte cp.async
//                         copies into the swizzled stage layout, was built and measured: correct, but the
//                         load/store path holds about 20 KB in flight per SM against the ring's 192 KB by TMA, and
//                         every block of a row tile fetches the same rows: 18.5 us per call against 14.6 us.)
//   score_mlp_tc_kernel   one block per (64 or 128 rollouts x 64 hidden units, or 128 x 128); shared memory is one ring of stages
//                         (the tile's 64 columns of X and of W1 per K step of 64), filled by four TMA producer threads,
//                         two for X and two for W1, on alternate K steps (one thread for all of W1 takes 300 cycles a step:
//                         N = 2,048, d = 2,048, h = 256, rows in place 8.7 -> 12.6 us).  Two (tiles of 128) or four (64) issuing
//                         warps take the K steps round robin: one warp's wait -> four MMAs -> commit round costs nearly 500
//                         cycles, the MMAs of a 128 x 64 x 64 step 128, and a step's operands come in in about 290.  K step ks
//                         goes to accumulator ks mod 4.  The ring's length is a multiple of the number of issuers, so that a
//                         stage always belongs to the same one: a parity wait cannot tell a round from the one before the last.
//                         Epilogue by all sixteen warps (with eight, two a scheduler, the chains of erff wait for themselves:
//                         3.0 us for 64 units): thread = rollout x a quarter of the tile's hidden units; accumulators added in
//                         index order, then sum_j w2_j gelu(u_j + b1_j) over 32 units in index order, two such sums added
//                         low + high -> a partial sum per 64 units and rollout, whatever the tile's width.
//                         The blocks of a row tile are a cluster and put their partial sums into the first block's shared
//                         memory, which adds them in index order, adds b2 and applies the probability map.  Without clusters
//                         (more than eight blocks of 128 hidden units, or where clusters would take more waves) the partial sums
//                         go through global memory and the last block to arrive (a counter per row tile) adds them.  The result
//                         does not depend on block order, nor on which of the two it was.  Per call of 20 in a graph, partial
//                         sums through global memory -> cluster: N = 2,048, d = 2,048, h = 256 13.5 -> 12.0 us (rows in place
//                         10.3 -> 8.7); 4,096, 4,096, 512 29.1 -> 26.5; 394, 1,664, 256 10.8 -> 9.3; 32, 256, 64 7.1 -> 6.0.
//   What the N = 2,048 call spent before the clusters (in-kernel stamps): 0.7 us to the first stage, 3.7 for 32 K steps (192 KB in flight
//   per SM and a copy's latency of 0.85 us), 1.6 of erff (45 instructions a unit and rollout), 2.2 in counting and adding up.
//   Packing inside this kernel, each block of a cluster a share of the row tile and the contraction following chunk by chunk,
//   was built and measured: 17.7 us, because every chunk's report waits 2 us for the stores before it.
// Every wait is bounded; on expiry the block records ARROL_DEV_WAIT_EXPIRED, drains and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include "arrol_internal.h"
#include "score_common.cuh"
#include "tc_common.cuh"

namespace {

constexpr int SUB_H = 64;                    // hidden units per partial sum: the same for every tile width
constexpr int S_ACCS = 4;                    // accumulators; K step ks goes to accumulator ks % 4
constexpr int S_PRODUCERS = 2;               // TMA producer threads per operand (lane 0 of the first warps)
constexpr int S_PRODUCER_WARPS = 4;          // warps before the issuers
constexpr int S_HELPER_WARP0 = 8;            // warps without a role in the contraction fetch what the epilogue needs
constexpr int S_HELPER_WARPS = 8;
constexpr int S_WARPS = S_HELPER_WARP0 + S_HELPER_WARPS, S_THREADS = S_WARPS * 32;     // the epilogue is all warps' work
constexpr uint32_t DRAIN_LIMIT = 1u << 16;   // tries per wait of a producer that gave up, for copies in flight
constexpr int MAX_SUBS = 16;                 // partial sums of a row tile whose blocks form a cluster: 8 blocks of 128 hidden units
// barriers, tensor-memory slot, flags | b1 and w2 of the tile, sums over 16 hidden units | sums over 32
// | the training step's ds of the tile's rollouts, sums over its warps
constexpr int S_TAIL_BYTES = 2560 + 2 * MAX_SUBS * 128 * 4 + 512 + 256;
constexpr int MAX_ROWS = 128;
// by tile: rollouts (MMA M: 64 or 128) x hidden units (MMA N: 64 or 128); 64 x 64, 128 x 64 and 128 x 128
template <int ROWS> __host__ __device__ constexpr int a_bytes() { return ROWS * BK * 2; }
template <int SBN, int ROWS> __host__ __device__ constexpr int ring_stages() { return SBN == 128 ? 6 : ROWS == 128 ? 8 : 12; }
template <int SBN> __host__ __device__ constexpr int issuers() { return SBN == 64 ? 4 : 2; }
template <int SBN, int ROWS> __host__ __device__ constexpr int stage_bytes() { return a_bytes<ROWS>() + SBN * BK * 2; }
template <int SBN, int ROWS> __host__ __device__ constexpr size_t smem_bytes() {
    return (size_t)ring_stages<SBN, ROWS>() * stage_bytes<SBN, ROWS>() + 1024 + S_TAIL_BYTES;
}

// one warp per 4 KB of a row (a grid row per slice, so that no warp divides): 16-byte copies, all of its loads in flight
// before the first store
constexpr int PACK_VECS = 256;
__global__ void __launch_bounds__(128)
pack_rows_kernel(const __nv_bfloat16* __restrict__ hidden, int64_t row_stride, const int64_t* __restrict__ row_index,
                 int N, int d, __nv_bfloat16* __restrict__ out, int64_t source_rows, uint32_t* d_status) {
    pdl_launch_dependents();
    pdl_wait();
    hidden = pdl_acquire(hidden); row_index = pdl_acquire(row_index);
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const int c0 = blockIdx.y * PACK_VECS + lane;
    if (i >= N) return;
    const int64_t row = row_index[i];
    const uint4* src = reinterpret_cast<const uint4*>(hidden + row * row_stride);
    uint4* dst = reinterpret_cast<uint4*>(out + (int64_t)i * d);
    const int nvec = d / 8;
    // outside the caller's buffer: never read, packed as zeros
    const bool read = !(source_rows > 0 && (row < 0 || row >= source_rows));
    if (!read && c0 == 0) atomicOr(d_status, ARROL_DEV_BAD_INDEX);
    uint4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = read && c0 + 32 * u < nvec ? __ldg(src + c0 + 32 * u) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int u = 0; u < 8; ++u)
        if (c0 + 32 * u < nvec) dst[c0 + 32 * u] = v[u];
}

struct ScoreTcParams {
    int N, h;
    int k_steps;                       // ceil(d / 64)
    const __nv_bfloat16* b1;           // [h] or NULL
    const __nv_bfloat16* w2;           // [h]
    const __nv_bfloat16* b2;           // [1] or NULL
    float* partial;                    // PARTIALS: [ceil(h / 64)][N]
    float* u_out;                      // [N][h] pre-activations (bias included) for the head training step, or NULL
    uint32_t* counters;                // [row tiles], zero between calls
    int B;
    const float* q_lut;
    float* score;
    float* prob;
    int32_t* bin;
    float* q;
    uint32_t* d_status;
    // TRAIN
    const float* rewards;
    const uint8_t* mask;               // or NULL
    __nv_bfloat16* du_hi;              // [N][h], du as the sum of two bf16 planes
    __nv_bfloat16* du_lo;
    float* tile_sums;                  // [2][row tiles][h]: sums of ds gelu(u) and of du over a tile's rollouts
    double* tile_loss;                 // [2][row tiles]: sums of the losses, divided by their number, and of ds
};

// PARTIALS: a row tile's blocks are on their own; the scores are finished through global memory.  SCORES: the blocks of a row tile
// (gridDim.y of them) are a cluster and finish the scores among themselves.  TRAIN: the head training step's forward and all
// of its backward but the dW1 contraction: as SCORES, but every block gets all partial sums, forms the scores' gradients ds and
// finishes its own hidden units: du = ds w2 gelu'(u), and the sums over the tile's rollouts that dw2 and db1 are made of, which the
// dW1 kernel adds up while it waits for its contraction.  Both addends go to the operand ring's shared memory, [unit][rollout], where
// the sums over rollouts are read along rows.  A kernel of its own with u through global memory between took 9.4 us at N = 2,048,
// h = 256 (ncu).
enum Mode { PARTIALS, SCORES, TRAIN };
template <int SBN, Mode MODE, int ROWS>
__global__ void __launch_bounds__(S_THREADS, 1)
score_mlp_tc_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                    const ScoreTcParams p) {
    constexpr int TM = ROWS, A_BYTES = a_bytes<ROWS>();
    constexpr int STAGES = ring_stages<SBN, ROWS>(), STAGE_BYTES = stage_bytes<SBN, ROWS>(), SB_BYTES = SBN * BK * 2;
    constexpr int ISSUERS = issuers<SBN>();
    static_assert(STAGES % ISSUERS == 0 && S_ACCS % ISSUERS == 0 && STAGES % S_PRODUCERS == 0,
                  "a stage and an accumulator belong to one issuer, a stage to one producer");
    constexpr int S_TMEM_COLS = S_ACCS * SBN;                    // a power of two >= 32
    constexpr bool CLUSTER = MODE != PARTIALS;
    constexpr int PITCH = TM == 128 ? TM : TM + 2;               // of the training step's planes: lanes l and l + 16 on different banks
    static_assert(2 * SBN * PITCH * 4 <= STAGES * STAGE_BYTES, "both planes fit the stages");
    static_assert(TM == 128 || (SBN == 64 && MODE != PARTIALS), "tiles of 64 rollouts: narrow ones, in clusters");
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* stage_a = smem;
    uint8_t* stage_b = smem + (size_t)STAGES * A_BYTES;
    uint8_t* tail = smem + (size_t)STAGES * STAGE_BYTES;
    uint64_t* full = reinterpret_cast<uint64_t*>(tail);          // [STAGES] producers -> MMA
    uint64_t* empty = full + STAGES;                             // [STAGES] MMA -> producers
    uint64_t* acc_full = empty + STAGES;                         // [1] every MMA of the block has finished
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    volatile uint32_t* is_last = tmem_slot + 2;
    float* b1_s = reinterpret_cast<float*>(tail + 512);          // [SBN]
    float* w2_s = reinterpret_cast<float*>(tail + 1024);         // [SBN]
    float* half_s = reinterpret_cast<float*>(tail + 1536);       // [2][TM] sums over 16 hidden units of a tile of 64
    float* runs_s = reinterpret_cast<float*>(tail + 2560);       // [2 MAX_SUBS][TM] sums over 32 (of the row tile in the first block of a
                                                                 // cluster; TRAIN: in every block)
    float* ds_s = runs_s + 2 * MAX_SUBS * MAX_ROWS;                    // [TM]
    double* warp_d = reinterpret_cast<double*>(ds_s + TM);       // [2][4]
    int* warp_n = reinterpret_cast<int*>(warp_d + 8);            // [S_HELPER_WARPS]
    float* gelu_s = reinterpret_cast<float*>(smem);              // [SBN][PITCH] ds gelu(u), once every MMA has finished
    float* du_s = gelu_s + SBN * PITCH;                          // [SBN][PITCH]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * TM, j0 = blockIdx.y * SBN;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 2); mbar_init(&empty[s], 1); }
        mbar_init(acc_full, ISSUERS);
        *abort_flag = 0u;
        *is_last = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_w) : "memory");
    }
    if (warp == S_PRODUCER_WARPS) {         // first MMA warp owns the tensor-memory allocation
        tcgen05_alloc(tmem_slot, S_TMEM_COLS);
        tcgen05_relinquish();
    }
    tcgen05_fence_before();
    __syncthreads();
    if constexpr (CLUSTER) cluster_sync_all();      // the other blocks' barriers exist before anything arrives on them
    tcgen05_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_launch_dependents();
    pdl_wait();                  // set-up above overlaps the previous kernel; global memory is read from here on

    bool labelled = false;       // TRAIN: of rollout threadIdx.x - 256 of the tile
    float reward = 0.f;
    // K step ks uses stage ks % STAGES in round ks / STAGES of the ring, issuer ks % ISSUERS and accumulator ks % S_ACCS.
    if (warp < S_PRODUCER_WARPS) {
        if (lane == 0) {         // two threads for the rows, two for W1, on alternate K steps
            const bool rows = warp < S_PRODUCERS;
            int last = -1;
            bool ok = true;
            for (int ks = warp % S_PRODUCERS; ks < p.k_steps; ks += S_PRODUCERS) {
                const int st = ks % STAGES;
                const uint32_t round = (uint32_t)(ks / STAGES);
                if (!mbar_wait(&empty[st], (round & 1u) ^ 1u, abort_flag)) { ok = false; break; }
                if (rows) {
                    mbar_expect_tx(&full[st], A_BYTES);
                    tma_load_2d(stage_a + (size_t)st * A_BYTES, &map_x, ks * BK, m0, &full[st]);
                } else {
                    mbar_expect_tx(&full[st], SB_BYTES);
                    tma_load_2d(stage_b + (size_t)st * SB_BYTES, &map_w, ks * BK, j0, &full[st]);
                }
                last = ks;
            }
            if (!ok || *abort_flag) {   // let this thread's copies in flight land before the block's shared memory goes away
                for (int ks = last; ks >= 0 && ks > last - STAGES; ks -= S_PRODUCERS)
                    for (uint32_t it = 0; it < DRAIN_LIMIT; ++it)       // (the stage's other operand may never have been asked for)
                        if (mbar_try_wait(&full[ks % STAGES], (uint32_t)(ks / STAGES) & 1u)) break;
            }
        }
    } else if (warp < S_HELPER_WARP0) {
        const int r = warp - S_PRODUCER_WARPS;
        if (r < ISSUERS) {
            const uint32_t a0 = smem_u32(stage_a), b0 = smem_u32(stage_b);
            constexpr uint32_t idesc = make_idesc(TM, SBN);
            bool ok = true;
            for (int ks = r; ks < p.k_steps; ks += ISSUERS) {
                const int st = ks % STAGES;
                if (!mbar_wait_warp(&full[st], (uint32_t)(ks / STAGES) & 1u, abort_flag)) { ok = false; break; }
                tcgen05_fence_after();
                const uint64_t a_desc = make_smem_desc(a0 + st * A_BYTES);
                const uint64_t b_desc = make_smem_desc(b0 + st * SB_BYTES);
                const uint32_t d_tmem = tmem_base + (uint32_t)((ks % S_ACCS) * SBN);
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < BK / UMMA_K; ++k)
                        tcgen05_mma_bf16(d_tmem, a_desc + (uint64_t)(2 * k), b_desc + (uint64_t)(2 * k), idesc,
                                         (ks >= S_ACCS || k > 0) ? 1u : 0u);
                    tcgen05_commit(&empty[st]);
                }
                __syncwarp();
            }
            // Arrives once every MMA issued by this warp has finished: publishes its accumulators on the normal path, and on the
            // give-up path it is what this warp waits for before shared and tensor memory go away.
            if (elect_one()) tcgen05_commit(acc_full);
            __syncwarp();
            if (!ok || *abort_flag)
                for (uint32_t it = 0; it < SPIN_LIMIT; ++it)
                    if (mbar_try_wait(acc_full, 0u)) break;
        }
    } else {
        const int e = threadIdx.x - S_HELPER_WARP0 * 32;
        if (e < SBN) {          // the tile's slice of b1 and w2, zero past h so that padded columns add nothing
            const int j = j0 + e;
            b1_s[e] = (j < p.h && p.b1) ? __bfloat162float(pdl_acquire(p.b1)[j]) : 0.f;
            w2_s[e] = (j < p.h) ? __bfloat162float(pdl_acquire(p.w2)[j]) : 0.f;
        }
        if constexpr (MODE == TRAIN) {      // every block counts the labelled rollouts itself
            const uint8_t* mask = pdl_acquire(p.mask);
            if (e < TM && m0 + e < p.N) {
                labelled = !mask || mask[m0 + e];
                reward = pdl_acquire(p.rewards)[m0 + e];
            }
            const int c = __reduce_add_sync(0xffffffffu, mask ? count_labelled(mask, p.N, e, S_HELPER_WARPS * 32) : 0);
            if (lane == 0) warp_n[warp - S_HELPER_WARP0] = c;
        }
    }
    __syncwarp();

    // Epilogue: all warps; thread = rollout x UNITS hidden units.  128 rollouts: accumulator row r is tensor-memory lane r, a warp reads
    // the lanes of its number mod 4 and a quarter of the columns.  64 rollouts: row r is lane 32 (r / 16) + r mod 16, so that the upper
    // half of a warp's lanes holds nothing; it takes over the upper half of the warp's columns.
    constexpr int COLS = SBN / 4, UNITS = TM == 128 ? COLS : COLS / 2;
    const int quarter = warp & 3, cg = warp >> 2;
    const bool upper = TM == 64 && lane >= 16;
    const int r_tile = TM == 128 ? quarter * 32 + lane : quarter * 16 + (lane & 15), m = m0 + r_tile;
    const int unit0 = cg * COLS + (upper ? UNITS : 0);                     // of this thread's, in the tile
    const int used_accs = p.k_steps < S_ACCS ? p.k_steps : S_ACCS;         // an accumulator without K steps holds nothing
    bool ok = mbar_wait(acc_full, 0u, abort_flag);
    ok = __all_sync(0xffffffffu, ok && !*abort_flag) != 0;
    __syncthreads();                        // b1_s, w2_s
    float v[UNITS], cdf[UNITS];             // u = pre-activations, then gelu(u); 2 Phi(u)
    {
        float sum[COLS];
        if (ok) {
            tcgen05_fence_after();
            const uint32_t at = tmem_base + ((uint32_t)(quarter * 32) << 16) + cg * COLS;
            tcgen05_ld_32(at, sum);
            for (int a = 1; a < used_accs; ++a) {      // fixed order: ((acc0 + acc1) + acc2) + acc3
                float w[COLS];
                tcgen05_ld_32(at + a * SBN, w);
#pragma unroll
                for (int j = 0; j < COLS; ++j) sum[j] += w[j];
            }
        } else {
#pragma unroll
            for (int j = 0; j < COLS; ++j) sum[j] = 0.f;
        }
#pragma unroll
        for (int j = 0; j < UNITS; ++j) {
            v[j] = sum[j];
            if constexpr (TM == 64) {
                const float other = __shfl_sync(0xffffffffu, sum[UNITS + j], lane & 15);
                if (upper) v[j] = other;
            }
        }
    }
    float slope[MODE == TRAIN ? UNITS : 1];        // gelu'(u) w2
#pragma unroll
    for (int j = 0; j < UNITS; ++j) {
        const float u = v[j] + b1_s[unit0 + j];
        v[j] = u;
        cdf[j] = 1.0f + erff(u * 0.70710678118654752440f);
    }
    if constexpr (MODE == PARTIALS) {
        if (p.u_out && m < p.N) {
            float* urow = p.u_out + (int64_t)m * p.h + j0 + unit0;
#pragma unroll
            for (int j = 0; j < UNITS; j += 4)      // h % 4 == 0: a float4 never straddles the edge
                if (j0 + unit0 + j < p.h) *reinterpret_cast<float4*>(urow + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        }
    }
    // sum_j w2_j gelu(u_j) over 32 hidden units in index order; two of these, low + high, make a partial sum.  Of a tile of 64 two
    // threads (four where a tile has 64 rollouts) have a part each, and the next one goes on where the one before ends.
    const float* w2 = w2_s + unit0;
    auto go_on = [&](float part) {
        auto units = [&](float start) {
#pragma unroll
            for (int j = 0; j < UNITS; ++j) start = fmaf(w2[j], 0.5f * v[j] * cdf[j], start);
            return start;
        };
        part = units(part);
        if constexpr (TM == 64) part = units(__shfl_sync(0xffffffffu, part, lane & 15));     // the upper lanes' after the lower ones'
        return part;
    };
    const bool ends = TM == 128 || upper;       // this thread's part is the last one of its warp
    float part = 0.f;
    if constexpr (SBN == 64) {
        if ((cg & 1) == 0) {
            part = go_on(0.f);
            if (ends) half_s[(cg >> 1) * TM + r_tile] = part;
        }
        __syncthreads();
        if ((cg & 1) == 1) part = half_s[(cg >> 1) * TM + r_tile];
    }
    if (SBN == 128 || (cg & 1) == 1) {
        part = go_on(part);
        const int run = SBN == 128 ? cg : cg >> 1;                       // of 32 hidden units, in the tile
        const int all = MODE == PARTIALS ? run : (int)blockIdx.y * (SBN / 32) + run;
        if (ends && (MODE == PARTIALS || (all >> 1) * SUB_H < p.h)) {
            const uint32_t to = smem_u32(&runs_s[all * TM + r_tile]);
            if constexpr (MODE == PARTIALS) runs_s[all * TM + r_tile] = part;
            if constexpr (MODE == SCORES) st_shared_cluster_f32(map_to_cta(to, 0u), part);
            if constexpr (MODE == TRAIN)
                for (uint32_t b = 0; b < gridDim.y; ++b) st_shared_cluster_f32(map_to_cta(to, b), part);
        }
    }

    tcgen05_fence_before();
    if constexpr (MODE == PARTIALS) {
        __syncthreads();
        // The counter protocol runs whatever happened above, so the counters are back at zero after every launch
        // (after an expired wait the scores of the call are not meaningful and the status word says so).
        const int sub = (int)blockIdx.y * (SBN / SUB_H) + cg;
        if (cg < SBN / SUB_H && m < p.N && sub * SUB_H < p.h)
            p.partial[(int64_t)sub * p.N + m] = runs_s[2 * cg * TM + r_tile] + runs_s[(2 * cg + 1) * TM + r_tile];
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            const uint32_t done = atomicAdd(&p.counters[blockIdx.x], 1u);
            if (done == gridDim.y - 1) {
                *is_last = 1u;
                p.counters[blockIdx.x] = 0u;    // every block of this row tile has arrived: ready for the next call
            }
        }
        __syncthreads();
        if (*is_last && cg == 0 && m < p.N) {
            __threadfence();
            float s = 0.f;
            for (int t = 0; t * SUB_H < p.h; ++t) s += __ldcg(&p.partial[(int64_t)t * p.N + m]);
            if (p.b2) s += __bfloat162float(p.b2[0]);
            probability_map(s, m, p.B, p.q_lut, p.score, p.prob, p.bin, p.q);
        }
    } else {
        cluster_arrive();
        if constexpr (MODE == TRAIN) {          // what needs no score is done while the partial sums are on their way
#pragma unroll
            for (int j = 0; j < UNITS; ++j) {
                const float u = v[j], half_cdf = 0.5f * cdf[j];
                slope[j] = w2[j] * (half_cdf + u * (expf(-0.5f * u * u) * 0.39894228040143267794f));
                v[j] = u * half_cdf;
            }
        }
        cluster_wait();             // the partial sums are there; nobody's shared memory is written from here on
    }
    auto score_of = [&](int r) {
        float s = 0.f;
        for (int t = 0; t * SUB_H < p.h; ++t) s += runs_s[2 * t * TM + r] + runs_s[(2 * t + 1) * TM + r];
        return p.b2 ? s + __bfloat162float(pdl_acquire(p.b2)[0]) : s;
    };
    if constexpr (MODE == SCORES) {
        if (blockIdx.y == 0 && cg == 0 && !upper && m < p.N)
            probability_map(score_of(r_tile), m, p.B, pdl_acquire(p.q_lut), p.score, p.prob, p.bin, p.q);
    }
    if constexpr (MODE == TRAIN) {
        const bool live = m < p.N;
        const int labels = warp - S_HELPER_WARP0;                        // the first of these warps have the labels
        if (labels >= 0 && labels < TM / 32) {
            const int r = labels * 32 + lane;
            int n = p.N;
            if (p.mask) {
                n = 0;
#pragma unroll
                for (int w = 0; w < S_HELPER_WARPS; ++w) n += warp_n[w];
            }
            double l = 0.0, sd = 0.0;
            float ds = 0.f;
            if (labelled) {
                const float s = score_of(r);
                const float y = reward > 0.5f ? 1.f : 0.f;
                ds = (1.0f / (1.0f + expf(-s)) - y) / (float)n;
                sd = (double)ds;
                if (blockIdx.y == 0) l = (double)((s > 0.f ? s + log1pf(expf(-s)) : log1pf(expf(s))) - y * s);
            }
            ds_s[r] = ds;
            if (blockIdx.y == 0) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    l += __shfl_xor_sync(0xffffffffu, l, o);
                    sd += __shfl_xor_sync(0xffffffffu, sd, o);
                }
                if (lane == 0) { warp_d[labels] = n > 0 ? l / (double)n : 0.0; warp_d[4 + labels] = sd; }
            }
        }
        __syncthreads();
        if (blockIdx.y == 0 && threadIdx.x < 2) {
            const double* d = warp_d + 4 * threadIdx.x;
            p.tile_loss[threadIdx.x * gridDim.x + blockIdx.x] = TM == 128 ? ((d[0] + d[1]) + d[2]) + d[3] : d[0] + d[1];
        }
        const float g = ds_s[r_tile];
        const int64_t out = (int64_t)m * p.h + j0 + unit0;
#pragma unroll
        for (int jj = 0; jj < UNITS; jj += 8) {
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float d_u = g * slope[jj + k];
                const __nv_bfloat16 top = __float2bfloat16_rn(d_u);
                const uint32_t h16 = __bfloat16_as_ushort(top), l16 = __bfloat16_as_ushort(__float2bfloat16_rn(d_u - __bfloat162float(top)));
                hi[k >> 1] = (k & 1) ? hi[k >> 1] | h16 << 16 : h16;
                lo[k >> 1] = (k & 1) ? lo[k >> 1] | l16 << 16 : l16;
                gelu_s[(unit0 + jj + k) * PITCH + r_tile] = live ? g * v[jj + k] : 0.f;       // rows past N: zeros, whatever b1 made of them
                du_s[(unit0 + jj + k) * PITCH + r_tile] = live ? d_u : 0.f;
            }
            if (live && j0 + unit0 + jj < p.h) {                       // h % 8 == 0
                *reinterpret_cast<uint4*>(p.du_hi + out + jj) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                *reinterpret_cast<uint4*>(p.du_lo + out + jj) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            }
        }
        __syncthreads();
        constexpr int ABREAST = 4;              // a warp per hidden unit, four of them side by side
        for (int j = ABREAST * warp; j < SBN && j0 + j < p.h; j += ABREAST * S_WARPS) {
            float sum[2 * ABREAST];
#pragma unroll
            for (int i = 0; i < ABREAST; ++i) {
                const float* a = gelu_s + (j + i) * PITCH + lane;
                const float* b = du_s + (j + i) * PITCH + lane;
                sum[2 * i] = a[0] + a[32];
                sum[2 * i + 1] = b[0] + b[32];
                if constexpr (TM == 128) { sum[2 * i] += a[64] + a[96]; sum[2 * i + 1] += b[64] + b[96]; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int i = 0; i < 2 * ABREAST; ++i) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
            if (lane < 2)                       // j0 + j + 3 < h: h % 8 == 0
                *reinterpret_cast<float4*>(p.tile_sums + ((int64_t)lane * gridDim.x + blockIdx.x) * p.h + j0 + j) =
                    lane == 0 ? make_float4(sum[0], sum[2], sum[4], sum[6]) : make_float4(sum[1], sum[3], sum[5], sum[7]);
        }
    }
    if (threadIdx.x == 0 && *abort_flag) atomicOr(p.d_status, ARROL_DEV_WAIT_EXPIRED);
    if (warp == S_PRODUCER_WARPS) {
        tcgen05_fence_after();
        tcgen05_dealloc(tmem_base, S_TMEM_COLS);
    }
}

// Clusters of `blocks` blocks with tiles of ROWS rollouts x SBN hidden units that are resident at once (asked once per context and size).
template <int SBN, int ROWS>
int resident_clusters(arrol_ctx* ctx, int blocks, int* fit) {
    int& known = ctx->score_max_clusters[SBN == 128 ? 2 : ROWS == 64][blocks];
    if (known == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1, (unsigned)blocks);
        cfg.blockDim = dim3(S_THREADS);
        cfg.dynamicSmemBytes = smem_bytes<SBN, ROWS>();
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1;
        attr[0].val.clusterDim.y = (unsigned)blocks;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        ARROL_CUDA_OK(cudaOccupancyMaxActiveClusters(&known, score_mlp_tc_kernel<SBN, SCORES, ROWS>, &cfg));
    }
    *fit = known;
    return ARROL_OK;
}

}  // namespace

// Launches the packing kernel and the contraction in one of its modes; p holds the mode's own outputs.  ARROL_ERR_UNSUPPORTED
// (nothing launched) when the sizes do not fit the context's buffers, or the mode.
static int launch_mlp_tc(arrol_ctx* ctx, const void* hidden, int64_t row_stride, const int64_t* row_index, int N,
                         const arrol_head* head, bool train, ScoreTcParams& p, cudaStream_t s, int* tile_rows = nullptr) {
    const int d = head->d, h = head->h;
    const int subs = (h + SUB_H - 1) / SUB_H;
    int m_tiles = (N + 127) / 128;
    if ((size_t)N * (size_t)subs > ARROL_SCRATCH_FLOATS || m_tiles > ARROL_SCORE_ROW_TILES)
        return ARROL_ERR_UNSUPPORTED;
    const bool pack = row_index != nullptr;
    if (pack && (size_t)N * (size_t)d * 2 > ARROL_PACK_BYTES) return ARROL_ERR_UNSUPPORTED;
    if (!row_index && ((uint64_t)row_stride * 2) >= (1ull << 40)) return ARROL_ERR_UNSUPPORTED;
    if (!ctx->score_tc_smem_set) {      // once per context: this call is on the prune step's microsecond path
        for (const auto f : {score_mlp_tc_kernel<64, PARTIALS, 128>, score_mlp_tc_kernel<64, SCORES, 128>, score_mlp_tc_kernel<64, TRAIN, 128>})
            ARROL_CUDA_OK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<64, 128>()));
        for (const auto f : {score_mlp_tc_kernel<128, PARTIALS, 128>, score_mlp_tc_kernel<128, SCORES, 128>, score_mlp_tc_kernel<128, TRAIN, 128>})
            ARROL_CUDA_OK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<128, 128>()));
        for (const auto f : {score_mlp_tc_kernel<64, SCORES, 64>, score_mlp_tc_kernel<64, TRAIN, 64>})
            ARROL_CUDA_OK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<64, 64>()));
        ctx->score_tc_smem_set = true;
    }
    // Tiles of 64 hidden units while they fit one wave of blocks (more SMs share the way in for the operands), of 128 beyond
    // that (a third fewer operand bytes and half as many blocks); the bits are the same.  Without / with the wide tiles (rows packed
    // before, partial sums through global memory): N = 4,096, d = 4,096, h = 512 39.0 -> 28.4 us (8 of them the packing), N = 8,192
    // 80.7 -> 64.7, N = 3,000, d = 1,024 17.1 -> 14.6; within one wave they lose: N = 2,048, d = 2,048, h = 256 14.2 -> 15.1.
    // Up to eight blocks of 64 are a cluster, or of 128; nine to sixteen blocks of 64 that fit one wave stay without (N = 300, d = 4,096,
    // h = 1,024 15.7 us, as cluster of wide ones 17.1), but for the training step, which needs the cluster (N = 300, d = 512, h = 1,024
    // 23.8 -> 21.2).
    // As clusters fewer blocks fit, GPCs not being filled by clusters of any size: 45, 33, 26, 22, 15 and 15 of three to eight blocks.  A
    // cluster saves a call about 2 us, a wave more costs it more, so scores are clustered where that takes no more waves (asked
    // once per context).  Without / with clusters, one wave more: d = 512: N = 6,000, h = 320 12.0 / 16.1 us, 9,000, 512 19.1 / 24.0, 2,100,
    // 896 11.9 / 15.4, 14,000, 1,024 50.3 / 60.9; d = 3,072: 2,100, 1,024 24.0 / 29.7, 9,000, 768 67.0 / 77.4; as many: N = 3,000, d = 1,024,
    // h = 512 14.7 / 12.9, 20,000, 256, 512 40.8 / 39.0.  The training step saves more, and is clustered unless one wave of the widest
    // tile rows becomes two: h = 1,024, N = 2,100, d = 512 40.5 / 42.3, d = 3,072 75.9 / 81.5; but h = 896, N = 2,600 45.5 / 44.3 (2,100
    // 41.7 / 42.5), h = 576, N = 3,300 43.5 / 36.9, h = 1,024, N = 4,200 63.3 / 63.0.
    const int wide_tiles = (h + 127) / 128;
    bool wide = m_tiles * subs > ctx->sm_count && h > SUB_H;
    const int waves = (m_tiles * (wide ? wide_tiles : subs) + ctx->sm_count - 1) / ctx->sm_count;       // without clusters
    // Tiles of 64 rollouts where all of these fit at once: half as much of the epilogue per SM, and a third fewer operand bytes.  Graph
    // of 20 calls, tiles of 128 / 64: N = 394, d = 1,664, h = 256 9.5 / 8.8 us, 1,000, 1,000, 320 11.2 / 9.5, 283, 600, 512 8.5 / 7.4, 32, 256,
    // 64 6.0 / 5.4; training steps N = 2,048, d = 2,048, h = 256 26.8 / 25.4, 525, 2,880, 512 27.2 / 23.5.
    bool cluster = false, half_rows = false;
    int fit = 0;
    if (!p.u_out && subs <= 8) {        // clusters of more than eight blocks are not portable
        if (resident_clusters<64, 64>(ctx, subs, &fit) != ARROL_OK) return ARROL_ERR_CUDA;
        half_rows = (N + 63) / 64 <= fit;
        if (half_rows) {
            wide = false;
            m_tiles = (N + 63) / 64;
        } else if (!wide && subs > 1) {
            if (resident_clusters<64, 128>(ctx, subs, &fit) != ARROL_OK) return ARROL_ERR_CUDA;
        }
        cluster = half_rows || (!wide && (subs == 1 || m_tiles <= fit));
    }
    if (!p.u_out && !cluster && subs <= MAX_SUBS && (wide || train)) {
        if (resident_clusters<128, 128>(ctx, wide_tiles, &fit) != ARROL_OK) return ARROL_ERR_CUDA;
        cluster = fit > 0 && ((m_tiles + fit - 1) / fit <= waves || (train && (waves > 1 || wide_tiles < 8)));
        wide = wide || cluster;
    }
    if (train && (!cluster || h % 8 != 0)) return ARROL_ERR_UNSUPPORTED;
    if (tile_rows) *tile_rows = half_rows ? 64 : 128;
    const int tiles_h = wide ? wide_tiles : subs;
    const void* x = hidden;
    int64_t ld = row_stride;
    if (pack) {
        const int slices = (d / 8 + PACK_VECS - 1) / PACK_VECS;
        ARROL_CUDA_OK(arrol_launch_pdl(pack_rows_kernel, dim3((unsigned)((N + 3) / 4), (unsigned)slices), dim3(128), 0, s,
                                       static_cast<const __nv_bfloat16*>(hidden), row_stride, row_index, N, d,
                                       static_cast<__nv_bfloat16*>(ctx->d_pack), ctx->source_rows, ctx->d_status));
        ctx->launches += 1;
        x = ctx->d_pack;
        ld = d;
    }
    CUtensorMap map_x, map_w;
    if (make_map(ctx, &map_w, head->W1, (uint64_t)h, (uint64_t)d, wide ? 128 : 64) != ARROL_OK) return ARROL_ERR_CUDA;
    if (make_map_ld(ctx, &map_x, x, (uint64_t)N, (uint64_t)d, (uint64_t)ld, half_rows ? 64 : 128) != ARROL_OK) return ARROL_ERR_CUDA;

    p.N = N;
    p.h = h;
    p.k_steps = (d + BK - 1) / BK;
    p.b1 = static_cast<const __nv_bfloat16*>(head->b1);
    p.w2 = static_cast<const __nv_bfloat16*>(head->w2);
    p.b2 = static_cast<const __nv_bfloat16*>(head->b2);
    p.partial = ctx->d_scratch;
    p.counters = ctx->d_tile_counters;
    p.d_status = ctx->d_status;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)m_tiles, (unsigned)tiles_h);
    cfg.blockDim = dim3(S_THREADS);
    cfg.dynamicSmemBytes = half_rows ? smem_bytes<64, 64>() : wide ? smem_bytes<128, 128>() : smem_bytes<64, 128>();
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = tiles_h;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster ? 2 : 1;
    const Mode mode = train ? TRAIN : cluster ? SCORES : PARTIALS;
    const auto kernel = half_rows ? (mode == TRAIN ? score_mlp_tc_kernel<64, TRAIN, 64> : score_mlp_tc_kernel<64, SCORES, 64>)
                        : wide ? (mode == TRAIN ? score_mlp_tc_kernel<128, TRAIN, 128>
                                                : mode == SCORES ? score_mlp_tc_kernel<128, SCORES, 128> : score_mlp_tc_kernel<128, PARTIALS, 128>)
                               : (mode == TRAIN ? score_mlp_tc_kernel<64, TRAIN, 128>
                                                : mode == SCORES ? score_mlp_tc_kernel<64, SCORES, 128> : score_mlp_tc_kernel<64, PARTIALS, 128>);
    ARROL_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, map_x, map_w, p));
    ctx->launches += 1;
    return ARROL_OK;
}

// Scores of a bf16 MLP head on the tensor cores.  Returns ARROL_ERR_UNSUPPORTED (nothing launched) when the sizes
// do not fit the context's buffers; the caller then takes the SIMT path.  Indexed rows are left packed as bf16
// [N][d] in the context's packing buffer (the head training step's second contraction reads them there).
// u_out [N][h]: the pre-activations as well (never clustered).
int arrol_internal_score_mlp_tc(arrol_ctx* ctx, const void* hidden, int64_t row_stride, const int64_t* row_index,
                                int N, const arrol_head* head, int B, const float* q_lut, float* score, float* prob,
                                int32_t* bin, float* q, float* u_out, cudaStream_t s) {
    ScoreTcParams p = {};
    p.u_out = u_out;
    p.B = B;
    p.q_lut = q_lut;
    p.score = score;
    p.prob = prob;
    p.bin = bin;
    p.q = q;
    return launch_mlp_tc(ctx, hidden, row_stride, row_index, N, head, false, p, s);
}

// The head training step up to the dW1 contraction, for at most 1,024 hidden units, a multiple of 8: du as two bf16 planes [N][h]; per tile of
// *tile_rows rollouts (64 or 128) what dw2 and db1 (tile_sums [2][tiles][h]), loss and db2 (tile_loss [2][tiles]) are the sums of.  Rows as above.
int arrol_internal_head_train_tc(arrol_ctx* ctx, const void* hidden, int64_t row_stride, const int64_t* row_index, int N,
                                 const arrol_head* head, const float* rewards, const uint8_t* mask, void* du_hi, void* du_lo,
                                 float* tile_sums, double* tile_loss, int* tile_rows, cudaStream_t s) {
    ScoreTcParams p = {};
    p.rewards = rewards;
    p.mask = mask;
    p.du_hi = static_cast<__nv_bfloat16*>(du_hi);
    p.du_lo = static_cast<__nv_bfloat16*>(du_lo);
    p.tile_sums = tile_sums;
    p.tile_loss = tile_loss;
    return launch_mlp_tc(ctx, hidden, row_stride, row_index, N, head, true, p, s, tile_rows);
}
