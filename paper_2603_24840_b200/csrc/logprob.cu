// arrol_token_logprob: selected-token log-probability of every survivor token from the lm_head
// (Section 3: log pi_theta(o_t | o_<t); Algorithm 1 "log-probs on R'"), as a fused contraction
// hidden[T,d] x W_vocab[V,d]^T with an online max / log-sum-exp epilogue.  The T x V logits never leave the SM.
//
// One thread block per SM, persistent over work items.  By default the blocks work as PAIRS (clusters of two, tcgen05
// cta_group::2) on 256-row tiles, see PAIR below; described first is the one-block form on 128-row tiles, which the
// pair form extends.  A work item is a token tile and a range of the vocabulary, which the block walks in chunks of 256
// columns.  Warp roles:
//   warp 0      TMA producer: K-major, 128-byte-swizzled tiles of hidden (128 x 64) and W_vocab (256 x 64) into
//               a ring of shared-memory stages, completion on mbarriers
//   warp 1      tcgen05.mma issuer (the warp waits, one elected lane issues): 128 x 256 x 16 bf16 MMAs into one of two
//               256-column fp32 accumulators in tensor memory; tcgen05.commit releases stages / publishes accumulators
//   epilogue warps  a thread owns one token row of the tile; tcgen05.ld of its accumulator row, running maximum and sum
//               of 2^(z log2e - max), and the target column's logit, all in registers
// The two accumulators let the epilogue of chunk c overlap the MMAs of chunk c + 1.
//
// Body and tail.  Whole waves of (tile, vocabulary group) items are the body.  What is left over would keep only some of
// the blocks busy for one more wave.  These tiles are the tail: (vocabulary segment, tile) items, as many segments as
// SMs, dealt round robin, so that every unit gets the same number of segments give or take one (see WorkList).  A token's
// records are merged in one order whoever computed them (see VocabPlan), so neither the token count nor the assignment of
// work shows in the bits.  Measured as pairs at d = 2560, V = 151,936 against whole items only (with more vocabulary splits
// while there were fewer tiles than SMs): 128 tokens 451 -> 181 us, 1,777 1,241 -> 1,051 us, 5,000 4.12 -> 2.83 ms, 9,000
// 5.24 -> 5.08 ms, 20,000 13.6 -> 11.0 ms.
//
// Waves in step.  The resident blocks all stream the same W_vocab chunks; as long as they do so at about the same
// time a chunk comes from HBM once and from L2 147 times.  Nothing in a persistent kernel keeps them together,
// though: measured on 6.5 M tokens (1,373 work items per block), the blocks' start times spread from 0.02 of an item
// after two waves to 2 items after 50 and 40 items after 800; once a block lags by more than L2 holds it re-streams
// its chunks from HBM, falls further behind, and the extra HBM traffic costs power: the SM clock under the 1 kW cap
// fell from 1.40 GHz in the first waves to 0.72 GHz.  So the blocks are held in step: before issuing the loads of
// wave k (its k-th work item) every producer arrives on a counter in global memory and waits until all blocks have
// arrived for that wave.  Single blocks are launched cooperatively whenever there is more than one wave, so that they are
// all resident; of pairs no more are launched than cudaOccupancyMaxActiveClusters says fit at once (a cooperative launch of
// clusters that fills the GPU is the one launch the profiler cannot make), which another launch on another stream can
// still keep from being resident together.  The results do not depend on the step, so a producer waits half as long as its own
// last item took (side by side they are within a few per cent of one another), or STEP_WAIT_CYCLES if that is longer, then goes on
// and waits no more.
// Every other wait is bounded too; when one runs out the block records ARROL_DEV_WAIT_EXPIRED, drains and returns.
//
// Gathered variant (arrol_token_logprob_gathered; Section 4.3 (ii): the survivors are re-batched "to compute
// log-probabilities"): the token rows are read straight from the pre-prune source buffer, so the packed copy of the
// hidden rows never exists.  A 128-row token tile that lies inside one survivor is 128 consecutive source rows: its
// TMA box simply starts at that source row.  Only a tile that crosses a survivor boundary is not contiguous in the
// source; those tiles (at most one per survivor) are first copied into a small scratch block, slot = the survivor
// of the tile's first row, by pack_boundary_tiles_kernel, and the main kernel reads them from there through a second
// tensor map.  Every tile therefore costs the same single box per K step.  That matters beyond the tile itself: the
// resident blocks stream the same W_vocab chunks at about the same time and share them through L2, and a block that
// falls behind by more than the L2 holds has to re-fetch its chunks from HBM (measured with multi-box copies for the
// boundary tiles: +10 % cycles on those tiles spread the blocks out, HBM traffic and power rose, and the SM clock
// fell from 1.27 to 0.8 GHz under the power cap).
#include <cuda.h>
#include <cuda_bf16.h>
#include <float.h>

#include "arrol_internal.h"
#include "tc_common.cuh"
#include "vocab_plan.cuh"

namespace {

constexpr int BM = 128;          // token rows per tile  (MMA M)
constexpr int BN = CHUNK_COLUMNS;   // vocabulary columns per chunk (MMA N)
constexpr int SOLO_STAGES = 4;
constexpr int A_STAGE_BYTES = BM * BK * 2;   // 16 KB
constexpr int SOLO_B_STAGE_BYTES = BN * BK * 2;   // 32 KB
constexpr int SOLO_STAGE_BYTES = A_STAGE_BYTES + SOLO_B_STAGE_BYTES;
// pair variant (two blocks of a cluster on one 256-row tile): every block stages its 128 rows of A and its half of
// the B tile, so a stage is 32 KB and six of them fit
constexpr int PAIR_STAGES = 6;
constexpr int PAIR_B_ROWS = BN / 2;
constexpr int PAIR_B_STAGE_BYTES = PAIR_B_ROWS * BK * 2;   // 16 KB
constexpr int PAIR_STAGE_BYTES = A_STAGE_BYTES + PAIR_B_STAGE_BYTES;
static_assert(PAIR_STAGES * PAIR_STAGE_BYTES == SOLO_STAGES * SOLO_STAGE_BYTES, "both variants fill the same shared memory");
constexpr int TMEM_COLS = 512;   // two fp32 accumulators of BN columns
constexpr int num_threads(int halves) { return 64 + 128 * halves; }     // producer, issuer, four epilogue warps per column half
constexpr long long STEP_WAIT_CYCLES = 100000;   // what a producer waits at least for the others of its wave (50 us or more)
constexpr int ITEMS_AHEAD = 64;              // work items of a unit that are listed in shared memory
constexpr size_t SMEM_BYTES = (size_t)SOLO_STAGES * SOLO_STAGE_BYTES + 1024 /* alignment slack */ + 256 /* barriers */ +
                              ITEMS_AHEAD * 28 /* WorkItem */;

struct PartialLse {   // of one token over some columns: running maximum and sum in the base-2 domain, target logit,
    float m2, l, zy2, sumz;   // sum of the raw accumulators (only when the confidence is asked for)
};

// (M, L) <- (M, L) + (m, l): M = max, L = sum of 2^(. - M).  One rounding per operation, so that the main kernel (body)
// and the combining kernel (tail) get the same bits.  An empty record (below) changes nothing: L 2^0 + 0.
__device__ __forceinline__ void merge_lse(float& M, float& L, float m, float l) {
    const float Mn = fmaxf(M, m);
    L = __fadd_rn(__fmul_rn(L, ex2_approx(M - Mn)), __fmul_rn(l, ex2_approx(m - Mn)));
    M = Mn;
}
__device__ __forceinline__ void merge_record(PartialLse& a, const PartialLse& b) {
    merge_lse(a.m2, a.l, b.m2, b.l);
    a.zy2 = fmaxf(a.zy2, b.zy2);        // exactly one record holds the target column, the others hold -inf
    a.sumz = __fadd_rn(a.sumz, b.sumz);
}
// The maximum starts at the lowest finite number: columns that are all -inf then add 2^(-inf) = 0 and leave the record empty, while
// NaN columns, which no maximum shows, make the sum NaN.  (From -inf both would end as -inf - -inf = NaN.)
__device__ __forceinline__ PartialLse empty_record() { return PartialLse{-FLT_MAX, 0.f, -INFINITY, 0.f}; }

// Work of one launch on `tiles` token tiles (128 rows, or 256 for a pair of blocks).  32-bit throughout (fewer than 2^24 tiles
// and at most 64 groups): the divisions are on the way of every work item and of the combining kernel.
struct WorkList {
    int body_tiles, body_items, tail_tiles, tail_items, waves;   // tail_tiles: at most units / splits + 1;  waves: those of the
    float inv_tail_tiles;                                        // body, plus one for the tail
};
__host__ __device__ inline WorkList make_work_list(int tiles, int units, const VocabPlan& v) {
    WorkList w;
    w.body_tiles = tiles * v.splits / units * units / v.splits;    // whole waves only
    w.body_items = w.body_tiles * v.splits;
    w.tail_tiles = tiles - w.body_tiles;
    w.tail_items = w.tail_tiles * v.n_sub;
    w.inv_tail_tiles = w.tail_tiles > 0 ? 1.0f / (float)w.tail_tiles : 0.f;
    w.waves = (w.body_items + units - 1) / units + (w.tail_items > 0 ? 1 : 0);
    return w;
}
struct WorkItem {
    int tile, wave;
    int group, sub0, sub1;      // group < 0: a tail item
    int c0, c1;                 // chunks of columns
};
// k-th item of a unit; false when it has none left.  The tail walks the segments as the slow index: at any time the
// units work on neighbouring segments of all tail tiles and share W_vocab through L2.  The segments that are a chunk longer go
// first: dealt round robin, no unit then has a chunk more than it must.  In the order of the vocabulary they fell to some units
// more often (19 pair tiles x 160 chunks: 44 chunks on the busiest of 74 pairs against 42; 24 tiles 60 against 52).  Single
// launches at the full clock in that order / this one: d = 1,856, V = 40,945: 1,000 tokens 132 / 110 us, 4,645 458 / 441, 6,000
// 615 / 550; d = 2,560, V = 50,257: 3,000 517 / 474, 5,000 794 / 783.
__device__ __forceinline__ bool work_item(const WorkList& w, const VocabPlan& v, int unit, int units, int k, WorkItem& it) {
    int i = unit + k * units;                   // body items, then tail items, in one numbering
    it.wave = k < w.waves ? k : w.waves - 1;
    if (i < w.body_items) {
        it.tile = i / v.splits;
        it.group = i - it.tile * v.splits;
        it.sub0 = v.sub_of_group(it.group);
        it.sub1 = v.sub_of_group(it.group + 1);
        it.c0 = v.chunk_of_sub(it.sub0);
        it.c1 = v.chunk_of_sub(it.sub1);
        return true;
    }
    i -= w.body_items;
    if (i >= w.tail_items) return false;
    const int turn = quotient(i, w.inv_tail_tiles);
    it.sub0 = v.nth_sub(turn);
    it.sub1 = it.sub0 + 1;
    it.tile = w.body_tiles + (i - turn * w.tail_tiles);
    it.group = -1;
    it.c0 = v.chunk_of_sub(it.sub0);
    it.c1 = v.chunk_of_sub(it.sub1);
    return true;
}

struct LogprobParams {
    const int32_t* targets;
    const int64_t* d_T;
    int64_t T_max;
    int d, V;
    VocabPlan plan;
    WorkList work;         // of T_max tokens
    float scale2;          // inv_temperature * log2(e)
    PartialLse* body;      // [splits][column halves][T_max]: records of the tokens in whole waves
    PartialLse* tail;      // [token of the tail][n_sub][column halves]
    uint32_t spin_limit;   // tries per pipeline wait
    int mute_producer;     // test hook: the producer issues no copies
    uint32_t* d_status;
    const int32_t* tile_row;      // gathered variant: source row of every token tile, or ~(scratch row) of a pre-packed one
    unsigned int* wave_counter;   // producers that have arrived, over all waves of this launch (zeroed before a launch of several)
    unsigned long long* timing;   // test hook: per body item {globaltimer start, end, clock64 start, end}, or NULL
    int64_t timing_items;
};

__device__ __forceinline__ unsigned long long global_timer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// 32 columns pc0 ... of one token row into its running record.  2.5 instructions a column: maxima three at a time, the exponents'
// arguments and the sums two at a time in packed fp32, and four chains of either, so that a warp does not wait for its own additions.
template <bool CONF>
__device__ __forceinline__ void accumulate_piece(uint32_t (&raw)[32], int pc0, int y, int V, float scale2, PartialLse& r) {
    auto v = [&](int j) { return __uint_as_float(raw[j]); };
    if constexpr (CONF) {                   // sum of the valid logits of the piece (before masking)
        float ps[4] = {0.f, 0.f, 0.f, 0.f};           // four chains; only the last piece needs the mask
        if (pc0 + 32 <= V) {
#pragma unroll
            for (int j = 0; j < 32; ++j) ps[j & 3] += v(j);
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) ps[j & 3] += (pc0 + j < V) ? v(j) : 0.f;
        }
        r.sumz += (ps[0] + ps[1]) + (ps[2] + ps[3]);
    }
    if (pc0 + 32 > V) {
#pragma unroll
        for (int j = 0; j < 32; ++j) if (pc0 + j >= V) raw[j] = 0xff800000u;      // -inf
    }
    if ((unsigned)(y - pc0) < 32u) {
        const int jy = y - pc0;
#pragma unroll
        for (int j = 0; j < 32; ++j) if (j == jy) r.zy2 = v(j) * scale2;
    }
    float top[4] = {v(0), v(1), v(2), v(3)};
#pragma unroll
    for (int j = 4; j < 28; j += 8)
#pragma unroll
        for (int c = 0; c < 4; ++c) top[c] = fmaxf(fmaxf(top[c], v(j + c)), v(j + 4 + c));
#pragma unroll
    for (int c = 0; c < 4; ++c) top[c] = fmaxf(top[c], v(28 + c));
    const float bmax = fmaxf(fmaxf(top[0], top[1]), fmaxf(top[2], top[3]));
    const float m_new = fmaxf(r.m2, bmax * scale2);
    const uint64_t scale = pack_f32x2(scale2, scale2), minus_m = pack_f32x2(-m_new, -m_new);
    uint64_t sum[2] = {0ull, 0ull};
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
        float a, b;
        unpack_f32x2(fma_f32x2(((uint64_t)raw[j + 1] << 32) | raw[j], scale, minus_m), a, b);
        sum[(j >> 1) & 1] = add_f32x2(sum[(j >> 1) & 1], pack_f32x2(ex2_approx(a), ex2_approx(b)));
    }
    float s0, s1;
    unpack_f32x2(add_f32x2(sum[0], sum[1]), s0, s1);
    r.l = fmaf(r.l, ex2_approx(r.m2 - m_new), s0 + s1);
    r.m2 = m_new;
}

// Survivor of packed token row t: the last s in [0, S) with cu_seqlens[s] <= t (this skips empty survivors).
__device__ __forceinline__ int survivor_of_row(const int64_t* __restrict__ cu_seqlens, int S, int64_t t) {
    int lo = 0, hi = S;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (cu_seqlens[mid] <= t) lo = mid; else hi = mid;
    }
    return lo;
}

// GATHER: map_h covers the pre-prune source rows and map_s the scratch of pre-packed boundary tiles
// ([S_max * 128, d], slot s at rows 128 s ...); otherwise map_h covers the packed rows and map_s is unused.
// PAIR: the kernel runs as clusters of two blocks; a pair works on 256 token rows (block r of the pair owns rows
// 128 r ...), block 0 issues 256 x 256 x 16 MMAs (cta_group::2) that read both blocks' shared memory and write both
// blocks' tensor memory, every block loads its own 128 rows of A and its own 128 of the chunk's 256 W_vocab rows and
// runs the epilogue of its own rows.  Per block and K step 32 KB come in from L2 instead of 48 KB and the tensor
// core reads 8 KB of operands per MMA from shared memory instead of 12 KB.
// HALVES: epilogue warps per tensor-memory lane quarter; two share a chunk's columns between them.
template <bool CONF, bool GATHER, bool PAIR, int HALVES>
__global__ void __launch_bounds__(num_threads(HALVES), 1)
token_logprob_kernel(const __grid_constant__ CUtensorMap map_h, const __grid_constant__ CUtensorMap map_s,
                     const __grid_constant__ CUtensorMap map_w, const LogprobParams p) {
    constexpr int STAGES = PAIR ? PAIR_STAGES : SOLO_STAGES;
    constexpr int B_STAGE_BYTES = PAIR ? PAIR_B_STAGE_BYTES : SOLO_B_STAGE_BYTES;
    constexpr int STAGE_BYTES = A_STAGE_BYTES + B_STAGE_BYTES;
    constexpr int EPI_WARPS = 4 * HALVES, EPI_COLS = BN / HALVES, TILE_ROWS = PAIR ? 2 * BM : BM;
    extern __shared__ uint8_t smem_raw[];
    // stage buffers need 1024-byte alignment for the 128-byte swizzle pattern
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* stage_a = smem;
    uint8_t* stage_b = smem + (size_t)STAGES * A_STAGE_BYTES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)STAGES * STAGE_BYTES);
    uint64_t* full = bars;                    // [STAGES]  TMA -> MMA (pair: block 0's receive both blocks' bytes)
    uint64_t* empty = bars + STAGES;          // [STAGES]  MMA -> TMA
    uint64_t* acc_full = bars + 2 * STAGES;   // [2]       MMA -> epilogue
    uint64_t* acc_empty = acc_full + 2;       // [2]       epilogue -> MMA
    uint64_t* drain = acc_empty + 2;          // [1]       used only when giving up: MMAs in flight -> done
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    WorkItem* items_s = reinterpret_cast<WorkItem*>(smem + (size_t)STAGES * STAGE_BYTES + 256);   // [ITEMS_AHEAD] this unit's first items

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // pair: rank of this block in its cluster (block 0 leads), unit = cluster; otherwise unit = block
    const uint32_t rank = PAIR ? cluster_cta_rank() : 0u;
    const int unit = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
    const int units = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;

    const int k_steps = (p.d + BK - 1) / BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        // pair: the leading block's acc_empty collects the epilogue warps of both blocks
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], (PAIR ? 2 : 1) * EPI_WARPS); }
        mbar_init(drain, 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_h) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_w) : "memory");
        if constexpr (GATHER) asm volatile("prefetch.tensormap [%0];" ::"l"(&map_s) : "memory");
    }
    if (warp == 1) {
        if constexpr (PAIR) { tcgen05_alloc_pair(tmem_slot, TMEM_COLS); tcgen05_relinquish_pair(); }
        else { tcgen05_alloc(tmem_slot, TMEM_COLS); tcgen05_relinquish(); }
    }
    // The unit's first items, a thread each.  Every role would work them out for itself, one behind the other, and the first time
    // through that code costs a microsecond of instruction and constant fetches: here it overlaps the preceding kernel.
    WorkList work = p.work;
    auto list_items = [&] {
        if (threadIdx.x < ITEMS_AHEAD) {
            WorkItem it = {};
            if (!work_item(work, p.plan, unit, units, threadIdx.x, it)) it.c0 = it.c1 = -1;
            items_s[threadIdx.x] = it;
        }
    };
    list_items();
    auto get_item = [&](int k, WorkItem& it) {
        if (k >= ITEMS_AHEAD) return work_item(work, p.plan, unit, units, k, it);
        it = items_s[k];
        return it.c0 >= 0;
    };
    tcgen05_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();     // the peer's barriers exist before anything arrives on them
    tcgen05_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // pair: shared::cluster addresses, in the leading block, of the barriers both blocks signal
    uint32_t lead_full0 = 0, lead_acc_empty0 = 0;
    if constexpr (PAIR) {
        lead_full0 = map_to_cta(smem_u32(&full[0]), 0u);
        lead_acc_empty0 = map_to_cta(smem_u32(&acc_empty[0]), 0u);
    }
    pdl_launch_dependents();       // the combining kernel may be set up while this one runs
    pdl_wait();                    // the set-up above overlaps the end of the preceding kernel
    int64_t T = p.T_max;
    if (p.d_T) {
        const int64_t t = *pdl_acquire(p.d_T);
        T = t < 0 ? 0 : (t < T ? t : T);
        const int tiles = (int)((T + TILE_ROWS - 1) / TILE_ROWS);
        if (tiles != work.body_tiles + work.tail_tiles) {          // uniform over the block
            work = make_work_list(tiles, units, p.plan);
            list_items();
            __syncthreads();
        }
    }

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            uint32_t stage = 0, phase = 0;
            uint32_t issued = 0;
            bool ok = true;
            const int32_t* tile_row = pdl_acquire(p.tile_row);
            // first of the 128 source rows of this block's tile (gathered variant; requested one item ahead)
            auto source_row = [&](const WorkItem& it) {
                return tile_row[PAIR ? 2 * it.tile + (int)rank : it.tile];
            };
            WorkItem it, next;
            bool have = !p.mute_producer && get_item(0, it);
            int row = 0;
            if constexpr (GATHER) if (have) row = source_row(it);
            int arrived = 0, waited = 0;            // waves
            bool in_step = true;
            long long item_begun = clock64();
            for (int k = 0; !p.mute_producer; ++k) {
                // hold the blocks in step: arrive for the item's wave (one arrival per unit and wave), then wait for
                // everybody; a unit without an item in a partial wave arrives as well
                const int wave = have ? it.wave : work.waves - 1;
                for (; arrived < wave; ++arrived)
                    if (rank == 0) atomicAdd(p.wave_counter, 1u);
                if (!have) break;
                if (wave > waited && in_step) {
                    const unsigned int target = (unsigned int)wave * (unsigned int)units;
                    long long now = clock64();
                    const long long until = now + max((now - item_begun) / 2, STEP_WAIT_CYCLES);
                    while (ld_relaxed_u32(p.wave_counter) < target) {
                        if (now >= until) { in_step = false; break; }
                        __nanosleep(64);
                        now = clock64();
                    }
                    waited = wave;
                    item_begun = now;
                }
                const bool have_next = get_item(k + 1, next);
                int row_next = 0;
                if constexpr (GATHER) if (have_next) row_next = source_row(next);
                // where the tile's 128 rows come from: the packed rows, a run of source rows, or a scratch slot
                const CUtensorMap* a_map = &map_h;
                int a_row = (PAIR ? 2 * it.tile + (int)rank : it.tile) * BM;
                if constexpr (GATHER) {
                    a_row = row;
                    if (row < 0) { a_map = &map_s; a_row = ~row; }
                }
                for (int c = it.c0; c < it.c1 && ok; ++c) {
                    for (int ks = 0; ks < k_steps; ++ks) {
                        if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag, p.spin_limit)) { ok = false; break; }
                        if constexpr (PAIR) {
                            // both blocks' bytes are counted on the leading block's barrier
                            const uint32_t bar = lead_full0 + stage * (uint32_t)sizeof(uint64_t);
                            if (rank == 0) mbar_expect_tx(&full[stage], 2 * STAGE_BYTES);
                            tma_load_2d_pair(smem_u32(stage_a) + stage * A_STAGE_BYTES, a_map, ks * BK, a_row, bar);
                            tma_load_2d_pair(smem_u32(stage_b) + stage * B_STAGE_BYTES, &map_w, ks * BK,
                                             c * BN + (int)rank * (chunk_columns(p.V, c) / 2), bar);
                        } else {
                            mbar_expect_tx(&full[stage], STAGE_BYTES);
                            tma_load_2d(stage_a + (size_t)stage * A_STAGE_BYTES, a_map, ks * BK, a_row, &full[stage]);
                            tma_load_2d(stage_b + (size_t)stage * B_STAGE_BYTES, &map_w, ks * BK, c * BN, &full[stage]);
                        }
                        ++issued;
                        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                    }
                }
                if (!ok) break;
                it = next;
                have = have_next;
                row = row_next;
            }
            if (!ok && rank == 0) {
                // Gave up: let the copies already issued land before the block's shared memory goes away.
                // The last min(issued, STAGES) stages may still be in flight; wait for each (bounded).  (In a pair the
                // second block's copies are counted on the leading block's barriers; the cluster barrier at the end
                // of the kernel keeps its shared memory alive until the leading block has got here.)
                const uint32_t pending = issued < (uint32_t)STAGES ? issued : (uint32_t)STAGES;
                uint32_t s = stage, ph = phase;
                for (uint32_t i = 0; i < pending; ++i) {
                    if (s == 0) { s = STAGES - 1; ph ^= 1u; } else { --s; }
                    for (uint32_t it = 0; it < p.spin_limit; ++it)
                        if (mbar_try_wait(&full[s], ph)) break;
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        // The whole warp walks the loops and waits, one elected lane issues: with control flow that is uniform over the
        // warp the descriptors and the loop state stay in uniform registers.  Under a single-thread branch around the loop
        // every MMA's operands went through per-thread registers first, and issuing a K step's four MMAs took the thread
        // about the 512 cycles that they run.  200,000 tokens, d = 2048, V = 61,125 (pairs): 35.6 -> 34.8 ms; 100,000,
        // d = 4096, V = 151,936 (single blocks): 91.7 -> 90.6 ms.
        if (rank == 0) {
            const int k_last = (p.d - (k_steps - 1) * BK + UMMA_K - 1) / UMMA_K;     // K slices of the last K step
            const uint32_t a0 = smem_u32(stage_a), b0 = smem_u32(stage_b);
            uint32_t stage = 0, phase = 0;
            uint32_t acc = 0, acc_phase = 0;
            bool ok = true;
            WorkItem it;
            for (int k = 0; ok && get_item(k, it); ++k) {
                for (int c = it.c0; c < it.c1 && ok; ++c) {
                    const uint32_t idesc = make_idesc(PAIR ? 2 * BM : BM, chunk_columns(p.V, c));
                    if (!mbar_wait_warp(&acc_empty[acc], acc_phase ^ 1u, abort_flag, p.spin_limit)) { ok = false; break; }
                    tcgen05_fence_after();
                    const uint32_t d_tmem = tmem_base + acc * BN;
                    for (int ks = 0; ks < k_steps; ++ks) {
                        if (!mbar_wait_warp(&full[stage], phase, abort_flag, p.spin_limit)) { ok = false; break; }
                        tcgen05_fence_after();
                        const uint64_t a_desc = make_smem_desc(a0 + stage * A_STAGE_BYTES);
                        const uint64_t b_desc = make_smem_desc(b0 + stage * B_STAGE_BYTES);
                        if (elect_one()) {
                            // advancing K by 16 elements = 32 bytes inside the swizzle row: +2 in address units
                            auto mma = [&](int j) {
                                if constexpr (PAIR)
                                    tcgen05_mma_bf16_pair(d_tmem, a_desc + (uint64_t)(2 * j), b_desc + (uint64_t)(2 * j), idesc,
                                                          (ks | j) != 0 ? 1u : 0u);
                                else
                                    tcgen05_mma_bf16(d_tmem, a_desc + (uint64_t)(2 * j), b_desc + (uint64_t)(2 * j), idesc,
                                                     (ks | j) != 0 ? 1u : 0u);
                            };
                            if (ks + 1 < k_steps || k_last == BK / UMMA_K) {
#pragma unroll
                                for (int j = 0; j < BK / UMMA_K; ++j) mma(j);
                            } else {
                                for (int j = 0; j < k_last; ++j) mma(j);     // slices past d are zeros
                            }
                            // stage reusable (in both blocks of a pair) once these MMAs have read it; after the last K
                            // step the accumulator is complete
                            if constexpr (PAIR) tcgen05_commit_pair(&empty[stage], (uint16_t)3);
                            else tcgen05_commit(&empty[stage]);
                            if (ks + 1 == k_steps) {
                                if constexpr (PAIR) tcgen05_commit_pair(&acc_full[acc], (uint16_t)3);
                                else tcgen05_commit(&acc_full[acc]);
                            }
                        }
                        __syncwarp();
                        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
                    }
                    if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
                }
            }
            if (!ok && elect_one()) {
                // Gave up: wait (bounded) until the MMAs already issued have finished with shared and tensor memory.
                if constexpr (PAIR) tcgen05_commit_pair(drain, (uint16_t)1);
                else tcgen05_commit(drain);
                for (uint32_t it = 0; it < p.spin_limit; ++it)
                    if (mbar_try_wait(drain, 0u)) break;
            }
            __syncwarp();
        }
    } else {
        // ---------------- epilogue: one token row (and its share of the columns) per thread ----------------
        const int quarter = warp & 3;                       // TMEM lanes 32*quarter .. 32*quarter+31
        const int half = (warp - 2) >> 2;                   // columns EPI_COLS * half ... of every chunk
        const int row_in_tile = quarter * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        const int32_t* targets = pdl_acquire(p.targets);
        uint32_t acc = 0, acc_phase = 0;
        bool ok = true;
        auto token_of = [&](const WorkItem& it) { return (int64_t)(PAIR ? 2 * it.tile + (int)rank : it.tile) * BM + row_in_tile; };
        auto target_of = [&](const WorkItem& it) { const int64_t t = token_of(it); return t < T ? targets[t] : -1; };
        // The next item and its target are requested before this one's columns: an item of one chunk would wait for them longer
        // than a quarter of its time.
        WorkItem it, next;
        bool have = get_item(0, it), have_next = false;
        int y = have ? target_of(it) : -1, y_next = -1;
        for (int k = 0; ok && have; ++k, it = next, y = y_next, have = have_next) {
            have_next = get_item(k + 1, next);
            y_next = have_next ? target_of(next) : -1;
            const int64_t t = token_of(it);
            PartialLse sub = empty_record(), mid = empty_record(), group = empty_record();
            const int64_t stamp_at = (int64_t)it.tile * p.plan.splits + it.group;
            const bool stamp = p.timing != nullptr && threadIdx.x == 64 && rank == 0 && it.group >= 0 && stamp_at < p.timing_items;
            if (stamp) { p.timing[4 * stamp_at] = global_timer_ns(); p.timing[4 * stamp_at + 2] = (unsigned long long)clock64(); }
            int mid_i = it.group >= 0 ? p.plan.group_begin[it.group] : 0;
            int mid_end = p.plan.mid_begin[mid_i + 1];
            int c = it.c0;
            for (int s = it.sub0; s < it.sub1 && ok; ++s) {
                const int c1 = s + 1 == it.sub1 ? it.c1 : p.plan.chunk_of_sub(s + 1);
                for (; c < c1 && ok; ++c) {
                    ok = mbar_wait(&acc_full[acc], acc_phase, abort_flag, p.spin_limit);
                    ok = __all_sync(0xffffffffu, ok) != 0;     // keep the warp converged for the aligned tensor-memory loads
                    if (!ok) break;
                    tcgen05_fence_after();
                    const int col0 = c * BN + half * EPI_COLS;
                    const int pieces = min(EPI_COLS / 32, (p.V - col0 + 31) / 32);        // none past the vocabulary
                    auto hand_back = [&] {
                        tcgen05_fence_before();
                        __syncwarp();
                        if (lane == 0) {
                            if constexpr (PAIR) mbar_arrive_cluster(lead_acc_empty0 + acc * (uint32_t)sizeof(uint64_t));
                            else mbar_arrive(&acc_empty[acc]);
                        }
                    };
#pragma unroll 1
                    for (int piece = 0; piece < pieces; ++piece) {
                        uint32_t v[32];
                        tcgen05_ld_32x32_issue(tmem_base + lane_addr + acc * BN + half * EPI_COLS + piece * 32, v);
                        tcgen05_ld_wait(v);
                        if (piece + 1 == pieces) hand_back();
                        accumulate_piece<CONF>(v, col0 + piece * 32, y, p.V, p.scale2, sub);
                    }
                    if (pieces <= 0) hand_back();
                    if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
                }
                if (it.group >= 0) {                           // the segment is complete: segment -> block -> group
                    merge_record(mid, sub);
                    sub = empty_record();
                    if (s + 1 == mid_end) {
                        merge_record(group, mid);
                        mid = empty_record();
                        if (s + 1 < it.sub1) mid_end = p.plan.mid_begin[++mid_i + 1];
                    }
                }
            }
            if (stamp) { p.timing[4 * stamp_at + 1] = global_timer_ns(); p.timing[4 * stamp_at + 3] = (unsigned long long)clock64(); }
            if (ok && t < T) {
                const PartialLse& r = it.group >= 0 ? group : sub;
                PartialLse* dst;
                if (it.group >= 0) {
                    dst = p.body + ((int64_t)it.group * HALVES + half) * p.T_max + t;
                } else {
                    const int64_t tail_row = t - (int64_t)work.body_tiles * ((PAIR ? 2 : 1) * BM);
                    dst = p.tail + (tail_row * p.plan.n_sub + it.sub0) * HALVES + half;
                }
                *reinterpret_cast<float4*>(dst) = make_float4(r.m2, r.l, r.zy2, r.sumz);
            }
        }
    }

    tcgen05_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();     // neither block's shared or tensor memory goes away under the other
    if (threadIdx.x == 0 && *abort_flag) atomicOr(p.d_status, ARROL_DEV_WAIT_EXPIRED);
    if (warp == 1) {
        tcgen05_fence_after();
        if constexpr (PAIR) tcgen05_dealloc_pair(tmem_base, TMEM_COLS);
        else tcgen05_dealloc(tmem_base, TMEM_COLS);
    }
}

// Gathered variant, first kernel: copies every token tile that crosses a survivor boundary into its scratch slot.
// Block s looks at the tile that holds survivor s's last row: if that tile starts inside s (so s owns it) and runs on
// past the end of s, its rows are copied, run by run, with 16-byte loads/stores (eight in flight per thread).  Bound by latency: a
// pass of 32 KB takes a block about 2 us and a tile of d = 2,240 has 18 of them, so the passes of a tile are dealt to the blocks of a
// column of the grid while that leaves SMs without one.
constexpr int PACK_THREADS = 256, PACK_PASS = 8 * PACK_THREADS;
__global__ void __launch_bounds__(PACK_THREADS)
pack_boundary_tiles_kernel(const uint4* __restrict__ src_rows, const int64_t* __restrict__ cu_seqlens,
                           const int32_t* __restrict__ survivor_idx, const int64_t* __restrict__ src_tok_off,
                           const int64_t* __restrict__ d_num, int S_max, int64_t T_max, int vec_per_row,
                           uint4* __restrict__ scratch, int32_t* __restrict__ tile_row) {
    __shared__ int64_t src_row_of[BM];
    pdl_launch_dependents();
    pdl_wait();
    cu_seqlens = pdl_acquire(cu_seqlens); survivor_idx = pdl_acquire(survivor_idx); d_num = pdl_acquire(d_num);
    src_tok_off = pdl_acquire(src_tok_off); src_rows = pdl_acquire(src_rows);
    int64_t S64 = d_num[0], T = d_num[1];
    const int S = (int)(S64 < 0 ? 0 : (S64 > (int64_t)S_max ? (int64_t)S_max : S64));
    T = T < 0 ? 0 : (T < T_max ? T : T_max);
    // where every token tile's rows come from (an even number of entries: a pair's second tile may lie past T)
    const int64_t tiles = ((T + BM - 1) / BM + 1) / 2 * 2;
    const int64_t block = (int64_t)blockIdx.y * gridDim.x + blockIdx.x, blocks = (int64_t)gridDim.x * gridDim.y;
    for (int64_t i = block * PACK_THREADS + threadIdx.x; i < tiles; i += blocks * PACK_THREADS) {
        const int64_t t0 = i * BM;
        int32_t row = 0;
        if (t0 < T) {
            const int s0 = survivor_of_row(cu_seqlens, S, t0);
            const int64_t s_end = cu_seqlens[s0 + 1];
            // the tile runs on into the next survivor: its pre-packed copy
            if (s_end < t0 + BM && s_end < T) row = ~(s0 * BM);
            else row = (int32_t)(src_tok_off[survivor_idx[s0]] + (t0 - cu_seqlens[s0]));
        }
        tile_row[i] = row;
    }
    for (int s0 = blockIdx.x; s0 < S; s0 += gridDim.x) {
        const int64_t begin = cu_seqlens[s0], end = cu_seqlens[s0 + 1];
        if (end <= begin || end >= T) continue;                 // empty, or nothing follows
        const int64_t t0 = (end - 1) / BM * BM;                 // tile of the survivor's last row
        if (t0 < begin || t0 + BM <= end) continue;             // owned by an earlier survivor / ends with the tile
        const int rows = (int)min((int64_t)BM, T - t0);
        __syncthreads();                                        // src_row_of is free again
        for (int r = threadIdx.x; r < rows; r += PACK_THREADS) {
            const int64_t t = t0 + r;
            int sv = s0;
            while (sv + 1 < S && cu_seqlens[sv + 1] <= t) ++sv;
            src_row_of[r] = src_tok_off[survivor_idx[sv]] + (t - cu_seqlens[sv]);
        }
        __syncthreads();
        uint4* dst = scratch + (int64_t)s0 * BM * vec_per_row;
        const int total = rows * vec_per_row;
        for (int v0 = (int)blockIdx.y * PACK_PASS; v0 < total; v0 += (int)gridDim.y * PACK_PASS) {
            uint4 buf[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int vv = v0 + u * PACK_THREADS + threadIdx.x;
                if (vv < total) {
                    const int r = vv / vec_per_row;
                    buf[u] = __ldg(src_rows + src_row_of[r] * vec_per_row + (vv - r * vec_per_row));
                }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int vv = v0 + u * PACK_THREADS + threadIdx.x;
                if (vv < total) dst[vv] = buf[u];
            }
        }
    }
}

// Merges every token's records.  Tokens of the body: one thread each, splits x HALVES records.  Tokens of the tail: a block takes
// `group` consecutive ones, whose records lie one after another and come into shared memory by asynchronous copies; a thread
// merges the segments of one block of segments (and column half), then a thread per token and half walks the blocks in order.
// Bound by latency: one round trip for the length, the targets and the records together (where no call of T_max tokens has a body the
// records' place does not depend on the length), then some 25 dependent merges of 50 cycles.  Of calls with no more blocks than fit at once,
// registers and shared memory leave room for one beside the log-prob kernel's on every SM, where it waits; blocks past that would pile up
// on the SM that is free first.  A warp per token, its lanes the blocks of segments and then all of them the same chain of 16 merges, took 4.5 to 6.5 us
// of a call of 2,800 tokens on V = 4,096 (d = 256), and takes 2.8 to 3.4 now.  With the items listed ahead the whole call went from 18.9 to
// 14.4 us (graph of 20), 3,636 tokens at d = 320 on V = 14,170 from 41.9 to 35.0.
constexpr int COMBINE_THREADS = 256;
static_assert((MAX_SEGMENTS + MAX_SPLITS) * 2 * 16 + SMEM_BYTES + 2 * BLOCK_SMEM_RESERVED <= SM_SMEM, "a token's records fit beside the log-prob kernel");
template <int HALVES>
__global__ void __launch_bounds__(COMBINE_THREADS, COMBINE_BLOCKS)
combine_splits_kernel(const PartialLse* body, const PartialLse* tail, const int32_t* targets, const int64_t* d_T,
                      int64_t T_max, int V, VocabPlan plan, int tile_rows, int units, int group, int block_lanes, bool tail_only,
                      float* __restrict__ logp, float* __restrict__ lse, float* __restrict__ conf, float inv_temp, uint32_t* d_status) {
    extern __shared__ __align__(16) float4 records_s[];    // [group][n_sub][HALVES], then [group][n_mid][HALVES] where that is less
    pdl_wait();
    body = pdl_acquire(body); tail = pdl_acquire(tail); targets = pdl_acquire(targets); d_T = pdl_acquire(d_T);
    const int tid = threadIdx.x;
    const int per_token = plan.n_sub * HALVES;
    auto fetch = [&](int64_t row0, int n) {
        const float4* from = reinterpret_cast<const float4*>(tail + row0 * per_token);
        for (int i = tid; i < n * per_token; i += COMBINE_THREADS) cp_async_16(records_s + i, from + i);
    };
    const int64_t first = (int64_t)blockIdx.x * group;
    if (tail_only && first < T_max) fetch(first, (int)min((int64_t)group, T_max - first));
    int64_t T = T_max;
    if (d_T) { const int64_t t = *d_T; T = t < 0 ? 0 : (t < T ? t : T); }
    const WorkList work = make_work_list((int)(((unsigned)T + tile_rows - 1) / (unsigned)tile_rows), units, plan);   // T < 2^31
    const int64_t body_rows = min(T, (int64_t)work.body_tiles * tile_rows);
    auto load = [](const float4* p) {
        const float4 r = *p;
        return PartialLse{r.x, r.y, r.z, r.w};
    };
    auto finish = [&](int64_t t, int y, const PartialLse& r) {
        const float lse2 = r.m2 + log2f(r.l);
        const float ln2 = 0.69314718055994530942f;
        float out = 0.f;
        if (y >= 0) {
            if (y < V) out = (r.zy2 - lse2) * ln2;
            else atomicOr(d_status, ARROL_DEV_BAD_TARGET);
        }
        logp[t] = out;
        if (lse) lse[t] = lse2 * ln2;
        if (conf) conf[t] = (float)V * (lse2 * ln2) - r.sumz * inv_temp;
    };
    const int64_t thread = blockIdx.x * (int64_t)COMBINE_THREADS + tid;
    const int64_t threads = (int64_t)gridDim.x * COMBINE_THREADS;
    for (int64_t t = thread; t < body_rows; t += threads) {
        const int y = targets[t];
        PartialLse total[HALVES];
#pragma unroll
        for (int h = 0; h < HALVES; ++h) total[h] = empty_record();
        for (int g = 0; g < plan.splits; ++g)
#pragma unroll
            for (int h = 0; h < HALVES; ++h)
                merge_record(total[h], load(reinterpret_cast<const float4*>(body + ((int64_t)g * HALVES + h) * T_max + t)));
#pragma unroll
        for (int h = 1; h < HALVES; ++h) merge_record(total[0], total[h]);
        finish(t, y, total[0]);
    }
    const int per_block = plan.n_mid * HALVES, lanes = 1 << block_lanes;       // lanes >= per_block
    float4* blocks_s = plan.n_mid < plan.n_sub ? records_s + group * per_token : records_s;
    for (int64_t row0 = first; row0 < T - body_rows; row0 += (int64_t)gridDim.x * group) {
        const int n = (int)min((int64_t)group, T - body_rows - row0);
        if (!tail_only) fetch(row0, n);
        const int token = tid / HALVES, h = tid % HALVES;
        const int y = token < n ? targets[body_rows + row0 + token] : -1;           // requested now, used at the end
        cp_async_wait_all();
        __syncthreads();
        if (plan.n_mid < plan.n_sub) {
            const int i = tid & (lanes - 1), b = i / HALVES;
            if (i < per_block)
                for (int of = tid >> block_lanes; of < n; of += COMBINE_THREADS >> block_lanes) {
                    const float4* rec = records_s + of * per_token + i % HALVES;
                    PartialLse mine = empty_record();
                    const int s1 = plan.mid_begin[b + 1];
#pragma unroll 4
                    for (int s = plan.mid_begin[b]; s < s1; ++s) merge_record(mine, load(rec + s * HALVES));
                    blocks_s[of * per_block + i] = make_float4(mine.m2, mine.l, mine.zy2, mine.sumz);
                }
            __syncthreads();
        }
        // warps come along whole
        if (tid / 32 * 32 < n * HALVES) {
            PartialLse total = empty_record(), in_group = empty_record();
            if (token < n) {
                const float4* rec = blocks_s + token * per_block + h;
                for (int g = 0; g < plan.splits; ++g) {
                    const int b1 = plan.group_begin[g + 1];
#pragma unroll 4
                    for (int b = plan.group_begin[g]; b < b1; ++b) merge_record(in_group, load(rec + b * HALVES));
                    merge_record(total, in_group);
                    in_group = empty_record();
                }
            }
            if constexpr (HALVES == 2)
                merge_record(total, PartialLse{__shfl_down_sync(0xffffffffu, total.m2, 1), __shfl_down_sync(0xffffffffu, total.l, 1),
                                               __shfl_down_sync(0xffffffffu, total.zy2, 1), __shfl_down_sync(0xffffffffu, total.sumz, 1)});
            if (token < n && h == 0) finish(body_rows + row0 + token, y, total);
        }
        __syncthreads();                    // the records are overwritten by the next ones
    }
    cp_async_wait_all();                    // of a block past the live tokens: its copies land before its shared memory goes away
}

// How many vocabulary splits per token tile.  With one split every resident block streams a different token
// tile (128 x d x 2 bytes each) against the same W chunks; when those tiles together outgrow about half of L2
// the tiles are re-fetched from HBM once per chunk, so the vocabulary is split until they fit.
int splits_for(const arrol_ctx* ctx, int d, int V, bool pair) {
    const int total_chunks = (V + BN - 1) / BN;
    // Measured with the blocks in step (TFLOP/s, packed rows / rows read in place by the gathered variant):
    //   d = 2048: 1 split (148 resident tiles, 74 MB) 1,380 / 1,200;  2 splits (74 tiles, 37 MB) 1,377 / 1,378
    //   d = 2560: 1 split (95 MB) 1,041 / 1,070;  2 splits (47 MB) 1,392 / 1,391;  4 splits (24 MB) 1,362 / 1,362
    //   d = 4096: 1 split (148 MB) 990 / 987;  2 splits (74 MB) 1,391 / 1,377;  4 splits (37 MB) 1,363 / 1,363
    // and as pairs of blocks (cta_group::2), same order:
    //   d = 2048: 1 split 1,389 / 1,271;  2 splits 1,411-1,427 / 1,403-1,410
    //   d = 2560: 2 splits 1,428 / 1,413;  4 splits 1,403 / 1,396
    //   d = 4096: 2 splits (74 MB) 1,235 / 1,232;  4 splits (37 MB) 1,392 / 1,371;  8 splits 1,357 / 1,352
    // Token tiles beyond what L2 keeps are re-fetched from HBM once per chunk; every split beyond that streams
    // W_vocab from HBM once more per wave.  So: two splits (tiles read in place are scattered over the source buffer and
    // 148 of them do not stay resident even at 74 MB), more only while the resident tiles exceed 80 MB (one block per tile) or 50 MB (pairs).  The packed and the in-place variant follow
    // the same rule, so their results are bit-identical.
    if (ctx->logprob_splits > 0) return ctx->logprob_splits < total_chunks ? ctx->logprob_splits : total_chunks;
    int splits = 2;
    const double l2_budget = (pair ? 50.0 : 80.0) * 1024 * 1024;
    const double tile_bytes = (double)BM * d * 2;
    while (splits < 8 && (ctx->sm_count / splits) * tile_bytes > l2_budget) splits *= 2;
    return splits < total_chunks ? splits : total_chunks;
}

// The form of the kernel for these sizes (V = 61,125, 100,000 tokens; us as single blocks and as pairs, eight epilogue warps up to
// 896, four beyond):
//   d = 256   2,865 / 2,850    d = 320 (20,000 tokens, V = 40,000)  456 / 425    d = 384   3,757 / 3,530    d = 512   4,710 / 4,290
//   d = 768 (four / eight warps)  7,140 / 7,242, pairs 6,954 / 6,653             d = 1,024 9,376 / 8,798
//   d = 4,096 (V = 151,936, 287,000 tokens): single blocks with two splits 250.6 ms, pairs with four 247.9 ms
// A chunk's 128 x 256 exponentials take an SM's special-function units 2,048 cycles, its MMAs 8 d: at small d the epilogue
// sets the pace.  Two warps per scheduler then hide the latency of one another's tensor-memory loads, and single blocks
// hand an accumulator back without waiting for a peer's epilogue.  At larger d pairs move fewer operand bytes, and fewer
// epilogue warps draw less power.  A call of few tokens pays for a pair's 256-row tiles and its
// start (V = 32,379, single blocks / pairs): d = 320, 286 tokens 17.8 / 25.2, 2,000 47.8 / 48.2, 5,000 115 / 109; d = 512, 1,000 tokens
// 32.7 / 32.8, 2,000 66.2 / 58.9, 5,000 159 / 145.  The line is drawn by T_max, the live tokens being on the device: with V = 151,936, capacities of
// 2,500 and 5,000, a quarter / half / all of it live, d = 320: 56 / 65, 102 / 101, 195 / 190 and 102 / 101, 196 / 192, 389 / 368; d = 512:
// 82 / 90, 150 / 140, 283 / 259 and 150 / 139, 287 / 263, 555 / 504.  What few tokens lose is the half tile at their end.
constexpr int PAIR_MIN_WIDTH = 320, PAIR_ALWAYS_WIDTH = 513, EIGHT_WARPS_MAX_WIDTH = 896;
constexpr int64_t PAIR_MIN_WORK = 800000;      // T_max d, for widths in between
bool pair_for(const arrol_ctx* ctx, int64_t T_max, int d) {
    if (ctx->sm_count < 2 || ctx->logprob_pair == 0) return false;
    return ctx->logprob_pair == 1 || d >= PAIR_ALWAYS_WIDTH || (d >= PAIR_MIN_WIDTH && T_max >= (PAIR_MIN_WORK + d - 1) / d);
}
int halves_for(int d) { return d <= EIGHT_WARPS_MAX_WIDTH ? 2 : 1; }

VocabPlan plan_for(const arrol_ctx* ctx, int d, int V) {
    // the same for every token count: where the form depends on that, both forms' resident tiles are far below either budget
    return make_vocab_plan(ctx->sm_count, (V + BN - 1) / BN, splits_for(ctx, d, V, pair_for(ctx, INT64_MAX, d)));
}

// Workspace: wave counter, body records, tail records, source rows of the token tiles (gathered variant).  Every part
// grows with T_max alone, so a workspace sized for T_max serves any call on fewer tokens with the same d and V.
struct WorkspaceLayout { size_t body, tail, tile_row, total; };
WorkspaceLayout workspace_layout(const arrol_ctx* ctx, int64_t T_max, int d, int V) {
    const VocabPlan v = plan_for(ctx, d, V);
    WorkspaceLayout L;
    const int halves = halves_for(d);
    auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
    L.body = 256;
    L.tail = L.body + up((size_t)v.splits * halves * (size_t)T_max * sizeof(PartialLse));
    // tail tiles: at most units / splits + 1 tiles of 256 rows for pairs, of 128 rows for twice as many single blocks
    const int64_t most = ((int64_t)(ctx->sm_count / 2) / v.splits + 1) * 2 * BM;
    const int64_t rows = (T_max + 2 * BM - 1) / (2 * BM) * (2 * BM);
    L.tile_row = L.tail + up((size_t)(rows < most ? rows : most) * v.n_sub * halves * sizeof(PartialLse));
    L.total = L.tile_row + up((size_t)(rows / BM) * sizeof(int32_t));
    return L;
}

}  // namespace

extern "C" size_t arrol_token_logprob_workspace(arrol_ctx* ctx, int64_t T_max, int32_t d, int32_t V) {
    if (!ctx || T_max <= 0 || d <= 0 || V <= 0) return 0;
    return workspace_layout(ctx, T_max, d, V).total;
}

extern "C" int32_t arrol_token_logprob_form(arrol_ctx* ctx, int64_t T_max, int32_t d, int32_t V) {
    if (!ctx || T_max <= 0 || d <= 0 || V <= 0) return 0;
    return pair_for(ctx, T_max, d) ? 2 : 1;
}

extern "C" int32_t arrol_token_logprob_splits(arrol_ctx* ctx, int64_t T_max, int32_t d, int32_t V) {
    if (!ctx || T_max <= 0 || d <= 0 || V <= 0) return 0;
    return plan_for(ctx, d, V).splits;
}

// Gather description of the gathered variant: the token rows come from `hidden` = the source buffer of
// `source_rows` rows through (cu_seqlens, survivor_idx, src_tok_off); NULL = `hidden` is the packed [T_max, d] block.
struct GatherArgs {
    const int64_t* cu_seqlens;
    const int32_t* survivor_idx;
    const int64_t* src_tok_off;
    const int64_t* d_num;
    int64_t source_rows;
    int32_t S_max;
};

// bytes of the boundary-tile scratch, placed after the split records in the gathered variant's workspace
static size_t boundary_scratch_bytes(int32_t S_max, int32_t d) { return (size_t)S_max * BM * (size_t)d * 2; }

static int run_token_logprob(arrol_ctx* ctx, const void* hidden, const void* W_vocab, const int32_t* targets,
                             int64_t T_max, const int64_t* d_T, int32_t d, int32_t V, float inv_temperature,
                             float* logp, float* lse, float* conf, void* workspace, size_t workspace_bytes,
                             void* stream, const GatherArgs* ga = nullptr) {
    if (!ctx || T_max < 0 || d <= 0 || V <= 0 || !(inv_temperature > 0.f)) return ARROL_ERR_INVALID_ARG;
    if (T_max == 0) return ARROL_OK;
    if (!hidden || !W_vocab || !targets || !logp) return ARROL_ERR_INVALID_ARG;
    if (d % 8 != 0) return ARROL_ERR_UNSUPPORTED;
    if (!arrol_aligned(hidden, 16) || !arrol_aligned(W_vocab, 16)) return ARROL_ERR_INVALID_ARG;
    if (T_max > (int64_t)INT32_MAX - BM) return ARROL_ERR_UNSUPPORTED;   // TMA coordinates are 32-bit
    const WorkspaceLayout L = workspace_layout(ctx, T_max, d, V);
    const size_t split_bytes = L.total;
    const size_t need = split_bytes + (ga ? boundary_scratch_bytes(ga->S_max, d) : 0);
    if (!workspace || workspace_bytes < need || !arrol_aligned(workspace, 256)) return ARROL_ERR_WORKSPACE;

    ArrolDeviceGuard guard(ctx->device);
    if (!guard.ok) return ARROL_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;

    CUtensorMap map_h, map_s, map_w;
    void* scratch = static_cast<uint8_t*>(workspace) + split_bytes;      // a multiple of 256 bytes
    if (make_map(ctx, &map_h, hidden, (uint64_t)(ga ? ga->source_rows : T_max), (uint64_t)d, BM) != ARROL_OK)
        return ARROL_ERR_CUDA;
    if (ga) {
        if (make_map(ctx, &map_s, scratch, (uint64_t)ga->S_max * BM, (uint64_t)d, BM) != ARROL_OK) return ARROL_ERR_CUDA;
    } else {
        map_s = map_h;
    }
    // pair variant (clusters of two blocks): every block loads half of a chunk's W_vocab rows
    const bool pair = pair_for(ctx, T_max, d);
    if (make_map(ctx, &map_w, W_vocab, (uint64_t)V, (uint64_t)d, pair ? PAIR_B_ROWS : BN) != ARROL_OK) return ARROL_ERR_CUDA;

    LogprobParams p;
    p.targets = targets;
    p.d_T = d_T;
    p.T_max = T_max;
    p.d = d;
    p.V = V;
    p.plan = plan_for(ctx, d, V);
    p.scale2 = inv_temperature * 1.44269504088896340736f;
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    p.body = reinterpret_cast<PartialLse*>(ws + L.body);
    p.tail = reinterpret_cast<PartialLse*>(ws + L.tail);
    int32_t* tile_row = reinterpret_cast<int32_t*>(ws + L.tile_row);
    p.d_status = ctx->d_status;
    p.spin_limit = ctx->test_spin_limit ? ctx->test_spin_limit : SPIN_LIMIT;
    p.mute_producer = ctx->test_mute_producer;
    p.tile_row = tile_row;
    p.wave_counter = reinterpret_cast<unsigned int*>(ws);      // in the call's own workspace: calls on several streams do not share it
    p.timing = ctx->logprob_timing;
    p.timing_items = ctx->logprob_timing_items;

    const int64_t m_tiles = (T_max + BM - 1) / BM;
    typedef void (*KernelFn)(CUtensorMap, CUtensorMap, CUtensorMap, LogprobParams);
    // [pair][two column halves][plain, with confidence, rows in place]
    static const KernelFn kernels[2][2][3] = {
        {{token_logprob_kernel<false, false, false, 1>, token_logprob_kernel<true, false, false, 1>, token_logprob_kernel<false, true, false, 1>},
         {token_logprob_kernel<false, false, false, 2>, token_logprob_kernel<true, false, false, 2>, token_logprob_kernel<false, true, false, 2>}},
        {{token_logprob_kernel<false, false, true, 1>, token_logprob_kernel<true, false, true, 1>, token_logprob_kernel<false, true, true, 1>},
         {token_logprob_kernel<false, false, true, 2>, token_logprob_kernel<true, false, true, 2>, token_logprob_kernel<false, true, true, 2>}}};
    if (!ctx->logprob_smem_set) {
        for (const auto& form : kernels)
            for (const auto& width : form)
                for (const KernelFn f : width)
                    ARROL_CUDA_OK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES));
        ctx->logprob_smem_set = true;
    }
    const int halves = halves_for(d);
    const int variant = ga ? 2 : (conf ? 1 : 0);
    const KernelFn fn = kernels[pair ? 1 : 0][halves - 1][variant];
    // the units that take the work items: blocks, or pairs of blocks on 256 rows
    const int64_t tiles_max = pair ? (m_tiles + 1) / 2 : m_tiles;
    int64_t units = pair ? ctx->sm_count / 2 : ctx->sm_count;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(num_threads(halves));
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = s;
    cudaLaunchAttribute attr[3];
    int n_attr = 0;
    if (pair) {
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr].val.clusterDim.x = 2;
        attr[n_attr].val.clusterDim.y = 1;
        attr[n_attr].val.clusterDim.z = 1;
        ++n_attr;
        // Pairs are kept in step per wave, so no more of them than fit the GPU at once (asked once per context and kernel
        // variant).  The cooperative attribute would have the driver see to it that they also are resident at once, but the
        // profiler cannot launch a cooperative grid of clusters that fills the GPU ("LaunchFailed"; the same grid without the
        // attribute profiles), and the waits do without (see the top of this file).
        if (ctx->pair_max_clusters[halves - 1][variant] == 0) {
            cfg.gridDim = dim3((unsigned)(2 * units));
            cfg.attrs = attr;
            cfg.numAttrs = n_attr;
            int fit = 0;
            ARROL_CUDA_OK(cudaOccupancyMaxActiveClusters(&fit, fn, &cfg));
            if (fit < 1) return ARROL_ERR_CUDA;
            ctx->pair_max_clusters[halves - 1][variant] = fit;
        }
        if (units > ctx->pair_max_clusters[halves - 1][variant]) units = ctx->pair_max_clusters[halves - 1][variant];
    }
    if (units > tiles_max * p.plan.n_sub) units = tiles_max * p.plan.n_sub;
    const int64_t grid = pair ? 2 * units : units;
    // more than one wave: the blocks are kept in step, and should all be resident (single blocks: cooperative launch)
    p.work = make_work_list((int)tiles_max, (int)units, p.plan);
    const bool several_waves = p.work.waves > 1;
    if (several_waves) ARROL_CUDA_OK(cudaMemsetAsync(p.wave_counter, 0, sizeof(unsigned int), s));
    if (several_waves && !pair) {
        attr[n_attr].id = cudaLaunchAttributeCooperative;
        attr[n_attr].val.cooperative = 1;
        ++n_attr;
    } else {
        attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
        ++n_attr;
    }
    cfg.gridDim = dim3((unsigned)grid);
    cfg.attrs = attr;
    cfg.numAttrs = n_attr;
    if (ga) {
        const int blocks = ga->S_max < ctx->sm_count * 4 ? ga->S_max : ctx->sm_count * 4;
        const int passes = (BM * (d / 8) + PACK_PASS - 1) / PACK_PASS;
        int columns = ctx->sm_count * 4 / blocks;
        if (columns > passes) columns = passes;
        ARROL_CUDA_OK(arrol_launch_pdl(pack_boundary_tiles_kernel, dim3((unsigned)blocks, (unsigned)columns), dim3(PACK_THREADS), 0, s,
                                       static_cast<const uint4*>(hidden), ga->cu_seqlens, ga->survivor_idx,
                                       ga->src_tok_off, ga->d_num, ga->S_max, T_max, d / 8, static_cast<uint4*>(scratch), tile_row));
        ctx->launches += 1;
    }
    ARROL_CUDA_OK(cudaLaunchKernelEx(&cfg, fn, map_h, map_s, map_w, p));
    ctx->launches += 1;
    ARROL_CUDA_OK(cudaGetLastError());
    // a thread per token of the body; tokens of the tail a few per block, so that the blocks are as many as SMs if they can be
    const int64_t tile_rows = (pair ? 2 : 1) * BM;
    const bool tail_only = p.work.body_tiles == 0;      // fewer tokens have none either
    int64_t tail_rows = (tiles_max < units / p.plan.splits + 1 ? tiles_max : units / p.plan.splits + 1) * tile_rows;
    if (tail_rows > T_max) tail_rows = T_max;
    const int group = combine_group(p.plan, halves, tail_rows, ctx->sm_count, SMEM_BYTES);
    int64_t blocks = (tail_rows + group - 1) / group;
    int block_lanes = 0;
    while ((1 << block_lanes) < p.plan.n_mid * halves) ++block_lanes;
    if (!tail_only) {
        if (blocks < (T_max + COMBINE_THREADS - 1) / COMBINE_THREADS) blocks = (T_max + COMBINE_THREADS - 1) / COMBINE_THREADS;
        if (blocks > (int64_t)ctx->sm_count * 8) blocks = (int64_t)ctx->sm_count * 8;
    }
    const auto combine = halves == 2 ? combine_splits_kernel<2> : combine_splits_kernel<1>;
    ARROL_CUDA_OK(arrol_launch_pdl(combine, dim3((unsigned)blocks), dim3(COMBINE_THREADS), (size_t)group * combine_bytes(p.plan, halves), s,
                                   static_cast<const PartialLse*>(p.body), static_cast<const PartialLse*>(p.tail), targets, d_T,
                                   T_max, V, p.plan, (int)tile_rows, (int)units, group, block_lanes, tail_only, logp, lse, conf, inv_temperature, ctx->d_status));
    ctx->launches += 1;
    return ARROL_OK;
}

extern "C" int arrol_token_logprob(arrol_ctx* ctx, const void* hidden, const void* W_vocab, const int32_t* targets,
                                   int64_t T_max, const int64_t* d_T, int32_t d, int32_t V, float inv_temperature,
                                   float* logp, float* lse, void* workspace, size_t workspace_bytes,
                                   void* stream) {
    return run_token_logprob(ctx, hidden, W_vocab, targets, T_max, d_T, d, V, inv_temperature, logp, lse, nullptr,
                             workspace, workspace_bytes, stream);
}

extern "C" int arrol_token_logprob_conf(arrol_ctx* ctx, const void* hidden, const void* W_vocab, const int32_t* targets,
                                        int64_t T_max, const int64_t* d_T, int32_t d, int32_t V, float inv_temperature,
                                        float* logp, float* lse, float* token_conf, void* workspace,
                                        size_t workspace_bytes, void* stream) {
    if (T_max > 0 && !token_conf) return ARROL_ERR_INVALID_ARG;
    return run_token_logprob(ctx, hidden, W_vocab, targets, T_max, d_T, d, V, inv_temperature, logp, lse, token_conf,
                             workspace, workspace_bytes, stream);
}

extern "C" size_t arrol_token_logprob_gathered_workspace(arrol_ctx* ctx, int32_t S_max, int64_t T_max, int32_t d,
                                                         int32_t V) {
    if (!ctx || S_max <= 0 || T_max <= 0 || d <= 0 || V <= 0) return 0;
    return arrol_token_logprob_workspace(ctx, T_max, d, V) + boundary_scratch_bytes(S_max, d);
}

extern "C" int arrol_token_logprob_gathered(arrol_ctx* ctx, const void* src_rows, int64_t source_rows,
                                            const void* W_vocab, const int32_t* targets, const int64_t* cu_seqlens,
                                            const int32_t* survivor_idx, const int64_t* src_tok_off,
                                            const int64_t* d_num, int32_t S_max, int64_t T_max, int32_t d, int32_t V,
                                            float inv_temperature, float* logp, float* lse, void* workspace,
                                            size_t workspace_bytes, void* stream) {
    if (!ctx || S_max < 0 || source_rows < 0 || T_max < 0) return ARROL_ERR_INVALID_ARG;
    if (T_max == 0 || S_max == 0) return ARROL_OK;
    if (!cu_seqlens || !survivor_idx || !src_tok_off || !d_num || source_rows == 0) return ARROL_ERR_INVALID_ARG;
    if (source_rows > (int64_t)INT32_MAX - BM || (int64_t)S_max * BM > (int64_t)INT32_MAX - BM)
        return ARROL_ERR_UNSUPPORTED;                                            // TMA coordinates are 32-bit
    GatherArgs ga = {cu_seqlens, survivor_idx, src_tok_off, d_num, source_rows, S_max};
    return run_token_logprob(ctx, src_rows, W_vocab, targets, T_max, d_num + 1, d, V, inv_temperature, logp, lse,
                             nullptr, workspace, workspace_bytes, stream, &ga);
}
