// arrol_lm_head_backward: gradient of the selected-token log-probs through the lm_head (Section 3: the policy
// update differentiates log pi_theta(o_t | o_<t); Algorithm 1 "Backprop ... on policy").
//
//   z = inv_temp H W^T,  logp_t = z_{t,y_t} - lse_t,  given g_t = dL/dlogp_t and lse_t from the forward call:
//   dz_{t,v} = g_t inv_temp ([v = y_t] - exp(z_{t,v} - lse_t)),   dH = dz W,   dW = dz^T H.
//
// The tokens are processed in chunks of TC rows.  Per chunk, three tensor-core kernels with the same
// TMA -> shared memory -> tcgen05.mma -> tensor memory pipeline as the forward kernel:
//   dz_kernel     recomputes the chunk's logits tile by tile and turns each accumulator tile into dz (bf16),
//                 written once as dZ [TC, V]
//   gemm_kernel   dH[chunk] = dZ . W       A = dZ K-major (K = V contiguous), B = W MN-major (N = d contiguous)
//   gemm_kernel   dW       (+)= dZ^T . H   A = dZ MN-major (M = V contiguous), B = H chunk MN-major
// The MN-major operands are read by the tensor core straight from their row-major storage (transpose bits in the
// instruction descriptor, MN-major shared-memory descriptors), so nothing is transposed in memory and the T x V
// matrix exists only one chunk at a time, once, in the workspace.
//
// All three work as PAIRS of blocks (clusters of two, tcgen05 cta_group::2) on 256 x 256 tiles: block r of a pair owns
// the tile's rows 128 r ..., brings them and half of the tile's 256 columns of B, and runs the epilogue of its rows;
// block 0 issues the MMAs for both.  Per block and K step 32 KB come in from L2 instead of the 48 KB of a 128 x 256 tile of
// its own.  These kernels are bound by the board's power cap and by the SM-to-L2 path, which their results share with
// the operands, not by the issue of MMAs (a warp-uniform issuer alone changed nothing), so fewer operand bytes are what
// helps.  Whole call against single blocks (which also walked the dead tiles of a partly live chunk): 47,360 tokens,
// d = 2048, V = 128,256 59.0 -> 56.8 ms; 28,000, d = 4096, V = 151,936 85.8 -> 78.6 ms; 3,000, d = 2048 6.78 -> 3.92 ms; 600,
// d = 1024, V = 30,000 689 -> 221 us.
#include "arrol_internal.h"
#include "tc_common.cuh"

namespace {

constexpr int BM = 128, BN = CHUNK_COLUMNS;   // rows of a block, columns of a tile
constexpr int TILE_ROWS = 2 * BM;        // rows of a pair's tile
constexpr int A_STAGE_BYTES = BM * BK * 2;
constexpr int B_STAGE_BYTES = BN / 2 * BK * 2;
constexpr int STAGE_BYTES = A_STAGE_BYTES + B_STAGE_BYTES;
constexpr int MN_BLOCK_BYTES = BK * 128;   // one 64-element MN block of an MN-major stage: BK rows of 128 bytes
constexpr int TMEM_COLS = 512;
constexpr int STAGES = 6;
constexpr int EPI_WARPS = 8;            // two warps per tensor-memory lane quarter, each takes half of the columns
constexpr int NUM_THREADS = 64 + 32 * EPI_WARPS;
constexpr int EPI_PIECES = BN / 32 / (EPI_WARPS / 4);   // 32-column pieces per epilogue warp and accumulator
// one 32-row x 128-byte staging tile per epilogue warp behind the barrier block (1 KB), 1024-byte aligned: results go through it to
// leave in whole 128-byte lines
constexpr int EPI_STAGE_TILE = 32 * 128;
constexpr size_t EPI_STAGE_OFFSET = (size_t)STAGES * STAGE_BYTES + 1024;
constexpr size_t SMEM_BYTES = EPI_STAGE_OFFSET + (size_t)EPI_WARPS * EPI_STAGE_TILE + 1024;
constexpr int TC = 37 * TILE_ROWS;      // tokens per chunk: 37 tiles of a pair, so that TC/256 x d/256 tiles fill 74 pairs evenly

struct PipeSmem {
    uint8_t* stage_a;
    uint8_t* stage_b;
    uint64_t *full, *empty, *acc_full, *acc_empty, *drain;
    uint32_t* tmem_slot;
    volatile uint32_t* abort_flag;
    volatile uint32_t* lock_seen;            // copy of the lock-step counter, 16 bytes
    uint32_t rank;                           // of this block in its pair (0 leads)
    uint32_t tmem_base;
    uint32_t lead_full, lead_acc_empty;      // shared::cluster addresses in the leading block
};

// Common prologue: barriers, tensor-memory allocation, then the wait for the preceding kernel (everything before it
// overlaps that kernel's end).
__device__ __forceinline__ PipeSmem pipe_setup(uint8_t* smem_raw, const CUtensorMap* ma, const CUtensorMap* mb) {
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    PipeSmem ps;
    ps.stage_a = smem;
    ps.stage_b = smem + (size_t)STAGES * A_STAGE_BYTES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)STAGES * STAGE_BYTES);
    ps.full = bars;
    ps.empty = bars + STAGES;
    ps.acc_full = bars + 2 * STAGES;
    ps.acc_empty = ps.acc_full + 2;
    ps.drain = ps.acc_empty + 2;
    ps.tmem_slot = reinterpret_cast<uint32_t*>(ps.drain + 1);
    ps.abort_flag = ps.tmem_slot + 1;
    ps.lock_seen = reinterpret_cast<uint32_t*>(smem + (size_t)STAGES * STAGE_BYTES + 512);
    ps.rank = cluster_cta_rank();
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&ps.full[s], 1); mbar_init(&ps.empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&ps.acc_full[b], 1); mbar_init(&ps.acc_empty[b], 2 * EPI_WARPS); }
        mbar_init(ps.drain, 1);
        *ps.abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(ma) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(mb) : "memory");
    }
    if ((threadIdx.x >> 5) == 1) {
        tcgen05_alloc_pair(ps.tmem_slot, TMEM_COLS);
        tcgen05_relinquish_pair();
    }
    tcgen05_fence_before();
    __syncthreads();
    cluster_sync_all();                      // the peer's barriers exist before anything arrives on them
    tcgen05_fence_after();
    ps.tmem_base = *ps.tmem_slot;
    ps.lead_full = map_to_cta(smem_u32(&ps.full[0]), 0u);
    ps.lead_acc_empty = map_to_cta(smem_u32(&ps.acc_empty[0]), 0u);
    pdl_launch_dependents();
    pdl_wait();
    return ps;
}

__device__ __forceinline__ void pipe_teardown(const PipeSmem& ps, uint32_t* d_status) {
    tcgen05_fence_before();
    __syncthreads();
    cluster_sync_all();                      // neither block's shared or tensor memory goes away under the other
    if (threadIdx.x == 0 && *ps.abort_flag) atomicOr(d_status, ARROL_DEV_WAIT_EXPIRED);
    if ((threadIdx.x >> 5) == 1) {
        tcgen05_fence_after();
        tcgen05_dealloc_pair(ps.tmem_base, TMEM_COLS);
    }
}

// Pairs in step.  The pairs of a launch share operand panels through L2, but only while they read them at about the same
// time, and nothing in a persistent kernel keeps them together: measured at d = 4,096, the dH contraction of a chunk read 33 GB
// from HBM where 11 would do and ran at 1.09 GHz under the power cap, the dz kernel beside it, with its little traffic, at 1.27.
// So about every EPOCH K steps the leading producer of a pair reports on a counter in global memory and waits until there are
// as many reports as all pairs make up to two epochs ago: no pair gets more than two epochs ahead of the average.  (A single
// straggler is not waited for by name: the reports of the pairs ahead stand in for its own.)  The counter is fetched an epoch
// ahead by an asynchronous copy into shared memory, so a pair that is not ahead does not wait for memory either.
// (A plain load of the counter by one thread at every epoch cost the tensor pipe 6-14 % of the cycles.)  One chunk alone, without
// and with it: d = 2,048, V = 128,256 HBM reads of dH 12.0 -> 6.8 GB, of dW 8.9 -> 6.1, the three kernels 10.4 -> 10.0 ms; d = 4,096,
// V = 151,936 34 -> 17 and 25 -> 15.5 GB, 25.7 -> 24.0 ms.  Over seconds, where the power cap evens it out, an update of a
// DAPO-shaped micro-batch takes 70.3 -> 69.4 ms.  Epochs of 8 steps reach the least traffic (4.9 and 4.7 GB, 11.7 and 11.2) but
// gain nothing more over seconds.
//   The results do not depend on it, and nothing may: the pairs of another launch, on another stream, can hold the SMs that some
// of these pairs still need, and wait for their own absent pairs in turn.  So the wait is a short one, far above what pairs
// that run side by side ever wait, and a pair that has waited that long goes on, reports as before and waits no more.
constexpr int EPOCH = 16;
constexpr uint32_t LOCK_TRIES = 128;   // of half a microsecond or more; an epoch takes about three
// The counters of a call, one per kernel, in one 16-byte group.  Each kernel zeroes the next one's, which its last user, a
// chunk ago, is done with and its next one, the following launch, has not begun to use.
enum LockWord { LOCK_DZ, LOCK_DH, LOCK_DW, LOCK_WORDS };
constexpr size_t LOCK_BYTES = 16;
struct Lockstep {
    unsigned int* words;        // 16-byte aligned; this kernel's is zero before the launch
    int word;
    uint32_t units, epochs;     // epochs of the pair with the most work
    int items_per_epoch;        // > 1 when a tile has few K steps
    bool on;                    // false: the pairs go as they like, and the counter is not touched
};
// `body` items of k_steps K steps each, then `tail` items of at most tail_steps (the same number where k_steps < EPOCH)
__device__ __forceinline__ Lockstep lockstep_for(unsigned int* words, int word, int64_t units, int64_t body, int k_steps, int64_t tail,
                                                 int tail_steps) {
    Lockstep l;
    l.words = words;
    l.word = word;
    l.units = (uint32_t)units;
    l.on = true;
    l.items_per_epoch = k_steps >= EPOCH ? 1 : EPOCH / max(k_steps, 1);
    const int64_t most = (body + units - 1) / units, most_tail = (tail + units - 1) / units;
    l.epochs = (uint32_t)(k_steps >= EPOCH ? most * ((k_steps + EPOCH - 1) / EPOCH) + most_tail * ((tail_steps + EPOCH - 1) / EPOCH)
                                           : (most + most_tail + l.items_per_epoch - 1) / l.items_per_epoch);
    return l;
}
// One thread, at the beginning of its pair's epoch `epoch`.  False: waited in vain.
__device__ __forceinline__ bool begin_epoch(const Lockstep& lock, volatile uint32_t* seen, uint32_t epoch) {
    unsigned int* counter = lock.words + lock.word;
    atomicAdd(counter, 1u);
    cp_async_wait_all();
    const uint32_t target = epoch < 2 ? 0u : (epoch - 1) * lock.units;       // the average pair has begun epoch - 2
    if (seen[lock.word] < target)
        for (uint32_t spin = 0; ld_relaxed_u32(counter) < target; ++spin) {
            if (spin >= LOCK_TRIES) return false;
            __nanosleep(32);
        }
    cp_async_16(seen, lock.words);                                            // looked at when the next epoch begins
    return true;
}

// One accumulator tile's operands: origin of the tile's rows (A) and columns (B), the columns that the MMA computes, the K steps
// [k0, k1), and where the result goes: the output (slot < 0) or a slot of partial sums.
struct TileAt { int a0, b0, n, k0, k1, slot; };

// Producer role (one warp of each block; the warp walks the loops and waits, one elected lane issues).  For every accumulator tile `coords(it, tile)` gives the operands' MN origins
// (false when the list is exhausted); this block loads rows a0 + 128 rank ... of A and b0 + (n / 2) rank ... of B.  Per K step
//   K-major operand:  one box  [128 MN rows x 64 K columns]      at (x = k, y = mn0)
//   MN-major operand: 2 blocks [64 K rows x 64 MN columns], BK*128 bytes apart: one three-dimensional box
//                     (64 elements, 64 K rows, 2 blocks) at (0, k, mn0/64) when the map is of that kind
//                     (a3d / b3d), else one two-dimensional box per block at (x = mn0 + 64 b, y = k).
// Both blocks' bytes are counted on the leading block's barrier.
template <bool A_MN, bool B_MN, typename Coords>
__device__ __forceinline__ void producer_loop(const PipeSmem& ps, const CUtensorMap* ma, const CUtensorMap* mb,
                                              const Lockstep& lock, Coords coords, bool a3d = false, bool b3d = false,
                                              const CUtensorMap* mb_tail = nullptr, int tail_ks = -1) {
    const uint32_t a0 = smem_u32(ps.stage_a), b0 = smem_u32(ps.stage_b);
    uint32_t stage = 0, phase = 0, issued = 0, epoch = 0;
    bool ok = true, in_step = lock.on;
    TileAt tile;
    int to_epoch = 0;                     // items until the next epoch
    if (blockIdx.x == 0 && elect_one()) lock.words[(lock.word + 1) % LOCK_WORDS] = 0u;
    for (int64_t it = 0; ok && coords(it, tile); ++it) {
        const int ay = tile.a0 + (int)ps.rank * BM, by = tile.b0 + (int)ps.rank * (tile.n / 2);
        for (int ks0 = tile.k0; ks0 < tile.k1 && ok; ks0 += EPOCH) {
            if (ks0 > tile.k0 || to_epoch == 0) {
                if (lock.on && ps.rank == 0) {
                    if (elect_one()) {
                        if (in_step) in_step = begin_epoch(lock, ps.lock_seen, epoch);
                        else atomicAdd(lock.words + lock.word, 1u);
                    }
                    in_step = __all_sync(0xffffffffu, in_step) != 0;
                }
                ++epoch;
                if (ks0 == tile.k0) to_epoch = lock.items_per_epoch;
            }
            const int ks1 = min(ks0 + EPOCH, tile.k1);
            for (int ks = ks0; ks < ks1; ++ks) {
                if (!mbar_wait_warp(&ps.empty[stage], phase ^ 1u, ps.abort_flag)) { ok = false; break; }
                if (elect_one()) {
                    const uint32_t bar = ps.lead_full + stage * (uint32_t)sizeof(uint64_t);
                    if (ps.rank == 0) mbar_expect_tx(&ps.full[stage], 2 * STAGE_BYTES);
                    const uint32_t sa = a0 + stage * A_STAGE_BYTES, sb = b0 + stage * B_STAGE_BYTES;
                    if constexpr (A_MN) {
                        if (a3d) {
                            tma_load_3d_pair(sa, ma, 0, ks * BK, ay >> 6, bar);
                        } else {
#pragma unroll
                            for (int b = 0; b < BM / 64; ++b)
                                tma_load_2d_pair(sa + b * MN_BLOCK_BYTES, ma, ay + 64 * b, ks * BK, bar);
                        }
                    } else {
                        tma_load_2d_pair(sa, ma, ks * BK, ay, bar);
                    }
                    if constexpr (B_MN) {
                        // the K step that holds the last, partly live block of rows is read from its zero-padded copy
                        const bool tail = ks == tail_ks;
                        const CUtensorMap* m = tail ? mb_tail : mb;
                        const int ky = tail ? 0 : ks * BK;
                        if (b3d) {
                            tma_load_3d_pair(sb, m, 0, ky, by >> 6, bar);
                        } else {
#pragma unroll
                            for (int b = 0; b < BN / 2 / 64; ++b)
                                tma_load_2d_pair(sb + b * MN_BLOCK_BYTES, m, by + 64 * b, ky, bar);
                        }
                    } else {
                        tma_load_2d_pair(sb, mb, ks * BK, by, bar);
                    }
                }
                __syncwarp();
                ++issued;
                if (++stage == STAGES) { stage = 0; phase ^= 1u; }
            }
        }
        --to_epoch;
    }
    if (lock.on && ps.rank == 0 && elect_one()) {
        cp_async_wait_all();
        if (epoch < lock.epochs) atomicAdd(lock.words + lock.word, lock.epochs - epoch);   // done: nobody waits for this pair
    }
    if (!ok && ps.rank == 0 && elect_one()) {
        // gave up: let the copies already issued land before shared memory goes away (bounded); the peer's copies are
        // counted here too, and the cluster barrier at the end keeps its shared memory alive until then
        const uint32_t pending = issued < (uint32_t)STAGES ? issued : (uint32_t)STAGES;
        uint32_t s = stage, ph = phase;
        for (uint32_t i = 0; i < pending; ++i) {
            if (s == 0) { s = STAGES - 1; ph ^= 1u; } else { --s; }
            for (uint32_t spin = 0; spin < SPIN_LIMIT; ++spin)
                if (mbar_try_wait(&ps.full[s], ph)) break;
        }
    }
    __syncwarp();
}

// MMA role (one warp of the leading block): the accumulator tiles that `coords(it, tile)` lists (false: no more), the last of all
// k_steps K steps having k_last slices of 16, alternating the two accumulators.  The whole warp
// walks the loops and waits, one elected lane issues.
// Inside a stage the four K = 16 slices are 32 bytes apart for a K-major operand (columns of the swizzled row) and
// 16 rows = 2048 bytes apart for an MN-major one.
template <bool A_MN, bool B_MN, typename Coords>
__device__ __forceinline__ void mma_loop(const PipeSmem& ps, int k_steps, int k_last, Coords coords) {
    constexpr uint64_t a_step = A_MN ? (UMMA_K * 128) >> 4 : (UMMA_K * 2) >> 4;
    constexpr uint64_t b_step = B_MN ? (UMMA_K * 128) >> 4 : (UMMA_K * 2) >> 4;
    const uint32_t a0 = smem_u32(ps.stage_a), b0 = smem_u32(ps.stage_b);
    uint32_t stage = 0, phase = 0, acc = 0, acc_phase = 0;
    bool ok = true;
    TileAt tile;
    for (int64_t it = 0; ok && coords(it, tile); ++it) {
        const uint32_t idesc = make_idesc(TILE_ROWS, tile.n, A_MN, B_MN);
        if (!mbar_wait_warp(&ps.acc_empty[acc], acc_phase ^ 1u, ps.abort_flag)) { ok = false; break; }
        tcgen05_fence_after();
        const uint32_t d_tmem = ps.tmem_base + acc * BN;
        const int k0 = tile.k0, k1 = tile.k1;
        for (int ks = k0; ks < k1; ++ks) {
            if (!mbar_wait_warp(&ps.full[stage], phase, ps.abort_flag)) { ok = false; break; }
            tcgen05_fence_after();
            const uint32_t sa = a0 + stage * A_STAGE_BYTES, sb = b0 + stage * B_STAGE_BYTES;
            const uint64_t a_desc = A_MN ? make_smem_desc_mn(sa, BK) : make_smem_desc(sa);
            const uint64_t b_desc = B_MN ? make_smem_desc_mn(sb, BK) : make_smem_desc(sb);
            if (elect_one()) {
                if (ks + 1 < k_steps || k_last == BK / UMMA_K) {
#pragma unroll
                    for (int k = 0; k < BK / UMMA_K; ++k)
                        tcgen05_mma_bf16_pair(d_tmem, a_desc + a_step * k, b_desc + b_step * k, idesc, ((ks - k0) | k) != 0 ? 1u : 0u);
                } else {
                    for (int k = 0; k < k_last; ++k)         // slices past the end of K are zeros
                        tcgen05_mma_bf16_pair(d_tmem, a_desc + a_step * k, b_desc + b_step * k, idesc, ((ks - k0) | k) != 0 ? 1u : 0u);
                }
                tcgen05_commit_pair(&ps.empty[stage], (uint16_t)3);
                if (ks + 1 == k1) tcgen05_commit_pair(&ps.acc_full[acc], (uint16_t)3);
            }
            __syncwarp();
            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
    if (!ok && elect_one()) {
        tcgen05_commit_pair(ps.drain, (uint16_t)1);
        for (uint32_t spin = 0; spin < SPIN_LIMIT; ++spin)
            if (mbar_try_wait(ps.drain, 0u)) break;
    }
    __syncwarp();
}

__device__ __forceinline__ int64_t live_tokens(const int64_t* d_T, int64_t T_max) {
    int64_t T = T_max;
    if (d_T) { const int64_t t = *pdl_acquire(d_T); T = t < 0 ? 0 : (t < T ? t : T); }
    return T;
}

// ---- dz: recompute logits, write the softmax gradient of one token chunk --------------------------------------
// Work item = (vocabulary chunk of 256 columns, token tile), the chunk as the slow index: the pairs share W_vocab chunks and
// token tiles through L2, and a chunk with few live tiles still spreads evenly.  When the token tiles of the whole chunk
// outgrow L2's share (50 MB, as in the forward kernel), they go in groups of `group_tiles`, each with its own pass over W_vocab.
struct DzParams {
    const int32_t* targets;
    const float* grad_logp;
    const float* lse;
    const int64_t* d_T;
    int64_t T_max, t0;        // chunk = tokens [t0, t0 + TC)
    int d, V;
    int group_tiles;
    float scale2, inv_temp;
    const uint16_t* hidden;
    unsigned int* lock_words;
    int lock_on;
    uint16_t* dz;             // [TC, ldz]
    int64_t ldz;
    uint16_t* tail;           // [63, d]: the last, partly live 64-row block of the chunk's hidden rows, zero-padded
    uint32_t* d_status;
};

__device__ __forceinline__ bool dz_item(int64_t i, int m_tiles, int total_chunks, int group_tiles, int& m, int& c) {
    const int64_t per_group = (int64_t)group_tiles * total_chunks;
    const int64_t g = i / per_group;
    const int first = (int)g * group_tiles;
    if (first >= m_tiles) return false;
    const int size = min(group_tiles, m_tiles - first);
    i -= g * per_group;
    if (i >= (int64_t)size * total_chunks) return false;
    c = (int)(i / size);
    m = first + (int)(i - (int64_t)c * size);
    return true;
}

// What bounds it: the MMAs (8 d cycles of an SM per tile) from d of about 400 on.  Below that the epilogue: 32,768 exponentials a tile and
// SM take the special-function units 2,048 cycles, and what a warp does for its 32 x 128 share takes it about 3,800.  It took 5,500 to
// 8,000 while results left by TMA tile stores, which queue behind the operand copies in flight, from a staging tile that had to be free
// again; while the accumulator was handed back by a release, which waited for those stores; and while the row's target and gradient
// were fetched when the tile had already arrived.  Now whole lines are read back from the staging tile and stored directly, rows are
// requested a tile ahead, and an element costs 3 to 4 instructions: two at a time in packed fp32, the target column, which few
// pieces hold, by a loop of its own.  (Sixteen warps with less staging each: no gain with tile stores, 10 % slower with direct ones.)
// 700 tokens, d = 320, V = 151,936: whole update 358 -> 303 us, with the dH kernel's epilogue in the same manner; 12,000, d = 512,
// V = 30,000 1,025 -> 970; 12,000, d = 2,048, V = 60,000 6,430 -> 6,250.
__global__ void __launch_bounds__(NUM_THREADS, 1)
dz_kernel(const __grid_constant__ CUtensorMap map_h, const __grid_constant__ CUtensorMap map_w, const DzParams p) {
    extern __shared__ uint8_t smem_raw[];
    const PipeSmem ps = pipe_setup(smem_raw, &map_h, &map_w);
    uint8_t* dz_stage = ps.stage_a + EPI_STAGE_OFFSET;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t T = live_tokens(p.d_T, p.T_max);
    const int live = (int)max((int64_t)0, min((int64_t)TC, T - p.t0));     // 0: chunk past the live tokens, nothing to do
    const int m_tiles = (live + TILE_ROWS - 1) / TILE_ROWS;
    const int k_steps = (p.d + BK - 1) / BK;
    const int k_last = (p.d - (k_steps - 1) * BK + UMMA_K - 1) / UMMA_K;
    const int total_chunks = (p.V + BN - 1) / BN;
    const int64_t unit = blockIdx.x >> 1, units = gridDim.x >> 1;
    auto coords = [&](int64_t it, TileAt& t) {
        int m, c;
        if (!dz_item(unit + it * units, m_tiles, total_chunks, p.group_tiles, m, c)) return false;
        t.a0 = (int)p.t0 + m * TILE_ROWS;
        t.b0 = c * BN;
        t.n = chunk_columns(p.V, c);
        t.k0 = 0;
        t.k1 = k_steps;
        return true;
    };

    if (warp == 0) {
        Lockstep lock = lockstep_for(p.lock_words, LOCK_DZ, units, (int64_t)m_tiles * total_chunks, k_steps, 0, 0);
        lock.on = p.lock_on != 0;
        producer_loop<false, false>(ps, &map_h, &map_w, lock, coords);
    } else if (warp == 1) {
        if (ps.rank == 0) mma_loop<false, false>(ps, k_steps, k_last, coords);
    } else {
        // The last, partly live 64-row block of the chunk's hidden rows, padded with zeros, for the dW contraction: rows past
        // the live tokens (caller memory that may hold anything) never reach the tensor core.  At most 63 rows live in it; the
        // copy fills the 64th with zeros by itself.
        if (live % BK != 0) {
            const int r0 = live / BK * BK, vec_per_row = p.d / 8;
            const uint16_t* hidden = pdl_acquire(p.hidden);
            for (int i = (int)blockIdx.x * 32 * EPI_WARPS + (int)threadIdx.x - 64; i < (BK - 1) * vec_per_row; i += (int)gridDim.x * 32 * EPI_WARPS) {
                const int r = i / vec_per_row, v = i - r * vec_per_row;
                uint4 x = make_uint4(0u, 0u, 0u, 0u);
                if (r0 + r < live) x = *reinterpret_cast<const uint4*>(hidden + (p.t0 + r0 + r) * p.d + v * 8);
                *reinterpret_cast<uint4*>(p.tail + (int64_t)r * p.d + v * 8) = x;
            }
        }
        const int32_t* targets = pdl_acquire(p.targets);
        const float* grad_logp = pdl_acquire(p.grad_logp);
        const float* lse = pdl_acquire(p.lse);
        const int quarter = warp & 3;
        const int col_half = (warp - 2) >> 2;           // which half of the accumulator's columns
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        // dz leaves through shared memory: the warp's 32 rows x 64 columns (two pieces, 128 bytes per row, 128-byte
        // swizzle) are staged and written in whole 128-byte lines.  (16-byte stores straight from the registers touch 32 lines per
        // instruction and cost the kernel 14 %.)  Columns past V go as far as the row's padding, which nobody reads.
        uint8_t* stg = dz_stage + (size_t)(warp - 2) * EPI_STAGE_TILE;
        uint32_t acc = 0, acc_phase = 0;
        bool ok = true;
        int m, c, m_next = 0, c_next = 0;
        // the row's target, gradient and log-sum-exp, requested a tile ahead
        int y_raw = -1;
        float grad_raw = 0.f, lse_raw = 0.f;
        auto request_row = [&](int tile) {
            const int64_t t = p.t0 + tile * TILE_ROWS + (int)ps.rank * BM + quarter * 32 + lane;
            y_raw = -1;
            if (t < T) {
                y_raw = targets[t];
                grad_raw = grad_logp[t];
                lse_raw = lse[t];
            }
        };
        int64_t item = unit;
        bool have = dz_item(item, m_tiles, total_chunks, p.group_tiles, m, c);
        if (have) request_row(m);
        while (ok && have) {
            item += units;
            const bool have_next = dz_item(item, m_tiles, total_chunks, p.group_tiles, m_next, c_next);
            const int row0 = m * TILE_ROWS + (int)ps.rank * BM + quarter * 32, first_col = c * BN;
            const bool valid = y_raw >= 0 && y_raw < p.V;
            const int y = valid ? y_raw : -1;
            const float coef = valid ? grad_raw * p.inv_temp : 0.f;
            const float lse2 = valid ? lse_raw * 1.44269504088896340736f : 0.f;
            if (have_next) request_row(m_next);
            ok = mbar_wait(&ps.acc_full[acc], acc_phase, ps.abort_flag);
            ok = __all_sync(0xffffffffu, ok) != 0;
            if (!ok) break;
            tcgen05_fence_after();
            const uint32_t tacc = ps.tmem_base + lane_addr + acc * BN;
            const uint32_t live_mask = coef == 0.f ? 0u : ~0u;    // rows that carry no gradient are zeros whatever their logits and lse hold
            const uint64_t scale_2 = pack_f32x2(p.scale2, p.scale2), lse_2 = pack_f32x2(-lse2, -lse2), coef_2 = pack_f32x2(-coef, -coef);
            // dz = coef ([v = y] - 2^(z log2e - lse log2e)), two columns at a time
            auto to_dz = [&](const uint32_t (&raw)[32], int piece, uint32_t (&packed)[16]) {
                const int pc0 = first_col + piece * 32;
#pragma unroll
                for (int j = 0; j < 32; j += 2) {
                    float e0, e1, d0, d1;
                    unpack_f32x2(fma_f32x2(((uint64_t)raw[j + 1] << 32) | raw[j], scale_2, lse_2), e0, e1);
                    unpack_f32x2(mul_f32x2(pack_f32x2(ex2_approx(e0), ex2_approx(e1)), coef_2), d0, d1);
                    const __nv_bfloat162 h2 = __floats2bfloat162_rn(d0, d1);
                    packed[j >> 1] = *reinterpret_cast<const uint32_t*>(&h2) & live_mask;
                }
                if (__any_sync(0xffffffffu, (unsigned)(y - pc0) < 32u)) {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (pc0 + j == y) {
                            const float e = fmaf(__uint_as_float(raw[j]), p.scale2, -lse2);
                            const __nv_bfloat16 h = __float2bfloat16_rn(-coef * ex2_approx(e) + coef);
                            const uint32_t bits = (uint32_t)*reinterpret_cast<const uint16_t*>(&h) & live_mask;
                            packed[j >> 1] = (j & 1) ? (packed[j >> 1] & 0xffffu) | (bits << 16) : (packed[j >> 1] & 0xffff0000u) | bits;
                        }
                }
            };
            auto stage_piece = [&](const uint32_t (&packed)[16], int piece) {
                const int chunk0 = (piece & 1) * 4;               // 16-byte chunks of the 128-byte staging row
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4)
                    *reinterpret_cast<uint4*>(stg + lane * 128 + (((chunk0 + q4) ^ (lane & 7)) << 4)) =
                        make_uint4(packed[4 * q4], packed[4 * q4 + 1], packed[4 * q4 + 2], packed[4 * q4 + 3]);
            };
            // Two register buffers: the tensor-memory load of piece i + 1 is in flight while piece i is turned into dz and staged.
            // The accumulator is handed back as soon as its last piece has been read.
            static_assert(EPI_PIECES % 2 == 0, "pieces go in pairs");
            const int p0 = col_half * EPI_PIECES;
            uint32_t ra[32], rb[32];
            tcgen05_ld_32x32_issue(tacc + p0 * 32, ra);
#pragma unroll 1
            for (int piece = p0; piece < p0 + EPI_PIECES; piece += 2) {
                uint32_t pa[16], pb[16];
                tcgen05_ld_wait(ra);
                tcgen05_ld_32x32_issue(tacc + (piece + 1) * 32, rb);
                to_dz(ra, piece, pa);
                tcgen05_ld_wait(rb);
                if (piece + 2 < p0 + EPI_PIECES) {
                    tcgen05_ld_32x32_issue(tacc + (piece + 2) * 32, ra);
                } else {
                    tcgen05_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(ps.lead_acc_empty + acc * (uint32_t)sizeof(uint64_t));
                }
                to_dz(rb, piece + 1, pb);
                const int col0 = first_col + piece * 32;
                __syncwarp();                                     // the staging tile has been read
                stage_piece(pa, piece);
                stage_piece(pb, piece + 1);
                __syncwarp();
                const int q = lane & 7;                           // eight lanes per row
                uint16_t* out = p.dz + (int64_t)(row0 + (lane >> 3)) * p.ldz + col0 + 8 * q;
                uint4 line[8];                                    // all of them read before the first store
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int row = 4 * i + (lane >> 3);
                    line[i] = *reinterpret_cast<const uint4*>(stg + row * 128 + ((q ^ (row & 7)) << 4));
                }
                if (col0 + 8 * q < p.ldz) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) *reinterpret_cast<uint4*>(out + 4 * i * p.ldz) = line[i];
                }
            }
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
            have = have_next;
            m = m_next;
            c = c_next;
        }
    }
    pipe_teardown(ps, p.d_status);
}

// ---- C[M,N] (+)= op(A) op(B): bf16 operands in either orientation, fp32 result ------------------------------------
//   A_MN = false: A stored [M, K] row-major;  A_MN = true: A stored [K, M] row-major (used as its transpose)
//   B_MN = false: B stored [N, K] row-major;  B_MN = true: B stored [K, N] row-major
// Tiles of 256 x 256, dealt to the pairs in groups of `group_n` column tiles: within a group consecutive pairs share the
// A panel and walk the B panels.  group_n keeps the B panels of a group (for dW a whole chunk of hidden rows) in L2 and the
// wave of 74 tiles near square, which is what it reads least bytes per K step with.
//   Whole waves of tiles are the body; the tiles left over (all of them where there are fewer than pairs) would keep part of the
// pairs busy for a whole wave, which is what a call of a few hundred tokens, with dH tiles of thousands of K steps on a handful
// of pairs, spent its time on.  So they are cut (GemmWork): for dH into ranges of K, the first of which writes dH and the others
// partial sums (in the rows of dZ that the chunk's tokens leave unused), added to dH in the order of the ranges by the epilogue
// warps of the dW kernel, which wait for their first tile at that time.  How they are cut depends on the sizes alone, so results are
// the same from run to run.
struct SumParams {            // dW kernel: the dH contraction whose partial sums it adds up
    const float* part;
    float* out;
    int M, N, K, group_n, slots;
    int64_t units;
};
struct GemmParams {
    int M, N, K;
    int group_n;
    int accumulate;           // 1: C += ..., 0: C = ...
    // rows of M (dH) or extent of K (dW) that count the chunk's tokens: only the live ones (T - t0) are contracted; dead rows
    // of C are written as zeros
    int m_is_tokens, k_is_tokens;
    int zero_if_dead;         // chunk without a live token: C = 0 instead of leaving it alone
    int a3d, b3d;             // the MN-major operand's maps are three-dimensional (one copy per stage)
    const int64_t* d_T;
    int64_t T_max, t0;
    unsigned int* lock_words;
    int lock_word;
    float* c;                 // [M, N], for direct stores
    float* part;              // partial sums of a tile, 256 x 256 each (dH): as many as fit the workspace
    int slots;
    SumParams sum;
    uint32_t* d_status;
};

struct GemmTile { int m, n; };
__device__ __forceinline__ bool gemm_item(int64_t i, int m_tiles, int n_tiles, int group_n, GemmTile& t) {
    const int64_t per_group = (int64_t)m_tiles * group_n;
    if (per_group == 0) return false;
    const int64_t g = i / per_group;
    const int first = (int)g * group_n;
    if (first >= n_tiles) return false;
    const int size = min(group_n, n_tiles - first);
    i -= g * per_group;
    t.m = (int)(i / size);
    if (t.m >= m_tiles) return false;
    t.n = first + (int)(i - (int64_t)t.m * size);
    return true;
}

// How the tiles of a launch are dealt.  Items [0, body) are whole tiles in the order of gemm_item; then the tail, by range of K and
// tile, the tile as the fast index, so that the pairs that work at the same time share operand panels.  (A column tile of half the
// width counts like the others: a K step takes the issuing warp about 500 cycles whatever the MMAs' width.)
constexpr int MIN_SEG = 16;              // K steps of a range at least: an epoch of the lock-step
// K steps that a wave of ranges costs beside its own (writing and adding 256 KB a pair).  Policy loss and backward with 0 / 12 / 40 (us): d = 320,
// V = 8,192, 2,500 tokens 71 / 68 / 68, 5,000 127 / 113 / 124; d = 1,024, 1,200 78 / 72 / 72, 2,500 124 / 112 / 123; d = 320, V = 30,000, 1,200
// 113 / 101 / 101, 4,700 320 / 320 / 324, and the one shape found where it is not the best, 2,400 180 / 185 / 181.
constexpr int SEG_COST = 12;
struct GemmWork {
    int m_tiles, n_tiles, group_n, k_steps;
    int body, tail, segs, items;         // tiles, tail tiles, ranges of K per tail tile
};
__device__ __forceinline__ GemmWork make_gemm_work(int m_tiles, int n_tiles, int group_n, int k_steps, int units, int slots) {
    GemmWork w;
    w.m_tiles = m_tiles; w.n_tiles = n_tiles; w.group_n = group_n; w.k_steps = k_steps;
    const int tiles = m_tiles * n_tiles, tail = tiles % units;
    w.segs = 1;
    int best = k_steps;
    if (tail > 0 && slots > 0)
#pragma unroll 1
        for (int waves = 1; waves <= 3; ++waves) {
            const int s = min(waves * units / tail, min(k_steps / MIN_SEG, slots / tail + 1));
            const int cost = waves * ((k_steps + s - 1) / max(s, 1) + SEG_COST);
            if (s > 1 && cost < best) { best = cost; w.segs = s; }
        }
    w.tail = w.segs > 1 ? tail : 0;      // nothing to gain: whole tiles to the end
    w.body = tiles - w.tail;
    w.items = w.body + w.tail * w.segs;
    return w;
}
__device__ __forceinline__ GemmTile gemm_tail_tile(const GemmWork& w, int idx) {
    GemmTile g;
    if (w.body > 0) gemm_item(w.body + idx, w.m_tiles, w.n_tiles, w.group_n, g);
    else { g.n = idx / w.m_tiles; g.m = idx - g.n * w.m_tiles; }
    return g;
}
// slot of range seg > 0 of tail tile idx
__device__ __forceinline__ int gemm_slot(const GemmWork& w, int idx, int seg) { return (seg - 1) * w.tail + idx; }
__device__ __forceinline__ bool gemm_work_item(const GemmWork& w, int N, int64_t item, TileAt& t) {
    if (item >= w.items) return false;
    GemmTile g;
    t.k0 = 0;
    t.k1 = w.k_steps;
    t.slot = -1;
    if (item < w.body) {
        gemm_item(item, w.m_tiles, w.n_tiles, w.group_n, g);
    } else {
        const int i = (int)item - w.body, seg = i / w.tail, idx = i - seg * w.tail;
        t.k0 = (int)((unsigned)seg * (unsigned)w.k_steps / (unsigned)w.segs);          // segs <= 3 units, k_steps < 2^20
        t.k1 = (int)((unsigned)(seg + 1) * (unsigned)w.k_steps / (unsigned)w.segs);
        if (seg > 0) t.slot = gemm_slot(w, idx, seg);
        g = gemm_tail_tile(w, idx);
    }
    t.a0 = g.m * TILE_ROWS;
    t.b0 = g.n * BN;
    t.n = N - t.b0 > BN / 2 ? BN : BN / 2;     // 64 columns per block at least: the granularity of an MN-major B tile's blocks
    return true;
}

// How results leave.  dH (written once, partial sums too): as 16-byte stores of whole lines, because a pair often has a single tile
// and its last store is what the kernel waits for.  dW: by TMA tile stores and reductions, beside the MMAs of the next tile; direct
// stores were no faster there (400 tokens, d = 512, V = 60,000 whole update 120 us, 124 with them; 12,000, d = 1,024, V = 30,000 1,662, 1,700).
template <bool A_MN, bool B_MN>
__global__ void __launch_bounds__(NUM_THREADS, 1)
gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
            const __grid_constant__ CUtensorMap map_b_tail, const __grid_constant__ CUtensorMap map_c,
            const GemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    const PipeSmem ps = pipe_setup(smem_raw, &map_a, &map_b);
    uint8_t* c_stage = ps.stage_a + EPI_STAGE_OFFSET;      // one 32 x 32 fp32 staging tile per epilogue warp
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t live = max((int64_t)0, live_tokens(p.d_T, p.T_max) - p.t0);
    const int n_tiles = (p.N + BN - 1) / BN;
    const int all_m_tiles = (p.M + TILE_ROWS - 1) / TILE_ROWS;
    const int K = p.k_is_tokens ? (int)min((int64_t)p.K, live) : p.K;
    const int k_steps = (K + BK - 1) / BK;
    const int k_last = (K - (k_steps - 1) * BK + UMMA_K - 1) / UMMA_K;
    // tiles that are contracted; the rest (rows of tokens that do not live) is written as zeros
    const int m_tiles = K == 0 ? 0 : p.m_is_tokens ? (int)min((int64_t)all_m_tiles, (live + TILE_ROWS - 1) / TILE_ROWS) : all_m_tiles;
    const int zero_m_tiles = live > 0 || p.zero_if_dead ? all_m_tiles - m_tiles : 0;
    const int64_t unit = blockIdx.x >> 1, units = gridDim.x >> 1;
    const GemmWork work = make_gemm_work(m_tiles, n_tiles, p.group_n, k_steps, (int)units, p.slots);
    auto coords = [&](int64_t it, TileAt& t) { return gemm_work_item(work, p.N, unit + it * units, t); };

    if (warp == 0) {
        const int tail_ks = (p.k_is_tokens && (K % BK) != 0) ? k_steps - 1 : -1;
        const Lockstep lock = lockstep_for(p.lock_words, p.lock_word, units, work.body, k_steps, work.items - work.body,
                                           (k_steps + work.segs - 1) / work.segs);
        producer_loop<A_MN, B_MN>(ps, &map_a, &map_b, lock, coords, p.a3d != 0, p.b3d != 0, &map_b_tail, tail_ks);
    } else if (warp == 1) {
        if (ps.rank == 0) mma_loop<A_MN, B_MN>(ps, k_steps, k_last, coords);
    } else {
        const int quarter = warp & 3;
        const int col_half = (warp - 2) >> 2;           // which half of the accumulator's columns
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        // The warp's 32 rows x 32 columns leave through shared memory (128-byte swizzle): as one TMA tile store, or as one TMA
        // reduction (global += tile) when the result is accumulated: whole 128-byte lines, no read of C by the SM, and rows / columns
        // past M / N are clipped by the copy; or as 16-byte stores of whole lines.
        constexpr bool DIRECT = !A_MN;
        uint8_t* stg = c_stage + (size_t)(warp - 2) * EPI_STAGE_TILE;
        auto store_tile = [&](const TileAt& t, bool zero, uint32_t tacc, auto release) {
            const bool partial = t.slot >= 0;
            const int row0 = (partial ? t.slot * TILE_ROWS : t.a0) + (int)ps.rank * BM + quarter * 32;
            const int pieces = t.n / 32 / (EPI_WARPS / 4);              // of this warp
#pragma unroll 1
            for (int i = 0; i < pieces; ++i) {
                const int piece = col_half * pieces + i;
                const bool inside = t.b0 + piece * 32 < p.N;
                const int pc0 = (partial ? 0 : t.b0) + piece * 32;
                float v[32];
                if (zero) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = 0.f;
                } else {
                    tcgen05_ld_32x32(tacc + piece * 32, v);
                    if (i + 1 == pieces) release();
                }
                if (!inside) continue;
                if (!DIRECT && lane == 0) bulk_wait_read_all();          // the previous tile copy has read the staging tile
                __syncwarp();
#pragma unroll
                for (int q4 = 0; q4 < 8; ++q4)
                    *reinterpret_cast<float4*>(stg + lane * 128 + ((q4 ^ (lane & 7)) << 4)) =
                        make_float4(v[4 * q4], v[4 * q4 + 1], v[4 * q4 + 2], v[4 * q4 + 3]);
                if constexpr (DIRECT) {
                    __syncwarp();
                    const int q = lane & 7;                              // eight lanes per row
                    const int64_t ld = partial ? BN : p.N;
                    float* out = (partial ? p.part : p.c) + (int64_t)(row0 + (lane >> 3)) * ld + pc0 + 4 * q;
                    float4 line[8];                                      // all of them read before the first store
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int row = 4 * k + (lane >> 3);
                        line[k] = *reinterpret_cast<const float4*>(stg + row * 128 + ((q ^ (row & 7)) << 4));
                    }
                    if (partial || pc0 + 4 * q < p.N) {                  // N is a multiple of 8
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (partial || row0 + 4 * k + (lane >> 3) < p.M) *reinterpret_cast<float4*>(out + 4 * k * ld) = line[k];
                    }
                } else {
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0 && row0 < p.M) {
                        if (p.accumulate) tma_reduce_add_2d(&map_c, pc0, row0, stg);
                        else tma_store_2d(&map_c, pc0, row0, stg);
                        bulk_commit_group();
                    }
                }
            }
        };
        if constexpr (A_MN) {       // dH += its partial sums, in the order of the ranges of K
            const SumParams& h = p.sum;
            const int h_tiles = (int)min((int64_t)((h.M + TILE_ROWS - 1) / TILE_ROWS), (live + TILE_ROWS - 1) / TILE_ROWS);
            const GemmWork hw = make_gemm_work(h_tiles, n_tiles, h.group_n, (h.K + BK - 1) / BK, (int)h.units, h.slots);
            if (hw.segs > 1) {
                constexpr int QUADS = TILE_ROWS * BN / 4;                // of a tile
                const float* part = pdl_acquire(h.part);
                const int stride = (int)gridDim.x * 32 * EPI_WARPS;
                for (int i = (int)blockIdx.x * 32 * EPI_WARPS + (int)threadIdx.x - 64; i < hw.tail * QUADS; i += stride) {
                    const int idx = i / QUADS, r = i / (BN / 4) % TILE_ROWS, q = i % (BN / 4);
                    const GemmTile g = gemm_tail_tile(hw, idx);
                    const int row = g.m * TILE_ROWS + r, col = g.n * BN + 4 * q;
                    if (row >= h.M || col >= h.N) continue;              // N is a multiple of 8
                    float4* out = reinterpret_cast<float4*>(h.out + (int64_t)row * h.N + col);
                    float4 v = __ldcg(out);
#pragma unroll 8
                    for (int seg = 1; seg < hw.segs; ++seg) {
                        const float4 x = __ldcg(reinterpret_cast<const float4*>(part + ((int64_t)gemm_slot(hw, idx, seg) * TILE_ROWS + r) * BN + 4 * q));
                        v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
                    }
                    *out = v;
                }
            }
        }
        uint32_t acc = 0, acc_phase = 0;
        bool ok = true;
        TileAt t;
        for (int64_t item = unit; ok && gemm_work_item(work, p.N, item, t); item += units) {
            ok = mbar_wait(&ps.acc_full[acc], acc_phase, ps.abort_flag);
            ok = __all_sync(0xffffffffu, ok) != 0;
            if (!ok) break;
            tcgen05_fence_after();
            store_tile(t, false, ps.tmem_base + lane_addr + acc * BN, [&]() {
                tcgen05_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(ps.lead_acc_empty + acc * (uint32_t)sizeof(uint64_t));
            });
            if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        GemmTile g;
        if (!p.accumulate)
            for (int64_t item = unit; gemm_item(item, zero_m_tiles, n_tiles, p.group_n, g); item += units)
                store_tile(TileAt{(m_tiles + g.m) * TILE_ROWS, g.n * BN, BN, 0, 0, -1}, true, 0u, []() {});
        if (lane == 0) bulk_wait_all();       // the tile copies have completed before the block's shared memory goes
    }
    pipe_teardown(ps, p.d_status);
}

int group_columns(int n_tiles) {          // column tiles per group: at most 10 (48 MB of B panels for K = 9,472), evenly
    const int groups = (n_tiles + 9) / 10;
    return (n_tiles + groups - 1) / groups;
}

// As many pairs as fit the GPU at once, whatever the work: in the dH kernel those without a tile of their own take part of another's, and in
// the dW kernel all of them add the partial sums.  Grids cut to the pairs with work do not leave more to a launch on another stream
// (two calls on one stream / two, us a call, all pairs and cut ones: T = 200, d = 256, V = 4,096 27.8 / 14.3, 29.8 / 15.2; 600, 512, 4,096 32.1 / 21.1,
// 33.9 / 20.4; 1,000, 256, 8,000 36.7 / 26.2, 36.4 / 25.8).
template <typename... KArgs, typename... Args>
cudaError_t launch_pairs(arrol_ctx* ctx, int which, void (*kernel)(KArgs...), cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(NUM_THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    // the pairs are persistent and kept in step: no more of them than the GPU holds at once (asked once per context and kernel)
    if (ctx->backward_max_pairs[which] == 0) {
        int fit = 0;
        cudaLaunchConfig_t ask = cfg;
        ask.gridDim = dim3((unsigned)(ctx->sm_count / 2 * 2));
        ask.numAttrs = 1;
        const cudaError_t e = cudaOccupancyMaxActiveClusters(&fit, kernel, &ask);
        if (e != cudaSuccess) return e;
        if (fit < 1) return cudaErrorInvalidConfiguration;
        ctx->backward_max_pairs[which] = fit;
    }
    cfg.gridDim = dim3((unsigned)(2 * ctx->backward_max_pairs[which]));
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

int raise_smem_limits(arrol_ctx* ctx) {
    if (ctx->backward_smem_set) return ARROL_OK;
    ARROL_CUDA_OK(cudaFuncSetAttribute(dz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES));
    ARROL_CUDA_OK(cudaFuncSetAttribute(gemm_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES));
    ARROL_CUDA_OK(cudaFuncSetAttribute(gemm_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES));
    ctx->backward_smem_set = true;
    return ARROL_OK;
}

constexpr int FREE_TILES = 16;         // tiles per pair that are not kept in step

// A kernel, not a memset: the dz kernel can be resident and set up while it waits for this one, and for the kernel before.
__global__ void clear_lock_kernel(unsigned int* words) {
    pdl_launch_dependents();
    pdl_wait();
    if (threadIdx.x < LOCK_WORDS) words[threadIdx.x] = 0u;
}

struct BackwardLayout {
    int64_t ldz;       // V rounded up to 8
    size_t dz, tail, lock, total;
};

BackwardLayout backward_layout(int d, int V) {
    BackwardLayout L;
    L.ldz = ((int64_t)V + 7) & ~(int64_t)7;
    L.dz = 0;
    L.tail = (((size_t)TC * L.ldz * 2) + 255) & ~(size_t)255;
    L.lock = L.tail + (size_t)(BK - 1) * d * 2;      // in the block's last row, which never holds a hidden row; d >= 8
    static_assert(LOCK_WORDS * sizeof(unsigned int) <= LOCK_BYTES && LOCK_BYTES <= 8 * 2, "the counters fit the narrowest row");
    L.total = L.tail + (((size_t)BK * d * 2 + 255) & ~(size_t)255);
    return L;
}

}  // namespace

extern "C" size_t arrol_lm_head_backward_workspace(arrol_ctx* ctx, int64_t T_max, int32_t d, int32_t V) {
    if (!ctx || T_max <= 0 || d <= 0 || V <= 0) return 0;
    return backward_layout(d, V).total;
}

extern "C" int arrol_lm_head_backward(arrol_ctx* ctx, const void* hidden, const void* W_vocab, const int32_t* targets,
                                      const float* grad_logp, const float* lse, int64_t T_max, const int64_t* d_T,
                                      int32_t d, int32_t V, float inv_temperature, float* dH, float* dW,
                                      void* workspace, size_t workspace_bytes, void* stream) {
    if (!ctx || T_max < 0 || d <= 0 || V <= 0 || !(inv_temperature > 0.f)) return ARROL_ERR_INVALID_ARG;
    if (!dW) return ARROL_ERR_INVALID_ARG;
    if (d % 8 != 0) return ARROL_ERR_UNSUPPORTED;
    if (T_max > (int64_t)INT32_MAX - TC) return ARROL_ERR_UNSUPPORTED;
    ArrolDeviceGuard guard(ctx->device);
    if (!guard.ok) return ARROL_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    if (T_max == 0) {
        ARROL_CUDA_OK(cudaMemsetAsync(dW, 0, sizeof(float) * (size_t)V * d, s));
        return ARROL_OK;
    }
    if (!hidden || !W_vocab || !targets || !grad_logp || !lse || !dH) return ARROL_ERR_INVALID_ARG;
    if (!arrol_aligned(hidden, 16) || !arrol_aligned(W_vocab, 16) || !arrol_aligned(dH, 16) || !arrol_aligned(dW, 16))
        return ARROL_ERR_INVALID_ARG;
    const BackwardLayout L = backward_layout(d, V);
    if (!workspace || workspace_bytes < L.total || !arrol_aligned(workspace, 256)) return ARROL_ERR_WORKSPACE;
    __nv_bfloat16* dZ = reinterpret_cast<__nv_bfloat16*>(static_cast<uint8_t*>(workspace) + L.dz);
    uint16_t* Htail = reinterpret_cast<uint16_t*>(static_cast<uint8_t*>(workspace) + L.tail);
    unsigned int* lock_words = reinterpret_cast<unsigned int*>(static_cast<uint8_t*>(workspace) + L.lock);
    // The dz kernel's counter has to be zero before the first chunk (the later ones are zeroed by the kernels).  Clearing it puts a
    // kernel's end and start, 3 us, before the dz kernel, and a memset 1.2 us more (backward, memset -> kernel: d = 512, V = 20,000, 2,048 tokens 121.8 ->
    // 120.5 us; 320, 40,000, 1,536 147.5 -> 146.6), so calls of which a pair has few tiles do without the step: they are over before pairs
    // drift apart.  Backward, in step / not: d = 512, V = 20,000, 2,048 tokens (8.5 tiles a pair) 120.9 / 118.4 us; 320, 40,000, 1,536 (12.7)
    // 146.8 / 144.0; 256, 60,000, 1,200 (15.9) 141.2 / 138.5; and past the line 512, 20,000, 5,000 (21) 266 / 264; 320, 151,936, 700 (24) 261.9 / 261.5;
    // 2,048, 60,000, 1,700 (22) 902 / 902; 4,096, 100,000, 1,000 (21) 1,801 / 1,803; 4,096, 10,000, 9,000 (19) 1,484 / 1,484.  At the line the
    // step is not yet worth its clearing; it stays well below the launches that drift.
    const bool first_in_step = (T_max + TILE_ROWS - 1) / TILE_ROWS * ((V + BN - 1) / BN) > (int64_t)FREE_TILES * (ctx->sm_count / 2);
    if (raise_smem_limits(ctx) != ARROL_OK) return ARROL_ERR_CUDA;

    // tensor maps: K-major operands are fetched as [128 MN rows x 64 K columns] boxes; MN-major ones (the same row-major
    // storage read the other way) as one three-dimensional box per stage when the MN extent is a whole number of
    // 64-element blocks, else as one [64 K rows x 64 MN columns] box per block
    CUtensorMap map_h_k, map_w_k, map_dz_k, map_w_mn, map_dz_mn, map_h_mn, map_h_tail;
    if (make_map(ctx, &map_h_k, hidden, (uint64_t)T_max, (uint64_t)d, BM) != ARROL_OK) return ARROL_ERR_CUDA;
    if (make_map(ctx, &map_w_k, W_vocab, (uint64_t)V, (uint64_t)d, BN / 2) != ARROL_OK) return ARROL_ERR_CUDA;
    if (make_map_ld(ctx, &map_dz_k, dZ, TC, (uint64_t)V, (uint64_t)L.ldz, BM) != ARROL_OK) return ARROL_ERR_CUDA;
    CUtensorMap map_dw;
    if (make_map_f32_tile(ctx, &map_dw, dW, (uint64_t)V, (uint64_t)d, (uint64_t)d) != ARROL_OK) return ARROL_ERR_CUDA;
    bool d3 = d % 64 == 0, v3 = V % 64 == 0;
    if (d3 && (make_map_mn3d(ctx, &map_w_mn, W_vocab, (uint64_t)V, (uint64_t)d, (uint64_t)d, BN / 2 / 64) != ARROL_OK ||
               make_map_mn3d(ctx, &map_h_tail, Htail, (uint64_t)BK - 1, (uint64_t)d, (uint64_t)d, BN / 2 / 64) != ARROL_OK))
        d3 = false;
    if (v3 && make_map_mn3d(ctx, &map_dz_mn, dZ, TC, (uint64_t)V, (uint64_t)L.ldz, BM / 64) != ARROL_OK) v3 = false;
    if (!d3) {
        if (make_map(ctx, &map_w_mn, W_vocab, (uint64_t)V, (uint64_t)d, BK) != ARROL_OK) return ARROL_ERR_CUDA;
        if (make_map(ctx, &map_h_tail, Htail, (uint64_t)BK - 1, (uint64_t)d, BK) != ARROL_OK) return ARROL_ERR_CUDA;
    }
    if (!v3 && make_map_ld(ctx, &map_dz_mn, dZ, TC, (uint64_t)V, (uint64_t)L.ldz, BK) != ARROL_OK) return ARROL_ERR_CUDA;

    if (first_in_step) {
        ARROL_CUDA_OK(arrol_launch_pdl(clear_lock_kernel, dim3(1), dim3(32), 0, s, lock_words));
        ctx->launches += 1;
    }
    const int n_tiles = (d + BN - 1) / BN;
    int m_groups = 1;
    while ((double)TC / m_groups * d * 2 > 50.0 * 1024 * 1024) ++m_groups;

    for (int64_t t0 = 0; t0 < T_max; t0 += TC) {
        const int64_t rows = (T_max - t0) < TC ? (T_max - t0) : (int64_t)TC;
        const int m_tiles = (int)((rows + TILE_ROWS - 1) / TILE_ROWS);
        // the chunk of hidden as an MN-major B operand: [rows (K), d (N)]; rows past T_max read as zero
        const void* h_chunk = static_cast<const uint8_t*>(hidden) + (size_t)t0 * d * 2;
        if ((d3 ? make_map_mn3d(ctx, &map_h_mn, h_chunk, (uint64_t)rows, (uint64_t)d, (uint64_t)d, BN / 2 / 64)
                : make_map(ctx, &map_h_mn, h_chunk, (uint64_t)rows, (uint64_t)d, BK)) != ARROL_OK)
            return ARROL_ERR_CUDA;

        DzParams zp;
        zp.targets = targets; zp.grad_logp = grad_logp; zp.lse = lse; zp.d_T = d_T; zp.T_max = T_max; zp.t0 = t0;
        zp.d = d; zp.V = V; zp.group_tiles = (TC / TILE_ROWS + m_groups - 1) / m_groups;
        zp.scale2 = inv_temperature * 1.44269504088896340736f; zp.inv_temp = inv_temperature;
        zp.lock_words = lock_words; zp.lock_on = t0 > 0 || first_in_step; zp.dz = reinterpret_cast<uint16_t*>(dZ); zp.ldz = L.ldz;
        zp.hidden = static_cast<const uint16_t*>(hidden); zp.tail = Htail; zp.d_status = ctx->d_status;
        ARROL_CUDA_OK(launch_pairs(ctx, 0, dz_kernel, s, map_h_k, map_w_k, zp));

        GemmParams gh = {};    // dH[chunk] = dZ . W
        gh.M = (int)rows; gh.N = d; gh.K = V; gh.group_n = group_columns(n_tiles);
        gh.m_is_tokens = 1; gh.b3d = d3; gh.lock_words = lock_words; gh.lock_word = LOCK_DH;
        gh.d_T = d_T; gh.T_max = T_max; gh.t0 = t0; gh.d_status = ctx->d_status;
        // partial sums of dH tiles lie in the rows of dZ that no tile of this chunk reaches
        constexpr size_t SLOT_BYTES = sizeof(float) * TILE_ROWS * BN;
        const size_t part_at = ((size_t)m_tiles * TILE_ROWS * L.ldz * 2 + 255) & ~(size_t)255;
        float* part = reinterpret_cast<float*>(static_cast<uint8_t*>(workspace) + L.dz + part_at);
        const size_t room = (L.tail - part_at) / SLOT_BYTES;
        gh.slots = room < 4096 ? (int)room : 4096;
        gh.part = part;
        gh.c = dH + t0 * d;
        ARROL_CUDA_OK(launch_pairs(ctx, 1, gemm_kernel<false, true>, s, map_dz_k, map_w_mn, map_w_mn, map_dw, gh));      // dH does not go through a map
        GemmParams gw = {};    // dW (+)= dZ^T . H[chunk]; the first chunk writes dW, zeros where no token lives
        gw.M = V; gw.N = d; gw.K = (int)rows; gw.group_n = group_columns(n_tiles);
        gw.accumulate = t0 > 0; gw.k_is_tokens = 1; gw.zero_if_dead = t0 == 0; gw.a3d = v3; gw.b3d = d3;
        gw.lock_words = lock_words; gw.lock_word = LOCK_DW;
        gw.d_T = d_T; gw.T_max = T_max; gw.t0 = t0; gw.d_status = ctx->d_status;
        gw.sum.part = part; gw.sum.out = dH + t0 * d; gw.sum.M = gh.M; gw.sum.N = gh.N; gw.sum.K = gh.K;
        gw.sum.group_n = gh.group_n; gw.sum.slots = gh.slots; gw.sum.units = ctx->backward_max_pairs[1];
        ARROL_CUDA_OK(launch_pairs(ctx, 2, gemm_kernel<true, true>, s, map_dz_mn, map_h_mn, map_h_tail, map_dw, gw));
        ctx->launches += 3;
    }
    return ARROL_OK;
}
