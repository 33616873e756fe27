// arrol_prune_step: score -> select -> compact from one call, for callers that want the prune-and-rebatch part of the
// step (Algorithm 1: quality check at the detection length, filter, re-batch) without host work between the launches.
//
// The chain is a handful of microsecond kernels, each a few dependent round trips to memory, so what it costs is
// launches and latency, not work.  Fast path: ONE grid runs scoring, selection, the survivor scan and the advantages,
// and a second launch writes the per-token outputs.
//   prune_fused_kernel   a block owns 32 / G whole groups (at most 32 rollouts, one warp each).  Linear head: every
//                        warp scores its rollout (the row reduction and probability map of score_linear_kernel) and
//                        leaves q in shared memory; MLP head: q comes from the scoring kernel that ran before (blocks
//                        of two warps then, always 32 / G groups each).  One or
//                        two warps run the per-group selection (select_lanes, as select_kernel) and write the keep
//                        flags.  The first warp then scans the block's rollouts (kept, kept length), adds the block's
//                        tokens to the sums of the blocks after it, waits until those before have added theirs to its
//                        own (a chained scan: every block only waits for lower-numbered blocks, of at most two per SM;
//                        how many rollouts they keep is known), and writes survivor_idx, cu_seqlens and the advantages
//                        of its own groups (group_statistics, as scan_adv_kernel); the last block writes {S, T}.
//                        Nothing is re-read from global memory and no block waits for the whole grid.  The second warp counts
//                        the blocks that are done with the chain; the last one clears it for the next call.
// The device functions are the ones the three separate kernels use, so the results are bit-identical to the three
// public calls, which remain the general path (more than SM-count blocks of 32 / G groups; group sizes above 32 are
// rejected by arrol_select either way).
#include <cuda_bf16.h>

#include "arrol_internal.h"
#include "prune_kernels.cuh"
#include "token_runs.cuh"

namespace {

struct FusedParams {
    // scoring (linear head) / its outputs
    const void* hidden;
    int64_t row_stride;
    const int64_t* row_index;
    const void* w;
    const void* bias;
    const float* q_lut;
    float *score, *prob, *q;
    int32_t* bin;
    int N, d, B;
    // selection
    int P, G, K, seg, gpb;     // gpb: groups per block
    double rho;
    uint8_t* keep;
    // scan + advantages
    const int32_t* lengths;
    const float* rewards;
    const int64_t* src_tok_off;
    double eps;
    int ddof;
    int64_t capacity, source_rows;
    int32_t* survivor_idx;
    int64_t* cu_seqlens;
    float* adv;
    int64_t* d_num;
    uint32_t* d_status;
    // chained scan: word [0] blocks that are done with it, from LEFT_ONE on those of which a kept rollout left the source (index
    // check), from EXPIRED_ONE on those that waited in vain; then from [2] a word per block, SUM_WORDS apart: the kept tokens of the blocks before
    // it, from ARRIVED_ONE on how many of these have added theirs; all zero between calls
    unsigned long long* chain;
    SurvivorRun* runs;         // or NULL: no per-token outputs
    uint32_t spin_limit;
    int rest_vecs;             // 16-byte vectors of a row past the first 256 that a warp has room for in shared memory: all of them, or 0
};

constexpr int LUT_STAGED = 1024;
constexpr int SUM_WORDS = ARROL_CHAIN_WORDS;       // a sector of its own for every block
constexpr unsigned long long ARRIVED_ONE = 1ull << 54, LEFT_ONE = 1ull << 32, EXPIRED_ONE = 1ull << 48;     // at most ARROL_CHAIN_BLOCKS of either

__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_add_u64(unsigned long long* p, unsigned long long v) {
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long count_acq_rel(unsigned long long* p, unsigned long long n) {
    unsigned long long before;
    asm volatile("atom.acq_rel.gpu.global.add.u64 %0, [%1], %2;" : "=l"(before) : "l"(p), "l"(n) : "memory");
    return before;
}

// SCORE: the block scores its rollouts itself (linear head, element type T); otherwise q was written by an earlier
// kernel on the stream.
template <typename T, bool SCORE>
__global__ void __launch_bounds__(SCAN_THREADS)
prune_fused_kernel(const FusedParams p) {
    __shared__ float q_s[32], rew_s[32];
    __shared__ uint8_t keep_s[32];
    __shared__ int32_t len_s[32];
    __shared__ int64_t src_s[32];
    __shared__ bool block_left, block_expired;               // a kept rollout of this block leaves the source; a wait ran out
    __shared__ double inv_count[SCAN_INV], g_mean[32], g_den[32];
    __shared__ float lut_s[LUT_STAGED];                      // the posterior table, or its first use would be one more round trip
    extern __shared__ uint4 w_stage[];                       // linear head: the weights, d * sizeof(T) bytes
    pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int group0 = blockIdx.x * p.gpb;
    const int groups_here = min(p.gpb, p.P - group0);
    const int first = group0 * p.G;
    const int n_here = groups_here * p.G;                   // rollouts of this block, one warp each
    if (threadIdx.x >= 1 && threadIdx.x < SCAN_INV) inv_count[threadIdx.x] = 1.0 / (double)threadIdx.x;
    pdl_wait();
    bool bad_index = false;
    if (warp == 1 && lane < n_here) {                        // the block's lengths and rewards, while the others score
        const int i = first + lane;
        len_s[lane] = max(pdl_acquire(p.lengths)[i], 0);
        rew_s[lane] = pdl_acquire(p.rewards)[i];
        if (p.runs || p.source_rows > 0) src_s[lane] = pdl_acquire(p.src_tok_off)[i];
    }
    if constexpr (SCORE) {
        // every warp fetches its row number while the block stages the head's weights
        constexpr int VN = Vec16<T>::N;
        typedef typename Vec16<T>::Raw Raw;
        Raw* w_s = reinterpret_cast<Raw*>(w_stage);
        const int i = first + warp;
        int64_t row = 0;
        if (warp < n_here) {
            const int64_t* row_index = pdl_acquire(p.row_index);
            row = row_index ? row_index[i] : (int64_t)i;
        }
        const T* w = pdl_acquire(static_cast<const T*>(p.w));
        const float* q_lut = pdl_acquire(p.q_lut);
        const bool lut_staged = q_lut && p.B <= LUT_STAGED;
        for (int c = threadIdx.x; c < p.d / VN; c += blockDim.x) w_s[c] = Vec16<T>::load_raw(w + (int64_t)c * VN);
        if (lut_staged)
            for (int c = threadIdx.x; c < p.B; c += blockDim.x) lut_s[c] = q_lut[c];
        const T* x = pdl_acquire(static_cast<const T*>(p.hidden)) + row * p.row_stride;
        const T* bias_ptr = pdl_acquire(static_cast<const T*>(p.bias));
        const float bias = bias_ptr ? to_f32(bias_ptr[0]) : 0.f;
        int nvec = warp < n_here ? p.d / VN : 0;
        if (nvec && p.source_rows > 0 && (row < 0 || row >= p.source_rows)) {   // never read, scored as zeros
            if (lane == 0) atomicOr(p.d_status, ARROL_DEV_BAD_INDEX);
            nvec = 0;
        }
        // the whole row is on its way while the block waits for the weights: 4 KB in registers, what is past them by asynchronous
        // copies (a second round trip to HBM after the first one otherwise)
        Raw xr[8];
        Raw* rest_s = p.rest_vecs > 0 ? w_s + p.d / VN + warp * p.rest_vecs : nullptr;
        linear_row_begin<T>(x, nvec, lane, xr);
        if (rest_s) linear_row_rest<T>(x, nvec, lane, rest_s);
        __syncthreads();
        if (warp < n_here) {
            float s = linear_row_dot_ws<T>(x, xr, w_s, nvec, lane, rest_s);
            if (lane == 0) {
                if (bias_ptr) s += bias;
                q_s[warp] = probability_map(s, i, p.B, lut_staged ? lut_s : q_lut, p.score, p.prob, p.bin, p.q);
            }
        }
    } else {
        if (threadIdx.x < n_here) q_s[threadIdx.x] = pdl_acquire(p.q)[first + threadIdx.x];
    }
    __syncthreads();
    // selection on the block's groups: a group per segment of `seg` lanes
    const int groups_per_warp = 32 / p.seg;
    if (warp * groups_per_warp < groups_here) {
        const int gl = warp * groups_per_warp + lane / p.seg;
        const int j = lane & (p.seg - 1);
        const bool member = gl < groups_here && j < p.G;
        const double qj = member ? (double)q_s[gl * p.G + j] : 0.0;
        const bool alive = select_lanes(qj, member, j, p.G, p.K, p.rho, p.seg);
        if (member) {
            keep_s[gl * p.G + j] = alive ? 1 : 0;
            p.keep[first + gl * p.G + j] = alive ? 1 : 0;
        }
    }
    __syncthreads();
    unsigned long long* sums = p.chain + 2;
    if (warp == 1) {
        // statistics of the block's groups, one lane per group, while the first warp scans
        if (lane < groups_here) {
            auto flag = [&](int r) { return keep_s[r] != 0; };
            auto rew = [&](int r) { return rew_s[r]; };
            double mean, den;
            group_statistics(lane * p.G, lane * p.G + p.G, p.ddof, p.eps, inv_count, flag, rew, mean, den);
            g_mean[lane] = mean;
            g_den[lane] = den;
        }
        __threadfence_block();
        named_barrier_arrive<1, 64>();
        // The block is done with the chain when the first warp has added its total to the sums of the blocks after it and read its
        // own.  The count's release is what the clearing rests on: every block's stores have been performed before the last one to be
        // counted zeroes the words.  Without it what a block adds to the sum of one that has given up waiting could land after the
        // zeros and be counted by a later call.  The release waits for
        // those stores, so it is this warp's, beside the outputs that the first one writes.  Graphs of 20 calls, this / with a fence and
        // the count in the first warp / with nothing between stores and count: 2,048 rollouts at d = 2,560 19.5 / 20.3 / 20.1 us, 4,096
        // after an MLP head 70.4 / 70.6 / 70.0, 32 rollouts 9.4 / 10.3 / 9.9.
        named_barrier_sync<2, 64>();
        unsigned long long done = 0;
        if (lane == 0) done = count_acq_rel(p.chain, 1ull + (block_left ? LEFT_ONE : 0ull) + (block_expired ? EXPIRED_ONE : 0ull));
        done = __shfl_sync(0xffffffffu, done, 0);
        if ((done & (LEFT_ONE - 1)) == gridDim.x - 1) {
            for (unsigned int b = lane; b < gridDim.x; b += 32) sums[b * SUM_WORDS] = 0ull;
            if (lane == 0) {
                const bool left = block_left || done % EXPIRED_ONE >= LEFT_ONE, expired = block_expired || done >= EXPIRED_ONE;
                if (left) atomicOr(p.d_status, ARROL_DEV_BAD_INDEX);
                if (expired) {                       // the survivors' list has holes: nobody is to follow it
                    atomicOr(p.d_status, ARROL_DEV_WAIT_EXPIRED);
                    p.d_num[0] = 0;
                    p.d_num[1] = 0;
                }
                p.d_status[1] = left || expired ? 1u : 0u;      // gate word: the gather kernels of this call copy nothing when set
                p.chain[0] = 0ull;
            }
        }
    }
    if (warp != 0) return;

    // ---- first warp: scan of the block's rollouts, chained over the blocks, outputs of the block's groups ----
    const bool kept = lane < n_here && keep_s[lane] != 0;
    const int64_t own_t = kept ? (int64_t)len_s[lane] : 0;
    if (kept && p.source_rows > 0) {
        const int64_t o = src_s[lane];
        bad_index = o < 0 || o + own_t > p.source_rows;
    }
    const unsigned int kept_lanes = __ballot_sync(0xffffffffu, kept);
    int64_t t = own_t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t ot = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += ot;
    }
    const int64_t block_t = __shfl_sync(0xffffffffu, t, 31);
    const int32_t block_c = __popc(kept_lanes);
    // The block adds its total to the sums of all blocks after it, and waits for its own sum to be complete: every block polls a word
    // of its own.  When each read all totals before it, 128 blocks polled the same lines, and the last total took 3.8 us to get
    // through to them (relaxed loads, eight at a time, 5 us: the more polls the later).  The additions grow with the square of the blocks;
    // at two blocks an SM, 43,660 of them: 592 prompts of 16 rollouts of 60 tokens at d = 512 26.2 -> 20.1 us, of 600 39.1 -> 32.0.
    for (unsigned int b = blockIdx.x + 1 + lane; b < gridDim.x; b += 32) red_add_u64(sums + (size_t)b * SUM_WORDS, ARRIVED_ONE + (unsigned long long)block_t);
    unsigned long long sum = 0;
    bool expired = false;
    if (lane == 0 && blockIdx.x > 0)
        for (uint32_t it = 0;;) {
            sum = ld_relaxed_u64(sums + (size_t)blockIdx.x * SUM_WORDS);
            if (sum / ARRIVED_ONE == blockIdx.x) break;
            if (++it >= p.spin_limit) { expired = true; break; }
        }
    const int64_t base_t = (int64_t)(__shfl_sync(0xffffffffu, sum, 0) % ARRIVED_ONE);
    const int32_t base_c = group0 * p.K;                     // every group before these keeps exactly K
    const bool any_bad = __any_sync(0xffffffffu, bad_index);
    const bool any_expired = __any_sync(0xffffffffu, expired);
    if (lane == 0) {
        block_left = any_bad;
        block_expired = any_expired;
        if (blockIdx.x == gridDim.x - 1) {                   // before the block is counted: the last one may take it back
            p.d_num[0] = base_c + block_c;
            p.d_num[1] = base_t + block_t;
            if (base_t + block_t > p.capacity) atomicOr(p.d_status, ARROL_DEV_CAPACITY);
        }
    }
    named_barrier_arrive<2, 64>();                           // done with the chain
    named_barrier_sync<1, 64>();                             // the groups' statistics
    if (kept) {
        const int pos = base_c + __popc(kept_lanes & ((1u << lane) - 1u));
        p.survivor_idx[pos] = first + lane;
        p.cu_seqlens[pos + 1] = base_t + t;
        const int g = lane / p.G;
        const float adv = (float)(((double)rew_s[lane] - g_mean[g]) * g_den[g]);      // den holds 1 / (std + eps), or 0
        p.adv[pos] = adv;
        if (p.runs) {
            const int64_t c0 = base_t + t - own_t, src0 = src_s[lane];
            int4* run = reinterpret_cast<int4*>(p.runs + pos);
            run[0] = make_int4((int)c0, (int)(c0 >> 32), (int)src0, (int)(src0 >> 32));
            run[1] = make_int4(len_s[lane], __float_as_int(adv), 0, 0);
        }
    }
    if (blockIdx.x == 0 && lane == 0) p.cu_seqlens[0] = 0;
}

}  // namespace

extern "C" int arrol_prune_step(arrol_ctx* ctx, const arrol_prune_step_args* a, void* stream) {
    if (!ctx || !a) return ARROL_ERR_INVALID_ARG;
    if (a->P < 0 || a->G < 1) return ARROL_ERR_INVALID_ARG;
    const int64_t N64 = (int64_t)a->P * a->G;
    if (N64 > INT32_MAX) return ARROL_ERR_UNSUPPORTED;
    const int32_t N = (int32_t)N64;

    // Everything is validated before the first launch, so that a bad argument of a later stage leaves nothing half done.
    if (N > 0) {
        int rc = arrol_internal_check_score(a->hidden, a->row_stride_elems, N, &a->head, &a->calib, a->score, a->prob, a->q);
        if (rc != ARROL_OK) return rc;
    }
    int rc = arrol_internal_check_select(a->q, a->P, a->G, a->K, a->rho, 0, a->keep);
    if (rc != ARROL_OK) return rc;
    rc = arrol_internal_check_compact(a->keep, a->lengths, a->src_tok_off, N, a->G, a->src_tokens, a->src_rows,
                                      a->row_bytes, a->rewards, a->eps, a->ddof, a->dst_capacity_tokens, a->dst_tokens,
                                      a->dst_rows, a->cu_seqlens, a->survivor_idx, a->adv, a->d_num);
    if (rc != ARROL_OK) return rc;
    if (N == 0)       // nothing to score or select; the scan still writes {0, 0}
        return arrol_compact(ctx, a->keep, a->lengths, a->src_tok_off, N, a->G, a->src_tokens, a->src_rows, a->row_bytes,
                             a->rewards, a->eps, a->ddof, a->dst_capacity_tokens, a->dst_tokens, a->dst_rows, a->cu_seqlens,
                             a->survivor_idx, a->adv, a->tok_adv, a->tok_seq, a->d_num, stream);

    const bool linear = a->head.h == 0;
    // groups per block: as many as 32 warps hold, fewer while that leaves most SMs without a block
    int gpb = 32 / a->G;
    while (gpb > 1 && (a->P + gpb - 1) / gpb < ctx->sm_count / 2) gpb = (gpb + 1) / 2;
    int threads = 32 * gpb * a->G;
    if (threads < 64) threads = 64;                          // warp 1 fetches the lengths and rewards
    if (!linear) {                                           // nothing to score: two warps per block, full blocks
        gpb = 32 / a->G;
        threads = 64;
    }
    const int64_t fused_blocks = ((int64_t)a->P + gpb - 1) / gpb;
    const size_t w_bytes = linear ? (size_t)a->head.d * (a->head.dtype == ARROL_F32 ? 4 : 2) : 0;
    // what is past the first 4 KB of a block's rows is staged too while the blocks of an SM have room for it side by side
    const size_t first_bytes = (size_t)ROW_BEGIN_VECS * 16;
    size_t rest_bytes = w_bytes > first_bytes ? (w_bytes - first_bytes) * (size_t)(threads / 32) : 0;
    if (rest_bytes + w_bytes > (fused_blocks > ctx->sm_count ? (size_t)96 : (size_t)200) * 1024) rest_bytes = 0;
    const size_t smem = w_bytes + rest_bytes;
    // blocks of the chained scan, which wait for lower-numbered ones: at most two per SM
    const int per_sm = 2048 / threads < 1 ? 1 : 2048 / threads;
    if (fused_blocks > (int64_t)ctx->sm_count * (per_sm > 2 ? 2 : per_sm) || fused_blocks > ARROL_CHAIN_BLOCKS ||
        w_bytes > 40 * 1024) {
        // more than the chained scan is made for, or a head too wide to stage: the three calls, back to back
        rc = arrol_score_partial(ctx, a->hidden, a->row_stride_elems, a->row_index, N, &a->head, &a->calib, a->score,
                                 a->prob, a->bin, a->q, stream);
        if (rc != ARROL_OK) return rc;
        rc = arrol_select(ctx, a->q, a->P, a->G, a->K, a->rho, 0, a->keep, stream);
        if (rc != ARROL_OK) return rc;
        return arrol_compact(ctx, a->keep, a->lengths, a->src_tok_off, N, a->G, a->src_tokens, a->src_rows, a->row_bytes,
                             a->rewards, a->eps, a->ddof, a->dst_capacity_tokens, a->dst_tokens, a->dst_rows, a->cu_seqlens,
                             a->survivor_idx, a->adv, a->tok_adv, a->tok_seq, a->d_num, stream);
    }
    if (!linear) {    // MLP head: its own kernels score; the fused kernel starts at the selection
        rc = arrol_score_partial(ctx, a->hidden, a->row_stride_elems, a->row_index, N, &a->head, &a->calib, a->score,
                                 a->prob, a->bin, a->q, stream);
        if (rc != ARROL_OK) return rc;
    }
    ArrolDeviceGuard guard(ctx->device);
    if (!guard.ok) return ARROL_ERR_CUDA;
    FusedParams p;
    p.hidden = a->hidden;
    p.row_stride = a->row_stride_elems;
    p.row_index = a->row_index;
    p.w = a->head.W1;
    p.bias = a->head.b1;
    p.q_lut = a->calib.q_lut;
    p.B = a->calib.B > 0 ? a->calib.B : 0;
    p.score = a->score; p.prob = a->prob; p.q = a->q; p.bin = a->bin;
    p.N = N; p.d = a->head.d;
    p.P = a->P; p.G = a->G; p.K = a->K; p.rho = a->rho;
    p.seg = 1;
    while (p.seg < a->G) p.seg <<= 1;
    p.gpb = gpb;
    p.keep = a->keep;
    p.lengths = a->lengths; p.rewards = a->rewards; p.src_tok_off = a->src_tok_off;
    p.eps = (double)a->eps; p.ddof = a->ddof;
    p.capacity = a->dst_capacity_tokens; p.source_rows = ctx->source_rows;
    p.survivor_idx = a->survivor_idx; p.cu_seqlens = a->cu_seqlens; p.adv = a->adv; p.d_num = a->d_num;
    p.d_status = ctx->d_status;
    p.chain = ctx->d_chain;
    p.runs = a->dst_tokens || a->tok_adv || a->tok_seq ? static_cast<SurvivorRun*>(ctx->d_runs) : nullptr;
    p.spin_limit = ctx->test_spin_limit ? ctx->test_spin_limit : (1u << 22);
    p.rest_vecs = (int)(rest_bytes / 16 / (size_t)(threads / 32));
    if (smem > 40 * 1024 && !ctx->prune_smem_set) {
        ARROL_CUDA_OK(cudaFuncSetAttribute(prune_fused_kernel<float, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        ARROL_CUDA_OK(cudaFuncSetAttribute(prune_fused_kernel<__nv_bfloat16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        ctx->prune_smem_set = true;
    }
    const dim3 grid((unsigned)fused_blocks), block((unsigned)threads);
    cudaStream_t s = (cudaStream_t)stream;
    if (!linear)
        ARROL_CUDA_OK(arrol_launch_pdl(prune_fused_kernel<float, false>, grid, block, 0, s, p));
    else if (a->head.dtype == ARROL_F32)
        ARROL_CUDA_OK(arrol_launch_pdl(prune_fused_kernel<float, true>, grid, block, smem, s, p));
    else
        ARROL_CUDA_OK(arrol_launch_pdl(prune_fused_kernel<__nv_bfloat16, true>, grid, block, smem, s, p));
    ctx->launches += 1;
    return arrol_internal_compact(ctx, a->keep, a->lengths, a->src_tok_off, N, a->G, a->src_tokens, a->src_rows,
                                  a->row_bytes, a->rewards, a->eps, a->ddof, a->dst_capacity_tokens, a->dst_tokens,
                                  a->dst_rows, a->cu_seqlens, a->survivor_idx, a->adv, a->tok_adv, a->tok_seq, a->d_num,
                                  stream, true, p.runs, a->P * a->K);
}
