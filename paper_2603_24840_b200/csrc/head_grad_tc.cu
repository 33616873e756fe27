// Weight gradient of a bf16 MLP head's first layer on the tensor cores: dW1[h, d] = du^T X (Section 4.2), du given as the sum of
// two bf16 planes (error 2^-17 relative), X the scored hidden rows.
//
// One block per (128 hidden units x TN columns) tile and K range; K counts rollouts.  Per K step of 64 rollouts a stage receives
// both planes' 64 x 128 values and 64 rows x TN columns of X, all MN-major (the row-major storage read the other way).  Both planes multiply the same X tile into one accumulator.  Bound by the
// operand bytes per SM (40 KB per step against 256 cycles of MMAs at TN = 64), so the reduction is split over a cluster's
// blocks while SMs are idle (their accumulators meet in shared memory, added in rank order) and TN is 128 where tiles of 64
// would need more than one wave.  N = 2,048, d = 2,048, h = 256: 12.7 us (7 of them launch, set-up and finish) against 35.7 for a
// launch per plane on eight 128 x 256 tiles; N = 4,096, d = 4,096, h = 512: 33 us.
// The epilogue warps, which wait for the contraction, add up the row tiles' sums that dw2, db1, db2 and the loss are made of (32 hidden units
// a block: by one block's threads alone 125 tiles took longer than its share of the contraction); the forward
// kernel's last blocks did, behind a fence, a counter and a reload (N = 2,048, d = 2,048, h = 256: whole call 32.3 -> 29.2 us).
// Every wait is bounded; on expiry the block records ARROL_DEV_WAIT_EXPIRED, drains and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include "arrol_internal.h"
#include "tc_common.cuh"

namespace {

constexpr int GM = 128;                           // hidden units per tile (MMA M)
constexpr int PLANE_BYTES = GM * BK * 2;          // one plane's part of a stage: two blocks of [64 rollouts x 64 units]
constexpr int G_THREADS = 192;                    // producer, issuer, four epilogue warps
constexpr int MN_BLOCK = BK * 128;                // bytes of a [64 x 64] MN-major block
constexpr int G_TAIL_BYTES = 512 + 2048;           // barriers | quarters of the row tiles' sums

template <int TN> __host__ __device__ constexpr int stage_bytes() { return 2 * PLANE_BYTES + TN * BK * 2; }
template <int TN> __host__ __device__ constexpr int stages() { return TN == 64 ? 5 : 4; }
template <int TN> __host__ __device__ constexpr size_t smem_bytes() { return (size_t)stages<TN>() * stage_bytes<TN>() + 1024 + G_TAIL_BYTES; }

struct Dw1Params {
    int N, d, h;
    int k_steps;                                  // ceil(N / 64)
    float* dW1;
    HeadTileSums sums;
    uint32_t* d_status;
};

template <int TN>
__global__ void __launch_bounds__(G_THREADS, 1)
head_dw1_kernel(const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
                const __grid_constant__ CUtensorMap map_x, const Dw1Params p) {
    constexpr int STAGES = stages<TN>(), STAGE_BYTES = stage_bytes<TN>();
    constexpr int PITCH = TN + 4;                 // floats per row of the accumulator's copy in shared memory
    static_assert(GM * PITCH * 4 <= STAGES * STAGE_BYTES, "the copy fits the stages");
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)STAGES * STAGE_BYTES);
    uint64_t* empty = full + STAGES;
    uint64_t* acc_full = empty + STAGES;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
    volatile uint32_t* abort_flag = tmem_slot + 1;
    double* quarter_s = reinterpret_cast<double*>(smem + (size_t)STAGES * STAGE_BYTES + 512);     // [2][4][32]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c0 = blockIdx.x * TN, j0 = blockIdx.y * GM;
    const int splits = gridDim.z, rank = blockIdx.z;              // the cluster's blocks: ranges of the K steps
    const int ks0 = (int)((int64_t)rank * p.k_steps / splits), ks1 = (int)((int64_t)(rank + 1) * p.k_steps / splits);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(acc_full, 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_hi) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_lo) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&map_x) : "memory");
    }
    if (warp == 1) {
        tcgen05_alloc(tmem_slot, TN);
        tcgen05_relinquish();
    }
    tcgen05_fence_before();
    __syncthreads();
    tcgen05_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_launch_dependents();
    pdl_wait();

    if (warp == 0) {
        int issued = 0;
        bool ok = true;
        for (int ks = ks0; ks < ks1; ++ks, ++issued) {
            const int st = issued % STAGES;
            if (!mbar_wait_warp(&empty[st], ((uint32_t)(issued / STAGES) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
            uint8_t* a = smem + (size_t)st * STAGE_BYTES;
            uint8_t* x = a + 2 * PLANE_BYTES;
            if (lane == 0) mbar_expect_tx(&full[st], STAGE_BYTES);
            __syncwarp();
            if (lane < 4)       // plane, block of 64 units
                tma_load_2d(a + lane * MN_BLOCK, lane < 2 ? &map_hi : &map_lo, j0 + 64 * (lane & 1), ks * BK, &full[st]);
            if (lane >= 4 && lane < 4 + TN / 64)
                tma_load_2d(x + (lane - 4) * MN_BLOCK, &map_x, c0 + 64 * (lane - 4), ks * BK, &full[st]);
        }
        if (!ok) {              // let the copies in flight land before the block's shared memory goes away
            for (int i = issued - 1; i >= 0 && i >= issued - STAGES; --i)
                for (uint32_t it = 0; it < SPIN_LIMIT; ++it)
                    if (mbar_try_wait(&full[i % STAGES], (uint32_t)(i / STAGES) & 1u)) break;
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = make_idesc(GM, TN, true, true);
        constexpr uint64_t step = (UMMA_K * 128) >> 4;             // 16 rollouts of an MN-major block
        const uint32_t base = smem_u32(smem);
        bool ok = true;
        for (int i = 0; i < ks1 - ks0; ++i) {
            const int st = i % STAGES;
            if (!mbar_wait_warp(&full[st], (uint32_t)(i / STAGES) & 1u, abort_flag)) { ok = false; break; }
            tcgen05_fence_after();
            const uint64_t hi = make_smem_desc_mn(base + st * STAGE_BYTES, BK);
            const uint64_t lo = make_smem_desc_mn(base + st * STAGE_BYTES + PLANE_BYTES, BK);
            const uint64_t x = make_smem_desc_mn(base + st * STAGE_BYTES + 2 * PLANE_BYTES, BK);
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < BK / UMMA_K; ++k) {
                    tcgen05_mma_bf16(tmem_base, hi + step * k, x + step * k, idesc, (i | k) != 0 ? 1u : 0u);
                    tcgen05_mma_bf16(tmem_base, lo + step * k, x + step * k, idesc, 1u);
                }
                tcgen05_commit(&empty[st]);
            }
            __syncwarp();
        }
        // arrives when every MMA issued has finished: publishes the accumulator, or is what a block that gave up waits for
        if (elect_one()) tcgen05_commit(acc_full);
        __syncwarp();
        if (!ok)
            for (uint32_t it = 0; it < SPIN_LIMIT; ++it)
                if (mbar_try_wait(acc_full, 0u)) break;
    } else {
        // thread = one hidden unit: its TN sums go to shared memory (the stages are free: every MMA has finished)
        const int quarter = warp & 3, r = quarter * 32 + lane;
        if (p.sums.tile_sums) {          // the row tiles' sums, while the contraction runs: 32 hidden units a block, a quarter of the tiles a warp
            const int tiles = p.sums.tiles, w = warp - 2;
            const int block = (int)blockIdx.x * splits + rank, blocks = (int)gridDim.x * splits;
            const float* tile_sums = pdl_acquire(p.sums.tile_sums);
            for (int u0 = block * 32; u0 < GM && j0 + u0 < p.h; u0 += blocks * 32) {
                const int j = j0 + u0 + lane;
                double w2 = 0.0, b1 = 0.0;           // up to 1,024 tiles
                if (j < p.h)
#pragma unroll 8
                    for (int t = w; t < tiles; t += 4) {
                        w2 += (double)tile_sums[(int64_t)t * p.h + j];
                        b1 += (double)tile_sums[(int64_t)(tiles + t) * p.h + j];
                    }
                quarter_s[w * 32 + lane] = w2;
                quarter_s[128 + w * 32 + lane] = b1;
                named_barrier_sync<1, 128>();
                if (w < 2 && j < p.h) {
                    const double* q = quarter_s + 128 * w + lane;
                    (w == 0 ? p.sums.dw2 : p.sums.db1)[j] = (float)(((q[0] + q[32]) + q[64]) + q[96]);
                }
                named_barrier_sync<1, 128>();
            }
            if (j0 == 0 && block == blocks - 1 && w >= 2) {
                const double* tile_loss = pdl_acquire(p.sums.tile_loss) + (w - 2) * tiles;
                double t = 0.0;
#pragma unroll 4
                for (int i = lane; i < tiles; i += 32) t += tile_loss[i];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                if (lane == 0) {
                    if (w == 2) *p.sums.loss = t;
                    else *p.sums.db2 = (float)t;
                }
            }
        }
        bool ok = mbar_wait(acc_full, 0u, abort_flag);
        ok = __all_sync(0xffffffffu, ok && !*abort_flag) != 0;
        float* row = reinterpret_cast<float*>(smem) + r * PITCH;
        if (ok) {
            tcgen05_fence_after();
#pragma unroll 1
            for (int piece = 0; piece < TN / 32; ++piece) {
                float v[32];
                tcgen05_ld_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + piece * 32, v);
#pragma unroll
                for (int j = 0; j < 32; j += 4)
                    *reinterpret_cast<float4*>(row + piece * 32 + j) =
                        ks0 < ks1 ? make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
    }
    tcgen05_fence_before();
    __syncthreads();
    cluster_sync_all();
    // every block of the cluster finishes its share of the tile's rows
    const int rows_each = GM / splits;
#pragma unroll 4
    for (int i = threadIdx.x; i < rows_each * (TN / 4); i += G_THREADS) {
        const int r = rank * rows_each + i / (TN / 4), c = i % (TN / 4) * 4;
        const uint32_t at = smem_u32(reinterpret_cast<float*>(smem) + r * PITCH + c);
        float4 sum = ld_shared_cluster_v4(map_to_cta(at, 0u));
        for (int z = 1; z < splits; ++z) {
            const float4 v = ld_shared_cluster_v4(map_to_cta(at, (uint32_t)z));
            sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
        }
        if (j0 + r < p.h && c0 + c < p.d) *reinterpret_cast<float4*>(p.dW1 + (int64_t)(j0 + r) * p.d + c0 + c) = sum;   // d % 8 == 0
    }
    cluster_sync_all();                 // nobody's shared memory goes away while it is being read
    if (threadIdx.x == 0 && *abort_flag) atomicOr(p.d_status, ARROL_DEV_WAIT_EXPIRED);
    if (warp == 1) {
        tcgen05_fence_after();
        tcgen05_dealloc(tmem_base, TN);
    }
}

template <int TN>
int launch_dw1(arrol_ctx* ctx, const CUtensorMap& hi, const CUtensorMap& lo, const CUtensorMap& x, const Dw1Params& p,
               cudaStream_t s) {
    if (!ctx->head_dw1_smem_set[TN == 128]) {
        ARROL_CUDA_OK(cudaFuncSetAttribute(head_dw1_kernel<TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<TN>()));
        ctx->head_dw1_smem_set[TN == 128] = true;
    }
    const int tiles = ((p.d + TN - 1) / TN) * ((p.h + GM - 1) / GM);
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(G_THREADS);
    cfg.dynamicSmemBytes = smem_bytes<TN>();
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    auto shape = [&](int splits) {
        cfg.gridDim = dim3((p.d + TN - 1) / TN, (p.h + GM - 1) / GM, splits);
        attr[0].val.clusterDim.z = splits;
    };
    // Blocks per cluster: at least four K steps each, and no more blocks than SMs; eight only where so many clusters fit at once
    // (asked once per context).  N = 5,000, d = 520, h = 72 (nine tiles) with four / eight: 28.5 / 24.5 us; where they do not fit, N = 8,000,
    // d = 1,024, h = 64 (16 tiles) 30.3 / 35.8.
    int splits = 1;
    while (splits < 4 && tiles * splits * 2 <= ctx->sm_count && p.k_steps >= splits * 2 * 4) splits *= 2;
    if (splits == 4 && tiles * 8 <= ctx->sm_count && p.k_steps >= 32) {
        int& fit = ctx->head_dw1_max_clusters[TN == 128];
        if (fit == 0) {
            shape(8);
            cfg.numAttrs = 1;
            ARROL_CUDA_OK(cudaOccupancyMaxActiveClusters(&fit, head_dw1_kernel<TN>, &cfg));
        }
        if (tiles <= fit) splits = 8;
    }
    shape(splits);
    cfg.numAttrs = 2;
    ARROL_CUDA_OK(cudaLaunchKernelEx(&cfg, head_dw1_kernel<TN>, hi, lo, x, p));
    ctx->launches += 1;
    return ARROL_OK;
}

}  // namespace

int arrol_internal_head_dw1(arrol_ctx* ctx, const void* du_hi, const void* du_lo, const void* X, int64_t ldx, int N, int d,
                            int h, float* dW1, const HeadTileSums& sums, cudaStream_t s) {
    CUtensorMap map_hi, map_lo, map_x;
    if (make_map(ctx, &map_hi, du_hi, (uint64_t)N, (uint64_t)h, BK) != ARROL_OK) return ARROL_ERR_CUDA;
    if (make_map(ctx, &map_lo, du_lo, (uint64_t)N, (uint64_t)h, BK) != ARROL_OK) return ARROL_ERR_CUDA;
    if (make_map_ld(ctx, &map_x, X, (uint64_t)N, (uint64_t)d, (uint64_t)ldx, BK) != ARROL_OK) return ARROL_ERR_CUDA;
    Dw1Params p;
    p.N = N; p.d = d; p.h = h;
    p.k_steps = (N + BK - 1) / BK;
    p.dW1 = dW1;
    p.sums = sums;
    p.d_status = ctx->d_status;
    const int tiles64 = ((d + 63) / 64) * ((h + GM - 1) / GM);
    return tiles64 > ctx->sm_count ? launch_dw1<128>(ctx, map_hi, map_lo, map_x, p, s)
                                   : launch_dw1<64>(ctx, map_hi, map_lo, map_x, p, s);
}
