// arrol_head_grad: one training step's gradients for the quality head (Section 4.2: trained on the fly with a
// cross-entropy loss on (score, final reward); Section 4.3 (iii): gradients stop at the head).
//   loss = (1/n) sum_i [log(1 + exp(s_i)) - y_i s_i],  ds_i = (sigmoid(s_i) - y_i) / n  over the masked-in rollouts;
//   linear head:  dw = sum_i ds_i x_i, db = sum_i ds_i
//   MLP head:     dw2_j = sum_i ds_i gelu(u_ij), db2 = sum_i ds_i, du_ij = ds_i w2_j gelu'(u_ij),
//                 dW1 = du^T X, db1_j = sum_i du_ij.
// All reductions run in a fixed order (the only atomics count arrivals), so the gradients are reproducible run to run.
#include <cuda_bf16.h>

#include "arrol_internal.h"
#include "score_common.cuh"
#include "tc_common.cuh"

namespace {

constexpr int DU_RUNS = 32;          // runs of rollouts of head_du_kernel

__device__ __forceinline__ float widen(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ float widen(float x) { return x; }
// eight consecutive elements of a row as they are loaded
template <typename T> struct Row8;
template <> struct Row8<__nv_bfloat16> {
    uint4 v;
    __device__ __forceinline__ void load(const __nv_bfloat16* p) { v = __ldg(reinterpret_cast<const uint4*>(p)); }
    __device__ __forceinline__ void widen(float (&o)[8]) const {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) { o[2 * i] = __uint_as_float(w[i] << 16); o[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
    }
};
template <> struct Row8<float> {
    float4 a, b;
    __device__ __forceinline__ void load(const float* p) {
        a = __ldg(reinterpret_cast<const float4*>(p));
        b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    }
    __device__ __forceinline__ void widen(float (&o)[8]) const {
        o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w; o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
    }
};

__device__ __forceinline__ void load_vector(const __nv_bfloat16* p, float (&o)[8]) {
    Row8<__nv_bfloat16> x;
    x.load(p);
    x.widen(o);
}
__device__ __forceinline__ void load_vector(const float* p, float (&o)[4]) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}

// Linear head, first kernel: ds_i = (sigmoid(s_i) - y_i) / n of the row-chunk's rollouts (every block counts the labelled ones itself), their losses
// and sum, and partial[c][k] = sum over the rows of row-chunk c of ds_i x_ik, in index order.  Thread = 8 consecutive columns.  Bound by
// the latency of its loads: the row numbers come with what ds is made of, and sixteen rows are in flight.  Rows without a factor are
// not read.  Second kernel: the chunks' sums.  As three kernels, ds by one block, blocks of 2,048 columns with eight rows in flight, a thread per
// column for the sums, a whole call took 19.6 us where it takes 9.4 now (graph of 20, N = 2,048, d = 2,048, bf16; 172, 1,464 15.2 -> 7.7; 8,192,
// 4,096 48.6 -> 25.6; 8,192, 512, fp32 30.4 -> 11.5).  What every block's counting costs grows with the square of the rollouts: N = 65,536, d = 4,096
// 215 us without a mask, 233 with one, 301 with one that is not 16-byte aligned (448 when one block counted, and formed ds for all).
constexpr int LIN_ROWS = 32, LIN_AHEAD = 16, LIN_THREADS = 128;
template <typename T>
__global__ void __launch_bounds__(LIN_THREADS)
linear_dw_partial_kernel(const T* hidden, int64_t row_stride, const int64_t* row_index, int N, int d, const float* score, const float* rewards,
                         const uint8_t* mask, float* __restrict__ partial, double* __restrict__ chunk_loss /* [2][chunks]: losses / n, ds */) {
    __shared__ float g_s[LIN_ROWS];
    __shared__ int64_t row_s[LIN_ROWS];
    __shared__ int warp_n[LIN_THREADS / 32];
    pdl_launch_dependents();
    pdl_wait();
    hidden = pdl_acquire(hidden); row_index = pdl_acquire(row_index); score = pdl_acquire(score); rewards = pdl_acquire(rewards);
    mask = pdl_acquire(mask);
    const int k0 = (blockIdx.x * LIN_THREADS + threadIdx.x) * 8;
    const int i0 = blockIdx.y * LIN_ROWS, i = i0 + (int)threadIdx.x;
    const bool mine = threadIdx.x < LIN_ROWS && i < N;           // the first warp's lanes: a rollout each
    bool labelled = false;
    float s = 0.f, y = 0.f;
    if (mine) {
        labelled = !mask || mask[i];
        s = score[i];
        y = rewards[i] > 0.5f ? 1.f : 0.f;
        row_s[threadIdx.x] = row_index ? row_index[i] : (int64_t)i;
    }
    const int c = __reduce_add_sync(0xffffffffu, mask ? count_labelled(mask, N, threadIdx.x, LIN_THREADS) : 0);
    if ((threadIdx.x & 31) == 0) warp_n[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x < LIN_ROWS) {
        int n = mask ? 0 : N;
#pragma unroll
        for (int w = 0; w < LIN_THREADS / 32; ++w) n += warp_n[w];
        float v = 0.f;
        double l = 0.0, sd = 0.0;
        if (labelled) {
            const float softplus = s > 0.f ? s + log1pf(expf(-s)) : log1pf(expf(s));
            l = (double)(softplus - y * s) / (double)n;
            v = (1.0f / (1.0f + expf(-s)) - y) / (float)n;
            sd = (double)v;
        }
        g_s[threadIdx.x] = v;
        if (blockIdx.x == 0) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                l += __shfl_xor_sync(0xffffffffu, l, o);
                sd += __shfl_xor_sync(0xffffffffu, sd, o);
            }
            if (threadIdx.x == 0) { chunk_loss[blockIdx.y] = l; chunk_loss[gridDim.y + blockIdx.y] = sd; }
        }
    }
    __syncthreads();
    if (k0 >= d) return;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int r0 = 0; r0 < LIN_ROWS; r0 += LIN_AHEAD) {
        Row8<T> x[LIN_AHEAD];
#pragma unroll
        for (int r = 0; r < LIN_AHEAD; ++r)
            if (g_s[r0 + r] != 0.f) x[r].load(hidden + row_s[r0 + r] * row_stride + k0);
#pragma unroll
        for (int r = 0; r < LIN_AHEAD; ++r)
            if (g_s[r0 + r] != 0.f) {
                float w[8];
                x[r].widen(w);
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[e] = fmaf(g_s[r0 + r], w[e], acc[e]);
            }
    }
    float* out = partial + (int64_t)blockIdx.y * d + k0;
    *reinterpret_cast<float4*>(out) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    *reinterpret_cast<float4*>(out + 4) = make_float4(acc[4], acc[5], acc[6], acc[7]);
}

// A block per 32 columns: eight warps take every eighth chunk, their sums are added in order.  The first block's last warp: loss and db.
__global__ void __launch_bounds__(288)
column_sum_kernel(const float* partial, const double* chunk_loss, int chunks, int d, float* __restrict__ out, double* __restrict__ loss,
                  float* __restrict__ dbias) {
    __shared__ float sums[8][32];
    pdl_launch_dependents();
    pdl_wait();
    partial = pdl_acquire(partial); chunk_loss = pdl_acquire(chunk_loss);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + lane;
    if (warp < 8) {
        float s = 0.f;
        if (k < d)
#pragma unroll 8
            for (int c = warp; c < chunks; c += 8) s += partial[(int64_t)c * d + k];
        sums[warp][lane] = s;
    } else if (blockIdx.x == 0) {
        double l = 0.0, sd = 0.0;
#pragma unroll 4
        for (int c = lane; c < chunks; c += 32) { l += chunk_loss[c]; sd += chunk_loss[chunks + c]; }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            l += __shfl_xor_sync(0xffffffffu, l, o);
            sd += __shfl_xor_sync(0xffffffffu, sd, o);
        }
        if (lane == 0) { *loss = l; *dbias = (float)sd; }
    }
    __syncthreads();
    if (warp == 0 && k < d) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) s += sums[w][lane];
        out[k] = s;
    }
}

// MLP heads whose forward does not form du itself (fp32, h not a multiple of 8, and where the tensor-core forward goes without clusters):
// everything between the forward and the dW1 contraction in one launch: ds_i, the loss, du_ij, and per hidden unit
// the sums dw2_j = sum_i ds_i gelu(u_ij), db1_j = sum_i du_ij.  (It was four launches: ds by one block, du, two column sums,
// 22 us at N = 2,048, h = 256 against 9.)  Block (x, y): 32 hidden units, a run of rollouts.  Every block counts the labelled
// rollouts itself and forms the ds of its own run; the last block of a column tile to arrive (a counter per tile, zero again when that
// block is through) adds the runs' sums in index order, the one of tile 0 the loss and db2 as well.  The score is given, or the sum of
// the forward's tile partials + b2.
// du goes out as float (SIMT contraction) or as the sum of two bf16 planes (error 2^-17 relative: the tensor-core operand).
constexpr int DU_THREADS = 256;
template <typename T>
__global__ void __launch_bounds__(DU_THREADS)
head_du_kernel(const float* u, const float* score, const float* partial, int h_tiles, const T* b2, const float* rewards,
               const uint8_t* mask, const T* w2, int N, int h, int rows_per_run, float* __restrict__ du,
               __nv_bfloat16* __restrict__ du_hi, __nv_bfloat16* __restrict__ du_lo, float* run_sums /* [2][runs][h] */,
               double* run_loss /* [2][runs] */, uint32_t* counters, float* __restrict__ dw2, float* __restrict__ db1,
               double* __restrict__ loss, float* __restrict__ db2) {
    extern __shared__ float ds_s[];            // [rows_per_run]; NaN-free: 0 for rollouts that do not count
    __shared__ float sums[2][8][33];
    __shared__ double warp_d[2][DU_THREADS / 32];
    __shared__ int warp_n[DU_THREADS / 32], is_last;
    pdl_launch_dependents();
    pdl_wait();
    u = pdl_acquire(u); score = pdl_acquire(score); rewards = pdl_acquire(rewards); mask = pdl_acquire(mask);
    w2 = pdl_acquire(w2); partial = pdl_acquire(partial); b2 = pdl_acquire(b2);
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int runs = gridDim.y, run = blockIdx.y;
    const int i0 = run * rows_per_run, i1 = min(N, i0 + rows_per_run);
    const int j = blockIdx.x * 32 + tx;
    // everything that depends on nothing is requested first: the first pre-activations, then the labels to count
    constexpr int AHEAD = 8;
    float ahead[AHEAD];
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) {
        const int i = i0 + ty + 8 * k;
        ahead[k] = j < h && i < i1 ? u[(int64_t)i * h + j] : 0.f;
    }
    const float wj = j < h ? widen(w2[j]) : 0.f;
    {
        int c = mask ? count_labelled(mask, N, threadIdx.x, DU_THREADS) : 0;
        c = __reduce_add_sync(0xffffffffu, c);
        if (tx == 0) warp_n[ty] = c;
    }
    __syncthreads();
    int n = mask ? 0 : N;
#pragma unroll
    for (int w = 0; w < DU_THREADS / 32; ++w) n += warp_n[w];
    double l = 0.0, sd = 0.0;
    for (int i = i0 + threadIdx.x; i < i1; i += DU_THREADS) {
        float v = 0.f;
        if (!mask || mask[i]) {
            float s = 0.f;
            if (score) {
                s = score[i];
            } else {
                for (int t = 0; t < h_tiles; ++t) s += partial[(int64_t)t * N + i];
                if (b2) s += widen(b2[0]);
            }
            const float y = rewards[i] > 0.5f ? 1.f : 0.f;
            const float softplus = s > 0.f ? s + log1pf(expf(-s)) : log1pf(expf(s));
            l += (double)(softplus - y * s);
            v = (1.0f / (1.0f + expf(-s)) - y) / (float)n;
            sd += (double)v;
        }
        ds_s[i - i0] = v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        l += __shfl_xor_sync(0xffffffffu, l, o);
        sd += __shfl_xor_sync(0xffffffffu, sd, o);
    }
    if (tx == 0) { warp_d[0][ty] = l; warp_d[1][ty] = sd; }
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x < 2) {
        double t = 0.0;
        for (int w = 0; w < DU_THREADS / 32; ++w) t += warp_d[threadIdx.x][w];
        run_loss[threadIdx.x * runs + run] = t;
    }
    float a_w2 = 0.f, a_b1 = 0.f;
    if (j < h) {
        auto one = [&](int i, float a) {
            const float g = ds_s[i - i0];
            const float cdf = 0.5f * (1.0f + erff(a * 0.70710678118654752440f));
            const float pdf = expf(-0.5f * a * a) * 0.39894228040143267794f;
            const float d_u = g * wj * (cdf + a * pdf);
            if (du) {
                du[(int64_t)i * h + j] = d_u;
            } else {
                const __nv_bfloat16 hi = __float2bfloat16_rn(d_u);
                du_hi[(int64_t)i * h + j] = hi;
                du_lo[(int64_t)i * h + j] = __float2bfloat16_rn(d_u - __bfloat162float(hi));
            }
            a_w2 = fmaf(g, a * cdf, a_w2);
            a_b1 += d_u;
        };
#pragma unroll
        for (int k = 0; k < AHEAD; ++k)
            if (i0 + ty + 8 * k < i1) one(i0 + ty + 8 * k, ahead[k]);
#pragma unroll 4
        for (int i = i0 + ty + 8 * AHEAD; i < i1; i += 8) one(i, u[(int64_t)i * h + j]);
    }
    sums[0][ty][tx] = a_w2;
    sums[1][ty][tx] = a_b1;
    __syncthreads();
    if (ty < 2 && j < h) {
        float t = 0.f;
        for (int r = 0; r < 8; ++r) t += sums[ty][r][tx];
        run_sums[((int64_t)ty * runs + run) * h + j] = t;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        is_last = atomicAdd(&counters[blockIdx.x], 1u) == (uint32_t)runs - 1u ? 1 : 0;
        if (is_last) counters[blockIdx.x] = 0u;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    if (ty < 2 && j < h) {
        float t = 0.f;
#pragma unroll 8
        for (int r = 0; r < runs; ++r) t += __ldcg(&run_sums[((int64_t)ty * runs + r) * h + j]);
        (ty == 0 ? dw2 : db1)[j] = t;
    }
    if (blockIdx.x == 0 && threadIdx.x >= 64 && threadIdx.x < 66) {
        const int which = threadIdx.x - 64;
        double t = 0.0;
        for (int r = 0; r < runs; ++r) t += __ldcg(&run_loss[which * runs + r]);
        if (which == 0) *loss = n > 0 ? t / (double)n : 0.0;
        else *db2 = (float)t;
    }
}

// dW1[j][k] = sum_i du[i][j] x[i][k]: 64 x 64 output tile per block, 8 x 4 per thread, rollouts in chunks of 32.  A head has few such tiles (d = 512,
// h = 256: 32) and each contracts all rollouts, so the rollouts are cut into ranges over the blocks of a cluster, whose sums meet in
// shared memory and are added in rank order; and a chunk waits for its row numbers and then for its rows, so they are requested
// two chunks and one ahead.  N = 2,000, d = 512, h = 256 (fp32): this
// kernel 292 us under the profiler as 32 blocks that waited for every load; whole call, with the forward's K over a cluster
// too and the launches below, graph of 20: 235 -> 58 us, N = 8,000, d = 1,024, h = 256 957 -> 315,
// 5,000, 256, 64 488 -> 61, 283, 288, 64 55 -> 23.
constexpr int GT = 64, GK = 32, GPAD = 4, DW1_THREADS = 128, DW1_SPLITS = 8;
template <typename T>
__global__ void __launch_bounds__(DW1_THREADS)
mlp_dw1_kernel(const float* du, const T* hidden, int64_t row_stride, const int64_t* row_index, int N, int d, int h, float* __restrict__ dW1) {
    constexpr int VN = 16 / (int)sizeof(T);                      // columns per 16-byte vector of x
    constexpr int XV = GK * GT / VN / DW1_THREADS, AV = GK * GT / 4 / DW1_THREADS;       // vectors per thread and chunk
    constexpr int X_STEP = DW1_THREADS * VN / GT;                // rows between a thread's vectors of x
    __shared__ __align__(16) float as[2][GK][GT + GPAD];         // du rows
    __shared__ __align__(16) float bs[2][GK][GT + GPAD];         // x rows
    static_assert(sizeof(float) * GT * (GT + GPAD) <= sizeof(as), "the block's sums fit the du rows");
    const int tid = threadIdx.x, j0 = blockIdx.y * GT, c0 = blockIdx.x * GT;
    const int tx = tid & 15, ty = tid >> 4;
    const int splits = gridDim.z, rank = blockIdx.z;             // the cluster's blocks
    const int chunks = (N + GK - 1) / GK;
    const int first = (int)((int64_t)rank * chunks / splits), last = (int)((int64_t)(rank + 1) * chunks / splits);
    const int xr = tid * VN / GT, xc = c0 + tid * VN % GT;       // this thread's first vector of x
    const int ar = tid / (GT / 4), aj = j0 + tid % (GT / 4) * 4; // and of du
    pdl_launch_dependents();
    pdl_wait();
    du = pdl_acquire(du); hidden = pdl_acquire(hidden); row_index = pdl_acquire(row_index);
    int64_t row[XV];                                             // of the chunk that is requested next
    float4 a_next[AV];
    float x_next[XV][VN];
    auto rows_of = [&](int chunk) {
#pragma unroll
        for (int i = 0; i < XV; ++i) {
            const int r = chunk * GK + xr + X_STEP * i;
            row[i] = chunk < last && r < N ? (row_index ? row_index[r] : (int64_t)r) : -1;
        }
    };
    auto fetch = [&](int chunk) {
#pragma unroll
        for (int i = 0; i < AV; ++i) {
            const int r = chunk * GK + ar + 8 * i;
            a_next[i] = chunk < last && r < N && aj < h ? *reinterpret_cast<const float4*>(du + (int64_t)r * h + aj)    // h % 4 == 0
                                                        : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < XV; ++i) {
            const int r = chunk * GK + xr + X_STEP * i;
            if (chunk < last && r < N && xc < d) {
                load_vector(hidden + row[i] * row_stride + xc, x_next[i]);
            } else {
#pragma unroll
                for (int e = 0; e < VN; ++e) x_next[i][e] = 0.f;
            }
        }
    };
    float acc[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
    rows_of(first);
    fetch(first);
    rows_of(first + 1);
    int buf = 0;
    for (int c = first; c < last; ++c, buf ^= 1) {
#pragma unroll
        for (int i = 0; i < AV; ++i) *reinterpret_cast<float4*>(&as[buf][ar + 8 * i][aj - j0]) = a_next[i];
#pragma unroll
        for (int i = 0; i < XV; ++i)
#pragma unroll
            for (int e = 0; e < VN; e += 4)
                *reinterpret_cast<float4*>(&bs[buf][xr + X_STEP * i][xc - c0 + e]) = make_float4(x_next[i][e], x_next[i][e + 1], x_next[i][e + 2], x_next[i][e + 3]);
        fetch(c + 1);
        rows_of(c + 2);
        __syncthreads();                                         // the other buffer was last read before the previous one
#pragma unroll
        for (int kk = 0; kk < GK; ++kk) {
            const float4 a0 = *reinterpret_cast<const float4*>(&as[buf][kk][ty * 8]);
            const float4 a1 = *reinterpret_cast<const float4*>(&as[buf][kk][ty * 8 + 4]);
            const float4 b0 = *reinterpret_cast<const float4*>(&bs[buf][kk][tx * 4]);
            const float ar8[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float br4[4] = {b0.x, b0.y, b0.z, b0.w};
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(ar8[a], br4[b], acc[a][b]);
        }
    }
    __syncthreads();
    float* sums = &as[0][0][0];                                  // [GT][GT + GPAD]
#pragma unroll
    for (int a = 0; a < 8; ++a)
        *reinterpret_cast<float4*>(sums + (ty * 8 + a) * (GT + GPAD) + tx * 4) = make_float4(acc[a][0], acc[a][1], acc[a][2], acc[a][3]);
    cluster_sync_all();
    const int rows_each = GT / splits;                           // every block finishes its share of the tile's rows
    for (int i = tid; i < rows_each * (GT / 4); i += DW1_THREADS) {
        const int r = rank * rows_each + i / (GT / 4), c = i % (GT / 4) * 4;
        const uint32_t at = smem_u32(sums + r * (GT + GPAD) + c);
        float4 sum = ld_shared_cluster_v4(map_to_cta(at, 0u));
        for (int z = 1; z < splits; ++z) {
            const float4 v = ld_shared_cluster_v4(map_to_cta(at, (uint32_t)z));
            sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
        }
        if (j0 + r < h && c0 + c < d) *reinterpret_cast<float4*>(dW1 + (int64_t)(j0 + r) * d + c0 + c) = sum;      // d % 8 == 0
    }
    cluster_sync_all();                 // nobody's shared memory goes away while it is being read
}

struct GradLayout {
    size_t tmp3, ds, u, du, run_loss, run_sums, counters, partial, total;   // byte offsets
    size_t du_plane;                          // bytes of one bf16 plane of du (hi at du, lo at du + du_plane)
};
GradLayout grad_layout(int N, int d, int h) {
    GradLayout L;
    auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
    size_t o = 0;
    L.tmp3 = o; o = up(o + sizeof(float) * 3 * (size_t)N);
    L.ds = o; o = up(o + sizeof(float) * (size_t)N);
    L.u = o; o = up(o + sizeof(float) * (size_t)N * (size_t)(h > 0 ? h : 0));
    const size_t plane = up(sizeof(uint16_t) * (size_t)N * (size_t)(h > 0 ? h : 0));   // one bf16 plane of du
    L.du = o; o = up(o + (sizeof(float) * (size_t)N * (size_t)(h > 0 ? h : 0) > 2 * plane
                              ? sizeof(float) * (size_t)N * (size_t)(h > 0 ? h : 0) : 2 * plane));
    L.du_plane = plane;
    const size_t chunks = ((size_t)N + LIN_ROWS - 1) / LIN_ROWS;
    const size_t tiles = (size_t)((h > 0 ? h : 0) + ARROL_MLP_TH - 1) / ARROL_MLP_TH;
    size_t part = h > 0 ? tiles * (size_t)N : chunks * (size_t)d;
    L.run_loss = o; o = up(o + sizeof(double) * 2 * DU_RUNS);                                       // loss / db2 per run
    L.run_sums = o; o = up(o + sizeof(float) * 2 * (size_t)DU_RUNS * (size_t)(h > 0 ? h : 0));      // dw2 / db1 per run
    L.counters = o; o = up(o + sizeof(uint32_t) * (size_t)(((h > 0 ? h : 0) + 31) / 32));             // finished runs per column tile
    L.partial = o; o = up(o + sizeof(float) * part);
    L.total = o;
    return L;
}

template <typename T>
int run_head_grad(arrol_ctx* ctx, const void* hidden, int64_t row_stride, const int64_t* row_index, int N,
                  const arrol_head* head, const float* rewards, const uint8_t* mask, float* dW1, float* db1,
                  float* dw2, float* db2, double* loss, uint8_t* ws, const GradLayout& L, cudaStream_t s) {
    const T* hid = static_cast<const T*>(hidden);
    float* ds = reinterpret_cast<float*>(ws + L.ds);
    float* partial = reinterpret_cast<float*>(ws + L.partial);
    const int d = head->d, h = head->h;
    if (h == 0) {
        float* tmp = reinterpret_cast<float*>(ws + L.tmp3);
        const int rc = arrol_score_partial(ctx, hidden, row_stride, row_index, N, head, nullptr, tmp, tmp + N, nullptr,
                                           tmp + 2 * (size_t)N, s);
        if (rc != ARROL_OK) return rc;
        const int chunks = (N + LIN_ROWS - 1) / LIN_ROWS;
        double* chunk_loss = reinterpret_cast<double*>(ds);          // 16 bytes per 32 rollouts
        ARROL_CUDA_OK(arrol_launch_pdl(linear_dw_partial_kernel<T>, dim3((d / 8 + LIN_THREADS - 1) / LIN_THREADS, chunks), dim3(LIN_THREADS), 0, s, hid,
                                       row_stride, row_index, N, d, static_cast<const float*>(tmp), rewards, mask, partial, chunk_loss));
        ARROL_CUDA_OK(arrol_launch_pdl(column_sum_kernel, dim3((d + 31) / 32), dim3(288), 0, s, static_cast<const float*>(partial),
                                       static_cast<const double*>(chunk_loss), chunks, d, dW1, loss, db1));
        ctx->launches += 2;
    } else {
        float* u = reinterpret_cast<float*>(ws + L.u);
        float* du = reinterpret_cast<float*>(ws + L.du);
        const int rows_per = ((N + DU_RUNS - 1) / DU_RUNS + 7) / 8 * 8;
        const int runs = (N + rows_per - 1) / rows_per;
        auto launch_du = [&](const float* score, const float* tile_partial, int h_tiles, float* du_f, __nv_bfloat16* hi,
                             __nv_bfloat16* lo, uint32_t* counters) -> int {
            ARROL_CUDA_OK(arrol_launch_pdl(head_du_kernel<T>, dim3((h + 31) / 32, runs), dim3(DU_THREADS), sizeof(float) * rows_per, s,
                                           static_cast<const float*>(u), score, tile_partial, h_tiles,
                                           score ? nullptr : static_cast<const T*>(head->b2), rewards, mask,
                                           static_cast<const T*>(head->w2), N, h, rows_per, du_f, hi, lo,
                                           reinterpret_cast<float*>(ws + L.run_sums), reinterpret_cast<double*>(ws + L.run_loss),
                                           counters, dw2, db1, loss, db2));
            ctx->launches += 1;
            return ARROL_OK;
        };
        if constexpr (sizeof(T) == 2) {
            // bf16 head: both contractions on the tensor cores.  Forward with the pre-activations kept, du split into
            // two bf16 planes, dW1 = du_hi^T X + du_lo^T X with X the packed rows (or the rows in place).
            if (h % 8 == 0) {
                __nv_bfloat16* du_hi = reinterpret_cast<__nv_bfloat16*>(ws + L.du);
                __nv_bfloat16* du_lo = reinterpret_cast<__nv_bfloat16*>(ws + L.du + L.du_plane);
                // sums per tile of 64 rollouts or more: where the other path keeps those of its runs, of more tiles where it keeps u and ds
                const bool few = (N + 63) / 64 <= DU_RUNS;
                float* tile_sums = few ? reinterpret_cast<float*>(ws + L.run_sums) : u;
                double* tile_loss = few ? reinterpret_cast<double*>(ws + L.run_loss) : reinterpret_cast<double*>(ds);
                int tile_rows = 128;
                int rc = arrol_internal_head_train_tc(ctx, hidden, row_stride, row_index, N, head, rewards, mask, du_hi, du_lo,
                                                      tile_sums, tile_loss, &tile_rows, s);
                HeadTileSums sums = {(N + tile_rows - 1) / tile_rows, tile_sums, tile_loss, dw2, db1, loss, db2};
                if (rc == ARROL_ERR_UNSUPPORTED) {      // no clusters for these sizes, or beyond the context's buffers
                    float* tmp = reinterpret_cast<float*>(ws + L.tmp3);
                    sums.tile_sums = nullptr;
                    rc = arrol_internal_score_mlp_tc(ctx, hidden, row_stride, row_index, N, head, 0, nullptr, tmp, tmp + N, nullptr,
                                                     tmp + 2 * (size_t)N, u, s);
                    if (rc == ARROL_OK) rc = launch_du(tmp, nullptr, 0, nullptr, du_hi, du_lo, ctx->d_head_counters);
                }
                if (rc == ARROL_OK)
                    return arrol_internal_head_dw1(ctx, du_hi, du_lo, row_index ? ctx->d_pack : hidden,
                                                   row_index ? (int64_t)d : row_stride, N, d, h, dW1, sums, s);
                if (rc != ARROL_ERR_UNSUPPORTED) return rc;
            }
        }
        // this path works in the call's own workspace alone, so that calls on several streams do not meet; its counters too
        // (a call on the tensor cores shares the context's packing buffer and scoring counters with others anyway)
        uint32_t* counters = reinterpret_cast<uint32_t*>(ws + L.counters);
        const int rc = arrol_internal_mlp_tiles(ctx, hidden, row_stride, row_index, N, head, partial, u, counters, (h + 31) / 32, s);
        if (rc != ARROL_OK) return rc;
        const int rd = launch_du(nullptr, partial, (h + ARROL_MLP_TH - 1) / ARROL_MLP_TH, du, nullptr, nullptr, counters);
        if (rd != ARROL_OK) return rd;
        const int tiles = ((d + GT - 1) / GT) * ((h + GT - 1) / GT), row_chunks = (N + GK - 1) / GK;
        int splits = 1;                     // two chunks at least, and no more than about four blocks per SM
        while (splits < DW1_SPLITS && tiles * splits * 2 <= 4 * ctx->sm_count && row_chunks >= splits * 2 * 2) splits *= 2;
        // Launched while the du kernel runs where both kernels' blocks have an SM each: more of them would pile up on the SMs that the du
        // kernel leaves free.  When it has ended / while it runs: N = 64, d = 256, h = 64 (4 + 16 blocks) 19.9 / 18.2 us, 300, 512, 128 (64 + 76)
        // 27.5 / 26.6, 20,000, 256, 64 (32 + 64) 188 / 187; past the line 300, 1,024, 256 (256 + 152) 36.4 / 39.9, 4,000, 512, 128 (128 + 128)
        // 79 / 90, 7,000, 1,024, 64 (128 + 64) 131 / 167, 700, 1,024, 64 (128 + 60) 37.1 / 36.2.
        const bool early = tiles * splits + (h + 31) / 32 * runs <= ctx->sm_count;
        ARROL_CUDA_OK(arrol_launch_cluster(early, mlp_dw1_kernel<T>, dim3((d + GT - 1) / GT, (h + GT - 1) / GT, splits), dim3(DW1_THREADS),
                                           dim3(1, 1, splits), s, static_cast<const float*>(du), hid, row_stride, row_index, N, d, h, dW1));
        ctx->launches += 1;
    }
    ARROL_CUDA_OK(cudaGetLastError());
    return ARROL_OK;
}

}  // namespace

extern "C" size_t arrol_head_grad_workspace(arrol_ctx* ctx, int32_t N, int32_t d, int32_t h) {
    if (!ctx || N <= 0 || d <= 0 || h < 0) return 0;
    return grad_layout(N, d, h).total;
}

extern "C" int arrol_head_grad(arrol_ctx* ctx, const void* hidden, int64_t row_stride_elems, const int64_t* row_index,
                               int32_t N, const arrol_head* head, const float* rewards, const uint8_t* mask,
                               float* dW1, float* db1, float* dw2, float* db2, double* loss, void* workspace,
                               size_t workspace_bytes, void* stream) {
    if (!ctx || !head || N < 0) return ARROL_ERR_INVALID_ARG;
    if (!loss || !dW1 || !db1) return ARROL_ERR_INVALID_ARG;
    if (head->h > 0 && (!dw2 || !db2 || !head->w2)) return ARROL_ERR_INVALID_ARG;
    if (head->dtype != ARROL_F32 && head->dtype != ARROL_BF16) return ARROL_ERR_INVALID_ARG;
    if (head->d <= 0 || head->h < 0 || !head->W1) return ARROL_ERR_INVALID_ARG;
    if (head->d % 8 != 0 || head->h % 4 != 0 || head->h > ARROL_MAX_H) return ARROL_ERR_UNSUPPORTED;
    if (N > ARROL_MAX_MLP_N) return ARROL_ERR_UNSUPPORTED;
    if (N > 0 && (!hidden || !rewards)) return ARROL_ERR_INVALID_ARG;
    const int esz = head->dtype == ARROL_F32 ? 4 : 2;
    if (N > 0 && (row_stride_elems < head->d || (row_stride_elems * esz) % 16 != 0 || !arrol_aligned(hidden, 16)))
        return ARROL_ERR_INVALID_ARG;
    if (!arrol_aligned(dW1, 16)) return ARROL_ERR_INVALID_ARG;
    ArrolDeviceGuard guard(ctx->device);
    if (!guard.ok) return ARROL_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    if (N == 0) {   // nothing to learn from: zero loss and gradients
        const size_t hh = head->h > 0 ? (size_t)head->h : 1;
        ARROL_CUDA_OK(cudaMemsetAsync(loss, 0, sizeof(double), s));
        ARROL_CUDA_OK(cudaMemsetAsync(dW1, 0, sizeof(float) * hh * head->d, s));
        ARROL_CUDA_OK(cudaMemsetAsync(db1, 0, sizeof(float) * hh, s));
        if (head->h > 0) {
            ARROL_CUDA_OK(cudaMemsetAsync(dw2, 0, sizeof(float) * hh, s));
            ARROL_CUDA_OK(cudaMemsetAsync(db2, 0, sizeof(float), s));
        }
        return ARROL_OK;
    }
    const GradLayout L = grad_layout(N, head->d, head->h);
    if (!workspace || workspace_bytes < L.total || !arrol_aligned(workspace, 256)) return ARROL_ERR_WORKSPACE;
    uint8_t* ws = static_cast<uint8_t*>(workspace);
    if (head->dtype == ARROL_F32)
        return run_head_grad<float>(ctx, hidden, row_stride_elems, row_index, N, head, rewards, mask, dW1, db1, dw2,
                                    db2, loss, ws, L, s);
    return run_head_grad<__nv_bfloat16>(ctx, hidden, row_stride_elems, row_index, N, head, rewards, mask, dW1, db1,
                                        dw2, db2, loss, ws, L, s);
}
