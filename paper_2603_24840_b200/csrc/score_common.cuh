// Device functions shared by the scoring and the head training kernels.
#pragma once
#include <stdint.h>

// Probability map (Appendix A.4): s -> s' = sigmoid(s), b = min(B-1, floor(B s')), q = q_lut[b]
__device__ __forceinline__ float probability_map(float s, int i, int B, const float* __restrict__ q_lut,
                                                 float* score, float* prob, int32_t* bin, float* q) {
    float sp = 1.0f / (1.0f + expf(-s));
    int b = 0;
    if (B > 0) {
        b = (int)floorf((float)B * sp);
        b = min(max(b, 0), B - 1);
    }
    score[i] = s;
    prob[i] = sp;
    if (bin) bin[i] = b;
    const float qv = (q_lut != nullptr) ? q_lut[b] : sp;      // global or shared memory
    q[i] = qv;
    return qv;
}

// one of `threads` threads' share of the rollouts with a label
__device__ __forceinline__ int count_labelled(const uint8_t* mask, int N, int thread, int threads) {
    int c = 0;
    const int vec = (reinterpret_cast<uintptr_t>(mask) & 15) == 0 ? N / 16 : 0;
    for (int i = thread; i < vec; i += threads) {
        const uint4 v = reinterpret_cast<const uint4*>(mask)[i];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) c += __popc(__vcmpne4(w[k], 0u)) >> 3;
    }
    for (int i = vec * 16 + thread; i < N; i += threads) c += mask[i] ? 1 : 0;
    return c;
}
