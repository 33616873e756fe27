// Per-token outputs of the compaction (token ids, survivor ordinal, advantage): device code of the kernel that writes them
// alone (gather_tokens_kernel) and of the row gather, which writes them beside its copies while these fit L2 (gather_rows_bulk_kernel).
#pragma once
#include "arrol_internal.h"

struct TokenOutputs {
    const int32_t* src_tokens;     // with dst_tokens
    const float* adv;              // per survivor
    int32_t* dst_tokens;           // each of the three outputs may be NULL
    float* tok_adv;
    int32_t* tok_seq;
    int vector_stores;             // the outputs start on 16-byte boundaries, the ids on 4-byte ones
    __host__ __device__ bool any() const { return dst_tokens || tok_adv || tok_seq; }
};
inline TokenOutputs token_outputs(const int32_t* src_tokens, const float* adv, int32_t* dst_tokens, float* tok_adv, int32_t* tok_seq) {
    TokenOutputs o{src_tokens, adv, dst_tokens, tok_adv, tok_seq, 0};
    o.vector_stores = arrol_aligned(dst_tokens, 16) && arrol_aligned(tok_adv, 16) && arrol_aligned(tok_seq, 16) && arrol_aligned(src_tokens, 4);
    return o;
}

// A survivor's run of tokens, left by the fused prune step for the kernel that writes the per-token outputs.
struct alignas(16) SurvivorRun {
    int64_t c0, src0;              // where it begins in the packed outputs and in the source
    int32_t len;
    float adv;
    int32_t pad[2];
};
__device__ __forceinline__ SurvivorRun load_run(const SurvivorRun* p) {
    const int4 a = *reinterpret_cast<const int4*>(p), b = *(reinterpret_cast<const int4*>(p) + 1);
    SurvivorRun r;
    r.c0 = (int64_t)(uint32_t)a.x | (int64_t)a.y << 32;
    r.src0 = (int64_t)(uint32_t)a.z | (int64_t)a.w << 32;
    r.len = b.x;
    r.adv = __int_as_float(b.y);
    return r;
}

// A team of lanes per survivor walks its run of tokens, so nothing has to be searched.  Bound by the bytes it moves
// (16 per token, 12 of them written): all three outputs leave as 16-byte stores, four tokens per lane.  The source run is
// aligned differently from the destination, so a lane reads the two aligned 16-byte words that hold its four ids (the second
// one is its neighbour's first, in L1 by then) and picks them out, without a branch, so that a lane's loads are all in
// flight together.  The few ids whose words would reach outside the run go one by one.
// Prune step without a payload plane, 4-byte stores and 128 threads per survivor / this / 16-byte stores and 256 threads per
// survivor: 1,024 runs of 2,600 ids 26.1 / 22.0 / 22.9 us; 12,288 of 131 58.6 / 52.6 / 69.7; 2,048 of 600 19.9 / 19.7 / 22.0; 828 of
// 275 12.3 / 12.5 / 12.9; 8 of 1,240 12.3 / 12.1 / 12.0.  Beyond what L2 holds (6.5 M ids, 104 MB) the stores go at HBM's pace.
constexpr int TOKENS_QUADS = 2;          // groups of four tokens in flight per lane (3 or 4 spill at four blocks per SM: 24.4, 26.7 us on the first of these)
// Survivors first, first + step, ... by lane `lane` of a team of `lanes`; next_run(s) gives survivor s's run.
template <typename NextRun>
__device__ __forceinline__ void token_runs(const TokenOutputs& o, NextRun next_run, int S, int first, int step, int lane, int lanes) {
    const int32_t* __restrict__ src_tokens = o.src_tokens;
    int32_t* __restrict__ dst_tokens = o.dst_tokens;
    float* __restrict__ tok_adv = o.tok_adv;
    int32_t* __restrict__ tok_seq = o.tok_seq;
#pragma unroll 1
    for (int s = first; s < S; s += step) {
        const SurvivorRun run = next_run(s);
        const int64_t c0 = run.c0, src0 = run.src0;
        const int len = run.len;
        const float a = run.adv;
        auto load_one = [&](int t) { return dst_tokens ? __ldg(src_tokens + src0 + t) : 0; };
        auto store_one = [&](int t, int32_t id) {
            if (dst_tokens) dst_tokens[c0 + t] = id;
            if (tok_seq) tok_seq[c0 + t] = s;
            if (tok_adv) tok_adv[c0 + t] = a;
        };
        // [head, end): whole 16-byte groups of the outputs whose ids lie in words inside the run
        int head = (int)((4 - (c0 & 3)) & 3), end = len - (int)((c0 + len) & 3);
        const int shift = (int)((reinterpret_cast<uintptr_t>(src_tokens + src0 + head) & 15) >> 2);   // ids before src0 + head in its word
        if (shift > head) head += 4;
        if (shift && end - shift + 4 > len) end -= 4;
        if (!o.vector_stores || end <= head) {
#pragma unroll 1
            for (int t = lane; t < len; t += lanes) store_one(t, load_one(t));
            continue;
        }
        // at most 6 ids before and 6 after, a lane each; stored after the groups, or the first lanes' loads would wait for a
        // store that waits for its id
        const int edge = lane < head ? lane : (lane >= 8 && end + lane - 8 < len ? end + lane - 8 : -1);
        const int32_t edge_id = edge >= 0 ? load_one(edge) : 0;
        const int4* words = reinterpret_cast<const int4*>(src_tokens + src0 + head - shift);
        const int quads = (end - head) / 4, second = shift ? 1 : 0;
#pragma unroll 1
        for (int k0 = lane; k0 < quads; k0 += TOKENS_QUADS * lanes) {
            int4 lo[TOKENS_QUADS], hi[TOKENS_QUADS];
            if (dst_tokens) {
#pragma unroll
                for (int u = 0; u < TOKENS_QUADS; ++u) {
                    const int k = k0 + u * lanes;
                    if (k < quads) {
                        lo[u] = __ldg(words + k);
                        hi[u] = __ldg(words + k + second);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < TOKENS_QUADS; ++u) {
                const int k = k0 + u * lanes;
                if (k >= quads) break;
                const int64_t at = c0 + head + 4 * k;
                if (dst_tokens) {
                    const bool two = shift & 2, one = shift & 1;
                    const int32_t x0 = two ? lo[u].z : lo[u].x, x1 = two ? lo[u].w : lo[u].y, x2 = two ? hi[u].x : lo[u].z,
                                  x3 = two ? hi[u].y : lo[u].w, x4 = two ? hi[u].z : hi[u].x;
                    *reinterpret_cast<int4*>(dst_tokens + at) = make_int4(one ? x1 : x0, one ? x2 : x1, one ? x3 : x2, one ? x4 : x3);
                }
                if (tok_seq) *reinterpret_cast<int4*>(tok_seq + at) = make_int4(s, s, s, s);
                if (tok_adv) *reinterpret_cast<float4*>(tok_adv + at) = make_float4(a, a, a, a);
            }
        }
        if (edge >= 0) store_one(edge, edge_id);
    }
}

// the same, each run from the scan's outputs: two dependent round trips more than a SurvivorRun
__device__ __forceinline__ void token_runs(const TokenOutputs& o, const int64_t* __restrict__ cu_seqlens, const int32_t* __restrict__ survivor_idx,
                                           const int64_t* __restrict__ src_tok_off, int S, int first, int step, int lane, int lanes) {
    auto next_run = [&](int s) {
        SurvivorRun r;
        r.c0 = __ldg(cu_seqlens + s);
        r.len = (int)(__ldg(cu_seqlens + s + 1) - r.c0);
        r.src0 = __ldg(src_tok_off + __ldg(survivor_idx + s));
        r.adv = __ldg(o.adv + s);
        return r;
    };
    token_runs(o, next_run, S, first, step, lane, lanes);
}
