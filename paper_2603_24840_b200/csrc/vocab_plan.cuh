// How the log-prob kernels cut the vocabulary, and how much of an SM's shared memory their combining kernel may take.  Host and device; a
// plain C++ compiler takes it too (the host side is tested without a GPU).
#pragma once
#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define ARROL_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define ARROL_HOST_DEVICE inline
#endif

// a / b of small whole numbers by b's rounded reciprocal, taken half a unit above a: exact while a < 2^16 and b < 2^10 (the margin is
// 0.5 / b, the error a / b 2^-22).  An item of a small call would wait for the division of integers.
ARROL_HOST_DEVICE int quotient(int a, float inv_b) { return (int)(((float)a + 0.5f) * inv_b); }

// total_chunks chunks of columns -> n_sub segments -> n_mid blocks of segments -> splits
// groups.  A body item covers a whole group, a tail item one segment; a token's records are merged segment by segment
// into a block, block by block into a group, then group by group, by whichever kernel holds them.
constexpr int MAX_SPLITS = 64;
constexpr int MAX_SEGMENTS = 255;    // segments: their numbers are kept in 8 bits, and products of two in `quotient`
struct VocabPlan {
    int total_chunks, n_sub, n_mid, splits;
    int per_sub;          // whole chunks per segment, n_long segments hold one more
    int n_long;           // total_chunks mod n_sub
    float inv_sub, inv_long, inv_short;   // 1 / n_sub, 1 / n_long, 1 / (n_sub - n_long)
    uint8_t mid_begin[MAX_SPLITS + 1];    // first segment of every block of segments
    uint8_t group_begin[MAX_SPLITS + 1];  // first block of every group
    // floor(i total_chunks / n_sub), without a division
    ARROL_HOST_DEVICE int chunk_of_sub(int i) const { return i * per_sub + quotient(i * n_long, inv_sub); }
    // j-th segment in the order of dealing: the long ones first.  Segment i is long where floor(i n_long / n_sub) steps after i,
    // short where ceil(i (n_sub - n_long) / n_sub) does.
    ARROL_HOST_DEVICE int nth_sub(int j) const {
        const bool is_long = j < n_long;
        const int a = is_long ? (j + 1) * n_sub + n_long - 1 : (j - n_long) * n_sub;
        return quotient(a, is_long ? inv_long : inv_short) - (is_long ? 1 : 0);
    }
    ARROL_HOST_DEVICE int sub_of_group(int g) const { return mid_begin[group_begin[g]]; }
};

// 1 <= splits <= MAX_SPLITS
inline VocabPlan make_vocab_plan(int sm_count, int total_chunks, int splits) {
    VocabPlan v;
    v.total_chunks = total_chunks;
    v.splits = splits;
    // one segment per SM: then the tail's items fill the units (SMs, or half as many pairs) a whole number of times
    v.n_sub = total_chunks < sm_count ? total_chunks : sm_count;
    if (v.n_sub > MAX_SEGMENTS) v.n_sub = MAX_SEGMENTS;
    v.n_long = v.total_chunks % v.n_sub;
    v.inv_long = v.n_long > 0 ? 1.0f / (float)v.n_long : 0.f;
    v.inv_short = 1.0f / (float)(v.n_sub - v.n_long);
    v.per_sub = v.total_chunks / v.n_sub;
    v.inv_sub = 1.0f / (float)v.n_sub;
    if (v.n_sub < v.splits) v.splits = v.n_sub;
    // as many blocks as there are segments in each, so that the two chains of merges together are shortest
    int per_group = 1;
    while (v.splits * per_group * v.splits * per_group < v.n_sub) ++per_group;
    v.n_mid = v.splits * per_group < v.n_sub ? v.splits * per_group : v.n_sub;        // <= MAX_SPLITS
    for (int i = 0; i <= v.n_mid; ++i) v.mid_begin[i] = (uint8_t)(i * v.n_sub / v.n_mid);
    for (int g = 0; g <= v.splits; ++g) v.group_begin[g] = (uint8_t)(g * v.n_mid / v.splits);
    return v;
}

// The combining kernel: `group` tokens of the tail per block, whose records (16 bytes each) lie in the block's shared memory: a token's
// segments, and its blocks of segments where they are fewer.
constexpr size_t SM_SMEM = 228 * 1024, BLOCK_SMEM_RESERVED = 1024;      // of an SM; what the system takes of it for every block
constexpr int COMBINE_GROUP = 32, COMBINE_BLOCKS = 4;      // most tokens per block; blocks per SM
constexpr size_t COMBINE_SMEM = 32 * 1024;
inline size_t combine_bytes(const VocabPlan& v, int halves) { return (size_t)(v.n_sub + (v.n_mid < v.n_sub ? v.n_mid : 0)) * halves * 16; }
// As many as give every SM a block, within the room.  While there are no more blocks than four an SM, which fit at once, that is the room
// beside a block of the log-prob kernel (with `beside` bytes), where the first of them wait while that one runs; beyond that fewer blocks
// are worth more.  Rooms of 31,744 / 32,768 bytes, d = 256, V = 33,280 (six and seven tokens): 1,000 tokens 25.6 / 26.0 us, 1,300 30.2 /
// 30.6, 2,000 39.9 / 40.3, 3,000 53.8 / 54.0; past the line 3,990 70.5 / 68.4, 9,000 149.4 / 146.4.
inline int combine_group(const VocabPlan& v, int halves, int64_t tail_rows, int sm_count, size_t beside) {
    const int64_t room_beside = (int64_t)((SM_SMEM - beside - 2 * BLOCK_SMEM_RESERVED) / combine_bytes(v, halves));
    const int64_t room = (int64_t)(COMBINE_SMEM / combine_bytes(v, halves));
    int64_t group = (tail_rows + sm_count - 1) / sm_count;
    if (group > COMBINE_GROUP) group = COMBINE_GROUP;
    if (group > room) group = room;
    return (int)(group > room_beside && tail_rows <= room_beside * COMBINE_BLOCKS * sm_count ? room_beside : group);
}
