// Online binned calibrator and the deployed stochastic pruning rule (Appendix A.4; Algorithm 1).
//
// State (one caller-provided device buffer): two first-in-first-out rings of bin indices (positive / negative
// rollouts), their histogram counts c_b^+ / c_b^-, the posterior table q_lut and the bias delta of the survival
// probability p_i = clip(kappa + delta + lambda (rho - q_i), p_min, p_max).
//
// arrol_calib_update (one block): pushes a step's labelled rollouts in index order (a full ring drops its oldest
// entry), keeps the counts in step with the rings, rebuilds q_lut with the Laplace-smoothed Bayes rule and solves
// delta by 64 bisection steps so that the expected keep rate under the buffer distribution equals kappa.  The
// table and delta are evaluated in fp64 with one rounding per operation, in a fixed order, so they are
// reproducible bit for bit.
// arrol_select_stochastic: survive iff u_i < p_i; rollouts that never reached the detection length are kept.
#include "arrol_internal.h"

namespace {

struct CalibHeader {
    int32_t B, pad;
    int64_t cap;
    int64_t head_pos, n_pos, head_neg, n_neg;
    double alpha;
    double delta;
};
static_assert(sizeof(CalibHeader) == 64, "state header layout");

struct CalibLayout {
    size_t cpos, cneg, q_lut, ring_pos, ring_neg, total;
};

CalibLayout layout_of(int B, int64_t cap) {
    CalibLayout L;
    size_t o = sizeof(CalibHeader);
    L.cpos = o; o += sizeof(int64_t) * (size_t)B;
    L.cneg = o; o += sizeof(int64_t) * (size_t)B;
    L.q_lut = o; o += sizeof(float) * (size_t)B;
    o = (o + 15) & ~(size_t)15;
    L.ring_pos = o; o += sizeof(int16_t) * (size_t)cap;
    o = (o + 15) & ~(size_t)15;
    L.ring_neg = o; o += sizeof(int16_t) * (size_t)cap;
    L.total = (o + 255) & ~(size_t)255;
    return L;
}

constexpr int CAL_THREADS = 1024;
constexpr int MAX_BINS = 1024;

__device__ __forceinline__ double survival_of(double q, double kappa_plus_delta, double lambda, double rho,
                                              double p_min, double p_max) {
    double p = __dadd_rn(kappa_plus_delta, __dmul_rn(lambda, __dsub_rn(rho, q)));
    if (p < p_min) p = p_min;
    if (p > p_max) p = p_max;
    return p;
}

__global__ void calib_init_kernel(uint8_t* state, int B, int64_t cap, double alpha, CalibLayout L) {
    CalibHeader* hd = reinterpret_cast<CalibHeader*>(state);
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        hd->B = B; hd->pad = 0; hd->cap = cap;
        hd->head_pos = hd->n_pos = hd->head_neg = hd->n_neg = 0;
        hd->alpha = alpha;
        hd->delta = 0.0;
    }
    int64_t* cpos = reinterpret_cast<int64_t*>(state + L.cpos);
    int64_t* cneg = reinterpret_cast<int64_t*>(state + L.cneg);
    float* lut = reinterpret_cast<float*>(state + L.q_lut);
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < B; b += gridDim.x * blockDim.x) {
        cpos[b] = 0; cneg[b] = 0; lut[b] = 0.5f;    // empty buffers: prior 1/2, flat likelihoods
    }
}

// One block, bound by latency: a handful of dependent round trips to memory and a serial search.  Every input is read once
// (the labelled bins are kept in shared memory up to CAL_STAGED rollouts), a thread owns a run of consecutive rollouts so
// that one block scan ranks all of them, and the bisection is settled in two or three rounds of 31 points (see below) instead of 64
// steps.  Per call, in a graph of 36 over changing states, mean of six (always three rounds, and a replay of all steps, before), lambda = 0.5:
// N = 2,048, 128 bins 15.7 -> 11.3 us; N = 32, 64 bins 12.9 -> 9.1; N = 8,192, 256 bins 23.5 -> 17.2.  lambda = 0.3, whose replay takes all
// steps: N = 2,048, 128 bins 16.6 -> 13.9; N = 64, 256 bins 19.1 -> 14.2; N = 4,000, 256 bins 20.8 -> 18.6.  Where bins meet the clip limits
// the root may lie next to a breakpoint, which more rounds follow: lambda = 1 to 1.3 0.65 to 1.19 of the former time by the state, 0.9 of the
// rounds in the mean of 48 states each.  More rollouts go through shared memory in pieces of CAL_STAGED,
// after a pass that counts the labels, so that global memory is read in whole lines (a thread's own run read from there
// touches a line per lane: N = 262,144 660 us a call by itself against 246 in pieces, 1,048,576 2,470 against 870; one rollout
// per thread and scan, as it was before the runs, 460 and 1,570).  An instance each, because the pieces' code in the same one cost
// small calls 0.3 us and 12,000 rollouts 1.5 (graph of 20 calls: 2,048 25.6 / 25.4 us, 12,000 37.4 / 36.0).
constexpr int CAL_STAGED = 8192;
constexpr int CAL_POINTS = 31;                 // points per round, one warp each
__host__ __device__ inline int product_pitch(int B) { return B | 1; }      // odd: 31 lanes walk 31 rows without bank conflicts
constexpr int CAL_PRODUCT_BINS = 704;          // most bins whose products are held in shared memory (31 x 705 x 8 = 175 KB)
template <bool ONE_PIECE>
__global__ void __launch_bounds__(CAL_THREADS)
calib_update_kernel(uint8_t* state, CalibLayout L, const int32_t* __restrict__ bin, const float* __restrict__ rewards,
                    const uint8_t* __restrict__ mask, int N, double kappa, double lambda, double rho, double p_min,
                    double p_max, int B_arg, int64_t cap_arg, uint32_t* d_status) {
    CalibHeader* hd = reinterpret_cast<CalibHeader*>(state);
    const int B = B_arg;
    const int64_t cap = cap_arg;
    __shared__ int16_t staged[CAL_STAGED];      // 2 bin + label of a rollout that is pushed, -1 of one that is not
    __shared__ int32_t warp_sum[2][32];
    __shared__ int32_t hist[2][MAX_BINS];       // signed change of the counts
    __shared__ double term[MAX_BINS];           // lambda (rho - q_b)
    __shared__ double weight[MAX_BINS];         // c_b^+ + c_b^-
    __shared__ double point_at[32], point_sum[32], point_slope[32];
    __shared__ double round_lo, round_hi, round_at, round_unit;
    __shared__ int round_kind;
    enum { DONE, EVEN, AROUND, ADJACENT, TREE };        // of a round's points, see below
    extern __shared__ double products[];        // [31][B rounded up to odd]: c_b p_b of a round's points
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;

    auto code_of = [&](int64_t i) {             // the three loads do not wait for one another
        const bool on = !mask || mask[i];
        int b = bin[i];
        const bool positive = rewards[i] > 0.5f;
        b = b < 0 ? 0 : (b >= B ? B - 1 : b);
        return on ? 2 * b + (positive ? 1 : 0) : -1;
    };
    auto stage = [&](int64_t from) {
        const int n = (int)min((int64_t)CAL_STAGED, N - from);
#pragma unroll 4
        for (int j = tid; j < n; j += CAL_THREADS) staged[j] = (int16_t)code_of(from + j);
        return n;
    };
    pdl_launch_dependents();
    pdl_wait();
    hd = pdl_acquire(hd); bin = pdl_acquire(bin); rewards = pdl_acquire(rewards); mask = pdl_acquire(mask); state = pdl_acquire(state);
    const int32_t state_B = hd->B;
    const int64_t state_cap = hd->cap;
    const int64_t head0[2] = {hd->head_neg, hd->head_pos}, n0[2] = {hd->n_neg, hd->n_pos};
    const double alpha = hd->alpha;
    if constexpr (ONE_PIECE) stage(0);
    // The byte layout L comes from the call's (B, cap); the state must have been initialised with the same pair.
    // A mismatched or uninitialised state is left untouched and reported (uniform over the block: no barrier yet).
    if (state_B != B || state_cap != cap) {
        if (tid == 0) atomicOr(d_status, ARROL_DEV_BAD_STATE);
        return;
    }
    int64_t* cnt[2] = {reinterpret_cast<int64_t*>(state + L.cneg), reinterpret_cast<int64_t*>(state + L.cpos)};
    int16_t* ring[2] = {reinterpret_cast<int16_t*>(state + L.ring_neg), reinterpret_cast<int16_t*>(state + L.ring_pos)};
    float* lut = reinterpret_cast<float*>(state + L.q_lut);
    int64_t old_cnt[2] = {0, 0};                // B <= MAX_BINS = CAL_THREADS: thread b owns bin b
    int16_t oldest[2];                          // this thread's first candidates for eviction, requested before it is known how many go
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        const int64_t at = head0[l] + tid;      // head0 < cap
        oldest[l] = tid < n0[l] ? ring[l][at < cap ? at : at - cap] : (int16_t)0;
    }
    if (tid < B) { old_cnt[0] = cnt[0][tid]; old_cnt[1] = cnt[1][tid]; hist[0][tid] = 0; hist[1][tid] = 0; }
    __syncthreads();

    // Sums over the block of two counts per thread (one barrier), and the sums of the threads before this one.
    auto block_scan = [&](const int32_t (&mine)[2], int64_t (&before)[2], int64_t (&total)[2]) {
        int32_t incl[2];
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            int32_t v = mine[l];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t t = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += t;
            }
            incl[l] = v;
            if (lane == 31) warp_sum[l][wid] = v;
        }
        __syncthreads();
#pragma unroll
        for (int l = 0; l < 2; ++l) {            // every warp scans the warp totals for itself
            int32_t v = warp_sum[l][lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t t = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += t;
            }
            total[l] = __shfl_sync(0xffffffffu, v, 31);
            const int32_t warps_before = __shfl_sync(0xffffffffu, v, wid > 0 ? wid - 1 : 0);
            before[l] = (wid > 0 ? warps_before : 0) + incl[l] - mine[l];
        }
    };
    // This thread's run [j0, j1) of the n staged entries, and the rank of its first one among those of its label.  Both labels'
    // counts in one word, 16 bits each: at most CAL_STAGED entries.
    static_assert(CAL_STAGED < 1 << 15, "two counts in one word");
    auto rank_run = [&](int n, int& j0, int& j1, int64_t (&first_rank)[2], int64_t (&total)[2]) {
        const int per = (n + CAL_THREADS - 1) / CAL_THREADS;
        j0 = min(n, tid * per);
        j1 = min(n, j0 + per);
        int32_t mine = 0;
        for (int j = j0; j < j1; ++j) {
            const int c = staged[j];
            mine += c < 0 ? 0 : (c & 1) ? 1 << 16 : 1;
        }
        int32_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) warp_sum[0][wid] = incl;
        __syncthreads();
        int32_t v = warp_sum[0][lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t t = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += t;
        }
        const int32_t all = __shfl_sync(0xffffffffu, v, 31), warps_before = __shfl_sync(0xffffffffu, v, wid > 0 ? wid - 1 : 0);
        const int32_t before = (wid > 0 ? warps_before : 0) + incl - mine;
        first_rank[0] = before & 0xffff; first_rank[1] = before >> 16;
        total[0] = all & 0xffff; total[1] = all >> 16;
    };
    int j0 = 0, j1 = 0;
    int64_t total_new[2], first_rank[2];
    if constexpr (ONE_PIECE) {
        rank_run(N, j0, j1, first_rank, total_new);
    } else {                                     // how many there are of each label decides what is evicted and what stays
        int32_t mine[2] = {0, 0};
#pragma unroll 8
        for (int64_t i = tid; i < N; i += CAL_THREADS) {
            const bool on = !mask || mask[i], pos = rewards[i] > 0.5f;
            mine[0] += on && !pos ? 1 : 0;
            mine[1] += on && pos ? 1 : 0;
        }
        block_scan(mine, first_rank, total_new);
    }

    // evict the oldest entries that the push displaces (read the rings before they are overwritten)
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        const int64_t over = n0[l] + total_new[l] - cap;
        const int64_t evict = over <= 0 ? 0 : (over < n0[l] ? over : n0[l]);
        for (int64_t j = tid; j < evict; j += CAL_THREADS) {
            const int64_t at = head0[l] + j;     // head0, j < cap
            atomicSub(&hist[l][j == tid ? oldest[l] : ring[l][at < cap ? at : at - cap]], 1);
        }
    }
    __syncthreads();

    // entry r of m lands in slot (head + n + r) mod cap, and only the last `cap` of them survive the call
    {
        int64_t slot0[2] = {head0[0] + n0[0], head0[1] + n0[1]};         // below 2 cap
#pragma unroll
        for (int l = 0; l < 2; ++l) slot0[l] -= slot0[l] >= cap ? cap : 0;
        auto write_run = [&](const int64_t (&before)[2]) {
            int64_t r[2] = {before[0] + first_rank[0], before[1] + first_rank[1]};
            for (int j = j0; j < j1; ++j) {
                const int c = staged[j];
                if (c < 0) continue;
                const int l = c & 1;
                const int64_t rank = l ? r[1]++ : r[0]++;
                if (rank >= (l ? total_new[1] : total_new[0]) - cap) {
                    const int64_t at = (l ? slot0[1] : slot0[0]) + (rank < cap ? rank : rank % cap);
                    (l ? ring[1] : ring[0])[at < cap ? at : at - cap] = (int16_t)(c >> 1);
                    atomicAdd(&hist[l][c >> 1], 1);
                }
            }
        };
        int64_t before[2] = {0, 0};
        if constexpr (ONE_PIECE) write_run(before);
        else
            for (int64_t from = 0; from < N; from += CAL_STAGED) {
                int64_t here[2];
                const int n = stage(from);
                __syncthreads();
                rank_run(n, j0, j1, first_rank, here);
                write_run(before);
                before[0] += here[0];
                before[1] += here[1];
                __syncthreads();                 // the staged entries and the warp sums are overwritten by the next piece
            }
    }
    __syncthreads();

    // ring bookkeeping; every thread keeps the new sizes
    int64_t n1[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        const int64_t over = n0[l] + total_new[l] - cap;
        n1[l] = over > 0 ? cap : n0[l] + total_new[l];
        if (tid == CAL_THREADS - 1 - l) {        // a warp without a bin to work on, most often
            const int64_t h1 = over > 0 ? (head0[l] + over) % cap : head0[l];
            if (l == 0) { hd->head_neg = h1; hd->n_neg = n1[l]; } else { hd->head_pos = h1; hd->n_pos = n1[l]; }
        }
    }

    // posterior table (Laplace-smoothed likelihoods, Bayes rule), fp64, one rounding per operation
    const double n_pos = (double)n1[1], n_neg = (double)n1[0];
    const double n = __dadd_rn(n_pos, n_neg);
    if (tid < B) {
        const double prior = n > 0.0 ? __ddiv_rn(n_pos, n) : 0.5;
        const double den_pos = __dadd_rn(n_pos, __dmul_rn(alpha, (double)B));
        const double den_neg = __dadd_rn(n_neg, __dmul_rn(alpha, (double)B));
        const int64_t c_neg = old_cnt[0] + hist[0][tid], c_pos = old_cnt[1] + hist[1][tid];
        cnt[0][tid] = c_neg;
        cnt[1][tid] = c_pos;
        const double p1 = __ddiv_rn(__dadd_rn((double)c_pos, alpha), den_pos);
        const double p0 = __ddiv_rn(__dadd_rn((double)c_neg, alpha), den_neg);
        const double num = __dmul_rn(prior, p1);
        const double den = __dadd_rn(num, __dmul_rn(__dsub_rn(1.0, prior), p0));
        const float qb = (float)__ddiv_rn(num, den);
        lut[tid] = qb;
        term[tid] = __dmul_rn(lambda, __dsub_rn(rho, (double)qb));
        weight[tid] = (double)(c_neg + c_pos);
    }
    __syncthreads();

    // delta: 64 bisection steps on E[p](delta) = kappa.  The value that decides a step is the expected keep rate summed over
    // the bins in index order, one rounding per operation (so that delta agrees bit for bit with a plain loop).
    //   Rounded addition, multiplication, clamping and division are all monotone, so the decision "below" is a monotone
    // function of the midpoint x, bit for bit, and one of kappa + x (rounded), through which alone x enters: one evaluation at x
    // settles every midpoint whose kappa + x lies on its side.  So the block evaluates 31 points a round (one warp each, in
    // ascending order), whatever they are, and at the end the first warp replays the bisection against the two settled points next to
    // the threshold.  E is piecewise linear, and its root needs few rounds:
    //   EVEN      points evenly over the bracket: after it the piece that the root lies on is known
    //   AROUND    the root of that piece, with the sum as a butterfly gives it: 17 neighbouring values of kappa + x, then points at
    //             growing distances.  The sum in index order is a few roundings from the butterfly's, so that the threshold lies
    //             among the neighbours most often, and nothing is left to settle
    //   ADJACENT  where it does not: 31 neighbours around the root that the sum in index order at the best point gives
    // and, where that does not settle all (breakpoints next to the root, or no slope), the 31 midpoints of the replay's next five levels
    // (TREE) until it does: a round of those settles a step at least, so 64 of them are always enough.
    // (Before, midpoints only, but for one round around the linear root: six rounds where three do now, with two replays between.)
    //   One evaluation: the lanes form the per-bin products c_b p_b (all >= 0) and a butterfly sum S of them; the in-order sum
    // differs from S by at most (B + 8) 2^-53 S (both are within their standard error bounds of the exact sum), so when S is
    // further from kappa n than four times that bound plus the roundings of the division and of kappa n, S < kappa n already
    // is the decision.  Points closer than that need the serial chain of B additions: the first warp runs the chains of all
    // 31 points side by side, one per lane (an addition takes about 30 cycles, and chains in 31 warps would queue for the fp64
    // pipe).
    double delta = 0.0;
    if (n > 0.0) {                                   // uniform for the block
        const double u = 1.1102230246251565e-16;     // 2^-53
        const double goal = kappa * n;
        const double inf = __longlong_as_double(0x7ff0000000000000ll);
        const int pitch = product_pitch(B);
        auto midpoint = [](double a, double b) { return __dmul_rn(0.5, __dadd_rn(a, b)); };
        auto clipped = [&](double p) {
            if (p < p_min) p = p_min;
            if (p > p_max) p = p_max;
            return p;
        };
        // the first warp's: the bracket of the replay, the settled points next to the threshold, S and dS/d(delta) at the lower one
        double lo = -(1.0 + lambda), hi = 1.0 + lambda;
        const double first_lo = lo, first_hi = hi;
        double known_below = -inf, known_above = inf;
        double sum_at = 0.0, slope_at = 0.0;
        bool sum_in_order = false;
        // infinite lambda: the first midpoint is NaN, no comparison holds, and a plain loop ends at NaN.  (A finite bracket
        // never gets there: its midpoints can overflow, but not with opposite signs.)
        int step = isinf(lambda) ? 64 : 0;
        if (step) hi = midpoint(lo, hi);
        for (int round = 0; round <= 3 + 64; ++round) {
            if (wid == 0) {
                int kind = TREE;
                double a = fmax(known_below, first_lo), b = fmin(known_above, first_hi), at = 0.0, unit = 0.0;
                if (step >= 64) {
                    kind = DONE;
                } else if (round < 3 && !(__dadd_rn(kappa, known_above) <= nextafter(__dadd_rn(kappa, known_below), inf) ||
                                          known_above <= nextafter(known_below, inf))) {
                    kind = EVEN;
                    if (round > 0 && known_below > -inf && slope_at > 0.0) {
                        // kappa + at without rounding: neighbours taken from halfway between two values would round to every other one
                        at = fmin(fmax(known_below + (goal - sum_at) / slope_at, a), b);
                        at = __dsub_rn(__dadd_rn(kappa, at), kappa);
                        kind = round == 2 && sum_in_order ? ADJACENT : AROUND;
                        unit = scalbn(1.0, ilogb(fmax(fmax(fabs(kappa + at), fabs(at)), 1e-200)) - 52);
                    }
                } else {                             // replay as far as the settled points reach
                    const double base_below = __dadd_rn(kappa, known_below), base_above = __dadd_rn(kappa, known_above);
                    // The first midpoints are whole multiples of (1 + lambda) 2^-j, without rounding while their bits last: after j steps the bracket
                    // is the cell of that grid that holds the threshold, found at once where 1 + lambda has few bits (51 steps of
                    // lambda = 0.5; none of 0.3, whose midpoints are rounded from the third one on; none past 2^1023, where lo + hi can overflow).
                    const int used = 53 - min(52, __ffsll(__double_as_longlong(first_hi) | (1ll << 52)) - 1);      // bits of 1 + lambda
                    if (step == 0 && used < 44 && first_hi <= 0x1p1023 && known_below > first_lo && known_above < first_hi) {
                        const int jump = 53 - used;
                        const double cells = __longlong_as_double((long long)(1023 + jump) << 52), unit_cell = __longlong_as_double((long long)(1023 - jump) << 52);
                        const double at = floor((known_below / first_hi + 1.0) * 0.5 * cells);
#pragma unroll 1
                        for (int k = -1; k <= 1 && step == 0; ++k) {         // one of these three, or none
                            const double below_k = (2.0 * (at + k) - cells) * unit_cell * first_hi, above_k = (2.0 * (at + k + 1.0) - cells) * unit_cell * first_hi;
                            if (at + k >= 0.0 && at + k + 1.0 <= cells && (at + k == 0.0 || __dadd_rn(kappa, below_k) <= base_below) &&
                                (at + k + 1.0 == cells || __dadd_rn(kappa, above_k) >= base_above)) {
                                lo = below_k;
                                hi = above_k;
                                step = jump;
                            }
                        }
                    }
                    double m = midpoint(lo, hi);
                    while (step < 64) {              // both next midpoints while the comparison is under way
                        const double base = __dadd_rn(kappa, m), m_up = midpoint(m, hi), m_down = midpoint(lo, m);
                        const bool below = base <= base_below;
                        if (!(below || base >= base_above)) break;
                        const bool unchanged = below ? m == lo : m == hi;                          // then it stays unchanged
                        lo = below ? m : lo;
                        hi = below ? hi : m;
                        m = below ? m_up : m_down;
                        step = unchanged ? 64 : step + 1;
                    }
                    if (step >= 64) kind = DONE;
                    a = lo;
                    b = hi;
                }
                if (lane == 0) { round_kind = kind; round_lo = a; round_hi = b; round_at = at; round_unit = unit; }
            }
            __syncthreads();
            const int kind = round_kind;
            if (kind == DONE) break;
            // this warp's point, in ascending order
            double x = 0.0;
            const int i = wid - 15;                  // -15 .. 15
            if (kind == EVEN) {
                const double t = (double)(wid + 1) * 0.03125;
                x = (1.0 - t) * round_lo + t * round_hi;
            } else if (kind == AROUND && (i < -8 || i > 8)) {
                const int k = i < 0 ? -i : i;        // unit <= (1 + lambda + kappa) 2^-52: past the eighth neighbour
                const double off = scalbn(1.0 + lambda + fabs(kappa), k == 9 ? -46 : k == 10 ? -43 : k == 11 ? -40 : k == 12 ? -35 : k == 13 ? -28 : k == 14 ? -19 : -10);
                x = i < 0 ? round_at - off : round_at + off;
            } else if (kind == ADJACENT || kind == AROUND) {
                x = round_at + (double)i * round_unit;
            } else {                                 // in-order traversal of the tree of the next five levels' midpoints
                double a = round_lo, b = round_hi;
                const int want = wid < CAL_POINTS ? wid + 1 : 1;
                x = midpoint(a, b);
                for (int node = 16, half = 8; node != want; half >>= 1) {
                    if (want > node) { a = x; node += half; } else { b = x; node -= half; }
                    x = midpoint(a, b);
                }
            }
            if (wid < CAL_POINTS) {
                const double base = __dadd_rn(kappa, x);
                double part = 0.0, slope = 0.0;
#pragma unroll 4
                for (int k = lane; k < B; k += 32) {
                    const double raw = __dadd_rn(base, term[k]), p = clipped(raw);
                    const double v = __dmul_rn(weight[k], p);
                    if (B <= CAL_PRODUCT_BINS) products[wid * pitch + k] = v;
                    part += v;
                    if (p == raw) slope += weight[k];
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    part += __shfl_xor_sync(0xffffffffu, part, o);
                    slope += __shfl_xor_sync(0xffffffffu, slope, o);
                }
                if (lane == 0) { point_sum[wid] = part; point_slope[wid] = slope; }
                if (lane == 1) point_at[wid] = x;
            }
            __syncthreads();
            if (wid == 0) {
                const bool has = lane < CAL_POINTS;
                const double S = has ? point_sum[lane] : 0.0;
                const double slack = 4.0 * ((double)(B + 8) * u * S + 3.0 * u * (S + goal));
                const bool near = has && fabs(S - goal) <= slack;
                bool below = S < goal;
                double e = S;
                if (__any_sync(0xffffffffu, near)) {
                    e = 0.0;
                    if (B <= CAL_PRODUCT_BINS) {
                        const double* row = products + (has ? lane : 0) * pitch;
#pragma unroll 8
                        for (int k = 0; k < B; ++k) e = __dadd_rn(e, row[k]);
                    } else {
                        const double base = __dadd_rn(kappa, has ? point_at[lane] : 0.0);
#pragma unroll 4
                        for (int k = 0; k < B; ++k) e = __dadd_rn(e, __dmul_rn(weight[k], clipped(__dadd_rn(base, term[k]))));
                    }
                    if (near) below = __ddiv_rn(e, n) < kappa;
                    if (has) point_sum[lane] = e;
                    __syncwarp();
                }
                // ascending points: the ones below come first
                const int count = __popc(__ballot_sync(0xffffffffu, has && below));
                if (count > 0 && point_at[count - 1] > known_below) {
                    known_below = point_at[count - 1];
                    sum_at = point_sum[count - 1];
                    slope_at = point_slope[count - 1];
                    sum_in_order = __any_sync(0xffffffffu, near);
                }
                if (count < CAL_POINTS) known_above = fmin(known_above, point_at[count]);
            }
        }
        delta = midpoint(lo, hi);                    // meaningful in the first warp
    }
    if (tid == 0) hd->delta = delta;
}

__global__ void select_stochastic_kernel(const float* __restrict__ q, const float* __restrict__ u,
                                         const uint8_t* __restrict__ eligible, int64_t N, double kappa,
                                         const double* __restrict__ d_delta, double delta_value, double lambda,
                                         double rho, double p_min, double p_max, uint8_t* __restrict__ keep,
                                         float* __restrict__ p_out) {
    pdl_launch_dependents();
    pdl_wait();
    q = pdl_acquire(q); u = pdl_acquire(u); eligible = pdl_acquire(eligible); d_delta = pdl_acquire(d_delta);
    const double delta = d_delta ? *d_delta : delta_value;
    const double base = __dadd_rn(kappa, delta);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) {
        if (eligible && !eligible[i]) {
            keep[i] = 1;
            if (p_out) p_out[i] = 1.0f;
            continue;
        }
        const double p = survival_of((double)q[i], base, lambda, rho, p_min, p_max);
        keep[i] = ((double)u[i] < p) ? 1 : 0;
        if (p_out) p_out[i] = (float)p;
    }
}

bool survival_ok(const arrol_survival* sp) {
    return sp && sp->kappa >= 0.0 && sp->kappa <= 1.0 && sp->lambda >= 0.0 && sp->rho >= 0.0 && sp->rho <= 1.0 &&
           sp->p_min >= 0.0 && sp->p_max <= 1.0 && sp->p_min <= sp->p_max;
}

}  // namespace

extern "C" size_t arrol_calib_state_bytes(int32_t B, int64_t cap) {
    if (B <= 0 || B > MAX_BINS || cap <= 0) return 0;
    return layout_of(B, cap).total;
}

extern "C" int arrol_calib_layout(int32_t B, int64_t cap, size_t* offsets6) {
    if (B <= 0 || B > MAX_BINS || cap <= 0 || !offsets6) return ARROL_ERR_INVALID_ARG;
    const CalibLayout L = layout_of(B, cap);
    offsets6[0] = L.cpos; offsets6[1] = L.cneg; offsets6[2] = L.q_lut; offsets6[3] = L.ring_pos;
    offsets6[4] = L.ring_neg; offsets6[5] = L.total;
    return ARROL_OK;
}

extern "C" int arrol_calib_init(arrol_ctx* ctx, void* state, size_t state_bytes, int32_t B, int64_t cap, double alpha,
                                void* stream) {
    if (!ctx || !state || !(alpha >= 0.0)) return ARROL_ERR_INVALID_ARG;
    if (B <= 0 || cap <= 0) return ARROL_ERR_INVALID_ARG;
    if (B > MAX_BINS) return ARROL_ERR_UNSUPPORTED;
    const CalibLayout L = layout_of(B, cap);
    if (state_bytes < L.total || !arrol_aligned(state, 16)) return ARROL_ERR_WORKSPACE;
    ArrolDeviceGuard guard(ctx->device);
    if (!guard.ok) return ARROL_ERR_CUDA;
    calib_init_kernel<<<1, 256, 0, (cudaStream_t)stream>>>(static_cast<uint8_t*>(state), B, cap, alpha, L);
    ctx->launches += 1;
    ARROL_CUDA_OK(cudaGetLastError());
    return ARROL_OK;
}

extern "C" const float* arrol_calib_q_lut(void* state, int32_t B, int64_t cap) {
    if (!state || B <= 0 || B > MAX_BINS || cap <= 0) return nullptr;
    return reinterpret_cast<const float*>(static_cast<uint8_t*>(state) + layout_of(B, cap).q_lut);
}

extern "C" const double* arrol_calib_delta(void* state) {
    if (!state) return nullptr;
    return &reinterpret_cast<CalibHeader*>(state)->delta;
}

extern "C" int arrol_calib_update(arrol_ctx* ctx, void* state, int32_t B, int64_t cap, const int32_t* bin,
                                  const float* rewards, const uint8_t* mask, int32_t N, const arrol_survival* sp,
                                  void* stream) {
    if (!ctx || !state || N < 0 || !survival_ok(sp)) return ARROL_ERR_INVALID_ARG;
    if (B <= 0 || cap <= 0) return ARROL_ERR_INVALID_ARG;
    if (B > MAX_BINS) return ARROL_ERR_UNSUPPORTED;
    if (N > 0 && (!bin || !rewards)) return ARROL_ERR_INVALID_ARG;
    ArrolDeviceGuard guard(ctx->device);
    if (!guard.ok) return ARROL_ERR_CUDA;
    const auto one_piece = calib_update_kernel<true>, pieces = calib_update_kernel<false>;
    if (!ctx->calib_smem_set) {
        const int most = (int)(sizeof(double) * CAL_POINTS * product_pitch(CAL_PRODUCT_BINS));
        ARROL_CUDA_OK(cudaFuncSetAttribute(one_piece, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        ARROL_CUDA_OK(cudaFuncSetAttribute(pieces, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        ctx->calib_smem_set = true;
    }
    const size_t smem = B <= CAL_PRODUCT_BINS ? sizeof(double) * CAL_POINTS * product_pitch(B) : 0;
    ARROL_CUDA_OK(arrol_launch_pdl(N <= CAL_STAGED ? one_piece : pieces, dim3(1), dim3(CAL_THREADS), smem, (cudaStream_t)stream,
                                   static_cast<uint8_t*>(state), layout_of(B, cap), bin, rewards, mask, N, sp->kappa, sp->lambda,
                                   sp->rho, sp->p_min, sp->p_max, B, cap, ctx->d_status));
    ctx->launches += 1;
    return ARROL_OK;
}

extern "C" int arrol_select_stochastic(arrol_ctx* ctx, const float* q, const float* u, const uint8_t* eligible,
                                       int64_t N, const arrol_survival* sp, const double* d_delta, double delta,
                                       uint8_t* keep, float* p_out, void* stream) {
    if (!ctx || N < 0 || !survival_ok(sp)) return ARROL_ERR_INVALID_ARG;
    if (N == 0) return ARROL_OK;
    if (!q || !u || !keep) return ARROL_ERR_INVALID_ARG;
    ArrolDeviceGuard guard(ctx->device);
    if (!guard.ok) return ARROL_ERR_CUDA;
    int64_t blocks = (N + 255) / 256;
    if (blocks > (int64_t)ctx->sm_count * 8) blocks = (int64_t)ctx->sm_count * 8;
    ARROL_CUDA_OK(arrol_launch_pdl(select_stochastic_kernel, dim3((unsigned)blocks), dim3(256), 0, (cudaStream_t)stream, q, u, eligible,
                                   N, sp->kappa, d_delta, delta, sp->lambda, sp->rho, sp->p_min, sp->p_max, keep, p_out));
    ctx->launches += 1;
    return ARROL_OK;
}
