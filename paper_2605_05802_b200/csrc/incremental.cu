// Incremental gate: one new action per rollout per environment step, gate
// re-evaluated after every step (the paper gates at one fixed K, Appendix C.1; a
// per-step evaluation is what its "adaptive K" follow-up needs, Section 5).
//
// Per pair (i, j), i < j, with current lengths m = len_i (rows) and n = len_j
// (columns) of the edit-distance matrix D, the state keeps
//   VP / VN : bit r-1 set iff D[r][n] - D[r-1][n] is +1 / -1   (last column)
//   HP / HN : bit c-1 set iff D[m][c] - D[m][c-1] is +1 / -1   (last row)
// and D[m][n] = n + popc(VP) - popc(VN) is never stored.  When j appends y, one
// bit-parallel column step over the rows gives the new last column, and the
// horizontal delta of the bottom row is appended to the last row; when i appends x, the
// same step on the transposed roles gives the new last row, and the vertical delta that leaves
// it is appended to the last column.  When both append, the row comes first, so that the
// column step already runs over m + 1 rows and its last cell is the new corner.
//
// State buffer layout (position independent, byte-copyable):
//   [0, 256)        header: magic, n_groups, N, max_steps, steps taken so far (an upper
//                   bound of every rollout's length, known without reading the lengths)
//   lens   int32 [n_groups][N]
//   hist   int32 [n_groups][8][N][4]      actions emitted so far: action r of rollout i
//                                         sits at [r / 4][i][r % 4], so that the first
//                                         quads of all rollouts of a group (what a step
//                                         reads) are contiguous
//   pairs  uint4 [n_groups][P]            (VP, VN, HP, HN)
// every section starts on a 256-byte boundary.
#include "common.cuh"

namespace sr {

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

namespace {

constexpr uint32_t kMagic = 0x53524731u;   // "SRG1"
constexpr int kHistPitch = 32;
constexpr int kRollThreads = 128;

struct IncrLayout {
    size_t off_lens, off_hist, off_pairs, total;
};

IncrLayout incr_layout(int32_t n_groups, int32_t N) {
    IncrLayout L;
    size_t off = 256;
    L.off_lens = off;
    off = align_up(off + (size_t)n_groups * N * 4, 256);
    L.off_hist = off;
    off = align_up(off + (size_t)n_groups * N * kHistPitch * 4, 256);
    L.off_pairs = off;
    off = align_up(off + (size_t)n_groups * pairs_of(N) * 16, 256);
    L.total = off;
    return L;
}

__global__ void incr_init_kernel(unsigned char* state, IncrLayout L, int n_groups, int N,
                                 int max_steps) {
    grid_begin();
    const size_t tid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t nthr = (size_t)gridDim.x * blockDim.x;
    uint32_t* hdr = reinterpret_cast<uint32_t*>(state);
    if (tid < 64) {
        uint32_t v = 0;
        if (tid == 0) v = kMagic;
        if (tid == 1) v = (uint32_t)n_groups;
        if (tid == 2) v = (uint32_t)N;
        if (tid == 3) v = (uint32_t)max_steps;
        hdr[tid] = v;
    }
    // lengths and pair state start at zero; the history needs no clearing (only the
    // first len entries of a row are ever read)
    uint32_t* lens = reinterpret_cast<uint32_t*>(state + L.off_lens);
    for (size_t e = tid; e < (size_t)n_groups * N; e += nthr) lens[e] = 0u;
    uint4* pairs = reinterpret_cast<uint4*>(state + L.off_pairs);
    for (size_t e = tid; e < (size_t)n_groups * pairs_of(N); e += nthr)
        pairs[e] = make_uint4(0u, 0u, 0u, 0u);
}

// The bit-parallel column step on the last column (P, M) of `len` cells, whose match bits are `Eq`
// (bits at or above len are harmless: carries and shifts only move upwards, and the result is
// masked with `below`, the bits under len); `last` is bit len - 1.  The delta that leaves the last
// cell (+1 where there is none) is appended to the crossing vector (cP, cM) as bit `at`.
__device__ __forceinline__ void append_step(uint32_t Eq, uint32_t& P, uint32_t& M, int len, uint32_t last,
                                            uint32_t below, uint32_t& cP, uint32_t& cM, uint32_t at) {
    uint32_t Ph, Mh;
    word_column(Eq, P, M, Ph, Mh);
    P &= below;
    M &= below;
    if ((Ph & last) != 0u || len == 0) cP |= at;
    if ((Mh & last) != 0u) cM |= at;
}

__device__ __forceinline__ uint32_t bit_of(int k) {     // 1 << k for 0 <= k < 32, otherwise 0
    uint32_t r;
    asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(k));
    return r;
}

struct IncrArgs {
    unsigned char* state;
    IncrLayout L;
    const int32_t* new_actions;
    int n_groups, N;
    double threshold;
    int norm_mode;
    int32_t* pair_dist;
    int32_t* pair_sum;
    double* mean;
    uint8_t* stop;
    int32_t* status;
    int gpb;                                               // groups per CTA
    uint32_t inv_P, inv_N;                                 // ceil(2^20 / P), ceil(2^20 / N): x / P by multiply-shift, exact while x (P - 1) < 2^20 (x: pairs of a CTA, at most 1984)
    int off_dist, off_term, off_roll, off_eq, off_state;              // shared-memory offsets
    uint32_t one;                                          // 1, as a run-time value
};

__device__ __forceinline__ int div20(int x, uint32_t inv) { return (int)(((uint32_t)x * inv) >> 20); }

// Match masks of a pair's two new actions against the stored actions of the other
// rollout: bit r of eq_y set iff action r of rollout ri equals y, bit c of eq_x set iff
// action c of rollout rj equals x, over the first 4 * kQuads positions.  Positions at or
// past a rollout's length hold whatever the buffer holds; the caller's column step
// ignores those bits (carries and shifts only move upwards, the result is masked).
// `quads` points at the group's stored actions ([8][N] int4): one 16-byte load and four
// compare / set-bit pairs per quad, both rows' loads issued before the comparisons.
template <int kQuads>
__device__ __forceinline__ void match_masks(const int4* quads, int N, int ri, int rj, int32_t y,
                                            int32_t x, uint32_t one, uint32_t& eq_y, uint32_t& eq_x) {
    int4 vi[kQuads], vj[kQuads];
#pragma unroll
    for (int q = 0; q < kQuads; ++q) { vi[q] = quads[q * N + ri]; vj[q] = quads[q * N + rj]; }
    eq_y = 0u;
    eq_x = 0u;
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
        // `one` holds 1 but is a run-time value: the bits are set by multiply-adds, which
        // issue on the FMA pipe while the comparisons keep the integer ALU busy
        asm("{ .reg .pred e0, e1, e2, e3;\n\t"
            "setp.eq.s32 e0, %1, %5; setp.eq.s32 e1, %2, %5; setp.eq.s32 e2, %3, %5; setp.eq.s32 e3, %4, %5;\n\t"
            "@e0 mad.lo.u32 %0, %10, %6, %0; @e1 mad.lo.u32 %0, %10, %7, %0;\n\t"
            "@e2 mad.lo.u32 %0, %10, %8, %0; @e3 mad.lo.u32 %0, %10, %9, %0; }"
            : "+r"(eq_y)
            : "r"(vi[q].x), "r"(vi[q].y), "r"(vi[q].z), "r"(vi[q].w), "r"(y),
              "r"(1u << (4 * q)), "r"(2u << (4 * q)), "r"(4u << (4 * q)), "r"(8u << (4 * q)), "r"(one));
        asm("{ .reg .pred e0, e1, e2, e3;\n\t"
            "setp.eq.s32 e0, %1, %5; setp.eq.s32 e1, %2, %5; setp.eq.s32 e2, %3, %5; setp.eq.s32 e3, %4, %5;\n\t"
            "@e0 mad.lo.u32 %0, %10, %6, %0; @e1 mad.lo.u32 %0, %10, %7, %0;\n\t"
            "@e2 mad.lo.u32 %0, %10, %8, %0; @e3 mad.lo.u32 %0, %10, %9, %0; }"
            : "+r"(eq_x)
            : "r"(vj[q].x), "r"(vj[q].y), "r"(vj[q].z), "r"(vj[q].w), "r"(x),
              "r"(1u << (4 * q)), "r"(2u << (4 * q)), "r"(4u << (4 * q)), "r"(8u << (4 * q)), "r"(one));
    }
}

// Appends to one pair (x by rollout i, y by rollout j, where ai / aj), stores its state and returns its
// distance; m and n become the new lengths.
__device__ __forceinline__ int step_pair(uint4 st, bool ai, bool aj, int32_t x, int32_t y, uint32_t eq_x, uint32_t eq_y,
                                         int& m, int& n, uint4* where) {
    const uint32_t bm = bit_of(m), bn = bit_of(n);         // 0 at 32: the rollout is full
    uint32_t last = bit_of(m - 1), below = bm - 1u;
    if (ai) {
        append_step(eq_x, st.z, st.w, n, bit_of(n - 1), bn - 1u, st.x, st.y, bm);
        eq_y &= below;                                     // the new row's match bit is x == y
        if (x == y) eq_y |= bm;
        last = bm;
        below = 2u * bm - 1u;
        ++m;
    }
    if (aj) {
        append_step(eq_y, st.x, st.y, m, last, below, st.z, st.w, bn);
        ++n;
    }
    if (ai || aj) *where = st;
    return n + __popc(st.x) - __popc(st.y);
}

// Small batches: one thread per pair, `gpb` groups per CTA.  The header (hot in L2: every CTA reads it)
// says how many steps the state has taken, which bounds every length; with that, all a
// pair needs -- its state, the two lengths, the two new actions AND the stored actions of
// both rollouts -- is requested in ONE round of independent loads instead of waiting for
// the lengths first (a second trip to DRAM per step made the kernel latency-bound).  The
// stored actions are read straight from the state: the pairs of a group share N rows, so
// all but the first touch of a row hit L1 (staging them in shared memory with asynchronous
// copies was measured slower).  The CTA synchronises twice, before the appends and before
// the per-group sums.
// kN: the group size when it is known at compile time (8, the paper's G: row offsets and
// the pair count fold into immediates), 0 for any other size.
template <int kN>
__global__ void __launch_bounds__(512, 3)
incr_step_kernel(IncrArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int N = kN ? kN : a.N, P = pairs_of(N);
    const int tid = threadIdx.x;
    const int grp = (int)(((uint32_t)tid * a.inv_P) >> 20);
    const int pr = kPairs.v[N][min(tid - grp * P, P - 1)];     // a table: no need to wait for it
    grid_begin();
    const int g0 = blockIdx.x * a.gpb;
    const int ng = min(a.gpb, a.n_groups - g0);
    int32_t* s_dist = reinterpret_cast<int32_t*>(smem + a.off_dist);    // [gpb][P]
    double* s_term = reinterpret_cast<double*>(smem + a.off_term);      // [gpb][P]

    const uint4 hdr = *reinterpret_cast<const uint4*>(a.state);         // magic, n_groups, N, max_steps
    const uint32_t steps_taken = reinterpret_cast<const uint32_t*>(a.state)[4];
    int32_t* g_len = reinterpret_cast<int32_t*>(a.state + a.L.off_lens) + (size_t)g0 * N;
    int32_t* g_hist = reinterpret_cast<int32_t*>(a.state + a.L.off_hist) + (size_t)g0 * N * kHistPitch;
    uint4* g_pairs = reinterpret_cast<uint4*>(a.state + a.L.off_pairs) + (size_t)g0 * P;
    const int32_t* g_new = a.new_actions + (size_t)g0 * N;

    const bool bad = hdr.x != kMagic || hdr.y != (uint32_t)a.n_groups || hdr.z != (uint32_t)N;
    if (bad) {                                     // uniform over the grid: nothing is touched
        if (tid == 0 && a.status) atomicOr(a.status, SR_STATUS_BAD_STATE);
        return;
    }
    const int max_steps = (int)hdr.w;
    // quads of stored actions any rollout can hold by now (the same for the whole grid, or
    // one more where a CTA already sees this step's own count: either is an upper bound)
    const int nq = (min((uint32_t)max_steps, steps_taken) + 3u) >> 2;

    if (blockIdx.x == 0 && tid == 0 && steps_taken < 0x7FFFFFFFu)
        reinterpret_cast<uint32_t*>(a.state)[4] = steps_taken + 1u;
    const bool is_pair = tid < ng * P;
    uint4 st = make_uint4(0u, 0u, 0u, 0u);
    int ri = 0, rj = 0, m = 0, n = 0;
    int32_t x = SR_NO_ACTION, y = SR_NO_ACTION;
    if (is_pair) {
        ri = pr & 0xFF;
        rj = pr >> 8;
        st = g_pairs[tid];
        const int gi = grp * N + ri, gj = grp * N + rj;
        m = g_len[gi];
        n = g_len[gj];
        x = __ldg(g_new + gi);
        y = __ldg(g_new + gj);
    }
    uint32_t eq_y = 0u, eq_x = 0u;                 // match masks of y in rollout ri, of x in rollout rj
    if (is_pair) {
        const int4* quads = reinterpret_cast<const int4*>(g_hist) + (size_t)grp * 8 * N;
        switch (nq) {
            case 0: break;
            case 1: match_masks<1>(quads, N, ri, rj, y, x, a.one, eq_y, eq_x); break;
            case 2: match_masks<2>(quads, N, ri, rj, y, x, a.one, eq_y, eq_x); break;
            case 3: match_masks<3>(quads, N, ri, rj, y, x, a.one, eq_y, eq_x); break;
            case 4: match_masks<4>(quads, N, ri, rj, y, x, a.one, eq_y, eq_x); break;
            case 5: match_masks<5>(quads, N, ri, rj, y, x, a.one, eq_y, eq_x); break;
            case 6: match_masks<6>(quads, N, ri, rj, y, x, a.one, eq_y, eq_x); break;
            case 7: match_masks<7>(quads, N, ri, rj, y, x, a.one, eq_y, eq_x); break;
            default: match_masks<8>(quads, N, ri, rj, y, x, a.one, eq_y, eq_x); break;
        }
    }
    // appenders: thread e < ng*N owns rollout e of this CTA
    const bool is_roll = tid < ng * N;
    int my_len = 0;
    int32_t my_act = SR_NO_ACTION;
    if (is_roll) { my_len = g_len[tid]; my_act = __ldg(g_new + tid); }
    if (m >= max_steps) x = SR_NO_ACTION;          // rollout already full: the action is ignored
    if (n >= max_steps) y = SR_NO_ACTION;
    if (is_roll && my_act != SR_NO_ACTION && my_len >= max_steps) {
        my_act = SR_NO_ACTION;
        if (a.status) atomicOr(a.status, SR_STATUS_STEP_OVERFLOW);
    }

    __syncthreads();       // every thread has read the lengths (and the stored actions) before the appends
    if (is_roll && my_act != SR_NO_ACTION) {
        const int g = (int)(((uint32_t)tid * a.inv_N) >> 20), i = tid - g * N;
        g_hist[(((size_t)g * 8 + (my_len >> 2)) * N + i) * 4 + (my_len & 3)] = my_act;
        g_len[tid] = my_len + 1;
    }
    if (is_pair) {
        const int d = step_pair(st, x != SR_NO_ACTION, y != SR_NO_ACTION, x, y, eq_x, eq_y, m, n, g_pairs + tid);
        if (a.pair_sum) s_dist[tid] = d;
        s_term[tid] = a.norm_mode == SR_NORM_NONE ? (double)d : kQuot.v[d * 33 + max(m, n)];
        if (a.pair_dist) a.pair_dist[(size_t)g0 * P + tid] = d;
    }
    __syncthreads();
    if (tid < ng) {
        GateArgs out{};
        out.pair_sum = a.pair_sum; out.mean = a.mean; out.stop = a.stop; out.threshold = a.threshold;
        group_sum_and_gate(s_term + tid * P, s_dist + tid * P, P, out, (size_t)g0 + tid);
    }
}

// Rollouts of pair e of a CTA, numbered within it, and how many places apart they are in their group.
__device__ __forceinline__ void pair_at(int e, int N, int P, int kN, uint32_t inv_P, int& gi, int& gj, int& apart) {
    const int g = kN ? e / P : div20(e, inv_P), pr = kPairs.v[N][e - g * P];
    gi = g * N + (pr & 0xFF);
    gj = g * N + (pr >> 8);
    apart = gj - gi;
}

// Large batches: one thread per rollout for the match masks, then one per pair for the steps, in a loop.
// A rollout's stored actions are read once, by one thread, and compared with the new actions
// of the group's other rollouts (kMasks at a time); the masks go to the pairs through shared memory.  A
// thread per pair that does its own comparing reads every stored action N - 1 times: the
// return path of L1 (16 bytes a lane and load) and the indices of its loads were half of that kernel.
// 30 steps, a thread per pair / per rollout: 65536 groups of 8 792 / 612 us, 16384 groups of 16 1033 / 721 us.
// (Registers decide: with one pair state in flight 656 us at 56 registers, 612 at 48, 665 at 40; with four
// 706 at 60, and 884 at 48, where it spills.)
// kN: as above.
template <int kN, int kMasks, bool kStaged>
__global__ void __launch_bounds__(kRollThreads, kN ? 9 : 8)
incr_rollout_kernel(IncrArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int N = kN ? kN : a.N, P = pairs_of(N), tid = threadIdx.x;
    double* s_term = reinterpret_cast<double*>(smem + a.off_term);      // [gpb][P]
    int32_t* s_dist = reinterpret_cast<int32_t*>(smem + a.off_dist);    // [gpb][P]
    int2* s_roll = reinterpret_cast<int2*>(smem + a.off_roll);          // [gpb * N] length before, action or none
    uint32_t* s_eq = reinterpret_cast<uint32_t*>(smem + a.off_eq);      // [gpb * N][N - 1]
    uint4* s_state = reinterpret_cast<uint4*>(smem + a.off_state);      // [gpb][P] pair states
    const int g = kN ? tid / N : div20(tid, a.inv_N), i = tid - g * N;
    // the thread's first pair: indices and a table, no need to wait for them
    int gi, gj, ahead;
    pair_at(tid, N, P, kN, a.inv_P, gi, gj, ahead);
    grid_begin();
    const int g0 = blockIdx.x * a.gpb;
    const int ng = min(a.gpb, a.n_groups - g0);
    const uint4 hdr = *reinterpret_cast<const uint4*>(a.state);         // magic, n_groups, N, max_steps
    const uint32_t steps_taken = reinterpret_cast<const uint32_t*>(a.state)[4];
    int32_t* g_len = reinterpret_cast<int32_t*>(a.state + a.L.off_lens) + (size_t)g0 * N;
    int32_t* g_hist = reinterpret_cast<int32_t*>(a.state + a.L.off_hist) + (size_t)g0 * N * kHistPitch;
    uint4* g_pairs = reinterpret_cast<uint4*>(a.state + a.L.off_pairs) + (size_t)g0 * P;
    const int32_t* g_new = a.new_actions + (size_t)g0 * N;

    const bool is_roll = tid < ng * N;
    int my_len = 0;
    int32_t my_act = SR_NO_ACTION;
    if (is_roll) { my_len = g_len[tid]; my_act = __ldg(g_new + tid); }
    // the first pair's state is on its way while the masks are made (kStaged: all of the thread's, without registers)
    uint4 st = make_uint4(0u, 0u, 0u, 0u);
    if constexpr (kStaged) {
        for (int e = tid; e < ng * P; e += kRollThreads) {
            const uint32_t to = (uint32_t)__cvta_generic_to_shared(s_state + e);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to), "l"(g_pairs + e) : "memory");
        }
    } else if (tid < ng * P) {
        st = g_pairs[tid];
    }
    const bool bad = hdr.x != kMagic || hdr.y != (uint32_t)a.n_groups || hdr.z != (uint32_t)N;
    if (bad) {                                     // uniform over the grid: nothing is touched
        if (tid == 0 && a.status) atomicOr(a.status, SR_STATUS_BAD_STATE);
        return;
    }
    const int max_steps = (int)hdr.w;
    // quads of stored actions any rollout can hold by now (or one more where a CTA already
    // sees this step's own count)
    const int nq = (min((uint32_t)max_steps, steps_taken) + 3u) >> 2;
    if (blockIdx.x == 0 && tid == 0 && steps_taken < 0x7FFFFFFFu)
        reinterpret_cast<uint32_t*>(a.state)[4] = steps_taken + 1u;

    if (is_roll) {
        if (my_act != SR_NO_ACTION && my_len >= max_steps) {
            my_act = SR_NO_ACTION;
            if (a.status) atomicOr(a.status, SR_STATUS_STEP_OVERFLOW);
        }
        s_roll[tid] = make_int2(my_len, my_act);
        const int4* quads = reinterpret_cast<const int4*>(g_hist) + g * 8 * N + i;
        uint32_t* eq_out = s_eq + tid * (N - 1);
        for (int d0 = 0; d0 < N - 1; d0 += kMasks) {           // rollouts i + 1 + d0 ... , cyclically
            int32_t y[kMasks];
            uint32_t eq[kMasks];
#pragma unroll
            for (int k = 0; k < kMasks; ++k) {
                int j = i + 1 + (kN ? k : min(d0 + k, N - 2));
                if (j >= N) j -= N;
                y[k] = __ldg(g_new + g * N + j);
                eq[k] = 0u;
            }
            uint32_t bit = a.one;
#pragma unroll 2
            for (int q = 0; q < nq; ++q) {
                const int4 v = quads[q * N];
                const uint32_t b1 = 2u * bit, b2 = 4u * bit, b3 = 8u * bit;
#pragma unroll
                for (int k = 0; k < kMasks; ++k)
                    // `one` holds 1 but is a run-time value: the bits are set by multiply-adds, which
                    // issue on the FMA pipe while the comparisons keep the integer ALU busy
                    asm("{ .reg .pred e0, e1, e2, e3;\n\t"
                        "setp.eq.s32 e0, %1, %5; setp.eq.s32 e1, %2, %5; setp.eq.s32 e2, %3, %5; setp.eq.s32 e3, %4, %5;\n\t"
                        "@e0 mad.lo.u32 %0, %10, %6, %0; @e1 mad.lo.u32 %0, %10, %7, %0;\n\t"
                        "@e2 mad.lo.u32 %0, %10, %8, %0; @e3 mad.lo.u32 %0, %10, %9, %0; }"
                        : "+r"(eq[k])
                        : "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(y[k]), "r"(bit), "r"(b1), "r"(b2), "r"(b3), "r"(a.one));
                bit = 16u * bit;
            }
#pragma unroll
            for (int k = 0; k < kMasks; ++k)
                if (kN || d0 + k < N - 1) eq_out[d0 + k] = eq[k];
        }
        // nobody else reads this rollout's stored actions or length
        if (my_act != SR_NO_ACTION) {
            g_hist[((g * 8 + (my_len >> 2)) * N + i) * 4 + (my_len & 3)] = my_act;
            g_len[tid] = my_len + 1;
        }
    }
    if constexpr (kStaged) asm volatile("cp.async.wait_all;" ::: "memory");       // each thread reads what it has copied itself
    __syncthreads();
    auto pair = [&](int e, uint4 state) {
        const int2 A = s_roll[gi], B = s_roll[gj];
        int m = A.x, n = B.x;
        const uint32_t eq_y = s_eq[gi * (N - 1) + ahead - 1], eq_x = s_eq[gj * (N - 1) + N - 1 - ahead];
        const int d = step_pair(state, A.y != SR_NO_ACTION, B.y != SR_NO_ACTION, A.y, B.y, eq_x, eq_y, m, n, g_pairs + e);
        if (a.pair_sum) s_dist[e] = d;
        s_term[e] = a.norm_mode == SR_NORM_NONE ? (double)d : kQuot.v[d * 33 + max(m, n)];
        if (a.pair_dist) a.pair_dist[(size_t)g0 * P + e] = d;
    };
    if (tid < ng * P) pair(tid, kStaged ? s_state[tid] : st);
#pragma unroll 2
    for (int e = tid + kRollThreads; e < ng * P; e += kRollThreads) {
        st = kStaged ? s_state[e] : g_pairs[e];
        pair_at(e, N, P, kN, a.inv_P, gi, gj, ahead);
        pair(e, st);
    }
    __syncthreads();
    if (tid < ng) {
        GateArgs out{};
        out.pair_sum = a.pair_sum; out.mean = a.mean; out.stop = a.stop; out.threshold = a.threshold;
        group_sum_and_gate(s_term + tid * P, s_dist + tid * P, P, out, (size_t)g0 + tid);
    }
}

// Steps follow one another.  A step whose CTAs become resident while the one before still runs crowds onto the
// SMs that have room: fine while an SM holds little of either, and again when the grid is more than one
// wave, but in between some SMs get two CTAs and others none.  The kernel with a thread per pair then overlaps on
// a stream, where that still pays, and not in a graph; the one with a thread per rollout, whose CTAs last
// longer, in neither up to 800 threads per SM.  30 steps, overlapping / ordinary in us: graph, 30000 groups of 2 (405
// threads per SM) 202 / 134, 33333 of 3 (676) 208 / 152, 3571 of 8 (687) 128 / 114, 1071 of 8 (206) 91 / 98, 8928 of 8
// (1716) 167 / 180; stream, 3571 of 8 136 / 168; thread per rollout, 2173 of 24 (352) 608 / 351 and 615 / 404,
// 8333 of 16 (900) 457 / 437 and 470 / 491.
int sm_count(int& sms) {
    int dev = 0;
    SR_CUDA_TRY(cudaGetDevice(&dev));
    SR_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    return SR_OK;
}

}  // namespace

size_t incr_state_bytes(int32_t n_groups, int32_t N, int32_t max_steps) {
    if (n_groups < 0 || N < 2 || N > SR_MAX_N || max_steps < 1 || max_steps > SR_MAX_INCR_STEPS)
        return 0;
    return incr_layout(n_groups, N).total;
}

int launch_incr_init(void* state, size_t bytes, int32_t n_groups, int32_t N, int32_t max_steps,
                     cudaStream_t s) {
    const IncrLayout L = incr_layout(n_groups, N);
    if (bytes < L.total) return SR_ERR_STATE_SIZE;
    size_t work = (size_t)n_groups * pairs_of(N);
    int blocks = (int)((work + 255) / 256);
    if (blocks < 1) blocks = 1;
    if (blocks > 4096) blocks = 4096;
    SR_LAUNCH("incr_init_kernel", incr_init_kernel, blocks, 256, 0, s, static_cast<unsigned char*>(state), L, n_groups, N, max_steps);
    return SR_OK;
}

int launch_incr_step(void* state, size_t bytes, const int32_t* new_actions, int32_t n_groups,
                     int32_t N, double threshold, int32_t norm_mode, int32_t* pair_dist,
                     int32_t* pair_sum, double* mean, uint8_t* stop, int32_t* status,
                     cudaStream_t s) {
    IncrArgs a;
    a.L = incr_layout(n_groups, N);
    if (bytes < a.L.total) return SR_ERR_STATE_SIZE;
    if (n_groups == 0) return SR_OK;
    a.state = static_cast<unsigned char*>(state);
    a.new_actions = new_actions;
    a.n_groups = n_groups; a.N = N;
    a.threshold = threshold; a.norm_mode = norm_mode;
    a.pair_dist = pair_dist; a.pair_sum = pair_sum; a.mean = mean; a.stop = stop; a.status = status;
    const int P = pairs_of(N);
    a.one = 1u;
    a.inv_P = ((1u << 20) + (uint32_t)P - 1u) / (uint32_t)P;
    a.inv_N = ((1u << 20) + (uint32_t)N - 1u) / (uint32_t)N;
    int off = 0;
    auto take = [&](int b) { int o = off; off = (off + b + 15) & ~15; return o; };
    // the thread-per-rollout form has the longer chain per thread and pays off once several CTAs of it
    // share every SM (N = 8: from 17000 groups on, 30 steps on 19600 275 and 250 us, on 14000 215 and 241; N = 16: from about 5000)
    if ((long long)n_groups * P >= (N == 8 ? 470000 : 550000)) {
        a.gpb = kRollThreads / N;
        a.off_dist = take(pair_sum ? a.gpb * P * 4 : 0);
        a.off_term = take(a.gpb * P * 8);
        a.off_roll = take(a.gpb * N * 8);
        a.off_eq = take(a.gpb * N * (N - 1) * 4);
        // Groups of 8 up to a little over two waves (nine CTAs an SM): the loads of one CTA's states are what the others of its SM wait for as well
        // (30 steps on 20000 groups 264 -> 249 us, 46000 449 -> 434, 65536 614 -> 617; 5000 of 16 370 -> 398).
        const bool staged = N == 8 && (long long)n_groups * P < 1300000;
        a.off_state = take(staged ? a.gpb * P * 16 : 0);
        auto kernel = N == 8 ? (staged ? incr_rollout_kernel<8, 7, true> : incr_rollout_kernel<8, 7, false>) : (N <= 5 ? incr_rollout_kernel<0, 4, false>
                                  : (N <= 8 ? incr_rollout_kernel<0, 7, false> : incr_rollout_kernel<0, 8, false>));
        const int blocks = (n_groups + a.gpb - 1) / a.gpb;
        int sms = 0;
        const int rc = sm_count(sms);
        if (rc != SR_OK) return rc;
        return launch_as((long long)blocks * kRollThreads > 800LL * sms, 1, "incr_rollout_kernel", kernel, blocks, kRollThreads, off, s, a);
    }
    int gpb = 256 / P;
    if (gpb < 1) gpb = 1;
    if (gpb > 32) gpb = 32;
    while (gpb > 1 && gpb * N > 256) --gpb;      // one appending thread per rollout
    a.gpb = gpb;
    a.off_dist = take(gpb * P * 4);
    a.off_term = take(gpb * P * 8);
    int threads = (gpb * P + 31) & ~31;
    if (threads < gpb * N) threads = (gpb * N + 31) & ~31;
    if (threads < 64) threads = 64;
    const int blocks = (n_groups + gpb - 1) / gpb;
    bool early = true;
    if (blocks > 64) {                           // 64 CTAs leave most SMs empty
        int sms = 0;
        const int rc = sm_count(sms);
        if (rc != SR_OK) return rc;
        const long long all = (long long)blocks * threads;
        early = all <= 384LL * sms || all > 1536LL * sms || !captured(s);
    }
    return launch_as(early, 1, "incr_step_kernel", N == 8 ? incr_step_kernel<8> : incr_step_kernel<0>, blocks, threads, off, s, a);
}

}  // namespace sr
