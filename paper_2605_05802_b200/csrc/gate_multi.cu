// Multi-word gate: prefixes of 33..SR_MAX_K symbols (token-level gate; same
// d_K of Section 3.2 of the paper, applied to token IDs).
//
// The edit-distance matrix of a pair is cut into 32-row blocks of the pattern; a
// block keeps its +1 / -1 vertical deltas in two 32-bit words and is advanced one
// text column at a time by the bit-vector recurrence, with the horizontal delta
// leaving a block entering the block below.  The work is organised as a pipeline
// of launches on the caller's stream, sharing a caller-provided workspace:
//
//   names    one CTA per group: gives every symbol a 16-bit name, the position of one of its
//            holders.
//   prep     one CTA per (group, pattern rollout): an array over the names holds the
//            pattern's positions, and every text paired with it is translated into a
//            "loc" stream: for text column c the position of the column's symbol in
//            the pattern (0x7FFF: absent).  A block's match word is then just
//            1 << (loc - first_row_of_block), no table lookup.  A symbol with several
//            occurrences gets a row of match words instead, and the stream names the row.
//            Bounds of the pair's distance fall out of the look-ups: the columns without any
//            match in the pattern from below, the differing positions from above.
//   bin      pairs with few matches get their distance from these alone, a warp each; the others
//            a team shape (what the band of their bounds costs at least, see
//            shape_of_pair) and bin counts.
//   order    counting sort of the pairs by bin: longest warp tasks first, one team
//            shape and similar durations per bin; warp-task table.  (One launch does both for
//            batches of up to a thousand pairs.)
//   dp       one CTA an SM; its warps are dealt their first tasks and pull the others.  A task is a warp of 32/T teams; a team of
//            T lanes owns one pair, a lane holding R <= 4 consecutive blocks (32*R rows) in
//            registers.  Lanes are skewed by four columns; the
//            delta bits of a lane's last block reach the next lane by warp shuffles.
//            All pairs of a task share (T, R) and have similar lengths, so the warp's
//            lanes stay busy.
//   finish   one thread per pair for the terms, one per group: ordered fp64 sum of the normalised
//            terms, threshold, outputs.
//
// A batch that leaves most of the GPU idle (runs_in_pairs) takes the names and one launch: prep keeps streams and rows in
// shared memory, the distances are computed right there, both ways from the ends of the text, and the
// last CTA of a group evaluates it (where there are even fewer, it names the symbols too, and the gate is one launch).
//
// Band.  With bounds lb <= d <= ub of a pair's distance an optimal alignment stays on a band of
// diagonals (band_of), and where the bounds meet nothing is left to compute.  Rollouts that have
// converged differ in few positions: their bands are narrow, and the T lanes of a team form a ring that
// follows the band down the pattern instead of covering all of it.  Cells outside the band are
// over-estimated at its edges, which leaves every cell on an optimal path exact (the banded block
// scheme of Sosic and Sikic 2017).  In decide mode the threshold caps how large a distance can
// still matter, and the pair's upper bound with it: a result within the bound is the exact
// distance, a result above it only says "more than the bound".
//
// Which rollout of a pair is the pattern is fixed by a round-robin tournament on the
// indices, so that every pattern CTA of `prep` serves the same number of texts.
#include <atomic>

#include <cooperative_groups.h>

#include "common.cuh"
#include "stream_words.cuh"

namespace sr {
namespace {

constexpr int kMostPrepThreads = 256;      // a thread for every four positions of a pattern
constexpr int kTextThreads = 16 * SR_MAX_N;  // a warp for every text of a pattern
constexpr int kTwoWarpThreads = 64;
static_assert(4 * kMostPrepThreads >= SR_MAX_K, "");
constexpr int kNumClasses = 21;     // team shapes (T lanes x R blocks), see class_of
constexpr int kTimeBuckets = 96;    // buckets of estimated task duration
constexpr float kLongTask = 2000.0f;  // tasks that last longer than it takes to see who is due for one, see multi_dp_kernel
constexpr int kNumBins = 2048;      // kTimeBuckets * kNumClasses of them used
constexpr int kOrderThreads = 1024;
constexpr int kAlonePairs = 1024;   // batches of up to this many pairs are ordered by one CTA
constexpr uint32_t kLocChain = 0xC000u;   // | first position of the symbol's occurrence chain
constexpr uint32_t kChainEnd = 0xFFFFu;
constexpr int kDpWarps = 12, kMostDpWarps = 16;   // of an SM, see multi_dp_kernel
constexpr uint32_t kBinMask = 0x7FFu;
constexpr uint32_t kListed = 0x800u;          // see multi_bin_kernel
constexpr uint32_t kHasChains = 0x40000000u;
constexpr int32_t kCappedFlag = 0x40000000;   // decide mode: the pair's distance exceeds its cap
constexpr int kStripShift = 12, kRowsShift = 22;
constexpr uint32_t kNeedsDp = 0x80000000u;
static_assert(kNumBins <= (int)kBinMask + 1 && kTimeBuckets * kNumClasses <= kNumBins, "bin index must fit its field");

struct PairDesc {          // 16 bytes
    uint32_t mn;           // m | n << 16
    uint32_t pat_row;      // g * patterns + pattern rollout
    uint32_t bin;          // bits 0..10 bin index; bit 11 listed for its few matches; bits 12..21 stripped common prefix (symbols,
                           // a multiple of 4); bits 22..29 mask rows of the pattern; bit 30 = the
                           // pattern has chains; bit 31 = pair needs the dp kernel
    uint32_t lower;        // bits 0..15 a lower bound of the pair's distance (decide mode),
                           // bits 16..31 an upper bound (mismatching positions + length
                           // difference; in decide mode also capped by what the threshold
                           // still allows): the band of the pair follows from it
};

struct Ctl {               // control block in the workspace
    unsigned long long work;                   // lane-time of the pairs for the recurrence, about
    unsigned long long maybe_work, few_work;   // of those that are counted next
    int32_t open;                              // how many they are
    int32_t maybe;                             // pairs for it or for their few matches, listed from the end of where the order goes
    int32_t few;                               // pairs for their few matches, listed from there on
    int32_t failed;                            // and how many of the listed ones had too many
    int32_t hist[kNumBins];
    int32_t fill[kNumBins];                    // what comes before here starts at zero
    int32_t start[kNumBins];
    int32_t task_start[kNumBins + 1];          // first warp task of every bin
    int32_t task_counter;
    int32_t total_tasks;
    int32_t alike;                             // whether the tasks take about as long each: no less than 0.6 of the longest on average
};

struct MultiWs {
    size_t off_dist, off_desc, off_loc, off_next, off_order, off_ctl, off_flag, off_rows, off_names, total;
    int pitch;             // uint16 elements per loc / chain row
    int row_words;         // 32-bit words of a mask row: one per 32 pattern positions
    int patterns;          // rollouts of a group that serve as patterns
    int row_cap;           // mask rows a pattern may have
    int rows_pitch;        // 32-bit words from one pattern's mask rows to the next's: a multiple of four
    int warps;             // warps of the recurrence for which the shapes are chosen
    uint32_t inv_patterns; // 2^32 / patterns, rounded up
    int text_warps, text_stride;   // prep: warps to a text, texts that the CTA's warps take at a time
    uint32_t inv_text_warps;       // 2^32 / text_warps, rounded up
    bool alone;            // one CTA orders the batch, and adds up its work itself
    bool rows_later;       // decide mode: prep leaves only the positions' rows, and multi_bin_kernel makes them for open groups
};

// Mask rows for an eighth of the positions: symbols with at least eight occurrences always
// fit, and 1/rank token frequencies put no more than about K / 10 symbols above one.
int full_row_cap(int32_t K) { return (K + 7) >> 3; }
// Prefixes from which rows that frequent symbols leave are handed to others in groups of four and five, whose rows serve two texts: below, chains cost those
// few columns no more than the rows cost prep (20000 groups of 4 of 64 over 100 symbols 235 us with them, 222 without, texts alike; 6000 of texts of 256
// 114 and 120).  In groups of eight they pay from the start (12000 of 48 1 %).
constexpr int kHandOut = 97;

MultiWs multi_layout(int32_t n_groups, int32_t N, int32_t K, int row_cap) {
    MultiWs w;
    const size_t P = pairs_of(N);
    w.pitch = (K + 7) & ~7;
    w.patterns = N & 1 ? N : N - 1;       // the last rollout of an even group is never a pattern
    w.warps = 1;
    w.text_warps = w.text_stride = 1;
    w.inv_text_warps = 0u;
    w.inv_patterns = (uint32_t)(((1ull << 32) + w.patterns - 1) / w.patterns);
    w.alone = w.rows_later = false;
    size_t off = 0;
    w.off_ctl = off;   off = align_up(off + sizeof(Ctl), 256);
    w.off_flag = off;  off = align_up(off + (size_t)n_groups, 256);
    w.off_dist = off;  off = align_up(off + (size_t)n_groups * P * 4, 256);
    w.off_desc = off;  off = align_up(off + (size_t)n_groups * P * sizeof(PairDesc), 256);
    w.off_order = off; off = align_up(off + (size_t)n_groups * P * 4, 256);
    w.off_next = off;  off = align_up(off + (size_t)n_groups * w.patterns * w.pitch * 2, 256);
    w.off_loc = off;   off = align_up(off + (size_t)n_groups * P * w.pitch * 2, 256);
    // a team's lanes cover up to 31 words more than the pattern has: slack after the last row
    w.row_words = (K + 3 + 31) >> 5;      // the pattern and what pads its texts to whole quads
    w.row_cap = row_cap;
    w.rows_pitch = (w.row_cap * w.row_words + 3) & ~3;
    w.off_rows = off;
    off = align_up(off + (size_t)n_groups * w.patterns * w.rows_pitch * 4 + 256, 256);
    w.off_names = off;
    off = align_up(off + (size_t)n_groups * N * w.pitch * 2, 256);
    w.total = off;
    return w;
}

// Class of a team shape: T = 1, 2, 4, 8 with R = 1..4, T = 16 with R = 1..3, T = 32 with R = 1, 2.
// (R = 5 and 6 amortise the work per column over more blocks, but with six bodies of the task
// loop the instruction cache no longer holds what an SM's warps run side by side.)
__host__ __device__ inline int max_blocks(int tlog) { return tlog < 4 ? 4 : 7 - tlog; }
__host__ __device__ inline int class_of(int tlog, int R) { return (tlog < 5 ? 4 * tlog : 19) + R - 1; }
__host__ __device__ inline void shape_of_class(int cls, int& tlog, int& R) {
    tlog = cls < 19 ? cls >> 2 : 5;
    R = cls - (cls < 19 ? 4 * tlog : 19) + 1;
}

// Diagonals d = row - column an optimal alignment of an m x n pair can visit when its
// distance is at most ub and at least lb.  A path that strays x diagonals beyond those between
// the corners spends x insertions and x deletions more than the length difference asks for:
// |m - n| + 2 x <= ub; and lb is a bound of what is spent besides x: lb + x <= ub (with m >= n a
// path has x insertions and at least as many other edits as lb counts: m - n deletions and one
// edit per text column without a match; with n > m it has x deletions besides those columns).
// At least two diagonals wide, so that a stripe always starts while the stripe above it is
// still running.
__host__ __device__ inline void band_of(int m, int n, int lb, int ub, int& dlo, int& dhi) {
    const int D = m - n, aD = D < 0 ? -D : D;
    int e = (ub - aD) >> 1;
    if (ub - lb < e) e = ub - lb;
    if (e < 0) e = 0;
    dlo = (D < 0 ? D : 0) - e;
    dhi = (D > 0 ? D : 0) + e;
    if (dhi == dlo) ++dhi;
}

// Cost of an iteration (a quad of columns on R blocks) in units of four issue cycles: measured
// 26 cycles per block and column with three warps per scheduler, and what does not depend on R.
__host__ __device__ inline int quad_cost(int R, bool ring) { return 26 * R + (ring ? 30 : 22); }

struct Shape { int tlog, R, time; };

// Quads of match words that a lane has under way (see dp_task).
__host__ __device__ constexpr int quads_ahead(int R) { return R <= 2 ? 2 : 1; }

// Team shape of a pair of m rows x n columns (what is left after the common prefix) whose
// distance lies in lb..ub.  Either the team's lanes hold the whole pattern, or, where the
// band is narrow enough, they form a ring that follows it: stripe g + T may only enter
// the band 2 quads_ahead(R) + 1 iterations after stripe g has left it, w + 32 R + 3 + 8 quads_ahead(R) < T (32 R + 4) for a
// band of w + 1 diagonals.  The shape with the least lane-time wins, where one that takes longer than
// the goal's limit counts for more in the proportion by which it does, and lanes that would be
// idle otherwise are free.
struct ShapeGoal { float limit, free_lanes; };
__device__ inline Shape shape_of_pair(int m, int n, int lb, int ub, ShapeGoal goal) {
    const int W = (m + 31) >> 5, nq = (n + 3) >> 2;
    int dlo, dhi;
    band_of(m, n, lb, ub, dlo, dhi);
    const int w = dhi - dlo;
    Shape best{0, 1, 0};
    float best_score = 3.0e38f;
#pragma unroll
    for (int t = 0; t <= 5; ++t) {
        const int T = 1 << t, room = w + 11 - 4 * T, far = room + 8;
        // all blocks on the team's lanes; a ring of stripes as low as the band allows
        const int full_R = (W + T - 1) >> t, ring_R = t == 0 ? 99 : far < 64 * (T - 1) ? (far < 0 ? 1 : far / (32 * (T - 1)) + 1) : max(room / (32 * (T - 1)) + 1, 3);
        static_assert(quads_ahead(2) == 2 && quads_ahead(3) == 1, "");
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int R = k ? ring_R : full_R;
            if (R > max_blocks(t) || (k && W <= T * R)) continue;
            // stripes of a ring: ceil(W / R)
            const int G = (int)((uint32_t)((W + R - 1) * (R == 3 ? 21846 : 65536 >> (R >> 1))) >> 16);
            const int time = (nq + (k ? G : T) - 1) * quad_cost(R, k);
            const float score = (float)time * fmaxf((float)T, goal.free_lanes) * fmaxf((float)time, goal.limit);
            if (score < best_score) {
                best = Shape{t, R, time};
                best_score = score;
            }
        }
    }
    return best;
}

// About the lane-time of the pair's cheapest shape.
__device__ inline int work_of_pair(int m, int n, int lb, int ub) {
    int dlo, dhi;
    band_of(m, n, lb, ub, dlo, dhi);
    return ((n + 3) >> 2) * min((m + 31) >> 5, (dhi - dlo + 128) >> 5) * 36;
}

// Bins order the pairs by the estimated running time of their warp task, longest first, and,
// within one duration bucket, by team shape: all pairs of a bin share the shape and have similar
// text lengths, and warps that pull tasks in bin order start the longest tasks first, which
// keeps the finishing times of the warps close together.  Buckets are 7 % wide (ten and a half to the octave).
__device__ inline int bin_of_shape(const Shape& s) {
    const int bucket = min(max((int)(10.5f * (15.2f - __log2f((float)s.time))), 0), kTimeBuckets - 1);
    return bucket * kNumClasses + class_of(s.tlog, s.R);
}
__device__ inline float time_of_bucket(int bucket) { return exp2f(15.2f - (float)bucket / 10.5f); }

// The pair of a descriptor, rows and columns extended to whole quads.
struct PairSize { int m, n, lb, ub; };
__device__ __forceinline__ PairSize size_of_desc(const PairDesc& d) {
    const int strip = (int)((d.bin >> kStripShift) & 0x3FFu), m = (int)(d.mn & 0xFFFFu), n = (int)(d.mn >> 16);
    const int pad = -n & 3;                                    // strip is a multiple of four
    return PairSize{m + pad - strip, n + pad - strip, (int)(d.lower & 0xFFFFu), (int)(d.lower >> 16)};
}

__device__ __forceinline__ int clamp_len(const int32_t* lens, size_t idx, int K, bool& neg) {
    int len = lens ? lens[idx] : K;
    if (len < 0) { len = 0; neg = true; }
    return min(len, K);
}

// ----------------------------------------------------------------------- names
// Names for the symbols of a group: all holders of a symbol agree on one of their positions (rollout x
// pitch + place).  Every position writes itself to the slot of a table that its symbol hashes to
// (whichever write lands last stays), and if the position found there afterwards holds the same symbol,
// that is the name; the symbols that lost their slot to another one go on with another hash, and every
// round names at least one symbol of each slot.  One CTA per group.  With the names, 16 bits
// each, a pattern's look-up table is an array: no hashing, no probing, no comparing in prep, which serves
// every text (N - 1) / 2 times.  Names and prep together, 1024 groups of 8 token prefixes: 82 us, 107 us at full
// length.  Bound: the latency between the barriers here (four CTAs of 48 KB per SM), instruction issue in prep.
constexpr uint32_t kHashMul = 0x9E3779B1u;
constexpr int kMaxTexts = SR_MAX_N / 2;        // texts a pattern is paired with
constexpr int kMaxPairs = SR_MAX_N * (SR_MAX_N - 1) / 2;
constexpr int kMostOwnPatterns = 8;            // of groups whose CTAs are a cluster: the portable size
constexpr int kMaxOwnPairs = kMostOwnPatterns * (kMostOwnPatterns + 1) / 2;

// s_sym: [N][pitch], s_table: [1 << table_log], s_len: the prefixes' lengths, out: [N][pitch].  All threads of a CTA, after a barrier.
__device__ __forceinline__ void name_symbols(const GateArgs& a, int g, const int* s_len, int32_t* s_sym, uint16_t* s_table, int table_log,
                                             int pitch, uint32_t inv_row, uint2* out) {
    const int N = a.N, tid = threadIdx.x, nthr = blockDim.x;
    const int row_quads = pitch >> 2, items = N * row_quads, shift = 32 - table_log;
    const int32_t* seqs = a.seqs + (size_t)g * N * a.stride;
#pragma unroll 4
    for (int e = tid; e < items; e += nthr) {
        const int i = (int)__umulhi((uint32_t)e, inv_row), q = e - i * row_quads, live = s_len[i] - 4 * q;
        if (live <= 0) continue;
        const int4 v = __ldg(reinterpret_cast<const int4*>(seqs + (size_t)(uint32_t)i * (uint32_t)a.stride) + q);
        reinterpret_cast<int4*>(s_sym)[e] = v;
        s_table[((uint32_t)v.x * kHashMul) >> shift] = (uint16_t)(4 * e);
        if (live > 1) s_table[((uint32_t)v.y * kHashMul) >> shift] = (uint16_t)(4 * e + 1);
        if (live > 2) s_table[((uint32_t)v.z * kHashMul) >> shift] = (uint16_t)(4 * e + 2);
        if (live > 3) s_table[((uint32_t)v.w * kHashMul) >> shift] = (uint16_t)(4 * e + 3);
    }
    __syncthreads();
    uint32_t open = 0u;                            // the thread's positions without a name, four bits an item
    int b = 0;
#pragma unroll 2
    for (int e = tid; e < items; e += nthr, b += 4) {
        const int i = (int)__umulhi((uint32_t)e, inv_row), q = e - i * row_quads, live = s_len[i] - 4 * q;
        if (live <= 0) continue;
        const int4 v = reinterpret_cast<const int4*>(s_sym)[e];
        const int32_t sym[4] = {v.x, v.y, v.z, v.w};
        uint32_t name[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) name[k] = s_table[((uint32_t)sym[k] * kHashMul) >> shift];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (k >= live) name[k] = 0u;           // any name will do
            else if (s_sym[name[k]] != sym[k]) open |= 1u << (b + k);
        }
        out[e] = make_uint2(name[0] | (name[1] << 16), name[2] | (name[3] << 16));
    }
    uint32_t mul = kHashMul;
    for (int round = 0; round < SR_MAX_N * SR_MAX_K; ++round) {
        if (!__syncthreads_or(open != 0u)) break;
        mul = mul * 0x2C1B3C6Du + 0x297A2D3Au;     // stays odd
        for (uint32_t o = open; o; o &= o - 1u) {
            const int c = __ffs(o) - 1, pos = 4 * (tid + (c >> 2) * nthr) + (c & 3);
            s_table[((uint32_t)s_sym[pos] * mul) >> shift] = (uint16_t)pos;
        }
        __syncthreads();
        for (uint32_t o = open; o; o &= o - 1u) {
            const int c = __ffs(o) - 1, pos = 4 * (tid + (c >> 2) * nthr) + (c & 3);
            const uint32_t name = s_table[((uint32_t)s_sym[pos] * mul) >> shift];
            if (s_sym[name] != s_sym[pos]) continue;
            reinterpret_cast<uint16_t*>(out)[pos] = (uint16_t)name;
            open &= ~(1u << c);
        }
    }
}

__global__ void __launch_bounds__(1024)
multi_names_kernel(GateArgs a, uint16_t* names, int pitch, uint32_t inv_row, int table_log, int g_base, int32_t* arrived, uint4* zero, int n_zero) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_len[SR_MAX_N];
    const int N = a.N, tid = threadIdx.x;
    int32_t* s_sym = reinterpret_cast<int32_t*>(smem);
    grid_begin();
    const int g = g_base + blockIdx.x;
    if (tid < N) {
        bool neg = false;
        s_len[tid] = clamp_len(a.lens, (size_t)g * N + tid, a.K, neg);
        if (neg && a.status) atomicOr(a.status, SR_STATUS_NEG_LEN);
    }
    if (arrived && tid == 0) arrived[g] = 0;           // see arrive_last
    if (blockIdx.x == 0)                               // what the kernels add up starts at zero
        for (int e = tid; e < n_zero; e += blockDim.x) zero[e] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    name_symbols(a, g, s_len, s_sym, reinterpret_cast<uint16_t*>(s_sym + N * pitch), table_log, pitch, inv_row,
                 reinterpret_cast<uint2*>(names + (size_t)g * N * pitch));
}

// ------------------------------------------------------------------ recurrence
__device__ __forceinline__ uint32_t shl_clamp(uint32_t v, uint32_t s) {
    uint32_t r;   // PTX shl clamps shift amounts above 31: the result is 0
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
    return r;
}

// One bit-vector column step over the R blocks a lane owns.  `Eq` are the column's match
// words, (inP, inM) the pre-shift horizontal delta words of the
// block above (only their top bits matter); returns this lane's last block's words in
// (inP, inM).
template <int R>
__device__ __forceinline__ void column_step(const uint32_t (&Eq)[R],
                                            uint32_t (&Pv)[R], uint32_t (&Mv)[R],
                                            uint32_t& inP, uint32_t& inM, uint32_t two) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint32_t pv = Pv[r], mv = Mv[r];
        const uint32_t hm = inM >> 31;
        // D0: the cells whose value equals that of their upper left neighbour
        const uint32_t D0 = ((((Eq[r] | hm) & pv) + pv) ^ pv) | (Eq[r] | mv | hm);
        const uint32_t Ph = mv | ~(D0 | pv);
        const uint32_t Mh = pv & D0;
        const uint32_t Phs = __funnelshift_l(inP, Ph, 1);
        // `two` holds 2 but is a run-time value, so this shift-and-insert is a multiply-add:
        // it issues on the FMA pipe and leaves the integer ALU, the bottleneck, one
        // instruction lighter per block (measured: 8 % faster than a second funnel shift)
        const uint32_t Mhs = Mh * two + hm;              // (Mh << 1) | hm
        Pv[r] = Mhs | ~(D0 | Phs);
        Mv[r] = Phs & D0;
        inP = Ph;
        inM = Mh;
    }
}

// --------------------------------------------------------------------- matches
// Pairs with few matches.  Besides the main diagonal, on which the two prefixes are compared place by
// place, two rollouts over a large vocabulary have hardly a symbol in common: a pair of 1024 uniform
// tokens out of 150 000 has seven matches where a matrix of a million cells says the same.  Between two
// matches (c, p) that it uses, a path either goes straight, max(columns, rows) edits, or by way of
// the main diagonal, where it pays for the places that differ; so the distance is a shortest path over the
// matches off the diagonal (sparse dynamic programming: Eppstein, Galil, Giancarlo and Italiano 1992), one
// lane each.  A pair whose bounds are further apart than there are lanes has more such columns than that, and the
// recurrence has it; the others are listed by prep, a warp each.
constexpr int kMostMatches = 32;                         // a lane each
// Whether a pattern of m positions has so few repeated symbols that its pairs may have few matches: 1024 uniform
// tokens have three or four (of a vocabulary of 32 000 sixteen), as long a text more than a hundred, one of 48 words four.
__device__ __forceinline__ bool few_repeats(int repeats, int m) { return 32 * repeats <= m + 64; }
// And whether a warp finds them for less than the recurrence's `work` (see work_of_pair) on `length` places of which
// `differ` differ: there is a match or more to every column between the bounds, and where the two agree, one to every place of
// a repeated symbol.  The weights are the warp's, in the units of `work`, drawn from nine
// sets on 13 shapes of K = 48 to 1024 and 16 kinds of batch (all pairs listed: 8000 groups of 8 ragged texts of 48 362 us,
// 238 with this, 243 without any search; 3000 of 100 172, 122 and 124; 400 of 16 with 256 of 3000 symbols 144, 111 and 111).
__device__ __forceinline__ bool worth_listing(int columns, int repeats, int differ, int length, int work) {
    return (2000 + 1000 * columns + 700 * repeats) * length + 1300 * repeats * (length - differ) <= work * length;
}
// Columns between the bounds up to which a pair is taken for its matches where it is not worth it by itself (see below).
constexpr int kFewColumns = 12;
constexpr int kSpan = 128;                               // columns a warp looks through a trip
constexpr int kSpans = SR_MAX_K / kSpan + 1;             // and one that begins where the longest text ends
constexpr int kMatchWarps = 8;

// The columns of a pair's stream with matches off the main diagonal, with the column's stream entry (upper half: a mask
// row, or a position from `strip` on, so that no place before `strip` is ever asked for), in `entries`, and in `differ` a bit for every column from `strip` on that differs from the pattern: column
// strip + 128 s + 4 l + k in bit l of word k of differ[s].  Returns the number of those columns, or more than
// there are lanes for.
// (kShared: the stream and, below, the rows are in shared memory.)
template <bool kShared>
__device__ __forceinline__ int find_matches(const uint2* stream, const uint2* text, const uint2* pat, int m, int n, int strip,
                                            uint4* differ, uint32_t* entries) {
    const int lane = threadIdx.x & 31;
    int found = 0;
    auto fetch = [&](int s) {
        const int q = (strip >> 2) + 32 * s + lane;
        return 4 * q < n ? (kShared ? stream[q] : __ldg(stream + q)) : make_uint2(kLocNone * 0x10001u, kLocNone * 0x10001u);
    };
    uint2 ahead[2] = {fetch(0), fetch(1)};
    for (int s = 0; strip + kSpan * s < n; ++s) {
        const int q = (strip >> 2) + 32 * s + lane;
        const int left = min(max(n - 4 * q, 0), 4), both = min(left, max(m - 4 * q, 0));   // columns that exist, and of those with a row
        const uint2 v = ahead[0];
        ahead[0] = ahead[1];
        ahead[1] = fetch(s + 2);
        if (strip + kSpan * (s + 1) <= min(m, n) && __all_sync(0xFFFFFFFFu, (v.x & v.y) == kLocNone * 0x10001u && (v.x | v.y) == (v.x & v.y))) {
            if (lane == 0) differ[s] = make_uint4(~0u, ~0u, ~0u, ~0u);     // no column of these has a match
            continue;
        }
        const uint32_t at0 = (uint32_t)(4 * q * 0x10001 + 0x10000), at1 = at0 + 0x20002u;   // the places on the main diagonal
        uint32_t d0 = set_halves(v.x ^ at0), d1 = set_halves(v.y ^ at1);
        uint32_t off0 = matches_beside(v.x, at0, strip), off1 = matches_beside(v.y, at1, strip);
        if ((v.x | v.y) & (kLocRow * 0x10001u)) {      // a symbol that occurs more than once: the names tell
            const uint2 x = kShared ? text[q] : __ldg(text + q), o = kShared ? pat[q] : __ldg(pat + q);
            d0 = set_halves(x.x ^ o.x);
            d1 = set_halves(x.y ^ o.y);
        }
        if (left < 4) {
            off0 = left > 1 ? off0 : (left == 1 ? off0 & 0xFFFFu : 0u);
            off1 = left == 3 ? off1 & 0xFFFFu : 0u;
        }
        if (both < 4) {
            d0 = both > 1 ? d0 : (both == 1 ? d0 & 0xFFFFu : 0u);
            d1 = both == 3 ? d1 & 0xFFFFu : 0u;
        }
        const unsigned b0 = __ballot_sync(0xFFFFFFFFu, (d0 & 0x8000u) != 0u), b1 = __ballot_sync(0xFFFFFFFFu, (d0 >> 31) != 0u);
        const unsigned b2 = __ballot_sync(0xFFFFFFFFu, (d1 & 0x8000u) != 0u), b3 = __ballot_sync(0xFFFFFFFFu, (d1 >> 31) != 0u);
        if (lane == 0) differ[s] = make_uint4(b0, b1, b2, b3);
        if (!__any_sync(0xFFFFFFFFu, (off0 | off1) != 0u)) continue;
        const unsigned o0 = __ballot_sync(0xFFFFFFFFu, (off0 & 0x8000u) != 0u), o1 = __ballot_sync(0xFFFFFFFFu, (off0 >> 31) != 0u);
        const unsigned o2 = __ballot_sync(0xFFFFFFFFu, (off1 & 0x8000u) != 0u), o3 = __ballot_sync(0xFFFFFFFFu, (off1 >> 31) != 0u);
        const unsigned under = (1u << lane) - 1u;
        int at = found + __popc(o0 & under) + __popc(o1 & under) + __popc(o2 & under) + __popc(o3 & under);
        found += __popc(o0) + __popc(o1) + __popc(o2) + __popc(o3);
        if (found > kMostMatches) return found;
        if (off0 & 0x8000u) entries[at++] = (uint32_t)(4 * q) | (v.x << 16);      // by column
        if (off0 >> 31) entries[at++] = (uint32_t)(4 * q + 1) | (v.x & 0xFFFF0000u);
        if (off1 & 0x8000u) entries[at++] = (uint32_t)(4 * q + 2) | (v.y << 16);
        if (off1 >> 31) entries[at++] = (uint32_t)(4 * q + 3) | (v.y & 0xFFFF0000u);
    }
    __syncwarp();
    return found;
}

// The distance of a pair from what find_matches found.  upper: the distance along the main diagonal.  Negative: more
// matches than there are lanes for.
template <bool kShared>
__device__ __forceinline__ int distance_by_matches(uint32_t* entries, int count, const uint4* differ, const uint32_t* rows, int row_words,
                                                   int m, int n, int strip, int upper) {
    const int lane = threadIdx.x & 31;
    const int lo = min(m, n);
    // every entry's matches: one position, or those of a mask row
    uint32_t node = lane < count ? entries[lane] : 0u;
    const bool row = lane < count && (node >> 16) >= kLocRow;
    if (__any_sync(0xFFFFFFFFu, lane < count && (node >> 16) >= kLocChain)) return -1;
    int total = count;
    unsigned todo = __ballot_sync(0xFFFFFFFFu, row);
    if (todo) {
        const bool single = lane < count && !row;
        const unsigned singles = __ballot_sync(0xFFFFFFFFu, single);
        total = __popc(singles);
        if (single) entries[__popc(singles & ((1u << lane) - 1u))] = node;
        while (todo) {                                 // eight rows on their way before the first is looked at
            uint32_t bits[8], column[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                bits[k] = column[k] = 0u;
                if (todo == 0u) continue;
                const uint32_t e = __shfl_sync(0xFFFFFFFFu, node, __ffs(todo) - 1);
                todo &= todo - 1u;
                column[k] = e & 0xFFFFu;
                const uint32_t* row = rows + ((e >> 16) & 0x3FFFu) * row_words + lane;
                if (lane < row_words) bits[k] = kShared ? *row : __ldg(row);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                while (__any_sync(0xFFFFFFFFu, bits[k] != 0u)) {
                    const int p = bits[k] ? 32 * lane + __ffs(bits[k]) - 1 : -1;
                    bits[k] &= bits[k] - 1u;
                    const bool use = p >= strip && p != (int)column[k];
                    const unsigned b = __ballot_sync(0xFFFFFFFFu, use);
                    const int at = total + __popc(b & ((1u << lane) - 1u));
                    total += __popc(b);
                    if (use && at < kMostMatches) entries[at] = column[k] | ((uint32_t)p << 16);
                }
            }
            if (total > kMostMatches) return -1;
        }
        if (total == 0) return upper;
        __syncwarp();
        // by column again
        const uint32_t own = lane < total ? entries[lane] : 0xFFFFFFFFu;
        int rank = 0;
        for (int l = 0; l < total; ++l) {
            const uint32_t other = __shfl_sync(0xFFFFFFFFu, own, l);
            rank += (other & 0xFFFFu) < (own & 0xFFFFu) || ((other & 0xFFFFu) == (own & 0xFFFFu) && l < lane);
        }
        if (lane < total) entries[rank] = own;
        __syncwarp();
    }
    __syncwarp();
    node = lane < total ? entries[lane] : (uint32_t)strip * 0x10001u;
    const int c = (int)(node & 0xFFFFu), p = (int)(node >> 16);
    // places that differ before x, strip <= x <= lo: columns begin at strip, and so do the positions of all nodes
    int before = 0;
    if (lane < kSpans && strip + kSpan * lane < n) {
        const uint4 d = differ[lane];
        before = __popc(d.x) + __popc(d.y) + __popc(d.z) + __popc(d.w);
    }
#pragma unroll
    for (int d = 1; d < 16; d <<= 1) {
        const int up = __shfl_up_sync(0xFFFFFFFFu, before, d);
        if (lane >= d) before += up;
    }
    auto differing = [&](int x) {
        const int rel = x - strip, s = rel / kSpan, l = (rel % kSpan) >> 2, k = rel & 3;
        const uint4 d = differ[s];
        const uint32_t under = (1u << l) - 1u, with = under | (1u << l);
        const int sum = __shfl_sync(0xFFFFFFFFu, before, max(s - 1, 0));
        return (s > 0 ? sum : 0) + __popc(d.x & (k > 0 ? with : under)) + __popc(d.y & (k > 1 ? with : under)) +
               __popc(d.z & (k > 2 ? with : under)) + __popc(d.w & under);
    };
    const int off = abs(c - p);
    const int enter = min(c, p), leave = max(c, p) + 1;  // the last place of the diagonal before the match, the first after it
    const int at_enter = differing(enter), at_leave = differing(min(leave, lo)), at_end = differing(lo);
    int cost = off + at_enter;                            // up to the match and through it
    for (int l = 0; l + 1 < total; ++l) {
        const uint32_t from = __shfl_sync(0xFFFFFFFFu, node, l);
        const uint32_t paid = __shfl_sync(0xFFFFFFFFu, (uint32_t)cost | ((uint32_t)at_leave << 16), l);
        const int fc = (int)(from & 0xFFFFu), fp = (int)(from >> 16);
        int step = max(c - fc, p - fp) - 1;
        if (max(fc, fp) < enter) step = min(step, abs(fc - fp) + at_enter - (int)(paid >> 16) + off);
        if (c > fc && p > fp) cost = min(cost, (int)(paid & 0xFFFFu) + step);
    }
    int last = max(n - c, m - p) - 1;
    if (leave <= lo) last = min(last, off + at_end - at_leave + abs(n - m));
    const int d = lane < total ? cost + last : upper;
    return min(__reduce_min_sync(0xFFFFFFFFu, d), upper);
}

// ------------------------------------------------------------------- both ends
// Pairs by the latency of their columns, for batches that leave most of the GPU idle: one team of lanes runs the
// recurrence over the first half of the text's columns, another one next to it over the rest from the end
// backwards (both sequences reversed), so that the chain of columns is half as long; where they meet, the distance is
// the least sum over the rows of what the two paid (Hirschberg 1975).  A team has T <= 16 lanes of R blocks each, a
// lane for every stripe; a warp has 16 / T pairs.  Stream and mask rows are in shared memory, where no first use of
// a row costs a trip to L2, and what a column needs is as good as computed in the stream's entry.
// Bound: the latency of the columns' chain of operations, then the integer pipe.

// Rows and columns from which looking for few matches costs less than they do here.
constexpr int kWorthMatches = 512;

// What a stream entry is here: a position, kLocNone, kWideRow | first word of a mask row, or kWideChain | position.
constexpr uint32_t kWideRow = 0x80000000u, kWideChain = 0xC0000000u;
__device__ __forceinline__ uint32_t wide_entry(uint32_t e, int row_words) {
    if (e < kLocRow) return e;
    return e < kLocChain ? kWideRow | ((e & 0x3FFFu) * (uint32_t)row_words) : kWideChain | (e & 0x3FFFu);
}

// Loads a lane's R words of a mask row where the entry names one, without a branch.
template <int R>
__device__ __forceinline__ void load_wide_row(uint32_t entry, uint32_t row, uint32_t (&Eq)[R]) {
    static_assert(R >= 1 && R <= 3, "");
    if constexpr (R == 1)
        asm volatile("{ .reg .pred p; setp.lt.s32 p, %1, 0xC0000000; @p ld.shared.u32 %0, [%2]; }" : "+r"(Eq[0]) : "r"(entry), "r"(row));
    else if constexpr (R == 2)
        asm volatile("{ .reg .pred p; setp.lt.s32 p, %2, 0xC0000000; @p ld.shared.u32 %0, [%3]; @p ld.shared.u32 %1, [%3 + 4]; }"
            : "+r"(Eq[0]), "+r"(Eq[1]) : "r"(entry), "r"(row));
    else
        asm volatile("{ .reg .pred p; setp.lt.s32 p, %3, 0xC0000000; @p ld.shared.u32 %0, [%4]; @p ld.shared.u32 %1, [%4 + 4]; "
            "@p ld.shared.u32 %2, [%4 + 8]; }"
            : "+r"(Eq[0]), "+r"(Eq[1]), "+r"(Eq[2]) : "r"(entry), "r"(row));
}

// The signs of four words, one a byte, the first word's on top.
__device__ __forceinline__ uint32_t signs(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3) {
    uint32_t a, b, r;
    asm("prmt.b32 %0, %1, %2, 0xFB00;" : "=r"(a) : "r"(w1), "r"(w0));
    asm("prmt.b32 %0, %1, %2, 0x00FB;" : "=r"(b) : "r"(w3), "r"(w2));
    asm("prmt.b32 %0, %1, %2, 0x7610;" : "=r"(r) : "r"(b), "r"(a));
    return r;
}

// The distances of a warp's pairs, each in the first lane of its 2 T lanes.  Per pair: loc, its stream (16-bit entries),
// and wide, room for the wide one, of which it makes use afterwards; m, n: lengths; strip: common prefix to leave out (a
// multiple of 4, of 32 where the stream names rows); live: false for lanes without a pair.  rows: the pattern's mask
// rows, turned: the same with the order of a row's bits reversed; info: upper halves lead along the chains.
// kTwo: a team is a whole warp, the pair's other one the next warp (of an even one), and `tlog` the number of a barrier for
// the two; the distance is then in the even warp's first lane.  With 32 lanes a half of 1024 columns takes 159
// iterations of one block instead of 143 of two.
template <int R, bool kTwo = false>
__device__ __forceinline__ int distance_from_both_ends(const uint16_t* loc, uint4* wide, const uint32_t* rows, const uint32_t* turned, int row_words,
                                                       const uint32_t* info, bool chains, bool live, int m, int n, int strip, int tlog,
                                                       uint32_t two) {
    const int lane = threadIdx.x & 31, T = kTwo ? 32 : 1 << tlog, gl = (int)threadIdx.x & (2 * T - 1), lt = lane & (T - 1);
    auto meet = [&]() {
        if (kTwo) asm volatile("bar.sync %0, 64;" ::"r"(tlog) : "memory"); else __syncwarp();
    };
    const int pad = -n & 3;                            // both are extended to whole quads of columns
    m = live ? m + pad - strip : 0;
    n = live ? n + pad - strip : 0;
    const int W = (m + 31) >> 5, G = (W + R - 1) / R;  // blocks, stripes
    const int nq = n >> 2, ahead = (nq + 1) >> 1;      // quads, and those of the half that runs forwards
    const bool back = gl >= T, held = lt < G;
    const int quads = back ? nq - ahead : ahead;
    // the wide stream: quads from `ahead` on in the order in which the other half meets their columns; one without
    // matches at either end
    const uint2* quad = reinterpret_cast<const uint2*>(loc + strip);
    for (int k = gl; k < nq; k += 2 * T) {
        const uint2 q = quad[k];
        uint32_t e[4] = {q.x & 0xFFFFu, q.x >> 16, q.y & 0xFFFFu, q.y >> 16};
#pragma unroll
        for (int u = 0; u < 4; ++u) e[u] = wide_entry(e[u], row_words);
        wide[1 + k] = k < ahead ? make_uint4(e[0], e[1], e[2], e[3]) : make_uint4(e[3], e[2], e[1], e[0]);
    }
    if (gl == 0) wide[0] = make_uint4(kLocNone, kLocNone, kLocNone, kLocNone);
    if (gl == 1) wide[1 + nq] = make_uint4(kLocNone, kLocNone, kLocNone, kLocNone);
    meet();
    // Backwards, position strip + p is row 32 W - 1 - p: the rows beyond the pattern's end come first, and
    // with vertical deltas of zero they hand on the +1 of row 0 as it is.
    const uint32_t sign = back ? ~0u : 1u, four = two * two, next_column = two * 128u;
    const uint32_t origin = back ? (uint32_t)(32 * W - 1 + strip - 32 * R * lt) : (uint32_t)-(strip + 32 * R * lt);
    const uint32_t words = (uint32_t)__cvta_generic_to_shared(back ? turned + (row_words - (strip >> 5) - W + R * lt) : rows + ((strip >> 5) + R * lt));
    const uint4* from = back ? wide + nq : wide + 1;   // the half's first quad
    const int step = back ? -1 : 1, most = held ? quads : -1;
    uint32_t Pv[R], Mv[R], endP[R], endM[R];
#pragma unroll
    for (int r = 0; r < R; ++r) { Pv[r] = 0xFFFFFFFFu; Mv[r] = 0u; }
    if (back && lt == 0) Pv[0] = 0xFFFFFFFFu << (32 * W - m);
#pragma unroll
    for (int r = 0; r < R; ++r) { endP[r] = Pv[r]; endM[r] = Mv[r]; }
    // the quad for iteration j: none before the lane's first; after its last any will do
    auto fetch = [&](int j) { return from[step * min(max(j - lt, -1), most)]; };
    auto match = [&](const uint4& q, uint32_t (&Eq)[4][R]) {
        const uint32_t e[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t d0 = e[u] * sign + origin;
#pragma unroll
            for (int r = 0; r < R; ++r) Eq[u][r] = shl_clamp(1u, d0 - 32u * r);    // 0 for rows and chains
            load_wide_row<R>(e[u], e[u] * four + words, Eq[u]);
        }
        if (!chains) return;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (e[u] < kWideChain) continue;
            uint32_t p = e[u] & 0x3FFFu;
            for (int hop = 0; hop < SR_MAX_K && p < (uint32_t)SR_MAX_K; ++hop) {   // a chain ends at 0xFFFF
                const uint32_t d0 = p * sign + origin;
#pragma unroll
                for (int r = 0; r < R; ++r) Eq[u][r] |= shl_clamp(1u, d0 - 32u * r);
                p = info[p] >> 16;
            }
        }
    };
    uint32_t Eq[4][R];
    match(fetch(0), Eq);
    uint4 q1 = fetch(1);
    uint32_t outP = 0u, outM = 0u;                     // signs of the deltas that leave the stripe
    const int last = held ? lt + quads - 1 : -1;       // the iteration after which the words are kept
    const int iters = __reduce_max_sync(0xFFFFFFFFu, ahead + G - 1);
    for (int j = 0; j < iters; ++j) {
        const uint4 q = q1;                            // the quad after this one
        q1 = fetch(j + 2);
        // Deltas from the stripe above, which worked on this quad last iteration.  A lane whose first quad is still to come gets
        // zeros, has no matches, and so leaves its words alone.
        uint32_t wP = __shfl_up_sync(0xFFFFFFFFu, outP, 1), wM = __shfl_up_sync(0xFFFFFFFFu, outM, 1);
        if (lt == 0) { wP = 0xFFFFFFFFu; wM = 0u; }    // row 0: +1 everywhere
        uint32_t next[4][R], cP[4], cM[4];
        match(q, next);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            cP[u] = wP;
            cM[u] = wM;
            column_step<R>(Eq[u], Pv, Mv, cP[u], cM[u], two);
            wP *= next_column;
            wM *= next_column;
        }
        outP = signs(cP[0], cP[1], cP[2], cP[3]);
        outM = signs(cM[0], cM[1], cM[2], cM[3]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            endP[r] = j == last ? Pv[r] : endP[r];
            endM[r] = j == last ? Mv[r] : endM[r];
#pragma unroll
            for (int u = 0; u < 4; ++u) Eq[u][r] = next[u][r];
        }
    }
    // The vertical deltas of the column where the halves meet: forwards along rows 1..m, backwards turned round.
    uint2* met = reinterpret_cast<uint2*>(wide);
    meet();
    if (held && back) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int w = W - 1 - (R * lt + r);
            if (w >= 0) met[w] = make_uint2(__brev(endP[r]), __brev(endM[r]));
        }
    }
    meet();
    int sum = 0, least = 0, whole = 0;
    if (held && !back) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int w = R * lt + r;
            if (w >= W) continue;
            const uint32_t rows_here = low_mask(min(m - 32 * w, 32));
            const uint2 b = met[w];
            const uint32_t bp = b.x & rows_here, bm = b.y & rows_here, fp = endP[r] & rows_here, fm = endM[r] & rows_here;
            whole += __popc(bp) - __popc(bm);
            // one row further: the front pays for it, the back does not any more
#pragma unroll 8
            for (int k = 0; k < 32; ++k) {
                sum += (int)((fp >> k) & 1u) + (int)((bm >> k) & 1u) - (int)((fm >> k) & 1u) - (int)((bp >> k) & 1u);
                least = min(least, sum);
            }
        }
    }
    int incl = sum;
#pragma unroll
    for (int d = 1; d < (kTwo ? 32 : 16); d <<= 1) {
        const int up = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (gl >= d) incl += up;
    }
    least += incl - sum;
    if (back) least = 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        if (!kTwo && d >= 2 * T) break;
        whole += __shfl_xor_sync(0xFFFFFFFFu, whole, d);
        least = min(least, __shfl_xor_sync(0xFFFFFFFFu, least, d));
    }
    return n + whole + least;                          // row 0: nothing of the pattern at the front, all of it at the back
}

// Sum, threshold and outputs of group g by one CTA, from what distance(pair) and length(rollout) give.
template <class Distance, class Length>
__device__ __forceinline__ void evaluate_group(const GateArgs& a, int g, uint8_t* exact, Distance distance, Length length) {
    __shared__ double s_term[kMaxPairs];
    __shared__ int32_t s_d[kMaxPairs];
    const int N = a.N, P = pairs_of(N);
    for (int e = threadIdx.x; e < P; e += blockDim.x) {
        const int pr = kPairs.v[N][e];
        s_d[e] = distance(e);
        s_term[e] = pair_term(s_d[e], length(pr & 0xFF), length(pr >> 8), a.norm_mode);
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    double s = 0.0;
    int isum = 0;
#pragma unroll 4
    for (int p = 0; p < P; ++p) {
        s = __dadd_rn(s, s_term[p]);
        isum += s_d[p];
    }
    const double dk = __ddiv_rn(s, (double)P);
    if (a.pair_sum) a.pair_sum[g] = isum;
    if (a.mean) a.mean[g] = dk;
    a.stop[g] = dk < a.threshold ? 1 : 0;
    if (exact) exact[g] = 1;
}

// Decide mode: d_K of group g on its pairs' lower bounds, and where the mask is all that is wanted on the upper ones (see
// multi_bound_kernel).  True, in all threads, if that settles the group; its outputs are then written.
__device__ __forceinline__ int settle_group(const GateArgs& a, int g, uint8_t* exact, const int32_t* lower, const int32_t* upper, const int* len) {
    __shared__ double s_below[kMaxOwnPairs], s_above[kMaxOwnPairs];
    __shared__ int s_settled_here;
    const int N = a.N, P = pairs_of(N);
    for (int e = threadIdx.x; e < P; e += blockDim.x) {
        const int pr = kPairs.v[N][e], m = len[pr & 0xFF], n = len[pr >> 8];
        s_below[e] = pair_term(lower[e], m, n, a.norm_mode);
        s_above[e] = pair_term(upper[e], m, n, a.norm_mode);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double below = 0.0, above = 0.0;
        int isum = 0;
#pragma unroll 4
        for (int p = 0; p < P; ++p) {
            below = __dadd_rn(below, s_below[p]);
            above = __dadd_rn(above, s_above[p]);
            isum += lower[p];
        }
        const double dk = __ddiv_rn(below, (double)P);
        const bool mask_only = !a.pair_dist && !a.pair_sum && !a.mean && !exact;
        const bool cut = mask_only && __ddiv_rn(above, (double)P) < a.threshold;
        s_settled_here = !(dk < a.threshold) || cut;
        if (s_settled_here) {
            if (a.pair_sum) a.pair_sum[g] = isum;
            if (a.mean) a.mean[g] = dk;
            if (exact) exact[g] = 0;
            a.stop[g] = cut ? 1 : 0;
        }
    }
    __syncthreads();
    return s_settled_here;
}

// Whether this is the last of the group's `parts` CTAs to come here.  All threads of a CTA call it after writing their distances.
__device__ __forceinline__ bool arrive_last(int parts, int32_t* arrived) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(arrived, 1) == parts - 1;
        __threadfence();
    }
    __syncthreads();
    return s_last;
}

// Mask rows that frequent symbols leave, for those of a thread's four with fewer occurrences: behind theirs, whoever comes first.
__device__ __forceinline__ void hand_out_rest(uint4 more, uint2 names, uint32_t need, int* repeats, int row_cap, uint16_t* map, uint32_t* info) {
    const uint32_t m[4] = {more.x, more.y, more.z, more.w}, name[4] = {names.x & 0xFFFFu, names.x >> 16, names.y & 0xFFFFu, names.y >> 16};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (m[k] == 0u || m[k] >= need) continue;
        const int row = repeats[need - 1u] + atomicAdd(repeats + 4, 1);
        if (row >= row_cap) continue;
        map[name[k]] = (uint16_t)(kLocRow | (uint32_t)row);
        info[k] = kLocRow | (uint32_t)row;
    }
}
// (Where registers are what limits the CTAs of an SM: few patterns need it.  Inlined, decide mode takes 1 % longer; not inlined, the gate up to 3.)
__device__ __noinline__ void hand_out_rest_apart(uint4 more, uint2 names, uint32_t need, int* repeats, int row_cap, uint16_t* map, uint32_t* info) {
    hand_out_rest(more, names, need, repeats, row_cap, map, info);
}

// One CTA per pattern.  Per text it also counts the columns whose symbol does not occur in the
// pattern at all and the positions at which text and pattern differ: bounds of the pair's distance that
// cost next to nothing here.  Where they meet the pair is done.
// kThreads: the CTA's threads where they are the most there can be (known at compile time 82 us of the token-level
// batch of 1024 groups, at run time 84.5), 0 for fewer.
// kTextThreads: a warp for every text where there are more than eight and a pair takes a warp (kPairs, K > 253), while every CTA
// has an SM: the ninth text and those after it do not wait for the first eight (6 groups of 20 texts of 850 that differ in 2 % of
// their places: 120 -> 69 us, 107 sorted; with more CTAs than SMs three of 256 threads to an SM are as good or better, 18 groups of
// 18 diverging ones 112 and 123).
// kPairs: the whole gate after the names.  Streams and mask rows stay in shared memory, the distances are computed right
// there, and the last CTA of a group evaluates it.
// kOwnNames: the whole gate.  A group's CTAs are a cluster, and each of them names all of the group's symbols for itself.
// kDecide and kPairs: a group's CTAs are a cluster, whose first one sums up the pairs' bounds, as multi_bound_kernel does; no
// distance is computed for a group that they settle.
// kTwoWarps: patterns of more than 512 positions and no more than two texts, a CTA to an SM: a pair has two warps (40
// groups of 4 texts of 1024: 48 -> 37 us; with four texts the integer pipe is busy already, 16 groups of 8: 46 -> 48).
// Small batches of fewer threads a CTA than that: no more than 72 registers, or seven CTAs of 128 threads do not fit an SM (301 groups of
// 5 of 501 at 74 registers 65.3 us, at 72 60.5).
// Large batches: room for seven CTAs of 256 threads an SM at least (32 registers, which leave room for eight), whose barriers then cost
// less (1024 groups of uniform tokens of up to 1024 with five 115.2 us, six 109.9, seven 105.0, eight 105.0).  CTAs of four warps gain as
// well (8000 groups of 8 of 64 4 % over six), those of two lose more by 32 registers, spilled, than by fewer of them (20000 groups of 4 of 64
// over 100 symbols 242 us, 233 with 48).
template <bool kDecide, int kThreads, bool kPairs, bool kOwnNames>
struct PrepBounds {
    static constexpr bool kFew = kPairs && !kDecide && !kOwnNames && kThreads == 0;
    static constexpr int kMost = kThreads ? kThreads : kFew ? kMostPrepThreads - 32 : kMostPrepThreads;
    static constexpr int kCtas = kThreads > kMostPrepThreads ? 1 : kFew ? 4 : kPairs ? 3 : kThreads == kTwoWarpThreads ? 20 : 7;
};
template <bool kDecide, int kThreads, bool kPairs, bool kOwnNames, bool kTwoWarps = false>
__global__ void __launch_bounds__(PrepBounds<kDecide, kThreads, kPairs, kOwnNames>::kMost, PrepBounds<kDecide, kThreads, kPairs, kOwnNames>::kCtas)
multi_prep_kernel(GateArgs a, unsigned char* ws, MultiWs W, int32_t* dist_out, int g_base, uint8_t* exact, uint32_t inv_row, int table_log,
                  uint32_t two) {
    constexpr bool kCluster = kOwnNames || (kDecide && kPairs);
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t* s_info = reinterpret_cast<uint32_t*>(smem);             // [pitch] see below
    uint16_t* s_map = reinterpret_cast<uint16_t*>(s_info + W.pitch);  // [N * pitch] stream entry of every name
    // kPairs: [N / 2][pitch] streams, [2][rows_pitch] mask rows, and turned round
    uint16_t* s_loc = s_map + a.N * (W.pitch + 8) + 16;
    uint32_t* s_rows = reinterpret_cast<uint32_t*>(s_loc + (a.N >> 1) * W.pitch);
    // kOwnNames: [N][pitch] names, [N][pitch] symbols and their table
    uint16_t* s_names = reinterpret_cast<uint16_t*>(s_rows + (2 * W.rows_pitch + 8));
    __shared__ int64_t s_stream[kMaxTexts];                           // where a text's stream begins
    __shared__ int s_txt[kMaxTexts], s_len[kMaxTexts], s_cp[kMaxTexts];
    __shared__ uint32_t s_count[kMaxTexts];  // differing positions | absent columns << 16
    __shared__ uint32_t s_flag[kMaxTexts];   // the stream holds row or chain entries
    __shared__ int s_repeats[5];     // symbols with >= 2, 3, 4 occurrences; mask rows handed out to frequent ones, asked for by others

    const int N = a.N, K = a.K, P = pairs_of(N);
    const int tid = threadIdx.x, lane = tid & 31, nthr = kThreads ? kThreads : blockDim.x, warps = nthr >> 5;
    const int M = W.patterns;
    // (divisions by what only the host knows are its to prepare: five of them were a sixth of a warp's instructions)
    int gl = M > 1 ? (int)__umulhi(blockIdx.x, W.inv_patterns) : (int)blockIdx.x;
    if (gl * M > (int)blockIdx.x) --gl;
    const int g = g_base + gl, i = (int)blockIdx.x - gl * M;
    if (tid < 5) s_repeats[tid] = 0;
    for (int e = tid; 8 * e < N * W.pitch; e += nthr)
        reinterpret_cast<uint4*>(s_map)[e] = make_uint4(kLocNone * 0x10001u, kLocNone * 0x10001u, kLocNone * 0x10001u, kLocNone * 0x10001u);
    for (int e = tid; 4 * e < W.pitch; e += nthr) reinterpret_cast<uint4*>(s_info)[e] = make_uint4(0u, 0u, 0u, 0u);
    grid_begin();
    if (kCluster) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");     // the wait: before the first distance
    bool neg = false;
    const int m = clamp_len(a.lens, (size_t)g * N + i, K, neg);
    const uint16_t* names = kOwnNames ? s_names : reinterpret_cast<const uint16_t*>(ws + W.off_names) + (size_t)g * N * W.pitch;
    const uint16_t* pat = names + i * W.pitch;
    // kCluster: the group's lengths, and in the cluster's first CTA its distances (and upper bounds).  (The others write
    // there once it has started.)
    __shared__ int s_all_len[kCluster ? SR_MAX_N : 1];
    __shared__ int32_t s_all_dist[kCluster ? kMaxOwnPairs : 1];
    __shared__ int32_t s_all_upper[kCluster && kDecide ? kMaxOwnPairs : 1];
    __shared__ int s_settled;
    const auto cluster = cooperative_groups::this_cluster();
    if constexpr (kCluster) {
        if (tid < N) {
            bool negative = false;
            s_all_len[tid] = clamp_len(a.lens, (size_t)g * N + tid, K, negative);
            if (kOwnNames && negative && i == 0 && a.status) atomicOr(a.status, SR_STATUS_NEG_LEN);
        }
    }
    if constexpr (kOwnNames) {
        __syncthreads();
        int32_t* s_sym = reinterpret_cast<int32_t*>(s_names + N * W.pitch);
        name_symbols(a, g, s_all_len, s_sym, reinterpret_cast<uint16_t*>(s_sym + N * W.pitch), table_log, W.pitch, inv_row, reinterpret_cast<uint2*>(s_names));
    }
    // Which rollout of a pair is the pattern follows a round-robin tournament: with M = N
    // for odd N and N - 1 otherwise, rollout i < M is the pattern against the `half` rollouts
    // after it (cyclically among the first M) and, for even N, against the last rollout,
    // which is a text for everyone.  Every pattern so serves floor(N / 2) texts.  In
    // ascending order the texts of pattern i are: the rollouts more than `half` places
    // before it, the `half` places after it, and the last rollout of an even group.
    const int half = (M - 1) / 2;
    const int n_before = max(0, i - half), n_after = min(i + half, M - 1) - i;
    const int ntxt = n_before + n_after + ((N & 1) ? 0 : 1);
    // The texts, one warp per text.  The warp measures the common prefix of pattern and text (256
    // positions per trip, stopping at the first mismatch): rollouts of one group start from
    // the same state and often agree on their first symbols, and the edit distance of two
    // sequences equals that of what is left after a common prefix is removed, so those rows
    // and columns are never looked up nor run through the recurrence.
    for (int t = tid >> 5; t < ntxt; t += warps) {
        const int j = t < n_before ? t : (t < n_before + n_after ? i + 1 + (t - n_before) : N - 1);
        const int n = clamp_len(a.lens, (size_t)g * N + j, K, neg);
        const int lo = min(m, n);
        int cp = lo;                                  // first mismatch; min(m, n) = none found
        for (int base = 0; base < lo && cp == lo; base += 256) {
            const int at = base + 8 * lane;
            int eq = 8;                               // names of the lane's eight that agree
            if (at < lo) {
                const uint4 u = *reinterpret_cast<const uint4*>(pat + at);
                const uint4 v = *reinterpret_cast<const uint4*>(names + j * W.pitch + at);
                const uint32_t x[4] = {u.x ^ v.x, u.y ^ v.y, u.z ^ v.z, u.w ^ v.w};
#pragma unroll
                for (int w = 3; w >= 0; --w)
                    if (x[w]) eq = 2 * w + ((x[w] & 0xFFFFu) ? 0 : 1);
            }
            const unsigned b = __ballot_sync(0xFFFFFFFFu, eq < 8);
            if (b) {
                const int first = __ffs(b) - 1;
                cp = min(base + 8 * first + __shfl_sync(0xFFFFFFFFu, eq, first), lo);
            }
        }
        if (lane == 0) {
            s_txt[t] = j;
            s_len[t] = n;
            s_stream[t] = ((int64_t)g * P + pair_index(min(i, j), max(i, j), N)) * W.pitch;
            s_count[t] = 0u;
            s_flag[t] = 0u;
            s_cp[t] = cp >= lo ? -1 : cp;             // -1: one prefix is the start of the other, nothing is left to do
        }
    }
    __syncthreads();
    // Every position claims its name's entry; those that find another one there count as further
    // occurrences with the position that stayed (s_info[claimant]).  Four positions per thread.
    const int p0 = 4 * tid, mine = min(max(m - p0, 0), 4);
    uint32_t my_name[4] = {0u, 0u, 0u, 0u}, my_first[4];
    if (mine > 0) {
        const uint2 v = *reinterpret_cast<const uint2*>(pat + p0);
        my_name[0] = v.x & 0xFFFFu; my_name[1] = v.x >> 16; my_name[2] = v.y & 0xFFFFu; my_name[3] = v.y >> 16;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (k < mine) s_map[my_name[k]] = (uint16_t)(p0 + k);
    __syncthreads();
    bool repeated = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        my_first[k] = p0 + k;
        if (k >= mine) continue;
        my_first[k] = s_map[my_name[k]];
        if (my_first[k] != (uint32_t)(p0 + k)) {
            atomicAdd(&s_info[my_first[k]], 1u);
            repeated = true;
        }
    }
    if (__syncthreads_or(repeated)) {
        // Symbols with several occurrences.  In written language a few tokens make up much of
        // every rollout (a third of the columns of such a text meet a symbol that occurs more
        // than once, the most common one dozens of times), so these get a row of match words,
        // one per 32 positions, which the recurrence reads in place of its one-hot word.  (Walking
        // a chain of occurrences makes the recurrence wait for the longest chain of the warp: 141 groups
        // of 8 such texts of 1024 tokens take 165 us, with a quarter of the rows and chains besides 426.)
        // The full pool has room for every symbol with at least eight occurrences; what does not fit
        // (the rarest of the repeated ones) is left as a chain of at most seven positions.  In a
        // smaller pool (see launch_gate_multi) the last symbols to ask get a chain of any length.  Where the rows suffice for all symbols
        // of three or of four occurrences, what these leave is handed to others (1024 groups of 8 of 1024
        // symbols out of 3000, 140 of which repeat in a pattern: 554 -> 416 us where they differ in 2 % of their places, 325 -> 284 diverging;
        // 438 of diverging texts of 200 71 -> 62).  Where they do not, the rows that symbols of eight leave stay empty, and the others are chains
        // (1024 positions of 150 to 300 equally frequent symbols).
        // From here on the lower half of s_info[claimant] is the symbol's stream entry, the upper half
        // the head of the chain of its further positions.
        // (only claimants of repeated symbols have a count)
        uint32_t more[4] = {0u, 0u, 0u, 0u};
        if (mine > 0) {
            const uint4 v = *reinterpret_cast<const uint4*>(s_info + p0);
            more[0] = v.x; more[1] = v.y; more[2] = v.z; more[3] = v.w;
        }
        const bool claims = (more[0] | more[1] | more[2] | more[3]) != 0u;
        const bool any_claims = __any_sync(0xFFFFFFFFu, claims);
        if (any_claims) {                              // symbols with >= 2, 3, 4 occurrences, ten bits each
            uint32_t occur = 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) occur += (more[k] > 0u ? 1u : 0u) + (more[k] > 1u ? 1u << 10 : 0u) + (more[k] > 2u ? 1u << 20 : 0u);
            occur = __reduce_add_sync(0xFFFFFFFFu, occur) >> (10 * min(lane, 2)) & 0x3FFu;
            if (lane < 3 && occur) atomicAdd(&s_repeats[lane], (int)occur);
        }
        __syncthreads();
        const uint32_t need = s_repeats[0] <= W.row_cap ? 1u : (s_repeats[1] <= W.row_cap ? 2u : (s_repeats[2] <= W.row_cap ? 3u : 7u));
        if (any_claims) {
            int asks = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) asks += more[k] >= need;
            int row = asks;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int up = __shfl_up_sync(0xFFFFFFFFu, row, d);
                if (lane >= d) row += up;
            }
            int first_row = 0;
            if (lane == 31 && row) first_row = atomicAdd(&s_repeats[3], row);
            row += __shfl_sync(0xFFFFFFFFu, first_row, 31) - asks;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (more[k] == 0u) continue;
                uint32_t code = (kChainEnd << 16) | kLocChain | (uint32_t)(p0 + k);
                if (more[k] >= need) {
                    if (row < W.row_cap) code = kLocRow | (uint32_t)row;
                    ++row;
                }
                s_map[my_name[k]] = (uint16_t)code;             // what the streams of the texts say
                s_info[p0 + k] = code;
            }
            if ((need == 2u || need == 3u) && (kThreads != kTwoWarpThreads || K >= kHandOut)) {
                constexpr auto hand_out = kPairs || kDecide ? hand_out_rest_apart : hand_out_rest;
                hand_out(make_uint4(more[0], more[1], more[2], more[3]), make_uint2(my_name[0] | (my_name[1] << 16), my_name[2] | (my_name[3] << 16)),
                         need, s_repeats, W.row_cap, s_map, s_info + p0);
            }
        }
        __syncthreads();
        uint32_t* rows = kPairs ? s_rows : reinterpret_cast<uint32_t*>(ws + W.off_rows) + ((size_t)g * M + i) * W.rows_pitch;
        const int n_rows = min(s_repeats[3] + s_repeats[4], W.row_cap);
        const bool later = kDecide && !kPairs && W.rows_later;
        for (int e = tid; !later && 4 * e < n_rows * W.row_words; e += nthr) {
            reinterpret_cast<uint4*>(rows)[e] = make_uint4(0u, 0u, 0u, 0u);
            if (kPairs) reinterpret_cast<uint4*>(rows + W.rows_pitch)[e] = make_uint4(0u, 0u, 0u, 0u);
        }
        if (!later) __syncthreads();
        uint32_t my_row[4] = {kLocNone, kLocNone, kLocNone, kLocNone};
        if (claims || repeated) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (more[k] == 0u && my_first[k] == (uint32_t)(p0 + k)) continue;
                const uint32_t p = p0 + k, f = my_first[k], info = s_info[f];
                if ((info & kLocChain) == kLocChain) {
                    if (f != p) s_info[p] = atomicExch(&s_info[f], (p << 16) | kLocChain | f);
                } else if (later) {
                    my_row[k] = info & 0xFFFFu;
                } else {
                    uint32_t* row = rows + (info & 0x3FFFu) * W.row_words;
                    atomicOr(row + (p >> 5), 1u << (p & 31));
                    if (kPairs) atomicOr(row + W.rows_pitch + W.row_words - 1 - (p >> 5), 0x80000000u >> (p & 31));
                }
            }
        }
        if (later && mine > 0) reinterpret_cast<uint2*>(rows + 4)[tid] = make_uint2(my_row[0] | (my_row[1] << 16), my_row[2] | (my_row[3] << 16));
        if (!kPairs && s_repeats[0] > n_rows) {        // some chains: leave them for the recurrence
            __syncthreads();
            uint16_t* g_next = reinterpret_cast<uint16_t*>(ws + W.off_next) + ((size_t)g * M + i) * W.pitch;
            for (int p = tid; p < m; p += nthr) g_next[p] = (uint16_t)(s_info[p] >> 16);
        }
    }
    const bool named = s_repeats[0] > 0;
    if (named) __syncthreads();                       // the map's entries are final

    // Match streams of all texts, four columns per lane and trip: one 8-byte load of names, four
    // look-ups, one 8-byte store.  As many warps to a text as there are for each (chunks dealt to all
    // warps in turn would be even, but then every warp sets up every text).
    uint16_t* locs = reinterpret_cast<uint16_t*>(ws + W.off_loc);
    const int per_text = W.text_warps, warp = tid >> 5, first_text = per_text > 1 ? (int)__umulhi((uint32_t)warp, W.inv_text_warps) : warp;
    const int part = warp - first_text * per_text;
    for (int t = first_text; t < ntxt; t += W.text_stride) {
        if (s_cp[t] < 0) continue;
        const int n = s_len[t];
        const uint2* in = reinterpret_cast<const uint2*>(names + s_txt[t] * W.pitch);
        const uint2* own = reinterpret_cast<const uint2*>(pat);
        uint2* out = reinterpret_cast<uint2*>(kPairs ? s_loc + t * W.pitch : locs + s_stream[t]);
        uint32_t differ = 0u, absent = 0u, seen = 0u;
        for (int q = ((s_cp[t] & ~31) >> 2) + 32 * part + lane; 4 * q < n; q += 32 * per_text) {
            const int left = n - 4 * q;                // columns of this quad that exist
            const uint2 v = in[q], o = own[q];         // past the pattern's end: still in the group's names or the rows after them
            uint32_t w0 = s_map[v.x & 0xFFFFu] | ((uint32_t)s_map[v.x >> 16] << 16);
            uint32_t w1 = s_map[v.y & 0xFFFFu] | ((uint32_t)s_map[v.y >> 16] << 16);
            // positions below both lengths whose symbol is not the pattern's symbol at the same place
            // (names have 15 bits: the sum of a half does not reach the other)
            uint32_t d0 = ((v.x ^ o.x) + 0x7FFF7FFFu) & 0x80008000u, d1 = ((v.y ^ o.y) + 0x7FFF7FFFu) & 0x80008000u;
            const int both = m - 4 * q;                // columns of this quad below the pattern's length
            if (left < 4 || both < 4) {
                const int k = min(left, both);
                d0 = k > 1 ? d0 : (k == 1 ? d0 & 0xFFFFu : 0u);
                d1 = k > 3 ? d1 : (k == 3 ? d1 & 0xFFFFu : 0u);
                // The last quad of a text is filled up with symbols of their own that the pattern is
                // extended by as well: a common suffix leaves the distance as it is, and the recurrence
                // always runs whole quads, whose four columns the compiler can then interleave.
                if (left == 1) w0 = (w0 & 0xFFFFu) | ((uint32_t)m << 16);
                if (left == 1) w1 = (uint32_t)(m + 1) | ((uint32_t)(m + 2) << 16);
                if (left == 2) w1 = (uint32_t)m | ((uint32_t)(m + 1) << 16);
                if (left == 3) w1 = (w1 & 0xFFFFu) | ((uint32_t)m << 16);
            }
            out[q] = make_uint2(w0, w1);
            seen |= w0 | w1;
            differ += __popc(d0) + __popc(d1);
            // columns without any match, 0x7FFF: the only entries with bit 14 and without bit 15
            absent += __popc(w0 & ~(w0 >> 1) & 0x40004000u) + __popc(w1 & ~(w1 >> 1) & 0x40004000u);
        }
        const uint32_t count = __reduce_add_sync(0xFFFFFFFFu, differ + (absent << 16));
        const bool row = __any_sync(0xFFFFFFFFu, (seen & (kLocRow * 0x10001u)) != 0u);
        if (lane == 0) {
            if (count) atomicAdd(&s_count[t], count);
            if (row) s_flag[t] = 1u;
        }
    }
    __syncthreads();
    // Bounds of a pair's distance.  Upper: substitute the differing positions, insert or delete the rest.  Lower:
    // every text column without a match costs an edit, and if the pattern is at least as long as the text,
    // m - n rows are deleted besides.
    auto bounds = [&](int t, int strip, int& lower, int& upper) {
        const int n = s_len[t];
        lower = upper = abs(m - n);                   // one prefix starts the other (or is empty)
        if (strip < 0) return;
        const int absent = (int)(s_count[t] >> 16);
        lower = m >= n ? m - n + absent : max(n - m, absent);
        upper += (int)(s_count[t] & 0xFFFFu);
    };
    // The removed prefix is a multiple of four symbols (the match stream is read in 8-byte
    // quads), and of 32 where the stream refers to mask rows (whose words start there).
    auto removed = [&](int t) { return s_cp[t] < 0 ? -1 : (s_cp[t] & (s_flag[t] ? ~31 : ~3)); };
    if constexpr (kPairs) {
        constexpr int kWarps = (kThreads > kMostPrepThreads ? kThreads : kMostPrepThreads) / 32;
        __shared__ uint4 s_differ[kWarps][kSpans];
        __shared__ uint32_t s_entries[kWarps][kMostMatches];
        __shared__ int s_dist[kMaxTexts];              // the distance, or -1: to be computed
        auto settle = [&](int t, int d) {
            const int pair = pair_index(min(i, s_txt[t]), max(i, s_txt[t]), N);
            if (kCluster) *cluster.map_shared_rank(s_all_dist + pair, 0) = d;
            if (!kCluster || a.pair_dist) dist_out[(size_t)g * P + pair] = d;
        };
        auto finish = [&]() {
            if constexpr (kCluster) {
                cluster.sync();
                if (i == 0) evaluate_group(a, g, exact, [&](int e) { return s_all_dist[e]; }, [&](int r) { return s_all_len[r]; });
            } else if (arrive_last(M, reinterpret_cast<int32_t*>(ws + W.off_order) + g)) {
                evaluate_group(a, g, exact, [&](int e) { return __ldcg(dist_out + (size_t)g * P + e); },
                               [&](int r) { bool negative = false; return clamp_len(a.lens, (size_t)g * N + r, K, negative); });
            }
        };
        if (kCluster) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        // first what the bounds and few matches settle
        for (int t = warp; t < ntxt; t += warps) {
            const int n = s_len[t], strip = removed(t);
            int lower, upper;
            bounds(t, strip, lower, upper);
            int d = lower < upper ? -1 : lower;
            if (kDecide) {                             // bounds first; few matches are no cheaper than what follows
                if (lane == 0) {
                    const int pair = pair_index(min(i, s_txt[t]), max(i, s_txt[t]), N);
                    *cluster.map_shared_rank(s_all_upper + pair, 0) = upper;
                    if (d < 0) settle(t, lower);
                }
            } else if (d < 0 && upper - lower <= kMostMatches && few_repeats(s_repeats[0], m) && n + m - 2 * strip > kWorthMatches) {
                __syncwarp();
                const int count = find_matches<true>(reinterpret_cast<const uint2*>(s_loc + t * W.pitch), reinterpret_cast<const uint2*>(names + s_txt[t] * W.pitch),
                                                     reinterpret_cast<const uint2*>(pat), m, n, strip, s_differ[warp], s_entries[warp]);
                if (count == 0) d = upper;
                else if (count <= kMostMatches)
                    d = distance_by_matches<true>(s_entries[warp], count, s_differ[warp], s_rows, W.row_words, m, n, strip, upper);
            }
            if (lane == 0) {
                s_dist[t] = d;
                if (d >= 0) settle(t, d);
            }
        }
        if constexpr (kDecide) {
            cluster.sync();
            if (i == 0) {
                const int settled = settle_group(a, g, exact, s_all_dist, s_all_upper, s_all_len);
                if (tid < M) *cluster.map_shared_rank(&s_settled, tid) = settled;
            }
            cluster.sync();
            if (s_settled) return;
        }
        __syncthreads();
        // Teams of as many lanes as the pattern has blocks, 16 at the most, and as many pairs to a warp as have room.
        const bool chains = s_repeats[0] > min(s_repeats[3] + s_repeats[4], W.row_cap);
        const uint32_t* turned = s_rows + W.rows_pitch;
        uint4* s_wide = reinterpret_cast<uint4*>(s_map);              // the map is not needed any more
        if constexpr (kTwoWarps) {
            const int t = warp >> 1;
            if (t < ntxt && s_dist[t] < 0) {
                const int n = s_len[t], strip = removed(t), high = (m + (-n & 3) - strip + 31) >> 5;
                const uint16_t* loc = s_loc + t * W.pitch;
                uint4* wide = s_wide + t * ((W.pitch + 8) >> 2);
                const int d = high <= 32 ? distance_from_both_ends<1, true>(loc, wide, s_rows, turned, W.row_words, s_info, chains, true, m, n, strip, 1 + t, two)
                                         : distance_from_both_ends<2, true>(loc, wide, s_rows, turned, W.row_words, s_info, chains, true, m, n, strip, 1 + t, two);
                if ((tid & 63) == 0) settle(t, d);
            }
            finish();
            return;
        }
        const int blocks = (m + 3 + 31) >> 5, tlog = min(32 - __clz(max(blocks, 1) - 1), 4), share = 16 >> tlog;
        for (int t0 = warp * share; t0 < ntxt; t0 += warps * share) {
            const int t = min(t0 + (lane >> (tlog + 1)), ntxt - 1);
            const bool live = t0 + (lane >> (tlog + 1)) < ntxt && s_dist[t] < 0;
            if (!__any_sync(0xFFFFFFFFu, live)) continue;
            const int n = s_len[t], strip = live ? removed(t) : 0;
            const uint16_t* loc = s_loc + t * W.pitch;
            // (lanes without a text share two quads of their own)
            uint4* wide = s_wide + (t0 + (lane >> (tlog + 1)) < ntxt ? t * ((W.pitch + 8) >> 2) : (N * (W.pitch + 8)) >> 3);
            const int high = __reduce_max_sync(0xFFFFFFFFu, live ? (m + (-n & 3) - strip + 31) >> 5 : 0);
            int d;
            if (high <= 16) d = distance_from_both_ends<1>(loc, wide, s_rows, turned, W.row_words, s_info, chains, live, m, n, strip, tlog, two);
            else if (high <= 32) d = distance_from_both_ends<2>(loc, wide, s_rows, turned, W.row_words, s_info, chains, live, m, n, strip, tlog, two);
            else d = distance_from_both_ends<3>(loc, wide, s_rows, turned, W.row_words, s_info, chains, live, m, n, strip, tlog, two);
            if (live && (lane & ((2 << tlog) - 1)) == 0) settle(t, d);
        }
        finish();
        return;
    }
    if (tid >= 32) return;                             // descriptors: the texts' threads are in the first warp
    if (kDecide && W.rows_later && tid == 0)
        reinterpret_cast<uint32_t*>(ws + W.off_rows)[((size_t)g * M + i) * W.rows_pitch] = (uint32_t)min(s_repeats[3] + s_repeats[4], W.row_cap) | ((uint32_t)m << 16);
    PairDesc* descs = reinterpret_cast<PairDesc*>(ws + W.off_desc);
    Ctl* ctl = reinterpret_cast<Ctl*>(ws + W.off_ctl);
    int work = 0, few = -1, maybe = -1;
    if (tid < ntxt) {
        const int j = s_txt[tid], n = s_len[tid];
        const int strip = removed(tid);
        const size_t idx = (size_t)g * P + pair_index(min(i, j), max(i, j), N);
        int lower, upper;
        bounds(tid, strip, lower, upper);
        PairDesc d{(uint32_t)m | ((uint32_t)n << 16), (uint32_t)(g * M + i), 0u, (uint32_t)lower | ((uint32_t)upper << 16)};
        if (lower < upper) {                          // otherwise that is the distance
            const int n_rows = min(s_repeats[3] + s_repeats[4], W.row_cap);
            d.bin = ((uint32_t)strip << kStripShift) | ((uint32_t)n_rows << kRowsShift) | kNeedsDp | (s_repeats[0] > n_rows ? kHasChains : 0u);
        }
        descs[idx] = d;
        if (kDecide || lower == upper) dist_out[idx] = lower;
        if (lower < upper) {
            const PairSize z = size_of_desc(d);
            work = work_of_pair(z.m, z.n, z.lb, z.ub);
            if (!kDecide && !W.alone && upper - lower <= kMostMatches && few_repeats(s_repeats[0], m)) {
                if (worth_listing(upper - lower, s_repeats[0], (int)(s_count[tid] & 0xFFFFu), min(m, n) - strip, work)) {
                    few = (int)idx;
                    descs[idx].bin = d.bin | kListed;
                } else if (upper - lower <= kFewColumns) {
                    maybe = (int)idx;
                }
            }
        }
    }
    if (kDecide || W.alone) return;                   // counted later: what the bounds leave; by the CTA that orders the batch
    int32_t* list = reinterpret_cast<int32_t*>(ws + W.off_order);
    auto note = [&](bool here, int32_t* count, unsigned long long* sum) {     // the place of this thread's pair among those noted
        const unsigned all = __ballot_sync(0xFFFFFFFFu, here);
        if (all == 0u) return 0;
        const int lane_time = __reduce_add_sync(0xFFFFFFFFu, here ? work : 0);
        int at = 0;
        if (tid == 0) {
            at = atomicAdd(count, __popc(all));
            atomicAdd(sum, (unsigned long long)lane_time);
        }
        return __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(all & ((1u << tid) - 1u));
    };
    const int at_few = note(few >= 0, &ctl->few, &ctl->few_work), at_maybe = note(maybe >= 0, &ctl->maybe, &ctl->maybe_work);
    if (few >= 0) list[at_few] = few;
    if (maybe >= 0) list[a.n_groups * P - 1 - at_maybe] = maybe;
    note(work > 0 && few < 0 && maybe < 0, &ctl->open, &ctl->work);
}

// ----------------------------------------------------------------------- order
// Exclusive prefix sum over the kOrderThreads threads of a CTA (one value per thread).
__device__ __forceinline__ int block_exclusive_scan(int v, int* s_part /* [32] */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int up = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += up;
    }
    if (lane == 31) s_part[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int w = s_part[lane];
        int wi = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int up = __shfl_up_sync(0xFFFFFFFFu, wi, d);
            if (lane >= d) wi += up;
        }
        s_part[lane] = wi - w;
    }
    __syncthreads();
    const int r = incl - v + s_part[warp];
    __syncthreads();                       // s_part may be reused at once
    return r;
}

// The longest a task should take: about what every resident warp has to do on average, so
// that none is still running long after the others (measured best among 0.6, 1.25 and 2.5 times
// on token-level batches of 1024 groups).  And how many lanes there are to a pair.
__device__ __forceinline__ ShapeGoal shape_goal(unsigned long long work, int open, int warps) {
    const float lanes = 32.0f * (float)warps;
    return ShapeGoal{1.25f * (float)work / lanes, lanes / (float)max(open, 1)};
}

// The first `bin_blocks` CTAs: every pair's shape and bin, and the bin counts.  The warps of the others go through the listed
// pairs, as many places apart as there are of them, and bin those with too many matches themselves.  (In one launch:
// a text, for which little or nothing is listed, does not wait for another one: 150 groups of 16 texts of 700 that differ in
// 2 % of their places 138 -> 134 us, 3000 of 8 ragged ones of 100 119 -> 117.  None are listed
// in decide mode: most pairs' groups are dismissed by their bounds.)
// Pairs that are not worth it by themselves are looked at if no pair has to go to the recurrence: the batch is then done
// here as a rule, and the latency of what comes after it is more than they cost (1024 groups of uniform tokens: 122 us, 142
// without these).  What fails then is shaped as if one in eight did.
// Decide mode: most groups are dismissed by their bounds before anyone reads a mask row, so prep leaves the rows of their positions
// (16 bits each, behind the number of rows and positions) where the rows will be, and the other CTAs make those of open groups
// (1024 groups of 8 texts of 1024 at 0.12: 218.6 -> 210.0 us, of which 156 are open; all settled 106 -> 98; all open 165 -> 169; K <= 256
// no gain).  From K = 257 on the rows' place has room for the list.
constexpr int kBinPairs = 32 * kMatchWarps;               // pairs that a CTA bins

// A warp: the mask rows of a pattern in place of its positions' rows.
__device__ __noinline__ void make_rows(uint32_t* rows, int row_words) {
    const int lane = threadIdx.x & 31, n_rows = (int)(rows[0] & 0xFFFFu), m = (int)(rows[0] >> 16);
    constexpr int kTrips = SR_MAX_K / 128;
    uint2 v[kTrips];
#pragma unroll
    for (int t = 0; t < kTrips; ++t) {
        const int q = lane + 32 * t;
        v[t] = n_rows > 0 && 4 * q < m ? reinterpret_cast<const uint2*>(rows + 4)[q] : make_uint2(kLocNone * 0x10001u, kLocNone * 0x10001u);
    }
    __syncwarp();
    for (int e = lane; 4 * e < n_rows * row_words; e += 32) reinterpret_cast<uint4*>(rows)[e] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
#pragma unroll
    for (int t = 0; t < kTrips; ++t) {
        const uint32_t row[4] = {v[t].x & 0xFFFFu, v[t].x >> 16, v[t].y & 0xFFFFu, v[t].y >> 16};
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (row[k] >= kLocRow) atomicOr(rows + (row[k] & 0x3FFFu) * row_words + ((lane + 32 * t) >> 3), 1u << ((4 * (lane + 32 * t) + k) & 31));
    }
}

__global__ void __launch_bounds__(32 * kMatchWarps, 5)
multi_bin_kernel(unsigned char* ws, MultiWs W, int N, int n_pairs, int bin_blocks, int32_t* dist_out, int row_patterns) {
    grid_begin();
    PairDesc* descs = reinterpret_cast<PairDesc*>(ws + W.off_desc);
    Ctl* ctl = reinterpret_cast<Ctl*>(ws + W.off_ctl);
    const bool any = ctl->open != 0;
    auto bin_of = [&](const PairDesc& d) {                   // (the goal anew for each: few need it where registers count)
        const unsigned long long lane_time = any ? ctl->work + ctl->maybe_work : (ctl->few_work + ctl->maybe_work) / 8;
        const ShapeGoal goal = shape_goal(lane_time, any ? ctl->open + ctl->maybe : (ctl->few + ctl->maybe) / 8, W.warps);
        const PairSize z = size_of_desc(d);
        return bin_of_shape(shape_of_pair(z.m, z.n, z.lb, z.ub, goal));
    };
    if ((int)blockIdx.x < bin_blocks) {
        if (!any) return;
        __shared__ int32_t s_hist[kNumBins];
        for (int b = threadIdx.x; b < kNumBins; b += 32 * kMatchWarps) s_hist[b] = 0;
        __syncthreads();
        const int idx = blockIdx.x * kBinPairs + threadIdx.x;
        if (idx < n_pairs) {
            const PairDesc d = descs[idx];
            if ((d.bin & (kNeedsDp | kListed)) == kNeedsDp) {
                const int bin = bin_of(d);
                descs[idx].bin = d.bin | (uint32_t)bin;
                atomicAdd(&s_hist[bin], 1);
            }
        }
        __syncthreads();
        for (int b = threadIdx.x; b < kNumBins; b += 32 * kMatchWarps)
            if (s_hist[b]) atomicAdd(&ctl->hist[b], s_hist[b]);
        return;
    }
    __shared__ uint4 s_differ[kMatchWarps][kSpans];
    __shared__ uint32_t s_entries[kMatchWarps][kMostMatches];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, P = pairs_of(N);
    if (W.rows_later) {
        if (!any) return;
        for (int p = ((int)blockIdx.x - bin_blocks) * kMatchWarps + warp; p < row_patterns; p += ((int)gridDim.x - bin_blocks) * kMatchWarps) {
            int g = W.patterns > 1 ? (int)__umulhi((uint32_t)p, W.inv_patterns) : p;
            if (g * W.patterns > p) --g;
            if ((ws + W.off_flag)[g]) make_rows(reinterpret_cast<uint32_t*>(ws + W.off_rows) + (size_t)p * W.rows_pitch, W.row_words);
        }
        return;
    }
    const int32_t* list = reinterpret_cast<const int32_t*>(ws + W.off_order);
    const int few = ctl->few, all = few + (any ? 0 : ctl->maybe);
    for (int e = ((int)blockIdx.x - bin_blocks) * kMatchWarps + warp; e < all; e += ((int)gridDim.x - bin_blocks) * kMatchWarps) {
        const int idx = list[e < few ? e : n_pairs - 1 - (e - few)];
        const PairDesc d = descs[idx];
        const int upper = (int)(d.lower >> 16);
        int dist = -1;
        const int m = (int)(d.mn & 0xFFFFu), n = (int)(d.mn >> 16), strip = (int)((d.bin >> kStripShift) & 0x3FFu);
        int g = W.patterns > 1 ? (int)__umulhi(d.pat_row, W.inv_patterns) : (int)d.pat_row;
        if (g * W.patterns > (int)d.pat_row) --g;
        const int i = (int)d.pat_row - g * W.patterns;
        const int pr = kPairs.v[N][idx - g * P], j = (pr & 0xFF) + (pr >> 8) - i;
        const uint16_t* names = reinterpret_cast<const uint16_t*>(ws + W.off_names) + (size_t)g * N * W.pitch;
        __syncwarp();                              // the pair before has been read
        const int count = find_matches<false>(reinterpret_cast<const uint2*>(reinterpret_cast<const uint16_t*>(ws + W.off_loc) + (size_t)idx * W.pitch),
                                       reinterpret_cast<const uint2*>(names + j * W.pitch), reinterpret_cast<const uint2*>(names + i * W.pitch),
                                       m, n, strip, s_differ[warp], s_entries[warp]);
        if (count == 0)
            dist = upper;
        else if (count <= kMostMatches)
            dist = distance_by_matches<false>(s_entries[warp], count, s_differ[warp],
                                       reinterpret_cast<const uint32_t*>(ws + W.off_rows) + (size_t)d.pat_row * W.rows_pitch,
                                       W.row_words, m, n, strip, upper);
        if (lane != 0) continue;
        if (dist >= 0) {
            descs[idx].bin = 0u;
            descs[idx].lower = (uint32_t)dist * 0x10001u;
            dist_out[idx] = dist;
        } else {
            const int bin = bin_of(d);
            descs[idx].bin = d.bin | (uint32_t)bin;
            atomicAdd(&ctl->hist[bin], 1);
            atomicAdd(&ctl->failed, 1);
        }
    }
}

__device__ __forceinline__ void sum_and_max(float& sum, float& most) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
        most = fmaxf(most, __shfl_xor_sync(0xFFFFFFFFu, most, d));
    }
}

// Counting sort of the pairs by bin: longest warp tasks first, one team shape and similar
// text lengths per bin.  Every CTA turns the bin counts into bin starts by itself (a scan
// of kNumBins values costs less than a launch) and places kOrderThreads pairs; the first CTA
// also leaves the tables the dp kernel reads.
// kAlone: one CTA sorts the whole batch, and bins it first.
template <bool kAlone>
__global__ void __launch_bounds__(kOrderThreads)
multi_order_kernel(PairDesc* descs, int32_t* order, Ctl* ctl, int n_pairs, int warps) {
    grid_begin();
    __shared__ int s_part[32];
    __shared__ int32_t s_start[kNumBins], s_hist[kNumBins];
    __shared__ unsigned long long s_work;
    __shared__ float s_time[32], s_longest[32];
    __shared__ int s_open;
    const int t = threadIdx.x;
    constexpr int kPer = kAlone ? kAlonePairs / kOrderThreads : 1;
    uint32_t bins[kPer];
    if (kAlone) {
        s_hist[2 * t] = s_hist[2 * t + 1] = 0;
        if (t == 0) { s_work = 0ull; s_open = 0; }
        __syncthreads();
        PairDesc d[kPer];
        int work = 0, open = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int idx = k * kOrderThreads + t;
            d[k].bin = 0u;
            if (idx < n_pairs) d[k] = descs[idx];
            if (d[k].bin & kNeedsDp) {
                const PairSize z = size_of_desc(d[k]);
                work += work_of_pair(z.m, z.n, z.lb, z.ub);
                ++open;
            }
        }
        work = __reduce_add_sync(0xFFFFFFFFu, work);
        open = __reduce_add_sync(0xFFFFFFFFu, open);
        if ((t & 31) == 0 && open) {
            atomicAdd(&s_work, (unsigned long long)work);
            atomicAdd(&s_open, open);
        }
        __syncthreads();
        const ShapeGoal goal = shape_goal(s_work, s_open, warps);
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            bins[k] = d[k].bin;
            if (d[k].bin & kNeedsDp) {
                const PairSize z = size_of_desc(d[k]);
                const int bin = bin_of_shape(shape_of_pair(z.m, z.n, z.lb, z.ub, goal));
                bins[k] |= (uint32_t)bin;
                atomicAdd(&s_hist[bin], 1);
            }
        }
        __syncthreads();
    } else {
        if (ctl->open == 0 && ctl->failed == 0) {      // bounds and matches have settled the whole batch
            if (blockIdx.x == 0 && t == 0) ctl->task_counter = ctl->total_tasks = 0;
            return;
        }
        s_hist[2 * t] = ctl->hist[2 * t];
        s_hist[2 * t + 1] = ctl->hist[2 * t + 1];
        const int idx = blockIdx.x * kOrderThreads + t;
        bins[0] = idx < n_pairs ? descs[idx].bin : 0u;
    }
    const int own[2] = {s_hist[2 * t], s_hist[2 * t + 1]};
    const int start = block_exclusive_scan(own[0] + own[1], s_part);
    s_start[2 * t] = start;
    s_start[2 * t + 1] = start + own[0];
    if (kAlone || blockIdx.x == 0) {
        // warp tasks per bin (32 / T pairs per task), exclusive prefix over the bins
        int tasks[2];
        float time = 0.0f, longest = 0.0f;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            int tl, rr;
            shape_of_class((2 * t + k) % kNumClasses, tl, rr);
            const int tpw = 32 >> tl;
            tasks[k] = (own[k] + tpw - 1) >> (5 - tl);
            if (tasks[k] == 0) continue;
            const float each = time_of_bucket((2 * t + k) / kNumClasses);
            time += each * (float)tasks[k];
            longest = fmaxf(longest, each);
        }
        // (in a fixed order: the same batch is run the same way every time)
        sum_and_max(time, longest);
        if ((t & 31) == 0) { s_time[t >> 5] = time; s_longest[t >> 5] = longest; }
        const int task_start = block_exclusive_scan(tasks[0] + tasks[1], s_part);
        ctl->start[2 * t] = start;
        ctl->start[2 * t + 1] = start + own[0];
        ctl->task_start[2 * t] = task_start;
        ctl->task_start[2 * t + 1] = task_start + tasks[0];
        if (kAlone) { ctl->hist[2 * t] = own[0]; ctl->hist[2 * t + 1] = own[1]; }
        if (t >= kOrderThreads - 32) {
            time = s_time[t & 31];
            longest = s_longest[t & 31];
            sum_and_max(time, longest);
        }
        if (t == kOrderThreads - 1) {
            ctl->task_start[kNumBins] = task_start + tasks[0] + tasks[1];
            ctl->total_tasks = task_start + tasks[0] + tasks[1];
            ctl->task_counter = 0;
            ctl->alike = longest >= kLongTask && time >= 0.6f * longest * (float)(task_start + tasks[0] + tasks[1]);
        }
    }
    if (!kAlone) {
        // The CTA's pairs of a bin stay together: pairs of a group read the same mask rows and streams, and what runs
        // side by side finds them in L1 and L2 (a global atomic to every pair, which
        // mixes the CTAs' pairs: 1024 groups that differ in 2 % of their places, over 3000 symbols 798 us, 664 with this, texts 433 and
        // 395; 8000 groups of diverging texts of 48 375 and 232).
        s_hist[2 * t] = s_hist[2 * t + 1] = 0;
        __syncthreads();
        const bool needs = bins[0] & kNeedsDp;
        const int bin = (int)(bins[0] & kBinMask);
        const int rank = needs ? atomicAdd(&s_hist[bin], 1) : 0;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (s_hist[2 * t + k]) s_start[2 * t + k] += atomicAdd(&ctl->fill[2 * t + k], s_hist[2 * t + k]);
        __syncthreads();
        if (needs) order[s_start[bin] + rank] = blockIdx.x * kOrderThreads + t;
        return;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if (!(bins[k] & kNeedsDp)) continue;
        order[atomicAdd(&s_start[bins[k] & kBinMask], 1)] = k * kOrderThreads + t;
    }
}

// -------------------------------------------------------------------------- dp
// Brings `bytes` bytes to L1, 32 a time, `lanes` lanes together.  (Not inlined: it is run once a task.)
__device__ __noinline__ void touch(const void* from, int bytes, int lane, int lanes) {
    for (int o = 32 * lane; o < bytes; o += 32 * lanes) {
        asm volatile("{ .reg .u32 x; ld.global.nc.u32 x, [%0]; }" ::"l"(static_cast<const char*>(from) + o));
    }
}

// Loads a lane's R words of a mask row where `p` is set, without a branch: the recurrence around
// it stays one block of straight-line code.
template <int R>
__device__ __forceinline__ void load_row_if(uint32_t p, const uint32_t* row, uint32_t (&Eq)[R]) {
    static_assert(R >= 1 && R <= 4, "");
    if constexpr (R == 1)
        asm("{ .reg .pred p; setp.ne.u32 p, %1, 0; @p ld.global.nc.u32 %0, [%2]; }" : "+r"(Eq[0]) : "r"(p), "l"(row));
    else if constexpr (R == 2)
        asm("{ .reg .pred p; setp.ne.u32 p, %2, 0; @p ld.global.nc.u32 %0, [%3]; @p ld.global.nc.u32 %1, [%3 + 4]; }"
            : "+r"(Eq[0]), "+r"(Eq[1]) : "r"(p), "l"(row));
    else if constexpr (R == 3)
        asm("{ .reg .pred p; setp.ne.u32 p, %3, 0; @p ld.global.nc.u32 %0, [%4]; @p ld.global.nc.u32 %1, [%4 + 4]; "
            "@p ld.global.nc.u32 %2, [%4 + 8]; }"
            : "+r"(Eq[0]), "+r"(Eq[1]), "+r"(Eq[2]) : "r"(p), "l"(row));
    else
        asm("{ .reg .pred p; setp.ne.u32 p, %4, 0; @p ld.global.nc.u32 %0, [%5]; @p ld.global.nc.u32 %1, [%5 + 4]; "
            "@p ld.global.nc.u32 %2, [%5 + 8]; @p ld.global.nc.u32 %3, [%5 + 12]; }"
            : "+r"(Eq[0]), "+r"(Eq[1]), "+r"(Eq[2]), "+r"(Eq[3]) : "r"(p), "l"(row));
}

// Match words of a text column for the R blocks a lane owns.  A position becomes a
// one-hot word; an entry that names a mask row is read from it (`words` points at the lane's
// first word of the pattern's first row).
template <int R>
__device__ __forceinline__ void match_words(uint32_t loc, uint32_t rowbase, const uint32_t* __restrict__ words,
                                            int row_words, uint32_t (&Eq)[R]) {
    const uint32_t d0 = loc - rowbase;
#pragma unroll
    for (int r = 0; r < R; ++r) Eq[r] = shl_clamp(1u, d0 - 32u * r);     // 0 for rows and chains
    load_row_if<R>((loc & kLocChain) == kLocRow, words + (loc & 0x3FFFu) * (uint32_t)row_words, Eq);
}

// The columns of a quad whose symbol is left as a chain of positions: walk it.
template <int R>
__device__ __forceinline__ void add_chains(uint2 q, uint32_t rowbase, const uint16_t* __restrict__ nxt, uint32_t (&Eq)[4][R]) {
    const uint32_t loc[4] = {q.x & 0xFFFFu, q.x >> 16, q.y & 0xFFFFu, q.y >> 16};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (loc[u] < kLocChain) continue;
        uint32_t p = loc[u] & 0x3FFFu;
        for (int hop = 0; hop < SR_MAX_K && p < (uint32_t)SR_MAX_K; ++hop) {   // a chain ends at 0xFFFF
            const uint32_t dd = p - rowbase;
#pragma unroll
            for (int r = 0; r < R; ++r) Eq[u][r] |= shl_clamp(1u, dd - 32u * r);
            p = __ldg(nxt + p);
        }
    }
}

// A warp task: 32/T teams of T lanes, one pair per team.  The pattern's blocks are grouped in
// stripes of R blocks, stripe g on lane g mod T.  Lanes are skewed by one QUAD of text columns:
// in iteration j stripe g works on columns 4(j-g) .. 4(j-g)+3.  The four
// columns are unrolled, so (a) a lane fetches its four stream entries with one
// 8-byte load, ahead of their use, (b) the deltas a lane needs from the stripe
// above (one +1 and one -1 bit per column, packed in two words) were produced a whole
// iteration earlier, so the shuffles never wait, and (c)
// the blocks of consecutive columns overlap in the pipeline.
//
// Where the team has a lane for every stripe, each runs over all columns.  Otherwise (G > T) the
// lanes form a ring that follows the band of the pair's bound: a stripe is run over the quads in
// which the band crosses it, and when the band has left it its lane takes the stripe T places
// further down, which starts from +1 vertical deltas below the stripe above; a stripe whose upper
// neighbour the band has left takes +1 horizontal deltas from above.  The distance is then the sum
// of the deltas along a path of cells that are all inside the band: down the first column of
// every stripe it enters, along a stripe's bottom row until the next stripe begins, at the end less the
// vertical deltas of the rows beyond the pattern's end.  A result above the pair's bound is
// reported as bound + 1 with kCappedFlag.
// (Not inlined on purpose: as separate functions the instantiations are
// scheduled independently, which measured 8 % faster than one merged kernel body.)
template <int R>
__device__ __noinline__ void dp_task(int tlog, int pos, bool valid, const PairDesc* descs,
                                        const int32_t* order, const uint16_t* locs,
                                        const uint16_t* nexts, const uint32_t* masks, MultiWs W,
                                        int32_t* dist_out, uint32_t two) {
    const int lane = threadIdx.x & 31;
    const int T = 1 << tlog;
    const int lt = lane & (T - 1);
    const int src = (lane & ~(T - 1)) | ((lt - 1) & (T - 1));      // the lane of the stripe above
    // m, n: rows and columns left after the common prefix of `strip` symbols, which neither
    // side runs through
    bool chains = false;
    int n_rows = 0;
    int idx = 0, m = 0, n = 0, strip = 0, lb = 0, ub = 0;
    const uint2* loc4 = reinterpret_cast<const uint2*>(locs);
    const uint16_t* nxt = nexts;
    const uint32_t* rows = masks;
    if (valid) {
        idx = order[pos];
        const PairDesc d = descs[idx];
        strip = (int)((d.bin >> kStripShift) & 0x3FFu);
        chains = d.bin & kHasChains;
        n_rows = (int)((d.bin >> kRowsShift) & 0xFFu);
        n = (int)(d.mn >> 16) - strip;
        m = (int)(d.mn & 0xFFFFu) - strip + (-n & 3);  // both extended to whole quads of columns
        n = (n + 3) & ~3;
        lb = (int)(d.lower & 0xFFFFu);
        ub = (int)(d.lower >> 16);
        // rows are 16-byte aligned and strip is a multiple of 4 entries: 8-byte loads
        loc4 = reinterpret_cast<const uint2*>(locs + (size_t)idx * W.pitch + strip);
        nxt = nexts + (size_t)d.pat_row * W.pitch;
        rows = masks + (size_t)d.pat_row * W.rows_pitch + (strip >> 5);
    }
    if (T >= 16 && valid) {
        // Few pairs: nothing else hides the latencies of this one, so all that it will read goes to L1 first,
        // the stream and the pattern's mask rows (the recurrence of 16 groups of 8 texts: 74 us, 78 without).
        touch(loc4, 2 * n, lt, T);
        touch(rows, 4 * n_rows * W.row_words, lt, T);
    }
    constexpr int H = 32 * R;                          // rows of a stripe
    const int nq = n >> 2;                             // quads of text columns
    const int G = (m + H - 1) / H;                     // stripes (0: no pair)
    const bool ring = G > T;
    const bool any_ring = __any_sync(0xFFFFFFFFu, ring), any_chains = __any_sync(0xFFFFFFFFu, chains);
    const int iters = __reduce_max_sync(0xFFFFFFFFu, G ? nq + G - 1 : 0);
    // Stripe g crosses the band in columns H g - dhi .. H (g + 1) - 1 - dlo: quads first .. last,
    // before they are clipped to the matrix.
    int dlo = -2 * SR_MAX_K, dhi = 2 * SR_MAX_K;
    if (ring) band_of(m, n, lb, ub, dlo, dhi);
    int g = lt;                                        // the stripe this lane holds
    int first = (H * g - dhi) >> 2, last = (H * (g + 1) - 1 - dlo) >> 2;
    // its first iteration and how many follow, the last iteration in which the stripe above feeds
    // it and in which its bottom row is part of the path, its first pattern position, and
    // where its stream (by iteration) and the mask rows' words begin
    int js, above_until, acc_until;
    uint32_t span, rowbase = (uint32_t)(strip + H * g);
    const uint2* stream = loc4 - g;
    const uint32_t* words = rows + R * g;
    auto enter = [&]() {
        js = max(first, 0) + g;
        span = (uint32_t)(min(last, nq - 1) + g - js);
        above_until = g > 0 ? last - H / 4 + g : -1;
        acc_until = (g == G - 1 ? nq : max(first + H / 4, 0)) + g - 1;
        if (g >= G) { js = 0x40000000; span = 0u; acc_until = -1; }
    };
    enter();
    uint32_t Pv[R], Mv[R];
#pragma unroll
    for (int r = 0; r < R; ++r) { Pv[r] = 0xFFFFFFFFu; Mv[r] = 0u; }
    uint32_t outP = 0u, outM = 0u;                     // deltas leaving the stripe, latest column in bit 0
    int acc = 0;
    const uint2 none = make_uint2(kLocNone | (kLocNone << 16), kLocNone | (kLocNone << 16));
    auto fetch = [&](int j) { return (uint32_t)(j - js) <= span ? __ldg(stream + j) : none; };
    // Match words are asked for kAhead iterations before they are used.  One is not enough for a trip to L2 where lanes hold
    // little of a pattern and an iteration is short: 1024 groups of 8 texts of 1024 that differ in 1 % of their places
    // 366 us, 316 with two; with two for R = 3 and 4 as well diverging ones 312, 338.
    constexpr int kAhead = quads_ahead(R);
    uint32_t words_of[kAhead][4][R];
    uint2 quads[kAhead];
#pragma unroll
    for (int s = 0; s < kAhead; ++s) {
        const uint2 q = fetch(s);
        const uint32_t loc[4] = {q.x & 0xFFFFu, q.x >> 16, q.y & 0xFFFFu, q.y >> 16};
#pragma unroll
        for (int u = 0; u < 4; ++u) match_words<R>(loc[u], rowbase, words, W.row_words, words_of[s][u]);
        if (any_chains) add_chains<R>(q, rowbase, nxt, words_of[s]);
        quads[s] = fetch(kAhead + s);
    }

    // The body is one block of straight-line code, so that the compiler can fill the latencies of
    // one column's chain of operations with the others' and with the next quad's match words:
    // a lane outside its stripe's quads runs along.  Before them it leaves its words alone by
    // itself (no matches, nothing coming in from above: all-ones stay all-ones); after them its
    // words are kept.
    auto step = [&](int j, uint32_t (&Eq)[4][R], uint2& next) {
        const uint2 q = next;                          // the quad kAhead after this one
        next = fetch(j + 2 * kAhead);
        const bool active = (uint32_t)(j - js) <= span;
        // deltas leaving the stripe above for this quad (it worked on it last iteration)
        uint32_t wP = __shfl_sync(0xFFFFFFFFu, outP, src) << 28, wM = __shfl_sync(0xFFFFFFFFu, outM, src) << 28;
        if (j > above_until) { wP = 0xF0000000u; wM = 0u; }    // row 0, or the band left the stripe above: +1 everywhere
        if (!active) wP = wM = 0u;
        uint32_t oldP[R], oldM[R];
#pragma unroll
        for (int r = 0; r < R; ++r) { oldP[r] = Pv[r]; oldM[r] = Mv[r]; }
        const uint32_t loc[4] = {q.x & 0xFFFFu, q.x >> 16, q.y & 0xFFFFu, q.y >> 16};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            uint32_t cP = wP, cM = wM;
            column_step<R>(Eq[u], Pv, Mv, cP, cM, two);
            outP = __funnelshift_l(cP, outP, 1);
            outM = __funnelshift_l(cM, outM, 1);
            wP *= two;                                 // shifts on the FMA pipe
            wM *= two;
            match_words<R>(loc[u], rowbase, words, W.row_words, Eq[u]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) { Pv[r] = active ? Pv[r] : oldP[r]; Mv[r] = active ? Mv[r] : oldM[r]; }
        if (any_chains) add_chains<R>(q, rowbase, nxt, Eq);
        if (any_ring && active) {
            if (ring && j <= acc_until) acc += __popc(outP & 0xFu) - __popc(outM & 0xFu);
            if (g + T < G && (uint32_t)(j - js) == span) {   // the band has left this stripe
                acc += H;
                g += T;
                first += T * (H / 4);
                last += T * (H / 4);
                rowbase += T * H;
                stream -= T;
                words += T * R;
                enter();
#pragma unroll
                for (int r = 0; r < R; ++r) { Pv[r] = 0xFFFFFFFFu; Mv[r] = 0u; }
            }
        }
    };
    // (two copies of the body, so that what is under way stays in its registers; the last may find no quad left)
    for (int j = 0; j < iters; j += kAhead) {
#pragma unroll
        for (int s = 0; s < kAhead; ++s) step(j + s, words_of[s], quads[s]);
    }
    if (!ring) {
        // D[m][n] = n + (sum of the vertical deltas of the last column over rows 1..m)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const uint32_t msk = low_mask(min(max(m - (H * lt + 32 * r), 0), 32));
            acc += __popc(Pv[r] & msk) - __popc(Mv[r] & msk);
        }
        if (lt == 0) acc += n;
    } else if (g < G) {                                // the lane's last stripe
        acc += H;
        if (g == G - 1) {                              // rows past the pattern's end
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const uint32_t past = ~low_mask(min(max(m - (H * g + 32 * r), 0), 32));
                acc -= __popc(Pv[r] & past) - __popc(Mv[r] & past);
            }
        }
    }
    for (int off = 1; off < T; off <<= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
    if (valid && lt == 0) dist_out[idx] = ring && acc > ub ? ((ub + 1) | kCappedFlag) : acc;
}

// Time of `total` tasks that all take as long, in tenths of what one takes of a scheduler's pipe, with so many warps a scheduler:
// full rounds, and what is left, evenly over the schedulers, of which one or two warps do not keep the pipe busy (1024 x 1024
// places on eight lanes of four blocks: four warps on a scheduler 248 us, three 187, two 131, one 96).
__device__ __forceinline__ int rounds_cost(int total, int schedulers, int warps) {
    const int round = schedulers * warps, left = (total % round + schedulers - 1) / schedulers;
    return 10 * (total / round * warps + left) + (left == 1 ? 6 : left == 2 ? 3 : 0);
}

// One CTA an SM, whose warps take the bins' warp tasks, longest first.  The first tasks are dealt out, four to an SM, then four
// more, so that every scheduler has the same number to within one, and neighbours, which run the same code on the same rows,
// are on one SM; the others are pulled.  (All of them pulled, by three CTAs of four warps, up to three ended up on one
// scheduler and none on others: decide mode at 0.12, 1024 groups of 8 texts of 1024, 1044 tasks, 234 -> 219 us; with
// twelve warps the 1796 tasks of 1024 groups over 3000 symbols took two rounds, 671 -> 550 us.)
// Sixteen warps where they hold all tasks.  Where there are more and they take about as long each, twelve or sixteen by
// rounds_cost, sixteen in doubt, for more of them hide more of the trips for rows (7000 groups of 256 over 100 symbols 876 us, 974 with twelve;
// 3000 of uniform tokens with 5 % edits, three rounds of twelve, 240 and 260).  Where they do not, twelve up to twice as many tasks, where few
// rounds end in a tail that is the longer the more warps share a scheduler (1024 groups of diverging ragged texts, 4148 tasks: 299 us, 331 with
// sixteen), sixteen above (6000 of 256 over 100 symbols, 10495 tasks, 806 and 739).
// Tasks that take as long: an SM's warps end a round together, and the first of them to ask took the whole next one, three
// tasks to one scheduler and none to others.  No scheduler has more than its share of the last round (400 groups of 8 uniform
// rollouts of 1024 with inserted and deleted tokens, 2802 tasks: 419 -> 370 us; 700 of texts with 2 % edits, 4906 tasks, 714 -> 648).
// (Over 30 shapes and nine kinds of batch 0.988 of the time without this, at worst 1.03 times it.  The order of
// tasks dealt out to the end, with no pulling: texts 5 to 8 % slower.)
// A CTA starts on an SM that is almost empty, so that tasks dealt to one which waits for another stream's kernel run after the
// others: 1024 groups of texts that differ in 2 % of their places take 307 us, 323 next to matrix products of 2048 places, 392 while sixteen
// SMs are held by a kernel that outlasts the call.  (Three CTAs of four warps, launched when the SMs were empty, took 392 alone, 450 next to the products and
// did not start before the other kernel's end.)
__global__ void __launch_bounds__(kMostDpWarps * 32, 1)
multi_dp_kernel(unsigned char* ws, MultiWs W, int32_t* dist_out, uint32_t two) {
    grid_begin();
    Ctl* ctl = reinterpret_cast<Ctl*>(ws + W.off_ctl);
    const PairDesc* descs = reinterpret_cast<const PairDesc*>(ws + W.off_desc);
    const int32_t* order = reinterpret_cast<const int32_t*>(ws + W.off_order);
    const uint16_t* locs = reinterpret_cast<const uint16_t*>(ws + W.off_loc);
    const uint16_t* nexts = reinterpret_cast<const uint16_t*>(ws + W.off_next);
    const uint32_t* masks = reinterpret_cast<const uint32_t*>(ws + W.off_rows);
    const int lane = threadIdx.x & 31;
    const int total = ctl->total_tasks;
    if (total == 0) return;                           // bounds and matches have settled the batch: 7 groups of 18 of 180, mask alone, 23.1 -> 22.3 us
    const int warp = (int)(threadIdx.x >> 5), most = kMostDpWarps * (int)gridDim.x;
    const bool at_once = total <= most;
    const bool fewer = !at_once && (ctl->alike ? 23 * rounds_cost(total, 4 * (int)gridDim.x, kDpWarps / 4) < 22 * rounds_cost(total, 4 * (int)gridDim.x, kMostDpWarps / 4)
                                               : total <= 2 * most);
    __shared__ int s_last, s_share, s_taken[4];       // first task of the last round, a scheduler's share of it and what each has had
    if (threadIdx.x == 0) {
        const int round = (fewer ? kDpWarps : kMostDpWarps) * (int)gridDim.x, left = ctl->alike ? total % round : 0;
        s_last = total - left;
        s_share = (left + 4 * (int)gridDim.x - 1) / (4 * (int)gridDim.x);
        for (int k = 0; k < 4; ++k) s_taken[k] = 0;
    }
    __syncthreads();
    if (fewer && warp >= kDpWarps) return;
    const int dealt = (fewer ? kDpWarps : kMostDpWarps) * (int)gridDim.x;
    // (Written like this on purpose: with the task kept from round to round, without a shuffle in the first one, or with the pulling
    // in a function of its own the recurrence itself comes out 10 % slower.)
    for (int round = 0;; ++round) {
        int task = 0;
        if (round == 0) task = 4 * ((int)blockIdx.x + (int)gridDim.x * (warp >> 2)) + (warp & 3);
        else if (at_once) task = total;
        else if (lane == 0) {
            // A scheduler that has had its share has done with the rest; the shares add up to no less than the round, and whoever has some
            // left comes back, so that every task is pulled.  (A task of the last round that is met unawares counts as well.)
            const bool ends = s_last < total && dealt + *reinterpret_cast<volatile int32_t*>(&ctl->task_counter) >= s_last;
            task = total;
            if (!ends || atomicAdd(&s_taken[warp & 3], 1) < s_share) {
                task = dealt + atomicAdd(&ctl->task_counter, 1);
                if (!ends && task >= s_last) atomicAdd(&s_taken[warp & 3], 1);
            }
        }
        task = __shfl_sync(0xFFFFFFFFu, task, 0);
        if (task >= total) break;
        int k = 0, hi = kNumBins;                     // last bin whose first task is <= task
        while (hi - k > 1) {
            const int mid = (k + hi) >> 1;
            if (ctl->task_start[mid] <= task) k = mid; else hi = mid;
        }
        int tlog, R;
        shape_of_class(k % kNumClasses, tlog, R);
        const int tpw = 32 >> tlog;
        const int pos = ctl->start[k] + (task - ctl->task_start[k]) * tpw + (lane >> tlog);
        const bool valid = pos < ctl->start[k] + ctl->hist[k];
        switch (R) {
            case 1: dp_task<1>(tlog, pos, valid, descs, order, locs, nexts, masks, W, dist_out, two); break;
            case 2: dp_task<2>(tlog, pos, valid, descs, order, locs, nexts, masks, W, dist_out, two); break;
            case 3: dp_task<3>(tlog, pos, valid, descs, order, locs, nexts, masks, W, dist_out, two); break;
            default: dp_task<4>(tlog, pos, valid, descs, order, locs, nexts, masks, W, dist_out, two); break;
        }
    }
}

// ----------------------------------------------------------------------- bound
// Decide mode.  Per group, d_K evaluated on the pairs' lower bounds, in the same order
// and arithmetic as the real thing: every term is <= the true term and rounded addition
// is monotone, so the result is <= the true d_K.  If it is already not below the
// threshold, the gate's answer is "continue" whatever the exact distances are: the
// group is finished here and its pairs never reach the bit-vector kernel.
// A group the bounds leave open still has a budget: with every other pair at its lower
// bound, pair p can only keep d_K below the threshold while its distance stays at or below
//     cap_p = L_p * (P * d_L - sum of the other pairs' bounded terms)
// (L_p the longer prefix, 1 for raw distances).  The pair's band is cut to that cap (plus a
// margin of two that swamps the rounding of this estimate); a pair whose banded result
// exceeds its cap is reported as "more than the cap", which is all Eq. 2 needs to know.
// mask_only (the caller wants nothing but the mask): a group whose d_K on the pairs' upper bounds, the distances
// along the main diagonal, is below the threshold is cut for certain, and finished here as well.  Converged texts
// reach those bounds: half of the groups that the lower bounds leave open are settled (1024 groups of 8 texts
// of 1024 at 0.12: 262 -> 244 us).
// One thread per pair, gpb groups per CTA (more pairs than threads: several per thread); one
// thread per group for the ordered sums.
constexpr int kGroupThreads = 256;

__global__ void __launch_bounds__(kGroupThreads)
multi_bound_kernel(GateArgs a, PairDesc* descs, Ctl* ctl, uint8_t* flag, uint8_t* exact, int gpb, bool alone, bool mask_only) {
    grid_begin();
    __shared__ double s_term[kMaxPairs], s_above[kMaxPairs], s_sum[kGroupThreads];
    __shared__ int s_lower[kMaxPairs], s_work, s_open;
    const int P = pairs_of(a.N), tid = threadIdx.x;
    const int g0 = blockIdx.x * gpb, ng = min(gpb, a.n_groups - g0);
    PairDesc* d = descs + (size_t)g0 * P;
    if (tid == 0) s_work = s_open = 0;
    for (int e = tid; e < ng * P; e += kGroupThreads) {
        const int m = (int)(d[e].mn & 0xFFFFu), n = (int)(d[e].mn >> 16);
        s_lower[e] = (int)(d[e].lower & 0xFFFFu);
        s_term[e] = pair_term(s_lower[e], m, n, a.norm_mode);        // max(m, n) is symmetric in the roles
        if (mask_only) s_above[e] = pair_term((int)(d[e].lower >> 16), m, n, a.norm_mode);
    }
    __syncthreads();
    if (tid < ng) {
        const int g = g0 + tid;
        double s = 0.0;
        int isum = 0;
        for (int p = 0; p < P; ++p) {
            isum += s_lower[tid * P + p];
            s = __dadd_rn(s, s_term[tid * P + p]);
        }
        const double dk = __ddiv_rn(s, (double)P);
        bool open = dk < a.threshold;                        // the bound alone cannot decide
        if (open && mask_only) {                             // but the upper ones may, by the same argument
            double above = 0.0;
            for (int p = 0; p < P; ++p) above = __dadd_rn(above, s_above[tid * P + p]);
            open = !(__ddiv_rn(above, (double)P) < a.threshold);
        }
        flag[g] = open ? 1 : 0;
        if (exact) exact[g] = open ? 1 : 0;
        s_sum[tid] = open ? s : __longlong_as_double(-1LL);  // NaN: settled
        if (!open) {
            if (a.pair_sum) a.pair_sum[g] = isum;
            if (a.mean) a.mean[g] = dk;
            a.stop[g] = dk < a.threshold ? 1 : 0;            // below: settled from above
        }
    }
    __syncthreads();
    const double budget = (double)P * a.threshold;
    int work = 0, open = 0;
    for (int e = tid; e < ng * P; e += kGroupThreads) {
        PairDesc x = d[e];
        if (!(x.bin & kNeedsDp)) continue;
        const double s = s_sum[e / P];
        if (s != s) {
            d[e].bin = x.bin & ~kNeedsDp;
            continue;
        }
        const int m = (int)(x.mn & 0xFFFFu), n = (int)(x.mn >> 16), lb = s_lower[e];
        const double longer = a.norm_mode == SR_NORM_NONE ? 1.0 : (double)max(m, n);
        const double room = (budget - (s - s_term[e])) * longer;
        // room < 2^31 here: an open group has s < budget, so room <= (budget + term) * longer
        const int ub = min((int)(x.lower >> 16), max(lb, (int)fmin(room, 1.0e9)) + 2);
        x.lower = (uint32_t)lb | ((uint32_t)ub << 16);
        d[e].lower = x.lower;
        const PairSize z = size_of_desc(x);
        work += work_of_pair(z.m, z.n, z.lb, z.ub);
        ++open;
    }
    if (open) {
        atomicAdd(&s_work, work);
        atomicAdd(&s_open, open);
    }
    __syncthreads();
    if (tid == 0 && s_open && !alone) {
        atomicAdd(&ctl->work, (unsigned long long)s_work);
        atomicAdd(&ctl->open, s_open);
    }
}

// ---------------------------------------------------------------------- finish
// One thread per pair turns its distance into a term of d_K (the loads and divisions of a
// group run side by side); one thread per group then adds the terms in pair order.
__global__ void __launch_bounds__(kGroupThreads)
multi_finish_kernel(GateArgs a, int32_t* dist, const uint8_t* flag, uint8_t* exact, int gpb) {
    grid_begin();
    __shared__ double s_term[kMaxPairs];
    __shared__ int32_t s_dist[kMaxPairs];
    const int N = a.N, P = pairs_of(N), tid = threadIdx.x;
    const int g0 = blockIdx.x * gpb, ng = min(gpb, a.n_groups - g0);
    for (int e = tid; e < ng * P; e += kGroupThreads) {
        const int g = e / P, pr = kPairs.v[N][e - g * P];
        bool neg = false;
        const int mi = clamp_len(a.lens, (size_t)(g0 + g) * N + (pr & 0xFF), a.K, neg);
        const int mj = clamp_len(a.lens, (size_t)(g0 + g) * N + (pr >> 8), a.K, neg);
        // decide mode marks a distance beyond its pair's cap: the value is then a lower bound
        const int raw = dist[(size_t)g0 * P + e];
        const int d = raw & ~kCappedFlag;
        if (raw != d) dist[(size_t)g0 * P + e] = d;
        s_dist[e] = raw;
        s_term[e] = pair_term(d, mi, mj, a.norm_mode);
    }
    __syncthreads();
    if (tid >= ng) return;
    const int g = g0 + tid;
    if (flag && flag[g] == 0) return;                        // decided from the bounds
    double s = 0.0;
    int isum = 0, capped = 0;
#pragma unroll 4
    for (int p = 0; p < P; ++p) {
        s = __dadd_rn(s, s_term[tid * P + p]);
        isum += s_dist[tid * P + p] & ~kCappedFlag;
        capped |= s_dist[tid * P + p] & kCappedFlag;
    }
    const double dk = __ddiv_rn(s, (double)P);
    if (a.pair_sum) a.pair_sum[g] = isum;
    if (a.mean) a.mean[g] = dk;
    a.stop[g] = dk < a.threshold ? 1 : 0;
    if (capped && exact) exact[g] = 0;                       // some distances are lower bounds
}

// The longest prefixes for which a team has no more than eight lanes there, and two pairs a warp.
constexpr int kMostEightLanes = 253;

// Which batches take every pair from both ends instead of sorting the pairs into warp tasks: those whose work leaves the SMs
// idle anyway.  Whole matrices are run there and bands in the other place, so the line lies where the batches that have the
// narrowest bands stop to gain (pairs with 2 % of their places substituted, or 5 % edited, of texts, uniform tokens, 3000 and 100
// symbols, and diverging texts, 2676 shapes of 2 to 32 rollouts and K = 33 to 1024; diverging batches would gain up to twice as
// many groups).  It falls with the lanes that a pair takes (up to 8, 16, 16 of two blocks), and where a CTA has only one text or
// two for its warps.  In the last fifth before the line the worst kind of
// batch takes 0.86 of the time it takes sorted, 1.05 at most, all kinds 0.74.
// With more than eight texts to a pattern a pair of 16 lanes waits for others of its CTA: then while there are SMs for
// all CTAs, or half of them (K <= 512).
// The decide mode does so for groups of up to eight, whose CTAs are a cluster that sums up the bounds first; clusters
// of three fit an SM's share worst, and the sorted way has fewer pairs to run.
bool runs_in_pairs(int n_groups, int N, int K, int sms, bool decide) {
    const long long n_pairs = (long long)n_groups * pairs_of(N), ctas = (long long)n_groups * (N & 1 ? N : N - 1);
    const int texts = N >> 1, lanes = K <= (texts == 1 ? 128 : kMostEightLanes) ? 0 : K <= 512 ? 1 : 2;
    if (decide) {
        constexpr int kMost[kMostOwnPatterns + 1][3] = {{}, {}, {4500, 1000, 1000}, {1000, 1000, 500}, {2400, 2400, 1000}, {2400, 2400, 1000},
                                                        {3500, 1900, 1700}, {3500, 1900, 1700}, {3500, 3200, 2100}};
        return N <= kMostOwnPatterns && n_pairs <= 7000 && n_pairs * (K + 384) <= 1000LL * kMost[N][lanes];
    }
    if (texts > 8 && lanes > 0) return ctas <= (lanes == 1 ? 2 : 1) * sms;
    constexpr int kMost[5][3] = {{4500, 1400, 1000}, {4500, 3900, 2900}, {6400, 3900, 2500}, {6400, 4200, 3400}, {4200, 0, 0}};
    return n_pairs * (K + 384) <= 1000LL * kMost[texts <= 3 ? texts - 1 : texts <= 8 ? 3 : 4][lanes];
}

// And which of them name a group's symbols in each of its CTAs, a cluster of them, and do without the launch and the latency
// of the names kernel: while the SMs have room for the work that is done several times (all 4 groups of 8 at K = 48
// 13.3 -> 11.6 us, 40 of them at 512 40.4 -> 33.7, 21 at 600 49.7 -> 40.7, but 80 at 512 48.5 -> 56.3, 16 at 1024 43 -> 57,
// and 400 at 100 44.2 -> 48.6).
bool names_for_itself(int n_groups, int patterns, int symbols, int sms) {
    const long long ctas = (long long)n_groups * patterns;
    return patterns <= kMostOwnPatterns && symbols <= 5000 && ctas <= 4 * sms && ctas * symbols <= 1200000LL;
}

// Shared memory that keeps more CTAs than its share off every SM.  They start early, on the SMs that the names kernel leaves
// first, and three of them there take longer than two on every SM (40 groups of 8 texts of 1024: 68 us, 60 with this; an
// ordinary launch spreads them as well, but costs small batches 2 us; 500 groups of 3 of 200, eleven CTAs an SM: 33.8, 30.0 with this).  Not for clusters, which then wait for
// seven SMs of one GPC with that much to spare (40 groups at 512: 33 us, 43 with this).
int even_smem(long long ctas, int sms) {
    constexpr int kSm = 227 * 1024, kDeclared = 10 * 1024;       // what an SM has; what the kernel declares and the driver adds
    const long long share = (ctas + sms - 1) / sms;
    return share < 2 || share > 20 ? 0 : kSm / (int)(share + 1) + 1024 - kDeclared;
}

// More than 48 KB of shared memory has to be asked for: the most that any call takes, once per device (noted,
// because asking is host time).
constexpr int kMostNamesSmem = 200 * 1024;
int allow_smem() {
    static std::atomic<bool> allowed[64];
    int dev = 0;
    SR_CUDA_TRY(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && allowed[dev].load(std::memory_order_relaxed)) return SR_OK;
    const int prep = SR_MAX_K * 4 + SR_MAX_N * SR_MAX_K * 2;
    SR_CUDA_TRY(cudaFuncSetAttribute(multi_names_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostNamesSmem));
    for (auto kernel : {multi_prep_kernel<true, 0, false, false>, multi_prep_kernel<true, kMostPrepThreads, false, false>, multi_prep_kernel<false, 0, false, false>, multi_prep_kernel<false, kMostPrepThreads, false, false>})
        SR_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, prep));
    for (auto kernel : {multi_prep_kernel<false, 0, true, false>, multi_prep_kernel<false, kMostPrepThreads, true, false>,
                        multi_prep_kernel<false, kTextThreads, true, false>,
                        multi_prep_kernel<false, 0, true, true>, multi_prep_kernel<false, kMostPrepThreads, true, true>,
                        multi_prep_kernel<false, kMostPrepThreads, true, false, true>, multi_prep_kernel<false, kMostPrepThreads, true, true, true>,
                        multi_prep_kernel<true, 0, true, false>, multi_prep_kernel<true, kMostPrepThreads, true, false>,
                        multi_prep_kernel<true, 0, true, true>, multi_prep_kernel<true, kMostPrepThreads, true, true>})
        SR_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostNamesSmem));
    if (dev >= 0 && dev < 64) allowed[dev].store(true, std::memory_order_relaxed);
    return SR_OK;
}

}  // namespace

size_t gate_multi_workspace_bytes(int32_t n_groups, int32_t N, int32_t K, int row_cap) {
    return multi_layout(n_groups, N, K, row_cap > 0 ? row_cap : full_row_cap(K)).total;
}

int launch_gate_multi(const GateArgs& a, void* ws_, size_t ws_bytes, cudaStream_t s,
                      const cudaEvent_t* ev, bool decide, uint8_t* exact, const GroupFeed* feed, int row_cap) {
    if (a.n_groups == 0) return SR_OK;
    MultiWs W = multi_layout(a.n_groups, a.N, a.K, row_cap > 0 ? row_cap : full_row_cap(a.K));
    if (ws_ == nullptr || ws_bytes < W.total || (reinterpret_cast<uintptr_t>(ws_) & 255) != 0)
        return SR_ERR_WORKSPACE;
    unsigned char* ws = static_cast<unsigned char*>(ws_);
    const int P = pairs_of(a.N);
    const long long n_pairs_ll = (long long)a.n_groups * P;
    if (n_pairs_ll > 0x7FFFFFFFLL) return SR_ERR_BAD_N;
    int dev = 0, sms = 0;
    SR_CUDA_TRY(cudaGetDevice(&dev));
    SR_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    W.warps = kDpWarps * sms;
    const int n_pairs = (int)n_pairs_ll;
    int32_t* dist = a.pair_dist ? a.pair_dist : reinterpret_cast<int32_t*>(ws + W.off_dist);
    Ctl* ctl = reinterpret_cast<Ctl*>(ws + W.off_ctl);

    const bool in_pairs = !feed && runs_in_pairs(a.n_groups, a.N, a.K, sms, decide);
    const bool clusters = in_pairs && decide;         // whose CTAs sum up their bounds together
    const bool own_names = in_pairs && names_for_itself(a.n_groups, W.patterns, a.N * W.pitch, sms);
    // names: at least two slots to a symbol while symbols and table fit; above 4096 symbols one, and four CTAs to an SM instead
    // of three (1024 groups of 8 of up to 1024: 122.0 -> 120.1 us)
    const int row_quads = W.pitch >> 2, sym_bytes = a.N * W.pitch * 4, names_most = a.N * W.pitch > 4 * 8 * 512 ? 1024 : 512;
    // A thread for every four positions of the group while 512 threads suffice; and for prep a warp for every 128
    // positions of the pattern and as many warps to every text, unless there are SMs for all patterns: more
    // threads only keep the next CTA waiting.  (512 and 256 whatever the shape: 28000 groups of 2 at K = 33 249 us
    // instead of 98, 4666 of 4 at K = 64 112 instead of 67, 1000 of 8 at K = 100 75 instead of 60.)
    const int names_threads = min((a.N * row_quads + 31) & ~31, names_most), texts = a.N >> 1;
    const int fewest = (max((a.K + 127) >> 7, texts) + texts - 1) / texts * texts;
    const bool an_sm_each = (long long)a.n_groups * W.patterns <= sms;
    const bool many_texts = in_pairs && !decide && an_sm_each && 32 * texts > kMostPrepThreads && a.K > kMostEightLanes;
    const int prep_threads = many_texts ? kTextThreads : an_sm_each ? kMostPrepThreads : min(32 * fewest, kMostPrepThreads);
    W.text_warps = max(1, (prep_threads >> 5) / texts);
    W.text_stride = (prep_threads >> 5) / W.text_warps;
    W.inv_text_warps = (uint32_t)(((1ull << 32) + W.text_warps - 1) / W.text_warps);
    int table_log = 8;
    while ((1 << table_log) < (a.N * a.K > 4096 ? 1 : 2) * a.N * a.K && sym_bytes + (4 << table_log) <= kMostNamesSmem) ++table_log;
    const int names_smem = sym_bytes + (2 << table_log);
    const uint32_t inv_row = (uint32_t)(((1ull << 32) + row_quads - 1) / row_quads);
    uint16_t* names = reinterpret_cast<uint16_t*>(ws + W.off_names);
    int prep_smem = W.pitch * 4 + a.N * W.pitch * 2;
    if (in_pairs) prep_smem += a.N * 16 + 32 + (a.N >> 1) * W.pitch * 2 + (2 * W.rows_pitch + 8) * 4;
    if (own_names) prep_smem += a.N * W.pitch * 2 + names_smem;
    else if (in_pairs && !clusters) prep_smem = max(prep_smem, even_smem((long long)a.n_groups * W.patterns, sms));
    if (names_smem > 47 * 1024 || prep_smem > 35 * 1024) {    // with what the kernels declare
        const int rc = allow_smem();
        if (rc != SR_OK) return rc;
    }

    if (ev) SR_CUDA_TRY(cudaEventRecord(ev[0], s));
    const bool alone = W.alone = n_pairs <= kAlonePairs;      // one CTA orders the batch, and needs nothing to be zero
    const bool mask_only = decide && !a.pair_dist && !a.pair_sum && !a.mean && !exact;
    // (with d_K wanted the groups that upper bounds would settle stay open too: 256 groups that differ in 1 % of their places 137 us, 143 so)
    W.rows_later = mask_only && !alone && !in_pairs && a.K > 256;
    static_assert(offsetof(Ctl, start) <= sizeof(Ctl) - 16, "the last zeros may reach into `start`, which is written later");
    int n_zero = alone || in_pairs ? 0 : (int)(offsetof(Ctl, start) + 15) / 16;       // (a launch of its own cost every call 2.5 us)
    uint8_t* flag = decide ? ws + W.off_flag : nullptr;
    // The match-stream pass works group by group, so when the groups arrive in pieces it runs
    // piece by piece: `feed->before` enqueues whatever makes groups [g0, g1) ready on `s`.
    const int pieces = feed ? feed->pieces : 1;
    for (int c = 0; c < pieces; ++c) {
        const int g0 = (int)((long long)a.n_groups * c / pieces);
        const int g1 = (int)((long long)a.n_groups * (c + 1) / pieces);
        if (g1 == g0) continue;
        if (feed) {
            const int rc = feed->before(feed->ctx, g0, g1, s);
            if (rc != SR_OK) return rc;
        }
        if (!own_names)
            SR_LAUNCH("multi_names_kernel", multi_names_kernel, g1 - g0, names_threads, names_smem, s, a, names, W.pitch, inv_row, table_log, g0,
                  in_pairs ? reinterpret_cast<int32_t*>(ws + W.off_order) : nullptr, reinterpret_cast<uint4*>(ctl), n_zero);
        n_zero = 0;
        const int cluster = own_names || clusters ? W.patterns : 1;
        const bool most = prep_threads == kMostPrepThreads;
        const bool two_warps = prep_threads == kTwoWarpThreads;
        const auto in_memory = decide ? (two_warps ? multi_prep_kernel<true, kTwoWarpThreads, false, false> : most ? multi_prep_kernel<true, kMostPrepThreads, false, false> : multi_prep_kernel<true, 0, false, false>)
                                      : (two_warps ? multi_prep_kernel<false, kTwoWarpThreads, false, false> : most ? multi_prep_kernel<false, kMostPrepThreads, false, false> : multi_prep_kernel<false, 0, false, false>);
        const auto pairs = decide ? (most ? multi_prep_kernel<true, kMostPrepThreads, true, false> : multi_prep_kernel<true, 0, true, false>)
                                  : (most ? multi_prep_kernel<false, kMostPrepThreads, true, false> : multi_prep_kernel<false, 0, true, false>);
        const auto alone_pairs = decide ? (most ? multi_prep_kernel<true, kMostPrepThreads, true, true> : multi_prep_kernel<true, 0, true, true>)
                                        : (most ? multi_prep_kernel<false, kMostPrepThreads, true, true> : multi_prep_kernel<false, 0, true, true>);
        const bool in_twos = in_pairs && most && !decide && a.K > 512 && texts <= 2 && an_sm_each;
        const auto prep = in_twos ? (own_names ? multi_prep_kernel<false, kMostPrepThreads, true, true, true> : multi_prep_kernel<false, kMostPrepThreads, true, false, true>)
                        : many_texts ? multi_prep_kernel<false, kTextThreads, true, false>
                        : own_names ? alone_pairs : in_pairs ? pairs : in_memory;
        const int rc = launch_as(true, cluster, "multi_prep_kernel", prep, (g1 - g0) * W.patterns, prep_threads, prep_smem, s,
                                 a, ws, W, dist, g0, exact, inv_row, table_log, 2u);
        if (rc != SR_OK) return rc;
    }
    if (in_pairs) {
        if (ev) for (int k = 1; k <= 4; ++k) SR_CUDA_TRY(cudaEventRecord(ev[k], s));
        return SR_OK;
    }
    const int gpb = P <= kGroupThreads ? kGroupThreads / P : 1;
    PairDesc* descs = reinterpret_cast<PairDesc*>(ws + W.off_desc);
    int32_t* order = reinterpret_cast<int32_t*>(ws + W.off_order);
    if (decide) {
        SR_LAUNCH("multi_bound_kernel", multi_bound_kernel, (a.n_groups + gpb - 1) / gpb, kGroupThreads, 0, s, a, descs, ctl, flag, exact, gpb, alone,
                  !a.pair_dist && !a.pair_sum && !a.mean && !exact);
    }
    if (ev) SR_CUDA_TRY(cudaEventRecord(ev[1], s));
    const int order_blocks = alone ? 1 : (n_pairs + kOrderThreads - 1) / kOrderThreads;
    const int bin_blocks = (n_pairs + kBinPairs - 1) / kBinPairs, match_blocks = decide ? (W.rows_later ? min((a.n_groups * W.patterns + kMatchWarps - 1) / kMatchWarps, 8 * sms) : 0)
                                                                               : min((n_pairs + kMatchWarps - 1) / kMatchWarps, 16 * sms);
    if (!alone) SR_LAUNCH("multi_bin_kernel", multi_bin_kernel, bin_blocks + match_blocks, 32 * kMatchWarps, 0, s, ws, W, a.N, n_pairs, bin_blocks, dist, a.n_groups * W.patterns);
    SR_LAUNCH("multi_order_kernel", alone ? multi_order_kernel<true> : multi_order_kernel<false>, order_blocks, kOrderThreads, 0, s, descs, order, ctl, n_pairs, W.warps);
    if (ev) SR_CUDA_TRY(cudaEventRecord(ev[2], s));
    const int blocks = n_pairs < sms ? n_pairs : sms;
    // (launched early like the others: one of its CTAs has the registers of most of an SM, so that no two can end up on one.  With the L1
    // that prep left, 1024 groups of 8 texts of 1024 over 100 symbols that differ in 2 % of their places took 973 us in the decide mode with d_K, 352 with
    // all of it; a launch that waits for empty SMs costs every sorted call 2.5 us.  The SMs have to be empty once more for the names kernel of the next call: 2 us of 45
    // for 400 groups of 8 of 1024 whose bounds settle the batch, nothing for 260, for 1024 or for shorter prefixes.  Half or a quarter
    // of the shared memory in place of none: no better than without, and the gate 10 % slower.  Bound, bin or order kernel asking in place of this one: the settled batches take as long
    // or up to 5 % longer, the others gain half as much)
    const int rc = launch_how(LaunchHow{true, 1, true}, "multi_dp_kernel", multi_dp_kernel, blocks, kMostDpWarps * 32, 0, s, ws, W, dist, 2u);
    if (rc != SR_OK) return rc;
    if (ev) SR_CUDA_TRY(cudaEventRecord(ev[3], s));
    SR_LAUNCH("multi_finish_kernel", multi_finish_kernel, (a.n_groups + gpb - 1) / gpb, kGroupThreads, 0, s, a, dist, flag, exact, gpb);
    if (ev) SR_CUDA_TRY(cudaEventRecord(ev[4], s));
    return SR_OK;
}

}  // namespace sr
