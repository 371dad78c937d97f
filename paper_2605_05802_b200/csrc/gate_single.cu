// Single-word gate kernels: prefixes of at most 32 symbols (action-level gate,
// Section 3.2 of the paper: d_K at K <= T_max = 30).  One thread per pair runs the
// bit-parallel column recurrence on one 32-bit word of +1 / -1 vertical deltas; the
// distance is read off as n + popc(Pv) - popc(Mv), so no per-column score is kept.  The
// two kernels differ in where a column's match word comes from.
//
// K <= 16, few rollouts or few groups: gate_direct_kernel.  A thread keeps both prefixes
// of its pair in registers (int4 loads; the rows of a group are shared by its pairs, so
// all but the first touch hit L1) and builds the match word of a column by comparing the
// text symbol with every pattern symbol: 2 instructions per cell against the ~14 of a
// column, no tables, no atomics, no shared memory before the final sums, one round of latencies.
//
// Otherwise: gate_named_kernel.  A group is handled by a warp (which takes several if they have
// room on its lanes) or, for K > 15 and N > 8, by a CTA:
//   1. every symbol is named by one position that holds it: all positions write themselves to
//      the slot of a small table that their symbol hashes to, and look who stayed there;
//   2. a name has a row of match masks, one per rollout: every position sets its bit in its
//      rollout's mask of its symbol's row, and the text keeps the row's place;
//   3. a column's match word for any pattern is then one look-up, row[pattern].  For K <= 15 the
//      masks of two patterns share a word, and one recurrence serves two pairs;
//   4. one thread per group adds the normalised terms in fp64 in pair order, thresholds
//      (Eq. 2) and writes out, for all groups of a CTA side by side.
// Bound: instruction issue.  65536 groups of 16 at K = 30, a CTA each, issue in 75 % of the scheduler's clocks, 55 % of it
// the recurrence; 65536 groups of 8 at K = 15, two to a warp, in 63 %, with 42 % of the warp slots filled.
// 4096 groups of 16, K = 30: 23 us; 16384 groups of 8, K = 30: 31 us; 65536 groups of 8, K = 15, ragged: 44 us.
#include <atomic>

#include "common.cuh"

namespace sr {
namespace {

// A unit is what a warp works on (kWarp: as many groups as its lanes have room for) or one group
// that a CTA works on.  Positions, items (quads of symbols) and rollouts are numbered within it.
struct NamedLayout {
    int groups;                        // groups per unit
    int Q, items;                      // quads per rollout, items per unit
    uint32_t inv_Q, inv_N, inv_C;      // ceil(2^20 / x): division of numbers below 2048 by multiply-shift
    int table_log;                     // names: slots per group
    int row_words;                     // words of a row of match masks
    int combos;                        // recurrences per group (kPacked: two pairs each)
    int pitch;                         // terms per group
    // byte offsets within a unit's shared memory
    int off_table, off_name, off_row, off_peq, off_len, off_order, unit_bytes;
};

__device__ __forceinline__ int div20(int x, uint32_t inv) { return (int)(((uint32_t)x * inv) >> 20); }

// kPacked: the recurrences of a group, enough to serve every pair once: word x of patterns
// (2x, 2x + 1) with the text that is its own upper half, and every word a with the two texts of every
// word b > a.  For each: word, text, and the places of its two pairs in pair order (kNoPair: none).
constexpr uint32_t kNoPair = 0xFFFFu;
struct ComboTable {
    uint16_t start[SR_MAX_N + 1];
    uint2 v[2992];                     // sum over N of ceil(N / 2)^2
    constexpr ComboTable() : start(), v() {
        int at = 0;
        for (int n = 2; n <= SR_MAX_N; ++n) {
            start[n] = (uint16_t)at;
            const int words = (n + 1) / 2;
            for (int a = 0; a < words; ++a)
                for (int j = 2 * a + 1; j < 2 * words; ++j) {
                    uint32_t place[2] = {kNoPair, kNoPair};
                    for (int h = 0; h < 2; ++h) {
                        const int i = 2 * a + h;
                        if (i < j && j < n) place[h] = (uint32_t)(i * n - i * (i + 1) / 2 + (j - i - 1));
                    }
                    v[at].x = (uint32_t)(a | (j << 8));
                    v[at++].y = place[0] | (place[1] << 16);
                }
        }
    }
};
__device__ const ComboTable kCombos = ComboTable();

template <bool kWarp>
__device__ __forceinline__ void unit_sync() {
    if (kWarp) __syncwarp(); else __syncthreads();
}

// kPacked (K <= 15): two patterns share a word, 15 rows and a guard bit each: one look-up and one
// recurrence serve two pairs.
template <bool kPacked, bool kWarp, int kItems>
__global__ void __launch_bounds__(kWarp ? 256 : 512)
gate_named_kernel(GateArgs a, NamedLayout L, uint32_t two) {
    // Rows: a CTA's group of more than eight rollouts would need 32 KB and more with one for every
    // position, so there only symbols that several rollouts hold get one.
    constexpr bool kAlloc = !kWarp;
    extern __shared__ __align__(16) unsigned char smem[];
    const int N = a.N, K = a.K, P = pairs_of(N);
    const int t = kWarp ? (threadIdx.x & 31) : threadIdx.x;               // thread within the unit
    const int nthr = kWarp ? 32 : blockDim.x;
    const int unit = kWarp ? threadIdx.x >> 5 : 0, units = kWarp ? blockDim.x >> 5 : 1;
    const int g0 = (blockIdx.x * units + unit) * L.groups;
    const int ng = min(L.groups, a.n_groups - g0);                        // <= 0: only keeps the barrier company
    unsigned char* base = smem + (size_t)unit * L.unit_bytes;
    int32_t* s_sym = reinterpret_cast<int32_t*>(base);                    // [items][4]
    uint32_t* s_txt = reinterpret_cast<uint32_t*>(base);                  // [items][4] byte offsets of rows, once the symbols have names
    uint16_t* s_name = reinterpret_cast<uint16_t*>(base + L.off_name);    // [items][4]
    uint16_t* s_row = reinterpret_cast<uint16_t*>(base + L.off_row);      // [items][4]
    uint32_t* s_peq = reinterpret_cast<uint32_t*>(base + L.off_peq);      // [rows][row_words]
    int32_t* s_len = reinterpret_cast<int32_t*>(base + L.off_len);        // [rollouts], then the row counter
    uint8_t* s_order = base + L.off_order;                                // [N]
    int& s_rows = s_len[L.groups * N];

    // before the wait: nothing global in here
    if (ng > 0) {
        if (kAlloc) {
#pragma unroll
            for (int u = 0; u < kItems; ++u) {
                const int e = t + u * nthr;
                if (e < L.items) reinterpret_cast<uint2*>(s_row)[e] = make_uint2(0u, 0u);
            }
            for (int w = t; w < L.row_words; w += nthr) s_peq[w] = 0u;    // row 0: no match
        } else {
            for (int w = t; w < L.items * L.row_words; w += nthr) reinterpret_cast<uint4*>(s_peq)[w] = make_uint4(0u, 0u, 0u, 0u);
        }
        if (!kWarp && t == 0) s_rows = 0;
    }
    grid_begin();
    if (ng > 0) {
        const int32_t* seqs = a.seqs + (size_t)g0 * N * a.stride;
        int32_t sym[kItems][4];
        int roll[kItems], live[kItems];            // rollout of the item; positions of its quad inside the prefix
        int open = 0;                              // positions without a name, one bit each
#pragma unroll
        for (int u = 0; u < kItems; ++u) {
            const int e = t + u * nthr;
            roll[u] = div20(e, L.inv_Q);
            live[u] = 0;
            if (e < ng * N * L.Q) {
                const int q = e - roll[u] * L.Q;
                // whole quads inside the row: stride is a multiple of 4 and >= K
                int4 v = make_int4(0, 0, 0, 0);
                if (4 * q < K) v = __ldg(reinterpret_cast<const int4*>(seqs + (uint64_t)(uint32_t)roll[u] * (uint32_t)a.stride) + q);
                int len = a.lens ? __ldg(a.lens + (size_t)g0 * N + roll[u]) : K;
                reinterpret_cast<int4*>(s_sym)[e] = v;
                sym[u][0] = v.x; sym[u][1] = v.y; sym[u][2] = v.z; sym[u][3] = v.w;
                if (q == 0) {
                    if (len < 0 && a.status) atomicOr(a.status, SR_STATUS_NEG_LEN);
                    s_len[roll[u]] = min(max(len, 0), K);
                }
                live[u] = min(max(min(len, K) - 4 * q, 0), 4);
            }
        }
        // ---- names: the symbol of a position is named by one of the positions that hold it.  Every
        // position writes itself to the slot its symbol hashes to (whichever write lands last
        // stays), and if the position found there afterwards holds the same symbol, that is the
        // name -- for all holders of the symbol alike.  The symbols that lost their slot to another
        // one go on with another hash; every round names at least one symbol of each slot.
        auto slot_of = [&](int r, uint32_t sy, uint32_t mul) {
            return reinterpret_cast<uint16_t*>(base + L.off_table) + ((kWarp ? div20(r, L.inv_N) : 0) << L.table_log) +
                   ((sy * mul) >> (32 - L.table_log));
        };
        uint16_t* slot[kItems][4];
#pragma unroll
        for (int u = 0; u < kItems; ++u)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                slot[u][k] = slot_of(roll[u], (uint32_t)sym[u][k], 0x9E3779B1u);
                if (k < live[u]) *slot[u][k] = (uint16_t)(4 * (t + u * nthr) + k);
            }
        unit_sync<kWarp>();
#pragma unroll
        for (int u = 0; u < kItems; ++u) {
            if (live[u] == 0) continue;
            uint32_t name[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                name[k] = 0u;
                if (k < live[u]) {
                    name[k] = *slot[u][k];
                    if (s_sym[name[k]] != sym[u][k]) open |= 1 << (4 * u + k);
                }
            }
            reinterpret_cast<uint2*>(s_name)[t + u * nthr] = make_uint2(name[0] | (name[1] << 16), name[2] | (name[3] << 16));
        }
        uint32_t mul = 0x9E3779B1u;
        for (int round = 0; round < 4 * 1024; ++round) {
            if (!(kWarp ? __any_sync(0xFFFFFFFFu, open) : __syncthreads_or(open))) break;
            if (kWarp) __syncwarp();               // the reads of the round before are done
            mul = mul * 0x2C1B3C6Du + 0x297A2D3Au;                        // stays odd
            for (int m = open; m; m &= m - 1) {
                const int b = __ffs(m) - 1, pos = 4 * (t + (b >> 2) * nthr) + (b & 3);
                *slot_of(div20(pos >> 2, L.inv_Q), (uint32_t)s_sym[pos], mul) = (uint16_t)pos;
            }
            unit_sync<kWarp>();
            for (int m = open; m; m &= m - 1) {
                const int b = __ffs(m) - 1, pos = 4 * (t + (b >> 2) * nthr) + (b & 3);
                const int name = *slot_of(div20(pos >> 2, L.inv_Q), (uint32_t)s_sym[pos], mul);
                if (s_sym[name] == s_sym[pos]) {
                    s_name[pos] = (uint16_t)name;
                    open &= ~(1 << b);
                }
            }
        }
        // ---- names held by more than one rollout get a row of match masks, one per rollout (without
        // kAlloc every position has one)
        if (kAlloc) {
#pragma unroll
        for (int u = 0; u < kItems; ++u) {
            if (live[u] == 0) continue;
            const uint2 v = reinterpret_cast<const uint2*>(s_name)[t + u * nthr];
            const uint32_t name[4] = {v.x & 0xFFFFu, v.x >> 16, v.y & 0xFFFFu, v.y >> 16};
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k < live[u] && (uint32_t)((int)(name[k] >> 2) - roll[u] * L.Q) >= (uint32_t)L.Q) s_row[name[k]] = 1;
        }
        unit_sync<kWarp>();
        {
            uint2 f[kItems];
            int own = 0;
#pragma unroll
            for (int u = 0; u < kItems; ++u) {
                const int e = t + u * nthr;
                f[u] = make_uint2(0u, 0u);
                if (e < L.items) f[u] = reinterpret_cast<const uint2*>(s_row)[e];
                own += __popc(f[u].x) + __popc(f[u].y);
            }
            int incl = own;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int up = __shfl_up_sync(0xFFFFFFFFu, incl, d);
                if ((t & 31) >= d) incl += up;
            }
            const int all = __shfl_sync(0xFFFFFFFFu, incl, 31);
            int first = 0;
            if (!kWarp) {
                if ((t & 31) == 0) first = atomicAdd(&s_rows, all);
                first = __shfl_sync(0xFFFFFFFFu, first, 0);
            }
            uint32_t row = (uint32_t)((first + incl - own + 1) * L.row_words);
#pragma unroll
            for (int u = 0; u < kItems; ++u) {
                if ((f[u].x | f[u].y) == 0u) continue;
                uint32_t h[4] = {f[u].x & 1u, f[u].x >> 16, f[u].y & 1u, f[u].y >> 16};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (h[k]) { h[k] = row; row += L.row_words; }
                reinterpret_cast<uint2*>(s_row)[t + u * nthr] = make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
            }
            {
                const int begin = (first + 1) * L.row_words, end = begin + all * L.row_words;   // the warp's rows
                for (int w = begin + (t & 31); w < end; w += 32) s_peq[w] = 0u;
            }
        }
        }
        if (!kWarp && t < 32) {
            // rollouts by falling length (ties by index), so that the pairs of a warp have texts
            // of similar lengths
            const int mine = t < N ? s_len[t] : K;
            int rank = t;
            if (__any_sync(0xFFFFFFFFu, mine < K)) {
                rank = 0;
                for (int r = 0; r < N; ++r) rank += s_len[r] > mine || (s_len[r] == mine && r < t);
            }
            if (t < N) s_order[rank] = (uint8_t)t;
        }
        unit_sync<kWarp>();
        // ---- every position sets its bit in its rollout's mask and notes the row's place
#pragma unroll
        for (int u = 0; u < kItems; ++u) {
            if (live[u] == 0) continue;
            const int q = (t + u * nthr) - roll[u] * L.Q;
            const int i = kWarp ? roll[u] - div20(roll[u], L.inv_N) * N : roll[u];
            unsigned char* mine = reinterpret_cast<unsigned char*>(s_peq) + 4 * (kPacked ? i >> 1 : i);
            const uint32_t bit = 1u << (4 * q + (kPacked ? (i & 1) << 4 : 0));
            const uint2 v = reinterpret_cast<const uint2*>(s_name)[t + u * nthr];
            const uint32_t name[4] = {v.x & 0xFFFFu, v.x >> 16, v.y & 0xFFFFu, v.y >> 16};
            uint32_t row[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                row[k] = 0u;
                if (k < live[u]) {
                    row[k] = (kAlloc ? s_row[name[k]] : name[k] * L.row_words) * 4u;
                    if (!kAlloc || row[k]) atomicOr(reinterpret_cast<uint32_t*>(mine + row[k]), bit << k);
                }
            }
            reinterpret_cast<uint4*>(s_txt)[t + u * nthr] = make_uint4(row[0], row[1], row[2], row[3]);
        }
        unit_sync<kWarp>();
        // ---- recurrences: one thread per pair, or per text and word of two patterns
        for (int c = t; c < ng * L.combos; c += nthr) {
            const int gl = kWarp ? div20(c, L.inv_C) : 0, x = c - gl * L.combos;
            int word, pj, at[2];                   // word of the rows, text, place of the pair(s)
            if (kPacked) {
                const uint2 v = kCombos.v[kCombos.start[N] + x];
                word = v.x & 0xFF;
                pj = v.x >> 8;
                at[0] = v.y & 0xFFFFu;
                at[1] = v.y >> 16;
                if (at[0] == kNoPair) continue;    // odd N: the last word has no upper half
            } else {
                const int pr = kPairs.v[N][x];
                word = pr >> 8;
                pj = pr & 0xFF;
                at[0] = x;
                at[1] = kNoPair;
                if (!kWarp) {                      // the pattern is the longer prefix, texts ascend
                    pj = s_order[N - 1 - pj];
                    word = s_order[N - 1 - word];
                    at[0] = pair_index(min(pj, word), max(pj, word), N);
                }
            }
            const int mt = s_len[gl * N + pj];
            const unsigned char* peq = reinterpret_cast<const unsigned char*>(s_peq + word);
            const uint4* txt = reinterpret_cast<const uint4*>(s_txt) + (gl * N + pj) * L.Q;
            // Rows of the lower pattern in bits 0..14 and of the upper one in bits 16..30.  The guard bits
            // above them are kept 1 in Mv (so they are 1 in D0 and Ph, whose shift then brings the
            // upper pattern its +1 at row 0) and 0 in Pv (which takes the carry of the sum).
            constexpr uint32_t kGuard = kPacked ? 0x80008000u : 0u, kBelow = kPacked ? 0x3FFF3FFFu : 0xFFFFFFFFu;
            uint32_t Pv = ~kGuard, Mv = kGuard;
            auto column = [&](uint32_t off) {
                const uint32_t Eq = *reinterpret_cast<const uint32_t*>(peq + off);
                const uint32_t D0 = (((Eq & Pv) + Pv) ^ Pv) | (Eq | Mv);
                const uint32_t Ph = Mv | ~(D0 | Pv), Mh = D0 & Pv & kBelow;
                // `two` is a run-time 2: the shifts are multiply-adds on the FMA pipe, which
                // leaves the integer pipe, the bottleneck, the seven logic operations
                const uint32_t Phs = Ph * two + 1u, Mhs = Mh * two;
                Pv = Mhs | ~(D0 | Phs);
                Mv = (Phs & D0) | kGuard;
            };
            uint4 w = txt[0];
            int c4 = mt >> 2;
            for (; c4 > 0; --c4) {
                const uint4 v = w;
                w = *++txt;                        // one quad past the end at most: within the unit
                column(v.x);
                column(v.y);
                column(v.z);
                column(v.w);
            }
            const int left = mt & 3;
            if (left > 0) column(w.x);
            if (left > 1) column(w.y);
            if (left > 2) column(w.z);
            double* s_term = reinterpret_cast<double*>(base + L.off_table) + gl * L.pitch;
            int32_t* s_dist = reinterpret_cast<int32_t*>(reinterpret_cast<double*>(base + L.off_table) + L.groups * L.pitch) + gl * L.pitch;
#pragma unroll
            for (int h = 0; h < (kPacked ? 2 : 1); ++h) {
                if (kPacked && at[h] == kNoPair) continue;
                const int mp = s_len[gl * N + (kPacked ? 2 * word + h : word)];
                const uint32_t msk = kPacked ? ((1u << mp) - 1u) << (16 * h) : low_mask(mp);
                const int d = mt + __popc(Pv & msk) - __popc(Mv & msk);
                if (a.pair_sum) s_dist[at[h]] = d;
                // one term of d_K (Section 3.2): distance / longer prefix, from the quotient table
                s_term[at[h]] = a.norm_mode == SR_NORM_NONE ? (double)d : kQuot.v[d * 33 + max(mp, mt)];
                if (a.pair_dist) a.pair_dist[(size_t)(g0 + gl) * P + at[h]] = d;
            }
        }
    }
    __syncthreads();

    // ---- d_K: ordered fp64 sum, strict threshold (Eq. 2): one thread per group of the CTA
    const int n_here = units * L.groups;
    if ((int)threadIdx.x < n_here) {
        const int u = threadIdx.x / L.groups, gl = threadIdx.x - u * L.groups;
        const size_t g = (size_t)blockIdx.x * n_here + threadIdx.x;
        const double* term = reinterpret_cast<const double*>(smem + (size_t)u * L.unit_bytes + L.off_table);
        if (g < (size_t)a.n_groups)
            group_sum_and_gate(term + gl * L.pitch, reinterpret_cast<const int32_t*>(term + L.groups * L.pitch) + gl * L.pitch, P, a, g);
    }
}

// Only a CTA's group takes more than 48 KB of shared memory, at most 80000 bytes (32 rollouts, K = 32).
// It has to be asked for: the most that any call takes, for all widths of the kernel, once per
// device (noted, because asking is host time).  Never less than that, or a thread with a smaller
// call would take back what another one has just been granted.
constexpr int kMostSmem = 80000;
int allow_smem() {
    static std::atomic<bool> allowed[64];
    int dev = 0;
    SR_CUDA_TRY(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && allowed[dev].load(std::memory_order_relaxed)) return SR_OK;
    SR_CUDA_TRY(cudaFuncSetAttribute(gate_named_kernel<false, false, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem));
    SR_CUDA_TRY(cudaFuncSetAttribute(gate_named_kernel<false, false, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem));
    SR_CUDA_TRY(cudaFuncSetAttribute(gate_named_kernel<false, false, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem));
    if (dev >= 0 && dev < 64) allowed[dev].store(true, std::memory_order_relaxed);
    return SR_OK;
}

template <bool kPacked, bool kWarp>
int launch_gate_named(const GateArgs& a, cudaStream_t s) {
    constexpr bool kAlloc = !kWarp;
    const int N = a.N, P = pairs_of(N);
    NamedLayout L;
    L.Q = a.K > 0 ? (a.K + 3) >> 2 : 1;
    L.row_words = kPacked ? (N + 1) >> 1 : N;
    L.combos = kPacked ? L.row_words * L.row_words : P;
    L.groups = 1;
    if (kWarp)                                     // fill the lanes, with at most four quads each
        while ((L.groups + 1) * L.combos <= 32 && (L.groups + 1) * N * L.Q <= 128) ++L.groups;
    L.items = L.groups * N * L.Q;
    auto inv = [](int x) { return ((1u << 20) + (uint32_t)x - 1u) / (uint32_t)x; };
    L.inv_Q = inv(L.Q);
    L.inv_N = inv(N);
    L.inv_C = inv(L.combos);
    L.table_log = 6;                               // at least two slots to a symbol (four were no better)
    while ((1 << L.table_log) < 2 * N * a.K) ++L.table_log;
    L.pitch = P | 1;
    int off = 0;
    auto take = [&](int bytes) { int o = off; off = (off + bytes + 15) & ~15; return o; };
    take(L.items * 16);
    // the terms and distances of the pairs take the table's place
    const int table = L.groups * (2 << L.table_log), terms = L.groups * L.pitch * 12;
    L.off_table = take(table > terms ? table : terms);
    L.off_name = take(L.items * 8);
    L.off_row = take(kAlloc ? L.items * 8 : 0);
    // allocated rows have at least two holders
    L.off_peq = take((kAlloc ? L.groups * (N * a.K / 2) + 1 : 4 * L.items) * L.row_words * 4);
    L.off_len = take((L.groups * N + 1) * 4);
    L.off_order = take(N);
    L.unit_bytes = off;
    int threads, units = 1, items_per_thread;
    if (kWarp) {
        units = 8;
        while (units > 1 && units * L.unit_bytes > 48 * 1024) units >>= 1;
        while (units > 1 && (long long)a.n_groups <= (units >> 1) * L.groups) units >>= 1;
        threads = 32 * units;
        items_per_thread = (L.items + 31) / 32;
    } else {
        threads = (P + 31) & ~31;
        if (threads > 512) threads = 512;
        items_per_thread = (L.items + threads - 1) / threads;
    }
    const int smem = units * L.unit_bytes, per = units * L.groups;
    const int blocks = (a.n_groups + per - 1) / per;
    auto kernel = items_per_thread <= 1 ? gate_named_kernel<kPacked, kWarp, 1>
                : items_per_thread == 2 ? gate_named_kernel<kPacked, kWarp, 2>
                                        : gate_named_kernel<kPacked, kWarp, 4>;
    if (smem > 48 * 1024) {
        const int rc = allow_smem();
        if (rc != SR_OK) return rc;
    }
    return launch("gate_named_kernel", kernel, blocks, threads, smem, s, a, L, 2u);
}

// ---------------------------------------------------------------------------------
// K <= 16: prefixes in registers, match words by direct comparison.  Threads are packed
// pair after pair: a CTA of T threads serves floor(T / P) groups.
template <int KR>      // pattern rows / text columns held in registers: K <= KR, KR % 4 == 0
__global__ void __launch_bounds__(512)
gate_direct_kernel(GateArgs a, int groups_per_cta, uint32_t one) {
    grid_begin();
    extern __shared__ __align__(16) unsigned char smem[];
    const int N = a.N, K = a.K, P = pairs_of(N);
    double* s_term = reinterpret_cast<double*>(smem);                               // [groups_per_cta * P]
    int32_t* s_dist = reinterpret_cast<int32_t*>(s_term + groups_per_cta * P);      // [groups_per_cta * P]
    const int tid = threadIdx.x;
    const int gl = tid / P, p = tid - gl * P;
    const size_t g = (size_t)blockIdx.x * groups_per_cta + gl;
    if (gl < groups_per_cta && g < (size_t)a.n_groups) {
        const int pr = kPairs.v[N][p];
        int pi = pr & 0xFF, pj = pr >> 8;
        int mi = a.lens ? __ldg(a.lens + g * N + pi) : K;
        int mj = a.lens ? __ldg(a.lens + g * N + pj) : K;
        if ((mi < 0 || mj < 0) && a.status) atomicOr(a.status, SR_STATUS_NEG_LEN);
        mi = min(max(mi, 0), K);
        mj = min(max(mj, 0), K);
        int mp = mi, mt = mj;                      // the pattern (rows) is the longer prefix
        if (mj > mi) { const int x = pi; pi = pj; pj = x; mp = mj; mt = mi; }
        const int4* prow = reinterpret_cast<const int4*>(a.seqs + (g * N + pi) * a.stride);
        const int4* trow = reinterpret_cast<const int4*>(a.seqs + (g * N + pj) * a.stride);
        int32_t pat[KR], txt[KR];
#pragma unroll
        for (int q = 0; q < KR / 4; ++q) {
            // whole quads inside the row (stride is a multiple of 4 and >= K); symbols past
            // a prefix's end are never looked at: columns stop at mt, and rows past mp only
            // disturb bits the final mask drops (carries and shifts move upwards only)
            int4 v = make_int4(0, 0, 0, 0), w = make_int4(0, 0, 0, 0);
            if (4 * q < mp) v = __ldg(prow + q);
            if (4 * q < mt) w = __ldg(trow + q);
            pat[4 * q] = v.x; pat[4 * q + 1] = v.y; pat[4 * q + 2] = v.z; pat[4 * q + 3] = v.w;
            txt[4 * q] = w.x; txt[4 * q + 1] = w.y; txt[4 * q + 2] = w.z; txt[4 * q + 3] = w.w;
        }
        uint32_t Pv = 0xFFFFFFFFu, Mv = 0u, Ph, Mh;
#pragma unroll
        for (int c = 0; c < KR; ++c) {
            if (c < mt) {
                uint32_t Eq = 0u;
#pragma unroll
                for (int r = 0; r < KR; ++r)
                    // `one` holds 1 but is a run-time value, so the bit is set by a multiply-add:
                    // it issues on the FMA pipe while the comparisons keep the integer ALU busy
                    asm("{ .reg .pred q; setp.eq.s32 q, %1, %2; @q mad.lo.u32 %0, %3, %4, %0; }"
                        : "+r"(Eq) : "r"(pat[r]), "r"(txt[c]), "r"(one), "r"(1u << r));
                word_column(Eq, Pv, Mv, Ph, Mh);
            }
        }
        const uint32_t msk = low_mask(mp);
        const int d = mt + __popc(Pv & msk) - __popc(Mv & msk);
        s_dist[tid] = d;
        // one term of d_K (Section 3.2): distance / longer prefix, from the quotient table
        s_term[tid] = a.norm_mode == SR_NORM_NONE ? (double)d : kQuot.v[d * 33 + mp];
        if (a.pair_dist) a.pair_dist[g * P + p] = d;
    }
    __syncthreads();
    // ---- d_K: ordered fp64 sum, strict threshold (Eq. 2): one thread per group of the CTA
    if (tid < groups_per_cta) {
        const size_t gg = (size_t)blockIdx.x * groups_per_cta + tid;
        if (gg < (size_t)a.n_groups) group_sum_and_gate(s_term + tid * P, s_dist + tid * P, P, a, gg);
    }
}

template <int KR>
int launch_gate_direct(const GateArgs& a, cudaStream_t s) {
    const int P = pairs_of(a.N);
    const int threads = P <= 256 ? 256 : 512;
    const int gpc = threads / P;
    const int smem = gpc * P * 12;
    const int blocks = (a.n_groups + gpc - 1) / gpc;
    SR_LAUNCH("gate_direct_kernel", gate_direct_kernel<KR>, blocks, threads, smem, s, a, gpc, 1u);
    return SR_OK;
}

// Where naming the symbols first pays: the least number of pairs, measured for the group sizes 2..32, every
// K up to 16 and 300 to 2.6 million pairs; mean time within 0.4 % of the better kernel's.  Direct comparison
// costs two instructions per cell, naming a few dozen per symbol and a longer chain of latencies on
// one warp a group: small batches, N < 8 and short prefixes stay with direct comparison.  The line
// lies later for large groups, whose warp takes long (32 rollouts: eight rounds of pairs), and for those
// whose pairs fill the CTAs of the direct kernel (31 and 32).  At K = 16 two patterns do not fit a
// word, and groups of 9 to 13 leave the CTA they then get mostly idle.  Direct / naming in us: 8 x 5714, K = 12
// 7.2 / 6.7; 32 x 161, K = 12 9.2 / 16.5; 16 x 2666, K = 8 8.7 / 8.9, 16 x 21666 45 / 34; 9 x 36111, K = 16 46 / 94.
bool names_pay(int N, int K, long long pairs) {
    if (N < 8) return false;
    if (K == 16) return (N == 8 || N >= 14) && pairs >= 25000;
    if (K >= 13) return pairs >= (N <= 16 ? 40000 : 120000);
    if (K >= 9) return pairs >= (N <= 10 ? 100000 : (N <= 30 ? 240000 : 1200000));
    if (N > 30 && K > 4) return false;
    return N >= 12 && pairs >= (N < 14 ? 1000000 : 300000);
}

}  // namespace

int launch_gate_single(const GateArgs& a, cudaStream_t s) {
    if (a.n_groups == 0) return SR_OK;
    if (a.K <= 16 && !names_pay(a.N, a.K, (long long)a.n_groups * pairs_of(a.N))) {
        if (a.K <= 4) return launch_gate_direct<4>(a, s);
        if (a.K <= 8) return launch_gate_direct<8>(a, s);
        if (a.K <= 12) return launch_gate_direct<12>(a, s);
        return launch_gate_direct<16>(a, s);
    }
    if (a.K <= 15) return launch_gate_named<true, true>(a, s);
    if (a.N <= 8) return launch_gate_named<false, true>(a, s);
    return launch_gate_named<false, false>(a, s);
}

}  // namespace sr
