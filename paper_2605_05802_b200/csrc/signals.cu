// Further per-group signals of the paper's Appendix B and the OR-rule extension.
#include <math.h>

#include <cooperative_groups.h>

#include "common.cuh"

namespace sr {
namespace {

// tau_K and Cut = [d_K < d_L] or [tau_K >= tau_H] (Eq. 3): one thread per group, N <= 32
// flags or lengths each.  A few bytes per rollout: bound by HBM bandwidth / launch latency.
__global__ void __launch_bounds__(256)
or_rule_kernel(const double* __restrict__ mean, const int32_t* __restrict__ lens,
               const uint8_t* __restrict__ done, int n_groups, int N, int K, double threshold,
               double tau_high, bool vec4, double* __restrict__ tau, uint8_t* __restrict__ stop) {
    grid_begin();
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n_groups) return;
    const double dk = mean[g];
    int finished = 0;
    if (vec4) {                                   // lengths only, rows 16-byte aligned
        const int4* row = reinterpret_cast<const int4*>(lens + (size_t)g * N);
        for (int q = 0; q < N / 4; ++q) {
            const int4 v = __ldg(row + q);
            finished += (v.x < K) + (v.y < K) + (v.z < K) + (v.w < K);
        }
    } else {
        for (int i = 0; i < N; ++i) {
            const size_t idx = (size_t)g * N + i;
            finished += done ? (done[idx] != 0) : (lens[idx] < K);
        }
    }
    const double t = __ddiv_rn((double)finished, (double)N);
    if (tau) tau[g] = t;
    stop[g] = (dk < threshold || t >= tau_high) ? 1 : 0;
}

constexpr int kClusterCtas = 8;                  // the portable size

// d / l for d <= 31 common bigrams of l <= 62 (0 when l == 0), correctly rounded as __ddiv_rn is.
struct JaccardTable {
    double v[32 * 63];
    constexpr JaccardTable() : v() {
        for (int d = 0; d < 32; ++d)
            for (int l = 0; l < 63; ++l) v[d * 63 + l] = l > 0 ? (double)d / (double)l : 0.0;
    }
};
__device__ const JaccardTable kJaccard = JaccardTable();

struct EntropyTerms {
    double plogp[SR_MAX_N + 1], ln_n;           // (c / N) ln (c / N), ln N
};
struct EntropyTable {                           // host side
    EntropyTerms of[SR_MAX_N + 1];
    EntropyTable() {
        for (int n = 1; n <= SR_MAX_N; ++n) {
            of[n].ln_n = log((double)n);
            of[n].plogp[0] = 0.0;
            for (int c = 1; c <= n; ++c) of[n].plogp[c] = ((double)c / n) * log((double)c / n);
        }
    }
};

// The other action-only signals of Appendix B.  One CTA per group, one thread per quad of
// symbols.  A bigram is named by one position at which it occurs: all positions write themselves to
// the slot of a small table that their bigram hashes to, and look who stayed there (the losers go on with
// another hash).  A name collects the rollouts that hold it; the names held by several are numbered, turned
// into a bit set per rollout by votes (32 names a step), and a pair's Jaccard term is a few popcounts.
// Two warps match the prefixes (by hash, then symbol by symbol) and the step-K actions; everything is added
// up in a fixed order.
// Bound: instruction issue (81 % of the scheduler's clocks for 65536 groups of 16 at K = 30, 205 us) and, in small
// batches, the latency between its barriers (4096 groups 17 us).
struct SignalLayout {
    int Q, items;                               // quads per rollout, items of the group
    uint32_t inv_Q;                             // ceil(2^20 / Q)
    int table_log;
    // byte offsets into dynamic shared memory
    int off_sym, off_name, off_table, off_mask, off_list, off_bits, off_small, off_term, off_plogp, total;
    int words;                                  // most words of a rollout's bit set
};

__device__ __forceinline__ bool same_prefix(const int32_t* a, const int32_t* b, int len) {
    for (int q = 0; 4 * q < len; ++q) {
        const int4 u = reinterpret_cast<const int4*>(a)[q], v = reinterpret_cast<const int4*>(b)[q];
        const int left = len - 4 * q;           // symbols of this quad inside the prefix
        if (u.x != v.x || (left > 1 && u.y != v.y) || (left > 2 && u.z != v.z) || (left > 3 && u.w != v.w)) return false;
    }
    return true;
}

__global__ void __launch_bounds__(256)
group_signals_kernel(const int32_t* __restrict__ seqs, const int32_t* __restrict__ lens, int N,
                     int stride, int K, EntropyTerms T, SignalLayout L,
                     double* upr, double* uar, double* ent, double* jac) {
    extern __shared__ __align__(16) unsigned char smem[];
    int32_t* s_sym = reinterpret_cast<int32_t*>(smem + L.off_sym);          // [items][4] and one more quad
    uint16_t* s_name = reinterpret_cast<uint16_t*>(smem + L.off_name);      // [items][4]
    uint16_t* s_table = reinterpret_cast<uint16_t*>(smem + L.off_table);    // [1 << table_log]
    uint32_t* s_mask = reinterpret_cast<uint32_t*>(smem + L.off_mask);      // [items][4] rollouts that hold the name
    uint32_t* s_list = reinterpret_cast<uint32_t*>(smem + L.off_list);      // masks of the names held by several
    uint32_t* s_bits = reinterpret_cast<uint32_t*>(smem + L.off_bits);      // [N][words]
    double* s_term = reinterpret_cast<double*>(smem + L.off_term);          // [P]
    int32_t* s_len = reinterpret_cast<int32_t*>(smem + L.off_small);        // 4 arrays of [N]
    int32_t* s_raw = s_len + N;
    uint32_t* s_hash = reinterpret_cast<uint32_t*>(s_raw + N);
    int32_t* s_card = s_raw + 2 * N;            // bigrams of the rollout's set
    int& s_shared = *(s_card + N);              // names held by several rollouts
    double* s_plogp = reinterpret_cast<double*>(smem + L.off_plogp);        // [N]
    const int g = blockIdx.x, tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31;
    const int P = pairs_of(N);
    // before the wait: nothing global in here
    if (tid < L.items) reinterpret_cast<uint4*>(s_mask)[tid] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < N) { s_hash[tid] = 0u; s_card[tid] = 0; }
    if (tid == 0) s_shared = 0;
    const int i = (int)(((uint32_t)tid * L.inv_Q) >> 20), q = tid - i * L.Q;      // rollout and quad of the thread's item
    grid_begin();
    int live = 0;                               // symbols of the quad inside the prefix
    int4 v = make_int4(0, 0, 0, 0);
    if (tid < N) {
        const int raw = lens ? __ldg(lens + (size_t)g * N + tid) : K;
        s_raw[tid] = raw;
        s_len[tid] = min(max(raw, 0), K);
    }
    int len = 0;
    if (tid < L.items && K > 0) {
        v = __ldg(reinterpret_cast<const int4*>(seqs + ((size_t)g * N + i) * stride) + q);
        len = lens ? __ldg(lens + (size_t)g * N + i) : K;
        len = min(max(len, 0), K);
        live = min(max(len - 4 * q, 0), 4);
        reinterpret_cast<int4*>(s_sym)[tid] = v;
    }
    __syncthreads();
    // hash of the prefix: any sum over positions and symbols will do
    const int32_t sym[4] = {v.x, v.y, v.z, v.w};
    if (live) {
        uint32_t h = 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < live) {
                const uint32_t x = ((uint32_t)sym[k] + (uint32_t)(4 * q + k) * 0x9E3779B1u) * 0x85EBCA77u;
                h += x ^ (x >> 15);
            }
        atomicAdd(&s_hash[i], h);
    }
    if (jac) {
        // bigram k of the item: symbols 4q + k and the next one, inside the prefix
        const int n_big = min(max(len - 1 - 4 * q, 0), 4);
        const int32_t next = tid < L.items ? s_sym[4 * tid + 4] : 0;       // one quad past the end at most
        const int32_t two[5] = {v.x, v.y, v.z, v.w, next};
        auto slot_of = [&](int32_t x, int32_t y, uint32_t mul) {
            return s_table + (((((uint32_t)x * mul) ^ ((uint32_t)x >> 15)) + (uint32_t)y * 0x85EBCA77u) * 0x2C1B3C6Du >> (32 - L.table_log));
        };
        int open = 0;
        uint16_t* slot[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            slot[k] = slot_of(two[k], two[k + 1], 0x9E3779B1u);
            if (k < n_big) *slot[k] = (uint16_t)(4 * tid + k);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < n_big) {
                const int name = *slot[k];
                s_name[4 * tid + k] = (uint16_t)name;
                if (s_sym[name] != two[k] || s_sym[name + 1] != two[k + 1]) open |= 1 << k;
            }
        uint32_t mul = 0x9E3779B1u;
        for (int round = 0; round < 1024; ++round) {           // every round names a bigram of each slot
            if (!__syncthreads_or(open)) break;
            mul = mul * 0x2C1B3C6Du + 0x297A2D3Au;              // stays odd
            for (int m = open; m; m &= m - 1) {
                const int pos = 4 * tid + __ffs(m) - 1;
                *slot_of(s_sym[pos], s_sym[pos + 1], mul) = (uint16_t)pos;
            }
            __syncthreads();
            for (int m = open; m; m &= m - 1) {
                const int k = __ffs(m) - 1, pos = 4 * tid + k;
                const int name = *slot_of(s_sym[pos], s_sym[pos + 1], mul);
                if (s_sym[name] == s_sym[pos] && s_sym[name + 1] == s_sym[pos + 1]) {
                    s_name[pos] = (uint16_t)name;
                    open &= ~(1 << k);
                }
            }
        }
        // the rollouts of every name; a rollout's set counts a bigram once
        if (n_big) {
            int fresh = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k < n_big) fresh += !(atomicOr(&s_mask[s_name[4 * tid + k]], 1u << i) >> i & 1u);
            if (fresh) atomicAdd(&s_card[i], fresh);
        }
    }
    __syncthreads();
    if (jac) {
        // numbers for the names that several rollouts hold
        uint32_t f[4] = {0u, 0u, 0u, 0u};
        int own = 0;
        if (tid < L.items) {
            const uint4 m = reinterpret_cast<const uint4*>(s_mask)[tid];
            f[0] = m.x; f[1] = m.y; f[2] = m.z; f[3] = m.w;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) own += (f[k] & (f[k] - 1u)) != 0u;
        int incl = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int up = __shfl_up_sync(0xFFFFFFFFu, incl, d);
            if (lane >= d) incl += up;
        }
        int first = 0;
        if (lane == 31) first = atomicAdd(&s_shared, incl);
        first = __shfl_sync(0xFFFFFFFFu, first, 31) + incl - own;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if ((f[k] & (f[k] - 1u)) != 0u) s_list[first++] = f[k];
    }
    // prefixes: rollouts with the same length and hash, and whether the first of them really agrees
    if (tid < 32) {
        const int mine = lane < N ? s_len[lane] : 0;
        const unsigned long long key = lane < N ? ((unsigned long long)s_hash[lane] << 32) | (unsigned)mine : ~0ull;
        const unsigned alike = __match_any_sync(0xFFFFFFFFu, key);
        bool first = true;
        for (unsigned m = lane < N ? alike & ((1u << lane) - 1u) : 0u; m && first; m &= m - 1u)
            first = !same_prefix(s_sym + 4 * L.Q * (__ffs(m) - 1), s_sym + 4 * L.Q * lane, mine);
        const int distinct = __popc(__ballot_sync(0xFFFFFFFFu, first && lane < N));
        if (lane == 0 && upr) upr[g] = kQuot.v[distinct * 33 + N];
    }
    // step-K actions: the rollouts that hold the same one; entropy terms, added up in order
    if (tid >= nthr - 32) {
        const bool has = lane < N && s_raw[lane] >= K && K >= 1;   // otherwise it shares the value "no action"
        const unsigned long long key = has ? (1ull << 32) | (uint32_t)s_sym[4 * L.Q * lane + K - 1] : (lane < N ? 0ull : ~0ull);
        const unsigned alike = __match_any_sync(0xFFFFFFFFu, key);
        const bool first = lane < N && __ffs(alike) - 1 == lane;
        const unsigned firsts = __ballot_sync(0xFFFFFFFFu, first);
        if (ent) {
            if (lane < N) s_plogp[lane] = first ? T.plogp[__popc(alike)] : 0.0;
            __syncwarp();
            if (lane == 0) {
                double h = 0.0;
                for (int r = 0; r < N; ++r) h = __dsub_rn(h, s_plogp[r]);      // - 0 where not the first
                ent[g] = __ddiv_rn(h, T.ln_n);
            }
        }
        if (lane == 0 && uar) uar[g] = kQuot.v[__popc(firsts) * 33 + N];
    }
    __syncthreads();
    if (jac) {
        const int shared = s_shared, words = (shared + 31) >> 5;
        for (int w = tid >> 5; w < words; w += nthr >> 5) {
            const uint32_t m = 32 * w + lane < shared ? s_list[32 * w + lane] : 0u;
            uint32_t mine = 0u;
            for (int r = 0; r < N; ++r) {
                const uint32_t b = __ballot_sync(0xFFFFFFFFu, m >> r & 1u);
                if (lane == r) mine = b;
            }
            if (lane < N) s_bits[lane * L.words + w] = mine;
        }
        __syncthreads();
        for (int p = tid; p < P; p += nthr) {
            const int pr = kPairs.v[N][p];
            const int a = pr & 0xFF, b = pr >> 8;
            int both = 0;
            for (int w = 0; w < words; ++w) both += __popc(s_bits[a * L.words + w] & s_bits[b * L.words + w]);
            const int uni = s_card[a] + s_card[b] - both;
            s_term[p] = uni > 0 ? __dsub_rn(1.0, kJaccard.v[both * 63 + uni]) : 0.0;
        }
    }
    __syncthreads();
    if (tid == 0 && jac) {
        double s = 0.0;
        int p = 0;
        for (; p + 8 <= P; p += 8) {            // loads ahead of the (necessarily sequential) additions
            double t[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) t[u] = s_term[p + u];
#pragma unroll
            for (int u = 0; u < 8; ++u) s = __dadd_rn(s, t[u]);
        }
        for (; p < P; ++p) s = __dadd_rn(s, s_term[p]);
        jac[g] = __ddiv_rn(s, (double)P);
    }
}

// Batch reductions (Section 4.5 dilution, Section 3.4 norm kept): grid-stride over the
// groups, fp64 partial sums per thread, warp shuffles, one set of atomics per CTA.
// N = 8 (the paper's G): four groups per trip, a grid stride apart (so that consecutive
// lanes read consecutive 32-byte rows), their eight 16-byte loads and four decision bytes
// issued before any arithmetic; the last trip takes whatever is left of the four with
// predicated loads.  Measured at 0.59 of the copy bandwidth: the warps wait on loads (17
// stall cycles per issue) while the fp32 -> fp64 conversions of the exact squares keep the
// conversion unit a third busy.  Tried and not faster: four consecutive groups per thread
// (uncoalesced 16-byte loads), eight groups per trip, larger CTAs, more CTAs (the five
// atomics per CTA start to cost from about 5000 CTAs on).
// kCluster: the grid is one cluster, whose CTAs hand their sums to the first one through distributed shared
// memory: it writes the outputs, which then need no clearing before and no atomics (4096 groups of
// 16: two clears and the kernel took 6.9 us, the cluster 4.5 us).
template <bool kCluster>
__global__ void __launch_bounds__(kCluster ? 1024 : 256)
batch_stats_kernel(const float* __restrict__ adv, const uint8_t* __restrict__ stop, int N,
                   int n_groups, bool vec4, unsigned long long* counts, double* sumsq) {
    grid_begin();
    double ss_all = 0.0, ss_kept = 0.0;
    unsigned z_all = 0, z_kept = 0, kept_groups = 0;
    const int stride = gridDim.x * blockDim.x;
    long long g = blockIdx.x * blockDim.x + threadIdx.x;     // 64-bit: g + 4 * stride may pass 2^31
    if (vec4 && N == 8) {
        for (; g < n_groups; g += 4LL * stride) {
            float4 v[4][2];
            unsigned char st[4];
            bool have[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const long long gg = g + (long long)u * stride;
                have[u] = gg < n_groups;
                v[u][0] = v[u][1] = make_float4(1.f, 1.f, 1.f, 1.f);
                st[u] = 0;
                if (have[u]) {
                    const float4* row = reinterpret_cast<const float4*>(adv + (size_t)gg * 8);
                    v[u][0] = __ldg(row);
                    v[u][1] = __ldg(row + 1);
                    st[u] = stop ? stop[gg] : 0;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (!have[u]) continue;
                const float f[8] = {v[u][0].x, v[u][0].y, v[u][0].z, v[u][0].w,
                                    v[u][1].x, v[u][1].y, v[u][1].z, v[u][1].w};
                double ss = 0.0;
                unsigned z = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {        // zero tests in fp32 (exact), squares in fp64
                    const double a = (double)f[i];
                    ss += __dmul_rn(a, a);
                    z += f[i] == 0.0f;
                }
                const bool kept = st[u] == 0;
                kept_groups += kept;
                ss_all += ss;
                z_all += z;
                if (kept) { ss_kept += ss; z_kept += z; }
            }
        }
    }
    for (; g < n_groups; g += stride) {            // any other group size: one group per trip
        const bool kept = !(stop && stop[g]);
        kept_groups += kept;
        const float* row = adv + (size_t)g * N;
        double ss = 0.0;
        unsigned z = 0;
        if (vec4) {
            for (int q = 0; q < N / 4; ++q) {
                const float4 v = __ldg(reinterpret_cast<const float4*>(row) + q);
                const double a0 = v.x, a1 = v.y, a2 = v.z, a3 = v.w;
                ss += __dmul_rn(a0, a0); ss += __dmul_rn(a1, a1); ss += __dmul_rn(a2, a2); ss += __dmul_rn(a3, a3);
                z += (a0 == 0.0) + (a1 == 0.0) + (a2 == 0.0) + (a3 == 0.0);
            }
        } else {
            for (int i = 0; i < N; ++i) {
                const double a = (double)__ldg(row + i);
                ss += __dmul_rn(a, a);
                z += a == 0.0;
            }
        }
        ss_all += ss;
        z_all += z;
        if (kept) { ss_kept += ss; z_kept += z; }
    }
    for (int off = 16; off > 0; off >>= 1) {
        ss_all += __shfl_xor_sync(0xFFFFFFFFu, ss_all, off);
        ss_kept += __shfl_xor_sync(0xFFFFFFFFu, ss_kept, off);
        z_all += __shfl_xor_sync(0xFFFFFFFFu, z_all, off);
        z_kept += __shfl_xor_sync(0xFFFFFFFFu, z_kept, off);
        kept_groups += __shfl_xor_sync(0xFFFFFFFFu, kept_groups, off);
    }
    // warp results -> shared memory -> one set of atomics per CTA
    __shared__ double s_ss[2][32];
    __shared__ unsigned s_cnt[3][32];
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        s_ss[0][w] = ss_all; s_ss[1][w] = ss_kept;
        s_cnt[0][w] = z_all; s_cnt[1][w] = z_kept; s_cnt[2][w] = kept_groups;
    }
    __syncthreads();
    __shared__ double s_sum[2];
    __shared__ unsigned long long s_total[3];
    if (threadIdx.x == 0) {
        double a = 0.0, k = 0.0;
        unsigned long long c0 = 0, c1 = 0, c2 = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
            a += s_ss[0][i]; k += s_ss[1][i];
            c0 += s_cnt[0][i]; c1 += s_cnt[1][i]; c2 += s_cnt[2][i];
        }
        if (kCluster) {
            s_sum[0] = a; s_sum[1] = k;
            s_total[0] = c0; s_total[1] = c1; s_total[2] = c2;
        } else {
            atomicAdd(&sumsq[0], a);
            atomicAdd(&sumsq[1], k);
            atomicAdd(&counts[0], c0);
            atomicAdd(&counts[1], c1);
            atomicAdd(&counts[2], c2);
        }
    }
    if (kCluster) {
        const auto cluster = cooperative_groups::this_cluster();
        cluster.sync();
        if (blockIdx.x == 0 && threadIdx.x < 5) {
            double a = 0.0;
            unsigned long long c = 0;
            for (unsigned b = 0; b < gridDim.x; ++b) {
                if (threadIdx.x < 2) a += cluster.map_shared_rank(s_sum, b)[threadIdx.x];
                else c += cluster.map_shared_rank(s_total, b)[threadIdx.x - 2];
            }
            if (threadIdx.x < 2) sumsq[threadIdx.x] = a;
            else counts[threadIdx.x - 2] = c;
        }
        cluster.sync();                        // nobody leaves while its sums are read
    }
}

}  // namespace

int launch_group_signals(const int32_t* seqs, const int32_t* lens, int32_t n_groups, int32_t N,
                         int32_t stride, int32_t K, double* upr, double* uar, double* ent,
                         double* jac, cudaStream_t s) {
    if (n_groups == 0) return SR_OK;
    // p ln p for the 1..N rollouts that may share an action, once per group size
    static const EntropyTable entropy;
    const EntropyTerms& T = entropy.of[N];
    SignalLayout L;
    L.Q = K > 0 ? (K + 3) >> 2 : 1;
    L.items = N * L.Q;
    L.inv_Q = ((1u << 20) + (uint32_t)L.Q - 1u) / (uint32_t)L.Q;
    L.table_log = 6;                                 // at least two slots to a bigram
    while ((1 << L.table_log) < 2 * N * K) ++L.table_log;
    L.words = (N * K / 2 + 31) >> 5 | 1;             // such a name has at least two holders; odd against bank conflicts
    int off = 0;
    auto take = [&](int bytes) { int o = off; off = (off + bytes + 15) & ~15; return o; };
    L.off_sym = take(L.items * 16 + 16);
    L.off_name = take(L.items * 8);
    L.off_table = take(2 << L.table_log);
    L.off_mask = take(L.items * 16);
    L.off_list = take((N * K / 2 + 1) * 4);
    L.off_bits = take(N * L.words * 4);
    L.off_small = take((4 * N + 1) * 4);
    L.off_plogp = take(N * 8);
    L.off_term = take(pairs_of(N) * 8);
    L.total = off;
    // A thread per quad; while every SM has four groups at most, one per pair too (in large batches the
    // extra warps only wait: 16384 groups of 32 at K = 5 take 91 us, with them 110).
    int threads = (L.items + 31) & ~31;
    if (jac && threads < pairs_of(N) && n_groups <= 1024) {
        int dev = 0, sms = 0;
        SR_CUDA_TRY(cudaGetDevice(&dev));
        SR_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        if (n_groups <= 4 * sms) threads = max(threads, min((pairs_of(N) + 31) & ~31, 256));
    }
    SR_LAUNCH("group_signals_kernel", group_signals_kernel, n_groups, threads, L.total, s, seqs, lens, N, stride, K, T, L, upr, uar, ent, jac);
    return SR_OK;
}

int launch_batch_stats(const float* adv, const uint8_t* stop, int32_t n_groups, int32_t N,
                       int64_t* counts, double* sumsq, cudaStream_t s) {
    const bool vec4 = (N % 4 == 0) && (reinterpret_cast<uintptr_t>(adv) & 15) == 0;
    unsigned long long* const c = reinterpret_cast<unsigned long long*>(counts);
    // One cluster while its eight SMs take no longer than clears, grid and atomics do (8 us).  That goes with the
    // bytes, sooner without 16-byte loads, and sooner where the rows of a warp's lanes fall on the
    // same lines of L1.  Cluster / grid in us: 16384 x 13 5.8 / 8.1, 16384 x 24 6.7 / 8.4, 12000 x 32 12.3 / 8.4;
    // rows off 16 bytes, 8192 x 20 5.6 / 8.4, 12000 x 16 12.4 / 8.2, 8192 x 32 20.8 / 10.8.
    const long long most = N % 16 == 0 ? (vec4 ? 1 << 18 : 1 << 17) : (vec4 ? 3 << 17 : 1 << 18);
    if (n_groups <= kClusterCtas * 1024 * 2 && (long long)n_groups * N <= most) {
        int ctas = 1;
        while (ctas < kClusterCtas && ctas * 256 < n_groups) ctas *= 2;
        int threads = 256;                           // up to two groups per thread
        if (n_groups > ctas * 256) threads = n_groups >= ctas * 1024 ? 1024 : ((n_groups + ctas - 1) / ctas + 31) & ~31;
        return launch_as(true, ctas, "batch_stats_kernel", batch_stats_kernel<true>, ctas, threads, 0, s, adv, stop, N, n_groups, vec4, c, sumsq);
    }
    SR_CUDA_TRY(cudaMemsetAsync(counts, 0, 3 * sizeof(int64_t), s));
    SR_CUDA_TRY(cudaMemsetAsync(sumsq, 0, 2 * sizeof(double), s));
    int dev = 0, sms = 0;
    SR_CUDA_TRY(cudaGetDevice(&dev));
    SR_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int want = (n_groups + 255) / 256;
    const int cap = sms * 16;
    const int blocks = want < cap ? want : cap;
    SR_LAUNCH("batch_stats_kernel", batch_stats_kernel<false>, blocks, 256, 0, s, adv, stop, N, n_groups, vec4, c, sumsq);
    return SR_OK;
}

int launch_or_rule(const double* mean, const int32_t* lens, const uint8_t* done, int32_t n_groups,
                   int32_t N, int32_t K, double threshold, double tau_high, double* tau,
                   uint8_t* stop, cudaStream_t s) {
    if (n_groups == 0) return SR_OK;
    const bool vec4 = done == nullptr && (N % 4 == 0) && (reinterpret_cast<uintptr_t>(lens) & 15) == 0;
    SR_LAUNCH("or_rule_kernel", or_rule_kernel, (n_groups + 255) / 256, 256, 0, s, mean, lens, done, n_groups, N, K, threshold, tau_high, vec4, tau, stop);
    return SR_OK;
}

}  // namespace sr
