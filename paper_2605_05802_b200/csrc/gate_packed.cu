// sr_gate_host_packed: the gate on HOST input in packed (ragged) form.  Rollout prefixes
// of very different lengths (token-level gates) waste a third or more of a padded
// [rows][stride] array, and over a host link the copy, not the kernels, sets the time of
// a call; here only the symbols that exist cross the link.  On the device a small kernel
// spreads them into the padded rows the gate kernels read.
#include "common.cuh"

namespace sr {
namespace {

constexpr int kUnpackThreads = 256;

// One warp per row: row r of the chunk holds symbols [start[r], start[r + 1]) of `packed`
// (indices relative to packed[0] of the whole batch); the first min(len, stride) of them
// go to the row's padded slot, the full length to lens.
__global__ void __launch_bounds__(kUnpackThreads)
unpack_rows_kernel(const int32_t* __restrict__ packed, const long long* __restrict__ start,
                   int rows, int stride, int32_t* __restrict__ seqs, int32_t* __restrict__ lens) {
    grid_begin();
    const int row = blockIdx.x * (kUnpackThreads / 32) + (threadIdx.x >> 5);
    if (row >= rows) return;
    const int lane = threadIdx.x & 31;
    const long long b = start[row], e = start[row + 1];
    const long long len = e - b;
    const int n = (int)(len < (long long)stride ? len : (long long)stride);
    const int32_t* src = packed + b;
    int32_t* dst = seqs + (size_t)row * stride;
    for (int t = lane; t < n; t += 32) dst[t] = __ldg(src + t);
    if (lane == 0) lens[row] = (int)(len < 0x7FFFFFFFLL ? len : 0x7FFFFFFFLL);
}

// What the pieces of a chunked transfer need on the kernels' stream: wait for the piece's
// copy, then spread its rows.
struct FeedCtx {
    const int32_t* d_packed;
    const long long* d_start;
    int32_t* d_seqs;
    int32_t* d_lens;
    int N, stride;
    cudaEvent_t* copied;      // one event per piece, recorded on the copy stream
    int pieces, n_groups;
    int first;                // the batch's group that is this feed's first
};

// Groups of a feed before its piece c, as the pipeline cuts them.
int piece_begin(int n_groups, int pieces, int c) { return (int)((long long)n_groups * c / pieces); }

int unpack_rows(const FeedCtx& f, int g0, int g1, cudaStream_t s) {
    const size_t row0 = (size_t)g0 * f.N;
    const int rows = (g1 - g0) * f.N;
    SR_LAUNCH("unpack_rows_kernel", unpack_rows_kernel, (rows + kUnpackThreads / 32 - 1) / (kUnpackThreads / 32), kUnpackThreads, 0, s,  f.d_packed, f.d_start + row0, rows, f.stride, f.d_seqs + row0 * f.stride, f.d_lens + row0);
    return SR_OK;
}

int feed_piece(void* ctx, int g0, int g1, cudaStream_t s) {
    const FeedCtx& f = *static_cast<const FeedCtx*>(ctx);
    // the piece index follows from g0 the same way the pipeline cut the groups
    int c = 0;
    while (c + 1 < f.pieces && piece_begin(f.n_groups, f.pieces, c + 1) <= g0) ++c;
    SR_CUDA_TRY(cudaStreamWaitEvent(s, f.copied[c], 0));
    return unpack_rows(f, f.first + g0, f.first + g1, s);
}

// Events of one call; destroyed when the call returns, whichever way (an event that is
// still pending is released by the driver once it has completed).
struct EventSet {
    cudaEvent_t ev[8];
    int n = 0;
    cudaError_t add() {
        const cudaError_t e = cudaEventCreateWithFlags(&ev[n], cudaEventDisableTiming);
        if (e == cudaSuccess) ++n;
        return e;
    }
    ~EventSet() { for (int k = 0; k < n; ++k) cudaEventDestroy(ev[k]); }
};

// Symbols from which they are sent in pieces: less is on the link for no longer than the launches of a pass per piece
// take (80 groups of 8 at K = 48 99 us in pieces, 38 in one; 200 at 256, 1.6 MB, 138 and 97; at 3 to 4 MB both are alike).
constexpr long long kPieceBytes = 2ll << 20;

// Symbols from which the gate itself runs in two parts, the first one under the copy of the second.  It pays once the copy of
// half the batch takes longer than the tails of a second set of launches: in one part / in two, 21 MB of ragged texts of
// 1024 743 / 688 us, 34 MB of full ones 1033 / 902, 17 MB of pairs of 700 478 / 472; 13 MB of groups of 4 432 / 455,
// 9 MB of ragged texts 420 / 453.
constexpr long long kPartBytes = 14ll << 20;

struct PackedArena {
    size_t off_packed, off_start, inner, total;     // `inner`: where the padded-input arena begins
};

PackedArena packed_arena(int32_t n_groups, int32_t N, int32_t stride, int32_t K) {
    PackedArena p;
    size_t off = 0;
    p.off_packed = off; off = align_up(off + (size_t)n_groups * N * stride * 4, 256);
    p.off_start = off;  off = align_up(off + ((size_t)n_groups * N + 1) * 8, 256);
    p.inner = off;
    p.total = off + host_arena(n_groups, N, stride, K).total;
    return p;
}

}  // namespace
}  // namespace sr

using namespace sr;

extern "C" {

size_t sr_gate_host_packed_arena_bytes(int32_t n_groups, int32_t N, int32_t stride, int32_t K) {
    if (n_groups < 0 || N < 2 || N > SR_MAX_N || stride < 0 || (stride & 3) || K < 0 || K > stride ||
        K > SR_MAX_K)
        return 0;
    return packed_arena(n_groups, N, stride, K).total;
}

int sr_gate_host_packed(const int32_t* symbols, const int64_t* row_start, int32_t n_groups, int32_t N,
                        int32_t stride, int32_t K, double threshold, int32_t norm_mode,
                        int32_t* pair_dist, int32_t* pair_sum, double* mean, uint8_t* stop,
                        int32_t* status, void* arena, size_t arena_bytes, void* stream,
                        void* copy_stream) {
    if (n_groups < 0 || N < 2 || N > SR_MAX_N) return SR_ERR_BAD_N;
    if (stride < 0 || (stride & 3) || K < 0 || K > stride || K > SR_MAX_K) return SR_ERR_BAD_K;
    if (norm_mode != SR_NORM_MAXLEN && norm_mode != SR_NORM_NONE) return SR_ERR_BAD_MODE;
    if (n_groups == 0) return SR_OK;
    if (row_start == nullptr || stop == nullptr) return SR_ERR_NULL;
    const size_t rows = (size_t)n_groups * N;
    // the offsets are host memory: checked here, before anything is enqueued
    if (row_start[0] != 0) return SR_ERR_BAD_OFFSETS;
    for (size_t r = 0; r < rows; ++r)
        if (row_start[r + 1] < row_start[r]) return SR_ERR_BAD_OFFSETS;
    const long long total = row_start[rows];
    if (total > 0 && symbols == nullptr) return SR_ERR_NULL;
    // a row longer than `stride` is legal (only its first K <= stride symbols matter), but the
    // packed staging area is sized for rows * stride symbols
    if ((unsigned long long)total > (unsigned long long)rows * (unsigned long long)stride)
        return SR_ERR_BAD_OFFSETS;
    const PackedArena pa = packed_arena(n_groups, N, stride, K);
    if (arena == nullptr || arena_bytes < pa.total || (reinterpret_cast<uintptr_t>(arena) & 255) != 0)
        return SR_ERR_WORKSPACE;
    unsigned char* d = static_cast<unsigned char*>(arena);
    unsigned char* di = d + pa.inner;
    const HostArena h = host_arena(n_groups, N, stride, K);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t P = pairs_of(N);
    int32_t* d_packed = reinterpret_cast<int32_t*>(d + pa.off_packed);
    long long* d_start = reinterpret_cast<long long*>(d + pa.off_start);
    int32_t* d_seqs = reinterpret_cast<int32_t*>(di + h.off_seqs);
    int32_t* d_lens = reinterpret_cast<int32_t*>(di + h.off_lens);
    GateArgs ga{d_seqs, d_lens, n_groups, N, stride, K, threshold, norm_mode,
                pair_dist ? reinterpret_cast<int32_t*>(di + h.off_dist) : nullptr,
                pair_sum ? reinterpret_cast<int32_t*>(di + h.off_sum) : nullptr,
                mean ? reinterpret_cast<double*>(di + h.off_mean) : nullptr,
                di + h.off_stop, status ? reinterpret_cast<int32_t*>(di + h.off_status) : nullptr};
    FeedCtx f{d_packed, d_start, d_seqs, d_lens, N, stride, nullptr, 1, n_groups, 0};
    if (status) SR_CUDA_TRY(cudaMemcpyAsync(di + h.off_status, status, 4, cudaMemcpyHostToDevice, s));
    cudaStream_t cs = static_cast<cudaStream_t>(copy_stream);
    // With a copy stream and long prefixes the symbols go over in pieces of whole groups, and the per-group pass of the gate
    // (match streams) runs on each piece while the next one is still on the link.  The rest of the gate runs once over the whole batch,
    // or, where there is enough to copy, once over the first half, while the second is on the link, and once over that.  The
    // two use the same workspace, one after the other.  (More parts lose: the few long pairs of a quarter set the time of its
    // recurrence.)
    if (cs != nullptr && cs != s && K > 32 && n_groups >= 64 && total * 4 >= kPieceBytes) {
        constexpr int kMostPieces = 4;
        const bool halves = total * 4 >= kPartBytes;
        const int parts = halves ? 2 : 1, pieces[2] = {halves ? 2 : kMostPieces, 1};
        const int cut[3] = {0, halves ? n_groups / 2 : n_groups, n_groups};
        EventSet events;                                  // [0] fork, then one for each piece that has been copied
        for (int k = 0; k < 1 + kMostPieces; ++k) SR_CUDA_TRY(events.add());
        // the copies must not overtake earlier work on `stream` that uses the arena
        SR_CUDA_TRY(cudaEventRecord(events.ev[0], s));
        SR_CUDA_TRY(cudaStreamWaitEvent(cs, events.ev[0], 0));
        SR_CUDA_TRY(cudaMemcpyAsync(d_start, row_start, (rows + 1) * 8, cudaMemcpyHostToDevice, cs));
        int at = 1;
        for (int p = 0; p < parts; ++p) {
            for (int c = 0; c < pieces[p]; ++c) {
                const size_t row0 = (size_t)(cut[p] + piece_begin(cut[p + 1] - cut[p], pieces[p], c)) * N;
                const size_t row1 = (size_t)(cut[p] + piece_begin(cut[p + 1] - cut[p], pieces[p], c + 1)) * N;
                const long long s0 = row_start[row0], s1 = row_start[row1];
                if (s1 > s0)
                    SR_CUDA_TRY(cudaMemcpyAsync(d_packed + s0, symbols + s0, (size_t)(s1 - s0) * 4,
                                                cudaMemcpyHostToDevice, cs));
                SR_CUDA_TRY(cudaEventRecord(events.ev[at++], cs));
            }
        }
        at = 1;
        for (int p = 0; p < parts; ++p) {
            const size_t g0 = cut[p], row0 = g0 * N;
            f.copied = events.ev + at;
            f.pieces = pieces[p];
            f.first = cut[p];
            f.n_groups = cut[p + 1] - cut[p];
            at += pieces[p];
            GateArgs part = ga;
            part.seqs += row0 * stride;
            part.lens += row0;
            part.n_groups = f.n_groups;
            if (part.pair_dist) part.pair_dist += g0 * P;
            if (part.pair_sum) part.pair_sum += g0;
            if (part.mean) part.mean += g0;
            part.stop += g0;
            const GroupFeed feed{f.pieces, feed_piece, &f};
            const int rc = launch_gate_multi(part, di + h.off_ws, h.total - h.off_ws, s, nullptr, false, nullptr, &feed);
            if (rc != SR_OK) return rc;
        }
    } else {
        SR_CUDA_TRY(cudaMemcpyAsync(d_start, row_start, (rows + 1) * 8, cudaMemcpyHostToDevice, s));
        if (total > 0)
            SR_CUDA_TRY(cudaMemcpyAsync(d_packed, symbols, (size_t)total * 4, cudaMemcpyHostToDevice, s));
        int rc = unpack_rows(f, 0, n_groups, s);
        if (rc != SR_OK) return rc;
        rc = sr_gate(ga.seqs, ga.lens, n_groups, N, stride, K, threshold, norm_mode, ga.pair_dist,
                     ga.pair_sum, ga.mean, ga.stop, ga.status, di + h.off_ws, h.total - h.off_ws, stream);
        if (rc != SR_OK) return rc;
    }
    if (pair_dist)
        SR_CUDA_TRY(cudaMemcpyAsync(pair_dist, di + h.off_dist, (size_t)n_groups * P * 4,
                                    cudaMemcpyDeviceToHost, s));
    if (pair_sum)
        SR_CUDA_TRY(cudaMemcpyAsync(pair_sum, di + h.off_sum, (size_t)n_groups * 4, cudaMemcpyDeviceToHost, s));
    if (mean)
        SR_CUDA_TRY(cudaMemcpyAsync(mean, di + h.off_mean, (size_t)n_groups * 8, cudaMemcpyDeviceToHost, s));
    SR_CUDA_TRY(cudaMemcpyAsync(stop, di + h.off_stop, (size_t)n_groups, cudaMemcpyDeviceToHost, s));
    if (status)
        SR_CUDA_TRY(cudaMemcpyAsync(status, di + h.off_status, 4, cudaMemcpyDeviceToHost, s));
    return SR_OK;
}

}  // extern "C"
