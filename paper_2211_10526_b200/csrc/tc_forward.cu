// Orchestration of the tensor-core path: state build -> split reduction -> apply, in stream order
// (the stream is the only synchronisation between the phases; no kernel waits on another).
#include "tc_host.cuh"
#include "state_splits.cuh"

#include <cstdlib>

namespace castling {
namespace tc {

namespace {
constexpr int kStateTile = 128;  // 128-byte rows per UMMA stage of the state kernel
// Automatic dispatch takes width-32 shapes that fit no 128-byte rows (odd grid widths or token counts, an odd number of heads
// side by side) from this many tokens in all planes on.  The kernels are faster below it too (300 tokens: 6 us against 17 us on
// the CUDA cores; 2 x 6 planes of 33 x 21: 8 us against 25 us), but the tests hold the smallest shapes to the CUDA-core family.
constexpr long long kNarrowMinTokens = 4096;
}

namespace {
// The non-default variants put two width-32 rows side by side in one of 128 bytes: two adjacent tokens of one head (tokens
// contiguous, even grid width), or the same token of two adjacent heads (head stride 32, as in a token-major [B,N,H,32]
// tensor with an even number of heads).
bool head_pairs(const Problem& p) {
    return p.d == 32 && p.H % 2 == 0 && p.hdiv == p.H && p.head0 == 0 && p.lq.head == 32 && p.lk.head == 32 &&
           p.lv.head == 32 && p.lo.head == 32;
}
}  // namespace

// Width-32 heads whose 64-byte rows lie next to one another in memory, token after token or head after head.
static bool dense_rows(const Problem& p) {
    return p.d == 32 && (p.contiguous_tokens() || (p.hdiv == p.H && p.lq.head == 32 && p.lk.head == 32 && p.lv.head == 32 && p.lo.head == 32));
}

// bf16, 3x3 or 5x5 filters, head width 64, or one of the width-32 arrangements above.
bool supports(const Problem& p) {
    if (!p.bf16 || (p.ksize != 3 && p.ksize != 5)) return false;
    return p.d == 64 || dense_rows(p);
}

int rows_per_head(int N, int d) { return d == 32 ? (N + 1) / 2 : N; }

// Planes of fewer than 48 tokens stay on the CUDA cores, where their operands are fp32 and where the tests hold them.  It is not the
// time that draws the line (CUDA cores / these kernels, from a graph): 64 x 12 planes of 4 x 4, width 32 13.6 / 12.8 us, 8 x 8 planes of
// 4 x 4 5.7 / 6.6, 64 x 8 of 6 x 6 14.1 / 10.0; width 64, 64 x 12 planes of 4 x 4 28.9 / 11.9.
bool preferred(const Problem& p) {
    return supports(p) && p.N >= 48 && (p.d == 64 || token_pairs(p) || head_pairs(p) || (long long)p.BH * p.N >= kNarrowMinTokens);
}

int choose_splits(int BH, int N) { return most_splits(BH, (N + kStateTile - 1) / kStateTile, device_sm_count()); }

// The state kernel on rows of 128 bytes per plane, split as the device holds the clusters.
static cudaError_t launch_split_state(const Problem& p, int rows, float* partial, float* state, unsigned* counters, unsigned* status, cudaStream_t stream) {
    const int tiles = (rows + kStateTile - 1) / kStateTile;
    const StateSplits s = state_splits(p.BH, tiles, device_sm_count(), p.d == 32, [](int P) { return state_clusters_at_once(P); });
    return launch_state(p, partial, state, counters, s.P, (tiles + s.P - 1) / s.P, s.clustered, status, stream);
}

// CASTLING_TC_ONE_KERNEL=1 in the environment selects the one-kernel forward (state and apply pipelines side
// by side in every CTA) instead of the separate state and apply kernels, which measure faster (read once).
static bool two_kernels() {
    static const bool one = [] { const char* e = getenv("CASTLING_TC_ONE_KERNEL"); return e && e[0] == '1'; }();
    return !one;
}

// CASTLING_TC_CLUSTER=1 in the environment selects the cluster-per-plane forward where the shape allows it.
static bool cluster_enabled() {
    static const bool on = [] { const char* e = getenv("CASTLING_TC_CLUSTER"); return e && e[0] == '1'; }();
    return on;
}

cudaError_t forward(const Problem& p_in, float* ws_state, float* ws_partial, unsigned* counters, unsigned* status,
                    cudaStream_t stream, int* launches, KernelTimer* timer) {
    *launches = 0;
    Problem p = p_in;
    // What the packed 128-byte rows do not take, and planes too small to fill their tiles, have the precision of fp32 operands, as
    // on the CUDA cores: unit keys and scaled states as pairs.  Relative error against 64 bits of the bf16 outputs, CUDA
    // cores / single bf16 / pairs: 64 x 8 planes of 7 x 7 1.65499e-3 / 1.67565e-3 / 1.65499e-3, 8 x 8 of 50 x 75, 5 x 5 filters,
    // 1.66210e-3 / 1.68312e-3 / 1.66210e-3, 64 x 8 of 8 x 8 1.65823e-3 / 1.67885e-3 / 1.65823e-3.  Time: 18.4 / 10.3 / 11.9 us,
    // 245 / 30.6 / 33.2, 21.4 / 10.7 / 12.6.
    p.fine = p.d == 32 && !head_pairs(p) && (!token_pairs(p) || p.N < 96);
    const bool fine = p.fine;
    cudaError_t e;
    if (!p.rownorm && fused_supports(p)) {  // a whole (b,h) fits in shared memory: one kernel, no workspace
        e = launch_fused(p, status, stream);
        if (e != cudaSuccess) return e;
        ++*launches;
        timer->mark(stream, "tc_fused");
        return cudaSuccess;
    }
    bool rows128 = p.d == 64 || token_pairs(p);   // every row of 128 bytes is full
    if (!rows128 && head_pairs(p)) {
        // heads (2m, 2m+1) side by side = one width-64 plane whose state is block diagonal
        p.d = 64; p.H /= 2; p.BH /= 2; p.hdiv = p.H; p.blockdiag = true;
        p.lq.head = p.lk.head = p.lv.head = p.lo.head = 64;
        rows128 = true;
    }
    rows128 = rows128 && !p.rownorm;   // the row sums are carried by the separate state and apply kernels only
    if (const int C = (cluster_enabled() && rows128) ? cluster_size(p) : 0) {
        e = launch_cluster(p, C, status, stream);
        if (e != cudaSuccess) return e;
        ++*launches;
        timer->mark(stream, "tc_cluster");
        return cudaSuccess;
    }
    if (!two_kernels() && rows128 && pipe_supports(p)) {
        // state and apply pipelines in one persistent kernel: V is read from memory once
        e = launch_pipe(p, ws_state, ws_partial, counters, status, stream);
        if (e != cudaSuccess) return e;
        ++*launches;
        timer->mark(stream, "tc_pipe");
    } else {
        p = p_in;   // width-32 heads in 64-byte rows of their own
        p.narrow = p.d == 32;
        p.fine = fine;
        e = launch_split_state(p, rows_per_head(p.N, p.d), ws_partial, ws_state, counters, status, stream);
        if (e != cudaSuccess) return e;
        ++*launches;
        timer->mark(stream, "tc_state");
        e = launch_apply(p, ws_state, status, stream);
        if (e != cudaSuccess) return e;
        ++*launches;
        timer->mark(stream, "tc_apply");
    }
    if (p.prefix > 0) {
        e = launch_prefix_rows(p, ws_state, stream);
        if (e != cudaSuccess) return e;
        ++*launches;
        timer->mark(stream, "tc_prefix_rows");
    }
    return cudaSuccess;
}

bool shard_supports(const Problem& p) {
    return p.bf16 && p.d == 64 && (p.ksize == 3 || p.ksize == 5) && p.prefix == 0 && !p.rownorm && p.N >= 48;
}

cudaError_t shard_state(const Problem& p, float* state_out, float* ws_partial, unsigned* counters, unsigned* status,
                        cudaStream_t stream, int* launches, KernelTimer* timer) {
    *launches = 0;
    const cudaError_t e = launch_split_state(p, p.N, ws_partial, state_out, counters, status, stream);
    if (e != cudaSuccess) return e;
    ++*launches;
    timer->mark(stream, "tc_state");
    return cudaSuccess;
}

cudaError_t shard_apply(const Problem& p, const float* state, unsigned* status, cudaStream_t stream, int* launches,
                        KernelTimer* timer) {
    *launches = 0;
    const cudaError_t e = launch_apply(p, state, status, stream);
    if (e != cudaSuccess) return e;
    ++*launches;
    timer->mark(stream, "tc_apply");
    return cudaSuccess;
}

}  // namespace tc
}  // namespace castling
