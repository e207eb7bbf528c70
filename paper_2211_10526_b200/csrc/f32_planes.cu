// fp32 forward of short planes (head width 32 or 64, 3x3 or 5x5 filters, at most 256 tokens):
//     out_t = (1/pi) q^_t (K^^T V) + 1/2 sum_n v_n + bias + DWConv(V)_t                    (Eq. 9)
// A cluster of 1, 2 or 4 CTAs per plane, each with a band of its grid rows (the first one with the leading off-grid tokens too) in
// shared memory: K and Q as tokens, V as the band with its halo (zero outside the grid), all by TMA.  One kernel does the following for its
// plane; where planes are few or of a column or two, one kernel stops after 2 and the other does 3, with bands and runs of its own.
//   1. rows of K to unit rows in place, the token sum of V, 1 / max(||q||, eps)
//   2. the band's state: a thread owns 8 x 8 of S and every G-th token (G groups of (D/8)^2 threads); the groups meet in shared memory,
//      the bands through distributed shared memory, both in a fixed order
//   3. a thread owns a run of 8 tokens (two kernels: 2) x 4 channels: the contraction over the key features, then the convolution, its window sliding
//      along the run
// What bounds it: the chain of these phases.  On one CTA a plane of 14 x 14 tokens, width 32, took 17 000 cycles (K and Q rows 5 600, one row
// at a time; state 2 800 and its parts 1 900; attention 3 700, convolution 1 700): so rows go four at a time and a few planes are
// shared by the CTAs of a cluster.
// Measured (from a graph, us; the two kernels of f32_kernels.cu, or simt_fused_kernel from 64 planes on, before): width 32, 14 x 14, 8 planes
// 10.4 -> 6.7 (9.8 with one CTA a plane), 64 planes 26.8 -> 8.3, 768 planes 106 -> 45; width 64, 8 planes 18.4 -> 10.0 (20.3), 144 planes 38 -> 22.
#include "tc_common.cuh"
#include "tc_host.cuh"

namespace castling {
namespace {

using tc::ffma2;
using tc::cluster_arrive;
using tc::cluster_wait;
using tc::ld_peer;
using tc::mbar_wait;

constexpr int kThreads = 256;
enum { kWhole, kState, kRows };   // the forward; its state and, in a second kernel, its output

template <int D, int KS> struct PlaneGeo {
    static constexpr int kSide = D / 8, kGroup = kSide * kSide, G = kThreads / kGroup;          // state: threads per group, groups
    static constexpr int kShuffled = kGroup < 32 ? 32 / kGroup : 1, kParts = G / kShuffled;     // groups added within a warp; what is left
    static constexpr int kChunks = D / 4, kRowsPass = kThreads / kChunks;                       // 16-byte chunks of a row, rows at a time
    static constexpr int kRuns = kThreads / kChunks;                                            // runs of tokens at a time
    static constexpr int R = KS / 2;
    // floats: S' | 1/2 s | bias | filters (tap-major) | sums of V by rows; then by size: 1/||q|| | K, later the groups' parts of S | Q | V
    static constexpr int kOffC = D * D, kOffB = kOffC + D, kOffW = kOffB + D, kOffSum = kOffW + KS * KS * D, kOffRq = kOffSum + kRowsPass * D;
};

struct F32PlaneParams {
    const float *w, *bias;
    float *out, *state;                           // state [BH][D*D + D]: S, s (two kernels)
    Layout lo;
    int H, head0, hdiv, prefix, gridH, gridW;
    int bands, band_rows, tokens;                 // CTAs per plane; rows of a band and tokens of its copies, at most
    int off_k, off_q, off_v, off_lead, off_bar;   // floats; V's leading tokens behind the grid with its halo
    float eps2;
    unsigned* status;
};

template <int D, int KS, int PART>
__global__ void __launch_bounds__(kThreads, D == 32 ? 2 : 1)
f32_plane_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmV,
                 const __grid_constant__ CUtensorMap tmLead, const F32PlaneParams prm) {
    using G = PlaneGeo<D, KS>;
    constexpr int R = G::R;
    constexpr unsigned kBit = tc::kStatusFusedTimeout;
    extern __shared__ uint8_t smem_raw[];
    float* smem = reinterpret_cast<float*>(tc::align_smem(smem_raw));
    float *k_s = smem + prm.off_k, *q_s = smem + prm.off_q, *v_s = smem + prm.off_v, *lead_s = smem + prm.off_lead, *rq_s = smem + G::kOffRq;
    uint64_t* kv_full = reinterpret_cast<uint64_t*>(smem + prm.off_bar);   // TMA: K and V landed
    uint64_t* q_full = kv_full + 1;                                        // TMA: Q landed
    volatile int* abort_flag = reinterpret_cast<volatile int*>(q_full + 1);
    const int tid = threadIdx.x, bh = blockIdx.x / prm.bands, rank = blockIdx.x % prm.bands;
    const int W = prm.gridW, pitch = W + 2 * R, h = (prm.head0 + bh) % prm.H;
    const int row0 = prm.gridH * rank / prm.bands, n_rows = prm.gridH * (rank + 1) / prm.bands - row0;
    const int lead_n = rank == 0 ? prm.prefix : 0, N = lead_n + n_rows * W;   // tokens of the band, the leading ones first
    const int first = rank == 0 ? 0 : prm.prefix + row0 * W;                  // token of the plane
    const int lc = (tid % G::kChunks) * 4, lr = tid / G::kChunks;

    if (tid == 0) {
        tc::mbar_init(kv_full, 1); tc::mbar_init(q_full, 1);
        *abort_flag = 0;
        tc::mbar_fence_init();
        tc::tma_prefetch_desc(&tmK); tc::tma_prefetch_desc(&tmV); tc::tma_prefetch_desc(&tmQ);
    }
    // Launched programmatically dependent on whatever precedes it in the stream, and so is what follows.  The second kernel loads Q and V
    // before the first one has finished, which lets it start only once what was before it has.
    if (PART == kWhole) tc::pdl_launch_dependents();
    if (PART != kRows) tc::pdl_wait_primary();
    if (PART != kWhole) tc::pdl_launch_dependents();
    if (tid == 0) {
        const int pb = bh / prm.hdiv, ph = bh - pb * prm.hdiv;
        tc::mbar_expect_tx(kv_full, ((PART != kRows ? prm.tokens : 0) + (prm.band_rows + 2 * R) * pitch + (lead_n ? 16 : 0)) * D * 4);
        if (PART != kRows) tc::tma_load_4d(k_s, &tmK, kv_full, 0, first, ph, pb);
        tc::tma_load_5d(v_s, &tmV, kv_full, 0, -R, row0 - R, ph, pb);
        if (lead_n) tc::tma_load_4d(lead_s, &tmLead, kv_full, 0, 0, ph, pb);
        if (PART != kState) {
            tc::mbar_expect_tx(q_full, prm.tokens * D * 4);
            tc::tma_load_4d(q_s, &tmQ, q_full, 0, first, ph, pb);
        }
    }
    if (PART != kState) {
    for (int i = tid; i < KS * KS * D; i += kThreads) smem[G::kOffW + i] = __ldg(prm.w + ((size_t)(h * D + i % D)) * (KS * KS) + i / D);
    if (tid < D) smem[G::kOffB + tid] = prm.bias ? __ldg(prm.bias + h * D + tid) : 0.f;
    }
    __syncthreads();   // the barriers are set up

    // V of the band's token n
    const uint32_t magic = 0xffffffffu / (uint32_t)W + 1;   // m / W is the high word of m * magic (W = 1: m itself)
    auto v_row = [&](int n) -> const float* {
        const int m = n - lead_n, y = W == 1 ? m : (int)__umulhi((uint32_t)m, magic);
        return m < 0 ? lead_s + n * D : v_s + (m + 2 * R * y + R * pitch + R) * D;
    };
    // f(row, this thread's chunk of it, 1 / max(norm, eps)), four rows at a time
    auto rows = [&](float* base, auto f) {
        for (int r0 = 0; r0 < N; r0 += 4 * G::kRowsPass) {   // whole warps: a row is shared by lanes
            float4 x[4];
            float ss[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = r0 + u * G::kRowsPass + lr;
                x[u] = r < N ? *reinterpret_cast<const float4*>(base + r * D + lc) : make_float4(0.f, 0.f, 0.f, 0.f);
                ss[u] = fmaf(x[u].x, x[u].x, fmaf(x[u].y, x[u].y, fmaf(x[u].z, x[u].z, x[u].w * x[u].w)));
            }
#pragma unroll
            for (int o = G::kChunks / 2; o > 0; o >>= 1)
#pragma unroll
                for (int u = 0; u < 4; ++u) ss[u] += __shfl_xor_sync(0xffffffffu, ss[u], o);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = r0 + u * G::kRowsPass + lr;
                const float f1 = inv_sqrt(fmaxf(ss[u], prm.eps2));
                if (r < N) f(r, x[u], f1);
            }
        }
    };
    bool ok = mbar_wait(kv_full, 0, abort_flag, prm.status, kBit);
    if (ok && PART != kRows) {
        rows(k_s, [&](int n, float4 x, float r) { *reinterpret_cast<float4*>(k_s + n * D + lc) = make_float4(x.x * r, x.y * r, x.z * r, x.w * r); });
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int n = lr; n < N; n += G::kRowsPass) {
            const float4 x = *reinterpret_cast<const float4*>(v_row(n) + lc);
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
        *reinterpret_cast<float4*>(smem + G::kOffSum + lr * D + lc) = s;
    }
    if (PART != kState) {
        ok = ok && mbar_wait(q_full, 0, abort_flag, prm.status, kBit);
        if (ok) rows(q_s, [&](int n, float4, float r) { if (lc == 0) rq_s[n] = r; });
    }
    // Giving up: the copies in flight land before shared memory goes away, and the barriers of the cluster are met all the same.
    ok = !__syncthreads_or(!ok);
    if (!ok && tid == 0) {
        for (int spin = 0; spin < (1 << 20) && !tc::mbar_try_wait(kv_full, 0); ++spin) {}
        for (int spin = 0; PART != kState && spin < (1 << 20) && !tc::mbar_try_wait(q_full, 0); ++spin) {}
    }

    if (PART != kRows) {   // ---- state ----
        const int g = tid / G::kGroup, t = tid % G::kGroup, ti = t / G::kSide, tj = t % G::kSide;
        float2 acc[8][4];
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int n = g; n < N; n += G::G) {
            const float* v = v_row(n);
            const float4 a0 = *reinterpret_cast<const float4*>(k_s + n * D + ti * 8), a1 = *reinterpret_cast<const float4*>(k_s + n * D + ti * 8 + 4);
            const float4 b0 = *reinterpret_cast<const float4*>(v + tj * 4), b1 = *reinterpret_cast<const float4*>(v + D / 2 + tj * 4);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float2 b[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
            for (int x = 0; x < 8; ++x)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[x][c] = ffma2(make_float2(a[x], a[x]), b[c], acc[x][c]);
        }
        if (G::kShuffled > 1) {
#pragma unroll
            for (int x = 0; x < 8; ++x)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    acc[x][c].x += __shfl_xor_sync(0xffffffffu, acc[x][c].x, G::kGroup);
                    acc[x][c].y += __shfl_xor_sync(0xffffffffu, acc[x][c].y, G::kGroup);
                }
        }
        __syncthreads();   // K is dead
        float* part = k_s + (g / G::kShuffled) * (D * D);
        if (g % G::kShuffled == 0) {
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                float* row = part + (ti * 8 + x) * D;
                *reinterpret_cast<float4*>(row + tj * 4) = make_float4(acc[x][0].x, acc[x][0].y, acc[x][1].x, acc[x][1].y);
                *reinterpret_cast<float4*>(row + D / 2 + tj * 4) = make_float4(acc[x][2].x, acc[x][2].y, acc[x][3].x, acc[x][3].y);
            }
        }
        __syncthreads();
        for (int i = tid * 4; i < D * D; i += kThreads * 4) {   // the parts in their order
            float4 s = *reinterpret_cast<const float4*>(k_s + i);
#pragma unroll
            for (int p = 1; p < G::kParts; ++p) {
                const float4 x = *reinterpret_cast<const float4*>(k_s + p * (D * D) + i);
                s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
            }
            *reinterpret_cast<float4*>(k_s + i) = s;
        }
        if (tid < D) {
            float s = 0.f;
#pragma unroll 8
            for (int r = 0; r < G::kRowsPass; ++r) s += smem[G::kOffSum + r * D + tid];
            smem[G::kOffSum + tid] = s;   // column tid is this thread's alone
        }
        // the bands of the plane
        if (prm.bands > 1) { cluster_arrive(); cluster_wait(); } else { __syncthreads(); }
        // (two kernels: each CTA its share of the words)
        const int share = PART == kState ? (D * D + D) / 4 / prm.bands : (D * D + D) / 4, begin = PART == kState ? rank * share : 0;
        for (int u = tid; u < share; u += kThreads) {
            const int i = (begin + u) * 4;
            const float* at = i < D * D ? k_s + i : smem + G::kOffSum + i - D * D;
            float4 s = prm.bands > 1 ? ld_peer(reinterpret_cast<const float4*>(at), 0) : *reinterpret_cast<const float4*>(at);
            for (int p = 1; p < prm.bands; ++p) {
                const float4 x = ld_peer(reinterpret_cast<const float4*>(at), p);
                s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
            }
            if (PART == kState) {
                *reinterpret_cast<float4*>(prm.state + (size_t)bh * (D * D + D) + i) = s;
            } else {
                const float f = i < D * D ? kInvPi : 0.5f;
                *reinterpret_cast<float4*>(smem + i) = make_float4(s.x * f, s.y * f, s.z * f, s.w * f);   // 1/2 s follows S'
            }
        }
        if (prm.bands > 1) cluster_arrive();   // the others' states have been read; waited for at the end
        if (PART == kState) { if (prm.bands > 1) cluster_wait(); return; }
        __syncthreads();
    }

    // ---- attention, convolution and output: runs of TOK tokens of a grid row, then of the leading tokens ----
    constexpr int TOK = PART == kRows ? 2 : 8;
    const int per_row = (W + TOK - 1) / TOK, grid_runs = per_row * n_rows, n_runs = ok ? grid_runs + (lead_n + TOK - 1) / TOK : 0;
    const float4 bs = *reinterpret_cast<const float4*>(smem + G::kOffB + lc);
    float* out = prm.out + plane_offset(prm.lo, bh, prm.hdiv) + first * prm.lo.token + lc;
    auto convolve = [&](int run, float2 (&acc)[TOK][2]) {   // of a run on the grid
        const int y = run / per_row, x0 = (run - y * per_row) * TOK;
        const float* vw = v_s + (y * pitch + x0) * D + lc;   // halo row 0, column 0
#pragma unroll 1
        for (int dy = 0; dy < KS; ++dy) {
            float4 f[KS];
#pragma unroll
            for (int dx = 0; dx < KS; ++dx) f[dx] = *reinterpret_cast<const float4*>(smem + G::kOffW + (dy * KS + dx) * D + lc);
#pragma unroll
            for (int c = 0; c < TOK + KS - 1; ++c) {
                const float4 x = *reinterpret_cast<const float4*>(vw + (dy * pitch + c) * D);
#pragma unroll
                for (int dx = 0; dx < KS; ++dx) {
                    const int j = c - dx;   // compile-time after unrolling
                    if (j < 0 || j >= TOK) continue;
                    acc[j][0] = ffma2(make_float2(f[dx].x, f[dx].y), make_float2(x.x, x.y), acc[j][0]);
                    acc[j][1] = ffma2(make_float2(f[dx].z, f[dx].w), make_float2(x.z, x.w), acc[j][1]);
                }
            }
        }
    };
    float2 conv[TOK][2];   // two kernels: the convolution of a run comes first, that of the first run before the state is there
    auto convolve_first = [&](int run) {
#pragma unroll
        for (int j = 0; j < TOK; ++j) { conv[j][0] = make_float2(bs.x, bs.y); conv[j][1] = make_float2(bs.z, bs.w); }
        if (run < grid_runs && run < n_runs) convolve(run, conv);
    };
    if (PART == kRows) {
        convolve_first(lr);
        tc::pdl_wait_primary();
        const float* st = prm.state + (size_t)bh * (D * D + D);
        for (int i = tid * 4; i < D * D + D; i += kThreads * 4) {
            const float4 s = __ldcg(reinterpret_cast<const float4*>(st + i));
            const float f = i < D * D ? kInvPi : 0.5f;
            *reinterpret_cast<float4*>(smem + i) = make_float4(s.x * f, s.y * f, s.z * f, s.w * f);
        }
        __syncthreads();
    }
    const float4 cs = *reinterpret_cast<const float4*>(smem + G::kOffC + lc);
    for (int run = lr; run < n_runs; run += G::kRuns) {
        const bool lead = run >= grid_runs;
        const int y = run / per_row, x0 = (run - y * per_row) * TOK;
        const int n0 = lead ? (run - grid_runs) * TOK : lead_n + y * W + x0, n_run = lead ? lead_n - n0 : W - x0;   // more than TOK: TOK
        float2 acc[TOK][2];
#pragma unroll
        for (int j = 0; j < TOK; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
        const float* q_run = q_s + n0 * D;   // tokens beyond the run are computed and dropped
#pragma unroll 2
        for (int i = 0; i < D; i += 4) {
            float4 a[TOK];
#pragma unroll
            for (int j = 0; j < TOK; ++j) a[j] = *reinterpret_cast<const float4*>(q_run + j * D + i);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 s = *reinterpret_cast<const float4*>(smem + (i + u) * D + lc);
#pragma unroll
                for (int j = 0; j < TOK; ++j) {
                    const float x = u == 0 ? a[j].x : u == 1 ? a[j].y : u == 2 ? a[j].z : a[j].w;
                    acc[j][0] = ffma2(make_float2(x, x), make_float2(s.x, s.y), acc[j][0]);
                    acc[j][1] = ffma2(make_float2(x, x), make_float2(s.z, s.w), acc[j][1]);
                }
            }
        }
        const float4 add = lead || PART == kRows ? cs : make_float4(cs.x + bs.x, cs.y + bs.y, cs.z + bs.z, cs.w + bs.w);
#pragma unroll
        for (int j = 0; j < TOK; ++j) {
            const float rq = rq_s[n0 + j];
            acc[j][0].x = fmaf(acc[j][0].x, rq, add.x); acc[j][0].y = fmaf(acc[j][0].y, rq, add.y);
            acc[j][1].x = fmaf(acc[j][1].x, rq, add.z); acc[j][1].y = fmaf(acc[j][1].y, rq, add.w);
        }
        if (PART == kRows) {
            if (run != lr) convolve_first(run);
#pragma unroll
            for (int j = 0; j < TOK; ++j)
#pragma unroll
                for (int c = 0; c < 2; ++c) { acc[j][c].x += lead ? 0.f : conv[j][c].x; acc[j][c].y += lead ? 0.f : conv[j][c].y; }
        } else if (!lead) {
            convolve(run, acc);
        }
#pragma unroll
        for (int j = 0; j < TOK; ++j)
            if (j < n_run) *reinterpret_cast<float4*>(out + (n0 + j) * prm.lo.token) = make_float4(acc[j][0].x, acc[j][0].y, acc[j][1].x, acc[j][1].y);
    }
    if (PART == kWhole && prm.bands > 1) cluster_wait();   // this band's state has been read
}

constexpr size_t kSmemLimit = 227 * 1024, kAlone = 116 * 1024;   // of which two do not fit a multiprocessor

// Bands of a plane, the shared memory of one, and where its parts begin (floats).
template <int D, int KS>
size_t plane_layout(const Problem& p, int part, F32PlaneParams* prm) {
    using G = PlaneGeo<D, KS>;
    prm->bands = 1;
    // As many CTAs as leave each a multiprocessor and about 40 tokens.  14 x 14, width 32, 8 planes on 1, 2, 4, 8 CTAs each 9.7, 8.0, 7.6, 8.6
    // us, 64 planes 11.7, 10.0; 7 x 7, 8 planes 7.0, 7.3.  Two CTAs of a cluster on one multiprocessor: 32 planes on 4 each 9.7, alone 7.9.
    if (part == kRows) {   // rows for one run per thread, as long as the CTAs are resident at once
        const int rows = G::kRuns / ((p.gridW + 1) / 2) < 1 ? 1 : G::kRuns / ((p.gridW + 1) / 2), want = (p.gridH + rows - 1) / rows;
        const int most = 2 * device_sm_count() / p.BH < 1 ? 1 : 2 * device_sm_count() / p.BH;
        prm->bands = want < most ? want : most;
    } else {
        while (2 * prm->bands * p.BH <= device_sm_count() && 2 * prm->bands <= p.gridH && p.N >= 40 * 2 * prm->bands) prm->bands *= 2;
    }
    prm->band_rows = (p.gridH + prm->bands - 1) / prm->bands;
    prm->tokens = p.prefix + prm->band_rows * p.gridW;
    auto align = [](int f) { return (f + 31) / 32 * 32; };   // 128 bytes: destinations of TMA copies
    const int halo = (p.gridW + KS - 1) * (prm->band_rows + KS - 1), parts = G::kParts * D * D;
    prm->off_k = align(G::kOffRq + prm->tokens + 8);
    prm->off_q = prm->off_k + (part == kRows ? 0 : prm->tokens * D > parts ? prm->tokens * D : parts);
    prm->off_v = prm->off_q + (prm->tokens + 8) * D;         // what a run reads beyond its last token
    prm->off_lead = prm->off_v + (halo + 8) * D;
    prm->off_bar = prm->off_lead + (p.prefix ? 16 * D : 0);
    const size_t bytes = 1024 + (size_t)prm->off_bar * 4 + 32;
    return part != kRows && prm->bands > 1 && bytes < kAlone ? kAlone : bytes;
}


template <int D, int KS, int PART>
cudaError_t launch_plane(const Problem& p, float* state, cudaStream_t st) {
    F32PlaneParams prm;
    const size_t smem = plane_layout<D, KS>(p, PART, &prm);
    CUtensorMap tmK, tmQ, tmV, tmLead;
    const uint64_t nb = (uint64_t)(p.BH / p.hdiv), hd = (uint64_t)p.hdiv;
    auto tokens = [&](CUtensorMap* m, const void* base, const Layout& l, int n) {   // [d, tokens, planes per batch step, batch steps]
        const uint64_t dims[4] = {(uint64_t)D, (uint64_t)p.N, hd, nb}, token = (uint64_t)l.token;
        const uint64_t strides[3] = {token, hd > 1 ? (uint64_t)l.head : token, nb > 1 ? (uint64_t)l.batch : token};
        const uint32_t box[4] = {(uint32_t)D, (uint32_t)n, 1, 1};
        return tc::make_tensor_map_f32(m, base, 4, dims, strides, box);
    };
    const uint64_t dims[5] = {(uint64_t)D, (uint64_t)p.gridW, (uint64_t)p.gridH, hd, nb}, token = (uint64_t)p.lv.token;
    const uint64_t strides[4] = {token, token * p.gridW, hd > 1 ? (uint64_t)p.lv.head : token, nb > 1 ? (uint64_t)p.lv.batch : token};
    const uint32_t box[5] = {(uint32_t)D, (uint32_t)(p.gridW + KS - 1), (uint32_t)(prm.band_rows + KS - 1), 1, 1};
    if (!tokens(&tmK, p.k, p.lk, prm.tokens) || !tokens(&tmQ, p.q, p.lq, prm.tokens) || (p.prefix && !tokens(&tmLead, p.v, p.lv, 16)) ||
        !tc::make_tensor_map_f32(&tmV, static_cast<const float*>(p.v) + p.prefix * p.lv.token, 5, dims, strides, box))
        return cudaErrorNotSupported;
    if (!p.prefix) tmLead = tmK;   // not read
    prm.w = static_cast<const float*>(p.w); prm.bias = static_cast<const float*>(p.bias);
    prm.out = static_cast<float*>(p.out); prm.state = state; prm.lo = p.lo;
    prm.H = p.H; prm.head0 = p.head0; prm.hdiv = p.hdiv; prm.prefix = p.prefix; prm.gridH = p.gridH; prm.gridW = p.gridW;
    prm.eps2 = p.eps2; prm.status = p.status;
    static PerDevice opt_in;
    const cudaError_t e = opt_in_smem(f32_plane_kernel<D, KS, PART>, kSmemLimit, opt_in);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.BH * prm.bands)); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)prm.bands; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = PART != kRows && prm.bands > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, f32_plane_kernel<D, KS, PART>, tmK, tmQ, tmV, tmLead, prm);
}

// A few planes: the second kernel's copies and convolution run beside the first one, on other multiprocessors.  14 x 14, two kernels / one, us
// from a graph: width 32, 8 planes 6.7 / 7.7, 16 planes 6.9 / 7.8, 32 planes 9.9 / 7.9; width 64, 8 planes 10.0 / 11.1, 24 planes 13.5 / 11.3.
// A run of the one kernel is eight tokens of a row, one of the two kernels' two, so these also take grids of one column (two at width 64, up to 64
// planes): 20 planes of 64 x 1, width 64, two kernels / one 9.2 / 20.5, 148 of 128 x 1, width 32, 12.1 / 16.1.  Not where many have few tokens:
// 96 of 4 x 1, width 64, 7.5 / 6.3, 148 of 16 x 1, 5x5 filters, 12.8 / 10.3.
bool one_kernel(const Problem& p) {
    const bool thin = p.N <= 16 && p.BH >= 64 ? false : p.gridW == 1 ? p.BH <= device_sm_count() : p.gridW == 2 && p.d == 64 && p.BH < 64;
    return p.BH >= 20 && !thin;
}

template <int D, int KS> bool fits(const Problem& p) {
    F32PlaneParams prm;
    for (int part : {kWhole, kRows}) {
        if (plane_layout<D, KS>(p, part, &prm) > kSmemLimit || prm.band_rows + KS - 1 > 256) return false;   // 256: boxes of TMA copies
    }
    // A band is one grid row at least: where that is more than three rounds of runs, the patches of the other kernels are faster.
    // From a graph, they / this one, us: width 32, 8 planes of 1 x 128 8.8 / 8.2, 1 x 200 10.4 / 11.2, 1 x 250 10.4 / 12.5; width 64, 1 x 128 13.9 / 17.5.
    return one_kernel(p) || prm.band_rows * ((p.gridW + 1) / 2) <= 3 * PlaneGeo<D, KS>::kRuns;
}

template <int D, int KS>
cudaError_t launch(const Problem& p, float* state, cudaStream_t st, int* launches, KernelTimer* timer) {
    const bool whole = one_kernel(p);
    cudaError_t e = whole ? launch_plane<D, KS, kWhole>(p, state, st) : launch_plane<D, KS, kState>(p, state, st);
    if (e != cudaSuccess) return e;
    *launches = 1;
    timer->mark(st, whole ? "f32_plane" : "f32_state");
    if (whole) return e;
    e = launch_plane<D, KS, kRows>(p, state, st);
    if (e != cudaSuccess) return e;
    *launches = 2;
    timer->mark(st, "f32_apply");
    return e;
}

}  // namespace

bool f32_plane_supports(const Problem& p) {
    if (p.bf16 || (p.d != 32 && p.d != 64) || (p.ksize != 3 && p.ksize != 5) || !p.status || p.rownorm || p.phase != kPhaseAll) return false;
    if (p.N > 256 || p.gridW + p.ksize - 1 > 256) return false;   // boxes of TMA copies
    // With more planes than multiprocessors their number over those in flight decides, two per multiprocessor at width 32 and mostly one at
    // width 64.  768 planes, the kernels there were / this one, us: width 32, 5 x 5 17.1 / 21.5, 7 x 7 (3072 planes) 80.7 / 79.6, 11 x 11 54.7 / 35.5,
    // 16 x 16 65.9 / 63.3; width 64, 6 x 6 44.9 / 45.2, 8 x 8 69.6 / 53.5, 10 x 10 133 / 89, 11 x 11 89 / 95, 14 x 14 112 / 129.
    if (p.BH > device_sm_count() && (p.N < 49 || (p.d == 64 && p.N > 100))) return false;
    // From 64 planes on the CUDA cores have one kernel too.  It is faster for the smallest planes of width 32 (96 of 1 x 16 5.4 / 6.2, 4 x 4 5.5 / 6.3)
    // and for many planes of one column (1536 of 64 x 1 50.9 / 79.4, width 64 116 / 226) or two (1536 of 25 x 2 45.5 / 52.8, 40 x 2 65.8 / 69.6, but 50 x 2
    // 78.4 / 80.7, 64 x 2 101 / 88, 149 of 120 x 2 28.8 / 33.3; width 64, 400 of 30 x 2 32.7 / 39.4, 40 x 2 72 / 51).
    if (p.BH >= 64 && p.d == 32 && p.N <= 16) return false;
    if (p.gridW == 1 && p.BH > device_sm_count()) return false;
    if (p.gridW == 2 && p.BH > (p.d == 32 ? 2 : 1) * device_sm_count() && p.N <= (p.d == 32 ? 80 : 64)) return false;
    if (p.gridW == 2 && p.BH > device_sm_count() && p.d == 32 && p.N >= 240) return false;
    if (p.d == 32) return p.ksize == 3 ? fits<32, 3>(p) : fits<32, 5>(p);
    return p.ksize == 3 ? fits<64, 3>(p) : fits<64, 5>(p);
}

cudaError_t f32_plane_forward(const Problem& p, float* state, cudaStream_t st, int* launches, KernelTimer* timer) {
    if (p.d == 32) return p.ksize == 3 ? launch<32, 3>(p, state, st, launches, timer) : launch<32, 5>(p, state, st, launches, timer);
    return p.ksize == 3 ? launch<64, 3>(p, state, st, launches, timer) : launch<64, 5>(p, state, st, launches, timer);
}

}  // namespace castling
