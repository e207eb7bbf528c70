// fp32 kernels of the linear-angular attention core for head widths 32, 64 and 128 and 3x3 or 5x5 filters (the 1e-5
// tolerance rules out bf16 operands; every other fp32 shape runs on simt_kernels.cu):
//   state kernel  S += k^^T v, s += v per (plane, token split): tiles of 64 tokens (128 at D = 32), brought by TMA, the next one on its way,
//                 K scaled to unit rows in place; a thread owns 8 x 8 of S and every G-th token (G groups of
//                 (D/8)^2 threads), the groups meet in shared memory at the end
//   apply kernel  persistent CTAs walk through patches of 8 rows x TX columns of tokens: Q and V with halo come by TMA (Q and V before
//                 the state kernel has finished; the next Q during the convolution, the next V during the contraction), S' = S / pi
//                 once per plane; a thread owns a run of 8 tokens x 4 channels: the contraction over the key features, then the
//                 convolution, its window sliding along the run
// Bound: fp32 FMA issue (4 d^2 flop per token and head at 128 FMA per cycle and multiprocessor: 62 us for 2 x 8 planes of
// 128 x 128, d = 64), which needs register tiles large enough for shared memory: 64 FMAs per four 16-byte loads in the state
// kernel, 128 per twelve in the apply kernel.
// Measured: 2 x 8 planes of 128 x 128, d = 64: 133 us per forward (392 on the kernels of simt_kernels.cu, whose threads issued 28
// instructions and eight 4-byte loads for 16 FMAs and read the convolution's window from global memory), the apply kernel 72 of
// them (88 with a CTA per patch that copied it in with 16-byte asynchronous copies: issuing those took 5 000 of its 23 000
// cycles), the state kernel 58 (63 with K through registers); 2 x 4 planes of 14 x 14, d = 32: 10.3 us in a replayed graph (22.7: one CTA per plane walked through seven tiles with
// three barriers and a trip to memory each).
#include "tc_common.cuh"
#include "tc_host.cuh"

namespace castling {
namespace {

using tc::ffma2;
using tc::mbar_wait;
using tc::pdl_launch_dependents;
using tc::pdl_wait_primary;

constexpr int kThreads = 256;
constexpr int kF32ApplyParts = 4; // partial states that the apply kernel adds up itself

// ---------------------------------------------------------------------------
// state kernel: grid (BH * P); CTA bh * P + p covers tokens [p * chunk, min(N, (p + 1) * chunk))
// ---------------------------------------------------------------------------
template <int D> struct StateGeo {
    static constexpr int kTok = D == 32 ? 128 : 64;   // tokens per tile
    static constexpr int kSide = D / 8, kGroup = kSide * kSide, G = kThreads / kGroup;   // threads per group, groups
    static constexpr int kChunks = D / 4, kRowsPass = kThreads / kChunks, kPasses = kTok / kRowsPass;   // 16-byte chunks
    static constexpr int kTileBytes = kTok * D * 4;
    static constexpr int kOffBar = 4 * kTileBytes > G * D * D * 4 ? 4 * kTileBytes : G * D * D * 4;   // after K, V twice
    static constexpr size_t kSmem = 1024 + kOffBar + 32;
};

template <int D, bool RN>
__global__ void __launch_bounds__(kThreads, D == 128 ? 1 : 2)
f32_state_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, float* __restrict__ dst, int N,
                 int chunk, int P, float eps2, int hdiv, unsigned* status) {
    using G = StateGeo<D>;
    constexpr int kWords = D * D + D + (RN ? D : 0), kTok = G::kTok;
    constexpr unsigned kBit = tc::kStatusStateTimeout;
    extern __shared__ uint8_t smem_raw[];
    float* smem = reinterpret_cast<float*>(tc::align_smem(smem_raw));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + G::kOffBar / 4);   // TMA: K and V of a tile landed
    volatile int* abort_flag = reinterpret_cast<volatile int*>(full + 2);
    const int tid = threadIdx.x, p = blockIdx.x % P, bh = blockIdx.x / P;
    const int n_begin = p * chunk, n_end = min(N, n_begin + chunk);
    const int pb = bh / hdiv, ph = bh - pb * hdiv;
    // sums over tokens: thread = 16-byte chunk lc of rows lr, lr + kRowsPass, ...
    const int lc = tid % G::kChunks, lr = tid / G::kChunks;
    float4 vsum = make_float4(0.f, 0.f, 0.f, 0.f), ksum = vsum;
    auto load = [&](int n0, int buf) {   // rows beyond N arrive as zeros
        float* ks = smem + 2 * buf * (kTok * D);
        tc::mbar_expect_tx(&full[buf], 2 * G::kTileBytes);
        tc::tma_load_4d(ks, &tmK, &full[buf], 0, n0, ph, pb);
        tc::tma_load_4d(ks + kTok * D, &tmV, &full[buf], 0, n0, ph, pb);
    };
    auto scale_k = [&](int buf) {   // unit rows, in place; two or four lanes per row, neighbouring rows from different chunks on (banks)
        constexpr int L = kThreads / kTok, kPer = G::kChunks / L;
        const int row = tid / L, l = tid % L;
        float* ks = smem + 2 * buf * (kTok * D) + row * D;
        float4 x[kPer];
        float ss = 0.f;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            x[i] = *reinterpret_cast<const float4*>(ks + (l + L * ((i + row) % kPer)) * 4);
            ss = fmaf(x[i].x, x[i].x, fmaf(x[i].y, x[i].y, fmaf(x[i].z, x[i].z, fmaf(x[i].w, x[i].w, ss))));
        }
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const float rk = inv_sqrt(fmaxf(ss, eps2));
#pragma unroll
        for (int i = 0; i < kPer; ++i)
            *reinterpret_cast<float4*>(ks + (l + L * ((i + row) % kPer)) * 4) = make_float4(x[i].x * rk, x[i].y * rk, x[i].z * rk, x[i].w * rk);
    };
    // computing: group g takes tokens g, g + G, ...; a thread owns rows 8 ti .. and columns {4 tj .., D/2 + 4 tj ..} of S
    const int g = tid / G::kGroup, t = tid % G::kGroup, ti = t / G::kSide, tj = t % G::kSide;
    // where a warp holds two groups (D = 32), whose rows lie in the same banks, the odd one takes its halves in reverse order
    const bool flip = G::kGroup < 32 && (g & 1);
    const int row_a = ti * 8 + (flip ? 4 : 0), row_b = ti * 8 + (flip ? 0 : 4);
    const int col_a = tj * 4 + (flip ? D / 2 : 0), col_b = tj * 4 + (flip ? 0 : D / 2);
    float2 acc[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = make_float2(0.f, 0.f);

    if (tid == 0) {
        tc::mbar_init(&full[0], 1); tc::mbar_init(&full[1], 1);
        *abort_flag = 0;
        tc::mbar_fence_init();
    }
    pdl_wait_primary();
    pdl_launch_dependents();
    if (tid == 0) load(n_begin, 0);
    __syncthreads();   // the barriers are set up
    int buf = 0;
    uint32_t phase = 0;
    for (int n0 = n_begin; n0 < n_end; n0 += kTok, phase ^= buf, buf ^= 1) {
        const bool ok = mbar_wait(&full[buf], phase, abort_flag, status, kBit);
        scale_k(buf);
        tc::fence_proxy_async_smem();       // TMA writes this buffer after the next tile's barrier
        if (__syncthreads_or(!ok)) break;   // this tile is ready; every thread has left the previous one
        if (tid == 0 && n0 + kTok < n_end) load(n0 + kTok, buf ^ 1);
        const float* ks = smem + 2 * buf * (kTok * D);
        const float* vs = ks + kTok * D;
#pragma unroll 2
        for (int n = g; n < kTok; n += G::G) {
            const float4 a0 = *reinterpret_cast<const float4*>(ks + n * D + row_a);
            const float4 a1 = *reinterpret_cast<const float4*>(ks + n * D + row_b);
            const float4 b0 = *reinterpret_cast<const float4*>(vs + n * D + col_a);
            const float4 b1 = *reinterpret_cast<const float4*>(vs + n * D + col_b);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float2 b[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
            for (int x = 0; x < 8; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = ffma2(make_float2(a[x], a[x]), b[y], acc[x][y]);
        }
#pragma unroll
        for (int r = 0; r < G::kPasses; ++r) {
            const float4 x = *reinterpret_cast<const float4*>(vs + (lr + r * G::kRowsPass) * D + lc * 4);
            vsum.x += x.x; vsum.y += x.y; vsum.z += x.z; vsum.w += x.w;
            if (RN) {
                const float4 z = *reinterpret_cast<const float4*>(ks + (lr + r * G::kRowsPass) * D + lc * 4);
                ksum.x += z.x; ksum.y += z.y; ksum.z += z.z; ksum.w += z.w;
            }
        }
    }
    if (tid == 0 && *abort_flag) {   // giving up: let the copies in flight land before their place is used
        for (int spin = 0; spin < (1 << 20) && !tc::mbar_try_wait(&full[buf], phase); ++spin) {}
    }
    float* out = dst + ((size_t)bh * P + p) * kWords;
    // groups meet in shared memory, in their order
    __syncthreads();
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        float* row = smem + (g * D + (x < 4 ? row_a + x : row_b + x - 4)) * D;
        *reinterpret_cast<float4*>(row + col_a) = make_float4(acc[x][0].x, acc[x][0].y, acc[x][1].x, acc[x][1].y);
        *reinterpret_cast<float4*>(row + col_b) = make_float4(acc[x][2].x, acc[x][2].y, acc[x][3].x, acc[x][3].y);
    }
    __syncthreads();
    for (int i = tid * 4; i < D * D; i += kThreads * 4) {
        float4 s = *reinterpret_cast<const float4*>(smem + i);
#pragma unroll
        for (int h = 1; h < G::G; ++h) {
            const float4 x = *reinterpret_cast<const float4*>(smem + h * D * D + i);
            s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
        }
        *reinterpret_cast<float4*>(out + i) = s;
    }
    __syncthreads();
    *reinterpret_cast<float4*>(smem + lr * D + lc * 4) = vsum;
    if (RN) *reinterpret_cast<float4*>(smem + (G::kRowsPass + lr) * D + lc * 4) = ksum;
    __syncthreads();
    if (tid < (RN ? 2 * D : D)) {
        const float* src = smem + (tid / D) * G::kRowsPass * D + tid % D;
        float s = 0.f;
#pragma unroll
        for (int r = 0; r < G::kRowsPass; ++r) s += src[r * D];
        out[D * D + tid] = s;
    }
}

// Sums P partial states per plane in index order; grid (BH, words / 256 rounded up).
__global__ void __launch_bounds__(kThreads)
f32_reduce_kernel(const float* __restrict__ partial, float* __restrict__ state, int words, int P) {
    pdl_wait_primary();
    pdl_launch_dependents();
    const int i = blockIdx.y * kThreads + threadIdx.x;
    if (i >= words) return;
    const float* src = partial + (size_t)blockIdx.x * P * words + i;
    float s = 0.f;
#pragma unroll 8
    for (int p = 0; p < P; ++p) s += __ldcg(src + (size_t)p * words);
    state[(size_t)blockIdx.x * words + i] = s;
}

// ---------------------------------------------------------------------------
// apply kernel: grid (BH * patches of a plane)
// ---------------------------------------------------------------------------
template <int D, int KS> struct ApplyGeo {
    static constexpr int kCG = D / 4;                     // channel groups of four
    static constexpr int kRuns = kThreads / kCG;          // runs of eight tokens
    static constexpr int TX = kRuns, TY = 8;              // patch: 8 rows x TX columns (TX / 8 runs per row)
    static constexpr int R = KS / 2, HX = TX + 2 * R, HY = TY + 2 * R;
    static constexpr int kTokens = TX * TY;
    // S' | 1/2 s | bias | sum k^ | filters (tap-major) | 1/||q|| | 1 / row sum | Q | V | barriers; TMA wants 128-byte boundaries
    static constexpr int kOffC = D * D, kOffB = kOffC + D, kOffZ = kOffB + D, kOffW = kOffZ + D, kOffRq = kOffW + KS * KS * D;
    static constexpr int kOffDen = kOffRq + kTokens, kOffQ = (kOffDen + kTokens + 31) / 32 * 32, kOffV = kOffQ + kTokens * D;
    static constexpr int kOffBar = kOffV + HX * HY * D;
    static constexpr size_t kSmem = 1024 + sizeof(float) * kOffBar + 32;
    static constexpr int kCtas = D < 128 && 2 * (kSmem + 1024) <= 228 * 1024 ? 2 : 1;   // per multiprocessor
    static_assert(kSmem <= 227 * 1024, "shared memory");
};

struct F32ApplyParams {
    const float *q, *w, *bias, *state;
    float* out;
    Layout lq, lo;
    int H, head0, hdiv, prefix, gridH, gridW, tilesX, patches;   // patches per plane: tiles, then one of leading tokens
    int total;             // patches of all planes
    int P;                 // partial states per plane to be summed here (1: the state is final)
    float eps2;
    int v_row0;            // row v_row0 of V is grid row 0
    unsigned* status;      // device status word
};

template <int D, int KS, bool RN>
__global__ void __launch_bounds__(kThreads, (ApplyGeo<D, KS>::kCtas))
f32_apply_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmV, const F32ApplyParams prm) {
    using G = ApplyGeo<D, KS>;
    constexpr int kWords = D * D + D + (RN ? D : 0);
    constexpr unsigned kBit = tc::kStatusApplyTimeout;
    extern __shared__ uint8_t smem_raw[];
    float* smem = reinterpret_cast<float*>(tc::align_smem(smem_raw));
    float* S_sm = smem;
    float* q_s = smem + G::kOffQ;
    float* v_s = smem + G::kOffV;
    uint64_t* q_full = reinterpret_cast<uint64_t*>(smem + G::kOffBar);   // TMA: Q of the patch landed
    uint64_t* v_full = q_full + 1;                                       // TMA: V of the patch landed
    volatile int* abort_flag = reinterpret_cast<volatile int*>(q_full + 2);
    const int tid = threadIdx.x, W = prm.gridW;
    // this CTA's run of patches, counted through all planes
    const int i_begin = (int)((long long)prm.total * blockIdx.x / gridDim.x), i_end = (int)((long long)prm.total * (blockIdx.x + 1) / gridDim.x);
    struct Patch { int bh, x0, y0; bool lead; };   // lead: the leading tokens of a plane, without grid position or convolution
    auto patch_at = [&](int i) {
        Patch t;
        t.bh = i / prm.patches;
        const int k = i - t.bh * prm.patches, py = k / prm.tilesX;
        t.lead = prm.prefix > 0 && k == prm.patches - 1;
        t.y0 = py * G::TY; t.x0 = (k - py * prm.tilesX) * G::TX;
        return t;
    };
    // one thread loads; rows and columns beyond the grid arrive as zeros
    auto load_q = [&](int i) {
        if (i >= i_end) return;
        const Patch t = patch_at(i);
        if (t.lead) return;   // copied by all threads when its turn has come
        const int pb = t.bh / prm.hdiv, ph = t.bh - pb * prm.hdiv;
        tc::mbar_expect_tx(q_full, G::kTokens * D * 4);
        tc::tma_load_5d(q_s, &tmQ, q_full, 0, t.x0, t.y0, ph, pb);
    };
    auto load_v = [&](int i) {
        if (i >= i_end) return;
        const Patch t = patch_at(i);
        if (t.lead) return;
        const int pb = t.bh / prm.hdiv, ph = t.bh - pb * prm.hdiv;
        tc::mbar_expect_tx(v_full, G::HX * G::HY * D * 4);
        tc::tma_load_5d(v_s, &tmV, v_full, 0, t.x0 - G::R, t.y0 - G::R + prm.v_row0, ph, pb);
    };
    if (tid == 0) {
        tc::mbar_init(q_full, 1); tc::mbar_init(v_full, 1);
        *abort_flag = 0;
        tc::mbar_fence_init();
        load_q(i_begin);   // Q, V and the filters were there before the state kernel started
        load_v(i_begin);
    }
    const int cg = tid % G::kCG, run = tid / G::kCG;   // this thread's channels 4 cg .. and run of tokens
    int plane = -1;
    uint32_t phase = 0;   // of both barriers: patches on the grid so far, modulo 2
    for (int it = i_begin; it < i_end; ++it) {
        const Patch cur = patch_at(it);
        const bool lead = cur.lead;
        const int bh = cur.bh;
        if (bh != plane) {   // every thread has left the previous plane: the barrier after its last convolution
            const int h = (prm.head0 + bh) % prm.H;
            for (int i = tid; i < KS * KS * D; i += kThreads)
                smem[G::kOffW + i] = __ldg(prm.w + ((size_t)(h * D + i % D)) * (KS * KS) + i / D);
            if (tid < D) smem[G::kOffB + tid] = prm.bias ? __ldg(prm.bias + h * D + tid) : 0.f;
            if (plane < 0) {
                pdl_wait_primary();
                pdl_launch_dependents();
            }
            plane = bh;
            const float* st = prm.state + (size_t)bh * prm.P * kWords;
            auto total = [&](int i, float f) {
                float4 s = __ldcg(reinterpret_cast<const float4*>(st + i));
                for (int p = 1; p < prm.P; ++p) {
                    const float4 x = __ldcg(reinterpret_cast<const float4*>(st + (size_t)p * kWords + i));
                    s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
                }
                return make_float4(s.x * f, s.y * f, s.z * f, s.w * f);
            };
            for (int i = tid * 4; i < kWords; i += kThreads * 4) {   // S / pi, 1/2 s, sum k^
                float* dst = smem + (i < D * D + D ? i : G::kOffZ + i - D * D - D);
                *reinterpret_cast<float4*>(dst) = total(i, i < D * D ? kInvPi : i < D * D + D ? 0.5f : 1.0f);
            }
        }
        if (lead) {
            const float* qp = prm.q + plane_offset(prm.lq, bh, prm.hdiv);
            for (int c = tid; c < prm.prefix * G::kCG; c += kThreads)
                *reinterpret_cast<float4*>(q_s + c * 4) = __ldg(reinterpret_cast<const float4*>(qp + (c / G::kCG) * prm.lq.token + (c % G::kCG) * 4));
        }
        __syncthreads();
        bool ok = lead || mbar_wait(q_full, phase, abort_flag, prm.status, kBit);
        {   // 1 / max(||q||, eps) of every token, one to four threads each; they walk a row from different chunks on, which lie in
            // different banks
            constexpr int L = kThreads / G::kTokens;
            const int r = tid / L, l = tid % L;
            float ss = 0.f, dot = 0.f;
#pragma unroll 4
            for (int c = 0; c < D / 4; c += L) {
                const int i = ((c + L * r + l) % (D / 4)) * 4;
                const float4 x = *reinterpret_cast<const float4*>(q_s + r * D + i);
                ss = fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, fmaf(x.w, x.w, ss))));
                if (RN) {
                    const float4 z = *reinterpret_cast<const float4*>(smem + G::kOffZ + i);
                    dot = fmaf(x.x, z.x, fmaf(x.y, z.y, fmaf(x.z, z.z, fmaf(x.w, z.w, dot))));
                }
            }
#pragma unroll
            for (int o = L / 2; o > 0; o >>= 1) {
                ss += __shfl_xor_sync(0xffffffffu, ss, o);
                if (RN) dot += __shfl_xor_sync(0xffffffffu, dot, o);
            }
            if (l == 0) {
                const float rq = inv_sqrt(fmaxf(ss, prm.eps2));
                smem[G::kOffRq + r] = rq;
                // Eq. 3's denominator for the kept kernel of Eq. 8: N/2 + q^ . (sum_j k^_j) / pi
                if (RN) smem[G::kOffDen + r] = 1.0f / fmaf(dot * rq, kInvPi, 0.5f * (float)(prm.prefix + prm.gridH * W));
            }
        }
        float2 acc[8][2];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j][0] = acc[j][1] = make_float2(0.f, 0.f);
        const float* q_run = q_s + run * 8 * D;
#pragma unroll 2
        for (int i = 0; i < D; i += 4) {
            float4 a[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) a[j] = *reinterpret_cast<const float4*>(q_run + j * D + i);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4 s = *reinterpret_cast<const float4*>(S_sm + (i + u) * D + cg * 4);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float x = u == 0 ? a[j].x : u == 1 ? a[j].y : u == 2 ? a[j].z : a[j].w;
                    acc[j][0] = ffma2(make_float2(x, x), make_float2(s.x, s.y), acc[j][0]);
                    acc[j][1] = ffma2(make_float2(x, x), make_float2(s.z, s.w), acc[j][1]);
                }
            }
        }
        ok = ok && (lead || mbar_wait(v_full, phase, abort_flag, prm.status, kBit));
        tc::fence_proxy_async_smem();          // a leading patch wrote Q, which TMA writes next
        if (__syncthreads_or(!ok)) break;      // the factors of every token are there, Q is dead
        if (tid == 0) load_q(it + 1);
        const float4 cs = *reinterpret_cast<const float4*>(smem + G::kOffC + cg * 4);
        float4 bs = *reinterpret_cast<const float4*>(smem + G::kOffB + cg * 4);
        if (lead) bs = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float rq = smem[G::kOffRq + run * 8 + j], inv = RN ? smem[G::kOffDen + run * 8 + j] : 1.0f;
            if (RN) {
                acc[j][0].x = fmaf(fmaf(acc[j][0].x, rq, cs.x), inv, bs.x); acc[j][0].y = fmaf(fmaf(acc[j][0].y, rq, cs.y), inv, bs.y);
                acc[j][1].x = fmaf(fmaf(acc[j][1].x, rq, cs.z), inv, bs.z); acc[j][1].y = fmaf(fmaf(acc[j][1].y, rq, cs.w), inv, bs.w);
            } else {
                acc[j][0].x = fmaf(acc[j][0].x, rq, cs.x + bs.x); acc[j][0].y = fmaf(acc[j][0].y, rq, cs.y + bs.y);
                acc[j][1].x = fmaf(acc[j][1].x, rq, cs.z + bs.z); acc[j][1].y = fmaf(acc[j][1].y, rq, cs.w + bs.w);
            }
        }
        if (!lead) {
            const float* vw = v_s + ((run / (G::TX / 8)) * G::HX + (run % (G::TX / 8)) * 8) * D + cg * 4;   // halo row 0, column 0
#pragma unroll 1
            for (int dy = 0; dy < KS; ++dy) {
                float4 f[KS];
#pragma unroll
                for (int dx = 0; dx < KS; ++dx) f[dx] = *reinterpret_cast<const float4*>(smem + G::kOffW + (dy * KS + dx) * D + cg * 4);
#pragma unroll
                for (int c = 0; c < 8 + KS - 1; ++c) {
                    const float4 x = *reinterpret_cast<const float4*>(vw + (dy * G::HX + c) * D);
#pragma unroll
                    for (int dx = 0; dx < KS; ++dx) {
                        const int j = c - dx;   // compile-time after unrolling
                        if (j < 0 || j >= 8) continue;
                        acc[j][0] = ffma2(make_float2(f[dx].x, f[dx].y), make_float2(x.x, x.y), acc[j][0]);
                        acc[j][1] = ffma2(make_float2(f[dx].z, f[dx].w), make_float2(x.z, x.w), acc[j][1]);
                    }
                }
            }
            phase ^= 1;
        }
        __syncthreads();   // V and the factors are dead
        if (tid == 0) load_v(it + 1);
        // tokens of the run: neighbours in memory
        const int y = cur.y0 + run / (G::TX / 8), x = cur.x0 + (run % (G::TX / 8)) * 8;
        const int n0 = lead ? run * 8 : prm.prefix + y * W + x, n_run = lead ? prm.prefix - n0 : y < prm.gridH ? W - x : 0;
        float* op = prm.out + plane_offset(prm.lo, bh, prm.hdiv) + n0 * prm.lo.token + cg * 4;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j < n_run) *reinterpret_cast<float4*>(op + j * prm.lo.token) = make_float4(acc[j][0].x, acc[j][0].y, acc[j][1].x, acc[j][1].y);
    }
    if (tid == 0 && *abort_flag) {   // giving up: let the copies in flight land before shared memory goes away
        for (int spin = 0; spin < (1 << 20) && !tc::mbar_try_wait(q_full, phase); ++spin) {}
        for (int spin = 0; spin < (1 << 20) && !tc::mbar_try_wait(v_full, phase); ++spin) {}
    }
}

template <typename Kernel, typename... Args>
cudaError_t launch_pdl(Kernel kernel, dim3 grid, size_t smem, cudaStream_t st, bool early, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = early;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int D, int KS, bool RN>
cudaError_t launch_f32(const Problem& p, float* ws_state, float* ws_partial, int P, cudaStream_t st, int* launches, KernelTimer* timer) {
    constexpr int kWords = D * D + D + (RN ? D : 0);
    using A = ApplyGeo<D, KS>;
    CUtensorMap tmQ, tmV;
    const int v_rows = p.v_rows > 0 ? p.v_rows : p.gridH;
    const uint64_t nb = (uint64_t)(p.BH / p.hdiv), hd = (uint64_t)p.hdiv;
    if (p.phase != kPhaseStateOnly) {
        // [d, columns, rows, planes per batch step, batch steps]: out-of-range coordinates read as zero
        auto map = [&](CUtensorMap* m, const void* base, const Layout& l, int rows, int bx, int by) {
            const uint64_t dims[5] = {(uint64_t)D, (uint64_t)p.gridW, (uint64_t)rows, hd, nb}, token = (uint64_t)l.token;
            const uint64_t strides[4] = {token, token * p.gridW, hd > 1 ? (uint64_t)l.head : token, nb > 1 ? (uint64_t)l.batch : token};
            const uint32_t box[5] = {(uint32_t)D, (uint32_t)bx, (uint32_t)by, 1, 1};
            return tc::make_tensor_map_f32(m, static_cast<const float*>(base) + p.prefix * l.token, 5, dims, strides, box);
        };
        if (!map(&tmQ, p.q, p.lq, p.gridH, A::TX, A::TY) || !map(&tmV, p.v, p.lv, v_rows, A::HX, A::HY)) return cudaErrorNotSupported;
    }
    const float* state = ws_state;
    int apply_parts = 1;
    cudaError_t e;
    if (p.phase != kPhaseApplyOnly) {
        using G = StateGeo<D>;
        const int tiles = (p.N + G::kTok - 1) / G::kTok, per = (tiles + P - 1) / P;
        P = (tiles + per - 1) / per;   // every split has tokens
        CUtensorMap tmK, tmV;   // [d, tokens, planes per batch step, batch steps]
        auto map = [&](CUtensorMap* m, const void* base, const Layout& l) {
            const uint64_t dims[4] = {(uint64_t)D, (uint64_t)p.N, hd, nb}, token = (uint64_t)l.token;
            const uint64_t strides[3] = {token, hd > 1 ? (uint64_t)l.head : token, nb > 1 ? (uint64_t)l.batch : token};
            const uint32_t box[4] = {(uint32_t)D, (uint32_t)G::kTok, 1, 1};
            return tc::make_tensor_map_f32(m, base, 4, dims, strides, box);
        };
        if (!map(&tmK, p.k, p.lk) || !map(&tmV, p.v, p.lv)) return cudaErrorNotSupported;
        static PerDevice opt_in;
        e = opt_in_smem(f32_state_kernel<D, RN>, G::kSmem, opt_in);
        if (e != cudaSuccess) return e;
        e = launch_pdl(f32_state_kernel<D, RN>, dim3((unsigned)(p.BH * P)), G::kSmem, st, true, tmK, tmV,
                       P > 1 ? ws_partial : ws_state, p.N, per * G::kTok, P, p.eps2, p.hdiv, p.status);
        if (e != cudaSuccess) return e;
        ++*launches;
        timer->mark(st, "f32_state");
        if (P > kF32ApplyParts || (P > 1 && p.phase == kPhaseStateOnly)) {
            e = launch_pdl(f32_reduce_kernel, dim3((unsigned)p.BH, (kWords + kThreads - 1) / kThreads), 0, st, true, ws_partial, ws_state, kWords, P);
            if (e != cudaSuccess) return e;
            ++*launches;
            timer->mark(st, "f32_reduce");
        } else if (P > 1) {
            state = ws_partial;   // few parts: the apply kernel adds them as it reads them
            apply_parts = P;
        }
        if (p.phase == kPhaseStateOnly) return cudaSuccess;
    }
    F32ApplyParams prm;
    prm.q = static_cast<const float*>(p.q);
    prm.w = static_cast<const float*>(p.w); prm.bias = static_cast<const float*>(p.bias);
    prm.state = state; prm.out = static_cast<float*>(p.out);
    prm.lq = p.lq; prm.lo = p.lo;
    prm.H = p.H; prm.head0 = p.head0; prm.hdiv = p.hdiv; prm.prefix = p.prefix; prm.gridH = p.gridH; prm.gridW = p.gridW;
    prm.tilesX = (p.gridW + A::TX - 1) / A::TX;
    prm.patches = prm.tilesX * ((p.gridH + A::TY - 1) / A::TY) + (p.prefix > 0 ? 1 : 0);
    prm.total = p.BH * prm.patches;
    prm.P = apply_parts; prm.eps2 = p.eps2;
    prm.v_row0 = p.v_row0; prm.status = p.status;
    const int resident = A::kCtas * device_sm_count();
    static PerDevice opt_in;
    e = opt_in_smem(f32_apply_kernel<D, KS, RN>, A::kSmem, opt_in);
    if (e != cudaSuccess) return e;
    // An apply pass on its own waits for whatever is before it in the stream, which may be writing Q and V; after the state
    // kernel they are there.
    e = launch_pdl(f32_apply_kernel<D, KS, RN>, dim3((unsigned)(prm.total < resident ? prm.total : resident)), A::kSmem, st,
                   p.phase != kPhaseApplyOnly, tmQ, tmV, prm);
    if (e != cudaSuccess) return e;
    ++*launches;
    timer->mark(st, "f32_apply");
    return cudaSuccess;
}

template <int D>
cudaError_t launch_f32_d(const Problem& p, float* s, float* part, int P, cudaStream_t st, int* n, KernelTimer* t) {
    if (p.ksize == 3) return p.rownorm ? launch_f32<D, 3, true>(p, s, part, P, st, n, t) : launch_f32<D, 3, false>(p, s, part, P, st, n, t);
    return p.rownorm ? launch_f32<D, 5, true>(p, s, part, P, st, n, t) : launch_f32<D, 5, false>(p, s, part, P, st, n, t);
}

}  // namespace

bool f32_supports(const Problem& p) { return !p.bf16 && f32_width(p.d) && (p.ksize == 3 || p.ksize == 5) && p.status; }

// The apply kernel takes a patch of 8 rows x TX columns whole, the one of simt_kernels.cu 64 tokens whatever their grid.  Where the
// patches hold much more than the grid, and there are more of them than run at a time, the latter is the faster one.  Whole
// forwards of 2 x 8 planes, this kernel / that one, us: 1 x 16384, d = 64 552 / 218, 2 x 8192 310 / 247, 4096 x 4 309 / 269 (patches four
// times the grid), 4096 x 4, d = 32 200 / 130 (eight times); apply kernels alone on this side of the line: 3 x 5461, d = 64 177 / 197 (2.7
// times), 2048 x 8, d = 32 96 / 102 (four times), 5 x 5 filters 119 / 171.
bool f32_thin(const Problem& p) {
    const long long tx = 4 * kThreads / p.d;   // ApplyGeo's TX
    const long long patches = ((p.gridW + tx - 1) / tx) * ((p.gridH + 7) / 8), places = patches * tx * 8, tokens = (long long)p.gridH * p.gridW;
    return p.BH * patches > 2 * device_sm_count() && (p.d == 32 ? places > 4 * tokens : 2 * places > 7 * tokens);
}

// Token splits of the state kernel: two CTAs per multiprocessor, at least 128 tokens each (the states of smaller grids need
// no workspace beyond the final one).  Up to kF32ApplyParts of them need no reduction in between.
int f32_choose_splits(int BH, int N) {
    int P = 2 * device_sm_count() / BH;
    if (P > N / 128) P = N / 128;
    if (P > 64) P = 64;
    return P < 1 ? 1 : P;
}

cudaError_t f32_forward(const Problem& p, float* ws_state, float* ws_partial, int P, cudaStream_t stream, int* launches,
                        KernelTimer* timer) {
    *launches = 0;
    if (p.d == 32) return launch_f32_d<32>(p, ws_state, ws_partial, P, stream, launches, timer);
    if (p.d == 64) return launch_f32_d<64>(p, ws_state, ws_partial, P, stream, launches, timer);
    return launch_f32_d<128>(p, ws_state, ws_partial, P, stream, launches, timer);
}

}  // namespace castling
