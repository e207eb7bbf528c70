// Whole forward pass in one kernel for short sequences (bf16; head width 64, at most 256 tokens per (b,h), or head width 32,
// at most 512):
//     out_t = (1/pi) q^_t (K^^T V) + 1/2 sum_n v_n + bias + DWConv(V)_t                    (Eq. 9)
// A plane (one (b,h)) fits in shared memory, so K, V and Q come from memory once, the state never
// leaves the SM and the forward is a single launch without workspace.  Several CTAs share an SM; each
// walks over planes blockIdx.x, blockIdx.x + gridDim.x, ...  Per plane
//   warp 0      TMA: K, V and Q as 128-token tiles (128-byte rows and swizzle, 64 bytes for width 32; rows beyond N are
//               zero-filled); once the state UMMAs have retired, V again without swizzle into
//               the K buffer (an L2 hit), which is what the convolution reads: the token grid with its halo, zero-filled outside (ROOMY),
//               or where that does not fit the tokens as they are, and words outside the grid are masked
//   workers     thread = 128-byte line (one token, or two of width 32): scale K rows by 1 / max(||k||, eps) in place;
//               1 / max(||q||, eps)
//   warp 1      one elected lane issues the state UMMAs, A = [K^ ; 1 0 0 ...] (M-major, the ones row makes
//               accumulator row 64 (32) the token sum of V), B = V (N-major): S and s land in TMEM
//   workers     read S and s from TMEM, write S' = S / pi as the bf16 B operand of the second
//               contraction and s as fp32
//   warp 1      apply UMMAs: acc[tile] = Q[tile] * S' into TMEM (the state's columns are reused)
//   workers     thread = token: accumulator rows from TMEM, times 1 / max(||q||, eps), to shared memory as fp32 (over the swizzled
//               V tiles and the Q tiles, both dead by then); then lane = channel pair (width 32: and column parity), warp = a
//               strip of two columns (four): depthwise convolution sliding down the strip with the filters in registers, the sums
//               of an output row starting from its accumulator + 1/2 s + bias, one rounding to bf16, rows stored
//               straight to memory; leading off-grid tokens get the attention terms only
// FINE (width 32 only): the unit keys and S' are two bf16 each, the value and what rounding it left off, contracted one after the
// other: as precise as fp32 operands.  The rest of K lies in the Q buffer, so Q comes with the second copy of V, once the state
// UMMAs have retired; the rest of S' lies in the V buffer, which is dead by then.  512 planes of 7 x 7: 11.7 us a call, 10.3
// with single operands.
//
// A plane is a serial chain of about 10 500 cycles (14 x 14 tokens, width 64, 4 600 of them the convolution), so the time of
// a call is the number of planes over those in flight.  Two shapes of CTA: 256 workers for planes of any size, two per SM;
// 128 workers for planes of at most 128 lines, three or four per SM, which finish a plane later but more of them at a time:
// taken when that saves a round of planes.
// Measured (from a graph, early launch included): 768 planes of 14 x 14 and a class token 28.7 us, 31.3 with every word of V masked, accumulators scaled one by one in the
// convolution, branches around its loads and stores and each tap's sum waiting for the last (12 300 cycles a plane); 12 planes 6.7 / 8.0; 256 planes
// of width 32 7.2 / 8.7; 512 planes of 7 x 7, width 32, 14.1 us a call with two tokens a line and large CTAs.
#include "tc_common.cuh"
#include "tc_host.cuh"

namespace castling {
namespace tc {
namespace {

constexpr int kTile = 128;                       // tokens per UMMA tile

// NARROW: width-32 heads in 64-byte rows, two tokens to a line.  WORKERS: worker threads, and lines a plane may have.
template <int KS, bool NARROW, int WORKERS, bool ROOMY = false> struct Geo {
    static constexpr int kW = NARROW ? 32 : 64;                  // head width
    static constexpr int kRow = kW * 2;                          // bytes of a token
    static constexpr int kTokens = WORKERS * (NARROW ? 2 : 1);   // tokens a plane may have
    static constexpr int kThreads = 64 + WORKERS;
    static constexpr int kCtas = KS != 3 ? (WORKERS == 256 ? 1 : 2) : WORKERS == 256 ? 2 : NARROW ? 4 : 3;   // per multiprocessor
    static constexpr int kTmemCols = kTokens / kTile * kW;       // outputs; the state uses the first kW columns before
    // Shared memory: S' | K | V | Q | ones | rq | s | barriers | filters.  After their first use the buffers change role: K holds
    // the unswizzled V plane, V and Q hold the fp32 accumulator rows.  The convolution's reads left of the plane's first token
    // fall into S'.
    static constexpr int kBuf = WORKERS * 128;
    // Bytes of an accumulator row.  ROOMY: the plane with its halo fits the K buffer, and its accumulator rows with 16 bytes of padding V's and Q's.
    static constexpr int kAccRow = kW * 4 + (ROOMY ? 16 : 0);
    static constexpr int kOffS = 0, kOffK = kW * kRow, kOffV = kOffK + kBuf, kOffQ = kOffV + kBuf;
    static_assert(kOffK % 1024 == 0 && kOffK >= KS / 2 * kRow, "swizzle atoms; room for the reads left of the plane");
    static constexpr int kOffOnes = kOffQ + kBuf;                // constant block of the A operand (after K: positive offset)
    static constexpr int kOffRq = kOffOnes + 16 * kRow;          // [kTokens] 1 / max(||q||, eps)
    static constexpr int kOffSum = kOffRq + kTokens * 4;         // [kW] token sum of V
    static constexpr int kOffBar = kOffSum + kW * 4;
    static constexpr int kOffW = kOffBar + 128;                  // filters of the plane's head, [taps][kW] fp32, and its bias
    static constexpr size_t kSmem = 1024 + kOffW + (KS * KS + 1) * kW * 4;
};

struct FusedParams {
    const __nv_bfloat16* w;     // [H*d][KS][KS]
    const __nv_bfloat16* bias;  // [H*d] or nullptr
    __nv_bfloat16* out;         // token n of plane i at plane_offset(lo, i, hdiv) + n * lo.token
    Layout lo;
    int H, head0, BH, hdiv, prefix, N, gridH, gridW;  // N = prefix + gridH * gridW
    bool turned;                // filters with rows and columns exchanged
    float eps2;
    unsigned* status;
};

// OUT_PACKED: the output's token rows are contiguous, which keeps the row addresses of the
// store loop compile-time offsets.
template <int KS, bool OUT_PACKED, bool NARROW, int WORKERS, bool FINE, bool ROOMY>
__global__ void __launch_bounds__((Geo<KS, NARROW, WORKERS>::kThreads), (Geo<KS, NARROW, WORKERS>::kCtas))
tc_fused_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmVplain,
                const FusedParams prm) {
    using G = Geo<KS, NARROW, WORKERS, ROOMY>;
    constexpr int R = KS / 2, kW = G::kW, kRow = G::kRow, kTileBytes = kTile * kRow, kWarps = WORKERS / 32, kHalves = WORKERS / 128;
    constexpr uint32_t kHigh = NARROW ? kDescHigh64 : kDescHigh;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_smem(smem_raw);
    uint8_t* K_s = smem + G::kOffK;
    uint8_t* V_s = smem + G::kOffV;
    uint8_t* Q_s = smem + G::kOffQ;
    uint8_t* S_s = smem + G::kOffS;
    uint8_t* ones = smem + G::kOffOnes;
    float* rq_s = reinterpret_cast<float*>(smem + G::kOffRq);
    float* sum_s = reinterpret_cast<float*>(smem + G::kOffSum);
    float* w_s = reinterpret_cast<float*>(smem + G::kOffW);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + G::kOffBar);
    uint64_t* k_full = bars + 0;      // TMA: K landed
    uint64_t* v_full = bars + 1;      // TMA: V (swizzled) landed
    uint64_t* q_full = bars + 2;      // TMA: Q landed
    uint64_t* vp_full = bars + 3;     // TMA: V (plain) landed in the K buffer
    uint64_t* k_scaled = bars + 4;    // K rows normalised (WORKERS)
    uint64_t* s_done = bars + 5;      // state UMMAs retired: S readable, K and V tiles no longer read
    uint64_t* sp_ready = bars + 6;    // S' and s written, state columns of TMEM read out (WORKERS)
    uint64_t* o_done = bars + 7;      // apply UMMAs retired: accumulators readable, Q tile no longer read
    uint64_t* tm_free = bars + 8;     // output accumulators read out of TMEM (WORKERS)
    uint64_t* plane_free = bars + 9;  // every buffer of the plane is free again (WORKERS)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 10);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int W = prm.gridW, N = prm.N;
    const int tiles = (N + kTile - 1) / kTile;
    const int n_planes = (prm.BH - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    constexpr unsigned kBit = kStatusFusedTimeout;

    if (tid == 0) {
        mbar_init(k_full, 1); mbar_init(v_full, 1); mbar_init(q_full, 1); mbar_init(vp_full, 1);
        mbar_init(k_scaled, WORKERS); mbar_init(s_done, 1); mbar_init(sp_ready, WORKERS);
        mbar_init(o_done, 1); mbar_init(tm_free, WORKERS); mbar_init(plane_free, WORKERS);
        *abort_flag = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmVplain);
    }
    if (warp == 1) tmem_alloc(tmem_slot, G::kTmemCols);
    if (warp >= 2 && tid - 64 < kRow) {
        // constant block of A: for each of 16 token rows, element kW (first of the second block along M) is 1.0 and the rest
        // 0; 16-byte chunk c of row r sits at chunk c ^ (r & 7), in rows of 64 bytes at c ^ ((r >> 1) & 3)
        const int t = tid - 64, r = t / (kRow / 16), c = t % (kRow / 16);
        uint4 val = make_uint4(0, 0, 0, 0);
        if ((c ^ (NARROW ? (r >> 1) & 3 : r & 7)) == 0) val.x = 0x3f80u;
        *reinterpret_cast<uint4*>(ones + t * 16) = val;
        fence_proxy_async_smem();
    }
    tcgen05_fence_before_sync();
    __syncthreads();
    tcgen05_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    // Launched programmatically dependent on whatever precedes it in the stream: all of the above ran while that kernel drained.  Every
    // thread waits for it here, also those that touch no memory: the limits of their waits are for this kernel's own work.  The next
    // forward may set itself up in the same way.
    pdl_launch_dependents();
    pdl_wait_primary();

    if (warp == 0) {
        if (lane == 0) {
            const uint64_t pol = l2_policy_evict_first();  // K and Q are read once
            int issued = 0, issued_vp = 0;
            for (int it = 0; it < n_planes; ++it) {
                const int bh = blockIdx.x + it * gridDim.x, pb = bh / prm.hdiv, ph = bh - pb * prm.hdiv;
                if (it > 0 && !mbar_wait(plane_free, (it - 1) & 1, abort_flag, prm.status, kBit)) break;
                mbar_expect_tx(k_full, tiles * kTileBytes);
                for (int t = 0; t < tiles; ++t) tma_load_4d_hint(K_s + t * kTileBytes, &tmK, k_full, 0, t * kTile, ph, pb, pol);
                mbar_expect_tx(v_full, tiles * kTileBytes);
                for (int t = 0; t < tiles; ++t) tma_load_4d(V_s + t * kTileBytes, &tmV, v_full, 0, t * kTile, ph, pb);
                auto load_q = [&]() {
                    mbar_expect_tx(q_full, tiles * kTileBytes);
                    for (int t = 0; t < tiles; ++t) tma_load_4d_hint(Q_s + t * kTileBytes, &tmQ, q_full, 0, t * kTile, ph, pb, pol);
                };
                if (!FINE) load_q();
                ++issued;
                // the K tiles are dead once the state UMMAs have retired: bring V in again, unswizzled
                if (!mbar_wait(s_done, it & 1, abort_flag, prm.status, kBit)) break;
                if (FINE) load_q();   // over the rest of K
                if (ROOMY) {
                    mbar_expect_tx(vp_full, (W + 2 * R) * (prm.gridH + 2 * R) * kRow);
                    tma_load_5d(K_s, &tmVplain, vp_full, 0, -R, -R, ph, pb);
                } else {
                    mbar_expect_tx(vp_full, tiles * kTileBytes);
                    for (int t = 0; t < tiles; ++t) tma_load_4d(K_s + t * kTileBytes, &tmVplain, vp_full, 0, t * kTile, ph, pb);
                }
                ++issued_vp;
            }
            if (*abort_flag) {
                // giving up: let the copies in flight land before shared memory goes away
                if (issued) {
                    const uint32_t ph = (issued - 1) & 1;
                    for (int spin = 0; spin < (1 << 20) && !mbar_try_wait(k_full, ph); ++spin) {}
                    for (int spin = 0; spin < (1 << 20) && !mbar_try_wait(v_full, ph); ++spin) {}
                }
                const int issued_q = FINE ? issued_vp : issued;
                if (issued_q) for (int spin = 0; spin < (1 << 20) && !mbar_try_wait(q_full, (issued_q - 1) & 1); ++spin) {}
                if (issued_vp) for (int spin = 0; spin < (1 << 20) && !mbar_try_wait(vp_full, (issued_vp - 1) & 1); ++spin) {}
            }
        }
    } else if (warp == 1) {
        // the whole warp walks through the planes, one elected lane issues
        constexpr uint32_t idesc_state = umma_idesc_bf16(NARROW ? 64 : 128, kW, true, true);
        constexpr uint32_t idesc_apply = umma_idesc_bf16(kTile, kW, false, true);
        const uint32_t k_addr = smem_u32(K_s), v_addr = smem_u32(V_s), q_addr = smem_u32(Q_s);
        const uint32_t s_addr = smem_u32(S_s), ones_addr = smem_u32(ones);
        // 16 tokens (rows) on; for A stepping adds to the address of K and takes the same off the distance to the constant block
        constexpr uint32_t kStepB = 16 * kRow >> 4, kStepA = kStepB - (kStepB << 16);
        const int steps = (N + 15) / 16;
        for (int it = 0; it < n_planes; ++it) {
            const uint32_t ph = it & 1;
            if (!mbar_wait_warp(v_full, ph, abort_flag, prm.status, kBit)) break;
            // the previous plane's output accumulators share TMEM columns with this plane's state
            if (it > 0 && !mbar_wait_warp(tm_free, (it - 1) & 1, abort_flag, prm.status, kBit)) break;
            if (!mbar_wait_warp(k_scaled, ph, abort_flag, prm.status, kBit)) break;
            tcgen05_fence_after_sync();
            if (elect_one()) {
                uint32_t a = desc_low(k_addr, ones_addr - k_addr), b = desc_low(v_addr);
                uint32_t rest = FINE ? desc_low(q_addr, ones_addr - q_addr) : 0;   // its row of ones counts the tokens a second time
#pragma unroll 4
                for (int j = 0; j < steps; ++j, a += kStepA, b += kStepB) {  // one UMMA per 16 tokens (K = 16)
                    umma_bf16_low<kHigh>(tmem, a, b, idesc_state, j != 0);
                    if (FINE) { umma_bf16_low<kHigh>(tmem, rest, b, idesc_state, 1u); rest += kStepA; }
                }
                umma_commit(s_done);
            }
            __syncwarp();
            if (!mbar_wait_warp(q_full, ph, abort_flag, prm.status, kBit)) break;
            if (!mbar_wait_warp(sp_ready, ph, abort_flag, prm.status, kBit)) break;
            tcgen05_fence_after_sync();
            if (elect_one()) {
                const uint32_t sl = desc_low(s_addr), sl_rest = desc_low(v_addr);
                for (int t = 0; t < tiles; ++t) {
                    const uint32_t q = desc_low(q_addr + t * kTileBytes);
#pragma unroll
                    for (int k = 0; k < kW / 16; ++k) umma_bf16_low<kHigh>(tmem + t * kW, q + k * 2, sl + k * kStepB, idesc_apply, k != 0);
#pragma unroll
                    for (int k = 0; FINE && k < kW / 16; ++k) umma_bf16_low<kHigh>(tmem + t * kW, q + k * 2, sl_rest + k * kStepB, idesc_apply, 1u);
                }
                umma_commit(o_done);
            }
            __syncwarp();
        }
    } else {
        const int wt = tid - 64;                    // the line this thread normalises
        const int ww = warp - 2;                    // worker warp
        const int quarter = warp & 3;               // TMEM lanes 32*quarter .. +31 are this warp's
        const int half = ww >> 2;                   // of kHalves warps with the same lanes
        const bool has_line = wt * (NARROW ? 2 : 1) < N;
        const float2 zero2 = make_float2(0.f, 0.f);
        // units of the convolution: strips of two output columns per lane, cut along y as long as there are fewer than warps
        const int n_strips = NARROW ? (W + 3) / 4 : (W + 1) / 2, cuts = min(prm.gridH, max(1, kWarps / n_strips));
        const int seg_rows = (prm.gridH + cuts - 1) / cuts, n_units = n_strips * ((prm.gridH + seg_rows - 1) / seg_rows);
        const int first_strip = ww % n_strips, first_seg = ww / n_strips;
        // 1 / max(norm, eps) of each half of this thread's line of K or Q: c[j] is 16-byte chunk j ^ (wt & 7) of the 128 bytes.
        // Two tokens: chunk c of token 2 wt (+ 1) sits at c ^ (wt & 3) of its half, so the walk meets all four chunks of token
        // 2 wt + bit 2 of wt first.
        auto sums = [&](const uint4 (&c)[8], float& sa, float& sb) {
            float2 ss[4] = {zero2, zero2, zero2, zero2};
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint32_t w4[4] = {c[j].x, c[j].y, c[j].z, c[j].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 p = make_float2(bf16lo(w4[e]), bf16hi(w4[e]));
                    ss[2 * (j >> 2) + (e & 1)] = ffma2(p, p, ss[2 * (j >> 2) + (e & 1)]);
                }
            }
            sa = (ss[0].x + ss[0].y) + (ss[1].x + ss[1].y);
            sb = (ss[2].x + ss[2].y) + (ss[3].x + ss[3].y);
        };
        for (int it = 0; it < n_planes; ++it) {
            const uint32_t ph = it & 1;
            const int bh = blockIdx.x + it * gridDim.x;
            const int h = (prm.head0 + bh) % prm.H;
            __nv_bfloat16* const out_bh = prm.out + plane_offset(prm.lo, bh, prm.hdiv);
            // this thread's share of the head's filters (and bias): on its way while the rows are normalised, into shared memory
            // once the state is ready.  Volatile: left to itself the compiler moves the loads down to their use.
            constexpr int kElems = kW * KS * KS, kShare = (kElems + WORKERS - 1) / WORKERS;
            unsigned short fraw[kShare], braw = 0;
            {
                const unsigned short* w0 = reinterpret_cast<const unsigned short*>(prm.w) + (size_t)h * kElems;
#pragma unroll
                for (int i = 0; i < kShare; ++i) {
                    fraw[i] = 0;
                    if (wt + i * WORKERS < kElems) asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(fraw[i]) : "l"(w0 + wt + i * WORKERS));
                }
                if (prm.bias && wt < kW)
                    asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(braw) : "l"(reinterpret_cast<const unsigned short*>(prm.bias) + h * kW + wt));
            }
            // A thread whose wait has run out goes straight to the barrier behind this block, where all of them leave.
            bool ok = false;
            do {
            // ---- K rows -> unit rows, in place ----
            if (!mbar_wait(k_full, ph, abort_flag, prm.status, kBit)) break;
            if (has_line) {
                uint8_t* row = K_s + wt * 128;
                uint4 c[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) c[j] = *reinterpret_cast<const uint4*>(row + ((j ^ (wt & 7)) << 4));
                float sa, sb;
                sums(c, sa, sb);
                const float rka = inv_sqrt(fmaxf(NARROW ? sa : sa + sb, prm.eps2));
                const float rkb = NARROW ? inv_sqrt(fmaxf(sb, prm.eps2)) : rka;
                // 3x3 filters: the row is read again, as it leaves too few registers for the rest.  From a graph, read again / kept: 12 planes of
                // 14 x 14, width 64, 6.7 / 7.2 us, 768 planes 28.7 / 30.8, width 32 15.5 / 15.3; 5x5 filters 53.8 / 53.1, width 32 26.2 / 25.0.
#pragma unroll(KS == 3 ? 4 : 8)
                for (int j = 0; j < 8; ++j) {
                    const uint4 c4 = KS == 3 ? *reinterpret_cast<const uint4*>(row + ((j ^ (wt & 7)) << 4)) : c[j];
                    const uint32_t w4[4] = {c4.x, c4.y, c4.z, c4.w};
                    const float2 rk2 = (j < 4) ? make_float2(rka, rka) : make_float2(rkb, rkb);
                    uint32_t o4[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 p = ffma2(make_float2(bf16lo(w4[e]), bf16hi(w4[e])), rk2, zero2);
                        o4[e] = pack_bf16x2(p.x, p.y);
                    }
                    *reinterpret_cast<uint4*>(row + ((j ^ (wt & 7)) << 4)) = make_uint4(o4[0], o4[1], o4[2], o4[3]);
                    if (FINE) {
                        uint32_t r4[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) r4[e] = rest_bf16x2(w4[e], rk2.x, o4[e]);
                        *reinterpret_cast<uint4*>(Q_s + wt * 128 + ((j ^ (wt & 7)) << 4)) = make_uint4(r4[0], r4[1], r4[2], r4[3]);
                    }
                }
                fence_proxy_async_smem();
            } else if (FINE && wt * 2 < (N + 15) / 16 * 16) {   // tokens beyond the plane that the UMMAs take along
#pragma unroll
                for (int j = 0; j < 8; ++j) *reinterpret_cast<uint4*>(Q_s + wt * 128 + (j << 4)) = make_uint4(0, 0, 0, 0);
                fence_proxy_async_smem();
            }
            mbar_arrive(k_scaled);

            // ---- 1 / max(||q||, eps) ----
            auto q_norms = [&]() {
                if (!has_line) return;
                const uint8_t* row = Q_s + wt * 128;
                uint4 c[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) c[j] = *reinterpret_cast<const uint4*>(row + ((j ^ (wt & 7)) << 4));
                float sa, sb;
                sums(c, sa, sb);
                if (NARROW) {
                    const int first = (wt >> 2) & 1;
                    rq_s[2 * wt + first] = rsqrtf(fmaxf(sa, prm.eps2));
                    rq_s[2 * wt + 1 - first] = rsqrtf(fmaxf(sb, prm.eps2));
                } else {
                    rq_s[wt] = rsqrtf(fmaxf(sa + sb, prm.eps2));
                }
            };
            if (!FINE) {
                if (!mbar_wait(q_full, ph, abort_flag, prm.status, kBit)) break;
                q_norms();
            }

            // ---- S, s out of TMEM -> S' (bf16 operand) and s ----
            if (!mbar_wait(s_done, ph, abort_flag, prm.status, kBit)) break;
            tcgen05_fence_after_sync();
            if (quarter < 3) {
                // rows 0..63 in lanes 0..63, row 64 in lane 64; M = 64 (NARROW): rows 16 q .. 16 q + 15 in lanes 32 q .. 32 q + 15
                const int row = NARROW ? (lane < 16 ? quarter * 16 + lane : kW + 1) : quarter * 32 + lane;
#pragma unroll
                for (int cc = 0; cc < kW / 16 / kHalves; ++cc) {
                    const int col = (half * (kW / 16 / kHalves) + cc) * 16;
                    float a[16];
                    tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + col, a);
                    tmem_ld_wait();
                    if (row < kW) {   // key feature `row`
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            uint4 o;
                            o.x = pack_bf16x2(a[8 * e + 0] * kInvPi, a[8 * e + 1] * kInvPi);
                            o.y = pack_bf16x2(a[8 * e + 2] * kInvPi, a[8 * e + 3] * kInvPi);
                            o.z = pack_bf16x2(a[8 * e + 4] * kInvPi, a[8 * e + 5] * kInvPi);
                            o.w = pack_bf16x2(a[8 * e + 6] * kInvPi, a[8 * e + 7] * kInvPi);
                            const int chunk = (col / 8 + e) ^ (NARROW ? (row >> 1) & 3 : row & 7);
                            *reinterpret_cast<uint4*>(S_s + row * kRow + (chunk << 4)) = o;
                            if (FINE) *reinterpret_cast<uint4*>(V_s + row * kRow + (chunk << 4)) =
                                make_uint4(rest_bf16x2(a[8 * e + 0], a[8 * e + 1], kInvPi, o.x), rest_bf16x2(a[8 * e + 2], a[8 * e + 3], kInvPi, o.y),
                                           rest_bf16x2(a[8 * e + 4], a[8 * e + 5], kInvPi, o.z), rest_bf16x2(a[8 * e + 6], a[8 * e + 7], kInvPi, o.w));
                        }
                    } else if (row == kW) {   // the token sum of V
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            *reinterpret_cast<float4*>(sum_s + col + 4 * e) = make_float4(a[4 * e], a[4 * e + 1], a[4 * e + 2], a[4 * e + 3]);
                    }
                }
            }
            if (FINE) {
                if (!mbar_wait(q_full, ph, abort_flag, prm.status, kBit)) break;
                q_norms();
            }
            fence_proxy_async_smem();
            tcgen05_fence_before_sync();
            mbar_arrive(sp_ready);
            // [tap][channel] as fp32, then the bias (every warp has left the previous plane's convolution: s_done followed its
            // arrival on k_scaled)
#pragma unroll
            for (int i = 0; i < kShare; ++i) {
                const int e = wt + i * WORKERS;
                if (e < kElems) w_s[(e % (KS * KS)) * kW + e / (KS * KS)] = __uint_as_float((uint32_t)fraw[i] << 16);
            }
            if (wt < kW) w_s[kElems + wt] = __uint_as_float((uint32_t)braw << 16);

            // ---- accumulator rows out of TMEM -> fp32 rows in shared memory ----
            // Row t, times 1 / max(||q_t||, eps), from the start of the V buffer on, through the Q buffer, which follows it.  ROOMY: rows
            // of 16 bytes more; else 16-byte chunk c at chunk c ^ (t & 7): conflict-free for these row-per-thread writes and for
            // the reads below.  All UMMAs and all row-norm reads of those buffers are done:
            // o_done follows sp_ready, which every worker reaches after its reads of Q.
            if (!mbar_wait(o_done, ph, abort_flag, prm.status, kBit) || !mbar_wait(sp_ready, ph, abort_flag, prm.status, kBit)) break;
            tcgen05_fence_after_sync();
            {
                const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
                const int n = tiles * (kW / 16);
                auto write = [&](int i, const float (&a)[16]) {
                    const int t = i / (kW / 16), cc = i % (kW / 16), r = t * kTile + quarter * 32 + lane;
                    if (r >= N) return;
                    const float rq = rq_s[r];
                    uint8_t* srow = V_s + r * G::kAccRow;
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        *reinterpret_cast<float4*>(srow + (((cc * 4 + e) ^ (ROOMY ? 0 : r & 7)) << 4)) =
                            make_float4(a[4 * e] * rq, a[4 * e + 1] * rq, a[4 * e + 2] * rq, a[4 * e + 3] * rq);
                };
                for (int i = half; i < n; i += 2 * kHalves) {   // two loads under way
                    float a[16], b[16];
                    const bool two = i + kHalves < n;
                    tmem_ld16(lanes + i * 16, a);
                    if (two) tmem_ld16(lanes + (i + kHalves) * 16, b);
                    tmem_ld_wait();
                    write(i, a);
                    if (two) write(i + kHalves, b);
                }
            }
            tcgen05_fence_before_sync();
            mbar_arrive(tm_free);
            ok = mbar_wait(vp_full, ph, abort_flag, prm.status, kBit);
            } while (false);
            if (named_barrier_any(1, WORKERS, !ok)) break;  // accumulator rows, rq, s and filters are visible to every worker

            // ---- convolution + combine ----
            // A unit is a strip of two output columns per lane over a run of grid rows: every word of V is loaded (a row ahead)
            // and unpacked once per strip, sums of the KS open output rows stay in registers.  NARROW: the half warps take the
            // even and the odd columns of four.
            const int par = NARROW ? lane >> 4 : 0, cp = NARROW ? lane & 15 : lane;   // column parity, channel pair
            constexpr int STEP = NARROW ? 2 : 1, NIN = STEP + KS;
            const float half = FINE ? 0.25f : 0.5f;   // FINE: the sums are of every token twice
            const float2 hs2 = make_float2(half * sum_s[2 * cp], half * sum_s[2 * cp + 1]);   // 1/2 s
            const float2 bias2 = *reinterpret_cast<const float2*>(w_s + kElems + 2 * cp);
            const float2 c2 = make_float2(hs2.x + bias2.x, hs2.y + bias2.y);  // + bias: grid tokens
            const bool turned = !NARROW && prm.turned;
            const int down = turned ? kW : KS * kW, right = turned ? KS * kW : kW;   // from tap to tap
            float2 wreg[KS][KS];
#pragma unroll
            for (int dy = 0; dy < KS; ++dy)
#pragma unroll
                for (int dx = 0; dx < KS; ++dx) wreg[dy][dx] = *reinterpret_cast<const float2*>(w_s + dy * down + dx * right + 2 * cp);
            uint32_t* out_plane = reinterpret_cast<uint32_t*>(out_bh) + cp;
            const long long out_tok = OUT_PACKED ? kW / 2 : prm.lo.token / 2;  // 32-bit words per token
            const uint32_t acc_s = smem_u32(V_s) + (ROOMY ? cp * 8 : 0);
            auto load_acc = [&](int t, float2& a2) {   // of token t, scaled
                lds64(acc_s + (uint32_t)(t * G::kAccRow + (ROOMY ? 0 : (((cp >> 1) ^ (t & 7)) << 4) + (cp & 1) * 8)), a2);
            };
            const int pitch = ROOMY ? W + 2 * R : W;      // tokens of a row of V in the K buffer
            const uint32_t v_base = smem_u32(K_s) + cp * 4;
            for (int u = ww; u < n_units; u += kWarps) {
                const int strip = u < kWarps ? first_strip : u % n_strips, y_first = (u < kWarps ? first_seg : u / n_strips) * seg_rows, n_rows = min(seg_rows, prm.gridH - y_first);
                const int x0 = strip * 2 * STEP + par;    // grid column of the lane's first output; the next is x0 + STEP
                const bool first = x0 < W, second = x0 + STEP < W;
                uint32_t cmask[NIN];      // of the words that lie in the grid's columns
#pragma unroll
                for (int o = 0; o < NIN; ++o) cmask[o] = (unsigned)(x0 + o - R) < (unsigned)W ? 0xffffffffu : 0u;
                float2 acc[KS][2];   // output row y of the unit in slot y % KS
#pragma unroll
                for (int k = 0; k < KS; ++k) acc[k][0] = acc[k][1] = zero2;
                uint32_t raw[NIN], rmask = 0;   // the words of the next halo row, all ones if it lies in the grid
                float2 next[2] = {zero2, zero2};   // the attention terms of the output row that starts with it
                uint32_t v_row = v_base + (uint32_t)((ROOMY ? y_first * pitch + x0 : prm.prefix + (y_first - R) * W + x0 - R) * kRow);
                const int t0 = prm.prefix + y_first * W + x0, t_last = t0 + (n_rows - 1) * W;   // tokens of the unit's first and last output row
                int t = t0;                                // of the output row that starts with the next halo row
                auto load_row = [&](int hy) {
                    uint32_t from = v_row;
                    if (!ROOMY) {
                        rmask = (unsigned)(y_first + hy - R) < (unsigned)prm.gridH ? 0xffffffffu : 0u;
                        from = rmask ? v_row : v_base;
                    }
#pragma unroll
                    for (int o = 0; o < NIN; ++o) raw[o] = lds32(from + (uint32_t)(o * kRow));
                    v_row += (uint32_t)(pitch * kRow);
                    load_acc(t, next[0]);
                    load_acc(t + STEP, next[1]);   // beyond the row it is some other token's
                    t = min(t + W, t_last);        // no output row starts with the last halo rows
                };
                load_row(0);
                uint32_t* to = out_plane + (t0 - (KS - 1) * W) * out_tok;   // of the output row that ends with the halo row
                const int last = n_rows + KS - 2;
                // halo row hy of the unit: the output row that started dy rows ago, in slot (k - dy) % KS, takes filter row dy
                auto row = [&](int hy, int k, bool ends) {
                    float2 in[NIN];
#pragma unroll
                    for (int o = 0; o < NIN; ++o) {
                        const uint32_t word = ROOMY ? raw[o] : raw[o] & cmask[o] & rmask;
                        in[o] = make_float2(bf16lo(word), bf16hi(word));
                    }
                    // output row hy starts here; it ends KS - 1 rows on
                    acc[k][0] = fadd2(next[0], c2);
                    acc[k][1] = fadd2(next[1], c2);
                    load_row(hy + 1);
#pragma unroll
                    for (int dx = 0; dx < KS; ++dx)
#pragma unroll
                        for (int dy = 0; dy < KS; ++dy)
#pragma unroll
                            for (int c = 0; c < 2; ++c)
                                acc[(k - dy + KS) % KS][c] = ffma2_in_order(wreg[dy][dx], in[STEP * c + dx], acc[(k - dy + KS) % KS][c]);
                    // predicates, no branches
                    stg32_if(ends && first, to, pack_bf16x2(acc[(k + 1) % KS][0].x, acc[(k + 1) % KS][0].y));
                    stg32_if(ends && second, to + STEP * out_tok, pack_bf16x2(acc[(k + 1) % KS][1].x, acc[(k + 1) % KS][1].y));
                    to += W * out_tok;
                };
                if (NARROW && !FINE) {
                    // one row of code and moving sums: units of width 32 have few rows.  1024 planes of 16 x 16 22.8 us, 25.5 unrolled; with 5 x 5
                    // filters, 14 x 14, 29.8 / 31.9; width 64 (768 planes of 14 x 14) 28.8 / 28.1
#pragma unroll 1
                    for (int hy = 0; hy <= last; ++hy) {
                        row(hy, KS - 1, hy >= KS - 1);
#pragma unroll
                        for (int j = 0; j + 1 < KS; ++j) { acc[j][0] = acc[j + 1][0]; acc[j][1] = acc[j + 1][1]; }
                    }
                } else {
                    bool done = false;
                    for (int h0 = 0; !done; h0 += KS) {
#pragma unroll
                        for (int k = 0; k < KS; ++k) {
                            row(h0 + k, k, h0 > 0 || k == KS - 1);
                            if (h0 + k == last) { done = true; break; }
                        }
                    }
                }
            }
            // off-grid leading tokens: the attention terms only
            for (int t = ww * STEP + par; t < prm.prefix; t += kWarps * STEP) {
                float2 a2;
                load_acc(t, a2);
                out_plane[t * out_tok] = pack_bf16x2(a2.x + hs2.x, a2.y + hs2.y);
            }
            fence_proxy_async_smem();
            mbar_arrive(plane_free);
        }
    }
    tcgen05_fence_before_sync();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, G::kTmemCols);
}

template <int KS, bool NARROW, int WORKERS, bool FINE, bool ROOMY>
cudaError_t launch_fused_room(const Problem& p, bool turned, unsigned* status, cudaStream_t st) {
    using G = Geo<KS, NARROW, WORKERS, ROOMY>;
    CUtensorMap tmK, tmV, tmQ, tmVplain;
    // [d, tokens, planes per batch step, batch steps]
    const uint64_t nb = (uint64_t)(p.BH / p.hdiv);
    const uint64_t dims[4] = {(uint64_t)G::kW, (uint64_t)p.N, (uint64_t)p.hdiv, nb};
    const uint32_t box[4] = {(uint32_t)G::kW, kTile, 1, 1};
    auto strides = [&](const Layout& l, uint64_t (&s)[3]) {
        s[0] = (uint64_t)l.token; s[1] = (uint64_t)l.head; s[2] = (uint64_t)(nb > 1 ? l.batch : l.head * p.hdiv);
    };
    uint64_t sq[3], sk[3], sv[3];
    strides(p.lq, sq); strides(p.lk, sk); strides(p.lv, sv);
    if (!make_tensor_map_bf16(&tmK, p.k, 4, dims, sk, box, G::kRow) || !make_tensor_map_bf16(&tmV, p.v, 4, dims, sv, box, G::kRow) ||
        !make_tensor_map_bf16(&tmQ, p.q, 4, dims, sq, box, G::kRow))
        return cudaErrorNotSupported;
    if (ROOMY) {   // the token grid, after the off-grid leading tokens of every plane: what lies outside is zero-filled
        const uint64_t dims_g[5] = {(uint64_t)G::kW, (uint64_t)p.gridW, (uint64_t)p.gridH, (uint64_t)p.hdiv, nb};
        const uint64_t sg[4] = {sv[0], sv[0] * (uint64_t)p.gridW, sv[1], sv[2]};
        const uint32_t box_g[5] = {(uint32_t)G::kW, (uint32_t)(p.gridW + KS - 1), (uint32_t)(p.gridH + KS - 1), 1, 1};
        if (!make_tensor_map_bf16(&tmVplain, static_cast<const __nv_bfloat16*>(p.v) + p.prefix * p.lv.token, 5, dims_g, sg, box_g, 0))
            return cudaErrorNotSupported;
    } else if (!make_tensor_map_bf16(&tmVplain, p.v, 4, dims, sv, box, 0)) {
        return cudaErrorNotSupported;
    }
    FusedParams prm;
    prm.w = static_cast<const __nv_bfloat16*>(p.w);
    prm.bias = static_cast<const __nv_bfloat16*>(p.bias);
    prm.out = static_cast<__nv_bfloat16*>(p.out);
    prm.lo = p.lo;
    prm.H = p.H; prm.head0 = p.head0; prm.BH = p.BH; prm.hdiv = p.hdiv; prm.prefix = p.prefix; prm.N = p.N;
    prm.gridH = p.gridH; prm.gridW = p.gridW; prm.turned = turned;
    prm.eps2 = p.eps2; prm.status = status;
    static PerDevice opt_in[2];  // per instantiation
    const bool packed = (p.lo.token == G::kW);
    const cudaError_t e = packed ? opt_in_smem(tc_fused_kernel<KS, true, NARROW, WORKERS, FINE, ROOMY>, G::kSmem, opt_in[1])
                                 : opt_in_smem(tc_fused_kernel<KS, false, NARROW, WORKERS, FINE, ROOMY>, G::kSmem, opt_in[0]);
    if (e != cudaSuccess) return e;
    const int resident = G::kCtas * device_sm_count();
    const int grid = p.BH < resident ? p.BH : resident;
    // CTAs that start while the kernel before drains lie on the multiprocessors in the order in which these became free, not one by one in
    // turn, so that some get more of the CTAs with a plane more than others.  Width 32, whose planes take the issue slots of a whole multiprocessor, gains
    // only where no CTA has a second plane; width 64 unless the last round has few enough planes for each multiprocessor to keep a CTA without one,
    // and not just a few.  Us a call with a new output, started early / not (width 64): 330 planes of 14 x 14 15.5 / 16.6, 444 19.1 / 18.6, 700 29.0 / 26.8, 768
    // 29.6 / 31.0, 1000 37.6 / 35.2, 1536 49.2 / 51.5, 444 of 16 x 16 24.0 / 22.0 (22.7 before there were early starts), 700 35.6 / 31.3 (32.0), 1184 of
    // 11 x 11, three to a multiprocessor, 31.1 / 29.1 (30.9); width 32 from a graph, 256 of 14 x 14 6.8 / 7.9, 1024 of 16 x 16 24.1 / 22.8, 1024 of
    // 16 x 32 44.0 / 40.0.  Planes handed out by a counter instead: 12 planes 7.2 against 6.9, 768 30.2 against 29.4.
    const int last = p.BH % grid;   // planes of the last round, 0 if it is full
    const bool uneven = 4 * last >= grid && last <= grid * (G::kCtas - 1) / G::kCtas + grid / 20;
    // In one round, CTAs that start while between a third and all of the multiprocessors are busy share some of them with one another, which only planes
    // with their halo, whose work is short, gain from (us a call, early / not): 110 planes of 16 x 16 11.4 / 10.5, 48 8.6 / 10.5, 148 9.0 / 11.3; of 14 x 14 9.8 / 10.4.
    const bool crowded = !ROOMY && !NARROW && 3 * p.BH > device_sm_count() && p.BH < device_sm_count();
    const bool early = grid == p.BH ? !crowded : !NARROW && !uneven;
    auto launch = [&](auto kernel) {
        return launch_programmatic(kernel, early, dim3((unsigned)grid), dim3(G::kThreads), G::kSmem, st, tmK, tmV, tmQ, tmVplain, prm);
    };
    return packed ? launch(tc_fused_kernel<KS, true, NARROW, WORKERS, FINE, ROOMY>) : launch(tc_fused_kernel<KS, false, NARROW, WORKERS, FINE, ROOMY>);
}

template <int KS, bool NARROW, int WORKERS, bool FINE>
cudaError_t launch_fused_ks(const Problem& p_in, unsigned* status, cudaStream_t st) {
    // A grid of one row is taken as one of one column, its filters turned to match: the strips of the convolution slide down columns.  From a graph, row /
    // column, us: 64 planes of 1 x 200 15.3 / 11.4, 1536 of 1 x 100 55.6 / 38.9, 768 with 5x5 filters 60.8 / 35.2.  Width 32, whose strips are twice as
    // wide, gains nothing: 768 of 1 x 100 19.2, of 100 x 1 23.5.
    Problem p = p_in;
    const bool turned = !NARROW && p.gridH == 1 && p.gridW > 1;
    if (turned) { p.gridH = p.gridW; p.gridW = 1; }
    using G = Geo<KS, NARROW, WORKERS, true>;
    const bool roomy = (p.gridW + KS - 1) * (p.gridH + KS - 1) * G::kRow <= G::kBuf && p.gridW + KS - 1 <= 256 && p.gridH + KS - 1 <= 256 &&
                       p.N * G::kAccRow <= 2 * G::kBuf;
    return roomy ? launch_fused_room<KS, NARROW, WORKERS, FINE, true>(p, turned, status, st)
                 : launch_fused_room<KS, NARROW, WORKERS, FINE, false>(p, turned, status, st);
}

template <int KS, bool NARROW, bool FINE>
cudaError_t launch_fused_width(const Problem& p, unsigned* status, cudaStream_t st) {
    // Small CTAs when the plane fits and they need fewer rounds of planes: a plane takes them about 1.2 times as long.  Measured,
    // large against small: 1000 planes of 7 x 7, width 32, 17.3 / 13.5 us; 3000 of 16 x 16 71.3 / 56.9; 320 of 11 x 11, width
    // 64, 13.7 / 11.8; 5x5 filters, 450 of 11 x 11, 29.4 / 23.8.  As many rounds with either: 148 planes of 11 x 11 8.1 / 9.5,
    // 450 15.7 / 17.9.
    auto rounds = [&](int ctas) { const int n = ctas * device_sm_count(); return (p.BH + n - 1) / n; };
    if (p.N <= Geo<KS, NARROW, 128>::kTokens && rounds(Geo<KS, NARROW, 128>::kCtas) < rounds(Geo<KS, NARROW, 256>::kCtas))
        return launch_fused_ks<KS, NARROW, 128, FINE>(p, status, st);
    return launch_fused_ks<KS, NARROW, 256, FINE>(p, status, st);
}

}  // namespace

// Width 32 token-major (heads side by side): up to 256 tokens; beyond, the separate kernels.
bool fused_supports(const Problem& p) {
    if (!p.bf16 || (p.ksize != 3 && p.ksize != 5)) return false;
    return p.d == 64 ? p.N <= 256 : p.d == 32 && p.N <= (p.contiguous_tokens() ? 512 : 256);
}

cudaError_t launch_fused(const Problem& p, unsigned* status, cudaStream_t st) {
    if (p.fine) return p.ksize == 3 ? launch_fused_width<3, true, true>(p, status, st) : launch_fused_width<5, true, true>(p, status, st);
    if (p.d == 32) return p.ksize == 3 ? launch_fused_width<3, true, false>(p, status, st) : launch_fused_width<5, true, false>(p, status, st);
    return p.ksize == 3 ? launch_fused_width<3, false, false>(p, status, st) : launch_fused_width<5, false, false>(p, status, st);
}

}  // namespace tc
}  // namespace castling
