// Apply kernel of the tensor-core path for width-32 heads in 64-byte rows (bf16): any grid width, any number of tokens,
// tokens or heads next to one another in memory:
//     out_t = (1/pi) q^_t S + 1/2 s + bias + DWConv(V)_t                         (Eq. 9)
// The roles are those of the width-64 apply kernel, on patches of 8 x 32 or 16 x 16 tokens (256 rows of 64 bytes):
//   warp 0      TMA: Q patch (64-byte swizzle) and V patch with its halo (out-of-grid rows and columns zero-filled, which is
//               the convolution's padding)
//   warp 1      four UMMAs per patch: acc[2 x 128 x 32] = Q S', S' = S / pi in bf16
//   warps 2..9  thread = token: ||q||, accumulator row from TMEM, out = acc / max(||q||, eps) + staged, one rounding; a warp
//               holds 32 tokens (one row of the patch, or two) and stores them with a TMA copy of its own, so no barrier joins the warps
//   warps 10..  depthwise convolution, lane = (column parity, channel pair): two columns at a time slide down the patch, every
//               word of V is loaded and unpacked once per pair of columns, sums of the KS open output rows in registers;
//               result (+ 1/2 s + bias) staged in shared memory as fp32
// FINE: S' is held as two bf16, the value and what rounding it left off, and contracted with Q (which is exact) one after the other.
// Bound: the packed FMAs of the convolution, 2.5 to 3 cycles each (5 x 5 filters: its warps are busy 3 100 of the 3 300 cycles of
// a patch, with four of them as with eight).
// Measured (per forward with the state kernel): 8 x 8 planes of 50 x 75, 5 x 5 filters 33 us (FINE; 31 otherwise; 245 on the
// CUDA-core kernels; 39 with the words of a row loaded right before their use); 64 x 64 27 us (37 with two tokens
// packed to a 128-byte row, where a lane's window slid two tokens per output and loaded 4.3 words per output instead of 3.1, and
// two CTA-wide barriers joined the warps per patch).
#include "tc_common.cuh"
#include "tc_host.cuh"

#include <type_traits>

namespace castling {
namespace tc {
namespace {

constexpr int kD = 32;
constexpr int kTile = 256;                     // tokens of a patch (TX columns x 256 / TX rows): two UMMA tiles of 128
constexpr int kQBytes = kTile * kD * 2;        // 16 KiB
constexpr int kStgStride = kD * 4 + 16;        // fp32 row + 16 B: conflict-free row-per-thread reads
constexpr int kStgBytes = kTile * kStgStride;
constexpr int kEpiThreads = 256;
constexpr int kStages = 3;
constexpr int kCols = 2;                       // columns per lane of the convolution

template <int KS, int kTX, bool FINE> struct Geo {
    static constexpr int R = KS / 2, kTY = kTile / kTX;
    // a convolution warp takes 8 rows of four columns
    static constexpr int kConvWarps = 8, kConvThreads = kConvWarps * 32, kRows = 8, kGroups = kTX / (2 * kCols);
    static constexpr int kThreads = 64 + kEpiThreads + kConvThreads;
    static constexpr int HY = kTY + 2 * R, HX = kTX + 2 * R;
    static constexpr int kVBytes = HY * HX * kD * 2;
    static constexpr int kStage = ((kQBytes + kVBytes + 1023) / 1024) * 1024;
    // S' | its second block (row sums) | the rest of both (FINE) | 1/2 s (row sums) | out rows | stages | staging x2 | barriers; the
    // swizzle repeats every 512 bytes
    static constexpr int kOffS = 0, kOffS2 = 2048, kRest = 4096, kOffHs = FINE ? 8192 : 4096;
    static constexpr int kOffOut = FINE ? kOffHs + 512 : 5120, kOffStages = kOffOut + kQBytes;
    static constexpr int kOffStg = kOffStages + kStages * kStage;
    static constexpr int kOffBar = kOffStg + 2 * kStgBytes;
    static constexpr size_t kSmem = 1024 + kOffBar + 256;
    static_assert(kSmem <= 227 * 1024, "shared memory");
};

struct Apply32Params {
    const float* state;            // [BH][32*32 + 32 (+ 32)]
    const __nv_bfloat16* w;        // [H*32][KS][KS]
    const __nv_bfloat16* bias;     // [H*32] or nullptr
    int column;                    // the grid is one column, taken as a row
    int flat;                      // the planes have one uniform stride: the tensor maps are 4-D, [.., plane]
    int H, head0, hdiv, tilesX, tilesY, n_tiles;
    float eps2;
    unsigned* status;
    int n_tokens;                  // tokens per sequence (row-sum normalisation)
};

// RN: row-sum normalisation, as in the width-64 kernel: column 32 of the accumulator is q . sum k^ / pi.
template <int KS, bool RN, int kTX, bool FINE>
__global__ void __launch_bounds__((Geo<KS, kTX, FINE>::kThreads), 1)
tc_apply32_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmV,
                  const __grid_constant__ CUtensorMap tmO, const Apply32Params prm) {
    using G = Geo<KS, kTX, FINE>;
    constexpr int kTY = G::kTY;
    constexpr int kSW = kD * kD + kD + (RN ? kD : 0);   // words of one state
    constexpr int kAccN = RN ? kD + 16 : kD;            // columns the UMMAs write per tile
    constexpr int kAccTile = RN ? 2 * kD : kD, kAcc = 2 * kAccTile;
    constexpr int kTmemCols = 2 * kAcc;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_smem(smem_raw);
    uint8_t* S_s = smem + G::kOffS;
    uint8_t* S2_s = smem + G::kOffS2;
    float* hs_s = reinterpret_cast<float*>(smem + G::kOffHs);   // [2][32]
    uint8_t* out_s = smem + G::kOffOut;
    uint8_t* stages = smem + G::kOffStages;
    uint8_t* stg = smem + G::kOffStg;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + G::kOffBar);  // [kStages] TMA landed
    uint64_t* empty = full + kStages;                                 // [kStages] stage consumed
    uint64_t* acc_full = empty + kStages;                             // [2] UMMAs retired
    uint64_t* conv_full = acc_full + 2;                               // [2] staging written
    uint64_t* buf_free = conv_full + 2;                               // [2] accumulator + staging read
    uint64_t* s_ready = buf_free + 2;                                 // S' of the current plane written
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_ready + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g_begin = (int)((long long)prm.n_tiles * blockIdx.x / gridDim.x);
    const int g_end = (int)((long long)prm.n_tiles * (blockIdx.x + 1) / gridDim.x);
    const int my_tiles = g_end - g_begin;
    constexpr unsigned kBit = kStatusApplyTimeout;

    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], G::kConvThreads + kEpiThreads + 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&conv_full[b], G::kConvThreads); mbar_init(&buf_free[b], kEpiThreads); }
        mbar_init(s_ready, kEpiThreads);
        *abort_flag = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmO);
    }
    if (warp == 1) tmem_alloc(tmem_slot, kTmemCols);
    tcgen05_fence_before_sync();
    __syncthreads();
    tcgen05_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    pdl_launch_dependents();   // the next forward's state kernel may set itself up; it waits before it touches memory

    // position of the CTA's current patch, advanced without divisions
    int bh = g_begin / (prm.tilesX * prm.tilesY), py, px;
    {
        const int rem = g_begin - bh * prm.tilesX * prm.tilesY;
        py = rem / prm.tilesX;
        px = rem - py * prm.tilesX;
    }
    auto step = [&]() { if (++px == prm.tilesX) { px = 0; if (++py == prm.tilesY) { py = 0; ++bh; } } };

    if (warp == 0) {
        if (lane == 0) {
            int issued = 0;
            const uint64_t pol_q = l2_policy_evict_first();  // Q is read once
            for (int it = 0; it < my_tiles; ++it, step()) {
                const int s = it % kStages, use = it / kStages;
                if (use > 0 && !mbar_wait(&empty[s], (use - 1) & 1, abort_flag, prm.status, kBit)) break;
                const int y0 = py * kTY, x0 = px * kTX;
                uint8_t* qs = stages + s * G::kStage;
                mbar_expect_tx(&full[s], kQBytes + G::kVBytes);
                if (prm.flat) {
                    tma_load_4d_hint(qs, &tmQ, &full[s], 0, x0, y0, bh, pol_q);
                    tma_load_4d(qs + kQBytes, &tmV, &full[s], 0, x0 - G::R, y0 - G::R, bh);
                } else {
                    const int pb = bh / prm.hdiv, ph = bh - pb * prm.hdiv;
                    tma_load_5d_hint(qs, &tmQ, &full[s], 0, x0, y0, ph, pb, pol_q);
                    tma_load_5d(qs + kQBytes, &tmV, &full[s], 0, x0 - G::R, y0 - G::R, ph, pb);
                }
                ++issued;
            }
            if (*abort_flag) {
                for (int i = max(0, issued - kStages); i < issued; ++i)
                    for (int spin = 0; spin < (1 << 20) && !mbar_try_wait(&full[i % kStages], (i / kStages) & 1); ++spin) {}
            }
        }
    } else if (warp == 1) {
        constexpr uint32_t idesc = umma_idesc_bf16(128, kAccN, false, true);
        const uint32_t s_addr = smem_u32(S_s);
        const uint32_t s_low = desc_low(s_addr, RN ? smem_u32(S2_s) - s_addr : 0);
        constexpr uint32_t kRest = G::kRest >> 4;   // to the rest of S'
        int prev_bh = -1, seg = 0;
        for (int it = 0; it < my_tiles; ++it, step()) {
            const int s = it % kStages, use = it / kStages, b = it & 1, ub = it >> 1;
            if (bh != prev_bh) {
                if (!mbar_wait_warp(s_ready, seg & 1, abort_flag, prm.status, kBit)) break;
                ++seg; prev_bh = bh;
            }
            if (!mbar_wait_warp(&full[s], use & 1, abort_flag, prm.status, kBit)) break;
            if (ub > 0 && !mbar_wait_warp(&buf_free[b], (ub - 1) & 1, abort_flag, prm.status, kBit)) break;
            tcgen05_fence_after_sync();
            if (elect_one()) {
                const uint32_t q_low = desc_low(smem_u32(stages + s * G::kStage));   // K-major rows of 64 B
#pragma unroll
                for (int t = 0; t < 2; ++t)
#pragma unroll
                    for (int k = 0; k < (FINE ? 2 : 1) * kD / 16; ++k) {   // the operand is N-major, 16 K-rows of 64 B per step
                        const int kk = k % (kD / 16);
                        umma_bf16_low<kDescHigh64>(tmem + b * kAcc + t * kAccTile, q_low + t * (kQBytes / 2 >> 4) + kk * 2,
                                                   s_low + kk * (1024u >> 4) + (k < kD / 16 ? 0u : kRest), idesc, k != 0);
                    }
                umma_commit(&acc_full[b]);
                umma_commit(&empty[s]);  // the same UMMAs have finished reading the Q patch
            }
            __syncwarp();
        }
    } else if (warp < 10) {
        // ------- epilogue: thread = token; a warp holds one grid row of the patch, or two half as long -------
        const int quarter = warp & 3, tile = (warp - 2) >> 2, row = tile * 128 + quarter * 32 + lane, et = tid - 64;
        const uint32_t acc_addr = tmem + ((uint32_t)(quarter * 32) << 16) + tile * kAccTile;
        uint8_t* orow = out_s + row * 64;
        const int sw = (row >> 1) & 3;   // 64-byte swizzle: chunk c of a row at chunk c ^ sw
        const uint64_t pol_o = l2_policy_evict_first();
        int prev_bh = -1;
        pdl_wait_primary();  // the state kernel's results are read below
        for (int it = 0; it < my_tiles; ++it, step()) {
            const int b = it & 1, ub = it >> 1, s = it % kStages, use = it / kStages;
            if (bh != prev_bh) {
                // every UMMA that read the previous S' has retired (its acc_full was waited on below)
                prev_bh = bh;
                const float* st = prm.state + (size_t)bh * kSW;
                const int i = (et & 127) >> 2, part = et & 3;   // row i of the operand, 8 columns from 8 * part on
                uint4 o = make_uint4(0, 0, 0, 0);
                if (et < 128) {
                    const float4 lo = __ldg(reinterpret_cast<const float4*>(st + i * kD + part * 8));
                    const float4 hi = __ldg(reinterpret_cast<const float4*>(st + i * kD + part * 8 + 4));
                    o.x = pack_bf16x2(lo.x * kInvPi, lo.y * kInvPi); o.y = pack_bf16x2(lo.z * kInvPi, lo.w * kInvPi);
                    o.z = pack_bf16x2(hi.x * kInvPi, hi.y * kInvPi); o.w = pack_bf16x2(hi.z * kInvPi, hi.w * kInvPi);
                    uint8_t* at = S_s + i * 64 + ((part ^ ((i >> 1) & 3)) << 4);
                    *reinterpret_cast<uint4*>(at) = o;
                    if (FINE) *reinterpret_cast<uint4*>(at + G::kRest) =
                        make_uint4(rest_bf16x2(lo.x, lo.y, kInvPi, o.x), rest_bf16x2(lo.z, lo.w, kInvPi, o.y),
                                   rest_bf16x2(hi.x, hi.y, kInvPi, o.z), rest_bf16x2(hi.z, hi.w, kInvPi, o.w));
                } else if (RN) {   // second block of the operand: sum k^ / pi in column 0
                    const float z = __ldg(st + kD * kD + kD + i);
                    if (part == 0) o.x = pack_bf16x2(z * kInvPi, 0.f) & 0xffffu;
                    uint8_t* at = S2_s + i * 64 + ((part ^ ((i >> 1) & 3)) << 4);
                    *reinterpret_cast<uint4*>(at) = o;
                    if (FINE) {
                        if (part == 0) o.x = rest_bf16x2(z, 0.f, kInvPi, o.x) & 0xffffu;
                        *reinterpret_cast<uint4*>(at + G::kRest) = o;
                    }
                }
                fence_proxy_async_smem();
                mbar_arrive(s_ready);
            }
            if (!mbar_wait_warp(&full[s], use & 1, abort_flag, prm.status, kBit)) break;
            float rq;
            {
                const uint8_t* qrow = stages + s * G::kStage + row * 64;
                float2 ss[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint4 c = *reinterpret_cast<const uint4*>(qrow + ((j ^ sw) << 4));
                    const uint32_t w4[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 p = make_float2(bf16lo(w4[e]), bf16hi(w4[e]));
                        ss[e & 1] = ffma2(p, p, ss[e & 1]);
                    }
                }
                mbar_arrive(&empty[s]);  // the Q row has been read
                rq = rsqrtf(fmaxf((ss[0].x + ss[0].y) + (ss[1].x + ss[1].y), prm.eps2));
            }
            if (!mbar_wait_warp(&acc_full[b], ub & 1, abort_flag, prm.status, kBit)) break;
            tcgen05_fence_after_sync();
            float a[2][16];
            tmem_ld16(acc_addr + b * kAcc, a[0]);
            tmem_ld16(acc_addr + b * kAcc + 16, a[1]);
            float x[16];  // RN: q . sum k^ / pi in x[0]
            if (RN) tmem_ld16(acc_addr + b * kAcc + kD, x);
            tmem_ld_wait();
            if (!mbar_wait_warp(&conv_full[b], ub & 1, abort_flag, prm.status, kBit)) break;
            if (lane == 0) tma_store_wait_read();   // this warp's previous copy has read its rows of out_s
            __syncwarp();
            const uint8_t* srow = stg + b * kStgBytes + row * kStgStride;
            const float inv = RN ? 1.0f / fmaf(x[0], rq, 0.5f * (float)prm.n_tokens) : 1.0f;
            const float* hrow = hs_s + b * kD;
#pragma unroll
            for (int e = 0; e < 4; ++e) {  // 8 channels -> one 16-byte chunk of the bf16 row
                const float4 c0 = *reinterpret_cast<const float4*>(srow + e * 32);
                const float4 c1 = *reinterpret_cast<const float4*>(srow + e * 32 + 16);
                const float* ae = &a[e >> 1][(e & 1) * 8];
                float v[8] = {ae[0], ae[1], ae[2], ae[3], ae[4], ae[5], ae[6], ae[7]};
                const float cv[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    // RN: (acc / ||q|| + 1/2 s) / (n / 2 + q^ . sum k^ / pi); the staged value is convolution + bias only
                    v[k] = RN ? fmaf(fmaf(v[k], rq, hrow[e * 8 + k]), inv, cv[k]) : fmaf(v[k], rq, cv[k]);
                *reinterpret_cast<uint4*>(orow + ((e ^ sw) << 4)) =
                    make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
            }
            tcgen05_fence_before_sync();
            mbar_arrive(&buf_free[b]);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                const int y = py * kTY + (tile * 4 + quarter) * (32 / kTX), x0 = px * kTX;   // rows below the grid are clipped by TMA
                const uint8_t* src = out_s + (tile * 128 + quarter * 32) * 64;
                if (prm.flat) {
                    tma_store_4d_hint(&tmO, src, 0, x0, y, bh, pol_o);
                } else {
                    const int pb = bh / prm.hdiv;
                    tma_store_5d_hint(&tmO, src, 0, x0, y, bh - pb * prm.hdiv, pb, pol_o);
                }
                tma_store_commit();
            }
        }
        if (lane == 0) tma_store_wait_all();
    } else {
        // ------- depthwise convolution: lane = (column parity, channel pair), two columns at a time down the patch -------
        const int cw = warp - 10, par = lane >> 4, cp = lane & 15;
        constexpr int NIN = 2 * (kCols - 1) + KS;   // columns of V that two output columns (two apart) need
        const int x0 = (cw % G::kGroups) * 2 * kCols + par, y0 = cw / G::kGroups * G::kRows;   // first column of this lane; the next is x0 + 2
        float2 wreg[KS][KS], bias2 = make_float2(0.f, 0.f);
        float2 cinit = bias2, hs2 = bias2;
        auto load_filters = [&]() {
            const int ch = ((prm.head0 + bh) % prm.H) * kD + 2 * cp;
#pragma unroll
            for (int dy = 0; dy < KS; ++dy)
#pragma unroll
                for (int dx = 0; dx < KS; ++dx)
                    wreg[dy][dx] = make_float2(__bfloat162float(prm.w[(size_t)ch * KS * KS + dy * KS + dx]),
                                               __bfloat162float(prm.w[(size_t)(ch + 1) * KS * KS + dy * KS + dx]));
            if (prm.column) {   // the filters' middle column, as the middle row: the only taps that meet the grid
#pragma unroll
                for (int dx = 0; dx < KS; ++dx)
                    wreg[G::R][dx] = make_float2(__bfloat162float(prm.w[(size_t)ch * KS * KS + dx * KS + G::R]),
                                                 __bfloat162float(prm.w[(size_t)(ch + 1) * KS * KS + dx * KS + G::R]));
            }
            if (prm.bias) bias2 = make_float2(__bfloat162float(prm.bias[ch]), __bfloat162float(prm.bias[ch + 1]));
        };
        load_filters();      // of the first plane, while the state kernel finishes
        int prev_bh = -1;
        pdl_wait_primary();  // the token sums of the state kernel are read below
        for (int it = 0; it < my_tiles; ++it, step()) {
            const int s = it % kStages, use = it / kStages, b = it & 1, ub = it >> 1;
            if (bh != prev_bh) {
                if (prev_bh >= 0) load_filters();
                prev_bh = bh;
                const float* sv = prm.state + (size_t)bh * kSW + kD * kD + 2 * cp;
                hs2 = make_float2(0.5f * __ldg(sv), 0.5f * __ldg(sv + 1));
                cinit = RN ? bias2 : make_float2(hs2.x + bias2.x, hs2.y + bias2.y);
            }
            if (!mbar_wait_warp(&full[s], use & 1, abort_flag, prm.status, kBit)) break;
            if (ub > 0 && !mbar_wait_warp(&buf_free[b], (ub - 1) & 1, abort_flag, prm.status, kBit)) break;
            const uint8_t* vh = stages + s * G::kStage + kQBytes + (y0 * G::HX + x0) * 64 + cp * 4;
            uint8_t* so = stg + b * kStgBytes + (y0 * kTX + x0) * kStgStride + cp * 8;
            float2 acc[KS][kCols];   // output row y in slot y % KS
            uint32_t raw[NIN];       // the row's words, loaded a row ahead
#pragma unroll
            for (int o = 0; o < NIN; ++o) raw[o] = lds32(vh + o * 64);
#pragma unroll
            for (int hy = 0; hy < G::kRows + 2 * G::R; ++hy) {
                float2 in[NIN];
#pragma unroll
                for (int o = 0; o < NIN; ++o) in[o] = make_float2(bf16lo(raw[o]), bf16hi(raw[o]));
                if (hy + 1 < G::kRows + 2 * G::R) {
#pragma unroll
                    for (int o = 0; o < NIN; ++o) raw[o] = lds32(vh + ((hy + 1) * G::HX + o) * 64);
                }
                if (hy < G::kRows) acc[hy % KS][0] = acc[hy % KS][1] = cinit;   // output row hy starts here
                // taps in the outer loop: consecutive FMAs go to different sums
#pragma unroll
                for (int dx = 0; dx < KS; ++dx)
#pragma unroll
                    for (int dy = 0; dy < KS; ++dy) {
                        const int y = hy - dy;   // compile-time after unrolling
                        if (y < 0 || y >= G::kRows) continue;
#pragma unroll
                        for (int c = 0; c < kCols; ++c) acc[y % KS][c] = ffma2(wreg[dy][dx], in[2 * c + dx], acc[y % KS][c]);
                    }
                if (hy >= KS - 1) {              // and output row hy - (KS - 1) ends here
                    const int y = hy - (KS - 1);
#pragma unroll
                    for (int c = 0; c < kCols; ++c) *reinterpret_cast<float2*>(so + (y * kTX + 2 * c) * kStgStride) = acc[y % KS][c];
                }
            }
            if (RN && warp == 10 && par == 0) *reinterpret_cast<float2*>(hs_s + b * kD + 2 * cp) = hs2;
            mbar_arrive(&empty[s]);      // the V patch of this stage is no longer needed
            mbar_arrive(&conv_full[b]);
        }
    }
    tcgen05_fence_before_sync();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

template <int KS, bool RN, int kTX, bool FINE>
cudaError_t launch_apply32_ks(const Problem& p, bool column, const float* state, unsigned* status, cudaStream_t st) {
    using G = Geo<KS, kTX, FINE>;
    constexpr int kTY = G::kTY;
    CUtensorMap tmQ, tmV, tmO;
    // [32, columns, grid rows, planes per batch step, batch steps]; with a single batch step the last dimension is dropped
    const uint64_t nb = (uint64_t)(p.BH / p.hdiv);
    const int rank = nb > 1 ? 5 : 4;
    const uint64_t dims[5] = {(uint64_t)kD, (uint64_t)p.gridW, (uint64_t)p.gridH, (uint64_t)p.hdiv, nb};
    const uint32_t boxq[5] = {kD, kTX, kTY, 1, 1}, boxv[5] = {kD, (uint32_t)G::HX, (uint32_t)G::HY, 1, 1}, boxo[5] = {kD, kTX, 32 / kTX, 1, 1};
    auto strides = [&](const Layout& l, uint64_t (&s)[4]) {
        s[0] = (uint64_t)l.token; s[1] = (uint64_t)(l.token * p.gridW); s[2] = (uint64_t)l.head;
        s[3] = (uint64_t)(nb > 1 ? l.batch : l.head * p.hdiv);
    };
    uint64_t sq[4], sv[4], so[4];
    strides(p.lq, sq); strides(p.lv, sv); strides(p.lo, so);
    // the token grid starts after the off-grid leading tokens of every plane
    const __nv_bfloat16* qg = static_cast<const __nv_bfloat16*>(p.q) + p.prefix * p.lq.token;
    const __nv_bfloat16* vg = static_cast<const __nv_bfloat16*>(p.v) + p.prefix * p.lv.token;
    __nv_bfloat16* og = static_cast<__nv_bfloat16*>(p.out) + p.prefix * p.lo.token;
    if (!make_tensor_map_bf16(&tmQ, qg, rank, dims, sq, boxq, 64) || !make_tensor_map_bf16(&tmO, og, rank, dims, so, boxo, 64) ||
        !make_tensor_map_bf16(&tmV, vg, rank, dims, sv, boxv, 0))
        return cudaErrorNotSupported;
    Apply32Params prm;
    prm.state = state;
    prm.column = column ? 1 : 0;
    prm.w = static_cast<const __nv_bfloat16*>(p.w);
    prm.bias = static_cast<const __nv_bfloat16*>(p.bias);
    prm.flat = (rank == 4) ? 1 : 0;
    prm.H = p.H; prm.head0 = p.head0; prm.hdiv = p.hdiv;
    prm.tilesX = (p.gridW + kTX - 1) / kTX; prm.tilesY = (p.gridH + kTY - 1) / kTY;
    prm.n_tiles = p.BH * prm.tilesX * prm.tilesY;
    prm.eps2 = p.eps2; prm.status = status; prm.n_tokens = p.N;
    static PerDevice opt_in;  // one per instantiation
    {
        const cudaError_t e = opt_in_smem(tc_apply32_kernel<KS, RN, kTX, FINE>, G::kSmem, opt_in);
        if (e != cudaSuccess) return e;
    }
    const int sms = device_sm_count();
    const int grid = prm.n_tiles < sms ? prm.n_tiles : sms;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(G::kThreads); cfg.dynamicSmemBytes = G::kSmem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, tc_apply32_kernel<KS, RN, kTX, FINE>, tmQ, tmV, tmO, prm);
}

template <int KS, bool RN, bool FINE>
cudaError_t launch_apply32_rn(const Problem& p, bool column, const float* state, unsigned* status, cudaStream_t st) {
    // Patches of 16 x 16 where they need fewer rounds of the device.  Measured, 32 columns wide against 16: 8 x 8 planes of
    // 50 x 75, 5 x 5 filters 31.4 / 30.6 us (10 rounds / 9), 25 x 38 18.0 / 16.1 (4 / 3), 3 x 3, 31 x 33 14.1 / 12.9 (4 / 3); as
    // many rounds: 64 x 64 27.4 / 27.6; fewer with 32: 100 x 150 84.4 / 88.5 (29 / 31), 64 x 8 planes of 24 x 24 28.1 / 31.5.
    auto rounds = [&](int tx) {
        const long long n = (long long)p.BH * ((p.gridW + tx - 1) / tx) * ((p.gridH + kTile / tx - 1) / (kTile / tx));
        return (n + device_sm_count() - 1) / device_sm_count();
    };
    return rounds(16) < rounds(32) ? launch_apply32_ks<KS, RN, 16, FINE>(p, column, state, status, st)
                                   : launch_apply32_ks<KS, RN, 32, FINE>(p, column, state, status, st);
}

}  // namespace

cudaError_t launch_apply32(const Problem& given, const float* state, unsigned* status, cudaStream_t st) {
    // A grid of one column is taken as one row, of which a patch holds 32 tokens or 16 instead of 8 or 16: 8 x 8 planes of
    // 16383 x 1, 5 x 5 filters 455 us (895 as a column), 3 x 3 319 (595).
    Problem p = given;
    const bool column = given.gridW == 1 && given.gridH > 1;
    if (column) { p.gridH = 1; p.gridW = given.gridH; }
    auto launch = [&](auto fine) {
        constexpr bool F = decltype(fine)::value;
        if (p.ksize == 3) return p.rownorm ? launch_apply32_rn<3, true, F>(p, column, state, status, st) : launch_apply32_rn<3, false, F>(p, column, state, status, st);
        return p.rownorm ? launch_apply32_rn<5, true, F>(p, column, state, status, st) : launch_apply32_rn<5, false, F>(p, column, state, status, st);
    };
    return p.fine ? launch(std::true_type{}) : launch(std::false_type{});
}

}  // namespace tc
}  // namespace castling
