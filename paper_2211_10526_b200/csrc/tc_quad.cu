// Attention with explicit weights on the tensor cores, bf16, head width 64: the exact angular kernel (Eq. 4-5)
//     out_t = sum_j (1 - arccos(q^_t . k^_j) / pi) v_j + bias + DWConv(V)_t
// and / or the masked softmax branch of training (Eq. 10) on top of either base kernel; quadratic in the number of
// tokens.  A work item is a plane and one or two tiles ("slots") of 128 queries, which share every tile of 128 keys.
//   warp 0       one thread keeps four rings of TMA copies going: Q tiles (an item ahead), K tiles, V tiles, and patches of
//                the token grid with their halo for the convolution
//   warps 4..7   scale every K row and every Q row to a unit row in place, as bf16
//   warp 1       issues C[128 x 128] = Q^ K^^T, slot after slot, into three TMEM buffers in turn
//   warps 8..23  thread = (query, 64 of the tile's keys): cosines out of TMEM, the weights back over them as bf16 (eight
//                warps per slot)
//   warp 2       issues O[128 x 64] += W[128 x 128] V, whose A operand W is read from TMEM
//   warps 24..31 while the sweep over the keys runs: bias and depthwise convolution of V for the item's queries (lane =
//                channel pair, warp = two columns of the patch) into shared memory as fp32; then thread = query: O out of
//                TMEM, add, round, 128-byte rows to memory
// Keys beyond the plane have k^ = 0 and v = 0 and need no mask in the weighted sum.  The masked branch takes a first
// sweep over the keys that only forms the cosines and adds up exp(cosine) per query (keys beyond the plane excluded); in
// the second sweep the weight of a pair is the base weight plus Mask_eps of its softmax probability.  When a plane has at
// most kResident key tiles they stay in shared memory between the two sweeps.
//
// What bounds it: the issue slots of the warps that turn cosines into weights and rows into unit rows, on top of the hand-over of a
// cosine buffer (first contraction, weights, second contraction), of which tensor memory has room for three.  2 x 8 planes of 64 x 64
// tokens, exact kernel: 115 us; in working copies, when it took 119, 97 with cosines written back as they are, 76 with rows left as they are as well: what
// the weights and the rows take comes on top of the chain, which waits for tensor memory and barriers.  So a weight has no square root where the cosines
// of a tile are small (127 us with 5 packed operations a pair, 135.5 with the square roots, whose unit has 16 lanes; 119 with one operation less a
// pair and rows scaled by a refined reciprocal root, 121.4 with a root and a quotient; 115 where a tile is looked through before, not step by step after).  Rows are scaled in fp32 with one rounding, as they are
// everywhere.  K scaled by the weight warps instead (its norms beside it, cosines not before a packed product): 133 against 127, as
// sixteen warps pay for what four did.  Four K stages, the convolution staged for one slot at a time: 117 against 119, but the masked branch 66 against 62.
// The two contractions have an issuing warp each: a ready wait costs 50 to 90 cycles and an issue 30 per UMMA, which one warp could not do in time.
// Eight weight warps instead of sixteen (with square roots): 151 us against 135; all sixteen on one slot at a time: 139.
// Masked branch, 64 x 12 planes of 14 x 14: 56.2 us.  61 with the cosines clamped pair by pair in both sweeps, and the keys that pad a tile left
// out one by one; now the padding's ones are taken off the sum.  Rows of Q that bring the factor log2(e) along to the contraction save 0.2 us, but
// round it to bf16 with them.
// No workspace; every wait is bounded.
#include "tc_common.cuh"
#include "tc_host.cuh"

#include <type_traits>

namespace castling {
namespace tc {
namespace {

constexpr int kD = 64;
constexpr int kTile = 128;                          // queries per slot, keys per tile
constexpr int kTileBytes = kTile * kD * 2;          // 16 KiB
constexpr int kKStages = 2, kVStages = 2;
constexpr int kResident = 2;                        // key tiles of a plane that stay between the sweeps
constexpr int kCBufs = 3;                           // cosine buffers
constexpr int kNormThreads = 128, kSlotThreads = 256, kConvThreads = 256;
constexpr int kThreads = 128 + kNormThreads + 2 * kSlotThreads + kConvThreads;
constexpr int kTmemCols = 512;
constexpr int kColO = kCBufs * kTile;               // outputs of the two slots behind the cosine buffers
constexpr int kStgStride = kD * 4 + 16;             // fp32 row + 16 B: conflict-free row-per-thread access
constexpr int kOffQ = 0, kOffK = 4 * kTileBytes, kOffV = kOffK + kKStages * kTileBytes;   // Q: [2 items][2 slots]
constexpr int kPatchX = 16, kPatchBytes = 10 * 18 * kD * 2;   // 8 rows (5 x 5 filters: 4) x 16 columns and their halo
constexpr int kOffPatch = kOffV + kVStages * kTileBytes, kOffStg = kOffPatch + kPatchBytes;
constexpr int kOffDen = kOffStg + 2 * kTile * kStgStride;   // softmax denominators [2 items][2 slots][2 halves][128]
constexpr int kOffW = kOffDen + 8 * kTile * 4;              // filters of the item's head: [taps][32 lanes] channel pairs
constexpr int kOffBar = kOffW + 25 * 32 * 4;
constexpr size_t kSmem = 1024 + kOffBar + 384;
static_assert(kSmem <= 227 * 1024, "shared memory");
static_assert(kColO + 2 * kD <= kTmemCols, "tensor memory");

struct QuadParams {
    __nv_bfloat16* out;
    const __nv_bfloat16* w;
    const __nv_bfloat16* bias;
    Layout lo;
    int hdiv, H, head0, N, gridH, gridW;
    int column;                  // the grid is one column, taken as a row (kOneRow): the filters are read transposed
    int slots;                   // query tiles per item (1 or 2)
    int groups;                  // items per plane
    int k_tiles, n_items;
    float eps2;
    unsigned* status;
    float sparse_eps;            // threshold of the mask (sparse sweeps only)
};

// D[tmem] (+)= A[tmem] * B[smem]: row i of A in lane i, two bf16 of the contracted index per 32-bit column.
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_low, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 db, {%2, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_low), "r"(idesc), "r"(kDescHigh), "r"(accumulate)
        : "memory");
}
// 8 consecutive 32-bit columns of this thread's TMEM lane, written.
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float2 dup2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float exp2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
constexpr float kLog2e = 1.4426950408889634f;

// 1 - arccos(x)/pi of a pair, any cosine: with t = 1 - |x| (clamped to [0, 1]: rounding can leave a cosine just outside [-1, 1]),
// arccos(|x|) = sqrt(t) * cubic(t) -- Abramowitz & Stegun 4.4.45 with its cubic in |x| expanded about |x| = 1, |error| <
// 7e-5 rad, far below the bf16 rounding of the weights -- and 1 - arccos(x)/pi = 1/2 + sign(x) (1/2 - arccos(|x|)/pi).
__device__ __forceinline__ float2 angular_weight2(float2 x) {
    const float2 t = make_float2(__saturatef(1.0f - fabsf(x.x)), __saturatef(1.0f - fabsf(x.y)));
    const float2 s = make_float2(sqrt_approx(t.x), sqrt_approx(t.y));
    float2 p = ffma2(dup2(-0.0187293f * kInvPi), t, dup2(-0.0180731f * kInvPi));
    p = ffma2(p, t, dup2(-0.1197803f * kInvPi));
    p = ffma2(p, t, dup2(-1.4141461f * kInvPi));
    const float2 h = ffma2(s, p, dup2(0.5f));
    const uint32_t sx = __float_as_uint(x.x) & 0x80000000u, sy = __float_as_uint(x.y) & 0x80000000u;
    return fadd2(make_float2(__uint_as_float((__float_as_uint(h.x) & 0x7fffffffu) | sx),
                             __uint_as_float((__float_as_uint(h.y) & 0x7fffffffu) | sy)), dup2(0.5f));
}
// The same where both |x| <= kNearLimit: 1/2 + arcsin(x)/pi with arcsin(x)/x quadratic in x^2 (|error| < 5e-5 rad, 1.2e-5 in the
// root mean square over cosines of independent rows; the general form 4.5e-5).  No square root and less than half the instructions
// of the general form, which is left to tiles that hold a larger cosine: between independent rows of 64 elements 0.6 is
// 4.8 standard deviations, and one tile in 4 000 has one.
constexpr float kNearLimit = 0.6f;
__device__ __forceinline__ float2 angular_weight2_near(float2 x) {
    const float2 u = ffma2(x, x, dup2(0.f));
    float2 p = ffma2(dup2(0.03577495f), u, dup2(0.05099359f));
    p = ffma2(p, u, dup2(0.31836814f));
    return ffma2(p, x, dup2(0.5f));
}
// A warp looks a tile's cosines through, 64 keys of 32 queries, before it takes one form or the other for all of them; once it has met a large
// one it takes the general form unseen for this many tiles, or to the item's end.  16 planes of 64 x 64, us a call: independent rows 115.1,
// cosines about 0.95 137.7, about 0.3 139.6, a large one in every 40th key 137.9; with the general form alone, in the kernel before there were two,
// 135.5.  Both forms in turn in every step of 16 keys with a large cosine instead: 117.7, 181.9, 145.6, 138.8.
constexpr int kLookAgain = 16;
// (x + 1) log2(e) + bias of a pair of cosines, clamped to [-1, 1].
__device__ __forceinline__ float2 exponent2(float2 x, float bias) {
    const float2 y = make_float2(__saturatef(fmaf(x.x, 0.5f, 0.5f)), __saturatef(fmaf(x.y, 0.5f, 0.5f)));
    return ffma2(y, dup2(2.0f * kLog2e), dup2(bias));
}
__device__ __forceinline__ float one_if_greater(float a, float b) {
    float r;
    asm("set.gt.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
// Largest magnitude of three.
__device__ __forceinline__ float max3_abs(float a, float b, float c) {
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// GRID.  kWide: rows longer than an item's queries, which then lie in one row, or at the end of one and the beginning of the next,
// and need not all columns of patches: 16 planes of 2 x 2048 (exact kernel) 155 us, 460 with all columns.  kOneRow: the same with
// patches of one row; a grid of one column is taken as one row: 16 planes of 1 x 4096 138 us (809 in patches of eight rows and all
// columns), 768 planes of 196 x 1 105 us (254 in patches of which one column is used).
enum { kOrdinary, kWide, kOneRow };
template <int KS, bool SPARSE, bool EXACT, int GRID>
__global__ void __launch_bounds__(kThreads, 1)
tc_quad_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
               const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmP, const QuadParams prm) {
    constexpr int R = KS / 2, kPatchY = GRID == kOneRow ? 1 : KS == 3 ? 8 : 4, HX = kPatchX + 2 * R, HY = kPatchY + 2 * R;
    static_assert(HX * HY * kD * 2 <= kPatchBytes, "patch");
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_smem(smem_raw);
    uint8_t* Q_s = smem + kOffQ;
    uint8_t* K_s = smem + kOffK;
    uint8_t* V_s = smem + kOffV;
    uint8_t* stg = smem + kOffStg;
    uint64_t* q_full = reinterpret_cast<uint64_t*>(smem + kOffBar);   // [2] by item
    uint64_t* q_ready = q_full + 2;              // [2] Q rows scaled (one arrival per warp, here and below)
    uint64_t* q_free = q_ready + 2;              // [2] the item's last cosine UMMAs have read Q
    uint64_t* k_full = q_free + 2;               // [kKStages]
    uint64_t* k_scaled = k_full + kKStages;      // [kKStages]
    uint64_t* k_empty = k_scaled + kKStages;     // [kKStages]
    uint64_t* v_full = k_empty + kKStages;       // [kVStages]
    uint64_t* v_empty = v_full + kVStages;       // [kVStages]
    uint64_t* c_full = v_empty + kVStages;       // [2][kCBufs] by slot: cosines written
    uint64_t* r_done = c_full + 2 * kCBufs;      // [kCBufs] cosines of a first sweep read
    uint64_t* p_full = r_done + kCBufs;          // [kCBufs] weights written
    uint64_t* pv_done = p_full + kCBufs;         // [kCBufs] weights read by the second contraction
    uint64_t* o_full = pv_done + kCBufs;         // [2] by slot
    uint64_t* o_free = o_full + 2;               // [2]
    uint64_t* patch_full = o_free + 2;
    uint64_t* patch_free = patch_full + 1;       // (one arrival per convolution warp)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(patch_free + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int my_items = ((int)blockIdx.x < prm.n_items) ? (prm.n_items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    const int T = prm.k_tiles, N = prm.N;
    constexpr int kSweeps = SPARSE ? 2 : 1;
    const bool resident = SPARSE && T <= kResident;
    const int k_loads = resident ? T : kSweeps * T;   // K tiles loaded per item
    constexpr unsigned kBit = kStatusFusedTimeout;
    // item number i of this CTA: plane, first token, active slots
    struct Item { int bh, t0, slots; };
    auto item_of = [&](int i) -> Item {
        const int item = blockIdx.x + i * gridDim.x, bh = item / prm.groups, t0 = (item - bh * prm.groups) * prm.slots * kTile;
        return {bh, t0, min(prm.slots, (N - t0 + kTile - 1) / kTile)};
    };
    // patches of the token grid that hold an item's queries
    struct Patches { int y0, nx, n; };
    auto patches_of = [&](const Item& im) -> Patches {
        const int y0 = im.t0 / prm.gridW, y1 = (min(N, im.t0 + im.slots * kTile) - 1) / prm.gridW;
        const int nx = (prm.gridW + kPatchX - 1) / kPatchX;
        if (GRID != kOrdinary) {   // from the first query's column of patches on; y1 - y0 is 0 or 1
            const int first = (im.t0 - y0 * prm.gridW) / kPatchX, last = (min(N, im.t0 + im.slots * kTile) - 1 - y1 * prm.gridW) / kPatchX;
            return {y0, nx, min(nx, last - first + 1 + (y1 - y0) * nx)};
        }
        return {y0, nx, nx * ((y1 - y0) / kPatchY + 1)};
    };
    // column of patch j of an item on such a grid: past the last one from the first on
    auto wide_column = [&](const Item& im, const Patches& pa, int j) -> int {
        const int c = (im.t0 - pa.y0 * prm.gridW) / kPatchX + j;
        return c < pa.nx ? c : c - pa.nx;
    };
    auto warp_arrive = [&](uint64_t* bar) { __syncwarp(); if (lane == 0) mbar_arrive(bar); };   // for all lanes of a warp
    auto warp_wait = [&](uint64_t* bar, uint32_t parity) -> bool {
        return mbar_wait_warp(bar, parity, abort_flag, prm.status, kBit);
    };

    if (tid == 0) {
        for (int b = 0; b < 2; ++b) { mbar_init(&q_full[b], 1); mbar_init(&q_ready[b], kNormThreads / 32); mbar_init(&q_free[b], 1); }
        for (int s = 0; s < kKStages; ++s) { mbar_init(&k_full[s], 1); mbar_init(&k_scaled[s], kNormThreads / 32); mbar_init(&k_empty[s], 1); }
        for (int s = 0; s < kVStages; ++s) { mbar_init(&v_full[s], 1); mbar_init(&v_empty[s], 1); }
        for (int b = 0; b < kCBufs; ++b) {
            mbar_init(&c_full[b], 1); mbar_init(&c_full[kCBufs + b], 1);
            mbar_init(&r_done[b], kSlotThreads / 32); mbar_init(&p_full[b], kSlotThreads / 32); mbar_init(&pv_done[b], 1);
        }
        for (int s = 0; s < 2; ++s) { mbar_init(&o_full[s], 1); mbar_init(&o_free[s], kTile / 32); }
        mbar_init(patch_full, 1); mbar_init(patch_free, kConvThreads / 32);
        *abort_flag = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmP);
    }
    if (warp == 1) tmem_alloc(tmem_slot, kTmemCols);
    tcgen05_fence_before_sync();
    __syncthreads();
    tcgen05_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    // Launched programmatically dependent on whatever precedes it in the stream, which every thread waits for here: the limits of the
    // waits below are for this kernel's own work.
    pdl_launch_dependents();
    pdl_wait_primary();

    if (warp == 0) {
        if (lane == 0) {
            // independent rings, polled in turn: none waits behind another
            int qi = 0, ki = 0, kj = 0, vi = 0, vj = 0;   // next item (and tile of it) of each ring
            int pi = 0, pj = 0;                           // next item (and patch of it) of the convolution
            int kn = 0, vn = 0, pn = 0;                   // tiles and patches issued
            unsigned long long t_last = 0;
            uint32_t idle = 0;
            while (qi < my_items || ki < my_items || vi < my_items || pi < my_items) {
                bool moved = false;
                if (pi < my_items && (pn == 0 || mbar_poll(patch_free, (pn - 1) & 1))) {
                    const Item im = item_of(pi);
                    const Patches pa = patches_of(im);
                    const int pb = im.bh / prm.hdiv, ph = im.bh - pb * prm.hdiv, y = GRID == kOrdinary ? pj / pa.nx : 0;
                    const int x = GRID == kOrdinary ? pj - y * pa.nx : wide_column(im, pa, pj);
                    mbar_expect_tx(patch_full, HX * HY * kD * 2);
                    tma_load_5d(smem + kOffPatch, &tmP, patch_full, 0, x * kPatchX - R, pa.y0 + y * kPatchY - R, ph, pb);
                    ++pn;
                    if (++pj == pa.n) { pj = 0; ++pi; }
                    moved = true;
                }
                if (qi < my_items && (qi < 2 || mbar_poll(&q_free[qi & 1], ((qi >> 1) - 1) & 1))) {
                    const Item im = item_of(qi);
                    const int pb = im.bh / prm.hdiv, ph = im.bh - pb * prm.hdiv, b = qi & 1;
                    mbar_expect_tx(&q_full[b], im.slots * kTileBytes);
                    for (int s = 0; s < im.slots; ++s)
                        tma_load_4d(Q_s + (2 * b + s) * kTileBytes, &tmQ, &q_full[b], 0, im.t0 + s * kTile, ph, pb);
                    ++qi;
                    moved = true;
                }
                if (ki < my_items) {
                    const int s = kn % kKStages, use = kn / kKStages;
                    if (use == 0 || mbar_poll(&k_empty[s], (use - 1) & 1)) {
                        const int bh = item_of(ki).bh, pb = bh / prm.hdiv, ph = bh - pb * prm.hdiv;
                        mbar_expect_tx(&k_full[s], kTileBytes);
                        tma_load_4d(K_s + s * kTileBytes, &tmK, &k_full[s], 0, (kj % T) * kTile, ph, pb);
                        ++kn;
                        if (++kj == k_loads) { kj = 0; ++ki; }
                        moved = true;
                    }
                }
                if (vi < my_items) {
                    const int s = vn % kVStages, use = vn / kVStages;
                    if (use == 0 || mbar_poll(&v_empty[s], (use - 1) & 1)) {
                        const int bh = item_of(vi).bh, pb = bh / prm.hdiv, ph = bh - pb * prm.hdiv;
                        mbar_expect_tx(&v_full[s], kTileBytes);
                        tma_load_4d(V_s + s * kTileBytes, &tmV, &v_full[s], 0, vj * kTile, ph, pb);
                        ++vn;
                        if (++vj == T) { vj = 0; ++vi; }
                        moved = true;
                    }
                }
                if (moved) { idle = 0; continue; }
                __nanosleep(100);
                if ((++idle & 255u) == 0) {
                    const unsigned long long now = global_ns();
                    if (idle == 256u) t_last = now;
                    if (*abort_flag) break;
                    if (now - t_last > kWaitLimitNs) { *abort_flag = 1; atomicOr(prm.status, kBit); break; }
                }
            }
            if (*abort_flag) {  // giving up: let the copies in flight land before shared memory goes away
                for (int i = max(0, kn - kKStages); i < kn; ++i)
                    for (int spin = 0; spin < (1 << 20) && !mbar_try_wait(&k_full[i % kKStages], (i / kKStages) & 1); ++spin) {}
                for (int i = max(0, vn - kVStages); i < vn; ++i)
                    for (int spin = 0; spin < (1 << 20) && !mbar_try_wait(&v_full[i % kVStages], (i / kVStages) & 1); ++spin) {}
                if (pn > 0) for (int spin = 0; spin < (1 << 20) && !mbar_try_wait(patch_full, (pn - 1) & 1); ++spin) {}
                for (int i = max(0, qi - 2); i < qi; ++i)
                    for (int spin = 0; spin < (1 << 20) && !mbar_try_wait(&q_full[i & 1], (i >> 1) & 1); ++spin) {}
            }
        }
    } else if (warp == 1) {
        // ---- cosines: the whole warp walks through the schedule, one elected lane issues ----
        constexpr uint32_t idesc_c = umma_idesc_bf16(kTile, kTile, false, false);   // Q^ (K-major) x K^ (K-major)
        const uint32_t q_low = desc_low(smem_u32(Q_s)), k_low = desc_low(smem_u32(K_s));
        uint32_t pv_pending = 0, rd_pending = 0;   // bit b: buffer b was last handed to the second contraction / to a first sweep
        uint32_t pv_parity = 0, rd_parity = 0;     // bit b: parity of the next completion of pv_done[b] / r_done[b]
        int b = 0, ks = 0;                         // next buffer and K stage
        uint32_t k_par = 0;
        bool ok = true;
        for (int i = 0; i < my_items && ok; ++i) {
            const int slots = item_of(i).slots;
            if (!(ok = warp_wait(&q_ready[i & 1], (i >> 1) & 1))) break;
            const int ks_item = ks;                // resident: the second sweep reads the stages of the first
            const uint32_t k_par_item = k_par;
            for (int u = 0; u < kSweeps * T && ok; ++u) {
                const bool last_sweep = u >= (kSweeps - 1) * T;
                if (SPARSE && resident && u == T) { ks = ks_item; k_par = k_par_item; }
                if (!(ok = warp_wait(&k_scaled[ks], k_par))) break;
                for (int s = 0; s < slots; ++s) {
                    const uint32_t bit = 1u << b;
                    if (pv_pending & bit) {
                        ok = warp_wait(&pv_done[b], (pv_parity & bit) != 0);
                        pv_parity ^= bit;
                    } else if (SPARSE && (rd_pending & bit)) {
                        ok = warp_wait(&r_done[b], (rd_parity & bit) != 0);
                        rd_parity ^= bit;
                    }
                    if (!ok) break;
                    if (last_sweep) { pv_pending |= bit; rd_pending &= ~bit; } else { rd_pending |= bit; pv_pending &= ~bit; }
                    tcgen05_fence_after_sync();
                    if (elect_one()) {
                        const uint32_t d = tmem + b * kTile, a = q_low + (2 * (i & 1) + s) * (kTileBytes >> 4);
                        const uint32_t k = k_low + ks * (kTileBytes >> 4);
                        umma_bf16_low(d, a, k, idesc_c, 0u);
                        umma_bf16_low(d, a + 2, k + 2, idesc_c, 1u);
                        umma_bf16_low(d, a + 4, k + 4, idesc_c, 1u);
                        umma_bf16_low(d, a + 6, k + 6, idesc_c, 1u);
                        umma_commit(&c_full[s * kCBufs + b]);
                        if (s == slots - 1) {
                            if (last_sweep || !resident) umma_commit(&k_empty[ks]);
                            if (u == kSweeps * T - 1) umma_commit(&q_free[i & 1]);
                        }
                    }
                    __syncwarp();
                    b = b == kCBufs - 1 ? 0 : b + 1;
                }
                if (++ks == kKStages) { ks = 0; k_par ^= 1; }
            }
        }
    } else if (warp == 2) {
        // ---- weighted sums ----
        constexpr uint32_t idesc_o = umma_idesc_bf16(kTile, kD, false, true);       // W (TMEM) x V (N-major)
        const uint32_t v_low = desc_low(smem_u32(V_s));
        int b = 0, vs = 0;
        uint32_t p_parity = 0, v_par = 0, o_used = 0, o_parity = 0;
        bool ok = true;
        for (int i = 0; i < my_items && ok; ++i) {
            const int slots = item_of(i).slots;
            if (SPARSE) b = (b + T * slots) % kCBufs;   // the buffers of the first sweep are not this warp's
            for (int j = 0; j < T && ok; ++j) {
                if (!(ok = warp_wait(&v_full[vs], v_par))) break;
                for (int s = 0; s < slots; ++s) {
                    const uint32_t bit = 1u << b;
                    if (j == 0) {   // the previous item's output has been read out of TMEM
                        if ((o_used >> s) & 1) { ok = warp_wait(&o_free[s], (o_parity >> s) & 1); o_parity ^= 1u << s; }
                        o_used |= 1u << s;
                    }
                    ok = ok && warp_wait(&p_full[b], (p_parity & bit) != 0);
                    if (!ok) break;
                    p_parity ^= bit;
                    tcgen05_fence_after_sync();
                    if (elect_one()) {
                        const uint32_t d = tmem + kColO + s * kD, a = tmem + b * kTile, v = v_low + vs * (kTileBytes >> 4);
                        umma_ts(d, a, v, idesc_o, j != 0);
#pragma unroll
                        for (int k = 1; k < kTile / 16; ++k)   // the weights of each half of the keys lie in its half of the columns
                            umma_ts(d, a + (k & 3) * 8 + (k >> 2) * (kTile / 2), v + k * 128, idesc_o, 1u);
                        umma_commit(&pv_done[b]);
                        if (s == slots - 1) umma_commit(&v_empty[vs]);
                        if (j == T - 1) umma_commit(&o_full[s]);
                    }
                    __syncwarp();
                    b = b == kCBufs - 1 ? 0 : b + 1;
                }
                if (++vs == kVStages) { vs = 0; v_par ^= 1; }
            }
        }
    } else if (warp == 3) {
        // spare: keeps the roles below aligned to groups of four warps
    } else if (warp < 8) {
        // ---- unit rows ----
        const int t = tid - 128;
        // row t of a tile times 1 / max(norm, eps); read twice: the whole row does not fit beside the rest
        auto scale_row = [&](uint8_t* row) {
            auto chunk = [&](int j) { return reinterpret_cast<uint4*>(row + ((j ^ (t & 7)) << 4)); };
            float2 ss[4] = {dup2(0.f), dup2(0.f), dup2(0.f), dup2(0.f)};
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const uint4 c = *chunk(j);
                const uint32_t w[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 p = make_float2(bf16lo(w[e]), bf16hi(w[e]));
                    ss[e] = ffma2(p, p, ss[e]);
                }
            }
            const float2 sum = fadd2(fadd2(ss[0], ss[1]), fadd2(ss[2], ss[3]));
            const float2 rk2 = dup2(inv_sqrt(fmaxf(sum.x + sum.y, prm.eps2)));
#pragma unroll 4
            for (int j = 0; j < 8; ++j) {
                const uint4 c = *chunk(j);
                const uint32_t w[4] = {c.x, c.y, c.z, c.w};
                uint32_t o[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 p = ffma2(make_float2(bf16lo(w[e]), bf16hi(w[e])), rk2, dup2(0.f));
                    o[e] = pack_bf16x2(p.x, p.y);
                }
                *chunk(j) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        };
        // The Q tiles of item i + 1 come after the first K tiles of item i: their copy starts once the cosines of item
        // i - 1 are done, whose K tiles were all scaled before those of item i, so this wait never holds up its own cause.
        auto scale_q = [&](int i) -> bool {
            if (!warp_wait(&q_full[i & 1], (i >> 1) & 1)) return false;
            const int slots = item_of(i).slots;
            for (int s = 0; s < slots; ++s) scale_row(Q_s + (2 * (i & 1) + s) * kTileBytes + t * 128);
            fence_proxy_async_smem();
            warp_arrive(&q_ready[i & 1]);
            return true;
        };
        int ks = 0;
        uint32_t k_par = 0;
        const int q_after = min(k_loads, 2) - 1;
        bool ok = my_items > 0 && scale_q(0);
        for (int i = 0; i < my_items && ok; ++i) {
            for (int j = 0; j < k_loads; ++j) {
                if (!(ok = warp_wait(&k_full[ks], k_par))) break;
                scale_row(K_s + ks * kTileBytes + t * 128);
                fence_proxy_async_smem();
                warp_arrive(&k_scaled[ks]);
                if (++ks == kKStages) { ks = 0; k_par ^= 1; }
                if (j == q_after && i + 1 < my_items && !(ok = scale_q(i + 1))) break;
            }
        }
    } else if (warp < 24) {
        // ---- weights: thread = query row of slot (warp - 8) / 8, half of the keys of every tile ----
        const int slot = (warp - 8) >> 3, half = ((warp - 8) >> 2) & 1, quarter = warp & 3;
        const uint32_t col0 = tmem + ((uint32_t)(quarter * 32) << 16) + half * (kTile / 2);
        int b = 0;                  // buffer of the next step of the CTA (this slot's or not)
        uint32_t par = 0;           // bit b: parity of the next completion of this slot's c_full[b]
        auto skip = [&](int n) { b = (b + n) % kCBufs; };
        auto wait_cosines = [&]() -> bool {
            const bool done = warp_wait(&c_full[slot * kCBufs + b], (par >> b) & 1);
            par ^= 1u << b;
            return done;
        };
        // with the mask too, both forms take more registers than there are: 16 planes of 64 x 64 334 us, 295 with the general one alone
        constexpr bool kNear = EXACT && !SPARSE;
        bool ok = true;
        // with the mask, a warp that has given up still meets the others at the next item's denominators, where all leave
        for (int i = 0; i < my_items && (ok || SPARSE); ++i) {
            const Item im = item_of(i);
            if (slot >= im.slots) { skip(kSweeps * T * im.slots); continue; }
            const bool live = im.t0 + slot * kTile + quarter * 32 < N;   // some row of this warp is a token
            float ebias = 0.f;   // exp(x) / den = exp2(x log2(e) + ebias); EXACT: exp2(y * 2 log2(e) + ebias), y = (x + 1) / 2
            skip(slot);
            if (SPARSE) {
                float2 den = dup2(0.f);
                for (int jt = 0; jt < T; ++jt) {
                    if (!(ok = ok && wait_cosines())) break;
                    const int left = N - jt * kTile - half * (kTile / 2);   // keys of the plane from this half on
                    if (live && left > 0) {
                        tcgen05_fence_after_sync();
                        float x[2][16];
                        tmem_ld16(col0 + b * kTile, x[0]);
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc) {
                            tmem_ld_wait();
                            if (cc < 3) tmem_ld16(col0 + b * kTile + (cc + 1) * 16, x[(cc + 1) & 1]);
                            if (cc * 16 >= left) continue;
#pragma unroll
                            for (int e = 0; e < 16; e += 2) {
                                const float* xe = &x[cc & 1][e];
                                const float2 a = EXACT ? exponent2(make_float2(xe[0], xe[1]), -kLog2e) : ffma2(make_float2(xe[0], xe[1]), dup2(kLog2e), dup2(0.f));
                                den = fadd2(den, make_float2(exp2_approx(a.x), exp2_approx(a.y)));
                            }
                        }
                        // keys beyond the plane: cosine 0, an exponential of 1 each
                        if (left < kTile / 2) den.x -= (float)(-left & 15);
                        tcgen05_fence_before_sync();
                    }
                    warp_arrive(&r_done[b]);
                    skip(im.slots);
                }
                // the two halves of a query meet in shared memory (by item parity: a thread is never two items ahead)
                float* den_s = reinterpret_cast<float*>(smem + kOffDen) + ((i & 1) * 4 + slot * 2) * kTile + quarter * 32 + lane;
                den_s[half * kTile] = den.x + den.y;
                if (named_barrier_any(2 + slot, kSlotThreads, !ok)) break;
                ebias = (EXACT ? -kLog2e : 0.f) - __log2f(den_s[0] + den_s[kTile]);
            }
            [[maybe_unused]] int unseen = 0;   // tiles of the item that take the general form without a look
            for (int jt = 0; jt < T; ++jt) {
                if (!(ok = wait_cosines())) break;
                if (live) {
                    tcgen05_fence_after_sync();
                    const uint32_t cb = col0 + b * kTile;
                    const int left = N - jt * kTile - half * (kTile / 2);
                    float x[2][16];
                    auto tile = [&](auto near_form) {
#pragma unroll
                        for (int cc = 0; cc < 4; ++cc) {
                            if (!kNear || cc == 2) tmem_ld_wait();
                            if (!kNear && cc < 3) tmem_ld16(cb + (cc + 1) * 16, x[(cc + 1) & 1]);
                            uint32_t o[8];
                            if (cc * 16 < left) {
                                auto weigh = [&](auto near) {
#pragma unroll
                                    for (int e = 0; e < 8; ++e) {
                                        const float2 xe = make_float2(x[cc & 1][2 * e], x[cc & 1][2 * e + 1]);
                                        float2 wv;
                                        if (EXACT) wv = decltype(near)::value ? angular_weight2_near(xe) : angular_weight2(xe);
                                        if (SPARSE) {
                                            float2 a;
                                            if (EXACT) {
                                                a = exponent2(xe, ebias);
                                            } else {
                                                wv = ffma2(xe, dup2(kInvPi), dup2(0.5f));   // 1/2 + x / pi
                                                a = ffma2(xe, dup2(kLog2e), dup2(ebias));
                                            }
                                            const float2 p = make_float2(exp2_approx(a.x), exp2_approx(a.y));
                                            // masked by a factor of 1 or 0: a pair takes three instructions, a predicate and an addition each four
                                            wv = ffma2(p, make_float2(one_if_greater(p.x, prm.sparse_eps), one_if_greater(p.y, prm.sparse_eps)), wv);
                                        }
                                        o[e] = pack_bf16x2(wv.x, wv.y);
                                    }
                                };
                                weigh(near_form);
                            } else {
#pragma unroll
                                for (int e = 0; e < 8; ++e) o[e] = 0u;   // keys beyond the plane: finite, times v = 0
                            }
                            if (kNear && cc < 2) tmem_ld16(cb + (cc + 2) * 16, x[cc]);
                            tmem_st8(cb + cc * 8, o);   // over cosines that this thread has already read
                        }
                    };
                    if constexpr (kNear) {
                        // the tile's cosines are looked through first; those of the first two steps stay
                        float m = 0.f, n = 0.f;   // NaN goes the general way
                        if (unseen == 0) {
                            tmem_ld16(cb + 32, x[0]);
                            tmem_ld16(cb + 48, x[1]);
                            tmem_ld_wait();
#pragma unroll
                            for (int e = 0; e < 16; e += 2) {
                                m = max3_abs(m, x[0][e], x[0][e + 1]);
                                n = max3_abs(n, x[1][e], x[1][e + 1]);
                            }
                        }
                        tmem_ld16(cb, x[0]);
                        tmem_ld16(cb + 16, x[1]);
                        tmem_ld_wait();
                        bool near = false;
                        if (unseen == 0) {
#pragma unroll
                            for (int e = 0; e < 16; e += 2) {
                                m = max3_abs(m, x[0][e], x[0][e + 1]);
                                n = max3_abs(n, x[1][e], x[1][e + 1]);
                            }
                            near = __all_sync(0xffffffffu, max3_abs(m, n, 0.f) <= kNearLimit);
                            if (!near) unseen = kLookAgain;
                        }
                        if (near) {
                            tile(std::true_type{});
                        } else {
                            --unseen;
                            tile(std::false_type{});
                        }
                    } else {
                        tmem_ld16(cb, x[0]);
                        tile(std::false_type{});
                    }
                    tmem_st_wait();
                    tcgen05_fence_before_sync();
                }
                warp_arrive(&p_full[b]);
                if (jt < T - 1) skip(im.slots);
            }
            skip(im.slots - slot);   // to the first step of the next item
        }
    } else {
        // ---- convolution of the item's queries, then their output rows ----
        const int cw = warp - 24, slot = cw >> 2, quarter = warp & 3;
        constexpr int NIN = KS + 1;       // columns of V that two output columns need
        uint32_t* w_s = reinterpret_cast<uint32_t*>(smem + kOffW) + lane;
        float2 wreg[9];                   // 3 x 3: the filters in registers
        float2 bias2 = dup2(0.f);
        int prev_head = -1, o_uses = 0, patch = 0;
        bool ok = true;
        const int W = prm.gridW;
        for (int i = 0; i < my_items; ++i) {
            const Item im = item_of(i);
            const int head = (prm.head0 + im.bh) % prm.H;
            if (head != prev_head) {
                prev_head = head;
                const unsigned short* w0 = reinterpret_cast<const unsigned short*>(prm.w) + (size_t)(head * kD + 2 * lane) * (KS * KS);
                for (int e = cw; e < KS * KS; e += kConvThreads / 32) {
                    const int tap = GRID == kOneRow && prm.column ? e % KS * KS + e / KS : e;
                    w_s[e * 32] = (uint32_t)__ldg(w0 + tap) | ((uint32_t)__ldg(w0 + KS * KS + tap) << 16);
                }
                if (prm.bias) {   // element by element, like the filters: neither need begin on a word boundary
                    const unsigned short* b0 = reinterpret_cast<const unsigned short*>(prm.bias) + head * kD + 2 * lane;
                    bias2 = make_float2(bf16lo(__ldg(b0)), bf16lo(__ldg(b0 + 1)));
                }
                named_barrier_sync(1, kConvThreads);
                if (KS == 3) {
#pragma unroll
                    for (int e = 0; e < 9; ++e) { const uint32_t fw = w_s[e * 32]; wreg[e] = make_float2(bf16lo(fw), bf16hi(fw)); }
                }
            }
            const Patches pa = patches_of(im);
            for (int pj = 0; pj < pa.n; ++pj, ++patch) {
                ok = ok && warp_wait(patch_full, patch & 1);
                if (!ok) break;
                // two columns slide down the patch; the words of a row are loaded a row ahead
                const int py = GRID == kOrdinary ? pj / pa.nx : 0, y0 = pa.y0 + py * kPatchY;
                const int x0 = (GRID == kOrdinary ? pj - py * pa.nx : wide_column(im, pa, pj)) * kPatchX + 2 * cw;
                const uint8_t* vh = smem + kOffPatch + 2 * cw * 128 + lane * 4;
                int tl = y0 * W + x0 - im.t0;          // token of the first output, within the item
                uint32_t raw[NIN];
                float2 acc[KS][2];                     // output row y in slot y % KS
#pragma unroll
                for (int o = 0; o < NIN; ++o) raw[o] = lds32(vh + o * 128);
#pragma unroll
                for (int hy = 0; hy < HY; ++hy) {
                    float2 in[NIN];
#pragma unroll
                    for (int o = 0; o < NIN; ++o) in[o] = make_float2(bf16lo(raw[o]), bf16hi(raw[o]));
                    if (hy + 1 < HY) {
#pragma unroll
                        for (int o = 0; o < NIN; ++o) raw[o] = lds32(vh + ((hy + 1) * HX + o) * 128);
                    }
                    if (hy < kPatchY) acc[hy % KS][0] = acc[hy % KS][1] = bias2;
#pragma unroll
                    for (int dx = 0; dx < KS; ++dx)
#pragma unroll
                        for (int dy = 0; dy < KS; ++dy) {
                            const int y = hy - dy;     // compile-time after unrolling
                            if (y < 0 || y >= kPatchY) continue;
                            float2 f;
                            if (KS == 3) f = wreg[(dy * KS + dx) % 9];
                            else { const uint32_t fw = w_s[(dy * KS + dx) * 32]; f = make_float2(bf16lo(fw), bf16hi(fw)); }
#pragma unroll
                            for (int c = 0; c < 2; ++c) acc[y % KS][c] = ffma2(f, in[c + dx], acc[y % KS][c]);
                        }
                    if (hy >= KS - 1) {
                        const int y = hy - (KS - 1);
#pragma unroll
                        for (int c = 0; c < 2; ++c)    // rows beyond the plane are beyond its last token
                            if (x0 + c < W && (unsigned)(tl + c) < 2u * kTile)
                                *reinterpret_cast<float2*>(stg + (tl + c) * kStgStride + lane * 8) = acc[y % KS][c];
                        tl += W;
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(patch_free);
            }
            named_barrier_sync(1, kConvThreads);   // the item's convolution is in shared memory
            if (slot < im.slots) {
                ok = ok && warp_wait(&o_full[slot], o_uses & 1);
                ++o_uses;
                if (ok) {
                    tcgen05_fence_after_sync();
                    const uint32_t o_base = tmem + ((uint32_t)(quarter * 32) << 16) + kColO + slot * kD;
                    uint8_t* srow = stg + (slot * kTile + quarter * 32 + lane) * kStgStride;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {   // 16 channels: fp32 read at 64 c, bf16 written behind it at 32 c
                        float a[16];
                        tmem_ld16(o_base + c * 16, a);
                        tmem_ld_wait();
                        uint4 pk[2];
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            const float4 s0 = *reinterpret_cast<const float4*>(srow + c * 64 + hf * 32);
                            const float4 s1 = *reinterpret_cast<const float4*>(srow + c * 64 + hf * 32 + 16);
                            pk[hf].x = pack_bf16x2(a[8 * hf + 0] + s0.x, a[8 * hf + 1] + s0.y);
                            pk[hf].y = pack_bf16x2(a[8 * hf + 2] + s0.z, a[8 * hf + 3] + s0.w);
                            pk[hf].z = pack_bf16x2(a[8 * hf + 4] + s1.x, a[8 * hf + 5] + s1.y);
                            pk[hf].w = pack_bf16x2(a[8 * hf + 6] + s1.z, a[8 * hf + 7] + s1.w);
                        }
                        *reinterpret_cast<uint4*>(srow + c * 32) = pk[0];
                        *reinterpret_cast<uint4*>(srow + c * 32 + 16) = pk[1];
                    }
                    tcgen05_fence_before_sync();
                    warp_arrive(&o_free[slot]);
                    __syncwarp();
                    __nv_bfloat16* op = prm.out + plane_offset(prm.lo, im.bh, prm.hdiv) + (lane & 7) * 8;
#pragma unroll
                    for (int it = 0; it < 8; ++it) {   // four whole 128-byte rows per instruction
                        const int r = slot * kTile + quarter * 32 + it * 4 + (lane >> 3);
                        const uint4 val = *reinterpret_cast<const uint4*>(stg + r * kStgStride + (lane & 7) * 16);
                        if (im.t0 + r < N) *reinterpret_cast<uint4*>(op + (long long)(im.t0 + r) * prm.lo.token) = val;
                    }
                }
            }
            named_barrier_sync(1, kConvThreads);   // the staging rows may be overwritten
        }
    }
    tcgen05_fence_before_sync();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

template <int KS, bool SPARSE, bool EXACT, int GRID>
cudaError_t launch_quad_grid(const Problem& p, int gridH, int gridW, int slots, unsigned* status, cudaStream_t st) {
    CUtensorMap tmQ, tmK, tmV, tmP;
    const uint64_t nb = (uint64_t)(p.BH / p.hdiv);
    const uint64_t dims[4] = {(uint64_t)kD, (uint64_t)p.N, (uint64_t)p.hdiv, nb};
    const uint32_t box[4] = {kD, kTile, 1, 1};
    auto strides = [&](const Layout& l, uint64_t (&s)[3]) {
        s[0] = (uint64_t)l.token; s[1] = (uint64_t)l.head; s[2] = (uint64_t)(nb > 1 ? l.batch : l.head * p.hdiv);
    };
    uint64_t sq[3], sk[3], sv[3];
    strides(p.lq, sq); strides(p.lk, sk); strides(p.lv, sv);
    if (!make_tensor_map_bf16(&tmQ, p.q, 4, dims, sq, box, 128) || !make_tensor_map_bf16(&tmK, p.k, 4, dims, sk, box, 128) ||
        !make_tensor_map_bf16(&tmV, p.v, 4, dims, sv, box, 128))
        return cudaErrorNotSupported;
    // [64, columns, grid rows, planes per batch step, batch steps]: columns and rows outside the grid are zero-filled
    const uint64_t dims_p[5] = {(uint64_t)kD, (uint64_t)gridW, (uint64_t)gridH, (uint64_t)p.hdiv, nb};
    const uint64_t strides_p[4] = {(uint64_t)p.lv.token, (uint64_t)(p.lv.token * gridW), sv[1], sv[2]};
    const uint32_t box_p[5] = {kD, kPatchX + 2 * (KS / 2), (GRID == kOneRow ? 1 : KS == 3 ? 8 : 4) + 2 * (KS / 2), 1, 1};
    if (!make_tensor_map_bf16(&tmP, p.v, 5, dims_p, strides_p, box_p, 0)) return cudaErrorNotSupported;
    QuadParams prm;
    prm.out = static_cast<__nv_bfloat16*>(p.out);
    prm.w = static_cast<const __nv_bfloat16*>(p.w);
    prm.bias = static_cast<const __nv_bfloat16*>(p.bias);
    prm.lo = p.lo;
    prm.hdiv = p.hdiv; prm.H = p.H; prm.head0 = p.head0; prm.N = p.N;
    prm.gridH = gridH; prm.gridW = gridW; prm.column = gridW != p.gridW ? 1 : 0;
    const int sms = device_sm_count(), q_tiles = (p.N + kTile - 1) / kTile;
    prm.slots = slots;
    prm.groups = (q_tiles + prm.slots - 1) / prm.slots;
    prm.k_tiles = q_tiles;
    prm.n_items = p.BH * prm.groups;
    prm.eps2 = p.eps2; prm.status = status;
    prm.sparse_eps = p.sparse_eps;
    static PerDevice opt_in;
    {
        const cudaError_t e = opt_in_smem(tc_quad_kernel<KS, SPARSE, EXACT, GRID>, kSmem, opt_in);
        if (e != cudaSuccess) return e;
    }
    const int grid = prm.n_items < sms ? prm.n_items : sms;
    return launch_programmatic(tc_quad_kernel<KS, SPARSE, EXACT, GRID>, true, dim3((unsigned)grid), dim3(kThreads), kSmem, st, tmQ, tmK, tmV, tmP, prm);
}

template <int KS, bool SPARSE, bool EXACT>
cudaError_t launch_quad_ks(const Problem& p, unsigned* status, cudaStream_t st) {
    // Two query tiles per item share the key tiles and keep both halves of the weight warps busy; an item of one tile takes
    // 0.7 (exact kernel) to 0.85 of its time: one tile each where that leaves (nearly) as few rounds.  Over 26 shapes of 1 to 768
    // planes and 128 to 4096 tokens this is the faster one with either kernel; closest to the line, one tile against two: exact, 24
    // planes of 32 x 64 (3 rounds / 2) 77.4 / 74.4 us, 16 of 32 x 32 (1 / 1) 18.3 / 23.9; masked, 192 planes of 14 x 14 (3 / 2)
    // 29.2 / 23.6, 48 of 14 x 14 (1 / 1) 12.0 / 14.7.
    const int sms = device_sm_count();
    const int q_tiles = (p.N + kTile - 1) / kTile;
    const long long one = (long long)p.BH * q_tiles, two = (long long)p.BH * ((q_tiles + 1) / 2);
    const int slots = ((one + sms - 1) / sms) * 3 < ((two + sms - 1) / sms) * 4 ? 1 : 2;
    const bool column = p.gridW == 1 && p.gridH > 1;
    const int gridH = column ? 1 : p.gridH, gridW = column ? p.gridH : p.gridW;
    if (gridH == 1) return launch_quad_grid<KS, SPARSE, EXACT, kOneRow>(p, gridH, gridW, slots, status, st);
    if (gridW > slots * kTile) return launch_quad_grid<KS, SPARSE, EXACT, kWide>(p, gridH, gridW, slots, status, st);
    return launch_quad_grid<KS, SPARSE, EXACT, kOrdinary>(p, gridH, gridW, slots, status, st);
}

}  // namespace

// bf16, head width 64 (16-byte aligned token rows), 3x3 or 5x5 filters, explicit weights (exact kernel and / or the
// masked softmax branch) without row-sum division, no leading tokens.
bool quad_supports(const Problem& p) {
    return p.bf16 && p.d == kD && (p.ksize == 3 || p.ksize == 5) && (p.exact_kernel || p.sparse) && !p.rownorm &&
           p.prefix == 0 && !p.blockdiag && (p.lv.token % 8) == 0 && (p.lo.token % 8) == 0;
}

cudaError_t launch_quad(const Problem& p, unsigned* status, cudaStream_t st) {
    if (p.sparse && p.exact_kernel)
        return p.ksize == 3 ? launch_quad_ks<3, true, true>(p, status, st) : launch_quad_ks<5, true, true>(p, status, st);
    if (p.sparse)
        return p.ksize == 3 ? launch_quad_ks<3, true, false>(p, status, st) : launch_quad_ks<5, true, false>(p, status, st);
    return p.ksize == 3 ? launch_quad_ks<3, false, true>(p, status, st) : launch_quad_ks<5, false, true>(p, status, st);
}

}  // namespace tc
}  // namespace castling
