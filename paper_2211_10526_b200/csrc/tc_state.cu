// State kernel of the tensor-core path (bf16, d = 64; d = 32: NARROW below): per (b,h) and token split,
//     S = sum_n k^_n^T v_n  (64 x 64)   and   s = sum_n v_n  (64)            (Eq. 9)
// as one tcgen05 contraction over tokens.  Per 128-token stage TMA brings the K and V tiles
// into 128-byte-swizzled shared memory; four warps scale every K row by 1 / max(||k||, eps) in
// place (the scale sits on the contracted index, so it cannot wait for an epilogue); one thread
// issues UMMAs with A = [K^ ; 1 0 0 ...] (128 x tokens, M-major: rows 0..63 are the key
// features, row 64 is all ones, which makes row 64 of the accumulator the token sum of V) and
// B = V (tokens x 64, N-major).  The fp32 accumulator lives in TMEM for the CTA's whole token
// range and is written once, as this split's partial state.
// RN (row-sum normalisation, Eq. 3's denominator on the kept kernel of Eq. 8) also needs sum_n k^_n: B gets a
// second 64-wide block along N from the same constant block ([V | 1 0 0 ...]), so column 64 of the accumulator is
// the row sum of A: rows 0..63 of it are sum_n k^_n, and the state has 64 more words.
#include "tc_common.cuh"
#include "tc_host.cuh"

namespace castling {
namespace tc {
namespace {

constexpr int kD = 64;
constexpr int kTile = 128;                   // 128-byte rows per stage
constexpr int kThreadRows = 128;             // normalising threads: one 128-byte row of a stage each
constexpr int kStages = 3;                  // 3 x 32 KiB: two CTAs fit on one SM
constexpr int kTileBytes = kTile * kD * 2;   // 16 KiB per operand tile
constexpr int kStageBytes = 2 * kTileBytes;  // K then V
constexpr int kOnesBytes = 2048;             // 16 token rows x 128 B: feature 64 = 1, 65..127 = 0
constexpr int kThreads = 192;                // warp 0 TMA, warp 1 UMMA, warps 2..5 scale + epilogue
constexpr int kTmemCols = 128;                // two 64-column accumulators: a CTA may serve several (b,h) (RN: twice that)
constexpr int kGroup = 4;                    // splits per first-level reduction group
constexpr int kFineStages = 2, kFineStageBytes = kStageBytes + kTileBytes;   // K, V, the rest of K
constexpr int kStagesBytes = kStages * kStageBytes;
static_assert(kFineStages * kFineStageBytes == kStagesBytes, "one size of shared memory");
constexpr size_t kSmemBytes = 1024 + kStagesBytes + kOnesBytes + 256;

// Rows are scaled in fp32, with one rounding to bf16; the factor as two bf16, packed bf16 operations, rounds one element in 1 300 another way and gains
// 0.1 us.  Sums and products in pairs and a refined reciprocal root instead of a root and a quotient, us per forward from a graph: 16 planes of 64 x 64
// 18.2 -> 17.9, of 128 x 128 42.9 -> 42.3, 64 of 50 x 75, width 32, 33.4 -> 33.1.
// NARROW serves width-32 heads: rows of 64 bytes, 64-byte swizzle, 256 tokens per stage (any grid width, any number of
// tokens), UMMAs of M = 64 (32 key features, then the row of ones) and N = 32, states of 32 x 32 + 32 words.  Two tokens
// packed to a 128-byte row instead, which wastes half of the contraction and needs an even grid width, took 19.8 us against
// 17.6 us (8 x 8 planes of 64 x 64 tokens).
// FINE (NARROW only): the unit keys are kept as two bf16, the value and what rounding it left off, and contracted one after the
// other, so that the state is as precise as one from fp32 keys; the second tile of K takes the place of a stage.
template <bool NARROW, bool RN, bool FINE>
__global__ void __launch_bounds__(kThreads, 2)
tc_state_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                float* __restrict__ dst, float* __restrict__ final_state, unsigned* __restrict__ counters,
                int N, int tiles_per_cta, int P, int clustered, int BH, int hdiv, int items_per_cta, float eps2, unsigned* status) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = align_smem(smem_raw);
    constexpr int kStages = FINE ? kFineStages : castling::tc::kStages, kStageBytes = FINE ? kFineStageBytes : castling::tc::kStageBytes;
    uint8_t* ones = smem + kStagesBytes;
    uint64_t* full = reinterpret_cast<uint64_t*>(ones + kOnesBytes);  // TMA bytes landed
    uint64_t* scaled = full + kStages;                                // K rows normalised (128 arrivals)
    uint64_t* empty = scaled + kStages;                               // UMMAs of the stage retired
    uint64_t* accum = empty + kStages;                                // [2] whole accumulation of an item retired
    uint64_t* acc_free = accum + 2;                                   // [2] accumulator read out (128 arrivals)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_free + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    constexpr int kW = NARROW ? 32 : kD;                   // width of the contraction's operands
    constexpr int kTok = NARROW ? 2 * kTile : kTile;       // rows (of kW elements) per stage
    constexpr int kAcc = RN ? 2 * kW : kW;                 // accumulator columns
    constexpr int kStateW = kW * kW + kW + (RN ? kW : 0);  // words of one state: S, s, (RN) sum of the unit key rows
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // Work items.  With P > 1 a CTA serves one (b,h, split).  With P == 1 (many heads, few tokens) a CTA
    // serves items_per_cta consecutive (b,h) one after another, so that barrier set-up, TMEM allocation
    // and the first load latency are paid once and the loads of the next (b,h) overlap the current one.
    const int total_tiles = (N + kTok - 1) / kTok;
    const int p = (P > 1) ? blockIdx.x % P : 0;
    const int bh0 = (P > 1) ? blockIdx.x / P : blockIdx.x * items_per_cta;
    const int n_items = (P > 1) ? 1 : min(items_per_cta, BH - bh0);
    const int t_begin = p * tiles_per_cta;
    const int n_tiles = min(total_tiles, t_begin + tiles_per_cta) - t_begin;  // per item, at least one
    const int bh = bh0;  // the (b,h) of the split reduction below (P > 1: the only item)
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&scaled[s], kThreadRows);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) { mbar_init(&accum[b], 1); mbar_init(&acc_free[b], kThreadRows); }
        *abort_flag = 0;
        mbar_fence_init();
        tma_prefetch_desc(&tmK);
        tma_prefetch_desc(&tmV);
    }
    if (warp == 1) tmem_alloc(tmem_slot, RN ? 2 * kTmemCols : kTmemCols);
    if (warp >= 2) {
        // constant block of A: for each of 16 token rows, element 64 (first of the second 64-wide
        // block along M) is 1.0 and the rest 0; 16-byte chunk c of row r sits at chunk c ^ (r & 7)
        // (rows of 64 bytes: element 32, chunk c of row r at chunk c ^ ((r >> 1) & 3), half as many threads; FINE: the other
        // half of the place is a block of zeros, which goes with the rest of K)
        const int t = tid - 64;  // 0..127 -> one 16-byte chunk each
        const int r = NARROW ? t >> 2 : t >> 3, c = NARROW ? t & 3 : t & 7;
        uint4 val = make_uint4(0, 0, 0, 0);
        if ((c ^ (NARROW ? (r >> 1) & 3 : r & 7)) == 0) val.x = 0x3f80u;  // logical chunk 0: bf16 1.0 in its first element
        if (NARROW && r >= 16) val.x = 0u;
        if (!NARROW || FINE || r < 16) *reinterpret_cast<uint4*>(ones + t * 16) = val;
        fence_proxy_async_smem();
    }
    tcgen05_fence_before_sync();
    __syncthreads();
    tcgen05_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    // Launched programmatically dependent on the kernel before it in the stream (which may let its dependents start long before it
    // ends): everything above ran while that kernel drained.  Every thread waits for it here; the limits of the waits below are for this
    // kernel's own work.  Global memory is first touched after this.
    pdl_wait_primary();

    if (warp == 0) {
        if (lane == 0) {
            int issued = 0;
            // Both tensors stream through L2 once here.  V is read again by the apply kernel, but at long sequences it
            // does not survive until then whatever the hint, and lines marked evict-last pile up and slow the streams
            // of both kernels (measured: 132 -> 125 us per forward at 2 x 8 planes of 256 x 256 tokens).
            const uint64_t pol_k = l2_policy_evict_first(), pol_v = l2_policy_evict_first();
            bool ok = true;
            // Only now may the apply kernel begin its prologue: it loads Q and V, which may be the output of the kernel
            // this grid has just waited for, as soon as it runs.
            pdl_launch_dependents();
            for (int item = 0; item < n_items && ok; ++item) {
                for (int it = 0; it < n_tiles; ++it, ++issued) {
                    const int s = issued % kStages, use = issued / kStages;
                    if (use > 0 && !mbar_wait(&empty[s], (use - 1) & 1, abort_flag, status, kStatusStateTimeout)) { ok = false; break; }
                    uint8_t* ks = smem + s * kStageBytes;
                    mbar_expect_tx(&full[s], 2 * kTileBytes);
                    const int plane = bh0 + item, pb = plane / hdiv, ph = plane - pb * hdiv;
                    tma_load_4d_hint(ks, &tmK, &full[s], 0, (t_begin + it) * kTok, ph, pb, pol_k);
                    tma_load_4d_hint(ks + kTileBytes, &tmV, &full[s], 0, (t_begin + it) * kTok, ph, pb, pol_v);
                }
            }
            if (*abort_flag) {
                // giving up: let copies already in flight land before the CTA's shared memory goes away
                for (int i = max(0, issued - kStages); i < issued; ++i)
                    for (int spin = 0; spin < (1 << 20) && !mbar_try_wait(&full[i % kStages], (i / kStages) & 1); ++spin) {}
            }
        }
    } else if (warp == 1) {
        // the whole warp walks through the tiles, one elected lane issues
        constexpr uint32_t idesc = umma_idesc_bf16(NARROW ? 64 : 128, kAcc, true, true);
        const uint32_t ones_addr = smem_u32(ones);
        // A: 128 bytes of K per token and, lbo bytes on, the constant block; stepping to the next 16 tokens adds to the
        // address and takes the same off the distance
        constexpr uint32_t kStepB = (16u * kW * 2) >> 4, kStep = kStepB - (kStepB << 16);
        bool ok = true;
        int s = 0;
        uint32_t par = 0;
        for (int item = 0; item < n_items && ok; ++item) {
            const int buf = item & 1;
            if (item >= 2) ok = mbar_wait_warp(&acc_free[buf], ((item >> 1) - 1) & 1, abort_flag, status, kStatusStateTimeout);
            for (int it = 0; it < n_tiles && ok; ++it) {
                ok = mbar_wait_warp(&scaled[s], par, abort_flag, status, kStatusStateTimeout);
                if (!ok) break;
                tcgen05_fence_after_sync();
                if (elect_one()) {
                    const uint32_t ka = smem_u32(smem + s * kStageBytes), va = ka + kTileBytes;
                    const uint32_t a = desc_low(ka, ones_addr - ka), b = desc_low(va, RN ? ones_addr - va : 0);
                    const uint32_t rest = FINE ? desc_low(va + kTileBytes, ones_addr + kOnesBytes / 2 - (va + kTileBytes)) : 0;
#pragma unroll
                    for (int j = 0; j < kTok / 16; ++j) {  // one UMMA per 16 tokens (K = 16)
                        umma_bf16_low<NARROW ? kDescHigh64 : kDescHigh>(tmem + buf * kAcc, a + j * kStep,
                                                                        b + j * (RN ? kStep : kStepB), idesc, (it | j) != 0);
                        if (FINE) umma_bf16_low<kDescHigh64>(tmem + buf * kAcc, rest + j * kStep, b + j * (RN ? kStep : kStepB), idesc, 1u);
                    }
                    umma_commit(&empty[s]);
                    if (it == n_tiles - 1) umma_commit(&accum[buf]);
                }
                __syncwarp();
                if (++s == kStages) { s = 0; par ^= 1; }
            }
        }
    } else {
        const int t = tid - 64;  // 128-byte row of the stage handled by this thread
        const int quarter = warp & 3;
        bool ok = true;
        // read the finished accumulator of `item` out of TMEM: rows 0..63 are S, row 64 is s; a warp reads
        // TMEM lanes 32*(warp%4)..+31.  Runs one item late, so that the UMMAs of an item overlap the
        // normalisation of the next item's tiles.
        auto flush = [&](int item) -> bool {
            const int buf = item & 1;
            if (!mbar_wait_warp(&accum[buf], (item >> 1) & 1, abort_flag, status, kStatusStateTimeout)) return false;
            tcgen05_fence_after_sync();
            if (quarter < 3) {
                // a cluster's partial state stays in shared memory, over the stages, which the UMMAs have read
                float* out = clustered ? reinterpret_cast<float*>(smem) : dst + ((size_t)(bh0 + item) * P + p) * kStateW;
                // M = 64 keeps rows 16 q .. 16 q + 15 in lanes 32 q .. 32 q + 15
                const int row = NARROW ? (lane < 16 ? quarter * 16 + lane : kW + 1) : quarter * 32 + lane;
#pragma unroll
                for (int cc = 0; cc < kW / 16; ++cc) {
                    float v[16];
                    tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + buf * kAcc + cc * 16, v);
                    tmem_ld_wait();
                    if (row <= kW) {
                        float4* o4 = reinterpret_cast<float4*>(out + row * kW + cc * 16);  // row kW lands on s
#pragma unroll
                        for (int e = 0; e < 4; ++e) o4[e] = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
                    }
                }
                if (RN) {  // column kW: the row sums of A; rows 0..kW - 1 are sum_n k^_n, stored behind s
                    float v[16];
                    tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + buf * kAcc + kW, v);
                    tmem_ld_wait();
                    if (row < kW) out[kW * kW + kW + row] = v[0];
                }
            }
            tcgen05_fence_before_sync();
            mbar_arrive(&acc_free[buf]);
            return true;
        };
        int gt = 0;  // tiles handled so far, over all items
        for (int item = 0; item < n_items && ok; ++item) {
            for (int it = 0; it < n_tiles; ++it, ++gt) {
                const int s = gt % kStages, use = gt / kStages;
                ok = mbar_wait_warp(&full[s], use & 1, abort_flag, status, kStatusStateTimeout);   // as a whole: flush() reads tensor memory
                if (!ok) break;
                // NARROW: the 128 bytes are tokens 2 t and 2 t + 1, whose chunk c sits at chunk c ^ (t & 3) of their half; the
                // same walk over the eight chunks as for a 128-byte swizzle meets all chunks of one of them first
                uint8_t* row = smem + s * kStageBytes + t * 128;
                uint4 c[8];
                const float2 zero2 = make_float2(0.f, 0.f);
                float2 sq[4] = {zero2, zero2, zero2, zero2};   // first / second half of the 128 bytes
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    c[j] = *reinterpret_cast<const uint4*>(row + ((j ^ (t & 7)) << 4));
                    const uint32_t w[4] = {c[j].x, c[j].y, c[j].z, c[j].w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 x = make_float2(bf16lo(w[e]), bf16hi(w[e]));
                        sq[2 * (j >> 2) + (e & 1)] = ffma2(x, x, sq[2 * (j >> 2) + (e & 1)]);
                    }
                }
                const float ssa = (sq[0].x + sq[0].y) + (sq[1].x + sq[1].y), ssb = (sq[2].x + sq[2].y) + (sq[3].x + sq[3].y);
                const float rka = inv_sqrt(fmaxf(NARROW ? ssa : ssa + ssb, eps2)), rkb = NARROW ? inv_sqrt(fmaxf(ssb, eps2)) : rka;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float rk = j < 4 ? rka : rkb;
                    auto times_rk = [&](uint32_t w) {
                        const float2 x = ffma2(make_float2(bf16lo(w), bf16hi(w)), make_float2(rk, rk), zero2);
                        return pack_bf16x2(x.x, x.y);
                    };
                    const uint4 o = make_uint4(times_rk(c[j].x), times_rk(c[j].y), times_rk(c[j].z), times_rk(c[j].w));
                    *reinterpret_cast<uint4*>(row + ((j ^ (t & 7)) << 4)) = o;
                    if (FINE) *reinterpret_cast<uint4*>(row + 2 * kTileBytes + ((j ^ (t & 7)) << 4)) =
                        make_uint4(rest_bf16x2(c[j].x, rk, o.x), rest_bf16x2(c[j].y, rk, o.y), rest_bf16x2(c[j].z, rk, o.z), rest_bf16x2(c[j].w, rk, o.w));
                }
                fence_proxy_async_smem();
                mbar_arrive(&scaled[s]);
            }
            if (ok && item > 0) ok = flush(item - 1);
        }
        if (ok) ok = flush(n_items - 1);
    }
    tcgen05_fence_before_sync();
    __syncthreads();  // every thread's part of this split's partial state has been stored
    if (warp == 1) tmem_dealloc(tmem, RN ? 2 * kTmemCols : kTmemCols);

    if (clustered) {   // the splits of a (b,h) are one cluster: each CTA adds its share of the words, in the splits' order
        constexpr int kWords4 = kStateW / 4;
        const int share = (kWords4 + P - 1) / P, end = min(kWords4, (p + 1) * share);
        cluster_arrive();
        cluster_wait();
        for (int i = p * share + tid; i < end; i += kThreads) {
            const float4* at = reinterpret_cast<const float4*>(smem) + i;
            float4 sum = ld_peer(at, 0);
            for (int m = 1; m < P; ++m) {
                const float4 x = ld_peer(at, m);
                sum.x += x.x; sum.y += x.y; sum.z += x.z; sum.w += x.w;
            }
            reinterpret_cast<float4*>(final_state + (size_t)bh * kStateW)[i] = sum;
        }
        cluster_arrive();   // this partial state has been read
        cluster_wait();
        return;
    }

    // Cross-split reduction without a second launch and without any waiting, as a two-level tree
    // driven by arrival counters: the splits of a (b,h) form groups of kGroup; the CTA that arrives
    // last in its group sums the group's partial states in index order into the group's first slot,
    // then the group that arrives last sums the group results in index order into the final state.
    // The order of the additions is fixed, so the result does not depend on which CTAs came last.
    // Every counter is put back to zero by the CTA that consumed it.
    if (P > 1 && !*abort_flag) {
        __shared__ int is_last;
        constexpr int kWords = kStateW, kWords4 = kWords / 4, kIter = (kWords4 + kThreads - 1) / kThreads;
        unsigned* cnt = counters + (size_t)bh * kCountersPerHead;
        const int n_groups = (P + kGroup - 1) / kGroup, grp = p / kGroup;
        const int first = grp * kGroup, members = min(kGroup, P - first);
        float4* base = reinterpret_cast<float4*>(dst + (size_t)bh * P * kWords);
        // One thread publishes for the CTA: its device-wide fence after the CTA barrier covers the stores the other
        // threads made before that barrier; its fence after the atomic, followed by a CTA barrier, lets every thread
        // read what the other CTAs of the group published the same way.
        if (tid == 0) {
            __threadfence();
            is_last = (atomicAdd(&cnt[grp], 1u) == (unsigned)(members - 1));
            __threadfence();
        }
        __syncthreads();
        if (!is_last) return;
        // a single group (at most kGroup splits): its sum is the final state, no second level
        float4* fin = reinterpret_cast<float4*>(final_state + (size_t)bh * kWords);
        float4* level1 = (n_groups == 1) ? fin : base + (size_t)first * kWords4;
        if (members > 1) {
            float4 acc[kIter];
#pragma unroll
            for (int j = 0; j < kIter; ++j) {
                const int i = tid + j * kThreads;
                if (i < kWords4) acc[j] = __ldcg(base + (size_t)first * kWords4 + i);
            }
            // every load of the group is issued before the first addition (one trip to L2, not one per member);
            // the additions keep the members' order
            float4 v[kGroup - 1][kIter];
#pragma unroll
            for (int m = 1; m < kGroup; ++m)
#pragma unroll
                for (int j = 0; j < kIter; ++j) {
                    const int i = tid + j * kThreads;
                    v[m - 1][j] = (m < members && i < kWords4) ? __ldcg(base + (size_t)(first + m) * kWords4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
            for (int m = 1; m < kGroup; ++m)
#pragma unroll
                for (int j = 0; j < kIter; ++j) {
                    if (m < members) { acc[j].x += v[m - 1][j].x; acc[j].y += v[m - 1][j].y; acc[j].z += v[m - 1][j].z; acc[j].w += v[m - 1][j].w; }
                }
#pragma unroll
            for (int j = 0; j < kIter; ++j) {
                const int i = tid + j * kThreads;
                if (i < kWords4) level1[i] = acc[j];
            }
        }
        if (n_groups == 1) {
            if (tid == 0) cnt[grp] = 0;
            return;
        }
        __syncthreads();
        if (tid == 0) {
            cnt[grp] = 0;
            __threadfence();
            is_last = (atomicAdd(&cnt[kCountersPerHead - 1], 1u) == (unsigned)(n_groups - 1));
            __threadfence();
        }
        __syncthreads();
        if (!is_last) return;
        float4 acc[kIter];
#pragma unroll
        for (int j = 0; j < kIter; ++j) {
            const int i = tid + j * kThreads;
            if (i < kWords4) acc[j] = __ldcg(base + i);
        }
        for (int g0 = 1; g0 < n_groups; g0 += 4) {  // four groups per trip to L2, added in the groups' order
            float4 v[4][kIter];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int j = 0; j < kIter; ++j) {
                    const int i = tid + j * kThreads;
                    v[u][j] = (g0 + u < n_groups && i < kWords4) ? __ldcg(base + (size_t)(g0 + u) * kGroup * kWords4 + i)
                                                                  : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int j = 0; j < kIter; ++j) {
                    if (g0 + u < n_groups) { acc[j].x += v[u][j].x; acc[j].y += v[u][j].y; acc[j].z += v[u][j].z; acc[j].w += v[u][j].w; }
                }
        }
#pragma unroll
        for (int j = 0; j < kIter; ++j) {
            const int i = tid + j * kThreads;
            if (i < kWords4) fin[i] = acc[j];
        }
        if (tid == 0) cnt[kCountersPerHead - 1] = 0;
    }
}

}  // namespace

// What a state CTA takes of a multiprocessor but for tensor memory: asked about a kernel that allocates some, the runtime counts one CTA per
// multiprocessor, and two of the state kernel's run on each.  Never launched.
static __global__ void __launch_bounds__(kThreads, 2) footprint_kernel() {}

int state_clusters_at_once(int P) {
    static std::atomic<int> known[kMaxDevices][9];   // the number and one more
    static PerDevice opt_in;
    int dev = 0, n = 0;
    if (P < 1 || P > 8 || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { (void)cudaGetLastError(); return 0; }
    if ((n = known[dev][P].load(std::memory_order_relaxed)) > 0) return n - 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)P); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)P; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    if (opt_in_smem(footprint_kernel, kSmemBytes, opt_in) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, footprint_kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    known[dev][P].store(n + 1, std::memory_order_relaxed);
    return n;
}

cudaError_t launch_state(const Problem& p, float* partial, float* final_state, unsigned* counters, int P,
                         int tiles_per_cta, bool clustered, unsigned* status, cudaStream_t st) {
    const bool narrow = p.d == 32;
    const int stage = narrow ? 2 * kTile : kTile;   // tokens
    if (P > 1 && (P - 1) * tiles_per_cta >= (p.N + stage - 1) / stage) return cudaErrorInvalidValue;   // a split without tokens: the kernel takes none
    CUtensorMap tmK, tmV;
    // [row, tokens, planes per batch step, batch steps]
    const uint64_t nb = (uint64_t)(p.BH / p.hdiv);
    const uint32_t width = narrow ? 32 : kD;
    const uint64_t dims[4] = {width, (uint64_t)p.N, (uint64_t)p.hdiv, nb};
    const uint32_t box[4] = {width, narrow ? 2u * kTile : kTile, 1, 1};
    const uint64_t sk[3] = {(uint64_t)p.lk.token, (uint64_t)p.lk.head, (uint64_t)(nb > 1 ? p.lk.batch : p.lk.head * p.hdiv)};
    const uint64_t sv[3] = {(uint64_t)p.lv.token, (uint64_t)p.lv.head, (uint64_t)(nb > 1 ? p.lv.batch : p.lv.head * p.hdiv)};
    const int swizzle = narrow ? 64 : 128;
    if (!make_tensor_map_bf16(&tmK, p.k, 4, dims, sk, box, swizzle) || !make_tensor_map_bf16(&tmV, p.v, 4, dims, sv, box, swizzle))
        return cudaErrorNotSupported;
    static PerDevice opt_in[6];
    float* dst = P > 1 ? partial : final_state;
    // P == 1: a CTA serves several consecutive (b,h); at most two CTAs per multiprocessor so all are resident
    int grid = p.BH * P, items = 1;
    const int resident = 2 * device_sm_count();
    if (P == 1 && p.BH > resident) {
        items = (p.BH + resident - 1) / resident;
        grid = (p.BH + items - 1) / items;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = kSmemBytes; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)P; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = clustered ? 2 : 1;
    auto launch = [&](auto kernel) {
        const cudaError_t e = opt_in_smem(kernel, kSmemBytes, opt_in[(p.fine ? 4 : narrow ? 2 : 0) + (p.rownorm ? 1 : 0)]);
        if (e != cudaSuccess) return e;
        return cudaLaunchKernelEx(&cfg, kernel, tmK, tmV, dst, final_state, counters, p.N, tiles_per_cta, P, clustered ? 1 : 0, p.BH, p.hdiv, items,
                                  p.eps2, status);
    };
    if (p.fine) return p.rownorm ? launch(tc_state_kernel<true, true, true>) : launch(tc_state_kernel<true, false, true>);
    if (narrow) return p.rownorm ? launch(tc_state_kernel<true, true, false>) : launch(tc_state_kernel<true, false, false>);
    return p.rownorm ? launch(tc_state_kernel<false, true, false>) : launch(tc_state_kernel<false, false, false>);
}

}  // namespace tc
}  // namespace castling
