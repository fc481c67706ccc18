// Gradients of the loss with respect to the weights of the feature networks (Section 5, "Training Details": the phi
// maps are trained with the rest of the model).  For one map, with dp = dfeat (.) 1[feat > 0] (the feature gradients the
// backward left in the workspace, masked by the features the forward kept):
//   h   = X W1 + b1,  G = GELU(h),  dg = dp W2^T,  dh = dg (.) GELU'(h)        (recomputed exactly as in the phi backward)
//   dW2 = G^T dp,   db2 = sum_t dp,   dW1 = X^T dh,   db1 = sum_t dh          (sums over all tokens of all heads)
//
// Both weight gradients contract over the tokens, so neither operand can stay in TMEM (a TMEM operand has one token per
// lane): the 16 arithmetic warps write the G and dh tiles to shared memory, where X^T, G^T (A operands) and dh, dp (B
// operands) are all read token-major ("MN-major").  Every CTA serves ONE map: the maps of a side share the grid, a contiguous run of
// CTAs each, so that a side leaves one partial per CTA.  (With every CTA walking all maps of its side one after the other the partials
// of three key maps were 33 MB at d = 128: 159 -> 139 us for the four launches of a call at 12 heads x 12600 tokens.)  It keeps
//   dW1     [d x d]   accumulator lane = input index, column = hidden unit
//   dW2ext  [d x 64]  accumulator lane = hidden unit, columns 0..5 = G^T dp_hi, 6..11 = G^T dp_lo
// in TMEM and leaves one partial in the workspace; a second kernel adds a map's partials in CTA order, so the result is
// bit-reproducible.
//
// warp 0: TMA loads, warp 1: dg, dW1 and dW2 MMAs, warp 2: h MMAs, warps 3..18: arithmetic (thread = token row x quarter
// of the hidden units), warps 19..22: column sums of the dh tile (db1), warps 23..26: dp tiles and db2 (thread = token row;
// off the arithmetic warps' instruction stream, which is what bounds the kernel).
#pragma once
#include "hla_tc_phi.cuh"

namespace hla {
namespace tc {

constexpr int kWgThreads = 27 * 32;
constexpr int kWgEpiWarp0 = 3, kWgSumWarp0 = 19, kWgDpWarp0 = 23;
constexpr int kWgColDg = 128, kWgColW1 = 256, kWgColW2 = 384;      // TMEM columns (h at 0)

template <int DV, int DP> struct WgCfg {
    static constexpr int kXBytes = 2 * kBlk;                     // two 64-column blocks per stage (the second stays zero for d = 64)
    static constexpr int kW1Bytes = DV * DV * 2;
    static constexpr int kDgSteps = DP == 6 ? 1 : 2;             // K = 16 steps of the dg product: [dp_hi | dp_lo] is 2 DP columns wide
    static constexpr int kW2tBlock = kDgSteps * 2048;
    static constexpr int kW2tBytes = (DV / 64) * kW2tBlock;      // [16 kDgSteps K rows][DV] bf16 (W2^T twice, halved; row 12 of the last step: b1)
    static constexpr int kOffX = 0;                              // 2 stages
    static constexpr int kOffW1 = 2 * kXBytes;                   // the map's W1
    static constexpr int kOffDp = kOffW1 + kW1Bytes;             // 3 dp blocks [128 tok][64]: K columns 0..5 dp_hi, 6..11 dp_lo; column 44 of block 0 is 1
    static constexpr int kOffW2t = kOffDp + 3 * kBlk;
    static constexpr int kOffG = ((kOffW2t + kW2tBytes + 1023) / 1024) * 1024;   // G tile, two 64-column blocks
    static constexpr int kOffDh = kOffG + 2 * kBlk;              // dh tile
    static constexpr int kOffBars = kOffDh + 2 * kBlk;
    static constexpr int kSmemUsed = 1024 + kOffBars + 256;
    static_assert(kSmemUsed <= 227 * 1024, "shared memory");
    static constexpr int kSmem = kSmemUsed > 120 * 1024 ? kSmemUsed : 120 * 1024;   // one CTA per SM (512 TMEM columns)
    static constexpr int kB1Row = 12;
    // one partial per CTA, in floats: dW1 [DV][DV], dW2ext [DV][kW2Cols], db1 [DV], db2 [4 token quarters][16]
    static constexpr int kW2Cols = 16 * kDgSteps;
    static constexpr int kPartW2 = DV * DV, kPartB1 = kPartW2 + DV * kW2Cols, kPartB2 = kPartB1 + DV, kPartFloats = kPartB2 + 64;
};

// The maps of one side: map i is served by the CTAs first[i] .. first[i + 1] - 1.
struct WgMaps {
    CUtensorMap x, w1[3];
    const __nv_bfloat16* b1[3];
    const __nv_bfloat16* W2[3];
    int first[4];
    int n;
};

// X [rows][DV] bf16.  feat / dfeat: key side (N > 0) [bh][n][N][DP], query side (N = 0) [rows][DP].  wpart: [gridDim.x][kPartFloats].
template <int DV, int DP>
__global__ void __launch_bounds__(kWgThreads, 1) tc_phi_wgrad_kernel(const __grid_constant__ WgMaps maps, const float* __restrict__ feat,
                                                                     const float* __restrict__ dfeat, float* __restrict__ wpart, long long rows, int N,
                                                                     int* status, bool beside) {
    using Cfg = WgCfg<DV, DP>;
    constexpr int HC = DV / 4;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Cfg::kOffBars);
    uint64_t* x_full = bars;           // [2] TMA
    uint64_t* x_empty = bars + 2;      // [2] MMA commit (dW1 of the unit has read the tile)
    uint64_t* w_full = bars + 4;       // TMA: W1 of the map
    uint64_t* h_full = bars + 6;       // MMA commit
    uint64_t* h_empty = bars + 7;      // 512 arrivals
    uint64_t* dp_full = bars + 8;      // [3] 128 arrivals
    uint64_t* dp_free = bars + 18;     // [3] MMA commit: the unit's products have read the block
    uint64_t* dg_full = bars + 11;     // MMA commit
    uint64_t* dg_empty = bars + 12;    // 512 arrivals
    uint64_t* gd_full = bars + 13;     // 512 arrivals: G and dh tiles written
    uint64_t* gd_empty = bars + 14;    // MMA commit + the column-sum warps
    uint64_t* acc_full = bars + 15;    // MMA commit after the last product
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 17);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int map = 0;
    while (map + 1 < maps.n && (int)blockIdx.x >= maps.first[map + 1]) ++map;
    const int slot = blockIdx.x - maps.first[map], nslots = maps.first[map + 1] - maps.first[map];
    const long long tiles = (rows + kTileTokens - 1) / kTileTokens;
    const long long t0 = tiles * slot / nslots, t1 = tiles * (slot + 1) / nslots;
    const int ntiles = (int)(t1 - t0);      // >= 1: a map has at most as many CTAs as there are tiles
    const __nv_bfloat16 *W2g = maps.W2[map], *b1g = maps.b1[map];
    const CUtensorMap* mapX = &maps.x;
    float* out_cta = wpart + (size_t)blockIdx.x * Cfg::kPartFloats;

    constexpr int kRows = 16 * Cfg::kDgSteps, kB1Abs = kRows - 16 + Cfg::kB1Row;
    for (int i = tid; i < 3 * kBlk / 16; i += kWgThreads) reinterpret_cast<uint4*>(smem + Cfg::kOffDp)[i] = make_uint4(0, 0, 0, 0);
    for (int i = tid; i < 2 * Cfg::kXBytes / 16; i += kWgThreads) reinterpret_cast<uint4*>(smem + Cfg::kOffX)[i] = make_uint4(0, 0, 0, 0);
    for (int i = tid; i < 4 * kBlk / 16; i += kWgThreads) reinterpret_cast<uint4*>(smem + Cfg::kOffG)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    for (int i = tid; i < kTileTokens; i += kWgThreads)      // K column 32 + kB1Row of dp block 0: the ones column of the bias step
        *reinterpret_cast<__nv_bfloat16*>(smem + Cfg::kOffDp + sw128_off(i, 4 + Cfg::kB1Row / 8) + (Cfg::kB1Row & 7) * 2) = __float2bfloat16_rn(1.f);
    fence_proxy_async();
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&x_full[i], 1);
            mbar_init(&x_empty[i], 1);
        }
        mbar_init(w_full, 1);
        mbar_init(h_full, 1);
        mbar_init(h_empty, 512);
        for (int i = 0; i < 3; ++i) {
            mbar_init(&dp_full[i], 128);
            mbar_init(&dp_free[i], 1);
        }
        mbar_init(dg_full, 1);
        mbar_init(dg_empty, 512);
        mbar_init(gd_full, 512);
        mbar_init(gd_empty, 1 + DV / 32);
        mbar_init(acc_full, 1);
        fence_mbar_init();
        prefetch_tmap(mapX);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_begin(beside);
    // (after the dependency wait: a kernel of the caller may have just written the weights)
    if (tid < DV) stage_w2t_column<DP, kRows, kB1Abs, Cfg::kW2tBlock>(smem + Cfg::kOffW2t, W2g, b1g, tid);
    fence_proxy_async();
    __syncthreads();
    bool ok = true;

    if (warp == 0) {
        if (elect_one()) {
            mbar_arrive_expect_tx(w_full, Cfg::kW1Bytes);
            for (int b = 0; b < DV / 64; ++b) tma_load_2d(smem + Cfg::kOffW1 + b * (DV * 128), &maps.w1[map], w_full, b * 64, 0);
            for (int unit = 0; unit < ntiles; ++unit) {
                const int st = unit & 1;
                if (!mbar_wait(&x_empty[st], ((unit >> 1) & 1) ^ 1)) { report_timeout(status, 1002); break; }
                mbar_arrive_expect_tx(&x_full[st], DV * kTileTokens * 2);
                for (int b = 0; b < DV / 64; ++b)
                    tma_load_2d(smem + Cfg::kOffX + st * Cfg::kXBytes + b * kBlk, mapX, &x_full[st], b * 64, (int)((t0 + unit) * kTileTokens));
            }
        }
    } else if (warp == 2) {
        if (elect_one()) {      // h = X * W1 + 1 * b1
            const uint32_t idesc1 = idesc_bf16(128, DV, false, true);    // X K-major, W1 [in][hidden] MN-major
            const uint64_t xd0 = smem_desc_sw128(smem_u32(smem + Cfg::kOffX), 16, 1024);
            const uint64_t wd = smem_desc_sw128(smem_u32(smem + Cfg::kOffW1), DV * 128, 1024);
            const uint64_t od = smem_desc_sw128(smem_u32(smem + Cfg::kOffDp) + 64, 16, 1024);
            const uint64_t bd0 = smem_desc_sw128(smem_u32(smem + Cfg::kOffW2t) + (Cfg::kDgSteps - 1) * 2048, Cfg::kW2tBlock, 1024);      // the K step with the b1 row
            bool good = mbar_wait(w_full, 0);
            for (int unit = 0; unit < ntiles && good; ++unit) {
                const int st = unit & 1;
                if (!(mbar_wait(&x_full[st], (unit >> 1) & 1) && mbar_wait(h_empty, (unit & 1) ^ 1))) { good = false; break; }
                // the unit's dg product must be complete too, so that h_full tells the arithmetic warps both
                if (!mbar_wait(dg_full, unit & 1)) { good = false; break; }
                tc_fence_after();
                const uint64_t xd = desc_advance(xd0, st * Cfg::kXBytes);
#pragma unroll
                for (int ks = 0; ks < DV / 16; ++ks)
                    umma_bf16(tmem, desc_advance(xd, (ks >> 2) * kBlk + (ks & 3) * 32), desc_advance(wd, ks * 2048), idesc1, ks > 0 ? 1u : 0u);
                umma_bf16(tmem, od, bd0, idesc1, 1u);      // + 1 * b1
                umma_commit(h_full);
            }
            if (!good) report_timeout(status, 1003);
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc_dg = idesc_bf16(128, DV, false, true);   // dg = dp (K-major) * W2^T (MN-major)
            const uint32_t idesc_w1 = idesc_bf16(128, DV, true, true);    // dW1 = X^T (MN-major, M = input index) * dh (MN-major, N = hidden)
            const uint32_t idesc_w2 = idesc_bf16(128, 64, true, true);    // dW2ext = G^T (MN-major, M = hidden) * dp block (MN-major, N = 64)
            const uint32_t dpa = smem_u32(smem + Cfg::kOffDp), xa = smem_u32(smem + Cfg::kOffX);
            const uint32_t ga = smem_u32(smem + Cfg::kOffG), da = smem_u32(smem + Cfg::kOffDh);
            const uint64_t vd0 = smem_desc_sw128(smem_u32(smem + Cfg::kOffW2t), Cfg::kW2tBlock, 1024);
            bool good = true;
            auto issue_dg = [&](int unit) -> bool {      // the arithmetic warps of unit - 1 must have taken their dg into registers
                if (unit > 0 && !mbar_wait(dg_empty, (unit - 1) & 1)) return false;
                if (!mbar_wait(&dp_full[unit % 3], (unit / 3) & 1)) return false;
                tc_fence_after();
#pragma unroll
                for (int ks = 0; ks < Cfg::kDgSteps; ++ks)
                    umma_bf16(tmem + kWgColDg, smem_desc_sw128(dpa + (unit % 3) * kBlk + ks * 32, 16, 1024), desc_advance(vd0, ks * 2048), idesc_dg,
                              ks > 0 ? 1u : 0u);
                umma_commit(dg_full);
                return true;
            };
            good = issue_dg(0);
            for (int unit = 0; unit < ntiles && good; ++unit) {
                const int st = unit & 1;
                if (unit + 1 < ntiles && !issue_dg(unit + 1)) { good = false; break; }
                if (!mbar_wait(gd_full, unit & 1)) { good = false; break; }
                tc_fence_after();
                const uint32_t xs = xa + st * Cfg::kXBytes, dps = dpa + (unit % 3) * kBlk;
#pragma unroll
                for (int ks = 0; ks < kTileTokens / 16; ++ks)
                    umma_bf16(tmem + kWgColW1, smem_desc_sw128(xs + ks * 2048, kBlk, 1024), smem_desc_sw128(da + ks * 2048, kBlk, 1024), idesc_w1,
                              (unit > 0 || ks > 0) ? 1u : 0u);
#pragma unroll
                for (int ks = 0; ks < kTileTokens / 16; ++ks)
                    umma_bf16(tmem + kWgColW2, smem_desc_sw128(ga + ks * 2048, kBlk, 1024), smem_desc_sw128(dps + ks * 2048, kBlk, 1024), idesc_w2,
                              (unit > 0 || ks > 0) ? 1u : 0u);
                umma_commit(gd_empty);
                umma_commit(&dp_free[unit % 3]);
                umma_commit(&x_empty[st]);
                if (unit == ntiles - 1) umma_commit(acc_full);
            }
            if (!good) report_timeout(status, 1004);
        }
    } else if (warp >= kWgSumWarp0 && warp < kWgDpWarp0) {
        // db1: column sums of the dh tile as the dW1 product sees it (bf16 values, fp32 sums).  Warp w owns the 32 hidden
        // units 32 w ..: one 16-byte load per lane and step, lane l adds the eight columns of chunk 4 w + (l & 3) over the
        // rows l >> 2, l >> 2 + 8, ... and keeps its partial sums; the lanes' sums meet after the last tile, in a fixed order.  (Two warps with one 4-byte load per row took as long as a whole unit: a lone warp issues
        // an instruction every five cycles or so.)
        const int sw = warp - kWgSumWarp0;
        if (sw < DV / 32) {
            const uint32_t da = smem_u32(smem + Cfg::kOffDh) + (sw >> 1) * kBlk;
            const int chunk = 4 * (sw & 1) + (lane & 3);
            float sm[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) sm[e] = 0.f;
            for (int unit = 0; unit < ntiles; ++unit) {
                if (ok && !mbar_wait(gd_full, unit & 1)) { ok = false; report_timeout(status, 1005); }
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
#pragma unroll 8
                for (int j = 0; j < kTileTokens / 8; ++j) {
                    uint32_t w[4];
                    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(da + sw128_off((lane >> 2) + 8 * j, chunk)) : "memory");
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        sm[2 * e] += __uint_as_float(w[e] << 16);
                        sm[2 * e + 1] += __uint_as_float(w[e] & 0xffff0000u);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(gd_empty);
                if (unit == ntiles - 1) {
                    float* o = out_cta + Cfg::kPartB1 + (sw >> 1) * 64 + 8 * chunk;
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        float v = sm[e];
#pragma unroll
                        for (int x = 4; x < 32; x <<= 1) v += __shfl_xor_sync(0xffffffffu, v, x);
                        if (lane < 4) o[e] = v;
                    }
                }
            }
        }
    } else if (warp >= kWgDpWarp0) {
        // dp = dfeat (.) 1[feat > 0] of one token row as [dp_hi | dp_lo] (two bf16 halves, so dg is exact to ~2^-17) into
        // block unit % 3, and db2 = sum over the tokens of dp (this warp's 32 tokens by shuffles: one partial per token quarter)
        const int quarter = warp - kWgDpWarp0, row = quarter * 32 + lane;
        const uint32_t dpblk = smem_u32(smem + Cfg::kOffDp);
        float b2s[DP];
#pragma unroll
        for (int i = 0; i < DP; ++i) b2s[i] = 0.f;
        for (int unit = 0; unit < ntiles; ++unit) {
            long long grow = (t0 + unit) * kTileTokens + row;
            const bool live = grow < rows;
            grow = live ? grow : rows - 1;
            size_t off;
            if (N > 0) {
                const uint32_t bh = (uint32_t)grow / (uint32_t)N, n = (uint32_t)grow - bh * (uint32_t)N;   // rows < 2^31 (checked on the host)
                off = (((size_t)bh * maps.n + map) * N + n) * DP;
            } else {
                off = (size_t)grow * DP;
            }
            uint32_t w[DP];      // [hi pairs | lo pairs]
#pragma unroll
            for (int i = 0; i < DP / 2; ++i) {
                const float2 f = __ldg(reinterpret_cast<const float2*>(feat + off) + i);
                const float2 g = __ldg(reinterpret_cast<const float2*>(dfeat + off) + i);
                const float d0 = (live && f.x > 0.f) ? g.x : 0.f, d1 = (live && f.y > 0.f) ? g.y : 0.f;
                const float l0 = d0 - __bfloat162float(__float2bfloat16_rn(d0)), l1 = d1 - __bfloat162float(__float2bfloat16_rn(d1));
                w[i] = pack_bf16(d0, d1);
                w[DP / 2 + i] = pack_bf16(l0, l1);
                b2s[2 * i] += d0;
                b2s[2 * i + 1] += d1;
            }
            if (ok && !mbar_wait(&dp_free[unit % 3], ((unit / 3) & 1) ^ 1)) { ok = false; report_timeout(status, 1010); }
            if (!ok) break;
            const uint32_t blk = dpblk + (unit % 3) * kBlk;
            if constexpr (DP == 6) {
                st_shared_v4(blk + sw128_off(row, 0), w[0], w[1], w[2], w[3]);
                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(blk + sw128_off(row, 1)), "r"(w[4]), "r"(w[5]) : "memory");
            } else {
#pragma unroll
                for (int c = 0; c < 3; ++c) st_shared_v4(blk + sw128_off(row, c), w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
            }
            fence_proxy_async();
            mbar_arrive(&dp_full[unit % 3]);
            if (unit == ntiles - 1) {      // the db2 partial of this token quarter
                float* o = out_cta + Cfg::kPartB2 + quarter * 16;
#pragma unroll
                for (int i = 0; i < DP; ++i) {
                    const float a = warp_sum(b2s[i]);
                    if (lane == 0) o[i] = a;
                }
                if (lane < 16 - DP) o[DP + lane] = 0.f;
            }
        }
    } else {
        const int quarter = warp & 3, part = (warp - kWgEpiWarp0) >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        for (int unit = 0; unit < ntiles && ok; ++unit) {
            // h_full(unit) also says that dg(unit) is complete (the thread that issues the h products waits for it first)
            if (!mbar_wait(h_full, unit & 1)) { ok = false; report_timeout(status, 1007); }
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            uint32_t dgr[HC];
#pragma unroll
            for (int c = 0; c < HC / 16; ++c) tmem_ld16(tmem + kWgColDg + lane_base + part * HC + 16 * c, *reinterpret_cast<uint32_t(*)[16]>(dgr + 16 * c));
            uint32_t hr[HC];
#pragma unroll
            for (int c = 0; c < HC / 16; ++c) tmem_ld16(tmem + lane_base + part * HC + 16 * c, *reinterpret_cast<uint32_t(*)[16]>(hr + 16 * c));
            tmem_ld_wait();
            tc_fence_before();
            mbar_arrive(dg_empty);
            mbar_arrive(h_empty);
            uint32_t gw[HC / 2], dw[HC / 2];
#pragma unroll
            for (int e = 0; e < HC / 2; ++e) {
                const float2 h = make_float2(__uint_as_float(hr[2 * e]), __uint_as_float(hr[2 * e + 1]));
                const float2 dg = make_float2(__uint_as_float(dgr[2 * e]), __uint_as_float(dgr[2 * e + 1]));
                float2 g, dh;
                gelu_both2(dg, h, g, dh);      // g = 2 GELU(h) (the factor 1/2 is applied when the partial is reduced); dg is halved (W2^T)
                gw[e] = pack_bf16(g.x, g.y);
                dw[e] = pack_bf16(dh.x, dh.y);
            }
            // the products of unit - 1 (and the column sums) have finished reading the two tiles
            if (!mbar_wait(gd_empty, (unit & 1) ^ 1)) { ok = false; report_timeout(status, 1008); }
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            const int col0 = part * HC;
            const uint32_t gblk = smem_u32(smem + Cfg::kOffG) + (col0 / 64) * kBlk, dblk = smem_u32(smem + Cfg::kOffDh) + (col0 / 64) * kBlk;
#pragma unroll
            for (int j = 0; j < HC / 8; ++j) {
                st_shared_v4(gblk + sw128_off(row, (col0 & 63) / 8 + j), gw[4 * j], gw[4 * j + 1], gw[4 * j + 2], gw[4 * j + 3]);
                st_shared_v4(dblk + sw128_off(row, (col0 & 63) / 8 + j), dw[4 * j], dw[4 * j + 1], dw[4 * j + 2], dw[4 * j + 3]);
            }
            fence_proxy_async();
            mbar_arrive(gd_full);
            if (unit == ntiles - 1) {
                // drain dW1 (lane = input index) and dW2ext (lane = hidden unit)
                if (!mbar_wait(acc_full, 0)) { ok = false; report_timeout(status, 1009); }
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                float* o = out_cta;
                if (row < DV) {
#pragma unroll
                    for (int c = 0; c < HC / 16; ++c) {
                        uint32_t r[16];
                        tmem_ld16(tmem + kWgColW1 + lane_base + col0 + 16 * c, r);
                        tmem_ld_wait();
                        float4* dst = reinterpret_cast<float4*>(o + (size_t)row * DV + col0 + 16 * c);
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            dst[q] = make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]), __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]));
                    }
                    if (part == 0) {
#pragma unroll
                        for (int c = 0; c < Cfg::kW2Cols / 16; ++c) {
                            uint32_t r[16];
                            tmem_ld16(tmem + kWgColW2 + lane_base + 16 * c, r);
                            tmem_ld_wait();
                            float4* dst = reinterpret_cast<float4*>(o + Cfg::kPartW2 + (size_t)row * Cfg::kW2Cols + 16 * c);
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                dst[q] = make_float4(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1]), __uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3]));
                        }
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, 512);
    grid_end(beside);
}

struct WgradOut {
    float* dW1[3];
    float* db1[3];
    float* dW2[3];
    float* db2[3];
    int first[4];      // map i: the partials first[i] .. first[i + 1] - 1
};
// Adds a map's partials in a fixed order (bit-reproducible) and writes its gradients (fp32, the shapes of the weights); grid = (blocks,
// maps).  A block owns 128 consecutive partial entries, a thread four of them: warp w adds the partials w, w + 8, ... of the map (512-byte
// reads, eight in flight), and the eight warp sums are added in warp order.  The entries of dW2 (its two halves) and db2 (its four token
// quarters) that make up one output lie in one block.  (With one entry per thread the two launches of a call took 16 us each for 11 MB.)
template <int DV, int DP>
__global__ void __launch_bounds__(256) tc_wgrad_reduce_kernel(const float* __restrict__ wpart, WgradOut out, bool beside) {
    using C1 = WgCfg<DV, DP>;
    constexpr int PF = C1::kPartFloats, oW2 = C1::kPartW2, oB1 = C1::kPartB1, oB2 = C1::kPartB2, W2C = C1::kW2Cols;
    static_assert(oW2 % 128 == 0 && 128 % W2C == 0 && PF % 4 == 0 && (oB2 % 128) + 64 <= 128, "entries of one output in one block");
    __shared__ __align__(16) float red[8][128];
    grid_begin(beside);
    const int m = blockIdx.y, base = blockIdx.x * 128;
    const int nctas = out.first[m + 1] - out.first[m];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, at = base + 4 * lane;
    const float* src = wpart + (size_t)out.first[m] * PF + at;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    if (at < PF) add_partials<8>(a, src, PF, warp, 8, nctas);
    *reinterpret_cast<float4*>(&red[warp][4 * lane]) = a;
    __syncthreads();
    const int i = threadIdx.x;
    if (i < 128) {
        float t = red[0][i];
#pragma unroll
        for (int w = 1; w < 8; ++w) t += red[w][i];
        red[0][i] = t;
    }
    __syncthreads();
    const int e = base + i;
    if (i < 128 && e < PF) {
        if (e < oW2) {
            out.dW1[m][e] = red[0][i];
        } else if (e < oB1) {
            const int j = (e - oW2) / W2C, o = (e - oW2) % W2C;
            if (o < DP) out.dW2[m][j * DP + o] = 0.5f * (red[0][i] + red[0][i + DP]);      // the G tile held 2 GELU(h); dp in two halves
        } else if (e < oB2) {
            out.db1[m][e - oB1] = red[0][i];
        } else if (e - oB2 < DP) {
            out.db2[m][e - oB2] = ((red[0][i] + red[0][i + 16]) + red[0][i + 32]) + red[0][i + 48];
        }
    }
    grid_end(beside);
}

// CTAs of the query map, and of each of n key maps: an even share of the SMs, and no more partials in all than three per tile (or four
// for a single tile), which bounds the workspace of short inputs.
inline int wgrad_query_ctas(long long tiles, int sm_count) { return (int)(tiles < sm_count ? tiles : sm_count); }
inline int wgrad_key_ctas(long long tiles, int sm_count, int n) {
    const int q = wgrad_query_ctas(tiles, sm_count), most = 2 * q < sm_count ? 2 * q : sm_count;
    return most / n > 1 ? most / n : 1;
}
inline size_t wgrad_part_bytes(int d, int n, long long rows, int sm_count) {
    const long long tiles = (rows + kTileTokens - 1) / kTileTokens;
    const size_t pf = d == 128 ? WgCfg<128, 12>::kPartFloats : WgCfg<64, 12>::kPartFloats;      // the larger of the two geometries
    return (size_t)(wgrad_query_ctas(tiles, sm_count) + n * wgrad_key_ctas(tiles, sm_count, n)) * pf * 4;
}

// dphi_q / dphi_k: fp32 device outputs with the shapes of the weights (dphi_k points to one entry per key map); either may be null.
// Both passes come first, the second beside the first (the partials of the sides have regions of their own), then both reductions, the
// second beside the first.
template <int DV, int F>
inline hla_status launch_phi_wgrad(const Dims& D, int BH, const hla_mlp* phi_q, const hla_mlp* phi_k, const void* Q, const void* K,
                                   const hla_mlp_grad* dphi_q, const hla_mlp_grad* dphi_k, char* ws, const hla_ws_layout& L, size_t off_wpart,
                                   int sm_count, LaunchRec& rec) {
    constexpr int NM = MT<F>::kMaps, DP = MT<F>::kDphi;
    const long long rows = (long long)BH * D.N;
    const long long tiles = (rows + kTileTokens - 1) / kTileTokens;
    int* status = reinterpret_cast<int*>(ws + L.status);
    if (!set_smem(tc_phi_wgrad_kernel<DV, DP>, WgCfg<DV, DP>::kSmem)) return HLA_ERR_CUDA;
    WgradOut out[2] = {};
    float* wpart[2];
    int nmaps[2] = {dphi_q ? 1 : 0, dphi_k ? NM : 0};
    bool first = true;
    for (int key = 0; key < 2; ++key) {
        const int n = nmaps[key];
        wpart[key] = reinterpret_cast<float*>(ws + off_wpart) + (key ? (size_t)wgrad_query_ctas(tiles, sm_count) * WgCfg<DV, DP>::kPartFloats : 0);
        if (n == 0) continue;
        const hla_mlp* w = key ? phi_k : phi_q;
        const hla_mlp_grad* g = key ? dphi_k : dphi_q;
        WgMaps maps{};
        WgradOut& o = out[key];
        if (!make_map_2d(&maps.x, key ? K : Q, (size_t)rows, DV, kTileTokens)) return HLA_ERR_CUDA;
        for (int i = 0; i < n; ++i) {
            if (!make_map_2d(&maps.w1[i], w[i].W1, DV, DV, DV)) return HLA_ERR_CUDA;
            maps.b1[i] = static_cast<const __nv_bfloat16*>(w[i].b1);
            maps.W2[i] = static_cast<const __nv_bfloat16*>(w[i].W2);
            o.dW1[i] = static_cast<float*>(g[i].dW1); o.db1[i] = static_cast<float*>(g[i].db1);
            o.dW2[i] = static_cast<float*>(g[i].dW2); o.db2[i] = static_cast<float*>(g[i].db2);
            maps.first[i + 1] = o.first[i + 1] = maps.first[i] + (key ? wgrad_key_ctas(tiles, sm_count, n) : wgrad_query_ctas(tiles, sm_count));
        }
        maps.n = n;
        const float* feat = reinterpret_cast<const float*>(ws + (key ? L.kf : L.qf));
        const float* dfeat = reinterpret_cast<const float*>(ws + (key ? L.dkf : L.dqf));
        const int per_head = key ? D.N : 0;
        rec.begin(key ? "tc_phi_wgrad_k" : "tc_phi_wgrad_q");
        launch_pdl(tc_phi_wgrad_kernel<DV, DP>, maps.first[n], dim3(kWgThreads), WgCfg<DV, DP>::kSmem, rec.st, maps, feat, dfeat, wpart[key], rows, per_head, status, !first);
        first = false;
        if (!rec.end()) return HLA_ERR_CUDA;
    }
    bool second = false;
    for (int key = 0; key < 2; ++key) {
        if (nmaps[key] == 0) continue;
        rec.begin("tc_wgrad_reduce");
        launch_pdl(tc_wgrad_reduce_kernel<DV, DP>, dim3((WgCfg<DV, DP>::kPartFloats + 127) / 128, nmaps[key]), dim3(256), 0, rec.st, (const float*)wpart[key], out[key], second);
        second = true;
        if (!rec.end()) return HLA_ERR_CUDA;
    }
    return HLA_OK;
}

inline hla_status phi_wgrad(const Dims& D, int BH, const hla_mlp* phi_q, const hla_mlp* phi_k, const void* Q, const void* K,
                            const hla_mlp_grad* dphi_q, const hla_mlp_grad* dphi_k, char* ws, const hla_ws_layout& L, size_t off_wpart, int sm_count,
                            LaunchRec& rec) {
    if (D.F == 3) {
        if (D.d == 128) return launch_phi_wgrad<128, 3>(D, BH, phi_q, phi_k, Q, K, dphi_q, dphi_k, ws, L, off_wpart, sm_count, rec);
        return launch_phi_wgrad<64, 3>(D, BH, phi_q, phi_k, Q, K, dphi_q, dphi_k, ws, L, off_wpart, sm_count, rec);
    }
    if (D.d == 128) return launch_phi_wgrad<128, 2>(D, BH, phi_q, phi_k, Q, K, dphi_q, dphi_k, ws, L, off_wpart, sm_count, rec);
    return launch_phi_wgrad<64, 2>(D, BH, phi_q, phi_k, Q, K, dphi_q, dphi_k, ws, L, off_wpart, sm_count, rec);
}

}  // namespace tc
}  // namespace hla
