// fp32 kernels for the paper's two geometries, (F, d_phi) = (3, 6) and (2, 12), at any head width d <= 128, d % 4 == 0: register-tiled
// products on the FMA units (fp32 inputs, and bf16 inputs of widths the tensor-core kernels do not take).  The kernels of hla_simt.cuh
// serve the other geometries.
//
// What bounds them is the FMA pipe, so each product is a tile of 8 tokens (or state rows) x 4 columns per thread that reads 16 bytes
// at a time from shared memory: 12 loads for 128 FMAs.  The kernels of hla_simt.cuh form 16-token tiles with one scalar load and one
// predicate per four FMAs and decode every index of T with divisions.
//
// The symmetry of the query tensor folds every contraction but one from P = 216 (144) products to M = 56 (78) monomials (the same
// argument as in hla_tc.cuh): the readout sees the state summed over index permutations, its gradient is the same for all
// permutations of an index, and so is G = X S^T of the key side.  Only the state itself is formed in full, because it is the layout
// the workspace promises (P rows); the folded rows are summed when a block stages the state.
//
// Measured on B200, fp32, F = 3, against the kernels of hla_simt.cuh: training step with B*H = 12, N = 3000, d = 64: 2602 -> 265 us (two
// state builds 1236 -> 63, two feature gradients 557 -> 46, two readouts 277 -> 35, feature networks backward 387 -> 94, forward 104 ->
// 63); forward with B*H = 2, N = 256, d = 16: 94 -> 19.8 us.  Of these, independent neighbours side by side, more splits of the gradient
// state and the small tiles: 431 -> 332 and 37 -> 25 us; loads without index divisions and without branches between them: 296 and 22.6;
// the state build as it is now: the rest.
#pragma once
#include "hla_simt.cuh"
#include "hla_tc.cuh"

namespace hla {
namespace simt {

// The per-token kernels work on tiles of TM = 8 R tokens, a thread holds the tokens tg + 8 i, i < R: R = 8 where that gives every SM a
// block, else R = 2 (512 rows: 32 blocks instead of 8, and a quarter of the serial work in each).
constexpr int kSbTok = 32;        // tokens per step of the state build
// State rows per block of the state build, in groups of 8 (a thread's rows): 72 of the 216 or 144 rows of the forward, all 56 or 78 of the
// gradient state.  (Blocks of 64 rows did a seventh of their work on padding.)
template <int F, bool BWD> constexpr int kSbGroups = !BWD ? 9 : (F == 3 ? 7 : 10);

template <int F> struct Geo {
    using M = tc::MT<F>;
    static constexpr int kDphi = M::kDphi, kN = M::kN, kKf = M::kKf;
    static constexpr int kNp = (kN + 3) / 4 * 4;             // rows of a folded operand, padded for 16-byte steps
    static constexpr int kP = F == 3 ? 216 : 144;
};

// The state row whose index digits are those of monomial m in ascending order.
template <int F> __host__ __device__ constexpr int first_row(int m) {
    int idx = 0;
    for (int a = 0; a < Geo<F>::kDphi; ++a)
        for (int b = a; b < Geo<F>::kDphi; ++b) {
            if (F == 2) {
                if (idx++ == m) return a * 12 + b;
            } else {
                for (int c = b; c < 6; ++c)
                    if (idx++ == m) return 36 * a + 6 * b + c;
            }
        }
    return 0;
}
template <int F> struct RowTable {
    short v[Geo<F>::kN];
    constexpr RowTable() : v() {
        for (int m = 0; m < Geo<F>::kN; ++m) v[m] = (short)first_row<F>(m);
    }
};
template <int F> __device__ constexpr RowTable<F> kRowTable{};

// ---- tiles -------------------------------------------------------------------------------------
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
    const uint2 w = __ldg(reinterpret_cast<const uint2*>(p));
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
}
__device__ __forceinline__ void store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16* p, float4 v) {
    *reinterpret_cast<uint2*>(p) = make_uint2(tc::pack_bf16(v.x, v.y), tc::pack_bf16(v.z, v.w));
}

// rows [row0, row0 + n) of a matrix [.][d] into a tile with row stride ld; rows from `limit` on are zero.  All threads of the block; a
// thread takes the columns 4 cg .. 4 cg + 3 of the rows tg, tg + 8, ...
template <int CG, typename T>
__device__ __forceinline__ void stage_rows(float* tile, int ld, const T* __restrict__ src, size_t row0, int n, size_t limit, int d) {
    const int c = 4 * (threadIdx.x % CG);
    if (c >= d) return;
#pragma unroll 8
    for (int r = threadIdx.x / CG; r < n; r += 8) {
        const float4 v = row0 + r < limit ? load4(src + (row0 + r) * d + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4*>(tile + r * ld + c) = v;
    }
}

// acc[i][j] += sum_k A[8 i][k] B[k][j], j < 4;  K a multiple of 4
template <int R> __device__ __forceinline__ void tile_nn(float (&acc)[R][4], const float* A, int lda, const float* B, int ldb, int K) {
#pragma unroll 1
    for (int k = 0; k < K; k += 4) {
        float4 b[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) b[e] = ld4(B + (k + e) * ldb);
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const float4 a = ld4(A + 8 * i * lda + k);
            const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                acc[i][0] = fmaf(av[e], b[e].x, acc[i][0]);
                acc[i][1] = fmaf(av[e], b[e].y, acc[i][1]);
                acc[i][2] = fmaf(av[e], b[e].z, acc[i][2]);
                acc[i][3] = fmaf(av[e], b[e].w, acc[i][3]);
            }
        }
    }
}
// The same (bit for bit) in packed instructions on pairs of columns: a multiplier is copied into both halves of a register pair, which leaves three
// issue slots where four single fmas were (the loads need them).  Feature networks forward, 12 heads x 3000 tokens, d = 64: 64.7 -> 62.6 us; in
// their backward, which is short of registers, 94.3 -> 95.7, and the readout is the same either way.  The forward call, 12 x 3000: d = 64 110.2 ->
// 107.1 us, 32 72.7 -> 70.0, 16 64.3 -> 62.0; up to d = 32 its two launches, which overlap, can also fit together worse: 12 x 4096, d = 32, 87.0 -> 89.6.
template <int R> __device__ __forceinline__ void tile_nn_packed(float (&acc)[R][4], const float* A, int lda, const float* B, int ldb, int K) {
    float2 p[R][2];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        p[i][0] = make_float2(acc[i][0], acc[i][1]);
        p[i][1] = make_float2(acc[i][2], acc[i][3]);
    }
#pragma unroll 1
    for (int k = 0; k < K; k += 4) {
        float4 b[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) b[e] = ld4(B + (k + e) * ldb);
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const float4 a = ld4(A + 8 * i * lda + k);
            const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 m = make_float2(av[e], av[e]);
                p[i][0] = __ffma2_rn(m, make_float2(b[e].x, b[e].y), p[i][0]);
                p[i][1] = __ffma2_rn(m, make_float2(b[e].z, b[e].w), p[i][1]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) {
        acc[i][0] = p[i][0].x; acc[i][1] = p[i][0].y;
        acc[i][2] = p[i][1].x; acc[i][3] = p[i][1].y;
    }
}
// The contraction of tile_nt below into a tile that starts at zero, even and odd k summed apart in packed instructions: half the issue
// slots, which the loads need, at the price of twice the accumulators.  Feature gradients of both sides, 12 heads x 3000 tokens, tile_nt -> this:
// d = 64 45 -> 43.5 us (F = 3), 66 -> 60 (F = 2), d = 128 78 -> 74, 95 -> 89; 12 x 2000, d = 96, 63.5 -> 57.5, 70.5 -> 64.  Not up to d = 32, where the
// registers of the two warps of a block decide how many blocks an SM holds (96 -> 158 with F = 3, 167 -> 219 with F = 2; 7 -> 6 and 5 -> 4 blocks): 40
// heads x 3000, d = 32, 76.6 -> 84.4 and 107 -> 119 us, the steps 423 -> 427.5 and 481 -> 492.5; 12 heads, d = 16, F = 2, the step 174.4 -> 182.4.
// Not in the networks' backward either, which keeps a dX tile besides: 94 -> 100 us.
template <int CG, int JN, int R> __device__ __forceinline__ void tile_nt_packed(float (&acc)[R][JN], const float* A, int lda, const float* B, int ldb, int K) {
    float2 p[R][JN];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < JN; ++j) p[i][j] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int k = 0; k < K; k += 4) {
        float4 b[JN];
#pragma unroll
        for (int j = 0; j < JN; ++j) b[j] = ld4(B + CG * j * ldb + k);
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const float4 a = ld4(A + 8 * i * lda + k);
#pragma unroll
            for (int j = 0; j < JN; ++j)
                p[i][j] = __ffma2_rn(make_float2(a.x, a.y), make_float2(b[j].x, b[j].y), __ffma2_rn(make_float2(a.z, a.w), make_float2(b[j].z, b[j].w), p[i][j]));
        }
    }
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < JN; ++j) acc[i][j] = p[i][j].x + p[i][j].y;
}
// acc[i][j] += sum_k A[8 i][k] B[CG j][k], j < JN  (rows of B past its end are the caller's padding)
template <int CG, int JN, int R> __device__ __forceinline__ void tile_nt(float (&acc)[R][JN], const float* A, int lda, const float* B, int ldb, int K) {
#pragma unroll 1
    for (int k = 0; k < K; k += 4) {
        float4 b[JN];
#pragma unroll
        for (int j = 0; j < JN; ++j) b[j] = ld4(B + CG * j * ldb + k);
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const float4 a = ld4(A + 8 * i * lda + k);
#pragma unroll
            for (int j = 0; j < JN; ++j) acc[i][j] = fmaf(a.x, b[j].x, fmaf(a.y, b[j].y, fmaf(a.z, b[j].z, fmaf(a.w, b[j].w, acc[i][j]))));
        }
    }
}

// The value-side tile: X = V, xz = 1 (forward), or X = r dO, xz = -r (dO . O), r = 1 / (eta + eps) (backward; CG lanes per row).
template <int CG, typename T, bool BWD>
__device__ __forceinline__ void stage_values(float* Xs, int ld, float* xz, const T* __restrict__ X, const T* __restrict__ O, const float* __restrict__ eta,
                                             const Dims& D, int bh, int tok0, int n, int limit) {
    if (!BWD) {
        stage_rows<CG>(Xs, ld, X + (size_t)bh * D.N * D.d, (size_t)tok0, n, (size_t)limit, D.d);
        for (int t = threadIdx.x; t < n; t += blockDim.x) xz[t] = tok0 + t < limit ? 1.f : 0.f;
        return;
    }
    const int cg = threadIdx.x % CG, c = 4 * cg;
#pragma unroll 4
    for (int t = threadIdx.x / CG; t < n; t += 8) {      // (n is a multiple of 8: all lanes of a warp take part in the sums)
        const int tok = tok0 + t;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        float s = 0.f, r = 0.f;
        if (tok < limit) {
            const size_t row = (size_t)bh * D.N + tok;
            r = 1.f / (__ldg(eta + row) + D.eps);
            if (c < D.d) {
                x = load4(X + row * D.d + c);
                const float4 o = load4(O + row * D.d + c);
                s = fmaf(x.x, o.x, fmaf(x.y, o.y, fmaf(x.z, o.z, x.w * o.w)));
            }
        }
#pragma unroll
        for (int o = CG / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (c < D.d) *reinterpret_cast<float4*>(Xs + t * ld + c) = make_float4(r * x.x, r * x.y, r * x.z, r * x.w);
        if (cg == 0) xz[t] = -r * s;
    }
}

// ---- state build -------------------------------------------------------------------------------
// Forward: rows = the P products T_k[p], X = V.  Backward: rows = the M monomials of q (the gradient is the same for every permutation
// of a row's indices), X = r dO, xz = -r (dO . O).  Block = (split, 8 RG rows, head), thread = 8 rows x 4 columns; the T tile of a step and
// its part of z are formed by threads that own one row each (CG / 8 threads per row, alternate tokens), so that a row's digits are decoded
// once per block.  The next step's inputs are on their way (in registers) while a step is computed: with the loads between two barriers of
// the same step, 18 % of the FMA rate; at B*H = 12, N = 3000, d = 64 that kernel took 62 us, of which 22 were a second wave of 24 blocks.
template <typename T, int F, int CG, bool BWD>
__global__ void __launch_bounds__(CG * kSbGroups<F, BWD>, CG == 32 ? 2 : 64 / CG) tiled_state_build_kernel(Dims D, const float* __restrict__ feat, const T* __restrict__ X,
                                                                                                const T* __restrict__ O, const float* __restrict__ eta,
                                                                                                float* __restrict__ part, int S, bool beside, int* __restrict__ clear) {
    using G = Geo<F>;
    constexpr int RG = kSbGroups<F, BWD>, NR = 8 * RG, NT = CG * RG, DP = G::kDphi, LD = 4 * CG + 4, LT = NR + 4, NF = BWD ? 1 : F, ROWS = BWD ? G::kN : G::kP;
    constexpr int PER = CG / 8;                            // threads per row of T
    constexpr int XI = (kSbTok + RG - 1) / RG;             // rows of X per thread and step
    constexpr int FQ = NF * kSbTok * DP / 2, FI = (FQ + NT - 1) / NT;      // float2 of features per step, and per thread
    __shared__ __align__(16) float Ts[kSbTok * LT];
    __shared__ __align__(16) float Xs[kSbTok * LD];
    __shared__ __align__(16) float fs[NF * kSbTok * DP];     // [map][token][feature]: each map's part is one run of the input
    __shared__ float xz[kSbTok];
    __shared__ float zs[PER * NR];
    const int s = blockIdx.x, row0 = blockIdx.y * NR, bh = blockIdx.z;
    const int cg = threadIdx.x % CG, rg = threadIdx.x / CG;      // columns 4 cg .., rows 8 rg ..
    const int steps = (D.N + kSbTok - 1) / kSbTok;
    const int t0 = (int)((long long)steps * s / S) * kSbTok, t1 = min(D.N, (int)((long long)steps * (s + 1) / S) * kSbTok);
    // the row this thread forms: offsets of its factors in fs
    const int trow = threadIdx.x % NR, row = row0 + trow, tpar = threadIdx.x / NR;
    int dig[F];
    {
        int rem = row < ROWS ? (BWD ? kRowTable<F>.v[row < ROWS ? row : 0] : row) : 0;
#pragma unroll
        for (int f = F - 1; f >= 0; --f) {
            dig[f] = rem % DP + (BWD ? 0 : f * (kSbTok * DP));
            rem /= DP;
        }
    }
    const float live = row < ROWS ? 1.f : 0.f;
    tc::grid_begin(beside);
    if (clear && s == 0 && blockIdx.y == 0 && bh == 0 && threadIdx.x < 16) clear[threadIdx.x] = 0;
    float2 acc[8][2];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
    float zacc = 0.f;
    if (4 * cg >= D.d) {      // columns past the head width: never staged, kept finite
        for (int t = rg; t < kSbTok; t += RG) *reinterpret_cast<float4*>(Xs + t * LD + 4 * cg) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float4 xn[XI], on[BWD ? XI : 1];
    float en[BWD ? XI : 1];
    float2 fn[FI];
    auto load_step = [&](int tok0) {
#pragma unroll
        for (int i = 0; i < XI; ++i) {
            const int t = rg + RG * i, tok = tok0 + t;
            const bool in = t < kSbTok && tok < t1;
            const size_t at = (size_t)bh * D.N + (in ? tok : t0);
            xn[i] = in && 4 * cg < D.d ? load4(X + at * D.d + 4 * cg) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (BWD) {
                on[i] = in && 4 * cg < D.d ? load4(O + at * D.d + 4 * cg) : make_float4(0.f, 0.f, 0.f, 0.f);
                en[i] = in ? 1.f / (__ldg(eta + at) + D.eps) : 0.f;
            }
        }
#pragma unroll
        for (int i = 0; i < FI; ++i) {
            const int e = threadIdx.x + NT * i, f = e / (kSbTok * DP / 2), j = e - f * (kSbTok * DP / 2);      // token j / (DP / 2)
            const bool in = e < FQ && 2 * j < (t1 - tok0) * DP;
            const size_t at = BWD ? ((size_t)bh * D.N + tok0) * DP : (((size_t)bh * F + (in ? f : 0)) * D.N + tok0) * DP;
            fn[i] = in ? __ldg(reinterpret_cast<const float2*>(feat + at) + j) : make_float2(0.f, 0.f);
        }
    };
    if (t0 < t1) load_step(t0);
    for (int tok0 = t0; tok0 < t1; tok0 += kSbTok) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < XI; ++i) {
            const int t = rg + RG * i;
            float4 x = xn[i];
            if (BWD) {
                const float r = en[i];
                float v = fmaf(x.x, on[i].x, fmaf(x.y, on[i].y, fmaf(x.z, on[i].z, x.w * on[i].w)));
                const unsigned lanes = CG == 32 ? 0xffffffffu : ((1u << (CG & 31)) - 1u) << (threadIdx.x & 31 & ~(CG - 1));      // the row's CG lanes
#pragma unroll
                for (int o = CG / 2; o > 0; o >>= 1) v += __shfl_xor_sync(lanes, v, o);
                if (cg == 0 && t < kSbTok) xz[t] = -r * v;
                x = make_float4(r * x.x, r * x.y, r * x.z, r * x.w);
            } else if (cg == 0 && t < kSbTok) {
                xz[t] = tok0 + t < t1 ? 1.f : 0.f;
            }
            if (t < kSbTok && 4 * cg < D.d) *reinterpret_cast<float4*>(Xs + t * LD + 4 * cg) = x;
        }
#pragma unroll
        for (int i = 0; i < FI; ++i)
            if (threadIdx.x + NT * i < FQ) reinterpret_cast<float2*>(fs)[threadIdx.x + NT * i] = fn[i];
        __syncthreads();
        if (tok0 + kSbTok < t1) load_step(tok0 + kSbTok);
#pragma unroll 8
        for (int t = tpar; t < kSbTok; t += PER) {
            const float* f = fs + t * DP;
            float v = live * f[dig[0]] * f[dig[1]];
            if (F == 3) v *= f[dig[F - 1]];
            Ts[t * LT + trow] = v;
            zacc = fmaf(v, xz[t], zacc);
        }
        __syncthreads();
#pragma unroll 4
        for (int t = 0; t < kSbTok; ++t) {
            const float4 a0 = ld4(Ts + t * LT + 8 * rg), a1 = ld4(Ts + t * LT + 8 * rg + 4), x = ld4(Xs + t * LD + 4 * cg);
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float2 x0 = make_float2(x.x, x.y), x1 = make_float2(x.z, x.w);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float2 a = make_float2(av[i], av[i]);
                acc[i][0] = __ffma2_rn(a, x0, acc[i][0]);
                acc[i][1] = __ffma2_rn(a, x1, acc[i][1]);
            }
        }
    }
    float* out = part + ((size_t)bh * S + s) * ROWS * D.ld;
    if (4 * cg < D.d) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (row0 + 8 * rg + i < ROWS) store4(out + (size_t)(row0 + 8 * rg + i) * D.ld + 4 * cg, make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y));
    }
    zs[threadIdx.x] = zacc;      // [PER][NR]
    __syncthreads();
    if (threadIdx.x < NR && row < ROWS) {
        float z = zs[threadIdx.x];
#pragma unroll
        for (int k = 1; k < PER; ++k) z += zs[k * NR + threadIdx.x];
        store4(out + (size_t)row * D.ld + D.d, make_float4(z, 0.f, 0.f, 0.f));
    }
    tc::grid_end(beside);
}

// Sum of the split partials in a fixed order (bit-reproducible) -> state [BH][P][ld].  FOLDED: the partials hold the M monomial rows;
// every row of the state takes the sum of its monomial.
template <int F, bool FOLDED>
__global__ void __launch_bounds__(256) tiled_reduce_kernel(float* __restrict__ out, const float* __restrict__ part, int BH, int S, int ld) {
    using G = Geo<F>;
    constexpr int ROWS = FOLDED ? G::kN : G::kP;
    const int q = ld >> 2, total = BH * ROWS * q;
    tc::grid_begin(false);
    for (int i = blockIdx.x * 256 + threadIdx.x; i < total; i += gridDim.x * 256) {
        const int c = i % q, row = (i / q) % ROWS, bh = i / (q * ROWS);
        const float4* src = reinterpret_cast<const float4*>(part) + ((size_t)bh * S * ROWS + row) * q + c;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        tc::add_partials<8>(a, reinterpret_cast<const float*>(src), (size_t)ROWS * ld, 0, 1, S);
        float4* o = reinterpret_cast<float4*>(out) + (size_t)bh * G::kP * q + c;
        if (!FOLDED) {
            o[(size_t)row * q] = a;
        } else {
            const int p = kRowTable<F>.v[row];
            if (F == 2) {
                o[(size_t)p * q] = a;
                o[(size_t)((p % 12) * 12 + p / 12) * q] = a;
            } else {
                const int d0 = p / 36, d1 = (p / 6) % 6, d2 = p % 6;
                const int perm[6] = {36 * d0 + 6 * d1 + d2, 36 * d0 + 6 * d2 + d1, 36 * d1 + 6 * d0 + d2, 36 * d1 + 6 * d2 + d0, 36 * d2 + 6 * d0 + d1, 36 * d2 + 6 * d1 + d0};
#pragma unroll
                for (int e = 0; e < 6; ++e) o[(size_t)perm[e] * q] = a;
            }
        }
    }
}

__device__ float4 g_no_row;      // zeros, read in place of a row that is left out; never written

// Folded rows of a head's state into a tile [kNp][ldt] (columns 0 .. d: d values, then z; the padding rows are zero).
//   SUM = true: sum over the distinct permutations of the row's indices (what the readout of q (x) .. (x) q sees);
//   SUM = false: the row itself (a gradient state, the same for all permutations).
template <int F, bool SUM> __device__ __forceinline__ void stage_state(float* tile, int ldt, const float* __restrict__ st, int ld) {
    using G = Geo<F>;
    const int q = ld >> 2;
    for (int i = threadIdx.x; i < G::kNp * q; i += blockDim.x) {
        const int m = i / q, c = 4 * (i - m * q);
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        if (m < G::kN) {
            // Every row is a load, those that repeat an index tuple one of zeros: independent loads instead of a chain of branches.  (A zero
            // factor made NaN of an infinite row; choosing or masking the loaded values took 21.5 us for a forward of 2 heads x 256 tokens
            // instead of 20.0.)
            const int p = kRowTable<F>.v[m];
            auto row = [&](int r, bool on = true) { return __ldg(on ? reinterpret_cast<const float4*>(st + (size_t)r * ld + c) : &g_no_row); };
            auto add = [&](float4 v) {
                a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
            };
            if (!SUM) {
                a = row(p);
            } else if (F == 2) {
                const int d0 = p / 12, d1 = p % 12;
                const float4 v0 = row(p), v1 = row(d1 * 12 + d0, d0 != d1);
                a = v0;
                add(v1);
            } else {
                const int d0 = p / 36, d1 = (p / 6) % 6, d2 = p % 6;      // d0 <= d1 <= d2
                const bool n01 = d0 != d1, n12 = d1 != d2;
                const float4 v0 = row(p), v1 = row(36 * d0 + 6 * d2 + d1, n12), v2 = row(36 * d1 + 6 * d0 + d2, n01), v3 = row(36 * d1 + 6 * d2 + d0, n01 && n12),
                             v4 = row(36 * d2 + 6 * d0 + d1, n01 && n12), v5 = row(36 * d2 + 6 * d1 + d0, n01 || n12);
                a = v0;
                add(v1);
                add(v2);
                add(v3);
                add(v4);
                add(v5);
            }
        }
        *reinterpret_cast<float4*>(tile + m * ldt + c) = a;
    }
}

// Features of one token into registers (key side: F sets).
template <int F, bool QSIDE> __device__ __forceinline__ void load_token(float* f, const float* __restrict__ feat, const Dims& D, int bh, int tok) {
    using G = Geo<F>;
    if (QSIDE) {
        tc::load_feat<G::kDphi>(f, feat + ((size_t)bh * D.N + tok) * G::kDphi);
    } else {
#pragma unroll
        for (int m = 0; m < F; ++m) tc::load_feat<G::kDphi>(f + m * G::kDphi, feat + (((size_t)bh * F + m) * D.N + tok) * G::kDphi);
    }
}

// ---- readout -----------------------------------------------------------------------------------
// QSIDE: Y = (mono Csym) / (eta + eps), eta = mono . zsym saved.  Key side: dV = Tsym_k dC.  Tile of 64 tokens, thread = 8 tokens x 4
// columns; the 64 operand rows are formed by 64 threads, one token each, from registers.
template <typename T, int F, int CG, int R, bool QSIDE>
__global__ void __launch_bounds__(CG * 8) tiled_readout_kernel(Dims D, const float* __restrict__ feat, const float* __restrict__ state, T* __restrict__ Y,
                                                               float* __restrict__ eta_out, bool beside) {
    using G = Geo<F>;
    constexpr int TM = 8 * R, LD = 4 * CG + 4, LA = G::kNp + 4;
    extern __shared__ __align__(16) float dyn[];
    float* Ss = dyn;                          // [kNp][LD]
    float* As = Ss + G::kNp * LD;             // [TM][LA]
    float* inv = As + TM * LA;               // [TM]
    const int bh = blockIdx.y, tok0 = blockIdx.x * TM;
    const int cg = threadIdx.x % CG, tg = threadIdx.x / CG;
    tc::grid_begin(beside);
    stage_state<F, QSIDE>(Ss, LD, state + (size_t)bh * G::kP * D.ld, D.ld);
    if (threadIdx.x < TM) {
        const int tok = tok0 + threadIdx.x;
        constexpr int KF = QSIDE ? G::kDphi : G::kKf;
        float f[KF], v[G::kN];
        load_token<F, QSIDE>(f, feat, D, bh, tok < D.N ? tok : D.N - 1);
        if constexpr (QSIDE) tc::query_monomials_t<F>(f, v);
        else tc::key_folded_t<F>(f, v);
        float* a = As + threadIdx.x * LA;
#pragma unroll
        for (int m = 0; m < G::kNp; ++m) a[m] = m < G::kN ? v[m < G::kN ? m : 0] : 0.f;
    }
    __syncthreads();
    if (QSIDE) {
        for (int t = threadIdx.x; t < TM; t += CG * 8) {
            float e0 = 0.f, e1 = 0.f;
#pragma unroll 4
            for (int m = 0; m < G::kN; m += 2) {
                e0 = fmaf(As[t * LA + m], Ss[m * LD + D.d], e0);
                e1 = fmaf(As[t * LA + m + 1], Ss[(m + 1) * LD + D.d], e1);
            }
            inv[t] = 1.f / (e0 + e1 + D.eps);
            if (tok0 + t < D.N) eta_out[(size_t)bh * D.N + tok0 + t] = e0 + e1;
        }
    }
    float acc[R][4];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    if (4 * cg < D.d) tile_nn(acc, As + tg * LA, LA, Ss + 4 * cg, LD, G::kNp);
    if (QSIDE) __syncthreads();
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int tok = tok0 + tg + 8 * i;
        const float r = QSIDE ? inv[tg + 8 * i] : 1.f;
        if (tok < D.N && 4 * cg < D.d) store4(Y + ((size_t)bh * D.N + tok) * D.d + 4 * cg, make_float4(acc[i][0] * r, acc[i][1] * r, acc[i][2] * r, acc[i][3] * r));
    }
    tc::grid_end(beside);
}

// ---- feature gradients -------------------------------------------------------------------------
// G[t][m] = sum_g X[t][g] S[m][g] + xz[t] S[m][d], then the product rule through the folded outer product, one token per thread.
// QSIDE: X = r dO, xz = -r (dO . O), S = (C|z) summed over permutations.  Key side: X = V, xz = 1, S = (dC|dz).
template <typename T, int F, int CG, int R, bool QSIDE>
__global__ void __launch_bounds__(CG * 8) tiled_feature_grad_kernel(Dims D, const float* __restrict__ feat, const T* __restrict__ X, const T* __restrict__ O,
                                                                    const float* __restrict__ eta, const float* __restrict__ state, float* __restrict__ dfeat, bool beside) {
    using G = Geo<F>;
    constexpr int TM = 8 * R, LD = 4 * CG + 4, JN = (G::kN + CG - 1) / CG, LG = G::kN + 1;
    extern __shared__ __align__(16) float dyn[];
    float* Xs = dyn;                          // [TM][LD]
    float* Ss = Xs + TM * LD;                // [CG * JN][LD] (kNp rows are staged; the columns of the rest are not used)
    float* xz = Ss + CG * JN * LD;            // [TM]
    float* Gs = xz + TM;                     // [TM][LG], an odd stride
    const int bh = blockIdx.y, tok0 = blockIdx.x * TM;
    const int cg = threadIdx.x % CG, tg = threadIdx.x / CG;
    tc::grid_begin(beside);
    stage_state<F, QSIDE>(Ss, LD, state + (size_t)bh * G::kP * D.ld, D.ld);
    stage_values<CG, T, QSIDE>(Xs, LD, xz, X, O, eta, D, bh, tok0, TM, D.N);
    __syncthreads();
    float acc[R][JN];
    if constexpr (CG == 8) {      // d <= 32
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < JN; ++j) acc[i][j] = 0.f;
        tile_nt<CG, JN, R>(acc, Xs + tg * LD, LD, Ss + cg * LD, LD, D.d);
    } else {
        tile_nt_packed<CG, JN, R>(acc, Xs + tg * LD, LD, Ss + cg * LD, LD, D.d);
    }
#pragma unroll
    for (int j = 0; j < JN; ++j) {
        const int m = cg + CG * j;
        if (m < G::kN) {
            const float z = Ss[m * LD + D.d];
#pragma unroll
            for (int i = 0; i < R; ++i) Gs[(tg + 8 * i) * LG + m] = fmaf(xz[tg + 8 * i], z, acc[i][j]);
        }
    }
    __syncthreads();
    const int tok = tok0 + threadIdx.x;
    if (threadIdx.x < TM && tok < D.N) {
        float g[G::kN];
#pragma unroll
        for (int m = 0; m < G::kN; ++m) g[m] = Gs[threadIdx.x * LG + m];
        if constexpr (QSIDE) {
            float q[G::kDphi], dq[G::kDphi];
            load_token<F, true>(q, feat, D, bh, tok);
            tc::query_monomials_grad_t<F>(q, g, dq);
            tc::store_feat<G::kDphi>(dfeat + ((size_t)bh * D.N + tok) * G::kDphi, dq);
        } else {
            float k[G::kKf], dk[G::kKf];
            load_token<F, false>(k, feat, D, bh, tok);
            tc::key_folded_grad_t<F>(k, g, dk);
#pragma unroll
            for (int m = 0; m < F; ++m) tc::store_feat<G::kDphi>(dfeat + (((size_t)bh * F + m) * D.N + tok) * G::kDphi, dk + m * G::kDphi);
        }
    }
    tc::grid_end(beside);
}

// ---- feature networks --------------------------------------------------------------------------
// feat = ReLU(W2^T GELU(W1^T x + b1) + b2) of 64 rows and one map (blockIdx.y).  rows = B*H*N; key side: out [bh][maps][N][d_phi].
template <typename T, int DP, int CG, int R, bool KSIDE>
__global__ void __launch_bounds__(CG * 8) tiled_phi_forward_kernel(const T* __restrict__ X, PhiWeights<T> W, float* __restrict__ out, size_t rows, int N, int d, bool beside) {
    constexpr int TM = 8 * R, NT = CG * 8, LD = 4 * CG + 4;
    extern __shared__ __align__(16) float dyn[];
    float* Xs = dyn;                  // [TM][LD]; the hidden layer later
    float* Ws = Xs + TM * LD;        // [d][LD]
    float* W2s = Ws + 4 * CG * LD;    // [DP][LD], transposed
    const size_t row0 = (size_t)blockIdx.x * TM;
    const int m = blockIdx.y, cg = threadIdx.x % CG, tg = threadIdx.x / CG;
    tc::grid_begin(beside);
    stage_rows<CG>(Xs, LD, X, row0, TM, rows, d);
    stage_rows<CG>(Ws, LD, W.W1[m], 0, d, (size_t)d, d);
    for (int i = threadIdx.x; i < d * DP; i += NT) W2s[(i % DP) * LD + i / DP] = ldf(W.W2[m] + i);
    __syncthreads();
    float acc[R][4];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
    const bool live = 4 * cg < d;
    if (live) {
        tile_nn_packed(acc, Xs + tg * LD, LD, Ws + 4 * cg, LD, d);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float b = ldf(W.b1[m] + 4 * cg + j);
#pragma unroll
            for (int i = 0; i < R; ++i) acc[i][j] = gelu_erf(acc[i][j] + b);
        }
    }
    __syncthreads();      // the input tile has been read
    if (live) {
#pragma unroll
        for (int i = 0; i < R; ++i) store4(Xs + (tg + 8 * i) * LD + 4 * cg, make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < TM * DP; i += NT) {
        const int t = i / DP, o = i - t * DP;
        float p0 = 0.f, p1 = 0.f;
        for (int j = 0; j < d; j += 4) {
            const float4 g = ld4(Xs + t * LD + j), w = ld4(W2s + o * LD + j);
            p0 = fmaf(g.x, w.x, fmaf(g.y, w.y, p0));
            p1 = fmaf(g.z, w.z, fmaf(g.w, w.w, p1));
        }
        const size_t row = row0 + t;
        if (row < rows) {
            const float v = fmaxf(p0 + p1 + ldf(W.b2[m] + o), 0.f);
            if (KSIDE) {
                const size_t bh = row / N, n = row - bh * N;
                out[((bh * W.nmaps + m) * N + n) * DP + o] = v;
            } else {
                out[row * DP + o] = v;
            }
        }
    }
    tc::grid_end(beside);
}

// dX[row][:] = sum over maps of W1 (GELU'(h) (.) (W2 (dfeat (.) [feat > 0]))), h recomputed, the ReLU mask from the kept features.
// (At least 16 warps per SM where shared memory allows it: at most 128 registers a thread.)
template <typename T, int DP, int CG, int R, bool KSIDE>
__global__ void __launch_bounds__(CG * 8, CG == 32 ? 1 : 64 / CG) tiled_phi_backward_kernel(const T* __restrict__ X, PhiWeights<T> W, const float* __restrict__ feat,
                                                                    const float* __restrict__ dfeat, T* __restrict__ dX, size_t rows, int N, int d, bool beside) {
    constexpr int TM = 8 * R, NT = CG * 8, LD = 4 * CG + 4, LP = DP + 2;
    extern __shared__ __align__(16) float dyn[];
    float* Xs = dyn;                          // [TM][LD]
    float* Ws = Xs + TM * LD;                // [4 CG][LD]
    float* Hs = Ws + 4 * CG * LD;             // [TM][LD] dh
    float* W2s = Hs + TM * LD;               // [DP][LD], transposed
    float* dps = W2s + DP * LD;               // [TM][LP]
    const size_t row0 = (size_t)blockIdx.x * TM;
    const int cg = threadIdx.x % CG, tg = threadIdx.x / CG;
    const bool live = 4 * cg < d;
    tc::grid_begin(beside);
    stage_rows<CG>(Xs, LD, X, row0, TM, rows, d);
    for (int i = threadIdx.x; i < (4 * CG - d) * (d >> 2); i += NT)      // rows of W1 past the head width: read by tile_nt, kept finite
        *reinterpret_cast<float4*>(Ws + (d + i / (d >> 2)) * LD + 4 * (i % (d >> 2))) = make_float4(0.f, 0.f, 0.f, 0.f);
    float dx[R][4];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) dx[i][j] = 0.f;
    for (int m = 0; m < W.nmaps; ++m) {
        if (m > 0) __syncthreads();      // the previous map's tiles have been read
        stage_rows<CG>(Ws, LD, W.W1[m], 0, d, (size_t)d, d);
        for (int i = threadIdx.x; i < d * DP; i += NT) W2s[(i % DP) * LD + i / DP] = ldf(W.W2[m] + i);
        for (int i = threadIdx.x; i < TM * DP; i += NT) {
            const int t = i / DP, o = i - t * DP;
            const size_t row = row0 + t;
            float g = 0.f;
            if (row < rows) {
                size_t at = row * DP + o;
                if (KSIDE) {
                    const size_t bh = row / N, n = row - bh * N;
                    at = ((bh * W.nmaps + m) * N + n) * DP + o;
                }
                g = __ldg(feat + at) > 0.f ? __ldg(dfeat + at) : 0.f;
            }
            dps[t * LP + o] = g;
        }
        __syncthreads();
        if (live) {
            float h[R][4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float b = ldf(W.b1[m] + 4 * cg + j);
#pragma unroll
                for (int i = 0; i < R; ++i) h[i][j] = b;
            }
            tile_nn(h, Xs + tg * LD, LD, Ws + 4 * cg, LD, d);
            float dg[R][4];
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) dg[i][j] = 0.f;
#pragma unroll
            for (int o = 0; o < DP; ++o) {
                const float4 w = ld4(W2s + o * LD + 4 * cg);
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const float p = dps[(tg + 8 * i) * LP + o];
                    dg[i][0] = fmaf(p, w.x, dg[i][0]);
                    dg[i][1] = fmaf(p, w.y, dg[i][1]);
                    dg[i][2] = fmaf(p, w.z, dg[i][2]);
                    dg[i][3] = fmaf(p, w.w, dg[i][3]);
                }
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
                store4(Hs + (tg + 8 * i) * LD + 4 * cg, make_float4(dg[i][0] * gelu_erf_grad(h[i][0]), dg[i][1] * gelu_erf_grad(h[i][1]),
                                                                    dg[i][2] * gelu_erf_grad(h[i][2]), dg[i][3] * gelu_erf_grad(h[i][3])));
        }
        __syncthreads();
        tile_nt<CG, 4, R>(dx, Hs + tg * LD, LD, Ws + cg * LD, LD, d);      // column cg + CG j of dX
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j)      // through shared memory: whole rows leave with 16-byte stores
#pragma unroll
        for (int i = 0; i < R; ++i) Hs[(tg + 8 * i) * LD + cg + CG * j] = dx[i][j];
    __syncthreads();
    if (live) {
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const size_t row = row0 + tg + 8 * i;
            if (row < rows) store4(dX + row * d + 4 * cg, ld4(Hs + (tg + 8 * i) * LD + 4 * cg));
        }
    }
    tc::grid_end(beside);
}

// ---- host --------------------------------------------------------------------------------------
inline bool tiled(const Dims& D) { return (D.F == 3 && D.dphi == 6) || (D.F == 2 && D.dphi == 12); }
// Token splits of a state build: as many blocks as the SMs hold at once (at least 64 / CG of CG x 9 threads; a wave that is nearly empty
// costs as much as a full one), but at least two steps of 32 tokens per block where that leaves every SM one.
inline int tiled_split_count(int blocks_per_split, int N, int d, int sm_count) {
    const int held = (d <= 32 ? 8 : (d <= 64 ? 4 : 2)) * sm_count, steps = (N + kSbTok - 1) / kSbTok;
    int S = held / blocks_per_split;
    if (S > steps) S = steps;
    if (S < 1) S = 1;
    const int per = (steps + S - 1) / S;      // the same longest run of steps with the fewest splits
    return (steps + per - 1) / per;
}
inline int tiled_splits(int BH, int N, int P, int d, int sm_count) { return tiled_split_count(BH * (P / 72), N, d, sm_count); }
// The gradient state has M instead of P rows: more splits, within the same bytes of partials.
template <int F> inline int tiled_gradient_splits(const Dims& D, int BH, int sm_count) {
    const int room = (int)((long long)D.S * Geo<F>::kP / Geo<F>::kN), S = tiled_split_count(BH, D.N, D.d, sm_count);
    return S < room ? S : room;
}
template <int F, int CG, int R> struct TiledSmem {
    using G = Geo<F>;
    static constexpr int LD = 4 * CG + 4, TM = 8 * R;
    static constexpr size_t readout = sizeof(float) * (G::kNp * LD + TM * (G::kNp + 4) + TM);
    static constexpr size_t grad = sizeof(float) * (TM * LD + (G::kN + CG - 1) / CG * CG * LD + TM + TM * (G::kN + 1));
    static_assert((G::kN + CG - 1) / CG * CG >= G::kNp, "staged rows");
    static constexpr size_t phi_fwd = sizeof(float) * (TM * LD + 4 * CG * LD + G::kDphi * LD);
    static constexpr size_t phi_bwd = sizeof(float) * (2 * TM * LD + 4 * CG * LD + G::kDphi * LD + TM * (G::kDphi + 2));
};

struct TiledArgs {
    Dims D;
    int BH;
    const void *Q, *K, *V, *O, *dO;
    void *Oout, *dQ, *dK, *dV;
    const float *qf, *kf;      // features: given, or in the workspace
    float *qf_out, *kf_out, *dqf, *dkf, *part, *state, *dstate, *eta;
    const hla_mlp *phi_q, *phi_k;      // null: features are given
    bool in_order;             // backward: gradients lie over inputs, no kernel may run beside another (see Tiled::backward)
    int* clear;                // status words, cleared by a kernel of the forward (none of these kernels waits, so none reports)
};

// Launch sequences.  Every kernel is launched with programmatic stream serialization and waits for its predecessor at its top.
template <typename T, int F, int CG, int R> struct Tiled {
    using G = Geo<F>;
    using S = TiledSmem<F, CG, R>;
    static constexpr int NT = CG * 8, TM = 8 * R;

    template <typename... KArgs, typename... Args>
    static bool launch(LaunchRec& rec, const char* name, void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, Args... args) {
        if (smem > 48 * 1024 && !tc::set_smem(kernel, (int)smem)) return false;
        rec.begin(name);
        tc::launch_pdl(kernel, grid, dim3(threads), smem, rec.st, KArgs(args)...);
        return rec.end();
    }
    static PhiWeights<T> weights(const hla_mlp* m, int n) {
        PhiWeights<T> w{};
        w.nmaps = n;
        for (int i = 0; i < n; ++i) {
            w.W1[i] = static_cast<const T*>(m[i].W1);
            w.b1[i] = static_cast<const T*>(m[i].b1);
            w.W2[i] = static_cast<const T*>(m[i].W2);
            w.b2[i] = static_cast<const T*>(m[i].b2);
        }
        return w;
    }
    static dim3 reduce_grid(const TiledArgs& a, int rows) {
        const long long n = (long long)a.BH * rows * (a.D.ld / 4), b = (n + 255) / 256;
        return dim3((unsigned)(b < 8192 ? b : 8192));
    }
    static const T* in(const void* p) { return static_cast<const T*>(p); }
    static T* out(void* p) { return static_cast<T*>(p); }

    static bool forward(const TiledArgs& a, int, LaunchRec& rec) {
        const Dims& D = a.D;
        const size_t rows = (size_t)a.BH * D.N;
        const unsigned rb = (unsigned)((rows + TM - 1) / TM), tb = (unsigned)((D.N + TM - 1) / TM);
        // the key maps run beside the query map
        if (a.phi_q) {
            if (!launch(rec, "simt_phi_forward", tiled_phi_forward_kernel<T, G::kDphi, CG, R, false>, dim3(rb, 1), NT, S::phi_fwd, in(a.Q), weights(a.phi_q, 1), a.qf_out,
                        rows, D.N, D.d, false))
                return false;
            if (!launch(rec, "simt_phi_forward", tiled_phi_forward_kernel<T, G::kDphi, CG, R, true>, dim3(rb, F), NT, S::phi_fwd, in(a.K), weights(a.phi_k, F), a.kf_out,
                        rows, D.N, D.d, true))
                return false;
        }
        return launch(rec, "simt_state_build", tiled_state_build_kernel<T, F, CG, false>, dim3(D.S, G::kP / 72, a.BH), CG * kSbGroups<F, false>, 0, D, a.kf, in(a.V),
                      in(nullptr), a.eta, a.part, D.S, false, a.clear) &&
               launch(rec, "simt_reduce_partials", tiled_reduce_kernel<F, false>, reduce_grid(a, G::kP), 256, 0, a.state, a.part, a.BH, D.S, D.ld) &&
               launch(rec, "simt_readout", tiled_readout_kernel<T, F, CG, R, true>, dim3(tb, a.BH), NT, S::readout, D, a.qf, a.state, out(a.Oout), a.eta, false);
    }
    static bool backward(const TiledArgs& a, int sm_count, LaunchRec& rec) {
        const Dims& D = a.D;
        const size_t rows = (size_t)a.BH * D.N;
        const unsigned rb = (unsigned)((rows + TM - 1) / TM), tb = (unsigned)((D.N + TM - 1) / TM);
        const int Sg = tiled_gradient_splits<F>(D, a.BH, sm_count);
        auto dq = [&]() {
            return launch(rec, "simt_feature_grad", tiled_feature_grad_kernel<T, F, CG, R, true>, dim3(tb, a.BH), NT, S::grad, D, a.qf, in(a.dO), in(a.O), a.eta, a.state,
                          a.dqf, false);
        };
        auto partials = [&](bool beside) {
            return launch(rec, "simt_state_build", tiled_state_build_kernel<T, F, CG, true>, dim3(Sg, 1, a.BH), CG * kSbGroups<F, true>, 0, D, a.qf, in(a.dO), in(a.O),
                          a.eta, a.part, Sg, beside, nullptr);
        };
        auto sum = [&]() { return launch(rec, "simt_reduce_partials", tiled_reduce_kernel<F, true>, reduce_grid(a, G::kN), 256, 0, a.dstate, a.part, a.BH, Sg, D.ld); };
        auto dk = [&]() {
            return launch(rec, "simt_feature_grad", tiled_feature_grad_kernel<T, F, CG, R, false>, dim3(tb, a.BH), NT, S::grad, D, a.kf, in(a.V), in(nullptr), a.eta, a.dstate,
                          a.dkf, false);
        };
        auto dv = [&](bool beside) {
            return launch(rec, "simt_readout", tiled_readout_kernel<T, F, CG, R, false>, dim3(tb, a.BH), NT, S::readout, D, a.kf, a.dstate, out(a.dV), a.eta, beside);
        };
        // dq, and beside it the partials of dC, dz;  their sum;  dk^f, and beside it dV;  the feature networks of Q (dq is long complete) beside
        // that, then those of K.  One after the other, each input is read for the last time before a gradient of its own shape is written
        // over it (dQ over Q, dK over K, dQ over V with the feature networks).
        const bool beside = !a.in_order;
        if (!(beside ? dq() && partials(true) && sum() && dk() && dv(true) : partials(false) && sum() && dq() && dv(false) && dk())) return false;
        if (!a.phi_q) return true;
        return launch(rec, "simt_phi_backward", tiled_phi_backward_kernel<T, G::kDphi, CG, R, false>, dim3(rb), NT, S::phi_bwd, in(a.Q), weights(a.phi_q, 1), a.qf, a.dqf,
                      out(a.dQ), rows, D.N, D.d, beside) &&
               launch(rec, "simt_phi_backward", tiled_phi_backward_kernel<T, G::kDphi, CG, R, true>, dim3(rb), NT, S::phi_bwd, in(a.K), weights(a.phi_k, F), a.kf, a.dkf,
                      out(a.dK), rows, D.N, D.d, false);
    }
};

// The column groups of a block: the smallest of 8, 16, 32 (x 4 columns) that covers the head width.
template <typename T, int F, int R> inline bool run_tiled_r(const TiledArgs& a, bool fwd, int sm_count, LaunchRec& rec) {
    if (a.D.d <= 32) return fwd ? Tiled<T, F, 8, R>::forward(a, sm_count, rec) : Tiled<T, F, 8, R>::backward(a, sm_count, rec);
    if (a.D.d <= 64) return fwd ? Tiled<T, F, 16, R>::forward(a, sm_count, rec) : Tiled<T, F, 16, R>::backward(a, sm_count, rec);
    return fwd ? Tiled<T, F, 32, R>::forward(a, sm_count, rec) : Tiled<T, F, 32, R>::backward(a, sm_count, rec);
}
template <typename T> inline bool run_tiled(const TiledArgs& a, bool fwd, int sm_count, LaunchRec& rec) {
    const bool few = (long long)a.BH * ((a.D.N + 63) / 64) < sm_count;
    if (a.D.F == 3) return few ? run_tiled_r<T, 3, 2>(a, fwd, sm_count, rec) : run_tiled_r<T, 3, 8>(a, fwd, sm_count, rec);
    return few ? run_tiled_r<T, 2, 2>(a, fwd, sm_count, rec) : run_tiled_r<T, 2, 8>(a, fwd, sm_count, rec);
}

}  // namespace simt
}  // namespace hla
