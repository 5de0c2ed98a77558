// k-blocked batched complex GEMM (SIMT, FP64 DFMA).
//
//   C_b (+)= alpha * sum_{c < nchunk} opA(A_{b,c}) opB(B_{b,c})      b < nbatch
//
// Every contraction of the periodic CCSD residual is a sum over one
// "chunk" momentum (k_e, k_n, k_m, ...) of dense orbital contractions between
// momentum blocks whose positions follow from momentum conservation (paper
// Sec. 3.2.5).  The position of block (b, c) of each operand is an element
// offset in a device table; inside a block the element (r, s) sits at
// row_off[r] + col_off[s], which expresses any index permutation of a
// row-major orbital block (all CCSD layouts are separable that way).  This
// replaces the paper's ALLTOALL "index changes" (Sec. 4.3.3): operands are
// read in place, whatever their storage order.
//
// GB300's FP64 pipe (2 FMAs per clock and SM, a 64th of its FP32 rate) bounds the FP64
// instance: a 16 x 16 tile already reads its operands in a tenth of the time its DFMAs
// take, so tiles and K splits are chosen for even load and little padding
// (zgemm_shapes.h), and warps outside the result issue none.  Large contractions run at
// 0.95 of the measured DFMA rate (2x2x2/o8/v32 ring: 343 ms; 362 ms on one resident
// 64 x 64 CTA per SM without prefetch).  Contractions with few outputs were bound by one
// CTA walking the whole K: 3 k points, o = 5, v = 13, one iteration 6.3 -> 1.5 ms; the
// 2x2x1/o8/v32 double-float F~_oo 2.41 -> 0.18 ms and its R1 terms 4.1 -> 0.7 ms.
//
// The kernel is instantiated for two arithmetic types: double (the FP64 form)
// and float (the mixed form's CUDA-core contractions: operands are read from
// complex64 copies where the plan has them, otherwise rounded from complex128
// on load; products accumulate in FP32 and the epilogue adds alpha * acc into
// the FP64 result).  Integrals stored complex64 are read through A32/B32 by
// both; the double instance widens them exactly.  On GB300 a double->float conversion issues on the slow
// FP64 pipe, so the complex64 copies matter for throughput, not only bytes.
#pragma once
#include "dfloat.cuh"
#include "tf32_split.cuh"
#include <cuda_runtime.h>
#include <stdint.h>
#include <type_traits>

namespace ccsdk {

struct GemmArgs {
    const double2* A; const long long* offA; const int* rowA; const int* colA;
    const double2* B; const long long* offB; const int* rowB; const int* colB;
    const float2* A32; const float2* B32;   // complex64 A / B (copies, or inputs stored so), used instead when set
    double2* C;       const long long* offC; const int* rowC; const int* colC;
    double2* work;    // split partials [nsplit][nbatch][M*N] when nsplit > 1
    int* cnt;         // finished splits per (batch, tile), zero between launches (nsplit > 1)
    const int* nchunk_b;   // per-batch chunk count (<= nchunk), or null for nchunk everywhere
    // antisymmetric mirror: each result is also subtracted at offC2[b] + rowC[m] + colC2[n]
    const long long* offC2; const int* colC2;
    int M, N, K, nbatch, nchunk, nsplit;
    int conjA, conjB, accumulate;
    double alpha_re, alpha_im;
    int tiles_m, tiles_n;
    // Affine operand tables (set on the host when every entry fits): element (m, k) of A
    // at offA + a0 + m * rAs + k * cAs, element (k, n) of B at offB + b0 + k * rBs + n * cBs.
    // Gathers then skip the table loads.
    int affA, affB;
    int dfA, dfB;          // A / B holds double-float pairs (copies for the df instance)
    int kfA, kfB;          // stage this operand K-fastest: its K index is the more contiguous one
    long long a0, b0;
    int rAs, cAs, rBs, cBs;
};

template <typename T> struct Cplx;
template <> struct Cplx<double> { using V = double2; };
template <> struct Cplx<float> { using V = float2; };
template <> struct Cplx<df> { using V = df2; };

// A complex128 operand element in the instance's arithmetic.  The FP32 instance rounds
// with integer operations (f32_rn; the double-float conversion does the same itself):
// on GB300 every FP64 operation, a conversion included, issues on a pipe of 2 per clock
// and SM.  The results are those of the plain conversions, bit for bit.
template <typename T> __device__ __forceinline__ T from_f64(double x) { return T(x); }
template <> __device__ __forceinline__ float from_f64<float>(double x) { return f32_rn(x); }

// A partial sum as a double; floats widen by integer operations.
__device__ __forceinline__ double to_f64(double x) { return x; }
__device__ __forceinline__ double to_f64(float x) { return f64_scaled(x); }
__device__ __forceinline__ double to_f64(df x) { return f64_scaled(x.h) + f64_scaled(x.l); }


// Shared-memory staging of one K step: the complex tiles, and for the FP64 and
// double-float instances also Re + Im of every element (the third factor of the 3M
// product).  Rows are padded by 16 bytes: an operand staged K-fastest is stored with
// consecutive lanes on consecutive rows, which without the shift all fall into one bank.
template <int BM, int BN, int BK, typename T>
struct ZgemmSmem {
    static constexpr int P = 16 / (int)sizeof(typename Cplx<T>::V), PS = 16 / (int)sizeof(T);
    typename Cplx<T>::V A[BK][BM + P];
    typename Cplx<T>::V B[BK][(BN + P - 1) / P * P + P];
    T As[sizeof(T) == 8 ? BK : 1][BM + PS];
    T Bs[sizeof(T) == 8 ? BK : 1][(BN + PS - 1) / PS * PS + PS];
};

// A staged operand element travels in registers from its load to the next stage store
// (the loads of a K step are in flight while the previous one is multiplied).  A
// complex64 element keeps its 64 bits in .x untouched.
// (df instance: split, the element is a stored double-float pair, read by its bits.)
// conj: 0, or 0x80000000 to negate the imaginary part (a flipped sign bit; a product with -1
// would be an FP64-pipe operation per element).
template <typename T>
__device__ __forceinline__ typename Cplx<T>::V zg_operand(double2 raw, bool c64, bool split, int conj) {
    typename Cplx<T>::V v;
    if constexpr (sizeof(v) == sizeof(df2) && sizeof(T) == sizeof(df) && !std::is_same<T, double>::value) {
        if (split) {
            v.x = df(__int_as_float(__double2loint(raw.x)), __int_as_float(__double2hiint(raw.x)));
            v.y = df(__int_as_float(__double2loint(raw.y) ^ conj), __int_as_float(__double2hiint(raw.y) ^ conj));
            return v;
        }
    }
    if (c64) {
        v.x = T(__int_as_float(__double2loint(raw.x)));
        v.y = T(__int_as_float(__double2hiint(raw.x) ^ conj));
    } else {
        v.x = from_f64<T>(raw.x);
        v.y = from_f64<T>(__hiloint2double(__double2hiint(raw.y) ^ conj, __double2loint(raw.y)));
    }
    return v;
}

// One output tile (tile, batch b, K split) of one GEMM; called by the plain
// kernel below and by the grouped persistent kernel of the batched form.
//
// FP64 instance: 3M complex products.  With a = ar + i ai, b = br + i bi,
//   t1 = sum ar br,  t2 = sum ai bi,  t3 = sum (ar + ai)(br + bi),
//   Re c = t1 - t2,  Im c = t3 - t1 - t2,
// three FP64 FMAs per complex multiply-add instead of four (the sums ar + ai
// and br + bi are formed once per element when the tile is staged).  The FP32
// instance keeps the four-product form, whose imaginary part has no
// cancellation (its operands are already rounded to FP32).
//
// KS > 1 (few outputs, long K): the CTA's threads form KS groups of (BM / TM) (BN / TN)
// threads; all of them stage each K step, group q multiplies rows q, q + KS, .. of it,
// and at the end the groups' partial sums are added in group order (deterministic)
// before the epilogue.
//
// K splits (nsplit > 1) share the flattened sum over (chunk, K) in units of ZG_KU
// terms, so a contraction with few outputs and one long chunk spreads over the chip as
// well as one with many chunks.  The CTA that finishes an output tile last adds the
// tile's partials in split order (the order does not depend on which CTA is last).
//
// A warp owns a compact sub-tile (up to 4 x 8 threads).  A warp whose sub-tile lies
// outside M x N stages operands but issues no products: on GB300's FP64 pipe (2 FMAs
// per clock and SM) a padded product costs as much as a real one, and a 65 x 65 block
// on 64 x 64 tiles would otherwise pay for 128 x 128.
constexpr int ZG_KU = 32;
constexpr int ZG_THREADS = 256;

template <int BM, int BN, int BK, int TM, int TN, typename T, int KS = 1>
__device__ __forceinline__ void zgemm_tile(const GemmArgs& g, int tile, long long b, int split,
                                           ZgemmSmem<BM, BN, BK, T>& sm)
{
    using V = typename Cplx<T>::V;
    constexpr bool k3M = sizeof(T) == 8;         // double and double-float: 3M products
    constexpr int TX = BN / TN, TY = BM / TM;
    constexpr int NT1 = TX * TY;                 // threads of one K group
    constexpr int NT = NT1 * KS;
    constexpr int KG = BK / KS;                  // K rows of a stage per group
    constexpr int WX = TX < 8 ? TX : 8, WY = 32 / WX;   // threads of a warp's sub-tile
    constexpr int EA = (BM * BK + NT - 1) / NT, EB = (BN * BK + NT - 1) / NT;
    static_assert(NT == ZG_THREADS && NT1 % 32 == 0 && TX % WX == 0 && TY % WY == 0, "whole warps tile a K group");
    static_assert(BK % KS == 0 && ZG_KU % BK == 0 && ZG_KU == 32, "each K group takes an equal share of a stage");
    const int m0 = (tile % g.tiles_m) * BM;
    const int n0 = (tile / g.tiles_m) * BN;
    const int tid = threadIdx.x;
    const int kgrp = tid / NT1;
    const int wrp = (tid % NT1) / 32, lane = tid & 31;
    const int tx = (wrp % (TX / WX)) * WX + lane % WX, ty = (wrp / (TX / WX)) * WY + lane / WX;
    const bool active = m0 + (wrp / (TX / WX)) * WY * TM < g.M && n0 + (wrp % (TX / WX)) * WX * TN < g.N;
    auto& As = sm.A;
    auto& Bs = sm.B;

    // 4M: (cr, ci); 3M: (cr, ci, cs) = (t1, t2, t3)
    T cr[TM][TN], ci[TM][TN], cs[TM][k3M ? TN : 1];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            cr[i][j] = T(0); ci[i][j] = T(0);
            if (k3M) cs[i][k3M ? j : 0] = T(0);
        }

    const int sa = g.conjA ? (int)0x80000000 : 0, sb = g.conjB ? (int)0x80000000 : 0;
    const bool a32 = g.A32 != nullptr, b32 = g.B32 != nullptr;
    const bool kfA = g.kfA != 0, kfB = g.kfB != 0;
    // this split's share of the flattened (chunk, K) sum
    const int nch = g.nchunk_b ? g.nchunk_b[b] : g.nchunk;
    const int upc = (g.K + ZG_KU - 1) / ZG_KU;
    const long long U = (long long)nch * upc;
    const long long u0 = U * split / g.nsplit, u1 = U * (split + 1) / g.nsplit;

    if (u0 < u1) {
        int c = (int)(u0 / upc), k0 = (int)(u0 % upc) * ZG_KU;
        const int cl = (int)((u1 - 1) / upc), kl = min(g.K, (int)((u1 - 1) % upc + 1) * ZG_KU);
        const long long* offA = g.offA + b * g.nchunk;
        const long long* offB = g.offB + b * g.nchunk;
        long long oa = offA[c], ob = offB[c];
        // row part (A) and column part (B) of this thread's staged elements
        long long pa[EA], pb[EB];
#pragma unroll
        for (int i = 0; i < EA; ++i) {
            const int e = tid + i * NT, m = m0 + (kfA ? e / BK : e % BM);
            pa[i] = m < g.M ? (g.affA ? g.a0 + (long long)m * g.rAs : (long long)g.rowA[m]) : -1;
        }
#pragma unroll
        for (int i = 0; i < EB; ++i) {
            const int e = tid + i * NT, n = n0 + (kfB ? e / BK : e % BN);
            pb[i] = n < g.N ? (g.affB ? g.b0 + (long long)n * g.cBs : (long long)g.colB[n]) : -1;
        }
        double2 ra[EA], rb[EB];
        auto fetch = [&](int kend) {
#pragma unroll
            for (int i = 0; i < EA; ++i) {
                const int e = tid + i * NT, k = k0 + (kfA ? e % BK : e / BM);
                ra[i] = make_double2(0.0, 0.0);
                if ((BM * BK % NT == 0 || e < BM * BK) && pa[i] >= 0 && k < kend) {
                    const long long q = oa + pa[i] + (g.affA ? (long long)k * g.cAs : (long long)g.colA[k]);
                    if (a32) ra[i].x = __ldg((const double*)g.A32 + q);
                    else ra[i] = __ldg(g.A + q);
                }
            }
#pragma unroll
            for (int i = 0; i < EB; ++i) {
                const int e = tid + i * NT, k = k0 + (kfB ? e % BK : e / BN);
                rb[i] = make_double2(0.0, 0.0);
                if ((BN * BK % NT == 0 || e < BN * BK) && pb[i] >= 0 && k < kend) {
                    const long long q = ob + pb[i] + (g.affB ? (long long)k * g.rBs : (long long)g.rowB[k]);
                    if (b32) rb[i].x = __ldg((const double*)g.B32 + q);
                    else rb[i] = __ldg(g.B + q);
                }
            }
        };
        int kend = c == cl ? kl : g.K;
        fetch(kend);
        for (bool more = true; more;) {
            const int kst = kend - k0;                // terms of the stage being stored
            __syncthreads();                          // the previous stage has been multiplied
#pragma unroll
            for (int i = 0; i < EA; ++i) {
                const int e = tid + i * NT;
                if (BM * BK % NT == 0 || e < BM * BK) {
                    const int mm = kfA ? e / BK : e % BM, kk = kfA ? e % BK : e / BM;
                    const V v = zg_operand<T>(ra[i], a32, g.dfA != 0, sa);
                    As[kk][mm] = v;
                    // (rows outside M x K: no sum, so a warp staging only those issues none)
                    if constexpr (k3M) sm.As[kk][mm] = pa[i] >= 0 && kk < kst ? v.x + v.y : T(0);
                }
            }
#pragma unroll
            for (int i = 0; i < EB; ++i) {
                const int e = tid + i * NT;
                if (BN * BK % NT == 0 || e < BN * BK) {
                    const int nn = kfB ? e / BK : e % BN, kk = kfB ? e % BK : e / BN;
                    const V v = zg_operand<T>(rb[i], b32, g.dfB != 0, sb);
                    Bs[kk][nn] = v;
                    if constexpr (k3M) sm.Bs[kk][nn] = pb[i] >= 0 && kk < kst ? v.x + v.y : T(0);
                }
            }
            __syncthreads();
            k0 += BK;
            if (k0 >= kend) {
                if (c == cl) more = false;
                else {
                    ++c;
                    k0 = 0;
                    kend = c == cl ? kl : g.K;
                    oa = offA[c];
                    ob = offB[c];
                }
            }
            if (more) fetch(kend);
            if (!active) continue;
#pragma unroll
            for (int kq = 0; kq < KG; ++kq) {
                const int kk = kq * KS + kgrp;
                if (kk >= kst) break;
                V a[TM], bb[TN];
#pragma unroll
                for (int i = 0; i < TM; ++i) a[i] = As[kk][ty * TM + i];
#pragma unroll
                for (int j = 0; j < TN; ++j) bb[j] = Bs[kk][tx * TN + j];
                if constexpr (k3M) {
                    T xa[TM], xb[TN];
#pragma unroll
                    for (int i = 0; i < TM; ++i) xa[i] = sm.As[kk][ty * TM + i];
#pragma unroll
                    for (int j = 0; j < TN; ++j) xb[j] = sm.Bs[kk][tx * TN + j];
#pragma unroll
                    for (int i = 0; i < TM; ++i)
#pragma unroll
                        for (int j = 0; j < TN; ++j) {
                            cr[i][j] = fma(a[i].x, bb[j].x, cr[i][j]);
                            ci[i][j] = fma(a[i].y, bb[j].y, ci[i][j]);
                            cs[i][k3M ? j : 0] = fma(xa[i], xb[j], cs[i][k3M ? j : 0]);
                        }
                } else {
#pragma unroll
                    for (int i = 0; i < TM; ++i)
#pragma unroll
                        for (int j = 0; j < TN; ++j) {
                            cr[i][j] = fma(a[i].x, bb[j].x, cr[i][j]);
                            cr[i][j] = fma(-a[i].y, bb[j].y, cr[i][j]);
                            ci[i][j] = fma(a[i].x, bb[j].y, ci[i][j]);
                            ci[i][j] = fma(a[i].y, bb[j].x, ci[i][j]);
                        }
                }
            }
        }
    }

    if constexpr (KS > 1) {
        // the groups' partial sums, added in group order by group 0
        constexpr int NV = TM * TN * (k3M ? 3 : 2);
        static_assert(sizeof(ZgemmSmem<BM, BN, BK, T>) >= sizeof(T) * NV * NT1 * (KS > 1 ? KS - 1 : 1),
                      "the partial sums of the K groups fit the stage buffers");
        __syncthreads();                              // the last stage has been multiplied
        T* red = (T*)&sm;
        const int t1 = tid % NT1;
        if (kgrp > 0) {
            T* dst = red + ((long long)(kgrp - 1) * NT1 + t1) * NV;
            int q = 0;
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    dst[q++] = cr[i][j];
                    dst[q++] = ci[i][j];
                    if (k3M) dst[q++] = cs[i][k3M ? j : 0];
                }
        }
        __syncthreads();
        if (kgrp == 0) {
            for (int gq = 1; gq < KS; ++gq) {
                const T* src = red + ((long long)(gq - 1) * NT1 + t1) * NV;
                int q = 0;
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int j = 0; j < TN; ++j) {
                        cr[i][j] = cr[i][j] + src[q++];
                        ci[i][j] = ci[i][j] + src[q++];
                        if (k3M) cs[i][k3M ? j : 0] = cs[i][k3M ? j : 0] + src[q++];
                    }
            }
        }
    }
    const bool writes = active && kgrp == 0;
    if (k3M && writes) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                const T t1 = cr[i][j], t2 = ci[i][j];
                cr[i][j] = t1 - t2;
                ci[i][j] = cs[i][k3M ? j : 0] - t1 - t2;
            }
    }
    double2* const Cb = g.C + g.offC[b];
    double2* const C2 = g.offC2 ? g.C + g.offC2[b] : nullptr;
    // a real alpha takes one FP64 operation per component: the plan's factors are +-1 and
    // +-1/2, whose products are exact, so the fused add rounds once as the separate one did
    const bool areal = g.alpha_im == 0.0;
    auto put = [&](int m, int n, double xr, double xi) {
        double2* p = Cb + (long long)g.rowC[m] + g.colC[n];
        if (areal && g.accumulate && !C2) {
            double2 o = *p;
            o.x = fma(g.alpha_re, xr, o.x);
            o.y = fma(g.alpha_re, xi, o.y);
            *p = o;
            return;
        }
        const double re = areal ? g.alpha_re * xr : g.alpha_re * xr - g.alpha_im * xi;
        const double im = areal ? g.alpha_re * xi : g.alpha_re * xi + g.alpha_im * xr;
        if (g.accumulate) { double2 o = *p; o.x += re; o.y += im; *p = o; }
        else *p = make_double2(re, im);
        if (C2) {
            double2* q = C2 + (long long)g.rowC[m] + g.colC2[n];
            double2 o = *q; o.x -= re; o.y -= im; *q = o;
        }
    };
    if (g.nsplit > 1) {
        const long long plane = (long long)g.nbatch * g.M * g.N;
        double2* W = g.work + b * (long long)g.M * g.N;
        if (writes) {
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const int m = m0 + ty * TM + i, n = n0 + tx * TN + j;
                    if (m < g.M && n < g.N)
                        __stcg(W + split * plane + (long long)m * g.N + n,
                               make_double2(to_f64(cr[i][j]), to_f64(ci[i][j])));
                }
        }
        // the last CTA of the tile adds the partials (the counter returns to zero for the
        // next launch)
        __shared__ int s_last;
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            int* cnt = g.cnt + b * g.tiles_m * g.tiles_n + tile;
            const int prev = atomicAdd(cnt, 1);
            s_last = prev == g.nsplit - 1 ? 1 : 0;
            if (s_last) *cnt = 0;
        }
        __syncthreads();
        if (!s_last) return;
        __threadfence();
        // every thread of the CTA takes elements of the tile (KS groups included)
        for (int e = tid; e < BM * BN; e += NT) {
            const int m = m0 + e / BN, n = n0 + e % BN;
            if (m >= g.M || n >= g.N) continue;
            const double2* w = W + (long long)m * g.N + n;
            double xr = 0.0, xi = 0.0;
#pragma unroll 4
            for (int s = 0; s < g.nsplit; ++s) {
                const double2 z = __ldcg(w + s * plane);
                xr += z.x; xi += z.y;
            }
            put(m, n, xr, xi);
        }
        return;
    }
    if (writes) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) {
                const int m = m0 + ty * TM + i, n = n0 + tx * TN + j;
                if (m < g.M && n < g.N) put(m, n, to_f64(cr[i][j]), to_f64(ci[i][j]));
            }
    }
}

template <int BM, int BN, int BK, int TM, int TN, typename T, int KS = 1>
__global__ void __launch_bounds__(ZG_THREADS)
zgemm_kb_kernel(const GemmArgs g)
{
    __shared__ ZgemmSmem<BM, BN, BK, T> sm;
    const int ntile = g.tiles_m * g.tiles_n;
    zgemm_tile<BM, BN, BK, TM, TN, T, KS>(g, blockIdx.x % ntile, blockIdx.x / ntile, blockIdx.y, sm);
}

// Grouped persistent form (batched solves): one launch covers the same plan
// step of many independent problems.  Work item w of the flattened list
// [member][split][batch][tile] maps to member i with prefix[i] <= w < prefix[i+1];
// every CTA strides through the list.  All members use this launch's tile shape.
template <int BM, int BN, int BK, int TM, int TN, typename T, int KS = 1>
__global__ void __launch_bounds__(ZG_THREADS)
zgemm_grouped_kernel(const GemmArgs* __restrict__ gs, const long long* __restrict__ prefix, int nmem, long long total)
{
    __shared__ ZgemmSmem<BM, BN, BK, T> sm;
    for (long long w = blockIdx.x; w < total; w += gridDim.x) {
        int lo = 0, hi = nmem - 1;
        while (lo < hi) {                       // last member whose prefix <= w
            const int mid = (lo + hi + 1) >> 1;
            if (prefix[mid] <= w) lo = mid; else hi = mid - 1;
        }
        const GemmArgs g = gs[lo];
        const long long local = w - prefix[lo];
        const long long ntile = (long long)g.tiles_m * g.tiles_n;
        const long long per_split = ntile * g.nbatch;
        const int split = (int)(local / per_split);
        const long long r = local % per_split;
        zgemm_tile<BM, BN, BK, TM, TN, T, KS>(g, (int)(r % ntile), r / ntile, split, sm);
        __syncthreads();                        // the next item reuses the stage buffers
    }
}

}  // namespace ccsdk
