// Tile shapes of the SIMT complex GEMM (zgemm_kb.cuh) and the rule that picks one, with
// its K split, for a contraction.  Host code, shared by the plan (ccsd_api.cu) and the
// launchers (zgemm_launch.cu).
#pragma once
#include <algorithm>

namespace ccsdk {

// (BM, BN, BK, TM, TN, KS), ZG_THREADS threads each
#define ZG_SHAPES(X)                                                                      \
    X(0, 64, 64, 8, 4, 4, 1)                                                              \
    X(1, 64, 32, 8, 4, 2, 1)                                                              \
    X(2, 128, 16, 8, 8, 1, 1)                                                             \
    X(3, 16, 16, 8, 1, 1, 1)                                                              \
    X(4, 32, 16, 8, 2, 1, 1)                                                              \
    X(5, 16, 16, 32, 2, 2, 4)                                                             \
    X(6, 32, 16, 32, 2, 2, 2)                                                             \
    X(7, 32, 32, 16, 2, 2, 1)                                                             \
    X(8, 128, 8, 8, 4, 1, 1)                                                              \
    X(9, 32, 8, 32, 2, 1, 2)                                                              \
    X(10, 8, 8, 32, 1, 1, 4)                                                              \
    X(11, 64, 1, 16, 1, 1, 4)

struct ZgShape { int bm, bn, bk, tm, tn, ks; };
constexpr ZgShape kZgShapes[] = {
#define X(id, bm, bn, bk, tm, tn, ks) {bm, bn, bk, tm, tn, ks},
    ZG_SHAPES(X)
#undef X
};
constexpr int kZgShapeCount = (int)(sizeof(kZgShapes) / sizeof(kZgShapes[0]));

// Arithmetic of an instance.
enum { ZG_FP64 = 0, ZG_FP32 = 1, ZG_DF = 2, ZG_ARITH = 3 };

// Rows and columns one warp covers (a warp outside M x N issues no products).
constexpr int zg_warp_rows(const ZgShape& s) { return 32 / (s.bn / s.tn < 8 ? s.bn / s.tn : 8) * s.tm; }
constexpr int zg_warp_cols(const ZgShape& s) { return (s.bn / s.tn < 8 ? s.bn / s.tn : 8) * s.tn; }

constexpr int kZgUnit = 32;            // K terms of one split unit (ZG_KU of the kernel)
constexpr int kZgMaxSplit = 64;
// Most partials of one launch (16 bytes each: 1 GiB).  Without the bound 3x3x3/o8/v24 took 4 GB
// of workspace beside 290 GB in use; at 2x2x2/o8/v32 the chosen splits need half of it.
constexpr long long kZgMaxPartials = 1LL << 26;
constexpr long long kZgFp32Chain = 8192;   // longest FP32 partial sum of the mixed form

struct ZgChoice { int shape, nsplit; double clocks; };

// Estimated time of one launch of shape s with nsplit K splits, in SM clocks.  The
// terms: products (padded to whole warps) at the arithmetic's rate, staging of the
// operand elements (an FP64 add per element for the 3M sums; for double-float three
// FP64-pipe conversions per complex128 component), the epilogue (FP64 conversions and
// adds per output, output read and written), the latency of a K step, waves of CTAs, and
// the CTA that adds a tile's partials.  c128: 0..2 operands are complex128 (the others
// complex64).  kZgFactor (a shape's products against the ideal rate: registers, resident
// CTAs and shared memory) and the other constants were fitted to the measured times of
// all shapes and splits on 41 contractions of 1 to 8 k points on GB300; the chosen shape
// is within 3 % (geometric mean) of the fastest one there, and within 3.6 % (at worst 1.6 times)
// on 120 contractions of other problems of that range.
// 0: not compiled.  Of 10^6 contractions drawn from M, N, K up to 8192, 729 chunks and 19683
// batches none took FP64's 64 x 64 tile (nor had it among the four that the batch autotuner
// times), or double-float's 64 x 32 and its 32 x 16 with two K groups (factors 4.0, 3.1, 2.4).
constexpr double kZgFactor[ZG_ARITH][kZgShapeCount] = {
    {0.0, 0.99, 2.6, 1.63, 1.13, 1.12, 1.12, 1.24, 1.08, 2.57, 1.2, 1.96},
    {1.2, 0.64, 4.0, 0.6, 2.4, 1.5, 1.7, 0.9, 1.4, 1.8, 0.6, 4.0},
    {2.3, 0.0, 1.5, 0.6, 0.89, 1.4, 0.0, 1.5, 1.2, 4.0, 0.6, 4.0}};
constexpr bool zg_built(int arith, int shape) { return kZgFactor[arith][shape] > 0.0; }
inline double zg_estimate(int arith, int shape, int nsplit, int M, int N, int K, long long nchunk,
                          long long nbatch, int c128, int sms) {
    const ZgShape& s = kZgShapes[shape];
    // clocks of the SM per product (a warp's products and its shared memory reads), per
    // staged element, per output; of a K step's latency; per four partials summed
    const double area = s.tm * s.tn * 32.0, reads = s.tm + s.tn;
    const double fma = kZgFactor[arith][shape] *
                       (arith == ZG_FP64 ? 1.52 : arith == ZG_FP32 ? (s.tm * s.tn + 0.5 * reads + 2.0) * 1.8 / area
                                                                   : (11.0 * s.tm * s.tn + reads + 2.0) * 1.25 / area);
    const double stage = arith == ZG_FP64 ? 0.7 : arith == ZG_FP32 ? 0.15 + 0.1 * c128 : 0.5 + 1.3 * c128;
    const double epi = arith == ZG_FP64 ? 3.0 : arith == ZG_FP32 ? 2.5 : 4.5;
    const double latency = arith == ZG_FP32 ? 1240.0 : 3200.0;
    const double mix = arith == ZG_FP32 ? 0.7 : 0.5, sum = 1650.0;
    const long long tm = (M + s.bm - 1) / s.bm, tn = (N + s.bn - 1) / s.bn;
    const int upc = (K + kZgUnit - 1) / kZgUnit;
    const long long units = nchunk * upc;
    const long long cta = tm * tn * nbatch * nsplit;
    const int wr = zg_warp_rows(s), wc = zg_warp_cols(s);
    // K steps and terms of one CTA and its products per term (the fullest tile, the mean)
    const double share = (double)((units + nsplit - 1) / nsplit) / upc;          // chunks
    const double steps = share * ((K + s.bk - 1) / s.bk);
    const double terms = share * ((K + s.ks - 1) / s.ks * s.ks);
    const double full = (double)std::min(s.bm, (M + wr - 1) / wr * wr) * std::min(s.bn, (N + wc - 1) / wc * wc);
    const double mean = (double)((M + wr - 1) / wr * wr) * ((N + wc - 1) / wc * wc) / (double)(tm * tn);
    const double work = (fma * mean + stage * (s.bm + s.bn)) * terms + epi * mean;
    const double top = (fma * full + stage * (s.bm + s.bn)) * terms + epi * full;
    const int resident = s.bm * s.bn >= 4096 ? (arith == ZG_FP32 ? 2 : 1) : s.bm * s.bn >= 2048 ? 2 : 4;
    const double per_sm = (double)((cta + sms - 1) / sms);
    const double waves = (double)((cta + (long long)sms * resident - 1) / ((long long)sms * resident));
    const double pipe = std::max((double)cta / sms * work, (per_sm > 1.0 ? per_sm - 1.0 : 0.0) * work + top);
    const double lat = waves * (steps * latency + 3000.0);
    const double bytes = (32.0 * M * N + (nsplit > 1 ? 32.0 * nsplit * M * N : 0.0)) * nbatch / 2000.0;
    double t = std::max(std::max(pipe, lat), bytes) + mix * std::min(pipe, lat) + 3000.0;
    if (nsplit > 1)         // the serial sum of the partials
        t += 1500.0 + nsplit / 4.0 * sum * std::max(1.0, (double)s.bm * s.bn / 256.0);
    return t;
}

// Splits that keep every FP32 partial sum of the mixed form within kZgFp32Chain terms.
inline long long zg_fp32_splits(int K, long long nchunk) {
    const long long units = nchunk * ((K + kZgUnit - 1) / kZgUnit);
    const long long most = std::max<long long>(1, kZgFp32Chain / std::min(K, kZgUnit));   // units per split
    return (units + most - 1) / most;
}

// The best K split of one shape: within the units there are, with FP32 sums as short as they must
// be, and with bounded partials.
inline ZgChoice zg_best_split(int arith, int shape, int M, int N, int K, long long nchunk, long long nbatch, int c128,
                              int sms) {
    const long long units = nchunk * ((K + kZgUnit - 1) / kZgUnit);
    const long long lo = arith == ZG_FP32 ? zg_fp32_splits(K, nchunk) : 1;
    ZgChoice best{shape, (int)lo, 1e300};
    static const int kSplits[] = {1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, kZgMaxSplit};
    for (int want : kSplits) {
        const long long ns = std::max<long long>(lo, std::min<long long>(want, units));
        if (ns > lo && ns * nbatch * M * N > kZgMaxPartials) continue;
        const double t = zg_estimate(arith, shape, (int)ns, M, N, K, nchunk, nbatch, c128, sms);
        if (t < best.clocks) best = ZgChoice{shape, (int)ns, t};
    }
    return best;
}

inline ZgChoice zg_choose(int arith, int M, int N, int K, long long nchunk, long long nbatch, int c128, int sms) {
    ZgChoice best{0, 1, 1e300};
    for (int i = 0; i < kZgShapeCount; ++i) {
        if (!zg_built(arith, i)) continue;
        const ZgChoice c = zg_best_split(arith, i, M, N, K, nchunk, nbatch, c128, sms);
        if (c.clocks < best.clocks) best = c;
    }
    return best;
}

}  // namespace ccsdk
