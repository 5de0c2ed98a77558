// Correlation energy without any device allocation.
//
// Some callers cannot allocate device memory while they use this library:
//  * code that runs inside a CUDA stream capture, where cudaMalloc is not
//    allowed;
//  * hosts whose allocator owns all device memory and forbids outside
//    allocations;
//  * latency-bound loops that must not pay for an allocation.
// ccsd_energy needs a handle, and ccsd_create allocates.  This entry point
// takes the problem data as plain device pointers instead.  Its only scratch
// -- a few partial sums per momentum block -- lives in a fixed array in this
// file, which every GPU that loads the library keeps until the process exits.
#include "../../include/ccsd.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

namespace {

constexpr int kMaxPartials = 32768;            // N_k^3 + 1 slots of 16 bytes: 512 KiB
constexpr int kMaxDevices = 64;

static __device__ __align__(256) double2 g_energy_partials[kMaxPartials];

std::mutex g_mu;
double2* g_partials_addr[kMaxDevices] = {};    // device address of the array, per device

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// nseg blocks per momentum block (ki,kj,ka) of t2; block (b, seg) writes its part of
//   sum_ijab <ij||ab> (1/4 t_ij^ab + [ka == ki] 1/2 t_i^a t_j^b)
// to partials[b * nseg + seg]; the last block writes sum_k sum_ia f_ia t_i^a.
// Every slot is overwritten, so nothing has to be cleared between calls.  Four FMAs per
// element on the FP64 pipe (2 per clock and SM) bound the sum, as in ccsd_energy; the
// element index is decoded only where there is a t1 term.
constexpr int kUnroll = 8;
__global__ void __launch_bounds__(256) energy_blocks(
    const double2* __restrict__ t1, const double2* __restrict__ t2, const double2* __restrict__ fov,
    const double2* __restrict__ oovv, int N, int o, int v, int nseg, double2* __restrict__ partials)
{
    __shared__ double2 sm[8];
    const int nblk = N * N * N;
    const int b = blockIdx.x / nseg, seg = blockIdx.x % nseg;
    double d0[2] = {}, d1[2] = {}, d2[2] = {}, d3[2] = {}, sr = 0.0, si = 0.0;
    if (b < nblk) {
        const long long blk = (long long)o * o * v * v;
        const int ka = b % N, kj = (b / N) % N, ki = b / (N * N);
        const double2* gp = oovv + (long long)b * blk;
        const double2* tp = t2 + (long long)b * blk;
        const long long unit = 256LL * kUnroll;
        for (long long e0 = seg * unit; e0 < blk; e0 += nseg * unit) {
            double2 g[kUnroll], t[kUnroll];
#pragma unroll
            for (int q = 0; q < kUnroll; ++q) {
                const long long e = e0 + q * 256 + threadIdx.x;
                g[q] = t[q] = make_double2(0.0, 0.0);
                if (e < blk) { g[q] = gp[e]; t[q] = tp[e]; }
            }
            if (ka == ki) {
                // t + 2 t_i^a t_j^b in place of t
#pragma unroll
                for (int q = 0; q < kUnroll; ++q) {
                    const long long e = e0 + q * 256 + threadIdx.x;
                    if (e >= blk) break;
                    int a, bb, i, j;
                    if (blk < (1LL << 31)) {
                        unsigned r = (unsigned)e;
                        bb = (int)(r % (unsigned)v); r /= (unsigned)v;
                        a = (int)(r % (unsigned)v); r /= (unsigned)v;
                        j = (int)(r % (unsigned)o); i = (int)(r / (unsigned)o);
                    } else {
                        long long r = e;
                        bb = (int)(r % v); r /= v;
                        a = (int)(r % v); r /= v;
                        j = (int)(r % o); i = (int)(r / o);
                    }
                    double2 x = t1[((long long)ki * o + i) * v + a];
                    const double2 y = t1[((long long)kj * o + j) * v + bb];
                    x.x += x.x; x.y += x.y;
                    t[q].x = fma(x.x, y.x, t[q].x); t[q].x = fma(-x.y, y.y, t[q].x);
                    t[q].y = fma(x.x, y.y, t[q].y); t[q].y = fma(x.y, y.x, t[q].y);
                }
            }
#pragma unroll
            for (int q = 0; q < kUnroll; ++q) {
                const int h = q & 1;
                d0[h] = fma(g[q].x, t[q].x, d0[h]); d1[h] = fma(g[q].y, t[q].y, d1[h]);
                d2[h] = fma(g[q].x, t[q].y, d2[h]); d3[h] = fma(g[q].y, t[q].x, d3[h]);
            }
        }
    } else {
        const long long n1 = (long long)N * o * v;
        for (long long e = threadIdx.x; e < n1; e += blockDim.x) {
            const double2 p = cmul(fov[e], t1[e]);
            sr += p.x; si += p.y;
        }
    }
    double er = fma(0.25, (d0[0] - d1[0]) + (d0[1] - d1[1]), sr);
    double ei = fma(0.25, (d2[0] + d3[0]) + (d2[1] + d3[1]), si);
    for (int off = 16; off > 0; off >>= 1) {
        er += __shfl_down_sync(0xffffffffu, er, off);
        ei += __shfl_down_sync(0xffffffffu, ei, off);
    }
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = make_double2(er, ei);
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) { er += sm[w].x; ei += sm[w].y; }
        partials[blockIdx.x] = make_double2(er, ei);
    }
}

// Fixed-order sum of the partials (one warp), divided by N_k (energy per unit cell).
__global__ void energy_finish(const double2* __restrict__ partials, int n, double inv_nk, double* __restrict__ out)
{
    double r = 0.0, im = 0.0;
    for (int i = threadIdx.x; i < n; i += 32) { r += partials[i].x; im += partials[i].y; }
    for (int off = 16; off > 0; off >>= 1) {
        r += __shfl_down_sync(0xffffffffu, r, off);
        im += __shfl_down_sync(0xffffffffu, im, off);
    }
    if (threadIdx.x == 0) {
        out[0] = r * inv_nk;
        out[1] = im * inv_nk;
    }
}

// Device address of the partials array on the current device, looked up once.
int partials_address(double2** out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return CCSD_ERR_CUDA; }
    if (dev < 0 || dev >= kMaxDevices) return CCSD_ERR_INVALID;
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_partials_addr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_energy_partials) != cudaSuccess || !p) { cudaGetLastError(); return CCSD_ERR_CUDA; }
        g_partials_addr[dev] = (double2*)p;
    }
    *out = g_partials_addr[dev];
    return CCSD_OK;
}

}  // namespace

extern "C" int ccsd_energy_noalloc(const int nk_dims[3], int nocc, int nvir, const void* f_ov, const void* oovv,
                                   const void* t1, const void* t2, void* e_out, void* stream)
{
    if (!nk_dims || !f_ov || !oovv || !t1 || !t2 || !e_out) return CCSD_ERR_INVALID;
    long long N = 1;
    for (int d = 0; d < 3; ++d) {
        // the bound ccsd_create applies; it also keeps N^3 below 2^63
        if (nk_dims[d] < 1 || nk_dims[d] > 64) return CCSD_ERR_INVALID;
        N *= nk_dims[d];
    }
    if (nocc < 1 || nvir < 1 || nocc > 256 || nvir > 512) return CCSD_ERR_INVALID;
    // one partial per momentum block of t2 plus one for the singles term
    if (N * N * N + 1 > kMaxPartials) return CCSD_ERR_INVALID;
    double2* partials = nullptr;
    int rc = partials_address(&partials);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    // blocks for a few waves of the chip, within the array and one unit of elements each
    const long long units = ((long long)nocc * nocc * nvir * nvir + 256 * kUnroll - 1) / (256 * kUnroll);
    const long long nseg = std::max(1LL, std::min({units, (kMaxPartials - 1) / (N * N * N), 2048 / (N * N * N) + 1}));
    const int nparts = (int)(N * N * N * nseg + 1);
    energy_blocks<<<nparts, 256, 0, st>>>((const double2*)t1, (const double2*)t2, (const double2*)f_ov,
                                          (const double2*)oovv, (int)N, nocc, nvir, (int)nseg, partials);
    energy_finish<<<1, 32, 0, st>>>(partials, nparts, 1.0 / (double)N, (double*)e_out);
    if (cudaGetLastError() != cudaSuccess) return CCSD_ERR_CUDA;
    return CCSD_OK;
}
