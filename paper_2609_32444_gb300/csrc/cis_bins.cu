// cis_bins.cu -- confidence-binned counts and sums of per-token values.
//
// The paper reports its statistics by bins of confidence: the sampled tokens
// binned by p_t with E[k_t - f_t] in each bin (Sec. 4.3, Fig. 5b), and
// logarithmic bins of 1 - p_t for the displacement and the log ratio (App.
// A.5).  cis_binned_sums takes any per-token key (p, 1 - p, ...) and up to four
// per-token values (k - f, the diagnostics' bias2 and dvar, ...) and gives
// each bin's count and the fp64 sums of the values; means are sum / count.
//
// Bound: HBM for long inputs (4 (NV + 1) bytes a token), launches for short ones.
// A thread adds its tokens to a column of bin accumulators of its own in shared
// memory, so a token costs one bin search and NV fp64 additions, whatever the
// number of bins, with no atomics and no exchange between threads: fp64
// additions run at 2 a clock and SM here, so their number decides.  (Summing
// every bin over every 256-token chunk in fixed fp64 butterflies, as before,
// took 345 us for 1,000,003 tokens in 18 bins with two values; this takes
// 18.9 us.)
//
// Deterministic: CTA c takes tokens c NT + i, then every grid NT further on;
// its columns are added in a fixed order, and a second kernel adds the CTAs'
// partial sums in a fixed tree.
#include <math.h>

#include <algorithm>

#include "cis_kernels.h"
#include "cis_nvtx.h"

namespace cis {
namespace {

constexpr int kBinTokens = 256;  // the workspace holds a partial sum per this many tokens
constexpr int kMaxBinCtas = 1024;
constexpr int kMaxBins = CIS_MAX_BINS;
constexpr int kMaxBinValues = CIS_MAX_BIN_VALUES;
constexpr int kBinMaxThreads = 256;
constexpr int kBinUnroll = 4;         // tokens a thread has in flight
constexpr int kCombineThreads = 256;  // one warp per (bin, field)

// edge[b], b < nbins: the smallest float that is >= the caller's edge, so that
// for a float key edge[b] <= key is the comparison of the fp64 values; last:
// the largest float <= the caller's last edge.
struct BinArgs {
    float edge[kMaxBins];
    float last;
    const float *values[kMaxBinValues];
    int nbins;
};

// The bin of a key: edge[b] <= key < edge[b + 1], the last bin closed on the
// right; -1 for a key outside [edge[0], last] or NaN.
__device__ __forceinline__ int bin_of(float key, const float *edge, float last, int nbins)
{
    if (!(key >= edge[0] && key <= last))
        return -1;
    int lo = 0, hi = nbins;  // edge[lo] <= key; the bin is in [lo, hi)
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (edge[mid] <= key)
            lo = mid;
        else
            hi = mid;
    }
    return lo;
}

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ long long warp_sum_i(long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// (double)f by its bits: the conversion instruction runs at the fp64 rate.
__device__ __forceinline__ double widen(float f)
{
    const uint32_t u = __float_as_uint(f);
    if (((u >> 23) & 255) - 1u < 254u)  // a normal number
        return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)),
                                (int)(u << 29));
    return (double)f;
}

// Shared memory of a CTA of NT threads: the sums' columns [nbins NV][NT], the
// counts' [nbins][NT].
size_t bin_smem(int nbins, int nvalues, int nt)
{
    return (size_t)nbins * (size_t)nt * (size_t)(8 * nvalues + 4);
}

// parts [nbins (NV + 1)][gridDim.x]: entry b (NV + 1) holds bin b's count (as an
// integer), the NV entries after it its sums.
template <int NV>
__global__ void __launch_bounds__(kBinMaxThreads)
    cis_binned_sums_kernel(const float *key, const uint8_t *mask, int64_t T,
                           const __grid_constant__ BinArgs a, double *parts)
{
    constexpr int kF = NV + 1;
    extern __shared__ __align__(16) double col[];
    __shared__ float edge[kMaxBins];
    const int NT = blockDim.x, tid = threadIdx.x, nbins = a.nbins;
    uint32_t *cnt = reinterpret_cast<uint32_t *>(col + (size_t)nbins * NV * NT);
    for (int k = 0; k < nbins * NV; ++k)
        col[k * NT + tid] = 0.0;
    for (int k = 0; k < nbins; ++k)
        cnt[k * NT + tid] = 0;
    for (int k = tid; k < nbins; k += NT)
        edge[k] = a.edge[k];
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * NT;
    for (int64_t t0 = (int64_t)blockIdx.x * NT + tid; t0 < T; t0 += kBinUnroll * step) {
        float k[kBinUnroll], v[NV > 0 ? NV : 1][kBinUnroll];
        bool on[kBinUnroll];
#pragma unroll
        for (int u = 0; u < kBinUnroll; ++u) {
            const int64_t t = t0 + u * step;
            on[u] = t < T && (mask == nullptr || mask[t] != 0);
            k[u] = t < T ? key[t] : NAN;
#pragma unroll
            for (int i = 0; i < NV; ++i)
                v[i][u] = t < T ? a.values[i][t] : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < kBinUnroll; ++u) {
            const int b = on[u] ? bin_of(k[u], edge, a.last, nbins) : -1;
            if (b >= 0) {
                ++cnt[b * NT + tid];
#pragma unroll
                for (int i = 0; i < NV; ++i)
                    col[(b * NV + i) * NT + tid] += widen(v[i][u]);
            }
        }
    }
    __syncthreads();
    // Every entry's columns are added 32 at a time, a warp per entry (lane l:
    // columns l, l + 32, ..., left in column l), then the 32 by one thread per
    // entry, each starting at a column of its own so that the threads' reads
    // fall in different banks.  (A butterfly would spend five fp64 additions of
    // all lanes on what one addition a column does.)
    const int lane = tid & 31, nsum = nbins * NV;
    for (int k = tid >> 5; k < nsum; k += NT / 32) {
        double s = col[k * NT + lane];
        for (int c = lane + 32; c < NT; c += 32)
            s += col[k * NT + c];
        col[k * NT + lane] = s;
    }
    for (int b = tid >> 5; b < nbins; b += NT / 32) {
        long long n = 0;
        for (int c = lane; c < NT; c += 32)
            n += cnt[b * NT + c];
        n = warp_sum_i(n);
        if (lane == 0)
            parts[(size_t)(b * kF) * gridDim.x + blockIdx.x] = __longlong_as_double(n);
    }
    __syncthreads();
    for (int k = tid; k < nsum; k += NT) {
        const double *src = col + k * NT;
        double s[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
            s[c] = src[(k + c) & 31];
#pragma unroll
        for (int c = 4; c < 32; ++c)
            s[c & 3] += src[(k + c) & 31];
        const int b = k / (NV > 0 ? NV : 1), i = k - b * NV;
        parts[(size_t)(b * kF + 1 + i) * gridDim.x + blockIdx.x] = (s[0] + s[1]) + (s[2] + s[3]);
    }
}

// One warp per entry: the CTAs' partial sums, lane by lane, then a butterfly.
__global__ void __launch_bounds__(kCombineThreads)
    cis_binned_combine_kernel(const double *parts, int ctas, int nbins, int nf,
                              int64_t *counts_out, double *sums_out)
{
    const int k = (int)((blockIdx.x * kCombineThreads + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (k >= nbins * nf)
        return;
    const int b = k / nf, f = k - b * nf;
    const double *src = parts + (size_t)k * ctas;
    if (f == 0) {
        long long n = 0;
        for (int c = lane; c < ctas; c += 32)
            n += __double_as_longlong(src[c]);
        n = warp_sum_i(n);
        if (lane == 0)
            counts_out[b] = n;
    } else {
        double s = 0.0;
        for (int c = lane; c < ctas; c += 32)
            s += src[c];
        s = warp_sum_d(s);
        if (lane == 0)
            sums_out[(size_t)(f - 1) * nbins + b] = s;
    }
}

// The most CTAs whose partial sums the workspace holds.
int64_t bin_ctas(int64_t T)
{
    const int64_t n = (T + kBinTokens - 1) / kBinTokens;
    return n < 1 ? 1 : (n > kMaxBinCtas ? kMaxBinCtas : n);
}

size_t bin_parts_bytes(int64_t T, int nbins, int nvalues)
{
    return (size_t)bin_ctas(T) * (size_t)nbins * (size_t)(nvalues + 1) * sizeof(double);
}

template <int NV>
cudaError_t launch_bins(const float *key, const uint8_t *mask, int64_t T, const BinArgs &a,
                        double *parts, int64_t *counts, double *sums, cudaStream_t s)
{
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    // As wide as about half of an SM's shared memory allows, two CTAs an SM;
    // 32 threads always fit: 64 bins of 4 values take 72 KB.  (T=1,000,003, 18
    // bins, two values: 18.9 us; one CTA an SM 21.8, 128 threads 22.2, four CTAs
    // of 128 20.4, one of 512 19.4.  T=4,000,000, 64 bins: 156 us; 292, 164, 186,
    // 152.)
    int nt = kBinMaxThreads;
    while (nt > 32 && bin_smem(a.nbins, NV, nt) > 100 * 1024)
        nt /= 2;
    const size_t smem = bin_smem(a.nbins, NV, nt);
    // a thread's columns cost it nbins additions at the end: give it some tokens
    const int64_t want = (T + (int64_t)nt * 8 - 1) / ((int64_t)nt * 8);
    int64_t ctas = std::min({want, (int64_t)2 * sms, bin_ctas(T)});
    ctas = ctas < 1 ? 1 : ctas;
    auto k = cis_binned_sums_kernel<NV>;
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
        cudaSuccess)
        return e;
    k<<<(unsigned)ctas, nt, smem, s>>>(key, mask, T, a, parts);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    const int entries = a.nbins * (NV + 1);
    cis_binned_combine_kernel<<<(unsigned)((entries + kCombineThreads / 32 - 1) /
                                           (kCombineThreads / 32)),
                                kCombineThreads, 0, s>>>(parts, (int)ctas, a.nbins, NV + 1,
                                                         counts, sums);
    return cudaGetLastError();
}

// The smallest float >= x, and the largest <= x (x not NaN).
float float_at_least(double x)
{
    const float f = (float)x;
    return (double)f >= x ? f : nextafterf(f, INFINITY);
}
float float_at_most(double x)
{
    const float f = (float)x;
    return (double)f <= x ? f : nextafterf(f, -INFINITY);
}

}  // namespace
}  // namespace cis

using namespace cis;

extern "C" {

CIS_API cis_status_t cis_binned_sums_workspace_size(int64_t T, int32_t nbins, int32_t nvalues,
                                                    size_t *bytes)
{
    if (bytes == nullptr || T < 0 || nbins < 1 || nbins > kMaxBins || nvalues < 0 ||
        nvalues > kMaxBinValues)
        return CIS_ERR_INVALID_ARG;
    *bytes = (bin_parts_bytes(T, nbins, nvalues) + 255) / 256 * 256 + 256;
    return CIS_OK;
}

CIS_API cis_status_t cis_binned_sums(const float *key, const uint8_t *mask, int64_t T,
                                     const double *edges, int32_t nbins,
                                     const float *const *values, int32_t nvalues,
                                     int64_t *counts_out, double *sums_out, void *workspace,
                                     size_t workspace_bytes, void *stream)
{
    NvtxRange nvtx_range("cis_binned_sums");
    size_t need = 0;
    if (cis_binned_sums_workspace_size(T, nbins, nvalues, &need) != CIS_OK || edges == nullptr ||
        counts_out == nullptr || (nvalues > 0 && (values == nullptr || sums_out == nullptr)) ||
        (T > 0 && key == nullptr) || workspace == nullptr || workspace_bytes < need ||
        (reinterpret_cast<uintptr_t>(workspace) & 255))
        return CIS_ERR_INVALID_ARG;
    BinArgs a = {};
    a.nbins = nbins;
    for (int b = 0; b <= nbins; ++b) {
        if (!(edges[b] == edges[b]) || (b > 0 && !(edges[b] > edges[b - 1])))
            return CIS_ERR_INVALID_ARG;  // NaN, or not strictly ascending
        if (b < nbins)
            a.edge[b] = float_at_least(edges[b]);
    }
    a.last = float_at_most(edges[nbins]);
    for (int i = 0; i < nvalues; ++i) {
        if (T > 0 && values[i] == nullptr)
            return CIS_ERR_INVALID_ARG;
        a.values[i] = values[i];
    }
    cudaStream_t s = (cudaStream_t)stream;
    double *parts = static_cast<double *>(workspace);
    cudaError_t e;
    switch (nvalues) {
    case 0: e = launch_bins<0>(key, mask, T, a, parts, counts_out, sums_out, s); break;
    case 1: e = launch_bins<1>(key, mask, T, a, parts, counts_out, sums_out, s); break;
    case 2: e = launch_bins<2>(key, mask, T, a, parts, counts_out, sums_out, s); break;
    case 3: e = launch_bins<3>(key, mask, T, a, parts, counts_out, sums_out, s); break;
    default: e = launch_bins<4>(key, mask, T, a, parts, counts_out, sums_out, s); break;
    }
    return e == cudaSuccess ? CIS_OK : CIS_ERR_CUDA;
}

}  // extern "C"
