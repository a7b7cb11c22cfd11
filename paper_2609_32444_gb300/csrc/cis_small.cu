// cis_small.cu -- the [T]-sized kernels of libcis.
//
//   cis_scales_kernel   the loss normaliser s_t: 1/n over the n valid tokens
//                   (Algorithm 1) or 1/(G |y_i|) per response (Eq. 1); it
//                   also clears the device status word of the call.
//   cis_weights_kernel  cis_weights: Algorithm 1 / Table 8, one thread per token.
//   cis_reduce_kernel   deterministic sums (one CTA per 256 tokens, then the
//                   last CTA in index order) of the per-token loss terms and the
//                   statistics the paper logs (App. D.1: share of tokens acted
//                   on, largest |log k|; App. D.5: the truncated excess).
#include "cis_kernels.h"

namespace cis {
namespace {

constexpr int kSmallThreads = 1024;
constexpr int kSeqThreads = 256;  // one CTA per response
constexpr int kMaxSeqInShared = 12000;

__device__ __forceinline__ bool is_valid(const uint8_t *mask, int64_t t)
{
    return mask == nullptr || mask[t] != 0;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The loss normaliser.  global_counts (device {N, G}, or null): the batch's
// counts over every shard, used in place of this call's own.
__global__ void __launch_bounds__(kSmallThreads)
    cis_scales_kernel(const uint8_t *mask, int64_t T, const int32_t *cu, int64_t B, int agg,
                  float *scale, int32_t *status, uint32_t *ticket, const int64_t *global_counts)
{
    __shared__ long long part[kSmallThreads / 32];
    __shared__ int cnt[kMaxSeqInShared];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    allow_next_grid();
    if (threadIdx.x == 0 && status)
        *status = 0;
    if (threadIdx.x == 0 && ticket)  // the reduction at the end of this call counts from 0
        *ticket = 0;
    if (agg == CIS_AGG_SEQ_MEAN_TOKEN_MEAN && cu != nullptr) {
        // valid tokens of each response (one warp per response)
        for (int64_t i = wid; i < B; i += kSmallThreads / 32) {
            int64_t lo = cu[i], hi = cu[i + 1];
            lo = lo < 0 ? 0 : (lo > T ? T : lo);
            hi = hi < lo ? lo : (hi > T ? T : hi);
            int c = 0;
            for (int64_t t = lo + lane; t < hi; t += 32)
                c += is_valid(mask, t);
            c = warp_sum(c);
            if (lane == 0)
                cnt[i] = c;
        }
        __syncthreads();
        long long g = 0;
        for (int64_t i = threadIdx.x; i < B; i += kSmallThreads)
            g += cnt[i] > 0;
        g = warp_sum(g);
        if (lane == 0)
            part[wid] = g;
        for (int64_t t = threadIdx.x; t < T; t += kSmallThreads)
            scale[t] = 0.0f;
        __syncthreads();
        long long G = 0;
        for (int i = 0; i < kSmallThreads / 32; ++i)
            G += part[i];
        if (global_counts)
            G = global_counts[1];
        for (int64_t i = wid; i < B; i += kSmallThreads / 32) {
            int64_t lo = cu[i], hi = cu[i + 1];
            lo = lo < 0 ? 0 : (lo > T ? T : lo);
            hi = hi < lo ? lo : (hi > T ? T : hi);
            const int n = cnt[i];
            const float s = n > 0 ? (float)(1.0 / ((double)G * (double)n)) : 0.0f;
            for (int64_t t = lo + lane; t < hi; t += 32)
                scale[t] = is_valid(mask, t) ? s : 0.0f;
        }
        return;
    }
    long long n = 0;
    for (int64_t t = threadIdx.x; t < T; t += kSmallThreads)
        n += is_valid(mask, t);
    n = warp_sum(n);
    if (lane == 0)
        part[wid] = n;
    __syncthreads();
    long long N = 0;
    for (int i = 0; i < kSmallThreads / 32; ++i)
        N += part[i];
    if (global_counts)
        N = global_counts[0];
    const float s = N > 0 ? (float)(1.0 / (double)N) : 0.0f;
    for (int64_t t = threadIdx.x; t < T; t += kSmallThreads)
        scale[t] = is_valid(mask, t) ? s : 0.0f;
}

// This call's {N, G}: valid tokens, and responses with a valid token (one
// warp per response), for the all-reduce of a token-sharded run.
__global__ void __launch_bounds__(kSmallThreads)
    cis_count_kernel(const uint8_t *mask, int64_t T, const int32_t *cu, int64_t B,
                     int64_t *counts)
{
    __shared__ long long part[2][kSmallThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    long long n = 0, g = 0;
    for (int64_t t = threadIdx.x; t < T; t += kSmallThreads)
        n += is_valid(mask, t);
    if (cu != nullptr) {
        for (int64_t i = wid; i < B; i += kSmallThreads / 32) {
            int64_t lo = cu[i], hi = cu[i + 1];
            lo = lo < 0 ? 0 : (lo > T ? T : lo);
            hi = hi < lo ? lo : (hi > T ? T : hi);
            int c = 0;
            for (int64_t t = lo + lane; t < hi; t += 32)
                c += is_valid(mask, t);
            c = warp_sum(c);
            if (lane == 0)
                g += c > 0;
        }
    }
    n = warp_sum(n);
    g = warp_sum(g);
    if (lane == 0) {
        part[0][wid] = n;
        part[1][wid] = g;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long N = 0, G = 0;
        for (int i = 0; i < kSmallThreads / 32; ++i) {
            N += part[0][i];
            G += part[1][i];
        }
        counts[0] = N;
        counts[1] = G;
    }
}

// VEC tokens a thread (4: one 16-byte load or store per array and thread, for
// arrays that are aligned for it).  Bound: the operator's and eps' arithmetic (two
// exponentials, up to four logarithms a token) more than HBM (8 bytes in, up to 9
// out).  The operator is a template parameter, so that its code alone is there:
// 1,000,003 tokens, band, with eps: 10.2 us against 12.9 with all operators and one
// token a thread.
template <int MODE, int VEC>
__global__ void __launch_bounds__(256)
    cis_weights_kernel(const float *lp_w, const float *lp_inf, const uint8_t *mask, int64_t T,
                       const __grid_constant__ DevParams P, float *w_out, uint8_t *trunc_out,
                       float *eps_out)
{
    auto one = [&](float lw, float li, bool on, float &w, uint8_t &tr, float &e) {
        w = 0.0f;
        tr = 0;
        e = 0.0f;
        if (on) {
            const TokenWeight tw = token_weight<true, MODE>(lw, 0.0f, li, P);
            w = tw.w;
            tr = tw.trunc;
            if (eps_out)
                e = token_eps(lw, li);
        }
    };
    const int64_t n = T / VEC, step = (int64_t)gridDim.x * blockDim.x;
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if constexpr (VEC == 4) {
        for (int64_t i = i0; i < n; i += step) {
            const float4 a = reinterpret_cast<const float4 *>(lp_w)[i];
            const float4 b = reinterpret_cast<const float4 *>(lp_inf)[i];
            const uchar4 m = mask ? reinterpret_cast<const uchar4 *>(mask)[i]
                                  : make_uchar4(1, 1, 1, 1);
            float4 w, e;
            uchar4 t;
            one(a.x, b.x, m.x != 0, w.x, t.x, e.x);
            one(a.y, b.y, m.y != 0, w.y, t.y, e.y);
            one(a.z, b.z, m.z != 0, w.z, t.z, e.z);
            one(a.w, b.w, m.w != 0, w.w, t.w, e.w);
            reinterpret_cast<float4 *>(w_out)[i] = w;
            if (trunc_out)
                reinterpret_cast<uchar4 *>(trunc_out)[i] = t;
            if (eps_out)
                reinterpret_cast<float4 *>(eps_out)[i] = e;
        }
    }
    for (int64_t t = (VEC == 4 ? 4 * n : 0) + i0; t < T; t += step) {
        float w, e;
        uint8_t tr;
        one(lp_w[t], lp_inf[t], is_valid(mask, t), w, tr, e);
        w_out[t] = w;
        if (trunc_out)
            trunc_out[t] = tr;
        if (eps_out)
            eps_out[t] = e;
    }
}

// One CTA per response: the fp64 sum of log k over its valid tokens in a
// fixed order (thread-strided partial sums, then a tree), then the response's
// weight for each of them (seq_weight, Table 8).
__global__ void __launch_bounds__(kSeqThreads)
    cis_seq_weights_kernel(const double *lw64, const float *lw32, const float *lp_inf,
                           const int32_t *ids, int64_t V, const uint8_t *mask,
                           const int32_t *cu, int64_t T, const DevParams P, float *w,
                           uint8_t *trunc)
{
    __shared__ double red[kSeqThreads];
    const int64_t i = blockIdx.x;
    allow_next_grid();
    int64_t b = cu[i], e = cu[i + 1];
    b = b < 0 ? 0 : (b > T ? T : b);
    e = e < b ? b : (e > T ? T : e);
    auto used = [&](int64_t t) {
        return is_valid(mask, t) && (ids == nullptr || (ids[t] >= 0 && (int64_t)ids[t] < V));
    };
    double acc = 0.0;
    for (int64_t t = b + threadIdx.x; t < e; t += kSeqThreads)
        if (used(t))
            acc += (lw64 ? lw64[t] : (double)lw32[t]) - (double)lp_inf[t];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int off = kSeqThreads / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off)
            red[threadIdx.x] += red[threadIdx.x + off];
        __syncthreads();
    }
    const TokenWeight tw = seq_weight(red[0], P);
    for (int64_t t = b + threadIdx.x; t < e; t += kSeqThreads)
        if (used(t)) {
            w[t] = tw.w;
            if (trunc)
                trunc[t] = tw.trunc;
        }
}

struct RedPart {
    double loss, excess, ent;
    long long nvalid, ntrunc;
    float maxlk;
};

// Sums over the tokens in fp64, deterministic and spread over many SMs: fp64
// additions run at 2 a clock and SM here, so one CTA summing every token, or
// butterflies in which every lane adds, are bound by them.  CTA b takes tokens
// [256 b, 256 b + 256), one per thread, and leaves their sums in parts[b]; the
// last CTA to finish (a ticket, zeroed by the scales kernel at the start of the
// call) adds the parts in index order the same way and writes the results.
//
// The CTA's sums, in thread 0: the values go through shared memory, warp 0 adds
// the losses, warp 1 the excesses, warp 2 the entropies (lane l: threads l, l +
// 32, ..., then a butterfly), warp 3 the rest.
struct RedShared {
    double v[3][kRedTokens];
    long long n[2][kRedTokens];
    float mx[kRedTokens];
    RedPart out;
};
__device__ __forceinline__ RedPart block_red(const RedPart &p, RedShared &sh)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    sh.v[0][tid] = p.loss;
    sh.v[1][tid] = p.excess;
    sh.v[2][tid] = p.ent;
    sh.n[0][tid] = p.nvalid;
    sh.n[1][tid] = p.ntrunc;
    sh.mx[tid] = p.maxlk;
    __syncthreads();
    if (wid < 3) {
        double s = sh.v[wid][lane];
#pragma unroll
        for (int k = 32; k < kRedTokens; k += 32)
            s += sh.v[wid][lane + k];
        s = warp_sum(s);
        if (lane == 0)
            (wid == 0 ? sh.out.loss : wid == 1 ? sh.out.excess : sh.out.ent) = s;
    } else if (wid == 3) {
        long long n = 0, m = 0;
        float mx = 0.0f;
#pragma unroll
        for (int k = 0; k < kRedTokens; k += 32) {
            n += sh.n[0][lane + k];
            m += sh.n[1][lane + k];
            mx = fmaxf(mx, sh.mx[lane + k]);
        }
        n = warp_sum(n);
        m = warp_sum(m);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) {
            sh.out.nvalid = n;
            sh.out.ntrunc = m;
            sh.out.maxlk = mx;
        }
    }
    __syncthreads();
    return sh.out;
}

__global__ void __launch_bounds__(kRedTokens)
    cis_reduce_kernel(const uint8_t *mask, int64_t T, const double *terms, const float *logk,
                  const float *w, const uint8_t *trunc, const float *entropy,
                  const int32_t *status, RedPart *parts, uint32_t *ticket, cis_stats_t *stats,
                  double *loss_out)
{
    __shared__ RedShared sh;
    __shared__ bool last;
    RedPart p{0.0, 0.0, 0.0, 0, 0, 0.0f};
    const int64_t t = (int64_t)blockIdx.x * kRedTokens + threadIdx.x;
    grid_wait();
    if (t < T) {
        p.loss = terms[t];
        if (is_valid(mask, t)) {
            p.nvalid = 1;
            const float lk = logk[t];
            p.maxlk = fabsf(lk);
            if (trunc[t]) {
                p.ntrunc = 1;
                p.excess = exp((double)lk) - (double)w[t];
            }
            if (entropy)
                p.ent = (double)entropy[t];
        }
    }
    p = block_red(p, sh);
    if (threadIdx.x == 0) {
        parts[blockIdx.x] = p;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last)
        return;
    __threadfence();
    const volatile RedPart *vp = parts;
    RedPart q{0.0, 0.0, 0.0, 0, 0, 0.0f};
    for (unsigned b = threadIdx.x; b < gridDim.x; b += kRedTokens) {
        RedPart x;
        x.loss = vp[b].loss;
        x.excess = vp[b].excess;
        x.ent = vp[b].ent;
        x.nvalid = vp[b].nvalid;
        x.ntrunc = vp[b].ntrunc;
        x.maxlk = vp[b].maxlk;
        q.loss += x.loss;
        q.excess += x.excess;
        q.ent += x.ent;
        q.nvalid += x.nvalid;
        q.ntrunc += x.ntrunc;
        q.maxlk = fmaxf(q.maxlk, x.maxlk);
    }
    __syncthreads();
    q = block_red(q, sh);
    if (threadIdx.x == 0) {
        if (loss_out)
            *loss_out = q.loss;
        if (stats) {
            stats->loss = q.loss;
            stats->trunc_excess = q.excess;
            stats->n_valid = q.nvalid;
            stats->n_truncated = q.ntrunc;
            stats->max_abs_logk = q.maxlk;
            stats->status = status ? *status : 0;
            stats->entropy_sum = q.ent;
        }
    }
}

}  // namespace

cudaError_t launch_scales(const uint8_t *mask, int64_t T, const int32_t *cu_seqlens, int64_t B,
                          int agg, float *scale, int32_t *status, uint32_t *ticket,
                          cudaStream_t s, const int64_t *global_counts)
{
    if (agg == CIS_AGG_SEQ_MEAN_TOKEN_MEAN && B > kMaxSeqInShared)
        return cudaErrorNotSupported;
    cis_scales_kernel<<<1, kSmallThreads, 0, s>>>(mask, T, cu_seqlens, B, agg, scale, status,
                                                  ticket, global_counts);
    return cudaGetLastError();
}

cudaError_t launch_count_valid(const uint8_t *mask, int64_t T, const int32_t *cu_seqlens,
                               int64_t B, int64_t *counts, cudaStream_t s)
{
    if (B > kMaxSeqInShared)
        return cudaErrorNotSupported;
    cis_count_kernel<<<1, kSmallThreads, 0, s>>>(mask, T, cu_seqlens, B, counts);
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_weights_mode(const float *lp_w, const float *lp_inf,
                                       const uint8_t *mask, int64_t T, const DevParams &P,
                                       float *w_out, uint8_t *trunc_out, float *eps_out,
                                       cudaStream_t s)
{
    auto off = [](const void *p, uintptr_t n) { return reinterpret_cast<uintptr_t>(p) & (n - 1); };
    // below this the SMs want the threads: T=40000 takes 1.9 us with one token each,
    // 2.9 with four; T=150000 2.5, 2.8; T=4000000 36, 22 (CIS)
    const bool vec = T >= (1 << 18) && !off(lp_w, 16) && !off(lp_inf, 16) && !off(w_out, 16) &&
                     !off(eps_out, 16) && !off(mask, 4) && !off(trunc_out, 4);
    int64_t blocks = (vec ? T / 4 : T) / 256 + 1;
    if (blocks > 4096)
        blocks = 4096;
    if (vec)
        cis_weights_kernel<MODE, 4><<<(unsigned)blocks, 256, 0, s>>>(lp_w, lp_inf, mask, T, P,
                                                                     w_out, trunc_out, eps_out);
    else
        cis_weights_kernel<MODE, 1><<<(unsigned)blocks, 256, 0, s>>>(lp_w, lp_inf, mask, T, P,
                                                                     w_out, trunc_out, eps_out);
    return cudaGetLastError();
}

cudaError_t launch_weights(const float *lp_w, const float *lp_inf, const uint8_t *mask,
                           int64_t T, const DevParams &P, float *w_out, uint8_t *trunc_out,
                           float *eps_out, cudaStream_t s)
{
    if (T == 0)
        return cudaSuccess;
#define CIS_WEIGHTS_CASE(M) \
    case M: return launch_weights_mode<M>(lp_w, lp_inf, mask, T, P, w_out, trunc_out, eps_out, s);
    switch (P.mode) {
        CIS_WEIGHTS_CASE(CIS_MODE_CIS)
        CIS_WEIGHTS_CASE(CIS_MODE_TIS)
        CIS_WEIGHTS_CASE(CIS_MODE_EXACT)
        CIS_WEIGHTS_CASE(CIS_MODE_BAND)
        CIS_WEIGHTS_CASE(CIS_MODE_ICEPOP)
        CIS_WEIGHTS_CASE(CIS_MODE_KPOP)
        CIS_WEIGHTS_CASE(CIS_MODE_SEQ_TIS)  // (and Seq-MIS: the response's weight comes after)
    case CIS_MODE_SEQ_MIS:
        return launch_weights_mode<CIS_MODE_SEQ_TIS>(lp_w, lp_inf, mask, T, P, w_out, trunc_out,
                                                     eps_out, s);
    default:
        return launch_weights_mode<CIS_MODE_NONE>(lp_w, lp_inf, mask, T, P, w_out, trunc_out,
                                                  eps_out, s);
    }
#undef CIS_WEIGHTS_CASE
}

cudaError_t launch_reduce(const PassArgs &a, cis_stats_t *stats, double *loss, cudaStream_t s)
{
    if (a.red_parts == nullptr || a.red_ticket == nullptr)
        return cudaErrorInvalidValue;
    static_assert(sizeof(RedPart) <= kRedPartBytes, "a partial sum must fit its slot");
    const int64_t blocks = a.T > 0 ? (a.T + kRedTokens - 1) / kRedTokens : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kRedTokens);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];  // it waits for the kernel before it itself
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = a.overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, cis_reduce_kernel, a.mask, a.T,
                              static_cast<const double *>(a.ws_terms),
                              static_cast<const float *>(a.ws_logk),
                              static_cast<const float *>(a.ws_w),
                              static_cast<const uint8_t *>(a.ws_trunc),
                              static_cast<const float *>(a.entropy_out),
                              static_cast<const int32_t *>(a.status),
                              static_cast<RedPart *>(a.red_parts), a.red_ticket, stats, loss);
}

cudaError_t launch_seq_weights(const double *lw64, const float *lw32, const float *lp_inf,
                               const int32_t *ids, int64_t V, const uint8_t *mask,
                               const int32_t *cu_seqlens, int64_t B, int64_t T,
                               const DevParams &P, float *w, uint8_t *trunc, cudaStream_t s)
{
    if (B <= 0 || T <= 0)
        return cudaSuccess;
    if (B > 0x7fffffffLL)
        return cudaErrorInvalidValue;
    cis_seq_weights_kernel<<<(unsigned)B, kSeqThreads, 0, s>>>(lw64, lw32, lp_inf, ids, V, mask,
                                                                cu_seqlens, T, P, w, trunc);
    return cudaGetLastError();
}

}  // namespace cis

