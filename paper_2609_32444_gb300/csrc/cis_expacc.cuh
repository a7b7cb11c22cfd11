// cis_expacc.cuh -- sums of exponentials over one row read straight into
// registers with aligned 16-byte loads (the forward kernel, the diagnostics).
//
// Per batch of vectors a thread takes one maximum (bf16 entries compared in
// pairs), moves its offset at most once, and then spends per entry an unpack,
// half a packed FMA, an exponential and half a packed add:
//   S = sum 2^{z log2e - c},  c = ceil(m log2e),
// with whole c, so that sums move between offsets by exact powers of two: the
// exponential instruction's error is one-sided (-4.9e-8 on average, measured), and a
// term that is rescaled on its way through threads and warps by it picks that up
// several times, the same way in every row.
#pragma once

#include "cis_common.cuh"

namespace cis {
namespace {

// 2^x for -1/8 < x < 9/8, to fp32 rounding.
__device__ __forceinline__ float exp2_accurate(float x)
{
    constexpr float ln2_lo = (float)(0.693147180559945309417 - (double)kLn2);
    const bool up = x > 0.5f;
    const float y = up ? x - 1.0f : x, h = y * kLn2;  // exact, then 2^x = (2) e^{y ln 2}
    float lo;
    const float hi = exp_pair(h, fmaf(y, kLn2, -h) + y * ln2_lo, lo);
    return up ? 2.0f * (hi + lo) : hi + lo;
}

// Running (m, S[, U]) of one thread in the exponent form above; U = sum e x with
// x = z log2e - c.  With |m| >= kHugeLogit x = (z - m) log2e and c is not used.
template <bool kEnt> struct ExpAcc {
    float m = -INFINITY, c = -INFINITY, S = 0.0f, U = 0.0f;

    __device__ __forceinline__ bool fast() const { return fabsf(m) < kHugeLogit; }
    // Raise the offset to a larger (or NaN) maximum, in whichever of the two forms
    // each of the maxima has.
    __device__ __forceinline__ void raise(float mx)
    {
        if (mx > m || mx != mx) {
            const float c1 = ceilf(mx * kLog2e);
            const bool now = fast(), then = fabsf(mx) < kHugeLogit;
            const float d = now ? (then ? c - c1 : fmaf(-mx, kLog2e, c))
                                : (then ? fmaf(m, kLog2e, -c1) : (m - mx) * kLog2e);
            const float f = ex2_ftz(d);
            if (kEnt)
                U = f == 0.0f ? 0.0f : fmaf(d, S, U) * f;
            S = f == 0.0f ? 0.0f : S * f;
            m = mx;
            c = c1;
        }
    }
    // The sum of 8 entries (those left out are -inf), as a pair, and of e x in u; the
    // offset covers them.
    __device__ __forceinline__ float2 sum8(const float2 (&z)[4], float2 &u) const
    {
        const float2 l2 = make_float2(kLog2e, kLog2e), nc = make_float2(-c, -c);
        float2 e[4];
        u = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 x = __ffma2_rn(z[i], l2, nc);
            e[i] = make_float2(ex2_ftz(x.x), ex2_ftz(x.y));
            if (kEnt)  // an entry at -inf adds 0, not 0 * -inf
                u = __ffma2_rn(e[i], make_float2(fmaxf(x.x, -1024.0f), fmaxf(x.y, -1024.0f)), u);
        }
        return __fadd2_rn(__fadd2_rn(e[0], e[1]), __fadd2_rn(e[2], e[3]));
    }
    // Add N such sums, to each other first: the growing sum is rounded at each addition,
    // and next to one large entry a thread's many small ones are lost to it, the more the
    // smaller they come (V=151936, a likely token and another one sampled: log p off by
    // 1.1e-7 on average; 3.4e-7 a vector at a time).
    template <int N> __device__ __forceinline__ void grow(float2 (&s)[N], float2 (&u)[N])
    {
#pragma unroll
        for (int w = 1; w < N; w <<= 1)
#pragma unroll
            for (int k = 0; k + w < N; k += 2 * w) {
                s[k] = __fadd2_rn(s[k], s[k + w]);
                if (kEnt)
                    u[k] = __fadd2_rn(u[k], u[k + w]);
            }
        S += s[0].x + s[0].y;
        if (kEnt)
            U += u[0].x + u[0].y;
    }
    // One entry, covered by the offset, in either form.
    __device__ __forceinline__ void add_entry(float z)
    {
        const float x = fast() ? fmaf(z, kLog2e, -c) : (z - m) * kLog2e, e = ex2_ftz(x);
        S += e;
        if (kEnt)
            U = fmaf(e, fmaxf(x, -1024.0f), U);
    }
    // As sums of e^{z - m}: m log2e - c is exact (an FMA), between -1 and 0 but
    // for the rounding of the product that c was taken from (2^-4 at most): above 0
    // where that product was rounded down to a whole number.
    __device__ __forceinline__ MaxSumU result() const
    {
        if (m == -INFINITY)
            return {m, 0.0f, 0.0f};
        const float err = fast() ? fmaf(m, kLog2e, -c) : 0.0f;
        const float f = fast() ? exp2_accurate(-err) : 1.0f;
        return {m, S * f, kEnt ? f * kLn2 * fmaf(-err, S, U) : 0.0f};
    }
};

// The CTA's threads' sums together, as sums of e^{z - m}; every thread gets them.
// red: NT / 32 slots.
template <int NT, bool kEnt>
__device__ __forceinline__ MaxSumU block_exp(const ExpAcc<kEnt> &acc, MaxSumU *red)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float M = acc.m;  // (a NaN is kept by its thread's sum)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    if (lane == 0)
        red[wid].m = M;
    __syncthreads();
    M = red[0].m;
#pragma unroll
    for (int w = 1; w < NT / 32; ++w)
        M = fmaxf(M, red[w].m);
    ExpAcc<kEnt> all;
    all.m = M;
    all.c = ceilf(M * kLog2e);
    if (M == -INFINITY)
        all.c = 0.0f;  // no entry: every sum is 0, or NaN
    // This thread's sums at the common offset: an exact power of two where both are
    // fast; a thread whose entries are all masked ones counts as 0.
    MaxSumU t = acc.result();
    float d, f;
    if (all.fast()) {
        d = acc.fast() ? acc.c - all.c : fmaf(acc.m, kLog2e, -all.c);
        t.s = acc.S;
        t.u = acc.U;
    } else {
        d = acc.m == -INFINITY ? -INFINITY : (acc.m - M) * kLog2e;
        t.u *= kLog2e;
    }
    f = ex2_ftz(d);
    float s = t.s * f, u = kEnt ? fmaf(fmaxf(d, -1e30f), t.s, t.u) * f : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        if (kEnt)
            u += __shfl_xor_sync(0xffffffffu, u, o);
    }
    if (lane == 0) {
        red[wid].s = s;
        red[wid].u = u;
    }
    __syncthreads();
    all.S = red[0].s;
    all.U = red[0].u;
#pragma unroll
    for (int w = 1; w < NT / 32; ++w) {
        all.S += red[w].s;
        all.U += red[w].u;
    }
    if (M == -INFINITY)
        return {M, all.S, all.U};
    MaxSumU o = all.result();
    if (!all.fast() && kEnt)
        o.u = all.U * kLn2;
    return o;
}

// One 16-byte vector: 8 bf16 or 4 fp32 entries.
template <typename InT> struct Vec;
template <> struct Vec<__nv_bfloat16> {
    static constexpr int kN = 8;
    static constexpr uint32_t kNone = 0xff80ff80u;  // entries at -inf
    uint4 q;
    __device__ __forceinline__ float entry(int i) const
    {
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
        return (i & 1) ? bf16_hi(w[i >> 1]) : bf16_lo(w[i >> 1]);
    }
    __device__ __forceinline__ void drop(int i)  // entry i to -inf
    {
        uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if ((i >> 1) == k)
                w[k] = (i & 1) ? (w[k] & 0x0000ffffu) | 0xff800000u
                               : (w[k] & 0xffff0000u) | 0x0000ff80u;
        q = make_uint4(w[0], w[1], w[2], w[3]);
    }
};
template <> struct Vec<float> {
    static constexpr int kN = 4;
    static constexpr uint32_t kNone = 0xff800000u;
    uint4 q;
    __device__ __forceinline__ float entry(int i) const
    {
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
        return __uint_as_float(w[i]);
    }
    __device__ __forceinline__ void drop(int i)
    {
        const uint32_t ninf = 0xff800000u;
        q.x = i == 0 ? ninf : q.x;
        q.y = i == 1 ? ninf : q.y;
        q.z = i == 2 ? ninf : q.z;
        q.w = i == 3 ? ninf : q.w;
    }
};

__device__ __forceinline__ __nv_bfloat162 as_bf2(uint32_t w)
{
    return *reinterpret_cast<const __nv_bfloat162 *>(&w);
}

// Maximum of N vectors (NaN propagates).
template <int N> __device__ __forceinline__ float vec_max(const Vec<__nv_bfloat16> (&v)[N])
{
    __nv_bfloat162 a = __hmax2_nan(as_bf2(v[0].q.x), as_bf2(v[0].q.y));
    __nv_bfloat162 b = __hmax2_nan(as_bf2(v[0].q.z), as_bf2(v[0].q.w));
#pragma unroll
    for (int k = 1; k < N; ++k) {
        a = __hmax2_nan(a, __hmax2_nan(as_bf2(v[k].q.x), as_bf2(v[k].q.y)));
        b = __hmax2_nan(b, __hmax2_nan(as_bf2(v[k].q.z), as_bf2(v[k].q.w)));
    }
    a = __hmax2_nan(a, b);
    return max_nan(__low2float(a), __high2float(a));
}
template <int N> __device__ __forceinline__ float vec_max(const Vec<float> (&v)[N])
{
    float m = -INFINITY;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        m = max_nan(m, max_nan(__uint_as_float(v[k].q.x), __uint_as_float(v[k].q.y)));
        m = max_nan(m, max_nan(__uint_as_float(v[k].q.z), __uint_as_float(v[k].q.w)));
    }
    return m;
}

template <bool kEnt, int N>
__device__ __forceinline__ void add_vecs(ExpAcc<kEnt> &acc, const Vec<__nv_bfloat16> (&v)[N])
{
    float2 s[N], u[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const uint4 q = v[k].q;
        const float2 z[4] = {make_float2(bf16_lo(q.x), bf16_hi(q.x)),
                             make_float2(bf16_lo(q.y), bf16_hi(q.y)),
                             make_float2(bf16_lo(q.z), bf16_hi(q.z)),
                             make_float2(bf16_lo(q.w), bf16_hi(q.w))};
        s[k] = acc.sum8(z, u[k]);
    }
    acc.grow(s, u);
}
template <bool kEnt, int N>
__device__ __forceinline__ void add_vecs(ExpAcc<kEnt> &acc, const Vec<float> (&v)[N])
{
    const float2 none = make_float2(-INFINITY, -INFINITY);
    float2 s[(N + 1) / 2], u[(N + 1) / 2];
#pragma unroll
    for (int k = 0; k < N; k += 2) {
        const uint4 a = v[k].q, b = v[k + 1 < N ? k + 1 : k].q;
        const float2 z[4] = {make_float2(__uint_as_float(a.x), __uint_as_float(a.y)),
                             make_float2(__uint_as_float(a.z), __uint_as_float(a.w)),
                             k + 1 < N ? make_float2(__uint_as_float(b.x), __uint_as_float(b.y))
                                       : none,
                             k + 1 < N ? make_float2(__uint_as_float(b.z), __uint_as_float(b.w))
                                       : none};
        s[k / 2] = acc.sum8(z, u[k / 2]);
    }
    acc.grow(s, u);
}

template <bool kEnt, int N, typename InT>
__device__ __forceinline__ void take(ExpAcc<kEnt> &acc, const Vec<InT> (&v)[N])
{
    acc.raise(vec_max<N>(v));
    if (acc.fast()) {
        add_vecs<kEnt, N>(acc, v);
    } else if (acc.m != -INFINITY) {
#pragma unroll
        for (int k = 0; k < N; ++k)
#pragma unroll
            for (int i = 0; i < Vec<InT>::kN; ++i)
                acc.add_entry(v[k].entry(i));
    }
}

// Where row's 16-byte vectors lie: the entries before the first whole one, and
// the number of whole ones.
template <typename InT>
__device__ __forceinline__ int row_head(const InT *row, int V)
{
    const int head =
        (int)((16 - (reinterpret_cast<uintptr_t>(row) & 15)) & 15) / (int)sizeof(InT);
    return head < V ? head : V;
}

}  // namespace
}  // namespace cis
