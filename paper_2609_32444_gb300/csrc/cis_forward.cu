// cis_forward.cu -- log p of the sampled tokens (cis_token_logprobs, and the
// first sweep of the sequence operators): one read of the logits, any layout.
//
// Bound: HBM for many rows (V entries read once, 12 bytes written a row), the
// latency of one row for few.  A row is read straight into registers with
// aligned 16-byte loads, kBatch of them in flight per thread; nothing is
// staged, since nothing is read twice.  The entries before the first 16-byte
// boundary and after the last one (rows of an odd V) are read one by one.
// Per batch a thread takes one maximum (bf16 entries compared in pairs), moves
// its offset at most once, and then spends per entry an unpack, half a packed
// FMA, an exponential and half a packed add:
//   S = sum 2^{z log2e - c},  c = fl(m log2e),
// the rounding residual of c being taken out once at the end.  The thread
// whose vector holds the sampled entry y puts -inf there, so the sums run over
// j != y (see cis_common.cuh for why).
//
// Few rows: the CTAs of a cluster share a row (fwd_plan), each leaving its
// (max, sum) in the shared memory of the cluster's first CTA, which finishes
// the row.
//
// Before (one 256-thread CTA a row, a maximum and 9 instructions an entry more
// per 8 entries, entries of unaligned rows one by one): T=8192, V=151936 took
// 508 us, with the entropy 807; T=24 33 us; T=2000, V=32003 63.5 us, now 25.
#include "cis_dsmem.cuh"
#include "cis_kernels.h"

namespace cis {
namespace {

constexpr int kBatch = 4;  // 16-byte loads in flight per thread

// Running (m, S[, U]) of one thread in the exponent form above; U = sum e x with
// x = z log2e - c.  With |m| >= kHugeLogit x = (z - m) log2e and c is not used.
template <bool kEnt> struct ExpAcc {
    float m = -INFINITY, c = -INFINITY, S = 0.0f, U = 0.0f;

    __device__ __forceinline__ bool fast() const { return fabsf(m) < kHugeLogit; }
    // Raise the offset to a larger (or NaN) maximum.
    __device__ __forceinline__ void raise(float mx)
    {
        if (mx > m || mx != mx) {
            const float c1 = mx * kLog2e;
            const float d = fast() && fabsf(mx) < kHugeLogit ? c - c1 : (m - mx) * kLog2e;
            const float f = ex2_ftz(d);
            if (kEnt)
                U = f == 0.0f ? 0.0f : fmaf(d, S, U) * f;
            S = f == 0.0f ? 0.0f : S * f;
            m = mx;
            c = c1;
        }
    }
    // Add 8 entries (those left out are -inf); the offset covers them.
    __device__ __forceinline__ void add8(const float2 (&z)[4])
    {
        const float2 l2 = make_float2(kLog2e, kLog2e), nc = make_float2(-c, -c);
        float2 e[4], u = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 x = __ffma2_rn(z[i], l2, nc);
            e[i] = make_float2(ex2_ftz(x.x), ex2_ftz(x.y));
            if (kEnt)  // an entry at -inf adds 0, not 0 * -inf
                u = __ffma2_rn(e[i], make_float2(fmaxf(x.x, -1024.0f), fmaxf(x.y, -1024.0f)), u);
        }
        const float2 s = __fadd2_rn(__fadd2_rn(e[0], e[1]), __fadd2_rn(e[2], e[3]));
        S += s.x + s.y;
        if (kEnt)
            U += u.x + u.y;
    }
    // One entry, covered by the offset, in either form.
    __device__ __forceinline__ void add_entry(float z)
    {
        const float x = fast() ? fmaf(z, kLog2e, -c) : (z - m) * kLog2e, e = ex2_ftz(x);
        S += e;
        if (kEnt)
            U = fmaf(e, fmaxf(x, -1024.0f), U);
    }
    // As sums of e^{z - m}: the residual of c is exact (an FMA).
    __device__ __forceinline__ MaxSumU result() const
    {
        if (m == -INFINITY)
            return {m, 0.0f, 0.0f};
        const float err = fast() ? fmaf(m, kLog2e, -c) : 0.0f, f = ex2_ftz(-err);
        return {m, S * f, kEnt ? f * kLn2 * fmaf(-err, S, U) : 0.0f};
    }
};

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
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const uint4 q = v[k].q;
        const float2 z[4] = {make_float2(bf16_lo(q.x), bf16_hi(q.x)),
                             make_float2(bf16_lo(q.y), bf16_hi(q.y)),
                             make_float2(bf16_lo(q.z), bf16_hi(q.z)),
                             make_float2(bf16_lo(q.w), bf16_hi(q.w))};
        acc.add8(z);
    }
}
template <bool kEnt, int N>
__device__ __forceinline__ void add_vecs(ExpAcc<kEnt> &acc, const Vec<float> (&v)[N])
{
    const float2 none = make_float2(-INFINITY, -INFINITY);
#pragma unroll
    for (int k = 0; k < N; k += 2) {
        const uint4 a = v[k].q, b = v[k + 1 < N ? k + 1 : k].q;
        const float2 z[4] = {make_float2(__uint_as_float(a.x), __uint_as_float(a.y)),
                             make_float2(__uint_as_float(a.z), __uint_as_float(a.w)),
                             k + 1 < N ? make_float2(__uint_as_float(b.x), __uint_as_float(b.y))
                                       : none,
                             k + 1 < N ? make_float2(__uint_as_float(b.z), __uint_as_float(b.w))
                                       : none};
        acc.add8(z);
    }
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

template <bool kEnt, int NT> struct FwdShared {
    MaxSumU part[kMaxCluster];  // the cluster's CTAs, in its first CTA
    MaxSumU redu[kEnt ? NT / 32 : 1];
    MaxSum red[kEnt ? 1 : NT / 32];
};

// A cluster of `cs` CTAs per row.
template <typename InT, bool kEnt, int NT>
__global__ void __launch_bounds__(NT) cis_logprob_kernel(const PassArgs a, unsigned cs)
{
    constexpr int EV = Vec<InT>::kN;
    __shared__ FwdShared<kEnt, NT> sh;
    const int64_t t = blockIdx.x / cs;
    const unsigned rank = blockIdx.x - (unsigned)t * cs;
    const int tid = threadIdx.x;
    const bool valid = a.mask == nullptr || a.mask[t] != 0;
    const int64_t y = a.ids[t];
    if (!valid || y < 0 || y >= a.V) {  // same branch in every CTA of the row
        if (rank == 0 && tid == 0) {
            const float lp = valid ? NAN : 0.0f;
            if (valid)
                set_status(a.status, kStatusBadId);
            if (a.lp_out) a.lp_out[t] = lp;
            if (a.lse_out) a.lse_out[t] = lp;
            if (a.lp64_out) a.lp64_out[t] = lp;
            if (kEnt) a.entropy_out[t] = lp;
        }
        return;
    }
    if (cs > 1)
        cluster_arrive_relaxed();  // waited for before the first store to a peer

    const InT *row = reinterpret_cast<const InT *>(a.logits) + t * a.ld;
    const float zy = to_f32(row[y]);
    const int V = (int)a.V;
    int head = (int)((16 - (reinterpret_cast<uintptr_t>(row) & 15)) & 15) / (int)sizeof(InT);
    head = head < V ? head : V;
    const int nvec = (V - head) / EV;
    const int v0 = (int)((int64_t)nvec * rank / cs), v1 = (int)((int64_t)nvec * (rank + 1) / cs);
    const uint4 *rv = reinterpret_cast<const uint4 *>(row + head);
    // the vector and the entry in it that hold y (none: vy is negative or past
    // the body)
    const int yb = (int)y - head;
    const int vy = yb >= 0 ? yb / EV : -1, iy = yb - vy * EV;

    ExpAcc<kEnt> acc;
    int v = v0 + tid;
    for (; v + (kBatch - 1) * NT < v1; v += kBatch * NT) {
        Vec<InT> x[kBatch];
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
            x[k].q = __ldcs(rv + v + k * NT);
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
            if (v + k * NT == vy)
                x[k].drop(iy);
        take<kEnt, kBatch>(acc, x);
    }
    if (v < v1) {  // the last, partial batch: absent vectors count as -inf
        Vec<InT> x[kBatch];
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
            x[k].q = v + k * NT < v1 ? __ldcs(rv + v + k * NT)
                                     : make_uint4(Vec<InT>::kNone, Vec<InT>::kNone,
                                                  Vec<InT>::kNone, Vec<InT>::kNone);
#pragma unroll
        for (int k = 0; k < kBatch; ++k)
            if (v + k * NT == vy)
                x[k].drop(iy);
        take<kEnt, kBatch>(acc, x);
    }
    if (rank == 0) {  // the ragged ends: fewer than 2 EV entries
        const int tail0 = head + nvec * EV;
        int j = -1;
        if (tid < head)
            j = tid;
        else if (tid - head < V - tail0)
            j = tail0 + tid - head;
        if (j >= 0 && j != (int)y) {
            const float z = to_f32(row[j]);
            acc.raise(z);
            if (acc.m != -INFINITY)
                acc.add_entry(z);
        }
    }
    MaxSumU o = acc.result();
    if constexpr (kEnt) {
        o = block_msu<NT, false>(o, sh.redu);
    } else {
        const MaxSum ms = block_ms<NT, false>(MaxSum{o.m, o.s}, sh.red);
        o = MaxSumU{ms.m, ms.s, 0.0f};
    }
    if (cs > 1) {
        cluster_wait();  // every CTA of the row has started
        if (tid == 0) {
            const uint32_t dst = map_rank(smem_u32(&sh.part[rank]), 0);
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst), "f"(o.m) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + 4), "f"(o.s) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + 8), "f"(o.u) : "memory");
        }
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (rank != 0)
            return;
        if (tid == 0) {  // in rank order
            o = sh.part[0];
            for (unsigned r = 1; r < cs; ++r) {
                if constexpr (kEnt) {
                    o = msu_combine(o, sh.part[r]);
                } else {
                    const MaxSum ms = ms_combine(MaxSum{o.m, o.s},
                                                 MaxSum{sh.part[r].m, sh.part[r].s});
                    o = MaxSumU{ms.m, ms.s, 0.0f};
                }
            }
        }
    }
    if (tid == 0) {
        const RowScalars rs = row_scalars(MaxSum{o.m, o.s}, zy);
        if (kEnt) a.entropy_out[t] = row_entropy(o, zy, rs.lp);
        if (a.lp_out) a.lp_out[t] = rs.lp;
        if (a.lse_out) a.lse_out[t] = rs.lse;
        if (a.lp64_out) a.lp64_out[t] = rs.lp64();
    }
}

// CTAs per row and their width, all measured with bf16 rows.
// - 256 threads and 4 loads in flight: T=8192, V=151936 takes 346 us (7.2 TB/s),
//   with the entropy 364; 128 threads 354 / 361, 512 threads 365 / 480, 2 loads
//   357 / 376, 8 loads 350 / 371.
// - 64 threads for rows of at most 512 vectors, which 256 threads would not fill
//   once: T=16384, V=4096 takes 26.6 us against 71.6.
// - 128 threads where 256 would leave a last, part-empty round of rows among few
//   (8 CTAs an SM, up to four rounds): T=2048, V=151936, a quarter masked, takes
//   81.7 us against 92.8; T=2000, V=32003 23.5 against 25.7.
// - A row is split over a cluster only while the clusters' CTAs stay within 608
//   (four a SM), since the exchange costs more than it gives once the SMs are
//   busy: V=151936 takes 33.2 us against 37.7 (one CTA a row, two) at T=512, 11.6
//   against 13.2 (four, eight) at T=128, and 5.8 against 33 for one CTA a row of
//   the kernel before at T=24.  A CTA keeps at least 512 vectors.
struct FwdPlan {
    int cs, nt;
};
FwdPlan fwd_plan(int64_t T, int64_t V, int in_bytes)
{
    const int64_t nvec = V * in_bytes / 16;
    FwdPlan p{1, nvec <= 512 ? 64 : (T > 1216 && T <= 4864 ? 128 : 256)};
    while (p.cs < kMaxCluster && T * p.cs * 2 <= 608 && nvec / (2 * p.cs) >= 512)
        p.cs *= 2;
    return p;
}

template <typename InT, bool kEnt, int NT>
cudaError_t launch_fwd(const PassArgs &a, int cs, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.T * cs), 1, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cs > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, cis_logprob_kernel<InT, kEnt, NT>, a, (unsigned)cs);
}

template <typename InT> cudaError_t launch_fwd_t(const PassArgs &a, cudaStream_t s)
{
    const FwdPlan p = fwd_plan(a.T, a.V, (int)sizeof(InT));
    const bool ent = a.entropy_out != nullptr;
    switch (p.nt) {
    case 64: return ent ? launch_fwd<InT, true, 64>(a, p.cs, s)
                        : launch_fwd<InT, false, 64>(a, p.cs, s);
    case 128: return ent ? launch_fwd<InT, true, 128>(a, p.cs, s)
                         : launch_fwd<InT, false, 128>(a, p.cs, s);
    default: return ent ? launch_fwd<InT, true, 256>(a, p.cs, s)
                        : launch_fwd<InT, false, 256>(a, p.cs, s);
    }
}

}  // namespace

cudaError_t launch_token_logprobs(const PassArgs &a, int dtype, cudaStream_t s)
{
    if (a.T == 0)
        return cudaSuccess;
    return dtype == CIS_BF16 ? launch_fwd_t<__nv_bfloat16>(a, s) : launch_fwd_t<float>(a, s);
}

}  // namespace cis
