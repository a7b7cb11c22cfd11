// cis_forward.cu -- log p of the sampled tokens (cis_token_logprobs, and the
// first sweep of the sequence operators): one read of the logits, any layout.
//
// Bound: HBM for many rows (V entries read once, 12 bytes written a row), the
// latency of one row for few.  A row is read straight into registers with
// aligned 16-byte loads, kBatch of them in flight per thread; nothing is
// staged, since nothing is read twice.  The entries before the first 16-byte
// boundary and after the last one (rows of an odd V) are read one by one.
// cis_expacc.cuh has the sums.  The thread whose vector holds the sampled entry
// y puts -inf there, so the sums run over j != y (see cis_common.cuh for why).
//
// Few rows: the CTAs of a cluster share a row (fwd_plan), each leaving its
// (max, sum) in the shared memory of the cluster's first CTA, which finishes
// the row.
//
// Before (one 256-thread CTA a row, a maximum and 9 instructions an entry more
// per 8 entries, entries of unaligned rows one by one): T=8192, V=151936 took
// 508 us, with the entropy 807; T=24 33 us; T=2000, V=32003 63.5 us, now 25.
#include "cis_dsmem.cuh"
#include "cis_expacc.cuh"
#include "cis_kernels.h"

namespace cis {
namespace {

constexpr int kBatch = 4;  // 16-byte loads in flight per thread

template <bool kEnt, int NT> struct FwdShared {
    MaxSumU part[kMaxCluster];  // the cluster's CTAs, in its first CTA
    MaxSumU red[NT / 32];
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
    const int head = row_head(row, V);
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
    MaxSumU o = block_exp<NT>(acc, sh.red);
    if (cs > 1) {
        cluster_wait();  // every CTA of the row has started
        if (tid == 0) {
            const uint32_t dst = map_rank(smem_u32(&sh.part[rank]), 0);
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst), "f"(o.m) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + 4), "f"(o.s) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + 8), "f"(o.u) : "memory");
        }
        __syncwarp();
        cluster_sync_data();
        if (rank != 0)
            return;
        if (tid == 0) {  // in rank order
            float M = sh.part[0].m;
            for (unsigned r = 1; r < cs; ++r)
                M = fmaxf(M, sh.part[r].m);
            o = MaxSumU{M, 0.0f, 0.0f};
            for (unsigned r = 0; r < cs; ++r) {
                const MaxSumU q = sh.part[r];
                const float d = q.m == -INFINITY ? -INFINITY : q.m - M, f = expf(d);
                o.s += q.s * f;
                o.u += fmaf(fmaxf(d, -1e30f), q.s, q.u) * f;
            }
        }
    }
    if (tid == 0) {
        const RowScalars rs = row_scalars(MaxSum{o.m, o.s}, zy, a.lp64_out != nullptr);
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
