// cis_cluster.cu -- the fused pass's fast path: cluster sizes and dispatch, and
// the launches for aligned rows (cis_cluster.cuh has the kernel).
#include <stdlib.h>

#include "cis_cluster.cuh"

namespace cis {
namespace {

// Whether the kernel's aligned form applies: whole groups of 8, every row of
// both tensors on a 16-byte boundary.
bool aligned_rows(const PassArgs &a, int ib, int ob)
{
    return a.V % 8 == 0 && (reinterpret_cast<uintptr_t>(a.logits) & 15) == 0 &&
           (a.ld * ib) % 16 == 0 && (reinterpret_cast<uintptr_t>(a.dz) & 15) == 0 &&
           (a.ld_out * ob) % 16 == 0;
}

int64_t slice_target_bytes()
{
    static int64_t v = [] {
        const char *e = getenv("CIS_SLICE_KB");
        long kb = e ? atol(e) : 80;
        if (kb < 8) kb = 8;
        if (kb > 200) kb = 200;
        return (int64_t)kb * 1024;
    }();
    return v;
}

// Cluster size forced for tuning sweeps (0: chosen from the slice target).
int forced_cluster()
{
    static int v = [] {
        const char *e = getenv("CIS_CLUSTER");
        const int c = e ? atoi(e) : 0;
        return (c >= 1 && c <= kMaxCluster) ? c : 0;
    }();
    return v;
}

// Smallest cluster size whose slices fit the target (any size 1..8).  Rows
// that fit one slice of the default 80 KB target but not one of 40 KB (a
// 32,000-entry bf16 row, for instance) run on two CTAs of 128 threads: at
// T=4096, V=32000 that took 106.6 us per step against 109.7 us for one CTA of
// 256 threads, and 256 threads on the two halves were slower still (122 us).
// Setting CIS_SLICE_KB or CIS_CLUSTER turns the rule off; CIS_CLUSTER_THREADS
// sets the width of its two CTAs.
bool make_plan(int64_t V, int in_bytes, ClusterPlan *p)
{
    const int64_t target = slice_target_bytes();
    const int forced = forced_cluster();
    for (int cs = forced ? forced : 1; cs <= kMaxCluster; ++cs) {
        const int64_t per = (V + cs - 1) / cs;
        const int64_t slice = (per + 7) / 8 * 8;
        if (forced || slice * in_bytes <= target || cs == kMaxCluster) {
            if (slice * in_bytes > 200 * 1024)
                return false;
            p->cs = cs;
            p->slice = slice;
            p->smem = (size_t)(slice * in_bytes) + 128;
            p->nt = 0;
            static const bool slice_set = getenv("CIS_SLICE_KB") != nullptr;
            if (!forced && !slice_set && cs == 1 && slice * in_bytes > 40 * 1024) {
                p->cs = 2;
                p->slice = ((V + 1) / 2 + 7) / 8 * 8;
                p->smem = (size_t)(p->slice * in_bytes) + 128;
                p->nt = 128;
            }
            return true;
        }
    }
    return false;
}

// CTA width forced for tuning sweeps (default 256 threads).
int cluster_threads()
{
    static int v = [] {
        const char *e = getenv("CIS_CLUSTER_THREADS");
        const int n = e ? atoi(e) : 256;
        return (n == 512 || n == 384 || n == 128) ? n : 256;
    }();
    return v;
}

// CTA width where make_plan leaves it open.  Short slices give 256 threads too
// little: with 128, more rows are on an SM at once (bf16, T=16384: V=1000 takes 57.6
// us against 84.8, V=4000 79 against 105; T=8192: V=16000 86 against 88, but V=20000
// 105.7 against 104.7, and V=151936 is 7% slower).  fp32 rows have half the entries
// a byte: 128 threads throughout (T=4096, V=151936: 718 us against 736; T=8192,
// V=1000: 28.6 against 43).
int plan_threads(const ClusterPlan &p, int in_bytes)
{
    return in_bytes == 4 || (p.cs == 1 && p.slice <= 16384) ? 128 : 256;
}

template <typename InT, typename OutT> struct Aligned {
    static cudaError_t run(const PassArgs &a, const ClusterPlan &p, cudaStream_t s)
    {
        if (a.entropy_out)
            return launch_cluster_ent<InT, OutT, false, Ops::kPlain>(a, p, s);
        switch (p.nt) {
        case 512: return launch_cluster_nt<InT, OutT, 512, false, false, Ops::kPlain>(a, p, s);
        case 384: return launch_cluster_nt<InT, OutT, 384, false, false, Ops::kPlain>(a, p, s);
        case 128: return launch_cluster_nt<InT, OutT, 128, false, false, Ops::kPlain>(a, p, s);
        default: return launch_cluster_nt<InT, OutT, 256, false, false, Ops::kPlain>(a, p, s);
        }
    }
};

}  // namespace

cudaError_t launch_cluster_aligned(const PassArgs &a, int dtype, int out_dtype,
                                   const ClusterPlan &p, cudaStream_t s)
{
    return by_type<Aligned>(dtype, out_dtype, a, p, s);
}

bool cluster_path_applies(const PassArgs &a, int dtype, int out_dtype)
{
    (void)out_dtype;
    if (a.T * 8 > 0x7fffffffLL)
        return false;
    ClusterPlan p;
    return make_plan(a.V, dtype == CIS_BF16 ? 2 : 4, &p);
}

cudaError_t launch_cluster_fwd_bwd(const PassArgs &a, int dtype, int out_dtype, cudaStream_t s)
{
    if (!cluster_path_applies(a, dtype, out_dtype))
        return cudaErrorNotSupported;
    if (a.T == 0)
        return cudaSuccess;
    ClusterPlan p;
    make_plan(a.V, dtype == CIS_BF16 ? 2 : 4, &p);
    static const bool width_set = getenv("CIS_CLUSTER_THREADS") != nullptr;
    if (p.nt == 0 || width_set)
        p.nt = width_set ? cluster_threads() : plan_threads(p, dtype == CIS_BF16 ? 2 : 4);
    const bool aligned = aligned_rows(a, dtype == CIS_BF16 ? 2 : 4, out_dtype == CIS_BF16 ? 2 : 4);
    const int m = a.P.mode;
    // the smallest variant that can do the call
    if (m == CIS_MODE_BAND || m == CIS_MODE_ICEPOP || m == CIS_MODE_KPOP)
        return launch_cluster_all(a, dtype, out_dtype, aligned, p, s);
    if (a.lp_old || a.w_in)
        return launch_cluster_given(a, dtype, out_dtype, aligned, p, s);
    return aligned ? launch_cluster_aligned(a, dtype, out_dtype, p, s)
                   : launch_cluster_ragged(a, dtype, out_dtype, p, s);
}

}  // namespace cis
