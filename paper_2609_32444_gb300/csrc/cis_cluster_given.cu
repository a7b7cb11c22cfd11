// cis_cluster_given.cu -- the cluster kernel's launches with l_old or a response's
// weight (CIS, TIS, exact, none and the sequence operators), for rows of any
// alignment.
#include "cis_cluster.cuh"

namespace cis {
namespace {

template <typename InT, typename OutT> struct GivenAligned {
    static cudaError_t run(const PassArgs &a, const ClusterPlan &p, cudaStream_t s)
    {
        if (a.entropy_out)
            return launch_cluster_ent<InT, OutT, false, Ops::kGiven>(a, p, s);
        return p.nt == 128 ? launch_cluster_nt<InT, OutT, 128, false, false, Ops::kGiven>(a, p, s)
                           : launch_cluster_nt<InT, OutT, 256, false, false, Ops::kGiven>(a, p, s);
    }
};

template <typename InT, typename OutT> struct GivenRagged {
    static cudaError_t run(const PassArgs &a, const ClusterPlan &p, cudaStream_t s)
    {
        if (a.entropy_out)
            return launch_cluster_ent<InT, OutT, true, Ops::kGiven>(a, p, s);
        return p.nt == 128 ? launch_cluster_nt<InT, OutT, 128, false, true, Ops::kGiven>(a, p, s)
                           : launch_cluster_nt<InT, OutT, 256, false, true, Ops::kGiven>(a, p, s);
    }
};

}  // namespace

cudaError_t launch_cluster_given(const PassArgs &a, int dtype, int out_dtype, bool aligned,
                               const ClusterPlan &p, cudaStream_t s)
{
    return aligned ? by_type<GivenAligned>(dtype, out_dtype, a, p, s)
                   : by_type<GivenRagged>(dtype, out_dtype, a, p, s);
}

}  // namespace cis
