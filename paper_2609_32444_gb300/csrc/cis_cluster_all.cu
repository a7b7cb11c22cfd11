// cis_cluster_all.cu -- the cluster kernel's launches with every operator (the
// band, IcePop and KPop come here), for rows of any alignment.
#include "cis_cluster.cuh"

namespace cis {
namespace {

template <typename InT, typename OutT> struct AllAligned {
    static cudaError_t run(const PassArgs &a, const ClusterPlan &p, cudaStream_t s)
    {
        if (a.entropy_out)
            return launch_cluster_ent<InT, OutT, false, Ops::kAll>(a, p, s);
        return p.nt == 128 ? launch_cluster_nt<InT, OutT, 128, false, false, Ops::kAll>(a, p, s)
                           : launch_cluster_nt<InT, OutT, 256, false, false, Ops::kAll>(a, p, s);
    }
};

template <typename InT, typename OutT> struct AllRagged {
    static cudaError_t run(const PassArgs &a, const ClusterPlan &p, cudaStream_t s)
    {
        if (a.entropy_out)
            return launch_cluster_ent<InT, OutT, true, Ops::kAll>(a, p, s);
        return p.nt == 128 ? launch_cluster_nt<InT, OutT, 128, false, true, Ops::kAll>(a, p, s)
                           : launch_cluster_nt<InT, OutT, 256, false, true, Ops::kAll>(a, p, s);
    }
};

}  // namespace

cudaError_t launch_cluster_all(const PassArgs &a, int dtype, int out_dtype, bool aligned,
                               const ClusterPlan &p, cudaStream_t s)
{
    return aligned ? by_type<AllAligned>(dtype, out_dtype, a, p, s)
                   : by_type<AllRagged>(dtype, out_dtype, a, p, s);
}

}  // namespace cis
