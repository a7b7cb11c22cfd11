// cis_cluster_ragged.cu -- the cluster kernel's launches for rows of any alignment
// and any V (T=4096, V=32003 bf16, a quarter masked: 78 us against 252 for
// one CTA a row reading entry by entry, twice).
#include "cis_cluster.cuh"

namespace cis {
namespace {

template <typename InT, typename OutT> struct Ragged {
    static cudaError_t run(const PassArgs &a, const ClusterPlan &p, cudaStream_t s)
    {
        if (a.entropy_out)
            return launch_cluster_ent<InT, OutT, true, Ops::kPlain>(a, p, s);
        return p.nt == 128 ? launch_cluster_nt<InT, OutT, 128, false, true, Ops::kPlain>(a, p, s)
                           : launch_cluster_nt<InT, OutT, 256, false, true, Ops::kPlain>(a, p, s);
    }
};

}  // namespace

cudaError_t launch_cluster_ragged(const PassArgs &a, int dtype, int out_dtype,
                                  const ClusterPlan &p, cudaStream_t s)
{
    return by_type<Ragged>(dtype, out_dtype, a, p, s);
}

}  // namespace cis
