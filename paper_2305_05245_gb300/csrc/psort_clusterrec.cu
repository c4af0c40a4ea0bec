// psort_clusterrec.cu -- one-launch sorts of (uint64 key, uint32 payload) records.
#include "psort_cluster_run.cuh"

namespace ps {
int run_cluster_rec(const SortArgs& a) { return ClusterSort<Rec>::run(a); }
template <>
cudaError_t cluster_blocks<Rec>(int xf, const GBuf<Rec>& src, const GBuf<Rec>& dst, const Inst& in, int64_t n_B, int64_t L,
                               cudaStream_t s)
{
    return ClusterSort<Rec>::blocks(xf, src, dst, in, n_B, L, s);
}
}  // namespace ps
