// psort_cluster64.cu -- one-launch sorts of 64-bit keys.
#include "psort_cluster_run.cuh"

namespace ps {
int run_cluster_u64(const SortArgs& a) { return ClusterSort<uint64_t>::run(a); }
template <>
cudaError_t cluster_blocks<uint64_t>(int xf, const GBuf<uint64_t>& src, const GBuf<uint64_t>& dst, const Inst& in, int64_t n_B, int64_t L,
                               cudaStream_t s)
{
    return ClusterSort<uint64_t>::blocks(xf, src, dst, in, n_B, L, s);
}
}  // namespace ps
