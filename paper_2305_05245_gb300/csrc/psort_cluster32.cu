// psort_cluster32.cu -- one-launch sorts of 32-bit keys.
#include "psort_cluster_run.cuh"

namespace ps {
int run_cluster_u32(const SortArgs& a) { return ClusterSort<uint32_t>::run(a); }
template <>
cudaError_t cluster_blocks<uint32_t>(int xf, const GBuf<uint32_t>& src, const GBuf<uint32_t>& dst, const Inst& in, int64_t n_B, int64_t L,
                               cudaStream_t s)
{
    return ClusterSort<uint32_t>::blocks(xf, src, dst, in, n_B, L, s);
}
}  // namespace ps
