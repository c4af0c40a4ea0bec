// psort_cluster32.cu -- one-launch sorts of 32-bit keys.
#include "psort_cluster_run.cuh"

namespace ps {
int run_cluster_u32(const SortArgs& a) { return ClusterSort<uint32_t>::run(a); }
}  // namespace ps
