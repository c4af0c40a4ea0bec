// psort_cluster64.cu -- one-launch sorts of 64-bit keys.
#include "psort_cluster_run.cuh"

namespace ps {
int run_cluster_u64(const SortArgs& a) { return ClusterSort<uint64_t>::run(a); }
}  // namespace ps
