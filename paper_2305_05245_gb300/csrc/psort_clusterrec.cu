// psort_clusterrec.cu -- one-launch sorts of (uint64 key, uint32 payload) records.
#include "psort_cluster_run.cuh"

namespace ps {
int run_cluster_rec(const SortArgs& a) { return ClusterSort<Rec>::run(a); }
}  // namespace ps
