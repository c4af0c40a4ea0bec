// psort_cluster64.cu -- one-launch sorts of 64-bit keys.
#include <atomic>

#include "psort_cluster_run.cuh"

namespace ps {
int run_cluster_u64(const SortArgs& a) { return ClusterSort<uint64_t>::run(a); }
template <>
cudaError_t cluster_blocks<uint64_t>(int xf, const GBuf<uint64_t>& src, const GBuf<uint64_t>& dst, const Inst& in, int64_t n_B, int64_t L,
                               cudaStream_t s)
{
    return ClusterSort<uint64_t>::blocks(xf, src, dst, in, n_B, L, s);
}

static std::atomic<int> g_placeable[64], g_cap{0};  // asked once per device; 0: not yet, no cap
void cluster_debug_cap(int ctas) { g_cap.store(ctas); }
int cluster_placeable()
{
    const int cap = g_cap.load(std::memory_order_relaxed);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return cap ? cap : 16;  // (no device: what the target has)
    }
    int best = g_placeable[dev].load(std::memory_order_relaxed);
    if (best == 0) {
        for (best = 16; best > 1; best /= 2)
            if (ClusterSort<uint64_t>::placeable(best)) break;
        g_placeable[dev].store(best, std::memory_order_relaxed);
    }
    return cap && cap < best ? cap : best;
}
}  // namespace ps
