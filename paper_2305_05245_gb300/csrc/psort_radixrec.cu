// psort_radixrec.cu -- the radix block sort of (uint64 key, uint32 payload) records.
#include "psort_radix_run.cuh"

namespace ps {
int run_radix_rec(const SortArgs& a) { return Radix<Rec>::run(a); }
size_t radix_bytes_rec(const SortArgs& a) { return Radix<Rec>::layout(a).total; }
int viol_read_radix_rec(unsigned long long* out) { return rx_viol_read(out); }
}  // namespace ps
