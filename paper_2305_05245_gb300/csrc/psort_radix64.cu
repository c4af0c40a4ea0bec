// psort_radix64.cu -- the radix block sort of 64-bit keys.
#include "psort_radix_run.cuh"

namespace ps {
int run_radix_u64(const SortArgs& a, char* ws, size_t cap) { return Radix<uint64_t>::run(a, ws, cap); }
size_t radix_bytes_u64(const SortArgs& a) { return Radix<uint64_t>::layout(a).total; }
int viol_read_radix_u64(unsigned long long* out) { return rx_viol_read(out); }
}  // namespace ps
