// psort_radix32.cu -- the radix block sort of 32-bit keys.
#include "psort_radix_run.cuh"

namespace ps {
int run_radix_u32(const SortArgs& a, char* ws, size_t cap) { return Radix<uint32_t>::run(a, ws, cap); }
size_t radix_bytes_u32(const SortArgs& a) { return Radix<uint32_t>::layout(a).total; }
int viol_read_radix_u32(unsigned long long* out) { return rx_viol_read(out); }
}  // namespace ps
