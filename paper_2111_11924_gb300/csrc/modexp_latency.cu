// More lanes per instance for small, latency-bound batches: each product
// spreads over more lanes, so one exponentiation finishes sooner when there
// are too few chunks to fill the GPU (the 100 KB workload of Table 2 has
// 101-807).  CRT residues of 1024-, 2048-, 4096-, 6144- and 8192-bit keys and the
// full width of 512-, 1024- and 3072-bit keys; chosen by the size of a call.
#include "modexp_kernels.cuh"

namespace pmk {

const ModexpEntry *modexp_entries_latency(int *count) {
  static const ModexpEntry entries[] = {
      make_entry<16, 4, true, 32>(kForm0),
      make_entry<16, 8, true, 32>(kForm0),
      make_entry<32, 16, true, 32>(kForm01),
      make_entry<64, 32, true, 32>(kForm0),
      make_entry<96, 32, true, 32>(kForm0),
      make_entry<128, 32, true, 32>(kForm0),
      make_entry<16, 4, false, 32>(kForm0),
      make_entry<16, 8, false, 32>(kForm0),
      make_entry<32, 16, false, 32>(kForm01),
      make_entry<96, 32, false, 32>(kForm0),
  };
  *count = (int)(sizeof(entries) / sizeof(entries[0]));
  return entries;
}

}  // namespace pmk
