// CRT residue kernels with the small odd-power table (8 odd powers, windows
// up to 4 bits): half the shared memory per exponentiation, so more are
// resident per SM, for a few percent more products.  Measured on GB300 it
// pays for 16 limbs on 2 lanes only (1024-bit CRT, 33,000 chunks 2.94 and
// 2.84 ms; at 32 limbs on 4 lanes 24.73 and 24.84 ms on 41,121 chunks, and
// 1-2.5% slower elsewhere); the autotuner decides per key set and batch size.
// The full-width kernels measured slower with it at every size and are not
// built with it.
#include "modexp_kernels.cuh"

namespace pmk {

const ModexpEntry *modexp_entries_small(int *count) {
  static const ModexpEntry entries[] = {
      make_entry<2, 2, true, dev::kThreads, kTableSmall>(kForm0),
      make_entry<4, 2, true, dev::kThreads, kTableSmall>(kForm0),
      make_entry<8, 2, true, dev::kThreads, kTableSmall>(kForm0),
      make_entry<16, 2, true, dev::kThreads, kTableSmall>(kForm0),
      make_entry<32, 4, true, 64, kTableSmall>(kForm01),
      make_entry<32, 8, true, dev::kThreads, kTableSmall>(kForm01),
      make_entry<48, 8, true, dev::kThreads, kTableSmall>(kForm01),
      make_entry<64, 8, true, dev::kThreads, kTableSmall>(kForm01),
      make_entry<64, 16, true, dev::kThreads, kTableSmall>(kForm01),
  };
  *count = (int)(sizeof(entries) / sizeof(entries[0]));
  return entries;
}

}  // namespace pmk
