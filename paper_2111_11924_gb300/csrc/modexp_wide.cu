// Wide-key instantiations: 6144- and 8192-bit full width (192 / 256 limbs),
// the CRT residues of two-prime 6144- and 8192-bit keys (96 / 128 limbs), and geometries
// with more lanes per instance for latency-bound small batches.
#include "modexp_kernels.cuh"

namespace pmk {

const ModexpEntry *modexp_entries_wide(int *count) {
  static const ModexpEntry entries[] = {
      make_entry<192, 16, false>(kForm01),
      make_entry<256, 16, false>(kForm01),
      make_entry<256, 32, false>(kForm0),
      make_entry<96, 8, true>(kForm0),
      make_entry<96, 16, true, 32>(kForm01),
      make_entry<128, 16, true>(kForm01),
      make_entry<96, 16, false, 32>(kForm01),
      make_entry<48, 16, true, 32>(kForm0),
      make_entry<128, 32, false, 32>(kForm0),
      make_entry<192, 32, false>(kForm0),
      make_entry<64, 32, false, 32>(kForm0),
  };
  *count = (int)(sizeof(entries) / sizeof(entries[0]));
  return entries;
}

}  // namespace pmk
