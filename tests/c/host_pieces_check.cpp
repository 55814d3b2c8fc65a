// Host check of how a long message is cut (host_pieces.h), over random
// lengths, widths and key counts; no GPU.  Every piece starts at a multiple of
// K and of 16 chunks; with more than one, each piece but the last is
// kPieceBytes of message or more, the last at least half of that, and each has
// kPieceRows chunks a key.
#include <cstdio>
#include <random>

#include "host_pieces.h"

int main() {
  std::mt19937_64 gen(7);
  long checks = 0, failures = 0, cut = 0;
  auto check = [&](size_t len, size_t nbits, uint32_t K) {
    const size_t payload = nbits / 8 - 1, n = (len + payload - 1) / payload;
    const size_t per = pmk::piece_chunks(len, n, K);
    bool ok = per > 0 && per <= n;
    if (per < n) {
      cut++;
      const size_t pieces = (n + per - 1) / per, last = n - (pieces - 1) * per;
      ok = ok && per % K == 0 && per % 16 == 0 && pieces <= pmk::kMaxPieces;
      ok = ok && per * payload + payload >= pmk::kPieceBytes;
      ok = ok && len - (pieces - 1) * per * payload >= pmk::kPieceBytes / 2 - payload;
      ok = ok && last >= pmk::kPieceRows * K;
    } else {
      // one piece only where two would be too short, a start being rounded by up to 16 K chunks
      ok = ok && (len < 2 * pmk::kPieceBytes || n < 2 * (pmk::kPieceRows + 16) * K);
    }
    checks++;
    if (!ok && failures++ < 20) std::printf("FAIL len %zu nbits %zu K %u per %zu n %zu\n", len, nbits, K, per, n);
  };
  check(65453669, 512, 1001);
  for (int i = 0; i < 400000; i++) {
    const size_t len = (size_t)1 << (gen() % 31);
    check(1 + gen() % len + len / 2, 128 << (gen() % 7), 1 + gen() % (1u << (gen() % 13)));
  }
  std::printf("%ld checks, %ld in pieces, %ld failures\n", checks, cut, failures);
  return failures != 0 || cut < 10000;
}
