// How a host encryption of a long message is cut into pieces (in_pieces in
// api.cpp); free of device calls.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace pmk {

// Encryption of a host message in pieces: each piece's copy in, kernels and
// copy out are queued on one of kPieceStreams streams, so that the copies of
// one piece run beside the kernels of the others and a piece's last blocks
// beside the next one's first.  A piece is at least kPieceBytes of message,
// enough to fill the GPU several times (the last one at least half of that),
// has kPieceRows chunks a key at least (a block serves one key: the last block
// of each is part empty), and starts at a multiple of K chunks (chunk t of the
// message is chunk t - start of the piece under the same key) and of 16 (aligned
// message bytes).  Host buffers
// that overlap go in one piece (all input is read before any output is
// written), and so does a call whose output is not page-locked, or whose stream
// has another priority than the pieces' own.
// Measured with page-locked buffers, one piece on one stream against pieces:
// 100 MiB at 2048 bits 8.04 and 7.14 ms, 50 MB at 1024 bits 2.29 and 1.90,
// 25 MiB at 4096 bits 3.79 and 3.61.  Decryption, where the copies are below 2%
// of the time, stays in one piece: in pieces, 25 MB with CRT 58.5 and 58.3, but
// 13 MiB full d at 4096 bits 475.8 and 494.7, 50 MiB at 2048 bits and 512 keys
// 473.5 and 485.5.
constexpr size_t kPieceBytes = 6u << 20, kPieceRows = 128, kMaxPieces = 8;

// Chunks per piece for a message of n chunks (n itself: one piece).  Rounded to
// piece starts, so the last piece is the shorter one: with many keys, fewer
// pieces are taken until it is half as long as the others and has its rows.
inline size_t piece_chunks(size_t msg_len, size_t n, uint32_t K) {
  size_t unit = K;
  while (unit % 16) unit *= 2;
  for (size_t pieces = std::min({kMaxPieces, msg_len / kPieceBytes, n / (kPieceRows * K)}); pieces >= 2; pieces--) {
    const size_t per = ((n + pieces - 1) / pieces + unit - 1) / unit * unit;
    if (per >= n) return n;
    const size_t last = (n - 1) % per + 1;
    if (last >= kPieceRows * K && 2 * last >= per) return per;
  }
  return n;
}

}  // namespace pmk
