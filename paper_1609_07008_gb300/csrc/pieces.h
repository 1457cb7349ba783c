// How the source kernel cuts a step's hub rows into pieces (source.cu); plain
// C++, so that the index arithmetic also compiles for the host.
#pragma once
#include <cstdint>

namespace mfbc {

constexpr int SRC_PIECE = 256;         // arcs of a piece

constexpr uint32_t src_pieces(int32_t len) { return len > 0 ? (uint32_t)(((int64_t)len + SRC_PIECE - 1) / SRC_PIECE) : 0u; }

// The arcs of piece i of a hub row with `out` out-arcs and `in` in-arcs: out-arcs
// first, then in-arcs (0 where one row serves both).  No arcs past the row's
// pieces: a step counts the pieces of every long row, also of those that its list
// has no room for, and these numbers fall to the last row listed.  They are bounded
// by the step's arcs only (2^23 and more), so offsets are formed in 64 bits.
struct HubPiece {
  bool in;                             // in-arcs rather than out-arcs
  int32_t first, count;                // arcs [first, first + count) of the row
};
constexpr HubPiece src_hub_piece(int32_t out, int32_t in, uint32_t i) {
  const uint32_t po = src_pieces(out);
  const bool is_in = i >= po;
  const int64_t len = is_in ? in : out, first = (int64_t)(is_in ? i - po : i) * SRC_PIECE;
  const int64_t left = len - first;
  if (left <= 0) return {is_in, 0, 0};
  return {is_in, (int32_t)first, (int32_t)(left < SRC_PIECE ? left : SRC_PIECE)};
}

}  // namespace mfbc
