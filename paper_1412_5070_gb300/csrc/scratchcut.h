// scratchcut.h -- how the static call cuts the scratch of one chunk out of what its
// fixed array leaves.  Plain C++ (a test exercises it without a GPU).
#pragma once

#include <algorithm>
#include <cstdint>

namespace f12host {

struct ScratchCut {
  int64_t keys_cap;    // ints
  int64_t part_thin;   // doubles of the items' partial rows when no Hermite rows are in use
  int64_t part_cap;    // ... and when they are
  int64_t rows_cap;    // doubles of Hermite rows
};

// room: bytes; nf: term families; item_pitch: doubles of an item's partial row
// (an item takes a key, a place in the order and that row).  big_pq: primitive
// quartets of the largest quartet; big_in, pitch: inner pairs and row doubles of
// the general quartets, at most (big_in = 0: there are none).  False when the list
// does not fit: the items of every quartet on its own, and the items and rows of
// one outer pair of every general one.
inline bool scratch_cut(int64_t room, bool direct, int64_t nf, int64_t item_pitch, int64_t big_pq, int64_t big_in,
                        int64_t pitch, ScratchCut *c) {
  const int64_t item_bytes = 8 + 8 * item_pitch;
  *c = ScratchCut{};
  if (room < big_pq * nf * item_bytes) return false;
  if (direct) {   // a key and a row per primitive quartet
    const int64_t n = room / (4 + 8 * pitch);
    c->keys_cap = n;
    c->rows_cap = n * pitch;
    return n >= big_in;
  }
  // items over the whole of it for the thin quartets; the general ones leave
  // its end to the rows: a quarter, within what one outer pair takes of either
  const int64_t items = room / item_bytes;
  c->keys_cap = items;
  c->part_thin = items * item_pitch;
  if (big_in == 0) return true;
  const int64_t least = (big_in * pitch + item_pitch - 1) / item_pitch * item_pitch;
  const int64_t most = c->part_thin - big_in * nf * item_pitch;
  if (least > most) return false;
  c->rows_cap = std::min(std::max(c->part_thin / 4 / item_pitch * item_pitch, least), most);
  c->part_cap = c->part_thin - c->rows_cap;
  return true;
}

}  // namespace f12host
