// lbm_halo.h -- layout of one face's halo buffer (host code).
#pragma once

#include <cstddef>

namespace lbm {

// Three parts: `fields` population planes of `seg` elements, the side planes,
// and (16-bit storage) the equilibrium records.  Each part starts at a multiple
// of its element size: an odd number of 2-byte elements ahead of the FP32 side
// planes is padded to whole words.
struct HaloLayout {
  size_t side, rec, bytes;      // byte offsets of the side planes and the records, size of the buffer
};
constexpr HaloLayout halo_layout(size_t fields, size_t seg, size_t store_bytes, size_t nside, size_t side_bytes,
                                 size_t rec_floats) {
  HaloLayout l{};
  l.side = (fields * seg * store_bytes + side_bytes - 1) / side_bytes * side_bytes;
  l.rec = l.side + nside * seg * side_bytes;
  l.bytes = l.rec + rec_floats * seg * sizeof(float);
  return l;
}

}  // namespace lbm
