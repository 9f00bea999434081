// Memory rule of the Galerkin product lists (host code without CUDA).
#pragma once

namespace rich {

// Whether lists of `slots` pairs (8 bytes each, a slice's padding included) for a product of
// nnz entries, with their offsets and the build's scratch, take at most half the free device
// memory.  Asked twice: with the number of products, before anything is laid out, and with
// the slots once the slices' widths are known.
inline bool plist_fits(double slots, double nnz, double free_bytes) {
  return 8.0 * slots + 24.0 * (nnz + 1.0) <= 0.5 * free_bytes;
}

}  // namespace rich
