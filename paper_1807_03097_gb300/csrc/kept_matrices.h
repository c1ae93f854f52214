// Whether the FP64 coupling matrices are kept as digits (host logic, checked in tests/kept_matrices_check.cpp).
#pragma once
#include <cstddef>

namespace efie {

// digits: bytes of the matrices; beside: bytes that this form needs beside them (fixed-point sources,
// partial results, offsets); free_bytes: free device memory.  store 0 keeps them when the matrices take at most half
// of it, store 2 whenever everything fits: matrices that fit without what belongs to them would
// end the setup, where the plain form, which needs nothing beside its smaller matrices, still runs.
inline bool keep_digits(int store, std::size_t digits, std::size_t beside, std::size_t free_bytes) {
  if (store == 1 || beside > free_bytes || digits > free_bytes - beside) return false;
  return store == 2 || digits <= free_bytes / 2;
}

}  // namespace efie
