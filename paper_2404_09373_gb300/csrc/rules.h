// Size rules of the tensor-core products, plain C++ (no CUDA types), so that they
// can be compiled and checked on any host.
#pragma once

#include <cstdint>

namespace isdf {

// k values from which a tile's sum of a 5- or 6-digit product may not fit 64 bits:
// it is kept in units of 2^-21 with 7 (S - 4) more bits below, at most 2^35 units
// a k value.  2^21 with 5 digits, 2^14 with 6.
constexpr int64_t oz_wide_k(int S) { return int64_t(1) << (28 - 7 * (S - 4)); }

}  // namespace isdf
