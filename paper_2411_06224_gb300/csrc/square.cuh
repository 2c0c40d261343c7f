// The domains of all levels as one list of jobs, for the kernels that invert them.
#pragma once

#include <stdint.h>

namespace gs {
namespace square {

struct Jobs {
  double* mat[8];      // per level: n_domains matrices of 3N x 3N, overwritten by their inverses
  uint8_t* dig[8];     // per level: digit matrices (bytes), or null
  int32_t* dexp[8];    // per level: their row exponents
  int32_t first[9];    // first job of each level
  int32_t n_items[8];  // real items per level (l >= 1)
  int L, N;
};

}  // namespace square
}  // namespace gs
