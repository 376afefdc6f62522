// matmul_tc.h -- exact integer matmul on the tcgen05 tensor cores (internal).
#pragma once

#include <cuda_runtime.h>

#include "ccm.h"

namespace ccm {

// True when every pair of widths that the capacities allow splits into exact
// digits (fields of up to 31 bits) and every sum stays inside int64.
bool matmul_tc_applies(const ccm_matrix& a, const ccm_matrix& b);
// Rows and columns of C that are taken at a time, by the room for the digit
// planes of A's rows and B's columns: all of them when the planes of both
// operands fit, {0, 0} when there is too little room.
struct Strips {
  uint64_t rows, cols;
};
Strips matmul_tc_strips(const ccm_matrix& a, const ccm_matrix& b, size_t room);
// A shape-only bound on the bytes of both operands' digit planes.
size_t matmul_tc_bytes_upper(uint64_t m, uint64_t k, uint64_t n);
// Writes the exact product into `c_scratch` (m x n, row-major; int32 when
// matmul_c32(c), else int64) and merges its width statistics into c's header.
// `ws`: the room that `s` = matmul_tc_strips(a, b, room) was found for.
int run_matmul_tc(const ccm_matrix& a, const ccm_matrix& b, const ccm_matrix& c, void* c_scratch,
                  void* ws, const Strips& s, cudaStream_t st);

}  // namespace ccm
