// matmul_tc.h -- exact integer matmul on the tcgen05 tensor cores (internal).
#pragma once

#include <cuda_runtime.h>

#include "ccm.h"

namespace ccm {

// True when every pair of widths that the capacities allow splits into exact
// digits (fields of up to 31 bits) and every sum stays inside int64.
bool matmul_tc_applies(const ccm_matrix& a, const ccm_matrix& b);
// Bytes of the digit planes of this product, and a shape-only bound on them.
size_t matmul_tc_bytes(const ccm_matrix& a, const ccm_matrix& b);
size_t matmul_tc_bytes_upper(uint64_t m, uint64_t k, uint64_t n);
// Writes the exact product into `c_scratch` (m x n, row-major; int32 when
// matmul_c32(c), else int64) and merges its width statistics into c's header.
// `ws`: matmul_tc_bytes(a, b) bytes.
int run_matmul_tc(const ccm_matrix& a, const ccm_matrix& b, const ccm_matrix& c, void* c_scratch,
                  void* ws, cudaStream_t st);

}  // namespace ccm
