// fmm_fp64.cuh -- launch sequence of the CTA-blocked FP64 far field (fmm_fp64.cu).
#pragma once

#include <cuda_runtime.h>

#include "fmm_passes.cuh"

namespace stk {
namespace fmm {

// Index of box a's offset from box b in the M2L kernel table (as in the kernel
// spectra), or -1 where the table has no entry: another depth, touching boxes,
// or boxes more than three apart.
FMM_HD int table_offset(const Tree &t, int32_t b, int32_t a) {
  if (t.depth[a] != t.depth[b]) return -1;
  int o[3];
  bool touch = true, far = false;
  for (int q = 0; q < 3; ++q) {
    o[q] = t.anchor[3 * a + q] - t.anchor[3 * b + q];
    touch = touch && o[q] >= -1 && o[q] <= 1;
    far = far || o[q] < -3 || o[q] > 3;
  }
  return touch || far ? -1 : (o[0] + 3) * 49 + (o[1] + 3) * 7 + (o[2] + 3);
}

cudaError_t far_field_fp64(const Pass &P, const int32_t *depth_ptr, int32_t max_depth, int sms,
                           cudaStream_t st);

}  // namespace fmm
}  // namespace stk
