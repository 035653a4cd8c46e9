// Arguments of one SRHT pass, shared by the kernels of srht.cu and srht64.cu.
#pragma once

#include "slse_internal.cuh"

namespace slse {

struct GroupArgs {
  const void *in;       // X (pass 1 / single) or W (pass 2)
  int64_t ldin;
  const void *in_y;     // Y or WY
  int64_t N;            // gather mode: rows >= N are the zero padding
  const int32_t *Psd;   // non-null: gather mode (sign-folded permutation)
  int64_t istride, igstride;  // input row j = rho * istride + g * igstride
  void *out;
  int64_t ldout;
  void *out_y;
  const int32_t *pos;   // non-null: output row = pos[k], skipped when < 0
  int64_t ostride, ogstride;  // output index k = kappa * ostride + g * ogstride
  int d;
  int nslab;
  int logq;
  int vec_in, vec_out;  // 1: rows allow VEC-wide vector access
  uint8_t *out_scale;   // FP8 form: block exponents, ld_scale bytes per row
  int64_t ld_scale;
  __nv_bfloat16 *hat_out;  // FP8 form: output rows >= hat_row0 go here in BF16 (nullable)
  int64_t hat_row0, hat_ld;
  double scale;
  void *copy_out;       // pass 1 reading host memory: every input row segment is also stored
                        // here at the same element offset (the device copy of X)
  unsigned *status;     // nullable: ST_TIMEOUT is raised here when a bounded wait gave up
};

// srht64.cu: the X columns of one FP64 pass over groups of 2^L rows (8 <= L <= 12) in 96-bit
// fixed point.  Tin = double, or float for pass 1 on FP32 storage.
template <class Tin> cudaError_t launch_group_fix(const GroupArgs &a, int L, int64_t ngroups, cudaStream_t s);

}  // namespace slse
