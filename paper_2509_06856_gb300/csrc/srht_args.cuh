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
  // input row of element rho of group g: rho * istride + (g >> iblk) * igstride + (g mod 2^iblk)
  int64_t istride, igstride;
  int iblk;
  void *out;
  int64_t ldout;
  void *out_y;
  const int32_t *pos;   // non-null: output row = pos[k], skipped when < 0
  // output index of element kappa: (kappa >> oblk) * ostride + (kappa mod 2^oblk) + g * ogstride
  int64_t ostride, ogstride;
  int oblk;
  int d;
  int nslab;
  int logq;
  int vec_in, vec_out;  // 1: rows allow VEC-wide vector access
  int pad_out;          // 1: output rows have room up to a multiple of 8 columns (the intermediate W)
  uint8_t *out_scale;   // FP8 form: block exponents, ld_scale bytes per row
  int64_t ld_scale;
  __nv_bfloat16 *hat_out;  // FP8 form: output rows >= hat_row0 go here in BF16 (nullable)
  int64_t hat_row0, hat_ld;
  double scale;
  void *copy_out;       // pass 1 reading host memory: every input row segment is also stored
                        // here at the same element offset (the device copy of X)
  unsigned *status;     // nullable: ST_TIMEOUT is raised here when a bounded wait gave up
  long long wait_polls; // tensor-core form: polls of a wait before it gives up (0: the built-in time limit)
};

__host__ __device__ __forceinline__ int64_t in_row(const GroupArgs &a, int64_t rho, int64_t g) {
  return rho * a.istride + (g >> a.iblk) * a.igstride + (g & ((int64_t(1) << a.iblk) - 1));
}
__host__ __device__ __forceinline__ int64_t out_row(const GroupArgs &a, int64_t kappa, int64_t g) {
  return (kappa >> a.oblk) * a.ostride + (kappa & ((int64_t(1) << a.oblk) - 1)) + g * a.ogstride;
}

// srht64.cu: the X columns of one FP64 pass over groups of 2^L rows (8 <= L <= 12) in 96-bit
// fixed point.  Tin = double, or float for pass 1 on FP32 storage.
template <class Tin> cudaError_t launch_group_fix(const GroupArgs &a, int L, int64_t ngroups, cudaStream_t s);

// srht_tc.cu: the X columns of one mixed-precision pass over groups of 2^10 or 2^11 rows on the
// tensor cores: FP32 rows gathered through Psd (pass 1) or BF16 rows (pass 2) in, BF16 rows out.
// The rows read are 16-byte aligned (ldin a multiple of 4 FP32 or 8 BF16 elements).
cudaError_t launch_group_tc(const GroupArgs &a, bool f32, int L, int64_t ngroups, cudaStream_t s);

}  // namespace slse
