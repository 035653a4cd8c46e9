// FP64 form of an SRHT pass (paper Sec. 3) in block fixed point on the integer pipe.
//
// What bounds it: this part's FP64 pipe retires two adds per clock and SM, so a pass of 2^10-row
// groups done with FP64 butterflies is bound by its 10 adds per element (0.97 of the FP64 add
// rate).  Here a column of a group is aligned once to its largest exponent and the butterflies run
// on 96-bit two's complement integers: three 32-bit adds with carry per output, exact, at the
// integer rate.  The result is rounded to FP64 once per pass (ten times per pass before), so the
// error of a pass is half an ulp of its output plus the alignment, which drops nothing within 2^29
// of the column's largest element and less than 2^-82 of it below that.
//
// One CTA holds a group (2^L rows x C columns): every thread loads 32 rows of one column
// (independent 8-byte loads, row segments of 8 C bytes), takes the top five row bits in registers,
// exchanges once through shared memory (three 32-bit planes) and takes the next five; sizes above
// 2^10 take the remaining bits with warp shuffles.  No cluster: the exchange stays on the SM.
//
// Measured at N' = 2^20, d = 200, FP64 (GB300): pass 1 4.44 -> 1.87 ms, pass 2 (1/16 of the rows
// kept) 4.40 -> 1.47 ms against FP64 butterflies on clusters; error of the sketch against 64-bit
// arithmetic 3.2e-16 -> 2.4e-16.
//
// A group with an infinity or a NaN takes FP64 butterflies in shared memory instead (CTA-uniform),
// which propagate them as FP64 arithmetic does.
#include "srht_args.cuh"

namespace slse {
namespace {

// Fixed-point position of the leading mantissa bit of the column's largest element:
// bit 52 + kShift = 82, so that 2^12 terms of it stay below 2^95.
constexpr int kShift = 30;
constexpr int kRows = 32;  // rows per thread

struct W96 {
  uint32_t w0, w1, w2;
};

// a + b and a - b, mod 2^96
__device__ __forceinline__ void butterfly(W96 &a, W96 &b) {
  W96 s, t;
  asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
      : "=&r"(s.w0), "=&r"(s.w1), "=r"(s.w2)
      : "r"(a.w0), "r"(a.w1), "r"(a.w2), "r"(b.w0), "r"(b.w1), "r"(b.w2));
  asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %7;\n\tsubc.u32 %2, %5, %8;"
      : "=&r"(t.w0), "=&r"(t.w1), "=r"(t.w2)
      : "r"(a.w0), "r"(a.w1), "r"(a.w2), "r"(b.w0), "r"(b.w1), "r"(b.w2));
  a = s;
  b = t;
}

// The double with words (hi, lo), its sign flipped by `flip` (0 or 2^31), in units of
// 2^(emax - 1075 - kShift) with emax >= 1 the column's largest (biased) exponent; bits below the
// unit are dropped.
__device__ __forceinline__ W96 to_fixed(uint32_t hi, uint32_t lo, uint32_t flip, int emax) {
  const int e = (int)((hi >> 20) & 0x7FFu);
  const uint32_t mh = (hi & 0xFFFFFu) | (e ? 0x100000u : 0u);
  const int t = emax - (e ? e : 1);  // right shift of mantissa << kShift
  uint32_t w0 = lo << kShift, w1 = __funnelshift_l(lo, mh, kShift), w2 = mh >> (32 - kShift);
  // variable 96-bit right shift: whole words first (rare), then within a word
  if (t >= 32) {
    w0 = w1; w1 = w2; w2 = 0u;
    if (t >= 64) {
      w0 = t >= 96 ? 0u : w1; w1 = 0u;
    }
  }
  W96 r;
  r.w0 = __funnelshift_r(w0, w1, t);
  r.w1 = __funnelshift_r(w1, w2, t);
  r.w2 = w2 >> (t & 31);
  const uint32_t s = (uint32_t)((int32_t)(hi ^ flip) >> 31);
  r.w0 ^= s; r.w1 ^= s; r.w2 ^= s;
  asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %3;\n\tsubc.u32 %2, %2, %3;"
      : "+&r"(r.w0), "+&r"(r.w1), "+r"(r.w2)
      : "r"(s));
  return r;
}

// v 2^(emax - 1075 - kShift + eadd), rounded to nearest even
__device__ __forceinline__ double from_fixed(W96 v, int emax, int eadd) {
  const uint32_t s = (uint32_t)((int32_t)v.w2 >> 31);
  v.w0 ^= s; v.w1 ^= s; v.w2 ^= s;
  asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %3;\n\tsubc.u32 %2, %2, %3;"
      : "+&r"(v.w0), "+&r"(v.w1), "+r"(v.w2)
      : "r"(s));
  int top = 95;  // position of the leading bit
  if (v.w2 == 0u) {
    v.w2 = v.w1; v.w1 = v.w0; v.w0 = 0u;
    top = 63;
    if (v.w2 == 0u) {
      v.w2 = v.w1; v.w1 = 0u;
      top = 31;
      if (v.w2 == 0u) return 0.0;
    }
  }
  const int n = __clz((int)v.w2);
  top -= n;
  const uint32_t h = __funnelshift_l(v.w1, v.w2, n), m = __funnelshift_l(v.w0, v.w1, n), l = v.w0 << n;
  // 53 leading bits: h and the top 21 of m; the rest decides the rounding
  uint32_t mh = h >> 11, ml = __funnelshift_r(m, h, 11);
  const uint32_t rest = (m & 0x7FFu) | (l != 0u ? 1u : 0u) | ((m & 0x800u) != 0u && (m & 0x7FFu) == 0x400u ? 1u : 0u);
  const uint32_t up = rest > 0x400u ? 1u : 0u;
  const int e = emax + eadd + top - 52 - kShift;  // biased exponent of the leading bit
  if (e >= 1 && e < 2046) {
    // mantissa with its leading bit, added to the exponent field less one: a carry of the rounding
    // moves into the exponent
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;"
        : "+&r"(ml), "+r"(mh)
        : "r"(up), "r"(((uint32_t)(e - 1) << 20)));
    return __hiloint2double((int)(mh | (s & 0x80000000u)), (int)ml);
  }
  // outside the normal range (rare)
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;" : "+&r"(ml), "+r"(mh) : "r"(up), "r"(1022u << 20));
  const double x = ldexp(__hiloint2double((int)mh, (int)ml), e - 1023);
  return s ? -x : x;
}

// Words of a stored element as an FP64 value.
__device__ __forceinline__ uint2 load_words(const double *p) {
  const double v = __ldcs(p);
  return make_uint2((uint32_t)__double2loint(v), (uint32_t)__double2hiint(v));
}
__device__ __forceinline__ uint2 load_words(const float *p) {
  const float f = __ldcs(p);
  const uint32_t u = __float_as_uint(f), a = u & 0x7FFFFFFFu, e = a >> 23;
  if ((e == 255u) | ((e == 0u) & (a != 0u))) {  // denormal, infinity, NaN
    const double v = (double)f;
    return make_uint2((uint32_t)__double2loint(v), (uint32_t)__double2hiint(v));
  }
  return make_uint2(u << 29, (u & 0x80000000u) | (a != 0u ? (a >> 3) + 0x38000000u : 0u));
}

template <class Tin, int L, int C>
__global__ void __launch_bounds__((1 << L) * C / kRows, L >= 11 ? 1 : ((1 << L) * C <= 4096 ? 4 : 2))
    k_group_fix(const GroupArgs a, int eadd, double mul) {
  constexpr int M = 1 << L;
  constexpr int NT = M * C / kRows;
  constexpr int NA = M / kRows;               // rows between two rows of a thread in stage A
  constexpr int PLANE = M * C + NA * C;       // C words of padding per 32 rows: no bank conflicts
  constexpr int BB = L - 5 < 5 ? L - 5 : 5;   // row bits of stage B in registers
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t *plane = reinterpret_cast<uint32_t *>(smem_raw);
  int32_t *s_idx = reinterpret_cast<int32_t *>(plane + 3 * PLANE);  // input rows, then output rows
  __shared__ uint32_t s_emax[C];

  const int t = threadIdx.x;
  const int slab = (int)(blockIdx.x % (unsigned)a.nslab);
  const int64_t g = (int64_t)(blockIdx.x / (unsigned)a.nslab);
  const int c = t % C, b = t / C;
  const int col = slab * C + c;
  const bool cv = col < a.d;
  const Tin *in = static_cast<const Tin *>(a.in);

  for (int l = t; l < M; l += NT) {
    const int64_t j = l * a.istride + g * a.igstride;
    s_idx[l] = a.Psd ? __ldg(a.Psd + j) : (int32_t)j;
  }
  if (t < C) s_emax[t] = 0u;
  __syncthreads();

  // stage A: rows b + NA k
  uint32_t lo[kRows], hi[kRows];
  const int64_t nin = a.Psd ? a.N : INT64_MAX;
  uint32_t flips = 0u;
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const int32_t v = s_idx[b + NA * k];
    const int64_t src = v < 0 ? (int64_t)(~v) : (int64_t)v;
    flips |= (v < 0 ? 1u : 0u) << k;
    uint2 x = make_uint2(0u, 0u);
    if (cv && src < nin) x = load_words(in + src * a.ldin + col);
    lo[k] = x.x;
    hi[k] = x.y;
  }
  if (a.copy_out) {  // pass 1 on host memory: the device copy of the rows read
    Tin *cpy = static_cast<Tin *>(a.copy_out);
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      const int32_t v = s_idx[b + NA * k];
      const int64_t src = v < 0 ? (int64_t)(~v) : (int64_t)v;
      if (cv && src < nin) cpy[src * a.ldin + col] = (Tin)__hiloint2double((int)hi[k], (int)lo[k]);
    }
  }
  uint32_t mx = 0u;
#pragma unroll
  for (int k = 0; k < kRows; ++k) mx = max(mx, hi[k] & 0x7FF00000u);
#pragma unroll
  for (int off = C; off < 32; off <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  if ((t & 31) < C) atomicMax(&s_emax[c], mx);
  __syncthreads();
  bool special = false;
#pragma unroll
  for (int q = 0; q < C; ++q) special |= s_emax[q] == 0x7FF00000u;
  int emax = (int)(s_emax[c] >> 20);
  emax = emax ? emax : 1;
  // the output rows replace the input rows (every thread has read its own)
  if (a.pos)
    for (int l = t; l < M; l += NT) s_idx[l] = __ldg(a.pos + l * a.ostride + g * a.ogstride);

  double *out = static_cast<double *>(a.out);
  if (special) {
    double *tile = reinterpret_cast<double *>(smem_raw);
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      const double x = __hiloint2double((int)hi[k], (int)lo[k]);
      tile[(b + NA * k) * C + c] = (flips >> k) & 1u ? -x : x;
    }
    __syncthreads();
    for (int h = 1; h < M; h <<= 1) {
      for (int p = t; p < M / 2 * C; p += NT) {
        const int q = p / C, r = (q / h) * 2 * h + q % h;
        double *u = tile + r * C + p % C;
        const double x = u[0], y = u[h * C];
        u[0] = x + y;
        u[h * C] = x - y;
      }
      __syncthreads();
    }
    for (int p = t; p < M * C; p += NT) {
      const int l = p / C, cc = slab * C + p % C;
      const int64_t dst = a.pos ? (int64_t)s_idx[l] : l * a.ostride + g * a.ogstride;
      if (dst >= 0 && cc < a.d) out[dst * a.ldout + cc] = tile[p] * a.scale;
    }
    return;
  }

  W96 v[kRows];
#pragma unroll
  for (int k = 0; k < kRows; ++k) v[k] = to_fixed(hi[k], lo[k], (flips >> k) << 31, emax);
#pragma unroll
  for (int h = 1; h < kRows; h <<= 1)
#pragma unroll
    for (int k = 0; k < kRows; ++k)
      if ((k & h) == 0) butterfly(v[k], v[k + h]);
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const int row = b + NA * k;
    const int idx = row * C + c + (row / kRows) * C;
    plane[idx] = v[k].w0;
    plane[PLANE + idx] = v[k].w1;
    plane[2 * PLANE + idx] = v[k].w2;
  }
  __syncthreads();
  // stage B: rows 32 b + k
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const int idx = (b * kRows + k) * C + c + b * C;
    v[k].w0 = plane[idx];
    v[k].w1 = plane[PLANE + idx];
    v[k].w2 = plane[2 * PLANE + idx];
  }
#pragma unroll
  for (int h = 1; h < (1 << BB); h <<= 1)
#pragma unroll
    for (int k = 0; k < kRows; ++k)
      if ((k & h) == 0) butterfly(v[k], v[k + h]);
  // row bits 5 .. L - 6 (the low bits of b: lanes C apart)
#pragma unroll
  for (int bit = 0; bit < L - 10; ++bit) {
    const bool up = (b >> bit) & 1;
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      W96 o;
      o.w0 = __shfl_xor_sync(0xffffffffu, v[k].w0, C << bit);
      o.w1 = __shfl_xor_sync(0xffffffffu, v[k].w1, C << bit);
      o.w2 = __shfl_xor_sync(0xffffffffu, v[k].w2, C << bit);
      W96 x = up ? o : v[k], y = up ? v[k] : o;
      butterfly(x, y);
      v[k] = up ? y : x;
    }
  }
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const int row = b * kRows + k;
    const int64_t dst = a.pos ? (int64_t)s_idx[row] : row * a.ostride + g * a.ogstride;
    if (dst >= 0 && cv) {
      double x = from_fixed(v[k], emax, eadd);
      if (mul != 1.0) x *= mul;
      out[dst * a.ldout + col] = x;
    }
  }
}

template <class Tin, int L, int C>
cudaError_t launch_fix(const GroupArgs &a0, int64_t ngroups, int eadd, double mul, cudaStream_t s) {
  constexpr int M = 1 << L;
  GroupArgs a = a0;
  a.nslab = (a.d + C - 1) / C;
  const size_t smem = 3 * (size_t)(M * C + M / kRows * C) * 4 + (size_t)M * 4;
  auto kern = k_group_fix<Tin, L, C>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)(ngroups * a.nslab), M * C / kRows, smem, s>>>(a, eadd, mul);
  return cudaGetLastError();
}

}  // namespace

// 8-byte row segments of C columns: 64 bytes (128 at 2^8 rows, 32 at 2^12), the widest whose planes
// leave room for two CTAs per SM (one from 2^11 rows on).
template <class Tin> cudaError_t launch_group_fix(const GroupArgs &a, int L, int64_t ngroups, cudaStream_t s) {
  // a power-of-two scale is an exponent offset, any other one multiply per output
  int ex = 0;
  const bool pow2 = frexp(a.scale, &ex) == 0.5;
  const int eadd = pow2 ? ex - 1 : 0;
  const double mul = pow2 ? 1.0 : a.scale;
  switch (L) {
    case 8: return launch_fix<Tin, 8, 16>(a, ngroups, eadd, mul, s);
    case 9: return launch_fix<Tin, 9, 8>(a, ngroups, eadd, mul, s);
    case 10: return launch_fix<Tin, 10, 8>(a, ngroups, eadd, mul, s);
    case 11: return launch_fix<Tin, 11, 8>(a, ngroups, eadd, mul, s);
    case 12: return launch_fix<Tin, 12, 4>(a, ngroups, eadd, mul, s);
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_group_fix<double>(const GroupArgs &, int, int64_t, cudaStream_t);
template cudaError_t launch_group_fix<float>(const GroupArgs &, int, int64_t, cudaStream_t);

}  // namespace slse
