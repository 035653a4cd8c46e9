// FP64 form of an SRHT pass (paper Sec. 3) in block fixed point on the integer pipe.
//
// What bounds it: this part's FP64 pipe retires two adds per clock and SM, so a pass of 2^10-row
// groups done with FP64 butterflies is bound by its 10 adds per element (0.97 of the FP64 add
// rate).  Here a column of a group is aligned once to its largest exponent and the butterflies run
// on 96-bit two's complement integers: three 32-bit adds with carry per output, exact, at the
// integer rate.  The result is rounded to FP64 once per pass (ten times per pass before), so the
// error of a pass is half an ulp of its output plus the alignment, which drops nothing within 2^30
// of the column's largest element and less than 2^-82 of it below that.
//
// One CTA holds a group (2^L rows x C columns): every thread loads 32 rows of one column
// (independent 8-byte loads, row segments of 8 C bytes), takes the top five row bits in registers,
// exchanges once through shared memory (three 32-bit planes) and takes the next five; sizes above
// 2^10 take the remaining bits with warp shuffles.  No cluster: the exchange stays on the SM.
//
// Measured (GB300), sketch of 10^6 x 200 FP64 (N' = 2^20, 1/16 of the rows kept): 9.27 -> 3.11 ms
// against FP64 butterflies on clusters, error against 64-bit arithmetic 3.2e-16 -> 2.4e-16;
// 2^20 x 256 11.3 -> 3.95 ms, 2^22 x 256 48.6 -> 18.1 ms, FP32 storage the same.  What bounds it
// now: 118 warp instructions per element at 16 warps per SM, with the loads of a group exposed
// (integer pipe 0.45 busy).
//
// A group with an infinity or a NaN takes FP64 butterflies in shared memory instead (CTA-uniform),
// which propagate them as FP64 arithmetic does.
#include <type_traits>

#include "srht_args.cuh"

namespace slse {
namespace {

constexpr int kRows = 32;  // rows per thread

// Fixed-point position of the leading mantissa bit of the column's largest element, for groups of
// 2^L rows: 84 (words 1 and 2 of the mantissa need no shift then), less what 2^L > 2^10 terms need.
constexpr int lead(int L) { return L > 10 ? 94 - L : 84; }

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

// The double with words (hi, lo) as a multiple of the unit 2^(eref - 1107), eref = emax + 84 - lead
// with emax >= 1 the column's largest biased exponent; bits below the unit are dropped (towards
// minus infinity).
__device__ __forceinline__ W96 to_fixed(uint32_t hi, uint32_t lo, int eref) {
  const uint32_t e = (hi >> 20) & 0x7FFu;
  uint32_t mh = (hi & 0xFFFFFu) | (min(e, 1u) << 20);
  const uint32_t t = (uint32_t)eref - max(e, 1u);  // right shift of the mantissa in words 1 and 2
  const uint32_t s = (uint32_t)((int32_t)hi >> 31);
  mh ^= s;
  lo ^= s;
  asm("sub.cc.u32 %0, %0, %2;\n\tsubc.u32 %1, %1, %2;" : "+&r"(lo), "+r"(mh) : "r"(s));
  uint32_t below = 0u;
  if (t >= 32u) {  // rare: an element 2^-30 of its column's largest
    const uint32_t fill = (uint32_t)((int32_t)mh >> 31);
    below = t >= 96u ? fill : (t >= 64u ? mh : lo);
    lo = t >= 64u ? fill : mh;
    mh = fill;
  }
  W96 r;
  r.w0 = __funnelshift_r(below, lo, t);
  r.w1 = __funnelshift_r(lo, mh, t);
  r.w2 = (uint32_t)((int32_t)mh >> (t & 31u));
  return r;
}

__device__ __forceinline__ void negate_if(W96 &v, uint32_t s) {
  v.w0 ^= s; v.w1 ^= s; v.w2 ^= s;
  asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %3;\n\tsubc.u32 %2, %2, %3;"
      : "+&r"(v.w0), "+&r"(v.w1), "+r"(v.w2)
      : "r"(s));
}

// v 2^(eout - 1118) for any |v| < 2^95: the cases the short form below leaves out (zero, a value
// below 2^64 units, a result outside the normal range).
__device__ __forceinline__ double from_fixed_rare(W96 v, int eout) {
  const uint32_t s = (uint32_t)((int32_t)v.w2 >> 31);
  negate_if(v, s);
  if ((v.w0 | v.w1 | v.w2) == 0u) return 0.0;
  while (v.w2 == 0u) {
    v.w2 = v.w1; v.w1 = v.w0; v.w0 = 0u;
    eout -= 32;
  }
  const int n = __clz((int)v.w2);
  const uint32_t h = __funnelshift_l(v.w1, v.w2, n), m = __funnelshift_l(v.w0, v.w1, n), l = v.w0 << n;
  const int e = eout - n;
  // more than 53 bits are only kept where the result is normal: ldexp rounds a subnormal once more,
  // so its 53 bits are cut with a sticky last bit instead of rounded
  const bool normal = e >= 1;
  uint32_t mh = h >> 11, ml = __funnelshift_r(m, h, 11);
  const uint32_t up = normal ? (m >> 10) & 1u : 0u;
  if (!normal) ml |= ((m & 0x7FFu) | l) != 0u ? 1u : 0u;
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;" : "+&r"(ml), "+r"(mh) : "r"(up), "r"(1022u << 20));
  const double x = ldexp(__hiloint2double((int)mh, (int)ml), e - 1023);
  return s ? -x : x;
}

// v 2^(eout - 1118), rounded to nearest (eout: the biased exponent of a value whose leading bit is
// bit 95): the 53 leading bits, rounded by the next one, with the exponent field added so that a
// carry of the rounding moves into it.  false: one of the rare cases, x is not set.
__device__ __forceinline__ bool from_fixed(W96 v, int eout, double &x) {
  const uint32_t s = (uint32_t)((int32_t)v.w2 >> 31);
  negate_if(v, s);
  const int n = __clz((int)v.w2);
  const int e = eout - n;
  if (n == 32 || (uint32_t)(e - 1) >= 2045u) return false;
  const uint32_t h = __funnelshift_l(v.w1, v.w2, n), m = __funnelshift_l(v.w0, v.w1, n);
  uint32_t mh = h >> 11, ml = __funnelshift_r(m, h, 11);
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;"
      : "+&r"(ml), "+r"(mh)
      : "r"((m >> 10) & 1u), "r"((uint32_t)(e - 1) << 20));
  x = __hiloint2double((int)(mh | (s & 0x80000000u)), (int)ml);
  return true;
}

// The words of a stored element as loaded (FP32: in the low word), and then as an FP64 value; `redo`
// is set for an FP32 denormal, infinity or NaN, which the caller widens again with the conversion
// instruction (a branch per element here would split the loads).
__device__ __forceinline__ uint2 load_words(const double *p) {
  const double v = __ldcs(p);
  return make_uint2((uint32_t)__double2loint(v), (uint32_t)__double2hiint(v));
}
__device__ __forceinline__ uint2 load_words(const float *p) { return make_uint2(__float_as_uint(__ldcs(p)), 0u); }

__device__ __forceinline__ void widen_words(uint32_t &lo, uint32_t &hi, bool &redo) {
  const double v = widen(__uint_as_float(lo), redo);
  lo = (uint32_t)__double2loint(v);
  hi = (uint32_t)__double2hiint(v);
}

// Row table of a group: byte offsets of its input rows with the sign of D in bit 0 and the padding
// rows marked in bit 1, then those of its output rows (-1: not sampled).  At 2^12 rows there is only
// room for 32-bit row indices, and the offsets are formed at each use.
template <int L> using RowEntry = std::conditional_t<(L <= 11), int64_t, int32_t>;

// MULT: the outputs are multiplied by `mul` (a scale that is not a power of two)
template <class Tin, int L, int C, bool MULT>
__global__ void __launch_bounds__((1 << L) * C / kRows, 512 / ((1 << L) * C / kRows))
    k_group_fix(const GroupArgs a, int eadd, double mul) {
  constexpr int M = 1 << L;
  constexpr int NT = M * C / kRows;
  constexpr int NA = M / kRows;               // rows between two rows of a thread in stage A
  constexpr int PLANE = M * C + NA * C;       // C words of padding per 32 rows: no bank conflicts
  constexpr int BB = L - 5 < 5 ? L - 5 : 5;   // row bits of stage B in registers
  using Entry = RowEntry<L>;
  constexpr bool kOff = sizeof(Entry) == 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Entry *s_row = reinterpret_cast<Entry *>(smem_raw);
  uint32_t *plane = reinterpret_cast<uint32_t *>(s_row + M);
  __shared__ uint32_t s_emax[C];

  const int t = threadIdx.x;
  const int slab = (int)(blockIdx.x % (unsigned)a.nslab);
  const int64_t g = (int64_t)(blockIdx.x / (unsigned)a.nslab);
  const int c = t % C, b = t / C;
  const int col = slab * C + c;
  const bool cv = col < a.d;
  const char *in = reinterpret_cast<const char *>(static_cast<const Tin *>(a.in) + (cv ? col : 0));
  const int64_t ldi = a.ldin * (int64_t)sizeof(Tin), ldo = a.ldout * (int64_t)sizeof(double);

  for (int l = t; l < M; l += NT) {
    const int64_t j = in_row(a, l, g);
    const int32_t v = a.Psd ? __ldg(a.Psd + j) : (int32_t)j;
    if constexpr (kOff) {
      const int64_t src = v < 0 ? (int64_t)(~v) : (int64_t)v;
      const bool pad = a.Psd && src >= a.N;
      s_row[l] = pad ? 2 : src * ldi + (v < 0 ? 1 : 0);
    } else {
      s_row[l] = v;
    }
  }
  if (t < C) s_emax[t] = 0u;
  __syncthreads();

  // stage A: rows b + NA k, the sign of D applied to the sign bit
  uint32_t lo[kRows], hi[kRows];
  auto row_in = [&](int k, int64_t &off, uint32_t &flip) -> bool {  // false: a padding row
    const Entry v = s_row[b + NA * k];
    if constexpr (kOff) {
      off = v & ~(int64_t)3;
      flip = (uint32_t)v << 31;
      return ((uint32_t)v & 2u) == 0u;
    } else {
      const int64_t src = v < 0 ? (int64_t)(~v) : (int64_t)v;
      off = src * ldi;
      flip = (uint32_t)v & 0x80000000u;
      return a.Psd == nullptr || src < a.N;
    }
  };
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    int64_t off;
    uint32_t flip;
    uint2 x = make_uint2(0u, 0u);
    if (row_in(k, off, flip) && cv) x = load_words(reinterpret_cast<const Tin *>(in + off));
    lo[k] = x.x;
    hi[k] = x.y;
  }
  if constexpr (sizeof(Tin) == 4) {
    uint32_t redo = 0u;
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      const uint32_t f = lo[k];
      bool special = false;
      widen_words(lo[k], hi[k], special);
      if (special) {  // keeps the stored word until it is converted below
        lo[k] = f;
        redo |= 1u << k;
      }
    }
    if (redo != 0u) {
#pragma unroll
      for (int k = 0; k < kRows; ++k)
        if ((redo >> k) & 1u) {
          const double v = (double)__uint_as_float(lo[k]);
          lo[k] = (uint32_t)__double2loint(v);
          hi[k] = (uint32_t)__double2hiint(v);
        }
    }
  }
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    int64_t off;
    uint32_t flip;
    row_in(k, off, flip);
    hi[k] ^= flip;
  }
  if (a.copy_out) {  // pass 1 on host memory: the device copy of the rows read
    char *cpy = reinterpret_cast<char *>(static_cast<Tin *>(a.copy_out) + (cv ? col : 0));
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      int64_t off;
      uint32_t flip;
      if (row_in(k, off, flip) && cv)
        *reinterpret_cast<Tin *>(cpy + off) = (Tin)__hiloint2double((int)(hi[k] ^ flip), (int)lo[k]);
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
  const int emax = max((int)(s_emax[c] >> 20), 1);
  // the output rows replace the input rows (every thread has read its own)
  for (int l = t; l < M; l += NT) {
    const int64_t kg = out_row(a, l, g);
    const int64_t dst = a.pos ? (int64_t)__ldg(a.pos + kg) : kg;
    if constexpr (kOff) s_row[l] = dst < 0 ? -1 : dst * ldo;
    else s_row[l] = (int32_t)dst;
  }
  auto row_out = [&](int row, int64_t &off) -> bool {  // false: not sampled
    const Entry v = s_row[row];
    off = kOff ? (int64_t)v : (int64_t)v * ldo;
    return v >= 0;
  };
  char *out = reinterpret_cast<char *>(static_cast<double *>(a.out) + (cv ? col : 0));

  if (special) {
    double *tile = reinterpret_cast<double *>(plane);
#pragma unroll
    for (int k = 0; k < kRows; ++k) tile[(b + NA * k) * C + c] = __hiloint2double((int)hi[k], (int)lo[k]);
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
    for (int l = b; l < M; l += NT / C) {
      int64_t off;
      if (row_out(l, off) && cv) *reinterpret_cast<double *>(out + off) = tile[l * C + c] * a.scale;
    }
    return;
  }

  W96 v[kRows];
#pragma unroll
  for (int k = 0; k < kRows; ++k) v[k] = to_fixed(hi[k], lo[k], emax + 84 - lead(L));
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
  // row bits 5 .. L - 6 (the low bits of b: lanes C apart): the upper row of a pair negates its own
  // value and adds the partner's
#pragma unroll
  for (int bit = 0; bit < L - 10; ++bit) {
    const uint32_t s = (b >> bit) & 1 ? 0xFFFFFFFFu : 0u;
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      W96 o;
      o.w0 = __shfl_xor_sync(0xffffffffu, v[k].w0, C << bit);
      o.w1 = __shfl_xor_sync(0xffffffffu, v[k].w1, C << bit);
      o.w2 = __shfl_xor_sync(0xffffffffu, v[k].w2, C << bit);
      negate_if(v[k], s);
      asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
          : "+&r"(v[k].w0), "+&r"(v[k].w1), "+r"(v[k].w2)
          : "r"(o.w0), "r"(o.w1), "r"(o.w2));
    }
  }
  const int eout = emax + eadd + 95 - lead(L);
  uint32_t rare = 0u;  // rows left to the general conversion
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    int64_t off;
    if (row_out(b * kRows + k, off) && cv) {
      double x;
      if (from_fixed(v[k], eout, x)) {
        if constexpr (MULT) x *= mul;
        *reinterpret_cast<double *>(out + off) = x;
      } else {
        rare |= 1u << k;
      }
    }
  }
  if (rare == 0u) return;
  // through this thread's own slots of the planes, in a loop that is not unrolled
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const int idx = (b * kRows + k) * C + c + b * C;
    plane[idx] = v[k].w0;
    plane[PLANE + idx] = v[k].w1;
    plane[2 * PLANE + idx] = v[k].w2;
  }
#pragma unroll 1
  for (; rare != 0u; rare &= rare - 1u) {
    const int k = __ffs((int)rare) - 1;
    const int idx = (b * kRows + k) * C + c + b * C;
    int64_t off;
    row_out(b * kRows + k, off);
    const double x = from_fixed_rare(W96{plane[idx], plane[PLANE + idx], plane[2 * PLANE + idx]}, eout);
    *reinterpret_cast<double *>(out + off) = MULT ? x * mul : x;
  }
}

template <class Tin, int L, int C>
cudaError_t launch_fix(const GroupArgs &a0, int64_t ngroups, int eadd, double mul, cudaStream_t s) {
  constexpr int M = 1 << L;
  GroupArgs a = a0;
  a.nslab = (a.d + C - 1) / C;
  const size_t smem = 3 * (size_t)(M * C + M / kRows * C) * 4 + (size_t)M * sizeof(RowEntry<L>);
  auto kern = mul != 1.0 ? k_group_fix<Tin, L, C, true> : k_group_fix<Tin, L, C, false>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)(ngroups * a.nslab), M * C / kRows, smem, s>>>(a, eadd, mul);
  return cudaGetLastError();
}

}  // namespace

// The registers hold 16384 elements of 96 bits per SM (128 registers a thread), so a group of 2^10
// rows leaves 16 columns (128-byte row segments), 2^11 rows 8 and 2^12 rows 4.  Narrower slabs with
// more CTAs per SM were slower (N = 2^20, d = 256: 16 columns 4.2 ms the sketch, 8 columns 4.4 ms,
// 4 columns 5.1 ms).
template <class Tin> cudaError_t launch_group_fix(const GroupArgs &a, int L, int64_t ngroups, cudaStream_t s) {
  // a power-of-two scale is an exponent offset, any other one multiply per output
  int ex = 0;
  const bool pow2 = frexp(a.scale, &ex) == 0.5;
  const int eadd = pow2 ? ex - 1 : 0;
  const double mul = pow2 ? 1.0 : a.scale;
  switch (L) {
    case 8: return launch_fix<Tin, 8, 16>(a, ngroups, eadd, mul, s);
    case 9: return launch_fix<Tin, 9, 16>(a, ngroups, eadd, mul, s);
    case 10: return launch_fix<Tin, 10, 16>(a, ngroups, eadd, mul, s);
    case 11: return launch_fix<Tin, 11, 8>(a, ngroups, eadd, mul, s);
    case 12: return launch_fix<Tin, 12, 4>(a, ngroups, eadd, mul, s);
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_group_fix<double>(const GroupArgs &, int, int64_t, cudaStream_t);
template cudaError_t launch_group_fix<float>(const GroupArgs &, int, int64_t, cudaStream_t);

}  // namespace slse
