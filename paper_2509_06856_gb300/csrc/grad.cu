// Fused one-pass residual-gradient kernels and the M-IHS update (paper Sec. 3,
// Eqs. (7) and (8); cost model "(4d+1) rows + 2d^2 + 5d" FLOPs per iteration).
//
// g = sum_i x_i^T (y_i - x_i beta) over the rows of X (2nd stage) or over the first
// m_i rows of the sampled sketch U (1st stage, scaled by N'/m_i).  One warp owns one
// row at a time: each lane holds a slice of the row (vector loads, 16 bytes per
// lane), forms its part of x_i beta, the warp reduces it with shuffles, and every
// lane then accumulates x_i r_i into its own slice of g.  Each row of X is read
// exactly once per pass.  Per-CTA partials are reduced in a fixed order (no atomics)
// so the result is deterministic.
//
// Mixed-precision 2nd stage (X stored FP32): the residual is formed against a base
// point beta_0 in FP64.  A "rebase" pass computes r0_i = y_i - x_i beta_0 with
// error-free transformations (TwoProd via FMA, TwoSum; beta_0 split into two FP32
// words) and stores r0 in FP32; later passes compute r_i = r0_i - x_i (beta - beta_0)
// in FP32, whose rounding error scales with ||beta - beta_0|| and vanishes as the
// iteration converges.  x_i r_i is accumulated in FP32 and folded every 16 rows into
// a two-word (TwoSum) accumulator.  The update kernel re-bases when the drift
// ||beta - beta_0|| exceeds both 2^-10 ||beta|| and 2^10 times the last step
// ||beta+ - beta||: the FP32 residual's error (~2^-24 of the drift) then stays below
// ~2^-14 of the step, i.e. of the iterate's current error, so passes far from the
// solution (the first steps from beta = 0) keep one base point instead of re-basing at
// every step, and the final base point lies within 2^-10 of the solution.
//
// Correction form of the mixed 2nd stage: exact passes stream X (the re-basing pass above or the
// plain FP32 pass); the reduction keeps their gradient g(beta_e).  The steps between exact ones
// use g(beta) = g(beta_e) - G_b (beta - beta_e) with the Gram matrix G_b = Xb^T Xb of the BF16 copy
// Xb of X, formed once on the tensor cores (gram.cu): a d x d product (in k_reduce) instead of a
// pass over X.  The update kernel schedules the next exact pass (a step below 1/100 of the first
// step after the last exact pass, a step above it, or one that meets the stopping test), makes it
// a re-basing pass only when the drift from beta_0 exceeds 2^-10 ||beta||, stops only on an exact
// step, and switches to the plain FP32 passes when a cycle gains less than plain steps would for
// the same cost.
#include "slse_internal.cuh"

namespace slse {
namespace {

constexpr int kGradThreads = 256;
constexpr int kWarps = kGradThreads / 32;
constexpr int kFlushRows = 16;

struct GradArgs {
  const void *X;
  int64_t ldx;
  const void *Y;
  int64_t nrows;
  int d;
  const double *beta_ring;
  DevState *st;
  const float *delta32;
  float *r0;
  double *beta0;
  double *partials;
  int check_done;
};

template <class T> __device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// Write the CTA partial: sum of the kWarps per-warp slices in a fixed order.
__device__ __forceinline__ void cta_partial(double (*sm)[512], int d, double *out) {
  __syncthreads();
  for (int c = threadIdx.x; c < d; c += blockDim.x) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) s += sm[w][c];
    out[c] = s;
  }
}

// ---------------------------------------------------------------- FP64 arithmetic
// Sums of R per-lane values (one per row) across the warp.  The first log2(R) levels are a
// transposed butterfly: at each level a lane keeps half of its rows and adds the partner's values
// of that half (one FP64 add per kept row instead of one per row), so after them lane l holds a
// partial of row rowsel(l); the remaining levels sum that one value.  FP64 adds hold this part's
// FP64 pipe for tens of cycles each, so the transposed form saves most of the reduction's cost
// (R = 4: 6 adds instead of 20).  Returns the full sum of every row to every lane (fixed order).
template <int R>
__device__ __forceinline__ void warp_sum_rows(double (&v)[R], int lane) {
  int off = 16;
#pragma unroll
  for (int n = R; n > 1; n >>= 1, off >>= 1) {
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int j = 0; j < n / 2; ++j) {
      const double send = upper ? v[j] : v[j + n / 2];
      const double keep = upper ? v[j + n / 2] : v[j];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
#pragma unroll
  for (; off > 0; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
  // lane l holds row sum((lane bit 16 >> k) * (R >> (k + 1))); broadcast each row's total
  double tot[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    int src = 0, o = 16;
#pragma unroll
    for (int n = R; n > 1; n >>= 1, o >>= 1)
      if (q % n >= n / 2) src |= o;
    tot[q] = __shfl_sync(0xffffffffu, v[0], src);
  }
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = tot[q];
}

// The FP64 pipe (two fused multiply-adds per clock and SM on this part) bounds this pass: x_i beta
// and x_i r_i are one each per element.  So x_i beta is formed on the integer pipes instead, beside
// the FP64 pipe, which is left with x_i r_i and a handful of operations per row group:
//  - beta_j = (bh 2^26 + bl) 2^(be - 1075), signed 27- and 26-bit parts, once per pass;
//  - the row's terms are aligned to the largest exponent F of x_ij beta_j over the row: x_ij's
//    mantissa becomes the 62-bit integer (zh 2^31 + zl) 2^(F - be ..), bits below 2^-61 of the
//    row's largest term are dropped;
//  - zh bh, zh bl and zl bh are summed exactly in 64 bits (three 32 x 32 + 64 bit multiply-adds), the
//    lanes' 96-bit sums are added exactly in 26-bit pieces, and the total is rounded to FP64 once;
//  - of zl bl the upper 32 bits are summed (FP64 storage; an FP32 mantissa fits zh, but for terms below
//    2^-7 of the row's largest).  It has the sign of its term: without it every x_i beta came out 2^-59
//    too small, an error of the gradient along X^T X beta that grew with the rows.  Residual 1e-3 of
//    X beta, 131072 x 10, error against a double-double sum: FP64 chain 2.6e-13, without zl bl 1.4e-12, with
//    it 1.8e-13.  It costs 2 % at 2^20 x 256, 5 % at 2^20 x 512 (with all 64 bits 5 and 5 to 7 %).
// The error of x_i beta is then below that of an FP64 chain (2^-53 of the partial sums at each of
// its d steps): sqrt(d) 2^-60 of the row's largest term, and half an ulp.  A row group with a
// denormal, an infinity or a NaN, or whose largest product is outside [2^-846, 2^954], takes the FP64
// sums (warp-uniform).  A row without a non-zero term has the sum zero and stays here (in
// the FP64 sums, which read X again element by element, a pass at beta = 0 took 2420 us at 2^20 x 512, FP32
// storage 3390; now 1190 and 1180).
// Measured (GB300), the whole call against the FP64 chain: N = 2^20, d = 256 FP64 1.10 -> 0.67 ms, d = 512
// FP64 2.02 -> 1.26 ms, FP32 storage 2.08 -> 1.25 ms.  What bounds it now: the FP64 pipe, 0.76
// busy (the integer pipe 0.67).  Before zl bl (0.63 ms at 2^20 x 256): 0.69 ms without
// the ring (rows prefetched into registers), 0.86 ms without any prefetch, 0.77 ms with three CTAs of
// 80 registers.
struct BetaFix {
  int bh, bl, be;
};

constexpr int kNoTerm = -(1 << 20);  // exponent of a zero term

__device__ __forceinline__ BetaFix beta_fix(double b) {
  const uint32_t hi = (uint32_t)__double2hiint(b), lo = (uint32_t)__double2loint(b);
  const int e = (int)((hi >> 20) & 0x7FFu);
  if (e == 0 || e == 0x7FF) return BetaFix{0, 0, e == 0 && ((hi << 1) | lo) == 0u ? kNoTerm : -kNoTerm};
  const uint32_t mh = (hi & 0xFFFFFu) | 0x100000u;
  const int h = (int)((mh << 6) | (lo >> 26)), l = (int)(lo & 0x3FFFFFFu);
  return (int)hi < 0 ? BetaFix{-h, -l, e} : BetaFix{h, l, e};
}

// a + b c, signed 32 x 32 bits into 64
__device__ __forceinline__ long long madw(int b, int c, long long a) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a) : "r"(b), "r"(c));
  return a;
}
// a + the upper 32 bits of b c
__device__ __forceinline__ int madh(int b, int c, int a) {
  asm("mad.hi.s32 %0, %1, %2, %0;" : "+r"(a) : "r"(b), "r"(c));
  return a;
}
// logical right shift that gives 0 from 32 on (the C operator does not define it)
__device__ __forceinline__ uint32_t shr_clamp(uint32_t v, uint32_t n) {
  asm("shr.u32 %0, %0, %1;" : "+r"(v) : "r"(n));
  return v;
}

// Biased FP64 exponent of x and, left-aligned at bit 63 of (ah, al), its mantissa with the leading
// bit; odd: neither a normal number nor zero.
__device__ __forceinline__ void split_x(double x, int &e, bool &zero, bool &odd, uint32_t &ah, uint32_t &al, int &sgn) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  e = (int)((hi >> 20) & 0x7FFu);
  zero = ((hi << 1) | lo) == 0u;
  odd = (uint32_t)(e - 1) >= 2046u && !zero;
  const uint32_t mh = (hi & 0xFFFFFu) | 0x100000u;
  ah = __funnelshift_l(lo, mh, 11);
  al = lo << 11;
  sgn = ((int)hi >> 31) | 1;
}
__device__ __forceinline__ void split_x(float x, int &e, bool &zero, bool &odd, uint32_t &ah, uint32_t &al, int &sgn) {
  const uint32_t u = __float_as_uint(x);
  const int e8 = (int)((u >> 23) & 0xFFu);
  zero = (u << 1) == 0u;
  odd = (uint32_t)(e8 - 1) >= 254u && !zero;
  e = e8 + 896;
  ah = (u << 8) | 0x80000000u;
  al = 0u;
  sgn = ((int)u >> 31) | 1;
}

// (p3 2^78 + p2 2^52 + p1 2^26 + p0) 2^(F - 2133), rounded to nearest; 1200 <= F <= 3000, |total| < 2^99
__device__ __forceinline__ double dot_total(uint32_t p0, uint32_t p1, uint32_t p2, int p3, int F) {
  const long long top = ((long long)p3 << 26) + (long long)p2;                             // units of 2^52
  const unsigned long long low = ((unsigned long long)p1 << 26) + (unsigned long long)p0;  // < 2^58
  unsigned long long L = ((unsigned long long)top << 52) + low;
  unsigned long long H = (unsigned long long)(top >> 12) + (L < low ? 1ull : 0ull);
  const bool neg = (long long)H < 0;
  if (neg) {
    L = 0ull - L;
    H = ~H + (L == 0ull ? 1ull : 0ull);
  }
  int pos = 127;  // of the leading bit
  if (H == 0ull) {
    H = L;
    L = 0ull;
    pos = 63;
  }
  if (H == 0ull) return 0.0;
  const int n = __clzll((long long)H);
  const unsigned long long m = n ? (H << n) | (L >> (64 - n)) : H;
  // the 53 leading bits, rounded by the next one; a carry moves into the exponent
  const unsigned long long bits = (m >> 11) + ((m >> 10) & 1ull) + ((unsigned long long)(uint32_t)(F - 2133 + 1022 + pos - n) << 52);
  return __longlong_as_double((long long)(bits | (neg ? 0x8000000000000000ull : 0ull)));
}

// Tx = double (X F64 or U F64) or float (X F32, widened exactly).  VW = elements per lane load,
// VMAX = lane loads per row (sized to d), RPW = rows per warp iteration.  BS: the parts of beta stay
// in shared memory (16 columns per lane leave no registers for them).  Two CTAs of 8 warps fit on an
// SM.  The rows of the next two groups are on their way meanwhile: every lane copies its own pieces
// (cp.async) into its warp's two-stage ring in shared memory, which costs no registers.
template <class Tx, int VW, int VMAX, int RPW, bool BS>
__global__ void __launch_bounds__(kGradThreads, 2) k_grad_f64(const GradArgs a) {
  extern __shared__ __align__(16) unsigned char ring_raw[];
  __shared__ __align__(16) double sm[kWarps][512];
  dependent_start();
  if (a.check_done && a.st->done) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t gw = (int64_t)blockIdx.x * kWarps + warp, nw = (int64_t)gridDim.x * kWarps;
  const int d = a.d;
  const double *beta = a.beta_ring + (size_t)(a.st->iter % 3) * d;
  const Tx *X = static_cast<const Tx *>(a.X);
  const Tx *Y = static_cast<const Tx *>(a.Y);
  constexpr int NB = BS ? 1 : VMAX * VW;
  // A row without a non-zero term: with the largest exponent kept above the terms' every shift is large and
  // the sums are zero by themselves (2^20 x 256 FP64 665 us, against 691 with the sum left out at the end;
  // 2^20 x 512 FP32 1252, 1294), but with beta in shared memory the other forms schedule worse so (2^20 x
  // 512 FP64 1350, 1254; 2^20 x 511 FP32 1534, 1408), and the narrowest tile, whose passes are short, feels its
  // latency (an FP64 fit of 20000 x 50 1221, 1157): there the sum is left out.
  constexpr bool kClamp = BS ? sizeof(Tx) == 4 && VW == 2 : VMAX >= 2;
  int rbh[NB], rbl[NB], rbe[NB];
  // shared-memory form: (bh, bl) pairs, then the exponents, in lane order
  int2 *sb = reinterpret_cast<int2 *>(&sm[0][0]);
  int *se = reinterpret_cast<int *>(sb + 32 * VMAX * VW);
  double g[VMAX][VW];
  bool beta_odd = false;
#pragma unroll
  for (int v = 0; v < VMAX; ++v)
#pragma unroll
    for (int e = 0; e < VW; ++e) {
      const int col = (v * 32 + lane) * VW + e;
      const BetaFix b = beta_fix(col < d ? beta[col] : 0.0);
      beta_odd |= b.be == -kNoTerm;
      if constexpr (BS) {
        if (warp == 0) {
          sb[(v * VW + e) * 32 + lane] = make_int2(b.bh, b.bl);
          se[(v * VW + e) * 32 + lane] = b.be;
        }
      } else {
        rbh[v * VW + e] = b.bh;
        rbl[v * VW + e] = b.bl;
        rbe[v * VW + e] = b.be;
      }
      g[v][e] = 0.0;
    }
  beta_odd = __any_sync(0xffffffffu, beta_odd);
  if constexpr (BS) __syncthreads();
  struct __align__(VW * sizeof(Tx)) Piece {
    Tx e[VW];
  };
  // this warp's ring: stage, row, load, lane
  Piece *ring = reinterpret_cast<Piece *>(ring_raw) + warp * (2 * RPW * VMAX * 32) + lane;
  auto load_rows = [&](int64_t i0, int stage) {  // rows past the end and columns past d as zeros
#pragma unroll
    for (int q = 0; q < RPW; ++q) {
      const int64_t i = i0 + q;
      const bool rv = i < a.nrows;
      const Tx *row = X + (rv ? i : 0) * a.ldx;
#pragma unroll
      for (int v = 0; v < VMAX; ++v) {
        const int col0 = (v * 32 + lane) * VW;
        const bool in = rv && col0 < d;
        const unsigned dst = (unsigned)__cvta_generic_to_shared(ring + ((stage * RPW + q) * VMAX + v) * 32);
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(dst), "l"(row + (in ? col0 : 0)),
                     "n"((int)sizeof(Piece)), "r"(in ? (int)sizeof(Piece) : 0)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  auto load_y = [&](int64_t i0) -> Tx {  // lane q: row q's
    return (lane < RPW && i0 + lane < a.nrows) ? Y[i0 + lane] : Tx(0);
  };
  const int64_t step = nw * RPW;
  load_rows(gw * RPW, 0);
  load_rows(gw * RPW + step, 1);
  Tx ny = load_y(gw * RPW);
  int stage = 0;
  for (int64_t i0 = gw * RPW; i0 < a.nrows; i0 += step, stage ^= 1) {
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    Tx x[RPW][VMAX][VW];
    const double y = (double)ny;
#pragma unroll
    for (int q = 0; q < RPW; ++q)
#pragma unroll
      for (int v = 0; v < VMAX; ++v) {
        const Piece t = ring[((stage * RPW + q) * VMAX + v) * 32];
#pragma unroll
        for (int e = 0; e < VW; ++e) x[q][v][e] = t.e[e];
      }
    load_rows(i0 + 2 * step, stage);
    ny = load_y(i0 + step);
    bool odd = false;
    uint32_t p0 = 0u, p1 = 0u, p2 = 0u;
    int p3 = 0, F = 1200;
#pragma unroll
    for (int q = 0; q < RPW; ++q) {
      int f[VMAX][VW], fmax = kNoTerm;
#pragma unroll
      for (int v = 0; v < VMAX; ++v)
#pragma unroll
        for (int e = 0; e < VW; ++e) {
          int ex, sgn;
          bool zero, od;
          uint32_t ah, al;
          split_x(x[q][v][e], ex, zero, od, ah, al, sgn);
          odd |= od;
          const int be = BS ? se[(v * VW + e) * 32 + lane] : rbe[BS ? 0 : v * VW + e];
          f[v][e] = zero ? kNoTerm : ex + be;
          fmax = max(fmax, f[v][e]);
        }
      fmax = __reduce_max_sync(0xffffffffu, fmax);
      if constexpr (kClamp) fmax = max(fmax, kNoTerm / 2);
      long long sh = 0, s1 = 0, s2 = 0;
      int s3 = 0;
#pragma unroll
      for (int v = 0; v < VMAX; ++v)
#pragma unroll
        for (int e = 0; e < VW; ++e) {
          int ex, sgn;
          bool zero, od;
          uint32_t ah, al;
          split_x(x[q][v][e], ex, zero, od, ah, al, sgn);
          const uint32_t t = (uint32_t)(fmax - f[v][e]) + 1u;  // right shift of (ah, al)
          const int zh = (int)shr_clamp(ah, t) * sgn;
          const int zl = (int)shr_clamp(__funnelshift_rc(al, ah, t), (uint32_t)max((int)t - 31, 1)) * sgn;
          int2 b;
          if constexpr (BS) b = sb[(v * VW + e) * 32 + lane];
          else b = make_int2(rbh[v * VW + e], rbl[v * VW + e]);
          sh = madw(zh, b.x, sh);
          s1 = madw(zl, b.x, s1);
          s2 = madw(zh, b.y, s2);
          if constexpr (sizeof(Tx) == 8) s3 = madh(zl, b.y, s3);
        }
      s1 += (long long)s3 << 6;
      // sh 2^31 + s1 + s2 2^5, in 96 bits
      const uint32_t hl = (uint32_t)sh, hh = (uint32_t)(sh >> 32);
      uint32_t w0 = hl << 31, w1 = __funnelshift_l(hl, hh, 31), w2 = (uint32_t)((int)hh >> 1);
      const uint32_t ml = (uint32_t)s2, mh = (uint32_t)(s2 >> 32);
      asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
          : "+&r"(w0), "+&r"(w1), "+r"(w2)
          : "r"((uint32_t)s1), "r"((uint32_t)(s1 >> 32)), "r"((uint32_t)(s1 >> 63)));
      asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
          : "+&r"(w0), "+&r"(w1), "+r"(w2)
          : "r"(ml << 5), "r"(__funnelshift_l(ml, mh, 5)), "r"((uint32_t)((int)mh >> 27)));
      // 26-bit pieces (the top one signed), each summed over the lanes; lane q keeps row q's
      const uint32_t q0 = __reduce_add_sync(0xffffffffu, w0 & 0x3FFFFFFu);
      const uint32_t q1 = __reduce_add_sync(0xffffffffu, __funnelshift_r(w0, w1, 26) & 0x3FFFFFFu);
      const uint32_t q2 = __reduce_add_sync(0xffffffffu, __funnelshift_r(w1, w2, 20) & 0x3FFFFFFu);
      const int q3 = __reduce_add_sync(0xffffffffu, (int)w2 >> 14);
      if (lane == q) { p0 = q0; p1 = q1; p2 = q2; p3 = q3; F = kClamp && fmax == kNoTerm / 2 ? 1200 : fmax; }
    }
    const bool rv = lane < RPW && i0 + lane < a.nrows;
    odd = __any_sync(0xffffffffu, odd);
    double r[RPW];
    const bool none = !kClamp && F < kNoTerm / 2;  // no non-zero term: a row of zeros, or beta = 0
    if (!beta_odd && !odd && !__any_sync(0xffffffffu, rv && !none && (uint32_t)(F - 1200) > 1800u)) {
      const double rl = rv ? (none ? y : y - dot_total(p0, p1, p2, p3, F)) : 0.0;
#pragma unroll
      for (int q = 0; q < RPW; ++q) r[q] = __shfl_sync(0xffffffffu, rl, q);
    } else {
      double t[RPW];
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        t[q] = 0.0;
        const int64_t i = i0 + q;
#pragma unroll 1
        for (int v = 0; v < VMAX * VW; ++v) {
          const int col = ((v / VW) * 32 + lane) * VW + v % VW;
          if (col < d && i < a.nrows) t[q] = fma((double)X[i * a.ldx + col], beta[col], t[q]);
        }
      }
      warp_sum_rows<RPW>(t, lane);
#pragma unroll
      for (int q = 0; q < RPW; ++q) r[q] = __shfl_sync(0xffffffffu, y, q) - t[q];
    }
    // rows past the end are zero rows: x = 0 adds nothing
    if (sizeof(Tx) == 4 && odd) {  // rare: values the integer widening does not take
#pragma unroll
      for (int q = 0; q < RPW; ++q)
#pragma unroll
        for (int v = 0; v < VMAX; ++v)
#pragma unroll
          for (int e = 0; e < VW; ++e) g[v][e] = fma((double)x[q][v][e], r[q], g[v][e]);
    } else {
      bool special = false;
#pragma unroll
      for (int q = 0; q < RPW; ++q)
#pragma unroll
        for (int v = 0; v < VMAX; ++v)
#pragma unroll
          for (int e = 0; e < VW; ++e) g[v][e] = fma(widen(x[q][v][e], special), r[q], g[v][e]);
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  if constexpr (BS) __syncthreads();  // the parts of beta share the array with the partials
#pragma unroll
  for (int v = 0; v < VMAX; ++v)
#pragma unroll
    for (int e = 0; e < VW; ++e) {
      const int col = (v * 32 + lane) * VW + e;
      if (col < d) sm[warp][col] = g[v][e];
    }
  cta_partial(sm, d, a.partials + (size_t)blockIdx.x * d);
}

// ---------------------------------------------------------------- 1st stage on BF16 sketch
// RPW consecutive rows per warp iteration (independent loads in flight); the BF16
// words stay packed in registers and are widened at use (exact).
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

template <int VMAX, int RPW>
__global__ void __launch_bounds__(kGradThreads, 2) k_grad_bf16v(const GradArgs a) {
  __shared__ double sm[kWarps][512];
  dependent_start();
  if (a.check_done && a.st->done) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t gw = (int64_t)blockIdx.x * kWarps + warp, nw = (int64_t)gridDim.x * kWarps;
  const int d = a.d;
  const double *beta = a.beta_ring + (size_t)(a.st->iter % 3) * d;
  const __nv_bfloat16 *U = static_cast<const __nv_bfloat16 *>(a.X);
  const __nv_bfloat16 *V = static_cast<const __nv_bfloat16 *>(a.Y);
  const int64_t ldu = a.ldx;
  float b[VMAX][8], g[VMAX][8];
#pragma unroll
  for (int v = 0; v < VMAX; ++v)
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int col = (v * 32 + lane) * 8 + e;
      b[v][e] = col < d ? (float)beta[col] : 0.f;
      g[v][e] = 0.f;
    }
  for (int64_t i0 = gw * RPW; i0 < a.nrows; i0 += nw * RPW) {
    uint4 raw[RPW][VMAX];
    float y[RPW];
#pragma unroll
    for (int q = 0; q < RPW; ++q) {
      const int64_t i = i0 + q;
      const bool rv = i < a.nrows;
#pragma unroll
      for (int v = 0; v < VMAX; ++v) {
        const int col0 = (v * 32 + lane) * 8;
        raw[q][v] = (rv && col0 < d) ? __ldg(reinterpret_cast<const uint4 *>(U + i * ldu + col0))
                                     : make_uint4(0u, 0u, 0u, 0u);
      }
      y[q] = rv ? __bfloat162float(V[i]) : 0.f;
    }
    float s[RPW];
#pragma unroll
    for (int q = 0; q < RPW; ++q) {
      float acc = 0.f;
#pragma unroll
      for (int v = 0; v < VMAX; ++v) {
        const uint32_t w[4] = {raw[q][v].x, raw[q][v].y, raw[q][v].z, raw[q][v].w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          acc = fmaf(bf_lo(w[k]), b[v][2 * k], acc);
          acc = fmaf(bf_hi(w[k]), b[v][2 * k + 1], acc);
        }
      }
      s[q] = acc;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
      for (int q = 0; q < RPW; ++q) s[q] += __shfl_xor_sync(0xffffffffu, s[q], off);
#pragma unroll
    for (int q = 0; q < RPW; ++q) {
      const float r = y[q] - s[q];  // padding columns are zero words, padding rows are zero
#pragma unroll
      for (int v = 0; v < VMAX; ++v) {
        const uint32_t w[4] = {raw[q][v].x, raw[q][v].y, raw[q][v].z, raw[q][v].w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          g[v][2 * k] = fmaf(bf_lo(w[k]), r, g[v][2 * k]);
          g[v][2 * k + 1] = fmaf(bf_hi(w[k]), r, g[v][2 * k + 1]);
        }
      }
    }
  }
#pragma unroll
  for (int v = 0; v < VMAX; ++v)
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int col = (v * 32 + lane) * 8 + e;
      if (col < d) sm[warp][col] = (double)g[v][e];
    }
  cta_partial(sm, d, a.partials + (size_t)blockIdx.x * d);
}

// Scalar-load variant for sketches whose rows are not 16-byte aligned.
template <int VMAX>
__global__ void __launch_bounds__(kGradThreads) k_grad_bf16s(const GradArgs a) {
  __shared__ double sm[kWarps][512];
  dependent_start();
  if (a.check_done && a.st->done) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t gw = (int64_t)blockIdx.x * kWarps + warp, nw = (int64_t)gridDim.x * kWarps;
  const int d = a.d;
  const double *beta = a.beta_ring + (size_t)(a.st->iter % 3) * d;
  const __nv_bfloat16 *U = static_cast<const __nv_bfloat16 *>(a.X);
  const __nv_bfloat16 *V = static_cast<const __nv_bfloat16 *>(a.Y);
  float b[VMAX], g[VMAX];
#pragma unroll
  for (int v = 0; v < VMAX; ++v) {
    const int col = v * 32 + lane;
    b[v] = col < d ? (float)beta[col] : 0.f;
    g[v] = 0.f;
  }
  for (int64_t i = gw; i < a.nrows; i += nw) {
    float x[VMAX];
#pragma unroll
    for (int v = 0; v < VMAX; ++v) {
      const int col = v * 32 + lane;
      x[v] = col < d ? __bfloat162float(U[i * a.ldx + col]) : 0.f;
    }
    float s = 0.f;
#pragma unroll
    for (int v = 0; v < VMAX; ++v) s = fmaf(x[v], b[v], s);
    s = warp_sum(s);
    const float r = __bfloat162float(V[i]) - s;
#pragma unroll
    for (int v = 0; v < VMAX; ++v) g[v] = fmaf(x[v], r, g[v]);
  }
#pragma unroll
  for (int v = 0; v < VMAX; ++v) {
    const int col = v * 32 + lane;
    if (col < d) sm[warp][col] = (double)g[v];
  }
  cta_partial(sm, d, a.partials + (size_t)blockIdx.x * d);
}

// ---------------------------------------------------------------- mixed 2nd stage (X F32)
// REBASE = 1: error-free residual against beta (FP64) and r0 written; REBASE = 0:
// residual r0 - x . delta32.  The device state (st->rebase) selects the one that runs.  The
// two-word accumulators (hi, lo) of each warp live in shared memory (float2 per column), folded
// every kFlushRows rows.
extern __shared__ __align__(16) unsigned char mixed_ring[];

template <int VW, int VMAX, int REBASE, int RPW>
__device__ __forceinline__ void grad_mixed_body(const GradArgs &a, double (*sm)[512]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t gw = (int64_t)blockIdx.x * kWarps + warp, nw = (int64_t)gridDim.x * kWarps;
  const int d = a.d;
  const double *beta = a.beta_ring + (size_t)(a.st->iter % 3) * d;
  const float *X = static_cast<const float *>(a.X);
  const float *Y = static_cast<const float *>(a.Y);
  float2 *acc = reinterpret_cast<float2 *>(&sm[warp][0]);  // (hi, lo) per column, this warp only
  for (int c = lane; c < 512; c += 32) acc[c] = make_float2(0.f, 0.f);
  float bh[VMAX][VW], bl[REBASE ? VMAX : 1][VW];
  float gacc[VMAX][VW];
#pragma unroll
  for (int v = 0; v < VMAX; ++v)
#pragma unroll
    for (int e = 0; e < VW; ++e) {
      const int col = (v * 32 + lane) * VW + e;
      if constexpr (REBASE) {
        const double bd = col < d ? beta[col] : 0.0;
        bh[v][e] = (float)bd;
        bl[v][e] = (float)(bd - (double)bh[v][e]);
      } else {
        bh[v][e] = col < d ? a.delta32[col] : 0.f;
      }
      gacc[v][e] = 0.f;
    }
  __syncwarp();
  int nacc = 0;
  // Aligned rows come through a two-stage ring of this warp in shared memory (cp.async, every lane its
  // own pieces), two groups ahead.  Measured at 2^21 x 256: re-basing pass 468 -> 432 us with the ring and
  // 356 us with it, packed arithmetic and the transposed butterfly (it issued 24 instructions per
  // element, and is within 1.15 of its bytes at the copy rate now).
  constexpr bool kRing = VW == 4;
  const int64_t step = nw * RPW;
  float4 *ring = reinterpret_cast<float4 *>(mixed_ring) + warp * (2 * RPW * VMAX * 32) + lane;
  auto load_rows = [&](int64_t i0, int stage) {
#pragma unroll
    for (int q = 0; q < RPW; ++q) {
      const int64_t i = i0 + q;
      const bool rv = i < a.nrows;
      const float *row = X + (rv ? i : 0) * a.ldx;
#pragma unroll
      for (int v = 0; v < VMAX; ++v) {
        const int col0 = (v * 32 + lane) * VW;
        const bool in = rv && col0 < d;
        const unsigned dst = (unsigned)__cvta_generic_to_shared(ring + ((stage * RPW + q) * VMAX + v) * 32);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(row + (in ? col0 : 0)),
                     "r"(in ? 16 : 0)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  // REBASE: the row of a group whose sums this lane ends up with (the butterfly below)
  int row_l = 0;
#pragma unroll
  for (int n = RPW, o = 16; n > 1; n >>= 1, o >>= 1) row_l += (lane & o) ? n / 2 : 0;
  constexpr int NY = REBASE ? 1 : RPW;
  float yn[NY];  // y of this lane's row, or r0 of the next group
  auto load_y = [&](int64_t i0) {
    if constexpr (REBASE) {
      yn[0] = i0 + row_l < a.nrows ? __ldcs(Y + i0 + row_l) : 0.f;
    } else {
#pragma unroll
      for (int q = 0; q < NY; ++q) yn[q] = i0 + q < a.nrows ? __ldcs(a.r0 + i0 + q) : 0.f;
    }
  };
  int stage = 0;
  if constexpr (kRing) {
    load_rows(gw * RPW, 0);
    load_rows(gw * RPW + step, 1);
    load_y(gw * RPW);
  }
  for (int64_t i0 = gw * RPW; i0 < a.nrows; i0 += step, stage ^= 1) {
    float x[RPW][VMAX][VW];
    if constexpr (kRing) {
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
#pragma unroll
      for (int q = 0; q < RPW; ++q)
#pragma unroll
        for (int v = 0; v < VMAX; ++v) {
          const float4 t = ring[((stage * RPW + q) * VMAX + v) * 32];
          x[q][v][0] = t.x; x[q][v][1] = t.y; x[q][v][2] = t.z; x[q][v][3] = t.w;
        }
      load_rows(i0 + 2 * step, stage);
    } else {
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        const int64_t i = i0 + q;
        const bool rv = i < a.nrows;
        const float *row = X + (rv ? i : 0) * a.ldx;
#pragma unroll
        for (int v = 0; v < VMAX; ++v) {
          const int col0 = (v * 32 + lane) * VW;
#pragma unroll
          for (int e = 0; e < VW; ++e) x[q][v][e] = (rv && col0 + e < d) ? __ldcs(row + col0 + e) : 0.f;
        }
      }
      load_y(i0);
    }
    float yr[NY];
#pragma unroll
    for (int q = 0; q < NY; ++q) yr[q] = yn[q];
    const float yl = yr[0];
    if constexpr (kRing) load_y(i0 + step);
    float r[RPW];
    if constexpr (REBASE) {
      // Dot2 (Ogita, Rump, Oishi 2005): s + c = -x . (bh + bl) with error-free products and sums
      float s[RPW], c[RPW];
      if constexpr (kRing) {
        // two columns at a time in the packed FP32 instructions
        const float2 m1 = make_float2(-1.f, -1.f);
#pragma unroll
        for (int q = 0; q < RPW; ++q) {
          float2 sp = make_float2(0.f, 0.f), cp = make_float2(0.f, 0.f);
#pragma unroll
          for (int v = 0; v < VMAX; ++v)
#pragma unroll
            for (int e = 0; e < VW; e += 2) {
              const float2 xp = make_float2(x[q][v][e], x[q][v][e + 1]);
              const float2 b = make_float2(bh[v][e], bh[v][e + 1]), nl = make_float2(-bl[v][e], -bl[v][e + 1]);
              const float2 nb = __fmul2_rn(b, m1);
              const float2 np = __fmul2_rn(xp, nb);
              const float2 pe = __ffma2_rn(xp, nb, __fmul2_rn(xp, b));  // (-x b) - np
              const float2 t = __fadd2_rn(sp, np), bb = __ffma2_rn(sp, m1, t);
              const float2 se = __fadd2_rn(__ffma2_rn(__ffma2_rn(bb, m1, t), m1, sp), __ffma2_rn(bb, m1, np));
              sp = t;
              cp = __ffma2_rn(xp, nl, __fadd2_rn(cp, __fadd2_rn(pe, se)));
            }
          float e;
          two_sum(sp.x, sp.y, s[q], e);
          c[q] = (cp.x + cp.y) + e;
        }
      } else {
#pragma unroll
        for (int q = 0; q < RPW; ++q) {
          s[q] = 0.f;
          c[q] = 0.f;
#pragma unroll
          for (int v = 0; v < VMAX; ++v)
#pragma unroll
            for (int e = 0; e < VW; ++e) {
              float pr, pe, se;
              two_prod(x[q][v][e], -bh[v][e], pr, pe);
              two_sum(s[q], pr, s[q], se);
              c[q] = fmaf(x[q][v][e], -bl[v][e], c[q] + (pe + se));
            }
        }
      }
      // Sums over the warp as a transposed butterfly: at each of the first levels a lane keeps half of
      // its rows, so that the rest of the tree sums one row per lane
      int off = 16;
      auto add = [&](float ks, float kc, float os, float oc, float &so, float &co) {
        float e;
        const float s2 = __shfl_xor_sync(0xffffffffu, os, off), c2 = __shfl_xor_sync(0xffffffffu, oc, off);
        two_sum(ks, s2, so, e);
        co = (kc + c2) + e;
      };
#pragma unroll
      for (int n = RPW; n > 1; n >>= 1, off >>= 1) {
        const bool upper = (lane & off) != 0;
#pragma unroll
        for (int j = 0; j < n / 2; ++j)
          add(upper ? s[j + n / 2] : s[j], upper ? c[j + n / 2] : c[j], upper ? s[j] : s[j + n / 2],
              upper ? c[j] : c[j + n / 2], s[j], c[j]);
      }
#pragma unroll
      for (; off > 0; off >>= 1) add(s[0], c[0], s[0], c[0], s[0], c[0]);
      // this lane's row: its residual, then every row's to every lane
      float rh, re;
      two_sum(yl, s[0], rh, re);
      const float rl = rh + (re + c[0]);
      if (a.r0 && (lane & (32 / RPW - 1)) == 0 && i0 + row_l < a.nrows) a.r0[i0 + row_l] = rl;
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        int src = 0, o = 16;
#pragma unroll
        for (int n = RPW; n > 1; n >>= 1, o >>= 1)
          if (q % n >= n / 2) src |= o;
        r[q] = __shfl_sync(0xffffffffu, rl, src);
      }
    } else {
      float s[RPW];
#pragma unroll
      for (int q = 0; q < RPW; ++q) {
        s[q] = 0.f;
#pragma unroll
        for (int v = 0; v < VMAX; ++v)
#pragma unroll
          for (int e = 0; e < VW; ++e) s[q] = fmaf(x[q][v][e], bh[v][e], s[q]);
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1)
#pragma unroll
        for (int q = 0; q < RPW; ++q) s[q] += __shfl_xor_sync(0xffffffffu, s[q], off);
#pragma unroll
      for (int q = 0; q < RPW; ++q) r[q] = yr[REBASE ? 0 : q] - s[q];
    }
#pragma unroll
    for (int q = 0; q < RPW; ++q)
#pragma unroll
      for (int v = 0; v < VMAX; ++v)
#pragma unroll
        for (int e = 0; e < VW; ++e) gacc[v][e] = fmaf(x[q][v][e], r[q], gacc[v][e]);
    nacc += RPW;
    if (nacc >= kFlushRows) {
      nacc = 0;
#pragma unroll
      for (int v = 0; v < VMAX; ++v)
#pragma unroll
        for (int e = 0; e < VW; ++e) {
          const int col = (v * 32 + lane) * VW + e;
          if (col < 512) {
            float2 h = acc[col];
            float sum, err;
            two_sum(h.x, gacc[v][e], sum, err);
            acc[col] = make_float2(sum, h.y + err);
          }
          gacc[v][e] = 0.f;
        }
    }
  }
  if constexpr (kRing) asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  // fold the remainder and convert each (hi, lo) pair in place to one double
#pragma unroll
  for (int v = 0; v < VMAX; ++v)
#pragma unroll
    for (int e = 0; e < VW; ++e) {
      const int col = (v * 32 + lane) * VW + e;
      if (col < 512) {
        const float2 h = acc[col];
        sm[warp][col] = ((double)h.x + (double)gacc[v][e]) + (double)h.y;
      }
    }
  if (REBASE && a.beta0 && blockIdx.x == 0) {
    for (int c = threadIdx.x; c < d; c += blockDim.x) a.beta0[c] = beta[c];
    if (threadIdx.x == 0) a.st->rebases += 1;
  }
  cta_partial(sm, d, a.partials + (size_t)blockIdx.x * d);
}

// One launch for both residual forms: a launch that returns at once still cost its start (1.4 us) and
// the host the call.
template <int VW, int VMAX, int RPW>
__global__ void __launch_bounds__(kGradThreads, 2) k_grad_mixed(const GradArgs a) {
  __shared__ __align__(16) double sm[kWarps][512];
  dependent_start();
  if (a.check_done && a.st->done) return;
  if (a.st->rebase) {
    grad_mixed_body<VW, VMAX, 1, RPW>(a, sm);
  } else {
    if (a.st->dc && a.st->bfnext) return;  // correction form: a correction step, not a pass
    grad_mixed_body<VW, VMAX, 0, RPW>(a, sm);
  }
}

// ---------------------------------------------------------------- reduction and update
struct ReduceArgs {
  const double *partials;
  int nblk, d;
  double scale;
  double *g;
  DevState *st;
  int check_done;
  double *g0;            // correction form: g(beta_e)
  const double *Gb;      // correction form: the Gram matrix and fl32(beta - beta_e)
  const float *delta_e;
  const double *rhs;     // added to the gradient of a pass
};

// g of this iteration, eight columns per CTA: the sum of the per-CTA partials of a pass, or, on a
// correction step, g0 - G_b delta_e (one warp per row of G_b).  Latency: every thread has all its
// partials (at most 12 per round) on their way at once, and the sums are short trees (an FP64 add
// takes 64 cycles on this part, a double shuffle and add 101).  5.1 -> 2.9 us at d = 37 against sums in
// four chains; the correction step's product used to be a launch of its own (2.6 us).
__global__ void __launch_bounds__(256) k_reduce(const ReduceArgs a) {
  __shared__ double sm[8][8];
  dependent_start();
  DevState *st = a.st;
  if (blockIdx.x == 0 && threadIdx.x == 0) st->t_red = device_ns();
  if (a.check_done && st->done) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, d = a.d;
  if (a.g0 && st->dc && st->bfnext && !st->rebase) {
    const int i = blockIdx.x * 8 + warp;
    if (i >= d) return;
    const double *row = a.Gb + (size_t)i * d;
    // four independent FP64 sums, fixed order
    double h0 = 0.0, h1 = 0.0, h2 = 0.0, h3 = 0.0;
    int k = lane;
    for (; k + 96 < d; k += 128) {
      h0 = fma(row[k], (double)a.delta_e[k], h0);
      h1 = fma(row[k + 32], (double)a.delta_e[k + 32], h1);
      h2 = fma(row[k + 64], (double)a.delta_e[k + 64], h2);
      h3 = fma(row[k + 96], (double)a.delta_e[k + 96], h3);
    }
    for (; k < d; k += 32) h0 = fma(row[k], (double)a.delta_e[k], h0);
    const double h = warp_sum((h0 + h1) + (h2 + h3));
    if (lane == 0) a.g[i] = a.g0[i] - h;
    return;
  }
  const int c = blockIdx.x * 8 + (lane & 7), b0 = threadIdx.x >> 3;  // column; partials b0, b0 + 32, ...
  double s = 0.0;
  if (c < d) {
    for (int base = b0; base < a.nblk; base += 32 * 12) {
      double v[12];
#pragma unroll
      for (int k = 0; k < 12; ++k) v[k] = base + 32 * k < a.nblk ? a.partials[(size_t)(base + 32 * k) * d + c] : 0.0;
#pragma unroll
      for (int k = 0; k < 6; ++k) v[k] += v[k + 6];
      s += ((v[0] + v[1]) + (v[2] + v[3])) + (v[4] + v[5]);
    }
  }
  s += __shfl_xor_sync(0xffffffffu, s, 8);
  s += __shfl_xor_sync(0xffffffffu, s, 16);
  if (lane < 8) sm[warp][lane] = s;
  __syncthreads();
  if (warp == 0) {
    double t = sm[lane >> 3][lane & 7] + sm[(lane >> 3) + 4][lane & 7];
    t += __shfl_xor_sync(0xffffffffu, t, 8);
    t += __shfl_xor_sync(0xffffffffu, t, 16);
    if (lane < 8 && c < d) {
      double v = a.scale * t;
      if (a.rhs) v += a.rhs[c];
      if (a.g0) a.g0[c] = v;  // exact pass: keep g(beta_e)
      a.g[c] = v;
    }
  }
}

struct UpdArgs {
  UpdateArgs u;
  double *part;  // 3 doubles per CTA
};

// beta+ = beta + mu H^{-1} g + eta (beta - beta_prev); one warp per row of H^{-1}.
__global__ void __launch_bounds__(256) k_update(const UpdArgs A, DevState *st) {
  const UpdateArgs &a = A.u;
  __shared__ double s_red[3][8];
  __shared__ int s_last;
  dependent_start();
  if (a.check_done && st->done) return;
  if (a.stage2 && blockIdx.x == 0 && threadIdx.x == 0) st->t_upd = device_ns();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int d = a.d;
  const int t = st->iter;
  const double *b = a.beta_ring + (size_t)(t % 3) * d;
  const double *bp = a.beta_ring + (size_t)((t + 2) % 3) * d;
  double *bn = a.beta_ring + (size_t)((t + 1) % 3) * d;
  const int i = blockIdx.x * 8 + warp;
  // correction form: whether this iteration's pass was exact (over X); read before the last block
  // of this kernel changes the state
  const bool corr_exact = a.stage2 && a.mixed && st->dc && (st->rebase || !st->bfnext);
  double ds = 0.0, nn = 0.0, dd = 0.0;
  if (i < d) {
    const double *Hrow = a.Hinv + (size_t)i * d;
    // four independent partial sums (the FP64 FMA latency is long on this part), fixed order
    double h0 = 0.0, h1 = 0.0, h2 = 0.0, h3 = 0.0;
    int k = lane;
    for (; k + 96 < d; k += 128) {
      h0 = fma(Hrow[k], a.g[k], h0);
      h1 = fma(Hrow[k + 32], a.g[k + 32], h1);
      h2 = fma(Hrow[k + 64], a.g[k + 64], h2);
      h3 = fma(Hrow[k + 96], a.g[k + 96], h3);
    }
    for (; k < d; k += 32) h0 = fma(Hrow[k], a.g[k], h0);
    double h = warp_sum((h0 + h1) + (h2 + h3));
    if (lane == 0) {
      const double mom = a.first ? 0.0 : a.eta * (b[i] - bp[i]);
      const double v = b[i] + a.mu * h + mom;
      bn[i] = v;
      ds = (v - b[i]) * (v - b[i]);
      nn = v * v;
      if (a.mixed) {
        const double del = v - a.beta0[i];
        a.delta32[i] = (float)del;
        dd = del * del;
        if (a.beta_e) {
          if (corr_exact) a.beta_e[i] = b[i];  // the gradient of this pass is g(b)
          a.delta_e[i] = (float)(v - a.beta_e[i]);
        }
      }
      if (a.hist && t < a.hist_cap) a.hist[(size_t)t * d + i] = v;
    }
  }
  if (lane == 0) { s_red[0][warp] = ds; s_red[1][warp] = nn; s_red[2][warp] = dd; }
  __syncthreads();
  if (warp == 0) {  // eight lanes per sum, a fixed tree
    double x = lane < 24 ? s_red[lane >> 3][lane & 7] : 0.0;
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    if (lane < 24 && (lane & 7) == 0) {
      A.part[3 * blockIdx.x + (lane >> 3)] = x;
      __threadfence();
    }
    __syncwarp();
    if (lane == 0) {
      const unsigned prev = atomicAdd(&st->upd_count, 1u);
      s_last = (prev == gridDim.x - 1);
    }
  }
  __syncthreads();
  if (!s_last || warp != 0) return;
  __threadfence();
  // the last CTA sums the per-CTA partials with its first warp: lane l takes CTAs l, l + 32, ...
  // in order, then a fixed shuffle tree (no serial chain of L2 round trips)
  double x0 = 0, x1 = 0, x2 = 0;
  for (unsigned c = lane; c < gridDim.x; c += 32) {
    x0 += __ldcg(A.part + 3 * c + 0);
    x1 += __ldcg(A.part + 3 * c + 1);
    x2 += __ldcg(A.part + 3 * c + 2);
  }
  x0 = warp_sum(x0);
  x1 = warp_sum(x1);
  x2 = warp_sum(x2);
  // correction form: a correction step more than twice the size of the cycle's first step is the
  // correction iteration diverging (an ill-conditioned X): it is not taken.  The kept iterate is
  // copied into the new slot (so the momentum of the next step is zero), the vectors of the base
  // points are formed from it, the norms are those of the kept iterate, and the next pass is exact.
  const bool reject = corr_exact == false && a.stage2 && a.mixed && st->dc && x0 > 4.0 * st->step_ref;
  if (reject) {
    double k1 = 0.0, k2 = 0.0;
    for (int i = lane; i < d; i += 32) {
      bn[i] = b[i];
      const double del = b[i] - a.beta0[i];
      a.delta32[i] = (float)del;
      if (a.beta_e) a.delta_e[i] = (float)(b[i] - a.beta_e[i]);
      if (a.hist && t < a.hist_cap) a.hist[(size_t)t * d + i] = b[i];
      k1 += b[i] * b[i];
      k2 += del * del;
    }
    x0 = 0.0;
    x1 = warp_sum(k1);
    x2 = warp_sum(k2);
  }
  if (lane != 0) return;
  st->upd_count = 0;
  // the relative step sqrt(x0 / x1) is compared squared: FP64 square roots, divisions and powers by one
  // thread took part of this kernel's time (with the sums as trees 8.5 -> 6.6 us at d = 37)
  const double n1 = x1 > 0.0 ? x1 : 1.0;
  st->step2 = x0;
  st->norm2 = n1;
  const bool small = a.thr > 0.0 && x0 <= a.thr * a.thr * n1;
  const int tn = t + 1;
  st->iter = tn;
  if (!isfinite(x0) || !isfinite(x1)) {
    st->status |= ST_NUMERIC;
    st->done = 1;
  }
  if (a.stage2) {
    // x2 = ||beta+ - beta_0||^2, x1 = ||beta+||^2, x0 = ||beta+ - beta||^2
    const bool corr = a.mixed && st->dc;
    const int exact = !corr || st->rebase || !st->bfnext;  // this iteration's pass was over X
    const int k2 = t - a.hist_base;
    if (k2 >= 0 && k2 < (int)sizeof(st->mode_hist)) st->mode_hist[k2] = exact ? 0 : 1;
    if (exact) st->ns_pass += st->t_red - st->t_mark;
    else st->ns_corr += st->t_upd - st->t_red;  // not the wait for the Gram matrix before the first one
    st->t_mark = device_ns();
    if (corr && exact) {
      // a cycle (exact pass + k correction steps, 1 + k c passes' worth of time for a correction
      // step costing c passes) that shrank the exact step by less than rho^(1 + k c), what plain
      // steps gain in that time, or by less than 10x: the BF16 Hessian term is too coarse for
      // these data (ill-conditioned X; its relative error, which sets a cycle's gain, is then
      // above 0.1, where the cycles, plain fixed-point steps without momentum, fall behind the
      // full form and the first cycle's gain, measured from the large first step of the 2nd
      // stage, overstates the gain in the error), so the remaining steps take the full form (its
      // next pass reads the r0 this exact pass wrote).  x0 and step_prev are squared norms.  A step
      // that meets the stopping test ends the fit either way and decides nothing.
      const double gain = a.gain[st->ninner < kMaxInner ? st->ninner : kMaxInner];
      if (st->step_prev > 0.0 && x0 > st->step_prev * gain && !small) {
        st->dc = 0;
        st->dc_fell_back = 1;
      }
      st->step_prev = x0;
      st->step_ref = x0;
      st->ninner = 0;
    } else if (corr) {
      st->ninner += 1;
    }
    const bool may_stop = !(corr && !exact);  // the correction form stops on exact steps only
    if (may_stop && small) st->done = 1;
    else if (tn >= a.T) {
      st->done = 1;
      if (a.thr > 0.0) st->status |= ST_NOTCONV;
    }
    if (a.mixed) {
      // next pass exact: the steps have shrunk to 1/10^4 of the cycle's first step (the correction
      // iteration has then settled at its fixed point, within ~1e-4 of the exact one on the
      // benchmark data), or one meets the stopping test (the stop itself waits for an exact step),
      // or a step grew beyond the cycle's first step (the correction iteration diverging on an
      // ill-conditioned X), or the cycle has taken 20 correction steps (twice what a contraction of
      // rho = 0.41 per step needs for 1e-4; steps count toward T); the exact pass
      // re-bases (error-free residuals) only when the drift from beta_0 exceeds 2^-10 ||beta||, so
      // that the FP32 residual r0 - X (beta - beta_0) stays within ~2^-34 ||X|| ||beta||
      if (st->dc) {
        const bool next_exact =
            !exact && (reject || x0 < 1e-8 * st->step_ref || x0 > st->step_ref || st->ninner >= kMaxInner || small);
        st->bfnext = next_exact ? 0 : 1;
        st->rebase = (next_exact && x2 > 0x1p-20 * x1) ? 1 : 0;
      } else {
        st->bfnext = 0;
        st->rebase = (x2 > 0x1p-20 * x1 && x2 > 0x1p20 * x0) ? 1 : 0;
      }
    }
    // the host polls this word (pinned host memory) for the iterations done and the stop flag
    if (a.mail)
      asm volatile("st.relaxed.sys.global.u32 [%0], %1;" ::"l"(a.mail), "r"((unsigned)tn << 1 | (unsigned)st->done) : "memory");
  }
}

__global__ void k_copy_beta(const double *ring, const DevState *st, int d, double *out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < d) out[c] = ring[(size_t)(st->iter % 3) * d + c];
}

template <class K>
cudaError_t launch1(K kern, int nblk, const GradArgs &a, cudaStream_t s, bool dep) {
  return launch_dep(kern, (unsigned)nblk, kGradThreads, 0, s, dep, a);
}

// FP64 kernel with its register tile sized to d (columns per lane) and several rows per warp
// iteration (fewer as the rows widen)
#define SLSE_GRAD64_VARIANTS(Tx, VW, F)                                              \
  F(1, 4, (k_grad_f64<Tx, VW, 1, 4, false>)) F(2, 4, (k_grad_f64<Tx, VW, 2, 4, false>)) \
  F(3, (VW == 1 ? 4 : 2), (k_grad_f64<Tx, VW, 3, (VW == 1 ? 4 : 2), false>))            \
  F(4, (VW == 1 ? 4 : 2), (k_grad_f64<Tx, VW, 4, (VW == 1 ? 4 : 2), false>))            \
  F(6, (VW == 1 ? 2 : 1), (k_grad_f64<Tx, VW, 6, (VW == 1 ? 2 : 1), (VW == 2)>))        \
  F(8, (VW == 1 ? 2 : 1), (k_grad_f64<Tx, VW, 8, (VW == 1 ? 2 : 1), (VW == 2)>))
#define SLSE_GRAD64_WIDE(Tx, V) (k_grad_f64<Tx, 1, V, 1, true>)
template <class Tx, int VW>
cudaError_t launch_f64(int d, int nblk, const GradArgs &a, cudaStream_t s, bool dep) {
  constexpr int per = 32 * VW;
  auto go = [&](auto kern, size_t row_bytes, int rows) -> cudaError_t {
    const size_t smem = (size_t)kWarps * 2 * rows * row_bytes;  // at most 64 KB
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_dep(kern, (unsigned)nblk, kGradThreads, smem, s, dep, a);
  };
#define SLSE_GRAD64_CASE(V, R, K) if (d <= V * per) return go(K, V * per * sizeof(Tx), R);
  SLSE_GRAD64_VARIANTS(Tx, VW, SLSE_GRAD64_CASE)
  if constexpr (VW == 1) {
    if (d <= 12 * per) return go(SLSE_GRAD64_WIDE(Tx, 12), 12 * per * sizeof(Tx), 1);
    if (d <= 16 * per) return go(SLSE_GRAD64_WIDE(Tx, 16), 16 * per * sizeof(Tx), 1);
  }
#undef SLSE_GRAD64_CASE
  return cudaErrorInvalidValue;
}

inline bool aligned(const void *p, int64_t ld, int64_t elem_bytes, int vw) {
  return (reinterpret_cast<uintptr_t>(p) % (size_t)(vw * elem_bytes) == 0) && (ld % vw == 0);
}

}  // namespace

int grad_grid(int nsm) { return 2 * nsm; }

cudaError_t launch_grad(int mode, int xdtype, const void *X, int64_t ldx, const void *Y, int64_t nrows, int d,
                        const double *beta_ring, DevState *st, const float *delta32, float *r0, double *beta0,
                        double *partials, int nblk, int check_done, cudaStream_t s, bool dep) {
  GradArgs a{X, ldx, Y, nrows, d, beta_ring, st, delta32, r0, beta0, partials, check_done};
  if (d > 512 || d < 1) return cudaErrorInvalidValue;
  switch (mode) {
    case GM_F64:
    case GM_STAGE1_F64:
      if (xdtype == SLSE_F64) {
        if (d % 2 == 0 && aligned(X, ldx, 8, 2)) return launch_f64<double, 2>(d, nblk, a, s, dep);
        return launch_f64<double, 1>(d, nblk, a, s, dep);
      } else {
        if (d % 2 == 0 && aligned(X, ldx, 4, 2)) return launch_f64<float, 2>(d, nblk, a, s, dep);
        return launch_f64<float, 1>(d, nblk, a, s, dep);
      }
    case GM_STAGE1_BF16:
      // the sketch buffer's padding columns are never written: the vector path requires
      // d % 8 == 0 so that no padding word is read
      // lanes cover 8 columns per word: one word per lane up to d = 256 (more rows in flight)
      if (d % 8 == 0 && ldx % 8 == 0 && aligned(X, ldx, 2, 8))
        return d <= 256 ? launch1(k_grad_bf16v<1, 6>, nblk, a, s, dep) : launch1(k_grad_bf16v<2, 4>, nblk, a, s, dep);
      return launch1(k_grad_bf16s<16>, nblk, a, s, dep);
    case GM_MIXED: {
      if (xdtype != SLSE_F32) return cudaErrorInvalidValue;
      const bool vec = d % 4 == 0 && aligned(X, ldx, 4, 4);
      // rows in flight per warp grow as d shrinks (the same 32 x-values per lane)
      if (!vec) return launch1(k_grad_mixed<1, 16, 1>, nblk, a, s, dep);
      auto go = [&](auto kern) -> cudaError_t {
        constexpr int smem = kWarps * 2 * 8 * 32 * 16;  // two stages of eight 16-byte pieces per lane
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        return launch_dep(kern, (unsigned)nblk, kGradThreads, smem, s, dep, a);
      };
      if (d <= 128) return go(k_grad_mixed<4, 1, 8>);
      if (d <= 256) return go(k_grad_mixed<4, 2, 4>);
      return go(k_grad_mixed<4, 4, 2>);
    }
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t preload_grad_kernels() {
  // every kernel launch_grad (modes GM_F64 and GM_MIXED) and launch_reduce can pick
  const void *k[] = {
#define SLSE_GRAD64_PTR(V, R, K) (const void *)K,
      SLSE_GRAD64_VARIANTS(double, 2, SLSE_GRAD64_PTR) SLSE_GRAD64_VARIANTS(double, 1, SLSE_GRAD64_PTR)
      SLSE_GRAD64_VARIANTS(float, 2, SLSE_GRAD64_PTR) SLSE_GRAD64_VARIANTS(float, 1, SLSE_GRAD64_PTR)
      (const void *)SLSE_GRAD64_WIDE(double, 12), (const void *)SLSE_GRAD64_WIDE(double, 16),
      (const void *)SLSE_GRAD64_WIDE(float, 12), (const void *)SLSE_GRAD64_WIDE(float, 16),
#undef SLSE_GRAD64_PTR
      (const void *)k_grad_mixed<1, 16, 1>, (const void *)k_grad_mixed<4, 1, 8>,
      (const void *)k_grad_mixed<4, 2, 4>, (const void *)k_grad_mixed<4, 4, 2>,
      (const void *)k_reduce};
  for (const void *f : k) {
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_reduce(const double *partials, int nblk, int d, double scale, double *g, DevState *st,
                          int check_done, cudaStream_t s, double *g0, const double *Gb, const float *delta_e,
                          const double *rhs, bool dep) {
  const ReduceArgs a{partials, nblk, d, scale, g, st, check_done, g0, Gb, delta_e, rhs};
  return launch_dep(k_reduce, (unsigned)(d + 7) / 8, 256, 0, s, dep, a);
}

cudaError_t launch_update(const UpdateArgs &a, DevState *st, cudaStream_t s, bool dep) {
  // per-CTA partial sums live right after the DevState's own cache line block
  UpdArgs A{a, reinterpret_cast<double *>(st + 1)};
  return launch_dep(k_update, (unsigned)(a.d + 7) / 8, 256, 0, s, dep, A, st);
}

cudaError_t launch_copy_beta(const double *beta_ring, DevState *st, int d, double *out, cudaStream_t s) {
  k_copy_beta<<<(d + 255) / 256, 256, 0, s>>>(beta_ring, st, d, out);
  return cudaGetLastError();
}

}  // namespace slse
