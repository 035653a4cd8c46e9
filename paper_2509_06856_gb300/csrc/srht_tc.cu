// Mixed-precision SRHT passes over groups of 2^10 and 2^11 rows on the tcgen05 tensor cores.
//
// What bounds the cluster form (srht.cu): 7/8 of every FP32 tile crosses the cluster through
// distributed shared memory, and a CTA's life is a chain of latencies.  Here the group stays on one
// SM: H_{2^L} = H_J (x) H_128 (row j = 128 jh + jl, J = 2^(L-7)), and H_128 down the rows jl is a
// matrix product with a constant +-1 matrix, D[kl][jh, c] = sum_jl H_128[kl][jl] X[jh, jl][c], whose
// FP32 accumulator (128 lanes x 512 columns: the whole group of 2^L rows x C = 512 / J columns)
// fills tensor memory.  H_J is then J adds and subtracts deep in registers, between values of one
// lane.  Products with +-1 are exact, so only the FP32 sums round, as the butterflies' did:
//  - pass 2 reads the BF16 intermediate, one product per element;
//  - pass 1 reads FP32 rows, each split exactly into three BF16 terms of 8 bits (by truncation), and
//    accumulates three products.
//
// One persistent CTA per SM, warps by role: eight producers load row segments (gathered through the
// signed permutation in pass 1) and write operand chunks of 16 jl x J jh x C columns into a ring of
// shared-memory stages in the 128-byte-swizzled MN-major layout (64 operand columns: two jh of 32 or
// one of 64 columns); one thread issues the MMAs; sixteen epilogue warps (four per 32 lanes of tensor
// memory) take a few columns of all J values at a time, transform, round to BF16 and park the packed
// words in tensor memory columns already read, so placed that a 16 x 256-bit load then gives each lane
// 16 contiguous bytes of an output row and four lanes a row segment.  The rings keep the loads running
// while the epilogue holds tensor memory: pass 2 copies straight into nine operand stages; pass 1
// copies FP32 rows into three stages of its own (96 KB on their way), from which the same threads
// split them into two operand stages.
// Measured (GB300) against the cluster form: N' = 2^22, d = 512, FP32 in, half the rows kept: pass 1
// 3.45 -> 3.05 ms, pass 2 3.22 -> 1.49 ms; sketch of 3000000 x 384 in BF16 5.43 -> 3.65 ms (0.25 of it
// by the draws' sort), its error against 64-bit arithmetic unchanged (2.4e-3, the BF16 roundings).  What bounds
// pass 1 now: the producers' splitting and the part of the epilogue that holds tensor memory (the loads
// alone would take 2.2 ms).  Tried on the way: eight producer warps loading into registers (32 KB on their way
// per SM: 3.39 ms at 3000000 x 384, 2.24 ms now), eight epilogue warps, H as an MN-major operand (the MMAs ran at
// half the rate), all output rows read back before the first store (spills).
// Every mbarrier wait is bounded (ST_TIMEOUT: the fit reports it, slse_sketch's output is NaN then);
// copies in flight are awaited and tensor memory is freed on that path too.
#include <climits>

#include "srht_args.cuh"
#include "tc_common.cuh"

namespace slse {
namespace {

constexpr int kProdWarps = 8, kEpiWarps = 16;
constexpr int kTcThreads = 32 * (kProdWarps + kEpiWarps + 1);
constexpr int kChunk = 16384;     // operand bytes of one chunk (one BF16 term)
constexpr int kHBytes = 32768;    // H_128 as the A operand
constexpr int kKSteps = 8;        // chunks of a group: 128 jl, 16 at a time
constexpr int kInFlight = 6;      // pass 2: chunks on their way per thread

constexpr int kRaw = 3;           // pass 1: FP32 chunks on their way or being split
constexpr int kRawBytes = 32768;  // of an FP32 chunk

template <bool F32> constexpr int ring_stages() { return F32 ? 2 : 9; }
template <bool F32> constexpr int stage_bytes() { return F32 ? 3 * kChunk : kChunk; }

struct TcPassArgs {
  GroupArgs a;
  int64_t ntiles;
  float scale;
};

// shared-memory descriptor of a 128-byte-swizzled operand, 1024 bytes between its 8-row groups (along
// K when it is MN-major, and lbo = bytes between 64-element groups along N; along M when it is K-major)
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr, uint32_t lbo) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}

// N consecutive columns of the thread's lane
template <int N> __device__ __forceinline__ void tmem_ld(uint32_t t, uint32_t *v) {
  if constexpr (N == 2)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(t) : "memory");
  else
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(t) : "memory");
}
// 16 lanes x 8 G columns: thread t gets, for each group of 8 columns, columns 2 (t mod 4), + 1 of lane
// t div 4 (v[4 g], v[4 g + 1]) and of lane t div 4 + 8 (v[4 g + 2], v[4 g + 3])
template <int G> __device__ __forceinline__ void tmem_ld_rows(uint32_t t, uint32_t *v) {
  if constexpr (G == 2)
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(t) : "memory");
  else
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                 "%13, %14, %15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(t) : "memory");
}
template <int N> __device__ __forceinline__ void tmem_st(uint32_t t, const uint32_t *v) {
  if constexpr (N == 1)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(t), "r"(v[0]) : "memory");
  else
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(t), "r"(v[0]), "r"(v[1]) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Byte offset in a chunk of 16-byte unit `p` of the segment of row (jh, k), k = jl mod 16: two jh
// (32 columns) or one (64) share a 128-byte line of the swizzled layout.
template <int L> __device__ __forceinline__ uint32_t chunk_off(int jh, int k, int p) {
  const int atom = L == 11 ? jh >> 1 : jh, unit = L == 11 ? ((jh & 1) << 2) + p : p;
  return (uint32_t)(atom * 2048 + k * 128 + ((unit ^ (k & 7)) << 4));
}

// Exact split of four FP32 values (signs of x flipped by sg) into three BF16 terms each (truncated:
// 8 + 8 + 8 bits), packed in pairs.  chk collects the last terms: it becomes NaN when a value is not
// finite, whose terms are then not meant (split3_rare).
__device__ __forceinline__ void split3(const float4 x, uint32_t sg, uint2 &h, uint2 &m, uint2 &l, float2 &chk) {
  const float2 m1 = make_float2(-1.f, -1.f);
  const uint32_t u[4] = {__float_as_uint(x.x) ^ sg, __float_as_uint(x.y) ^ sg, __float_as_uint(x.z) ^ sg,
                         __float_as_uint(x.w) ^ sg};
  uint32_t hw[2], mw[2], lw[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const float2 v = make_float2(__uint_as_float(u[2 * e]), __uint_as_float(u[2 * e + 1]));
    const float2 hb = make_float2(__uint_as_float(u[2 * e] & 0xFFFF0000u), __uint_as_float(u[2 * e + 1] & 0xFFFF0000u));
    const float2 r = __ffma2_rn(hb, m1, v);
    const float2 mb = make_float2(__uint_as_float(__float_as_uint(r.x) & 0xFFFF0000u),
                                  __uint_as_float(__float_as_uint(r.y) & 0xFFFF0000u));
    const float2 s = __ffma2_rn(mb, m1, r);
    chk = __fadd2_rn(chk, s);
    hw[e] = __byte_perm(u[2 * e], u[2 * e + 1], 0x7632);
    mw[e] = __byte_perm(__float_as_uint(r.x), __float_as_uint(r.y), 0x7632);
    lw[e] = __byte_perm(__float_as_uint(s.x), __float_as_uint(s.y), 0x7632);
  }
  h = make_uint2(hw[0], hw[1]);
  m = make_uint2(mw[0], mw[1]);
  l = make_uint2(lw[0], lw[1]);
}
// The same with an infinity or a NaN in the first term alone.
__device__ __noinline__ void split3_rare(const float4 x, uint32_t sg, uint2 &h, uint2 &m, uint2 &l) {
  const uint32_t u[4] = {__float_as_uint(x.x), __float_as_uint(x.y), __float_as_uint(x.z), __float_as_uint(x.w)};
  uint32_t w[3][4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float v = __uint_as_float(u[e] ^ sg);
    if ((u[e] & 0x7F800000u) == 0x7F800000u) {
      w[0][e] = v != v ? 0x7FC0u : (u[e] ^ sg) >> 16;
      w[1][e] = w[2][e] = 0u;
    } else {
      const float r = v - __uint_as_float((u[e] ^ sg) & 0xFFFF0000u);
      const float s = r - __uint_as_float(__float_as_uint(r) & 0xFFFF0000u);
      w[0][e] = (u[e] ^ sg) >> 16;
      w[1][e] = __float_as_uint(r) >> 16;
      w[2][e] = __float_as_uint(s) >> 16;
    }
  }
  h = make_uint2(w[0][0] | (w[0][1] << 16), w[0][2] | (w[0][3] << 16));
  m = make_uint2(w[1][0] | (w[1][1] << 16), w[1][2] | (w[1][3] << 16));
  l = make_uint2(w[2][0] | (w[2][1] << 16), w[2][2] | (w[2][3] << 16));
}

// POLLS: a test has set a limit to the waits (a form of its own: the test of the limit in every wait cost
// 30 us of 3.65 ms at 3000000 x 384)
template <bool F32, int L, bool POLLS>
__global__ void __launch_bounds__(kTcThreads, 1) k_group_tc(const TcPassArgs A) {
  constexpr int J = 1 << (L - 7);      // rows jh
  constexpr int C = 512 / J;           // columns of a group
  constexpr int NST = ring_stages<F32>();
  constexpr int CC = 32 / J;           // columns an epilogue thread transforms at a time
  extern __shared__ uint8_t smem_raw[];
  uint8_t *sm = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *ring = sm + kHBytes;
  uint8_t *raw = ring + NST * stage_bytes<F32>();  // pass 1: FP32 chunks
  uint64_t *full = reinterpret_cast<uint64_t *>(raw + (F32 ? kRaw * kRawBytes : 0));
  uint64_t *empty = full + NST, *tfull = empty + NST, *tempty = tfull + 1, *fin = tempty + 1;
  uint32_t *tslot = reinterpret_cast<uint32_t *>(fin + 1);
  volatile int *abort_f = reinterpret_cast<volatile int *>(tslot + 1);
  unsigned *dummy = reinterpret_cast<unsigned *>(tslot + 2);
  // pass 2: output rows of two groups (16-byte aligned)
  int32_t *s_pos = reinterpret_cast<int32_t *>((reinterpret_cast<uintptr_t>(tslot + 3) + 15) & ~uintptr_t(15));
  const GroupArgs &a = A.a;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned *status = a.status ? a.status : dummy;
  const int d = a.d;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], kProdWarps);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, kEpiWarps);
    mbar_init(fin, 1);
    *abort_f = 0;
    *dummy = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // H_128[m][k] = (-1)^popcount(m & k) as the K-major A operand (two halves of 64 k); symmetric, so
  // the roles of the two indices do not matter
  for (int e = threadIdx.x; e < 128 * 16; e += kTcThreads) {
    const int k = e >> 4, mg = e & 15;  // row k, elements m = 8 mg ..
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int m0 = 8 * mg + 2 * q;
      w[q] = ((__popc(m0 & k) & 1) ? 0xBF80u : 0x3F80u) | (((__popc((m0 + 1) & k) & 1) ? 0xBF80u : 0x3F80u) << 16);
    }
    *reinterpret_cast<uint4 *>(sm + (mg >> 3) * 16384 + k * 128 + (((mg & 7) ^ (k & 7)) << 4)) =
        make_uint4(w[0], w[1], w[2], w[3]);
  }
  fence_proxy_async_smem();
  if (warp == kProdWarps + kEpiWarps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tslot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  const int ntile = (int)((A.ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x);  // of this CTA
  const int nchunk = ntile * kKSteps;
  auto wait_one = [&](uint64_t *bar, uint32_t parity) -> bool {
    if constexpr (POLLS) return mbar_wait_polls(bar, parity, abort_f, status, a.wait_polls);
    else return mbar_wait(bar, parity, abort_f, status);
  };
  // a wait of a whole warp, with one result for all lanes
  auto wait_all = [&](uint64_t *bar, uint32_t parity) -> bool { return __all_sync(0xFFFFFFFFu, wait_one(bar, parity)); };
  auto tile_of = [&](int it, int64_t &g, int &col0) {
    const uint32_t item = blockIdx.x + (uint32_t)it * gridDim.x, gg = item / (uint32_t)a.nslab;
    g = (int64_t)gg;
    col0 = (int)(item - gg * (uint32_t)a.nslab) * C;
  };

  if (warp < kProdWarps) {
    if constexpr (!F32) {
      // 16-byte units of BF16 rows, straight into the operand layout
      constexpr int UR = C / 8;       // units per row segment
      const int p = lane % UR;
      const char *W = static_cast<const char *>(a.in);
      const int64_t rowb = a.ldin * 2;
      uint32_t dst[4];
      int64_t off[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int rid = i * (8 * 32 / UR) + warp * (32 / UR) + lane / UR;
        const int k = rid & 15, jh = rid >> 4;
        dst[i] = smem_u32(ring) + chunk_off<L>(jh, k, p);
        off[i] = (int64_t)(jh * 128 + k) * a.istride * rowb;
      }
      const int64_t kstep = 16 * a.istride * rowb;
      int64_t g = 0;
      int col0 = 0;
      int done = 0;
      for (int n = 0; n < nchunk; ++n) {
        const int ks = n % kKSteps, st = n % NST;
        if (ks == 0) tile_of(n / kKSteps, g, col0);
        if (n >= NST && !wait_all(&empty[st], (uint32_t)((n - NST) / NST) & 1u)) break;
        const int col = col0 + p * 8;
        const char *src = W + in_row(a, 0, g) * rowb + (int64_t)col * 2 + ks * kstep;
        const int bytes = col < d ? 16 : 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst[i] + (uint32_t)st * kChunk),
                       "l"(bytes ? src + off[i] : W), "r"(bytes)
                       : "memory");
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        if (n >= kInFlight) {
          asm volatile("cp.async.wait_group %0;\n" ::"n"(kInFlight) : "memory");
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(&full[done % NST]);
          ++done;
        }
      }
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0 && !*abort_f)
        for (; done < nchunk; ++done) mbar_arrive(&full[done % NST]);
    } else {
      // FP32 rows: every thread copies its own 16-byte pieces into its slots of the raw ring, two
      // chunks ahead (their indices three ahead), then splits them with the sign applied
      constexpr int LR = C / 4;              // lanes per row segment
      const int cq = lane % LR, lg = lane / LR;
      // row i of this thread: L = 11 (4 rows a warp): k = warp mod 4 + 4 lg, jh = warp / 4 + 2 i;
      // L = 10 (2 rows a warp): k = warp + 8 lg, jh = i (the 8-byte stores of a warp fall on all banks)
      const int k = L == 11 ? (warp & 3) + 4 * lg : warp + 8 * lg;
      const float *X = static_cast<const float *>(a.in);
      float *cpy = static_cast<float *>(a.copy_out);
      const int32_t nrows = (int32_t)a.N;
      auto jh_of = [&](int i) { return L == 11 ? (warp >> 2) + 2 * i : i; };
      float4 *slot = reinterpret_cast<float4 *>(raw) + threadIdx.x;  // stage, i, thread
      const uint32_t rowb = (uint32_t)a.ldin * 4u;
      int32_t idn[8];  // row indices of the next chunk to copy
      // the group whose indices are loaded next, and the one whose rows are copied next
      int64_t gi = 0, gc = 0;
      int ci = 0, cc = 0;
      auto load_idx = [&](int n) {
        if (n % kKSteps == 0) tile_of(n / kKSteps, gi, ci);
        const int32_t *q = a.Psd + in_row(a, 0, gi) + ((n % kKSteps) * 16 + k);
#pragma unroll
        for (int i = 0; i < 8; ++i) idn[i] = __ldg(q + jh_of(i) * 128);
      };
      // copies chunk n (rows of the padding and columns past d as zeros); the signs of its rows, row i
      // at bit 7 - i
      auto copy_x = [&](int n) -> uint32_t {
        if (n % kKSteps == 0) tile_of(n / kKSteps, gc, cc);
        const int col = cc + cq * 4;
        const int want = col + 4 <= d ? 16 : (col < d ? (d - col) * 4 : 0);
        const char *base = reinterpret_cast<const char *>(X + (want ? col : 0));
        const uint32_t dst = smem_u32(slot + (n % kRaw) * (8 * 256));
        uint32_t sg = 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int32_t src = idn[i] ^ (idn[i] >> 31);
          sg = __funnelshift_l((uint32_t)idn[i], sg, 1);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst + i * 4096),
                       "l"(base + (uint64_t)(uint32_t)src * rowb), "r"(src < nrows ? want : 0)
                       : "memory");
        }
        return sg;
      };
      uint32_t sgn[3] = {0u, 0u, 0u};  // chunks n, n + 1, n + 2
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        if (n < nchunk) {
          load_idx(n);
          sgn[n] = copy_x(n);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
      }
      if (nchunk > 2) load_idx(2);
      for (int n = 0; n < nchunk; ++n) {
        const int st = n % NST;
        if (n + 2 < nchunk) {
          sgn[2] = copy_x(n + 2);
          if (n + 3 < nchunk) load_idx(n + 3);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        if (n >= NST && !wait_all(&empty[st], (uint32_t)((n - NST) / NST) & 1u)) break;
        asm volatile("cp.async.wait_group 2;\n" ::: "memory");
        uint8_t *base = ring + (size_t)st * stage_bytes<true>() + (cq & 1) * 8;
        const float4 *mine = slot + (n % kRaw) * (8 * 256);
        if (cpy) {  // pass 1 on host memory: the device copy of the rows read
          int64_t g;
          int col0;
          tile_of(n / kKSteps, g, col0);
          const int col = col0 + cq * 4;
#pragma unroll 1
          for (int i = 0; i < 8; ++i) {
            const int32_t v = __ldg(a.Psd + in_row(a, 0, g) + (jh_of(i) * 128 + (n % kKSteps) * 16 + k));
            const int32_t src = v ^ (v >> 31);
            if (src >= nrows) continue;
            float *q = cpy + src * a.ldin + col;
            const float4 x = mine[i * 256];
            if (col + 4 <= d) *reinterpret_cast<float4 *>(q) = x;
            else if (col < d) {
              q[0] = x.x;
              if (col + 1 < d) q[1] = x.y;
              if (col + 2 < d) q[2] = x.z;
            }
          }
        }
        float2 chk = make_float2(0.f, 0.f);
        uint8_t *q0 = base + chunk_off<L>(jh_of(0), k, cq >> 1);  // row i: 2048 bytes on
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          uint2 h, m, l;
          split3(mine[i * 256], (sgn[0] << (24 + i)) & 0x80000000u, h, m, l, chk);
          *reinterpret_cast<uint2 *>(q0 + i * 2048) = h;
          *reinterpret_cast<uint2 *>(q0 + i * 2048 + kChunk) = m;
          *reinterpret_cast<uint2 *>(q0 + i * 2048 + 2 * kChunk) = l;
        }
        if (chk.x + chk.y != chk.x + chk.y) {  // rare: a value is not finite
#pragma unroll 1
          for (int i = 0; i < 8; ++i) {
            uint2 h, m, l;
            split3_rare(mine[i * 256], (sgn[0] << (24 + i)) & 0x80000000u, h, m, l);
            *reinterpret_cast<uint2 *>(q0 + i * 2048) = h;
            *reinterpret_cast<uint2 *>(q0 + i * 2048 + kChunk) = m;
            *reinterpret_cast<uint2 *>(q0 + i * 2048 + 2 * kChunk) = l;
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&full[st]);
        sgn[0] = sgn[1];
        sgn[1] = sgn[2];
      }
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
  } else if (warp == kProdWarps + kEpiWarps) {
    if (lane == 0) {
      const uint32_t id = umma_idesc_bf16(128, 256) | (1u << 16);  // B MN-major
      const uint32_t hb = smem_u32(sm);
      bool ok = true;
      for (int it = 0; it < ntile && ok; ++it) {
        if (it > 0 && !wait_one(tempty, (uint32_t)(it - 1) & 1u)) break;
        tc_fence_after();
        for (int ks = 0; ks < kKSteps; ++ks) {
          const int n = it * kKSteps + ks, st = n % NST;
          if (!wait_one(&full[st], (uint32_t)(n / NST) & 1u)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t xb = smem_u32(ring + (size_t)st * stage_bytes<F32>());
          const uint64_t ad = desc_sw128(hb + (uint32_t)((ks >> 2) * 16384 + (ks & 3) * 32), 16u);
#pragma unroll
          for (int s = 0; s < (F32 ? 3 : 1); ++s)
#pragma unroll
            for (int h = 0; h < 2; ++h)
              umma_bf16(tmem + 256u * h, ad, desc_sw128(xb + (uint32_t)(s * kChunk + h * 8192), 2048u), id,
                        (ks > 0 || s > 0) ? 1u : 0u);
          umma_commit(&empty[st]);
        }
        if (ok) umma_commit(tfull);
      }
      // every MMA has completed before tensor memory is freed, also after a failed wait
      umma_commit(fin);
      volatile int never = 0;
      mbar_wait(fin, 0u, &never, status);
    }
    __syncwarp();
  } else {
    const int quad = warp & 3, part = (warp - kProdWarps) >> 2;  // lanes 32 quad .., one of four warps there
    const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16);
    const float scale = A.scale;
    constexpr int U = C / 32;   // 16-byte units of an output row per lane
    constexpr int KH = J / 4;   // output row groups kh per warp
    // step t of warp `part`: columns c = 4 CC t + CC part ..; its packed words (CC / 2 per kh) go where
    // the row load gives unit u = c / 8 to lane u mod 4: group 2 (u / 4) + (c / 4) mod 2 (of 8 columns),
    // word 2 (u mod 4) + (c / 2) mod 2
    auto park = [&](int t) -> uint32_t {
      const int c = 4 * CC * t + CC * part, u = c >> 3;
      return (uint32_t)((2 * (u >> 2) + ((c >> 2) & 1)) * 8 + 2 * (u & 3) + ((c >> 1) & 1));
    };
    __nv_bfloat16 *out = static_cast<__nv_bfloat16 *>(a.out);
    for (int it = 0; it < ntile; ++it) {
      int64_t g;
      int col0;
      tile_of(it, g, col0);
      const bool ok = wait_all(tfull, (uint32_t)it & 1u);
      // a warp whose wait failed still meets the others here, and the four agree to stop
      uint32_t failed;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %2, 0;\n\tbarrier.red.or.pred q, %1, 128, p;\n\t"
          "selp.u32 %0, 1, 0, q;\n\t}"
          : "=r"(failed)
          : "r"(1 + quad), "r"(ok ? 0u : 1u)
          : "memory");
      if (failed) break;
      tc_fence_after();
      if (a.pos) {  // this quadrant's entries of the group's output rows, read back below
        const int tt = part * 32 + lane;
        if (tt < J * 8) {
          const int e = (tt >> 3) * 128 + quad * 32 + (tt & 7) * 4;
          asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(s_pos + (it & 1) * (128 * J) + e)),
                       "l"(a.pos + out_row(a, e, g))
                       : "memory");
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
      }
      // All words go to columns that steps 0 and 1 read, so step 0's are parked a step late, after a
      // barrier behind the loads of step 1.
      uint32_t w[J][CC / 2];
#pragma unroll 1
      for (int t = 0; t < 4; ++t) {
        uint32_t r[J][CC];
        const uint32_t c0 = tq + (uint32_t)(4 * CC * t + CC * part);
#pragma unroll
        for (int j = 0; j < J; ++j) tmem_ld<CC>(c0 + (uint32_t)(j * C), r[j]);
        tmem_wait_ld();
        if (t == 1) {
          tc_fence_before();
          asm volatile("barrier.sync %0, 128;" ::"r"(1 + quad) : "memory");
          tc_fence_after();
#pragma unroll
          for (int j = 0; j < J; ++j) tmem_st<CC / 2>(tq + (uint32_t)(j * C) + park(0), w[j]);
        }
        float2 v[J][CC / 2];
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
          for (int e = 0; e < CC / 2; ++e)
            v[j][e] = make_float2(__uint_as_float(r[j][2 * e]), __uint_as_float(r[j][2 * e + 1]));
        const float2 m1 = make_float2(-1.f, -1.f), sc = make_float2(scale, scale);
#pragma unroll
        for (int h = 1; h < J; h <<= 1)
#pragma unroll
          for (int j = 0; j < J; ++j)
            if ((j & h) == 0)
#pragma unroll
              for (int e = 0; e < CC / 2; ++e) {
                const float2 x = v[j][e], y = v[j + h][e];
                v[j][e] = __fadd2_rn(x, y);
                v[j + h][e] = __ffma2_rn(y, m1, x);
              }
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
          for (int e = 0; e < CC / 2; ++e) {
            const float2 o = F32 ? v[j][e] : __fmul2_rn(v[j][e], sc);  // pass 1 is not scaled
            const __nv_bfloat162 b = __floats2bfloat162_rn(o.x, o.y);
            w[j][e] = *reinterpret_cast<const uint32_t *>(&b);
          }
        if (t > 0)
#pragma unroll
          for (int j = 0; j < J; ++j) tmem_st<CC / 2>(tq + (uint32_t)(j * C) + park(t), w[j]);
      }
      tmem_wait_st();
      if (a.pos) asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      tc_fence_before();
      asm volatile("barrier.sync %0, 128;" ::"r"(1 + quad) : "memory");  // every word is parked
      tc_fence_after();
      // this warp's output rows kh in units of 16 kl: a quarter is read and stored, then the rest read
      // (more does not fit the registers), and tensor memory is free for the next group
      constexpr int NU = 2 * KH, N1 = NU / 4;
      const bool fast = a.vec_out && col0 + C <= d;
      // the last slab's units: whole while eight columns are left, and in W, whose rows are padded, up to the
      // end (2^22 x 112, the whole sketch: 2317 us with two-byte stores there, 1602 so; 2126 in the cluster
      // form)
      const int nvec = !a.vec_out ? INT_MAX : (a.pad_out ? 1 : 8);
      auto read_unit = [&](int z, uint32_t *u) {
        tmem_ld_rows<2 * U>(tq + ((uint32_t)(16 * (z & 1)) << 16) + (uint32_t)((part * KH + (z >> 1)) * C), u);
      };
      auto store_unit = [&](int z, const uint32_t *u) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int kappa = (part * KH + (z >> 1)) * 128 + quad * 32 + (lane >> 2) + 16 * (z & 1) + 8 * x;
          const int64_t dst = a.pos ? (int64_t)s_pos[(it & 1) * (128 * J) + kappa] : out_row(a, kappa, g);
          if (dst < 0) continue;
          __nv_bfloat16 *orow = out + dst * a.ldout + col0 + (lane & 3) * 8;
#pragma unroll
          for (int h = 0; h < U; ++h) {
            const uint32_t *f = u + 8 * h + 2 * x;
            const int n = d - (col0 + (lane & 3) * 8 + 32 * h);  // columns left
            if (fast || n >= nvec) {
              *reinterpret_cast<uint4 *>(orow + 32 * h) = make_uint4(f[0], f[1], f[4], f[5]);
            } else {
              const uint32_t e4[4] = {f[0], f[1], f[4], f[5]};
#pragma unroll
              for (int e = 0; e < 8; ++e)
                if (e < n) {
                  __nv_bfloat16_raw b;
                  b.x = (unsigned short)(e4[e >> 1] >> (16 * (e & 1)));
                  orow[32 * h + e] = __nv_bfloat16(b);
                }
            }
          }
        }
      };
      {
        uint32_t u[N1][8 * U];
#pragma unroll
        for (int z = 0; z < N1; ++z) read_unit(z, u[z]);
        tmem_wait_ld();
#pragma unroll
        for (int z = 0; z < N1; ++z) store_unit(z, u[z]);
      }
      uint32_t u[NU - N1][8 * U];
#pragma unroll
      for (int z = N1; z < NU; ++z) read_unit(z, u[z - N1]);
      tmem_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty);
#pragma unroll
      for (int z = N1; z < NU; ++z) store_unit(z, u[z - N1]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kProdWarps + kEpiWarps) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

template <bool F32, int L> cudaError_t launch_tc(const GroupArgs &a0, int64_t ngroups, int nsm, cudaStream_t s) {
  constexpr int C = 512 >> (L - 7);
  TcPassArgs A{a0, 0, (float)a0.scale};
  A.a.nslab = (A.a.d + C - 1) / C;
  A.ntiles = ngroups * A.a.nslab;
  const size_t smem = 1024 + kHBytes + (size_t)ring_stages<F32>() * stage_bytes<F32>() + (F32 ? kRaw * kRawBytes : 0) + 8 * (2 * ring_stages<F32>() + 3) + 32 +
                      (F32 ? 0 : 8 * (size_t)(1 << L));
  auto kern = a0.wait_polls > 0 ? k_group_tc<F32, L, true> : k_group_tc<F32, L, false>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)(A.ntiles < nsm ? A.ntiles : nsm), kTcThreads, smem, s>>>(A);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_group_tc(const GroupArgs &a, bool f32, int L, int64_t ngroups, cudaStream_t s) {
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (L == 11) return f32 ? launch_tc<true, 11>(a, ngroups, nsm, s) : launch_tc<false, 11>(a, ngroups, nsm, s);
  if (L == 10) return f32 ? launch_tc<true, 10>(a, ngroups, nsm, s) : launch_tc<false, 10>(a, ngroups, nsm, s);
  return cudaErrorInvalidValue;
}

}  // namespace slse
