// FP64 Householder QR by panels of eight columns (paper, Appendix "implementation details").
//
// What bounds the column-by-column form (linalg.cu, k_qr): two grid-wide barriers and two rounds
// through L2 per column, 12 us for 2.5 us of FP64 work at 3072 x 512.  Here a panel is factored by one
// cluster of 16 CTAs that keeps its rows in registers (one or a few rows of eight columns per thread):
// a column costs one exchange through distributed shared memory, its dot products with all eight
// columns of the panel (those with the reflectors so far give the factor T) in one reduction.  The
// rest of the matrix is updated by the whole GPU once per panel, Q^T A = A - V T^T (V^T A): one CTA
// takes one or two columns over all rows, so its inner products stay within the CTA.  The matrix is
// held column-major, so every access is along rows.
// Measured (GB300), slse_qr with the inverse: 3072 x 512 6.93 -> 4.33 ms, 1536 x 256 2.67 -> 1.50 ms, 300 x 50
// 0.50 -> 0.33 ms, 12000 x 200 3.54 -> 2.90 ms.  What bounds it now: the FP64 pipe in the update of the
// columns behind (55 us for the first panels, beside 28 us of panel and 10 us for the next panel's
// columns), then the panel chain; 0.5 ms are R^{-1} and H^{-1}.  Without the update running beside the
// next panel 5.0 ms.
#include "host_res.cuh"

namespace slse {
namespace {

constexpr int kNb = 8;         // panel columns
constexpr int kCluster = 16;   // CTAs of a panel
constexpr int kThreads = 256;
constexpr int kMaxRpt = 4;     // rows per thread of a panel, at most (16384 rows)

struct PanelArgs {
  double *A;      // d x ldr: column c at A + c ldr
  int64_t ldr;
  int64_t j0;     // first row and column of the panel
  int64_t rows;   // rows from j0 on
  int nb;         // columns of the panel (kNb, fewer in the last one)
  double *V;      // kNb x ldr: reflectors, from row j0 on, zero above their diagonal
  double *T;      // kNb x kNb, upper triangular
  DevState *st;
};

__device__ __forceinline__ void st_cluster(double *p, int rank, double v) {
  unsigned remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Sums of N (a power of two, at most 16) values over the warp: afterwards v[0] of lane l is the total
// of value bitsel(l), whose bits are lane bits 16, 8, .. from the top (half the adds of N plain sums).
template <int N> __device__ __forceinline__ void warp_sums(double (&v)[N], int lane) {
  int off = 16;
#pragma unroll
  for (int n = N; n > 1; n >>= 1, off >>= 1) {
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int q = 0; q < n / 2; ++q) {
      const double send = upper ? v[q] : v[q + n / 2], keep = upper ? v[q + n / 2] : v[q];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
#pragma unroll
  for (; off > 0; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
}

template <int RPT> __global__ void __launch_bounds__(kThreads) k_qr_panel(const PanelArgs a) {
  __shared__ double s_w[kThreads / 32][kNb];        // per-warp sums
  __shared__ double s_x[2][kCluster][kNb];          // sums of every CTA of the cluster
  __shared__ double s_piv[2][kNb];                  // row j of the panel
  __shared__ double s_own[kNb];
  __shared__ double s_tw[kNb], s_vj, s_alpha;
  __shared__ double s_S[kNb][kNb], s_tau[kNb];      // v_l . v_j and tau_j
  const int rank = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t per = (a.rows + kCluster - 1) / kCluster;
  for (int e = threadIdx.x; e < kThreads / 32 * kNb; e += blockDim.x) (&s_w[0][0])[e] = 0.0;  // warps not launched
  double x[RPT][kNb], diag = 0.0;
  int64_t ri[RPT];  // row in the panel, or beyond its end
#pragma unroll
  for (int k = 0; k < RPT; ++k) {
    const int64_t l = threadIdx.x + (int64_t)blockDim.x * k;
    ri[k] = l < per ? rank * per + l : a.rows;
    if (ri[k] > a.rows) ri[k] = a.rows;
#pragma unroll
    for (int c = 0; c < kNb; ++c) x[k][c] = (ri[k] < a.rows && c < a.nb) ? a.A[(a.j0 + c) * a.ldr + a.j0 + ri[k]] : 0.0;
  }
  cluster_sync();  // every CTA has started
#pragma unroll
  for (int j = 0; j < kNb; ++j) {
    if (j >= a.nb) break;
    const int buf = j & 1;
    double p[kNb];
#pragma unroll
    for (int c = 0; c < kNb; ++c) p[c] = 0.0;
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      const double xj = (ri[k] >= j && ri[k] < a.rows) ? x[k][j] : 0.0;
#pragma unroll
      for (int c = 0; c < kNb; ++c) p[c] = fma(xj, x[k][c], p[c]);
    }
    if (ri[0] == j) {
#pragma unroll
      for (int c = 0; c < kNb; ++c) s_own[c] = x[0][c];
    }
    warp_sums<kNb>(p, lane);
    if ((lane & 3) == 0) s_w[warp][((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] = p[0];
    __syncthreads();
    const int val = lane & 7, q = lane >> 3;
    if (warp == 0) {
      double t = s_w[q][val] + s_w[q + 4][val];
      t += __shfl_xor_sync(0xffffffffu, t, 8);
      t += __shfl_xor_sync(0xffffffffu, t, 16);
#pragma unroll
      for (int m = 0; m < kCluster / 4; ++m) {
        st_cluster(&s_x[buf][rank][val], q * 4 + m, t);
        if (rank == j / per) st_cluster(&s_piv[buf][val], q * 4 + m, s_own[val]);
      }
    }
    cluster_sync();
    if (warp == 0) {
      double f = (s_x[buf][q * 4][val] + s_x[buf][q * 4 + 1][val]) + (s_x[buf][q * 4 + 2][val] + s_x[buf][q * 4 + 3][val]);
      f += __shfl_xor_sync(0xffffffffu, f, 8);
      f += __shfl_xor_sync(0xffffffffu, f, 16);
      const double piv = s_piv[buf][val];
      const double nrm2 = __shfl_sync(0xffffffffu, f, j), ajj = __shfl_sync(0xffffffffu, piv, j);
      double alpha = 0.0, tau = 0.0, dot = 0.0;
      if (nrm2 > 0.0) {
        const double nrm = sqrt(nrm2);
        alpha = ajj >= 0.0 ? -nrm : nrm;
        tau = 1.0 / (nrm * (nrm + fabs(ajj)));  // 2 / v^T v
        dot = f - alpha * piv;                  // v^T x_c, also for the reflectors c < j
      } else if (rank == 0 && lane == 0) {
        atomicOr(&a.st->status, ST_NUMERIC);
      }
      if (lane < kNb) {
        s_tw[lane] = tau * dot;
        s_S[j][lane] = dot;
      }
      if (lane == 0) {
        s_vj = ajj - alpha;
        s_alpha = alpha;
        s_tau[j] = tau;
      }
    }
    __syncthreads();
    const double vj = s_vj;
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      if (ri[k] < j || ri[k] >= a.rows) continue;
      if (ri[k] == j) {
        diag = s_alpha;
        x[k][j] = vj;
      }
#pragma unroll
      for (int c = 0; c < kNb; ++c)
        if (c > j) x[k][c] = fma(-x[k][j], s_tw[c], x[k][c]);
    }
  }
#pragma unroll
  for (int k = 0; k < RPT; ++k) {
    if (ri[k] >= a.rows) continue;
#pragma unroll
    for (int c = 0; c < kNb; ++c) {
      a.V[(int64_t)c * a.ldr + ri[k]] = (c < a.nb && ri[k] >= c) ? x[k][c] : 0.0;
      if (c < a.nb && ri[k] <= c) a.A[(a.j0 + c) * a.ldr + a.j0 + ri[k]] = ri[k] == c ? diag : x[k][c];
    }
  }
  // T of the block reflector I - V T V^T, row i by lane i of the last CTA
  if (rank == kCluster - 1 && threadIdx.x < kNb) {
    const int i = threadIdx.x;
    double t[kNb];
#pragma unroll
    for (int j = 0; j < kNb; ++j) {
      t[j] = 0.0;
      if (j < a.nb && j >= i) {
        if (j == i) t[j] = s_tau[j];
        else {
          double s = 0.0;
#pragma unroll
          for (int l = 0; l < kNb; ++l)
            if (l >= i && l < j) s = fma(t[l], s_S[j][l], s);
          t[j] = -s_tau[j] * s;
        }
      }
      a.T[i * kNb + j] = t[j];
    }
  }
}

struct TrailArgs {
  double *A;
  int64_t ldr, j0, rows;
  int c0, c1;      // columns to update: [c0, c1)
  const double *V, *T;
};

// Columns c0 + CB (blockIdx.x / RS) ..: A -= V (T^T (V^T A)) over the rows from j0 on, the rows split
// over the RS CTAs of a cluster.
template <int CB, int RS> __global__ void __launch_bounds__(kThreads) k_qr_trail(const TrailArgs a) {
  __shared__ double s_w[kThreads / 32][kNb * CB];
  __shared__ double s_x[RS][kNb * CB];
  __shared__ double s_W[kNb * CB], s_T[kNb * kNb];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = a.c0 + (int)(blockIdx.x / RS) * CB, rank = (int)(blockIdx.x % RS);
  const int64_t per = (a.rows + RS - 1) / RS, i0 = rank * per, i1 = i0 + per < a.rows ? i0 + per : a.rows;
  double *col[CB];
  bool live[CB];
#pragma unroll
  for (int b = 0; b < CB; ++b) {
    live[b] = c + b < a.c1;
    col[b] = a.A + (int64_t)(live[b] ? c + b : c) * a.ldr + a.j0;
  }
  if (RS > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  if (threadIdx.x < kNb * kNb) s_T[threadIdx.x] = a.T[threadIdx.x];
  double w[kNb * CB];
#pragma unroll
  for (int q = 0; q < kNb * CB; ++q) w[q] = 0.0;
#pragma unroll 2
  for (int64_t i = i0 + threadIdx.x; i < i1; i += kThreads) {
    double v[kNb], x[CB];
#pragma unroll
    for (int q = 0; q < kNb; ++q) v[q] = __ldg(a.V + (int64_t)q * a.ldr + i);
#pragma unroll
    for (int b = 0; b < CB; ++b) x[b] = col[b][i];
#pragma unroll
    for (int q = 0; q < kNb; ++q)
#pragma unroll
      for (int b = 0; b < CB; ++b) w[q * CB + b] = fma(v[q], x[b], w[q * CB + b]);
  }
  warp_sums<kNb * CB>(w, lane);
  // value index: lane bits from the top
  constexpr int L2 = CB == 1 ? 3 : 4;
  if ((lane & ((32 >> L2) - 1)) == 0) {
    int idx = 0;
#pragma unroll
    for (int k = 0; k < L2; ++k) idx = idx * 2 + ((lane >> (4 - k)) & 1);
    s_w[warp][idx] = w[0];
  }
  if (RS > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // the peers have started
  __syncthreads();
  if (threadIdx.x < kNb * CB) {
    double t[kThreads / 32];
#pragma unroll
    for (int k = 0; k < kThreads / 32; ++k) t[k] = s_w[k][threadIdx.x];
    const double sum = ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
    if constexpr (RS == 1) {
      s_W[threadIdx.x] = sum;
    } else {
#pragma unroll
      for (int k = 0; k < RS; ++k) st_cluster(&s_x[rank][threadIdx.x], k, sum);
    }
  }
  if constexpr (RS > 1) {
    cluster_sync();
    if (threadIdx.x < kNb * CB) {
      double t = s_x[0][threadIdx.x];
#pragma unroll
      for (int k = 1; k < RS; ++k) t += s_x[k][threadIdx.x];
      s_W[threadIdx.x] = t;
    }
  }
  __syncthreads();
  // T^T W (T upper triangular), by every thread for its registers
  double y[kNb * CB];
#pragma unroll
  for (int b = 0; b < CB; ++b) {
    const int q = lane & 7;  // each lane of eight forms one entry, then all take all
    double s = 0.0;
#pragma unroll
    for (int l = 0; l < kNb; ++l)
      if (l <= q) s = fma(s_T[l * kNb + q], s_W[l * CB + b], s);
#pragma unroll
    for (int k = 0; k < kNb; ++k) y[k * CB + b] = __shfl_sync(0xffffffffu, s, k);
  }
#pragma unroll 2
  for (int64_t i = i0 + threadIdx.x; i < i1; i += kThreads) {
    double v[kNb], x[CB];
#pragma unroll
    for (int q = 0; q < kNb; ++q) v[q] = __ldg(a.V + (int64_t)q * a.ldr + i);
#pragma unroll
    for (int b = 0; b < CB; ++b) x[b] = col[b][i];
#pragma unroll
    for (int q = 0; q < kNb; ++q)
#pragma unroll
      for (int b = 0; b < CB; ++b) x[b] = fma(-v[q], y[q * CB + b], x[b]);
#pragma unroll
    for (int b = 0; b < CB; ++b)
      if (live[b]) col[b][i] = x[b];
  }
}

// At (d x ldr) = A^T (A r x d, ld lda)
__global__ void __launch_bounds__(256) k_qr_transpose(const double *A, int64_t lda, int64_t r, int d, double *At, int64_t ldr) {
  __shared__ double t[32][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32;
  const int c0 = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int k = ty; k < 32; k += 8) t[k][tx] = (i0 + k < r && c0 + tx < d) ? A[(i0 + k) * lda + c0 + tx] : 0.0;
  __syncthreads();
  for (int k = ty; k < 32; k += 8)
    if (c0 + k < d && i0 + tx < r) At[(int64_t)(c0 + k) * ldr + i0 + tx] = t[tx][k];
}

// R (d x d, non-negative diagonal, zero below it) and R^T from the factored columns
__global__ void k_qr_extract(const double *At, int64_t ldr, int d, double *R, double *Rt) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= d * d) return;
  const int k = e / d, i = e % d;  // consecutive threads along a column of At
  const double diag = At[(int64_t)i * ldr + i];
  const double v = k >= i ? (diag < 0.0 ? -1.0 : 1.0) * At[(int64_t)k * ldr + i] : 0.0;
  R[(int64_t)i * d + k] = v;
  Rt[(int64_t)k * d + i] = v;
}

// A panel's CTAs take their SMs for themselves: the FP64 pipe, which the update of the columns behind
// would share with them, sets their pace (a panel beside it 40 us instead of 30).
constexpr int kPanelSmem = 190 * 1024, kTrailSmem = 40 * 1024;

template <class... P>
cudaError_t launch_cluster(void (*kern)(P...), unsigned grid, unsigned threads, unsigned cluster, int smem, cudaStream_t s,
                           P... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Two columns per CTA while that fills the GPU (each CTA reads all of V), one below, and the rows of a
// column over a cluster when few columns are left: as many CTAs as there are SMs at most, until one column
// each does not fit.
cudaError_t launch_trail(const TrailArgs &a, int nsm, cudaStream_t s, int &launched) {
  const int n = a.c1 - a.c0;
  if (n <= 0) return cudaSuccess;
  ++launched;
  if (n <= nsm / 4) return launch_cluster(k_qr_trail<1, 4>, 4u * n, kThreads, 4, kTrailSmem, s, a);
  if (n <= nsm / 2) return launch_cluster(k_qr_trail<1, 2>, 2u * n, kThreads, 2, kTrailSmem, s, a);
  if (n <= nsm) k_qr_trail<1, 1><<<n, kThreads, kTrailSmem, s>>>(a);
  else k_qr_trail<2, 1><<<(n + 1) / 2, kThreads, kTrailSmem, s>>>(a);
  return cudaGetLastError();
}

inline size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }
int64_t ld_rows(int64_t r) { return (r + 31) / 32 * 32; }

}  // namespace

bool qr_panels_ok(int64_t r) { return r <= (int64_t)kCluster * kThreads * kMaxRpt; }

size_t qr_panels_ws_bytes(int64_t r, int d) {
  return al256((size_t)ld_rows(r) * d * 8) + 2 * al256((size_t)ld_rows(r) * kNb * 8) + 2 * al256(kNb * kNb * 8);
}

cudaError_t launch_qr_panels(const double *A, int64_t r, int d, int64_t lda, double *R, double *Rt, void *ws, DevState *st,
                             int nsm, cudaStream_t s, int &launched) {
  const int64_t ldr = ld_rows(r);
  char *p = static_cast<char *>(ws);
  double *At = reinterpret_cast<double *>(p);
  const size_t o_v = al256((size_t)ldr * d * 8), vb = al256((size_t)ldr * kNb * 8);
  double *V[2], *T[2];
  for (int k = 0; k < 2; ++k) {
    V[k] = reinterpret_cast<double *>(p + o_v + k * vb);
    T[k] = reinterpret_cast<double *>(p + o_v + 2 * vb + k * al256(kNb * kNb * 8));
  }
  k_qr_transpose<<<dim3((unsigned)((r + 31) / 32), (unsigned)((d + 31) / 32)), 256, 0, s>>>(A, lda, r, d, At, ldr);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  for (const void *k : {(const void *)k_qr_panel<1>, (const void *)k_qr_panel<2>, (const void *)k_qr_panel<4>})
    if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kPanelSmem)) != cudaSuccess)
      return e;
  // The panel chain (panel, update of the next panel's columns) runs on a stream of the highest
  // priority; the update of the columns behind those runs beside the next panel on the caller's
  // stream.  Reflectors are double-buffered: block p is read until the update of block p + 1 starts.
  Events E;
  cudaEvent_t e_chain = nullptr, e_rest = nullptr;
  SideStream chain;
  // One stream while the caller's is being captured (a stream of the thread's would stay part of the
  // capture after the call), and when every side stream has other work.
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) {
    cudaGetLastError();
    capture = cudaStreamCaptureStatusActive;
  }
  if (d > 2 * kNb && capture == cudaStreamCaptureStatusNone && (e = chain.open(true, s, true)) != cudaSuccess) return e;
  const bool ahead = chain.h != nullptr;
  if (ahead) {
    e_chain = E.make();
    e_rest = E.make();
    if (!e_chain || !e_rest) return cudaErrorUnknown;
    if ((e = cudaEventRecord(e_rest, s))) return e;
  }
  const cudaStream_t sc = ahead ? chain.h : s;
  for (int j0 = 0, blk = 0; j0 < d; j0 += kNb, blk ^= 1) {
    const int nb = d - j0 < kNb ? d - j0 : kNb, c0 = j0 + nb, c1 = c0 + kNb < d ? c0 + kNb : d;
    if (ahead && j0 == 0 && (e = cudaStreamWaitEvent(sc, e_rest, 0))) return e;
    const PanelArgs pa{At, ldr, j0, r - j0, nb, V[blk], T[blk], st};
    const int64_t per = (r - j0 + kCluster - 1) / kCluster;
    const unsigned threads = per >= kThreads ? kThreads : (unsigned)((per + 31) / 32 * 32);
    e = launch_cluster(per <= kThreads ? k_qr_panel<1> : (per <= 2 * kThreads ? k_qr_panel<2> : k_qr_panel<4>), kCluster,
                       threads, kCluster, kPanelSmem, sc, pa);
    if (e != cudaSuccess) return e;
    ++launched;
    TrailArgs ta{At, ldr, j0, r - j0, c0, c1, V[blk], T[blk]};
    // the block before has reached the next panel's columns
    if (ahead && j0 > 0 && (e = cudaStreamWaitEvent(sc, e_rest, 0))) return e;
    if ((e = launch_trail(ta, nsm, sc, launched)) != cudaSuccess) return e;
    ta.c0 = c1;
    ta.c1 = d;
    // the columns behind wait for that too: the next panel, of the higher priority, is placed first
    if (ahead && ((e = cudaEventRecord(e_chain, sc)) || (e = cudaStreamWaitEvent(s, e_chain, 0)))) return e;
    if ((e = launch_trail(ta, nsm, s, launched)) != cudaSuccess) return e;
    if (ahead && (e = cudaEventRecord(e_rest, s))) return e;
  }
  if (ahead) {
    if ((e = cudaEventRecord(e_chain, sc)) || (e = cudaStreamWaitEvent(s, e_chain, 0))) return e;
  }
  k_qr_extract<<<(d * d + 255) / 256, 256, 0, s>>>(At, ldr, d, R, Rt);
  launched += 2;  // with the transpose
  return cudaGetLastError();
}

}  // namespace slse
