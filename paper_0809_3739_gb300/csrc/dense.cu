// Dense n x n side of one iteration (Eq. 4 and the subspace step of
// Sec. III): the reduction of the Gram sums, Cholesky + triangular inverse and
// the symmetric eigen-decomposition, all FP64 (the contractions over the grid
// are in tc_gemm.cu and fx_gemm.cu).
#include <cooperative_groups.h>
#include <math.h>

#include "fx_scalar.cuh"
#include "itp_kernels.cuh"

namespace cg = cooperative_groups;

namespace itp {

namespace {

constexpr int kMaxM = 256;   // states of the n x n work at most

// ---------------------------------------------------------------------------
// G = scale * the sum of the chunks' partial sums: E entries per CTA, 256 / E
// slots over the chunks, the slots' sums added in integers.  It is bound by
// FP64 additions, 78 cycles of a sub-partition each, so few states (few
// entries) are spread over many CTAs: 10 and 24 states with 304 chunks 20 us
// with 32 entries per CTA, 6 with four; 57 13 and 7; 89 and 128 (152 chunks) 7
// and 9 either way, with the fewer CTAs.
constexpr int kReduceFewM = 64;
template <int E>
__global__ void __launch_bounds__(256) gram_reduce_kernel(const double* __restrict__ partial,
                                                          int n_chunks, int m, double scale,
                                                          int sym, double* __restrict__ G) {
  constexpr int kSlots = 256 / E;
  __shared__ double ss[E][kSlots + 1];
  const int el = threadIdx.x % E, slot = threadIdx.x / E;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int e = blockIdx.x * E + el;
  double s = 0.0, t = 0.0;
  if (e < m * m) {
    const int i = e / m, j = e - i * m;
    const double* p = partial + e;
    const double* q = partial + j * m + i;
#pragma unroll 4
    for (int c = slot; c < n_chunks; c += kSlots) {
      s += p[(long long)c * m * m];
      if (sym) t += q[(long long)c * m * m];
    }
  }
  ss[el][slot] = sym ? s + t : s;
  __syncthreads();
  for (int k = warp; k < E; k += 8) {
    double v = 0.0;
    for (int c = lane; c < kSlots; c += 32) v += ss[k][c];
    v = warp_sum64(v);
    const int o = blockIdx.x * E + k;
    if (lane == 0 && o < m * m) G[o] = (sym ? 0.5 * scale : scale) * v;
  }
}

// ---------------------------------------------------------------------------
// The O(m^3) kernels run on one CTA, or on a cluster of kClus for larger m:
// an SM retires about 1.7 FP64 FMAs per clock, so the work is spread over SMs
// once it outweighs the cluster barriers.  CTA r of n owns the rows i with
// i % n == r (the work per row grows or shrinks with i), in its shared memory.
constexpr int kClus = 8;            // CTAs per cluster (portable size)
constexpr int kClusThreads = 256;   // Cholesky: a panel row per thread
constexpr int kClusMinM = 28;       // from this m on the cluster is faster (24: even, 32: 10 %)
constexpr int kPanel = 8;           // columns per Cholesky panel

// d > 0 and finite, on the bits (a comparison of doubles takes the FP64 unit)
__device__ __forceinline__ bool is_pivot(double d) {
  const long long b = __double_as_longlong(d);
  return b > 0 && b < 0x7ff0000000000000LL;
}

// Cholesky S = L L^T and M = L^{-1}, in the form S = U D U^T (U unit lower
// triangular, D = diag d): M = D^{-1/2} U^{-1}, so that no square root lies on
// the chain from pivot to pivot.  Right-looking in panels of kPanel columns:
// every CTA gathers the panel (thread t holds row k0 + t) and factors it
// alike, one block barrier and a reciprocal per column; it completes the
// panel's rows of R = U^{-1}; then it updates its own rows below,
//   A[i][j] -= sum_c U[i][c] A[j][c]  (j <= i),   R[i][j] -= sum_c U[i][c] R[c][j].
// One cluster barrier per panel (the column-by-column form took one cluster
// and two block barriers, a square root and a division per column: 2.5 us;
// 57 states 0.118 -> 0.055 ms, 128 states 0.35 -> 0.148).
__global__ void __launch_bounds__(kClusThreads)
    cholesky_inverse_kernel(const double* __restrict__ S, int m, double* __restrict__ Minv,
                            int* status) {
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ double csh[];
  __shared__ double s_col[kPanel][kPanel];   // A[k0 + c'][k0 + c] when column c is eliminated
  __shared__ double s_rs[kPanel];            // 1 / sqrt(d) of the panel
  __shared__ int s_bad;
  const int nr = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int rp = (m + nr - 1) / nr, pitch = m + 1;
  double* A_ = csh;                        // [rp][pitch] own rows of S (lower part)
  double* Rr_ = A_ + (size_t)rp * pitch;   // [rp][pitch] own rows of R
  double* U = Rr_ + (size_t)rp * pitch;    // [m][kPanel + 1] panel of U
  double* Ac = U + (size_t)m * (kPanel + 1);   // [m][kPanel + 1] panel of A
  double* Rp = Ac + (size_t)m * (kPanel + 1);  // [kPanel][pitch] panel rows of R
  constexpr int UP = kPanel + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NT = kClusThreads, NW = NT / 32;
  if (tid == 0) s_bad = 0;
  for (int i = rank + nr * warp; i < m; i += nr * NW) {
    double* a = A_ + (size_t)(i / nr) * pitch;
    double* r = Rr_ + (size_t)(i / nr) * pitch;
    for (int j = lane; j < m; j += 32) {
      a[j] = S[(long long)i * m + j];
      r[j] = i == j ? 1.0 : 0.0;
    }
  }
  for (int k0 = 0; k0 < m; k0 += kPanel) {
    const int w = min(kPanel, m - k0);
    if (nr > 1) cl.sync();
    else __syncthreads();
    const int i = k0 + tid;   // this thread's panel row
    double a[kPanel];
    if (i < m) {
      const double* src = A_ + (size_t)(i / nr) * pitch + k0;
      if (nr > 1) src = cl.map_shared_rank(src, i % nr);
#pragma unroll
      for (int c = 0; c < kPanel; ++c) a[c] = c < w ? src[c] : 0.0;
    }
    for (int q = warp; q < w; q += NW) {
      const double* src = Rr_ + (size_t)((k0 + q) / nr) * pitch;
      if (nr > 1) src = cl.map_shared_rank(src, (k0 + q) % nr);
      for (int j = lane; j < k0 + w; j += 32) Rp[q * pitch + j] = src[j];
    }
#pragma unroll
    for (int c = 0; c < kPanel; ++c) {
      if (c < w) {   // uniform
        if (tid >= c && tid < w) s_col[c][tid] = a[c];
        __syncthreads();
        if (i > k0 + c && i < m) {
          double d = s_col[c][c];
          if (!is_pivot(d)) d = 1.0;
          const double u = a[c] * recip(d);
          U[i * UP + c] = u;
          Ac[i * UP + c] = a[c];
#pragma unroll
          for (int q = c + 1; q < kPanel; ++q)
            if (q < w && k0 + q <= i) a[q] = fma(-u, s_col[c][q], a[q]);
        }
      }
    }
    __syncthreads();
    // the panel's own rows of R, a column per thread; 1/sqrt(d) meanwhile
    if (tid < w) {
      const double d = s_col[tid][tid];
      const bool ok = is_pivot(d);
      if (!ok) s_bad = 1;
      s_rs[tid] = ok ? rsqrt64(d) : 1.0;
    }
    for (int j = tid; j < k0 + w; j += NT) {
      double x[kPanel];
#pragma unroll
      for (int c = 0; c < kPanel; ++c) {
        if (c < w) {
          double v = Rp[c * pitch + j];
#pragma unroll
          for (int q = 0; q < c; ++q) v = fma(-U[(k0 + c) * UP + q], x[q], v);
          x[c] = v;
          Rp[c * pitch + j] = v;
        }
      }
    }
    __syncthreads();
    for (int q = warp; q < w; q += NW)
      if ((k0 + q) % nr == rank)
        for (int j = lane; j < m; j += 32)
          Minv[(long long)(k0 + q) * m + j] = j <= k0 + q ? Rp[q * pitch + j] * s_rs[q] : 0.0;
    // own rows below the panel: one warp per row, lanes over columns
    const int first = k0 + w;
    for (int r = first + (rank - first % nr + nr) % nr + nr * warp; r < m; r += nr * NW) {
      double u[kPanel];
#pragma unroll
      for (int c = 0; c < kPanel; ++c) u[c] = c < w ? U[r * UP + c] : 0.0;
      double* ar = A_ + (size_t)(r / nr) * pitch;
      double* rr = Rr_ + (size_t)(r / nr) * pitch;
      for (int j = lane; j <= r; j += 32) {
        double* dst = j < first ? rr + j : ar + j;
        const double* src = j < first ? Rp + j : Ac + (size_t)j * UP;
        const int step = j < first ? pitch : 1;
        double v0 = *dst, v1 = 0.0;
#pragma unroll
        for (int c = 0; c < kPanel; c += 2) {
          if (c < w) v0 = fma(-u[c], src[c * step], v0);
          if (c + 1 < w) v1 = fma(-u[c + 1], src[(c + 1) * step], v1);
        }
        *dst = v0 + v1;
      }
    }
  }
  if (tid == 0 && s_bad) atomicOr(status, 1);
  if (nr > 1) cl.sync();   // no CTA leaves while another may still read its shared memory
}

// Householder tridiagonalisation (eigenvalues only).  An FP64 operation costs
// 78 cycles of its sub-partition and as much latency, so up to 128 states the
// CTA has one warp per sub-partition (two above), and the steps are arranged
// for a short chain of dependent operations.  Every CTA holds column k, x = A[k+1.., k], of the current
// matrix; groups of eight lanes of all warps but the last own rows of A.  Step k:
//   the groups form y = A x for their rows and publish y and their entries C
//   of column k + 1 to all CTAs, while the last warp forms the reflector
//   v = x - alpha e_1, beta = 2 / v^T v from x; (cluster) barrier;
//   A v = y - alpha C, so p = beta (y - alpha C), K = beta/2 v^T p and w = p -
//   K v follow from one dot product, and so does the next column, C - v w_1 -
//   w v_1, in every CTA alike; block barrier;
//   the groups apply A -= v w^T + w v^T to their rows and in the same pass form
//   the next y.
// Every warp forms p and its sum itself and a thread keeps its own entry: the
// count of FP64 instructions per warp (78 cycles each) and the length of the
// chain decide alike.  (The form with two cluster barriers, five block barriers
// and 256 threads took 5.4 us per step; now 24 states take 47 us, 57 122, 89
// 222 and 128 459; with FP64 scalars and warp sums and the dot product x^T y
// 24 states took 55 and 57 states 144 us.  From 128 states on the product y
// takes most of a step.)
template <int kTriThreads>
__global__ void __launch_bounds__(kTriThreads)
    tridiag_kernel(const double* __restrict__ H, int m, double* __restrict__ d,
                   double* __restrict__ e) {
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ double csh[];
  __shared__ double s_alpha[2], s_beta[2], s_hbeta[2], s_v0[2];
  const int nr = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int rp = (m + nr - 1) / nr, pitch = m + 1;
  double* A_ = csh;                       // [rp][pitch] own rows
  double* Y = A_ + (size_t)rp * pitch;    // [2][m] published y (step parity)
  double* C = Y + 2 * m;                  // [2][m] published column k + 1
  double* xf = C + 2 * m;                 // [2][m] x
  double* vf = xf + 2 * m;                // [m]
  double* wf = vf + m;                    // [m]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = kTriThreads / 32, kLanes = 8, kGroups = (NW - 1) * 32 / kLanes;
  for (int i = rank + nr * warp; i < m; i += nr * NW)
    for (int j = lane; j < m; j += 32)
      A_[(size_t)(i / nr) * pitch + j] = 0.5 * (H[(long long)i * m + j] + H[(long long)j * m + i]);
  for (int j = tid; j < m; j += kTriThreads) {
    xf[j] = 0.5 * (H[j] + H[(long long)j * m]);
    vf[j] = wf[j] = 0.0;
  }
  __syncthreads();
  if (nr > 1) cl.sync();   // every CTA has started before it is written to
  auto warp_sum = [](double v, int width) {
    for (int o = width / 2; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  const int group = tid / kLanes, gl = tid % kLanes;
  for (int k = 0; k + 2 < m; ++k) {
    const int n0 = k + 1, b = k & 1;
    const double* x = xf + b * m;
    double* Yb = Y + b * m;
    double* Cb = C + b * m;
    if (warp == NW - 1) {   // the reflector
      const double x0 = x[n0];
      double s = 0.0;
      for (int j = n0 + 1 + lane; j < m; j += 32) s = fma(x[j], x[j], s);
      const bool any = __any_sync(0xffffffffu, fx_bits(s) != 0);   // (no FP64 comparison)
      if (lane == 31) s = fma(x0, x0, s);
      long long t;
      int ex;
      const bool fast = fx_warp_sum(s, &t, &ex) && ex > 100;
      if (!fast) s = warp_sum(s, 32);
      if (lane == 0) {
        double alpha = x0, beta = 0.0, v0 = 0.0;
        if (any && fast) {
          fx_reflector(fx_normal((unsigned long long)t, ex - 1079), x0, &alpha, &beta, &v0);
        } else if (any) {
          const double nrm = sqrt(s);
          beta = 1.0 / fma(fabs(x0), nrm, s);
          alpha = x0 > 0 ? -nrm : nrm;
          v0 = x0 - alpha;
        }
        s_alpha[b] = alpha;
        s_beta[b] = beta;
        s_hbeta[b] = 0.5 * beta;
        s_v0[b] = v0;
        if (rank == 0) e[k] = alpha;
      }
    } else {
      // own rows i >= n0: the previous step's update (v, w from column k - 1;
      // zero before the first step), then y = A x
      const int il0 = (n0 - rank + nr - 1) / nr;   // first local row with i >= n0
      for (int il = il0 - il0 % kGroups + group; il - group < rp; il += kGroups) {
        const int i = rank + nr * il;
        const bool mine = il >= il0 && i < m;
        double s = 0.0, t = 0.0, c = 0.0;
        if (mine) {
          double* row = A_ + (size_t)il * pitch;
          const double vi = vf[i], wi = wf[i];
          for (int j = n0 + gl; j < m; j += 2 * kLanes) {
            const int j2 = j + kLanes;
            const double a = fma(-vi, wf[j], fma(-wi, vf[j], row[j]));
            row[j] = a;
            s = fma(a, x[j], s);
            if (j == n0) c = a;
            if (j2 < m) {
              const double a2 = fma(-vi, wf[j2], fma(-wi, vf[j2], row[j2]));
              row[j2] = a2;
              t = fma(a2, x[j2], t);
            }
          }
        }
        s = warp_sum(s + t, kLanes);
        c = __shfl_sync(0xffffffffu, c, lane & ~(kLanes - 1));
        if (mine && gl < nr) {
          double* y = Yb + i;
          double* cc = Cb + i;
          if (nr > 1) {
            y = cl.map_shared_rank(y, gl);
            cc = cl.map_shared_rank(cc, gl);
          }
          *y = s;
          *cc = c;
        }
      }
    }
    if (nr > 1) cl.sync();
    else __syncthreads();
    // scalars, in every warp alike
    const double alpha = s_alpha[b], beta = s_beta[b], v0 = s_v0[b];
    // p = beta (y - alpha C) and v^T p in every warp; lane l has the entries n0 + l
    // + 32 q and keeps that of q = warp, entry j = n0 + tid (m <= kTriThreads)
    double vp = 0.0, p1 = 0.0, vj = 0.0, pj = 0.0, cj = 0.0;
#pragma unroll
    for (int q = 0; q < NW; ++q) {
      if (n0 + 32 * q >= m) break;
      const int i = n0 + 32 * q + lane;
      double v = 0.0, p = 0.0, c = 0.0;
      if (i < m) {
        c = Cb[i];
        v = i == n0 ? v0 : x[i];
        p = beta * fma(-alpha, c, Yb[i]);
        vp = fma(v, p, vp);
      }
      if (q == 0) p1 = __shfl_sync(0xffffffffu, p, 0);
      if (q == warp) {
        vj = v;
        pj = p;
        cj = c;
      }
    }
    // the next column is C - v w_1 - w v_1 with w = p - K v, K = beta/2 v^T p: two
    // operations after the sum
    const int j = n0 + tid;
    const double cp = fma(-pj, v0, fma(-vj, p1, cj)), vv = vj * v0;
    const double sum = warp_sum64(vp), K2 = beta * sum, K = s_hbeta[b] * sum;
    if (tid == 0 && (n0 - 1) == 0 && rank == 0) d[0] = A_[0];
    if (j < m) {
      const double cn = fma(K2, vv, cp);
      vf[j] = vj;
      wf[j] = fma(-K, vj, pj);
      xf[(b ^ 1) * m + j] = cn;
      if (j == n0 && rank == 0) d[n0] = cn;
    }
    __syncthreads();
  }
  // the last 2 x 2 block: d[m - 2] is set above (m > 2), the update of the last
  // diagonal entry is still due
  const int last = m - 1;
  if (m == 1) {
    if (tid == 0 && rank == 0) d[0] = A_[0];
  } else if (last % nr == rank && tid == 0) {
    const double* row = A_ + (size_t)(last / nr) * pitch;
    if (m == 2) {
      e[0] = row[0];
      d[1] = row[1];
    } else {
      const double vl = vf[last], wl = wf[last];
      d[last] = fma(-vl, wl, fma(-wl, vl, row[last]));
      e[last - 1] = xf[((m - 2) & 1) * m + last];
    }
  }
  if (m == 2 && rank == 0 && tid == 0) d[0] = A_[0];
  if (nr > 1) cl.sync();   // no CTA leaves while another may still write to it
}

// Shared memory of the two kernels on a cluster of nr CTAs.
size_t cholesky_smem(int m, int nr) {
  return ((size_t)2 * ((m + nr - 1) / nr) * (m + 1) + (size_t)2 * m * (kPanel + 1) +
          (size_t)kPanel * (m + 1)) * sizeof(double);
}
size_t tridiag_smem(int m, int nr) {
  return ((size_t)((m + nr - 1) / nr) * (m + 1) + (size_t)8 * m) * sizeof(double);
}

// Launch on one cluster (of one CTA for small m).
template <typename K, typename... Args>
cudaError_t launch_cluster(K kernel, int nr, int threads, size_t smem, cudaStream_t st,
                           Args... args) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(nr);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = nr;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// ---------------------------------------------------------------------------
// Parallel cyclic Jacobi (round-robin pairing: m/2 disjoint rotations per
// round, m-1 rounds per sweep).  A in shared memory (pitch m+1), U^T in
// global memory (row p of U^T is eigenvector p).
__global__ void __launch_bounds__(1024) jacobi_kernel(const double* __restrict__ H, int m,
                                                      double* __restrict__ E,
                                                      double* __restrict__ Rt,
                                                      double* __restrict__ Ut,
                                                      double* __restrict__ Aglob, int* status) {
  extern __shared__ double sh[];
  const int mm = (m + 1) & ~1;          // even number of players (a dummy if m is odd)
  const int P = m + 1;
  // m x P working matrix: in shared memory, or (Aglob set: too large for
  // one CTA) in global memory, where it stays in L2
  double* A = Aglob ? Aglob : sh;
  double* cs = Aglob ? sh : sh + m * P;  // [mm/2] c, [mm/2] s
  int* pr = reinterpret_cast<int*>(cs + mm);   // [mm/2] p, [mm/2] q
  __shared__ double off_norm, tot_norm;
  __shared__ int done;
  const int tid = threadIdx.x, nthr = blockDim.x;
  for (int e = tid; e < m * m; e += nthr) {
    const int i = e / m, j = e - i * m;
    A[i * P + j] = 0.5 * (H[i * m + j] + H[j * m + i]);
    Ut[e] = (i == j) ? 1.0 : 0.0;
  }
  __syncthreads();
  const int npairs = mm / 2;
  int sweep;
  for (sweep = 0; sweep < 40; ++sweep) {
    if (tid == 0) { off_norm = 0.0; tot_norm = 0.0; }
    __syncthreads();
    double lo = 0.0, lt = 0.0;
    for (int e = tid; e < m * m; e += nthr) {
      const int i = e / m, j = e - i * m;
      const double v = A[i * P + j] * A[i * P + j];
      lt += v;
      if (i != j) lo += v;
    }
    atomicAdd(&off_norm, lo);
    atomicAdd(&tot_norm, lt);
    __syncthreads();
    // off-diagonal Frobenius norm <= 1e-13 of the total: eigenvalue errors
    // are then second order in it (~1e-26 |H|^2 / gap)
    if (tid == 0) done = (off_norm <= 1e-26 * tot_norm) || (off_norm == 0.0);
    __syncthreads();
    if (done) break;
    for (int round = 0; round < mm - 1; ++round) {
      for (int t = tid; t < npairs; t += nthr) {
        // players 0..mm-1; player 0 fixed, the others rotate
        const int a = (t == 0) ? 0 : 1 + (t - 1 + round) % (mm - 1);
        const int b = 1 + (mm - 2 - t + round) % (mm - 1);
        int p = min(a, b), q = max(a, b);
        double c = 1.0, s = 0.0;
        if (q < m) {
          const double apq = A[p * P + q];
          if (apq != 0.0) {
            const double app = A[p * P + p], aqq = A[q * P + q];
            const double zeta = (aqq - app) / (2.0 * apq);
            const double tt = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
            c = 1.0 / sqrt(1.0 + tt * tt);
            s = tt * c;
          }
        } else {
          p = q = -1;
        }
        cs[t] = c;
        cs[npairs + t] = s;
        pr[t] = p;
        pr[npairs + t] = q;
      }
      __syncthreads();
      // columns: A <- A J
      for (int e = tid; e < npairs * m; e += nthr) {
        const int t = e / m, r = e - t * m;
        const int p = pr[t], q = pr[npairs + t];
        if (p < 0) continue;
        const double c = cs[t], s = cs[npairs + t];
        const double arp = A[r * P + p], arq = A[r * P + q];
        A[r * P + p] = c * arp - s * arq;
        A[r * P + q] = s * arp + c * arq;
      }
      __syncthreads();
      // rows: A <- J^T A ; and U^T <- J^T U^T (rows p, q)
      for (int e = tid; e < npairs * m; e += nthr) {
        const int t = e / m, r = e - t * m;
        const int p = pr[t], q = pr[npairs + t];
        if (p < 0) continue;
        const double c = cs[t], s = cs[npairs + t];
        const double apr = A[p * P + r], aqr = A[q * P + r];
        A[p * P + r] = c * apr - s * aqr;
        A[q * P + r] = s * apr + c * aqr;
        const double up = Ut[p * m + r], uq = Ut[q * m + r];
        Ut[p * m + r] = c * up - s * uq;
        Ut[q * m + r] = s * up + c * uq;
      }
      __syncthreads();
    }
  }
  if (tid == 0 && sweep >= 40) atomicOr(status, 2);
  __syncthreads();
  // sort eigenvalues ascending (stable by index) and permute the rows of U^T
  for (int i = tid; i < m; i += nthr) {
    const double ei = A[i * P + i];
    int rank = 0;
    for (int j = 0; j < m; ++j) {
      const double ej = A[j * P + j];
      rank += (ej < ei) || (ej == ei && j < i);
    }
    E[rank] = ei;
    for (int r = 0; r < m; ++r) Rt[rank * m + r] = Ut[i * m + r];
  }
}

// ---------------------------------------------------------------------------
// Eigenvalues only: the tridiagonalisation above, then bisection on
// Sturm counts, one CTA of four warps per eigenvalue (128-point
// multisection: seven bits per round, one warp on each of the SM's four
// sub-partitions, whose FP64 units the counts keep busy).
constexpr int kBisWarps = 4;
constexpr int kBisPts = 32 * kBisWarps;   // points per round; the last is hi

// Biased binary exponent of a double (0 for zero and subnormals).
__device__ __forceinline__ int dexp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
// v * 2^k by its exponent field (v normal, the result normal).
__device__ __forceinline__ double dscale(double v, int k) {
  return __hiloint2double(__double2hiint(v) + (k << 20), __double2loint(v));
}

// Number of eigenvalues below x of the symmetric tridiagonal with diagonal
// d and squared off-diagonal e2 (e2[i] couples rows i and i+1), scaled so
// that |d_i|, |x| < 1 and e2_i <= 4.  The sign changes of the leading
// principal minors of T - x I,
//   p_0 = 1,  p_1 = d_0 - x,  p_{i+1} = (d_i - x) p_i - e2_{i-1} p_{i-1},
// i.e. the negative pivots p_{i+1}/p_i of its LDL^T factorisation.  No
// division: three FP64 operations per row, the rest on the integer pipe.
//  - A minor that vanishes against the previous one (|p_{i+1}| < 2^-599
//    |p_i|, zero included) becomes -2^-600 p_i: the pivot -2^-600, as a
//    zero pivot of the LDL^T recurrence is replaced by a tiny negative one.
//  - p_i and p_{i-1} are rescaled together by a power of two (exponent
//    arithmetic, exact) whenever |p_i| leaves [2^-256, 2^257).
// With the pivot rule |p_{i-1}| <= 2^600 |p_i|, so |p_{i+1}| < 2^603 |p_i|
// and every value stays a normal double between 2^-860 and 2^860.
__device__ __forceinline__ int sturm_count(const double* __restrict__ d,
                                           const double* __restrict__ e2, int m, double x) {
  double pm = 1.0, p = d[0] - x;
  int ep = dexp(p);
  if (ep < 1023 - 599) {
    p = -0x1p-600;
    ep = 1023 - 600;
  }
  int cnt = __double2hiint(p) < 0;
  if (ep < 1023 - 256) {
    p = dscale(p, 1023 - ep);
    pm = dscale(pm, 1023 - ep);
    ep = 1023;
  }
  for (int i = 1; i < m; ++i) {
    double pn = fma(d[i] - x, p, -(e2[i - 1] * pm));
    int en = dexp(pn);
    if (en < ep - 599) {
      pn = __hiloint2double((__double2hiint(p) ^ (int)0x80000000) - (600 << 20),
                            __double2loint(p));
      en = ep - 600;
    }
    cnt += (__double2hiint(pn) ^ __double2hiint(p)) < 0;
    pm = p;
    p = pn;
    ep = en;
    if ((unsigned)(en - (1023 - 256)) > 512u) {
      p = dscale(p, 1023 - en);
      pm = dscale(pm, 1023 - en);
      ep = 1023;
    }
  }
  return cnt;
}

// One CTA per eigenvalue index j (ascending): the Gershgorin interval of
// the tridiagonal, scaled by a power of two into (-1, 1), narrowed by
// 128-point multisection down to a few ulps.
__global__ void __launch_bounds__(kBisPts) bisect_kernel(const double* __restrict__ dg,
                                                          const double* __restrict__ eg, int m,
                                                          double* __restrict__ E) {
  __shared__ double sd[kMaxM], se2[kMaxM];
  __shared__ double s_lo, s_hi, s_scale;
  __shared__ unsigned s_ball[2][kBisWarps];
  __shared__ double s_x[2][kBisPts];   // the points of a round
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp == 0) {
    double lo = dg[0], hi = dg[0];
    for (int i = lane; i < m; i += 32) {
      const double r = (i > 0 ? fabs(eg[i - 1]) : 0.0) + (i + 1 < m ? fabs(eg[i]) : 0.0);
      lo = fmin(lo, dg[i] - r);
      hi = fmax(hi, dg[i] + r);
    }
    for (int o = 16; o; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) {
      const double span = fmax(hi - lo, 1e-300);
      lo -= 1e-14 * span + 1e-300;
      hi += 1e-14 * span + 1e-300;
      int k;
      frexp(fmax(fabs(lo), fabs(hi)), &k);   // max |.| = f 2^k, f in [1/2, 1)
      const double g = ldexp(1.0, -k);
      s_scale = g;
      s_lo = lo * g;
      s_hi = hi * g;
    }
  }
  __syncthreads();
  const double g = s_scale;
  for (int i = tid; i < m; i += blockDim.x) {
    sd[i] = dg[i] * g;
    const double ei = i + 1 < m ? eg[i] * g : 0.0;
    se2[i] = ei * ei;
  }
  __syncthreads();
  const int j = blockIdx.x;
  double lo = s_lo, hi = s_hi;
  const double part = (double)(tid + 1) / (double)kBisPts;
  for (int it = 0; it < 16; ++it) {
    // (positive doubles order as their bits; a comparison takes the FP64 unit)
    const double width = hi - lo;
    const long long al = fx_bits(lo) & 0x7fffffffffffffffLL, ah = fx_bits(hi) & 0x7fffffffffffffffLL;
    const double tol = fma(4.0 * 2.220446049250313e-16, fx_from_bits(al > ah ? al : ah), 0x1p-70);
    if (fx_bits(width) <= fx_bits(tol)) break;
    // points lo + width (t+1)/128, t < 127; point 127 is hi (count m + 1)
    const double x = fma(width, part, lo);
    s_x[it & 1][tid] = x;
    const int c = tid < kBisPts - 1 ? sturm_count(sd, se2, m, x) : m + 1;
    const unsigned ball = __ballot_sync(0xffffffffu, c > j);
    if (lane == 0) s_ball[it & 1][warp] = ball;
    __syncthreads();
    // the eigenvalue j lies in the first part whose right end has count > j
    int first = kBisPts - 1;
    for (int w = kBisWarps - 1; w >= 0; --w) {
      const unsigned b = s_ball[it & 1][w];
      if (b) first = 32 * w + __ffs(b) - 1;
    }
    if (first > 0) lo = s_x[it & 1][first - 1];
    if (first < kBisPts - 1) hi = s_x[it & 1][first];
  }
  if (tid == 0) E[j] = 0.5 * (lo + hi) / g;
}

__global__ void diag_kernel(const double* __restrict__ H, int m, double* __restrict__ E) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) E[i] = H[i * m + i];
}

// ---------------------------------------------------------------------------
// Residual norms of the adaptive iteration (Sec. III):
//   out_j = dV * sum_p (A[j][p] - c_j B[j][p])^2,
// c_j = exp(scale E_j) (mode 1: R^E with A = T psi, B = psi, scale = -tau) or
// c_j = E_j (mode 0: R^H with A = H psi, B = psi).  Chunks of points per
// CTA, the per-thread sums in the precision of the data, the rest in FP64,
// partial sums combined in a fixed order.
template <typename T> struct Vec4Of;
template <> struct Vec4Of<float> { using type = float4; static constexpr int W = 4; };
template <> struct Vec4Of<double> { using type = double2; static constexpr int W = 2; };

__device__ __forceinline__ float sqdiff_sum(const float4 a, const float4 b, float c) {
  const float d0 = a.x - c * b.x, d1 = a.y - c * b.y, d2 = a.z - c * b.z, d3 = a.w - c * b.w;
  return d0 * d0 + d1 * d1 + d2 * d2 + d3 * d3;
}
__device__ __forceinline__ double sqdiff_sum(const double2 a, const double2 b, double c) {
  const double d0 = a.x - c * b.x, d1 = a.y - c * b.y;
  return d0 * d0 + d1 * d1;
}

template <typename T>
__global__ void __launch_bounds__(256) residual_partial_kernel(
    const T* __restrict__ A, const T* __restrict__ B, const double* __restrict__ E,
    double scale, int mode, long long N, int chunks, double* __restrict__ partial) {
  using V = typename Vec4Of<T>::type;
  constexpr int W = Vec4Of<T>::W;
  const int j = blockIdx.y, c = blockIdx.x;
  const T cj = (T)(mode ? exp(scale * E[j]) : E[j]);
  const long long nv = N / W;
  const long long per = (nv + chunks - 1) / chunks;
  const long long v0 = (long long)c * per, v1 = min(nv, v0 + per);
  const V* a = reinterpret_cast<const V*>(A + (long long)j * N);
  const V* b = reinterpret_cast<const V*>(B + (long long)j * N);
  T acc = 0;
  for (long long v = v0 + threadIdx.x; v < v1; v += blockDim.x) acc += sqdiff_sum(a[v], b[v], cj);
  double s = (double)acc;
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ double ws[8];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += ws[w];
    partial[(long long)j * chunks + c] = t;
  }
}

__global__ void residual_final_kernel(const double* __restrict__ partial, int chunks, int m,
                                      double dV, double* __restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= m) return;
  double t = 0.0;
  for (int c = 0; c < chunks; ++c) t += partial[(long long)j * chunks + c];
  out[j] = t * dV;
}

template <typename TS, typename TD>
__global__ void convert_kernel(const TS* __restrict__ src, TD* __restrict__ dst, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = (TD)src[i];
}

}  // namespace

cudaError_t launch_gram_reduce(const double* partial, int n_chunks, int m, double scale, int sym,
                               double* G, cudaStream_t st) {
  if (m <= kReduceFewM)
    gram_reduce_kernel<4><<<(m * m + 3) / 4, 256, 0, st>>>(partial, n_chunks, m, scale, sym, G);
  else
    gram_reduce_kernel<32><<<(m * m + 31) / 32, 256, 0, st>>>(partial, n_chunks, m, scale, sym, G);
  return cudaGetLastError();
}

cudaError_t launch_cholesky_inverse(const double* S, int m, double* Minv, int* status,
                                    cudaStream_t st) {
  if (m < 1 || m > kMaxM) return cudaErrorInvalidValue;
  const int nr = m < kClusMinM ? 1 : kClus;
  return launch_cluster(cholesky_inverse_kernel, nr, kClusThreads, cholesky_smem(m, nr), st, S, m,
                        Minv, status);
}

cudaError_t launch_jacobi_eigh(const double* H, int m, double* E, double* Rt, double* work,
                               int* status, cudaStream_t st) {
  if (m < 1 || m > kMaxM) return cudaErrorInvalidValue;
  const int mm = (m + 1) & ~1;
  const size_t amat = (size_t)m * (m + 1) * sizeof(double);
  const size_t rest = (size_t)mm * sizeof(double) + (size_t)mm * sizeof(int);
  // the working matrix goes to global memory (after U^T in work) when it
  // does not fit one CTA's shared memory
  const bool global_a = amat + rest > 227 * 1024;
  const size_t smem = global_a ? rest : amat + rest;
  cudaError_t e = cudaFuncSetAttribute(jacobi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  jacobi_kernel<<<1, 1024, smem, st>>>(H, m, E, Rt, work,
                                       global_a ? work + (size_t)m * m : nullptr, status);
  return cudaGetLastError();
}

cudaError_t launch_tridiag(const double* H, int m, double* work, cudaStream_t st) {
  if (m < 1 || m > kMaxM) return cudaErrorInvalidValue;
  const int nr = m < kClusMinM ? 1 : kClus;
  if (m <= 128)
    return launch_cluster(tridiag_kernel<128>, nr, 128, tridiag_smem(m, nr), st, H, m, work,
                          work + m);
  return launch_cluster(tridiag_kernel<256>, nr, 256, tridiag_smem(m, nr), st, H, m, work,
                        work + m);
}

cudaError_t launch_bisect(const double* work, int m, double* E, cudaStream_t st) {
  if (m > kMaxM) return cudaErrorInvalidValue;
  bisect_kernel<<<m, kBisPts, 0, st>>>(work, work + m, m, E);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_residual_norms(const T* A, const T* B, const double* E, double scale,
                                  int mode, int m, long long N, double dV, int chunks,
                                  double* partial, double* out, cudaStream_t st) {
  if (m < 1 || chunks < 1 || (N % Vec4Of<T>::W)) return cudaErrorInvalidValue;
  residual_partial_kernel<T><<<dim3(chunks, m), 256, 0, st>>>(A, B, E, scale, mode, N, chunks,
                                                              partial);
  residual_final_kernel<<<(m + 127) / 128, 128, 0, st>>>(partial, chunks, m, dV, out);
  return cudaGetLastError();
}
template cudaError_t launch_residual_norms<float>(const float*, const float*, const double*,
                                                  double, int, int, long long, double, int,
                                                  double*, double*, cudaStream_t);
template cudaError_t launch_residual_norms<double>(const double*, const double*, const double*,
                                                   double, int, int, long long, double, int,
                                                   double*, double*, cudaStream_t);

template <typename R>
__global__ void axpby_kernel(R a, const R* __restrict__ X, R b, const R* Y, R* out,
                             long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = fma(b, Y[i], a * X[i]);
}

template <typename R>
cudaError_t launch_axpby(double a, const R* X, double b, const R* Y, R* out, long long n,
                         cudaStream_t st) {
  axpby_kernel<R><<<4 * 152, 256, 0, st>>>((R)a, X, (R)b, Y, out, n);
  return cudaGetLastError();
}
template cudaError_t launch_axpby<float>(double, const float*, double, const float*, float*,
                                         long long, cudaStream_t);
template cudaError_t launch_axpby<double>(double, const double*, double, const double*,
                                          double*, long long, cudaStream_t);

cudaError_t launch_diag(const double* H, int m, double* E, cudaStream_t st) {
  diag_kernel<<<(m + 127) / 128, 128, 0, st>>>(H, m, E);
  return cudaGetLastError();
}

template <typename TS, typename TD>
cudaError_t launch_convert(const TS* src, TD* dst, long long count, cudaStream_t st) {
  convert_kernel<TS, TD><<<4 * 152, 256, 0, st>>>(src, dst, count);
  return cudaGetLastError();
}

template cudaError_t launch_convert<float, double>(const float*, double*, long long, cudaStream_t);
template cudaError_t launch_convert<double, float>(const double*, float*, long long, cudaStream_t);
template cudaError_t launch_convert<double, double>(const double*, double*, long long, cudaStream_t);

}  // namespace itp
