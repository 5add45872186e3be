// FP32 contractions over the grid for few states, on the FP32 cores: the
// overlap / subspace matrix and the update of the mixed path where the state
// count is far below the 128 rows of a tensor-core tile.  The tensor-core
// kernels (tc_gemm.cu) convert and multiply 128 rows whatever m is; with
// 16 states on 256^3 they took 3.8 ms per Gram matrix and 7.4 ms per update
// for 1.1 and 2.1 GB of data.  At such counts the FP32 arithmetic is below the
// memory time, so these kernels stream.
//
// Precision: products and sums in FP32 over runs of 128 points, the runs
// added with the error-free TwoSum (a pair of FP32 values per entry), chunks
// in FP64; the update is a plain FP32 sum over the states.  The tensor-core
// forms split into TF32 parts and add 32-point tiles in FP32.
#include <cuda_runtime.h>
#include <stdint.h>

#include "itp_kernels.cuh"

namespace itp {

namespace {

// 16-byte asynchronous copy to shared memory, zeros where !valid.
__device__ __forceinline__ void copy16(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void copies_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void two_sum(float& s, float& e, float x) {
  const float t = s + x;
  const float bb = t - s;
  e += (s - (t - bb)) + (x - bb);
  s = t;
}

// ---------------------------------------------------------------------------
// Gram partial sums P[c][i][j] = sum_{p in chunk c} A[i][p] B[j][p], all of the
// m x m result in one CTA: 16 x 16 threads, TT x TT entries each (rows ty + 16
// q, columns tx + 16 r).  Tiles of 64 points come by asynchronous copies into
// a ring of buffers (deeper where a tile has few rows, to keep enough bytes in
// flight), [row][point] with a pitch of 68 (consecutive rows 4 banks apart,
// so that the 16-byte reads of eight rows meet no conflict).
constexpr int kGramPts = 64;
constexpr int kGramPitch = kGramPts + 4;
template <int TT> constexpr int kGramBufs = TT == 1 ? 8 : TT == 2 ? 6 : TT == 3 ? 4 : 3;

template <int TT>
constexpr size_t gram_smem(bool same) {
  return (size_t)kGramBufs<TT> * (same ? 1 : 2) * 16 * TT * kGramPitch * sizeof(float);
}

template <int TT>
__global__ void __launch_bounds__(256) f32_gram_kernel(const float* __restrict__ A,
                                                       const float* __restrict__ B, int m,
                                                       long long N, long long chunk,
                                                       double* __restrict__ partial, int same) {
  constexpr int ROWS = 16 * TT;
  extern __shared__ __align__(16) float fsm[];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int ops = same ? 1 : 2;
  const long long p_begin = (long long)blockIdx.x * chunk;
  const long long p_end = p_begin + chunk < N ? p_begin + chunk : N;
  const int ntile = p_begin < p_end ? (int)((p_end - p_begin + kGramPts - 1) / kGramPts) : 0;
  auto fetch = [&](int t) {   // tile t into buffer t % kGramBufs<TT> (N and chunk: multiples of 4)
    if (t < ntile) {
      float* buf = fsm + (size_t)(t % kGramBufs<TT>) * ops * ROWS * kGramPitch;
      const long long p = p_begin + (long long)t * kGramPts + 4 * tx;
      for (int op = 0; op < ops; ++op) {
        const float* X = op == 0 ? A : B;
#pragma unroll
        for (int q = 0; q < TT; ++q) {
          const int i = ty + 16 * q;
          const bool valid = i < m && p < p_end;
          copy16(buf + (op * ROWS + i) * kGramPitch + 4 * tx,
                 valid ? X + (long long)i * N + p : X, valid);
        }
      }
    }
    copies_commit();
  };
  float acc[TT][TT], s[TT][TT], e[TT][TT];
#pragma unroll
  for (int q = 0; q < TT; ++q)
#pragma unroll
    for (int r = 0; r < TT; ++r) acc[q][r] = s[q][r] = e[q][r] = 0.f;
  for (int t = 0; t < kGramBufs<TT> - 1; ++t) fetch(t);
  for (int t = 0; t < ntile; ++t) {
    copies_wait<kGramBufs<TT> - 2>();
    __syncthreads();   // tile t is here, tile t - 1 consumed
    fetch(t + kGramBufs<TT> - 1);
    const float* ta = fsm + (size_t)(t % kGramBufs<TT>) * ops * ROWS * kGramPitch;
    const float* tb = same ? ta : ta + ROWS * kGramPitch;
#pragma unroll 4
    for (int k = 0; k < kGramPts; k += 4) {
      float4 a[TT], b[TT];
#pragma unroll
      for (int q = 0; q < TT; ++q)
        a[q] = *reinterpret_cast<const float4*>(ta + (ty + 16 * q) * kGramPitch + k);
#pragma unroll
      for (int r = 0; r < TT; ++r)
        b[r] = *reinterpret_cast<const float4*>(tb + (tx + 16 * r) * kGramPitch + k);
#pragma unroll
      for (int q = 0; q < TT; ++q)
#pragma unroll
        for (int r = 0; r < TT; ++r) {
          float v = acc[q][r];
          v = fmaf(a[q].x, b[r].x, v);
          v = fmaf(a[q].y, b[r].y, v);
          v = fmaf(a[q].z, b[r].z, v);
          acc[q][r] = fmaf(a[q].w, b[r].w, v);
        }
    }
    if (t & 1) {   // a run of 128 points
#pragma unroll
      for (int q = 0; q < TT; ++q)
#pragma unroll
        for (int r = 0; r < TT; ++r) {
          two_sum(s[q][r], e[q][r], acc[q][r]);
          acc[q][r] = 0.f;
        }
    }
  }
  copies_wait<0>();
  double* out = partial + (long long)blockIdx.x * m * m;
#pragma unroll
  for (int q = 0; q < TT; ++q)
#pragma unroll
    for (int r = 0; r < TT; ++r) {
      const int i = ty + 16 * q, j = tx + 16 * r;
      if (i < m && j < m)
        out[i * m + j] = (double)s[q][r] + ((double)e[q][r] + (double)acc[q][r]);
    }
}

// ---------------------------------------------------------------------------
// Y = M X, m <= 4 RG: M in shared memory as FP32, [k][i]; tiles of PT = 1024 /
// RG points by asynchronous copies, [k][point]; 4 rows x 4 points per thread.
// lower: M[i][k] = 0 for k > i, a row group stops there.
constexpr int kApplyBufs = 3;

template <int RG>
__global__ void __launch_bounds__(256) f32_apply_kernel(const double* __restrict__ M, int m,
                                                        int lower, const float* __restrict__ X,
                                                        float* __restrict__ Y, long long N) {
  constexpr int ROWS = 4 * RG, TX = 256 / RG, PT = 4 * TX;
  extern __shared__ __align__(16) float fsm[];
  float* sM = fsm;                   // [ROWS k][ROWS i]
  float* sX = fsm + ROWS * ROWS;     // [kApplyBufs][ROWS k][PT]
  const int tid = threadIdx.x, ty = tid / TX, tx = tid - ty * TX;
  for (int q = tid; q < ROWS * ROWS; q += 256) {
    const int k = q / ROWS, i = q - k * ROWS;
    sM[q] = i < m && k < m ? (float)M[(long long)i * m + k] : 0.f;
  }
  const long long ntiles = (N + PT - 1) / PT;
  auto fetch = [&](long long tile, int buf) {
    if (tile < ntiles) {
      const long long p = tile * PT + 4 * tx;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = ty + RG * q;
        const bool valid = k < m && p < N;   // N is a multiple of 4
        copy16(sX + ((size_t)buf * ROWS + k) * PT + 4 * tx,
               valid ? X + (long long)k * N + p : X, valid);
      }
    }
    copies_commit();
  };
  const int kmax = lower ? (m < 4 * ty + 4 ? m : 4 * ty + 4) : m;
  for (int b = 0; b < kApplyBufs - 1; ++b) fetch(blockIdx.x + (long long)b * gridDim.x, b);
  int buf = 0;
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    copies_wait<kApplyBufs - 2>();
    __syncthreads();   // this tile is here, the previous one consumed
    const int ahead = buf + kApplyBufs - 1;
    fetch(tile + (long long)(kApplyBufs - 1) * gridDim.x,
          ahead >= kApplyBufs ? ahead - kApplyBufs : ahead);
    const float* xb = sX + (size_t)buf * ROWS * PT + 4 * tx;
    float acc[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < 4; ++r) acc[q][r] = 0.f;
#pragma unroll 4
    for (int k = 0; k < kmax; ++k) {
      const float4 a = *reinterpret_cast<const float4*>(sM + k * ROWS + 4 * ty);
      const float4 b = *reinterpret_cast<const float4*>(xb + k * PT);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[q][r] = fmaf(av[q], bv[r], acc[q][r]);
    }
    const long long p = tile * PT + 4 * tx;
    if (p < N) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (4 * ty + q < m)
          *reinterpret_cast<float4*>(Y + (long long)(4 * ty + q) * N + p) =
              make_float4(acc[q][0], acc[q][1], acc[q][2], acc[q][3]);
    }
    buf = buf + 1 == kApplyBufs ? 0 : buf + 1;
  }
  copies_wait<0>();
}

template <int TT>
cudaError_t gram_launch(const float* A, const float* B, int m, long long N, int n_chunks,
                        double* partial, cudaStream_t st) {
  const bool same = A == B;
  long long chunk = (N + n_chunks - 1) / n_chunks;
  chunk = (chunk + kGramPts - 1) / kGramPts * kGramPts;
  const size_t smem = gram_smem<TT>(same);
  cudaError_t e = cudaFuncSetAttribute(f32_gram_kernel<TT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)gram_smem<TT>(false));
  if (e != cudaSuccess) return e;
  f32_gram_kernel<TT><<<n_chunks, 256, smem, st>>>(A, B, m, N, chunk, partial, same ? 1 : 0);
  return cudaGetLastError();
}

template <int RG>
cudaError_t apply_launch(const double* M, int m, int lower, const float* X, float* Y, long long N,
                         cudaStream_t st) {
  constexpr int ROWS = 4 * RG, PT = 1024 / RG;
  const size_t smem = ((size_t)ROWS * ROWS + (size_t)kApplyBufs * ROWS * PT) * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(f32_apply_kernel<RG>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 152, per = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f32_apply_kernel<RG>, 256, smem);
  if (e != cudaSuccess) return e;
  const long long ntiles = (N + PT - 1) / PT, cap = (long long)sms * (per < 1 ? 1 : per);
  f32_apply_kernel<RG><<<(int)(ntiles < cap ? ntiles : cap), 256, smem, st>>>(M, m, lower, X, Y,
                                                                              N);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_f32_gram(const float* A, const float* B, int m, long long n_points,
                            int n_chunks, double* partial, cudaStream_t st) {
  if (m < 1 || m > kF32MaxM || (n_points & 3)) return cudaErrorInvalidValue;
  switch ((m + 15) / 16) {
    case 1: return gram_launch<1>(A, B, m, n_points, n_chunks, partial, st);
    case 2: return gram_launch<2>(A, B, m, n_points, n_chunks, partial, st);
    case 3: return gram_launch<3>(A, B, m, n_points, n_chunks, partial, st);
    default: return gram_launch<4>(A, B, m, n_points, n_chunks, partial, st);
  }
}

cudaError_t launch_f32_apply(const double* M, int m, int lower, const float* X, float* Y,
                             long long n_points, cudaStream_t st) {
  if (m < 1 || m > kF32MaxM || (n_points & 3)) return cudaErrorInvalidValue;
  if (m <= 16) return apply_launch<4>(M, m, lower, X, Y, n_points, st);
  if (m <= 32) return apply_launch<8>(M, m, lower, X, Y, n_points, st);
  return apply_launch<16>(M, m, lower, X, Y, n_points, st);
}

}  // namespace itp
