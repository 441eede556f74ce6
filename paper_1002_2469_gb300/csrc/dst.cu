// dst.cu -- the steps around the FFT of the Poisson driver's sine transform (orthonormal DST-I along the
// first axis of an [M, My] array, poisson.py).
//
// With N = M + 1 and a_0 = a_N = 0, y_k = sin(pi k / N) (a_k + a_{N-k}) + (a_k - a_{N-k}) / 2 has
// sum_k y_k exp(-2 pi i k m / N) = C_m - i S_m with X_{2m} = S_m and X_{2m+1} = C_0 / 2 + C_1 + ... + C_m.
// Every column has a real FFT of its own: two columns in one complex FFT would each carry rounding errors
// of the larger one's size, and its Inf and NaN.  (cuFFT itself takes two rows at a time at odd lengths above
// 256.  A Poisson solve of 2000 x 2319 1363 us, with pairs 1299; 1999 x 2319 922 and 765, 3071 x 3071 1565
// and 1342.)  The transform's scale sqrt(2 / N) (and the caller's) is folded into the coefficients
// c1 = scale (s + 1/2), c2 = scale (s - 1/2) of y_k = c1 a_k + c2 a_{N-k}, y_{N-k} = c2 a_k + c1 a_{N-k}.
//
// Each kernel reads and writes its arrays once (the torch expressions they replace made about 15 passes
// and strided ones among them).  Both move 16 bytes per element; the FP64 pipe (2 operations per clock
// and SM) bounds them too: 2 operations per element before the FFT, about 2 after it.
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/dichotomy.h"
#include "planner.cuh"

namespace dich {

// ---------------------------------------------------------------- before the FFT
// a [M][My] (row k - 1 holds a_k) -> z [My][N].  One CTA: 32 values of k and their
// mirror images, 64 columns; the tile is transposed in shared memory, so that rows of a are read in runs of
// 512 bytes and rows of z written in runs of 256.  coef[k] = (c1, c2), k = 0 .. N / 2.
constexpr int kPreK = 32, kPreJ = 64, kPrePitch = kPreJ + 1;

__global__ void __launch_bounds__(256) k_dst_pre(int64_t M, int64_t My, const double* a, const double2* coef,
                                                 double* z) {
  __shared__ double t1[kPreK * kPrePitch], t2[kPreK * kPrePitch];
  const int64_t N = M + 1, tiles_j = (My + kPreJ - 1) / kPreJ;   // one grid dimension: either may be long
  const int64_t k0 = blockIdx.x / tiles_j * kPreK, j0 = blockIdx.x % tiles_j * kPreJ;
  const int64_t half = N / 2;
  const int jj = threadIdx.x & 63;
  const bool jin = j0 + jj < My;
#pragma unroll
  for (int i = 0; i < kPreK / 4; ++i) {
    const int kk = (threadIdx.x >> 6) + 4 * i;
    const int64_t k = k0 + kk;
    double u = 0.0, v = 0.0;
    if (k >= 1 && k <= half && jin) {
      const double x = __ldcs(a + (k - 1) * My + j0 + jj), y = __ldcs(a + (N - k - 1) * My + j0 + jj);
      const double2 c = coef[k];
      u = fma(c.x, x, c.y * y);
      v = fma(c.y, x, c.x * y);
    }
    t1[kk * kPrePitch + jj] = u;
    t2[kk * kPrePitch + jj] = v;
  }
  __syncthreads();
  const int kk = threadIdx.x & 31;
  const int64_t k = k0 + kk;
  if (k > half) return;
#pragma unroll
  for (int i = 0; i < kPreJ / 8; ++i) {
    const int c = (threadIdx.x >> 5) + 8 * i;
    if (j0 + c >= My) break;
    double* row = z + (j0 + c) * N;
    row[k] = t1[kk * kPrePitch + c];
    if (k >= 1 && 2 * k != N) row[N - k] = t2[kk * kPrePitch + c];
  }
}

// ---------------------------------------------------------------- after the FFT
// Z [My][N / 2 + 1] -> X [M][My].  One CTA: eight pairs of columns, a warp each, marching over m in
// chunks of 128 (4 per lane) with the running sums carried along; the chunk's 256 rows by 16 columns
// leave through shared memory in runs of 128 bytes.  The next chunk's values are loaded before the
// current one is stored.
constexpr int kPostM = 128, kPostPairs = 8, kPostPitch = 2 * kPostPairs + 1;

__global__ void __launch_bounds__(256) k_dst_post(int64_t M, int64_t My, const double2* Z, double* X) {
  __shared__ double t[2 * kPostM * kPostPitch];
  const int64_t N = M + 1, pairs = (My + 1) / 2;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t p0 = (int64_t)blockIdx.x * kPostPairs, p = p0 + wid;
  const int64_t pitch = N / 2 + 1;
  const bool two = 2 * p + 1 < My;   // the pair's second column
  const double2* z0 = Z + (p < pairs ? 2 * p : 0) * pitch;
  const double2* z1 = z0 + (two ? pitch : 0);
  const int64_t last = M / 2;   // the largest m: X_{2m} up to M, X_{2m+1} up to M
  double2 q[4], r[4];           // Z_m of both columns, the lane's four m
  auto load = [&](int64_t m0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t m = m0 + 4 * lane + i;
      const bool in = m <= last && p < pairs;
      q[i] = in ? __ldcs(z0 + m) : make_double2(0.0, 0.0);
      r[i] = (in && two) ? __ldcs(z1 + m) : make_double2(0.0, 0.0);
    }
  };
  load(0);
  double run0 = 0.0, run1 = 0.0;   // the running sums of the two columns
  for (int64_t m0 = 0; m0 <= last; m0 += kPostM) {
    double c0[4], c1[4], s0[4], s1[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      c0[i] = q[i].x;
      c1[i] = r[i].x;
      s0[i] = -q[i].y;
      s1[i] = -r[i].y;
    }
    if (m0 + lane == 0) {   // C_0 / 2
      c0[0] *= 0.5;
      c1[0] *= 0.5;
    }
    if (m0 + kPostM <= last) load(m0 + kPostM);
    // inclusive sums over the lane's four, then the exclusive scan of the lanes' totals
#pragma unroll
    for (int i = 1; i < 4; ++i) {
      c0[i] += c0[i - 1];
      c1[i] += c1[i - 1];
    }
    double e0 = c0[3], e1 = c1[3];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const double y0 = __shfl_up_sync(0xffffffffu, e0, d), y1 = __shfl_up_sync(0xffffffffu, e1, d);
      if (lane >= d) {
        e0 += y0;
        e1 += y1;
      }
    }
    const double n0 = run0 + __shfl_sync(0xffffffffu, e0, 31), n1 = run1 + __shfl_sync(0xffffffffu, e1, 31);
    double b0 = __shfl_up_sync(0xffffffffu, e0, 1), b1 = __shfl_up_sync(0xffffffffu, e1, 1);
    b0 = lane ? run0 + b0 : run0;
    b1 = lane ? run1 + b1 : run1;
    run0 = n0;
    run1 = n1;
    // tile row 32 u + lane: u = 2 i for X_{2m}, 2 i + 1 for X_{2m+1} (m = m0 + 4 lane + i)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      double* te = t + (32 * (2 * i) + lane) * kPostPitch + 2 * wid;
      double* to = t + (32 * (2 * i + 1) + lane) * kPostPitch + 2 * wid;
      te[0] = s0[i];
      te[1] = s1[i];
      to[0] = b0 + c0[i];
      to[1] = b1 + c1[i];
    }
    __syncthreads();
    const int col = threadIdx.x & 15;
    const int64_t j = 2 * p0 + col;
    if (j < My)
#pragma unroll 4
      for (int row = threadIdx.x >> 4; row < 2 * kPostM; row += 16) {
        const int u = row >> 5;
        const int64_t K = 2 * (m0 + 4 * (row & 31) + (u >> 1)) + (u & 1);   // X_K
        if (K >= 1 && K <= M) __stcs(X + (K - 1) * My + j, t[row * kPostPitch + col]);
      }
    __syncthreads();
  }
}

}  // namespace dich

using namespace dich;
using namespace dich::plan;

extern "C" {

int dichotomy_dst_rows_pre(int64_t M, int64_t My, const double* d_a, const double* d_coef, double* d_z, void* stream) {
  if (M < 1 || My < 1 || !d_a || !d_coef || !d_z) return DICH_ERR_ARG;
  if (!aligned8(d_a) || ((uintptr_t)d_coef & 15u) != 0 || !aligned8(d_z)) return DICH_ERR_ARG;
  if (!is_device_ptr(d_a) || !is_device_ptr(d_coef) || !is_device_ptr(d_z)) return DICH_ERR_ARG;
  const int64_t gk = ((M + 1) / 2 + 1 + kPreK - 1) / kPreK, gj = (My + kPreJ - 1) / kPreJ;
  if (gk > INT32_MAX / gj) return DICH_ERR_UNSUPPORTED;
  k_dst_pre<<<(unsigned)(gk * gj), 256, 0, (cudaStream_t)stream>>>(M, My, d_a, (const double2*)d_coef, d_z);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DICH_OK : cuda_fail(e);
}

int dichotomy_dst_rows_post(int64_t M, int64_t My, const double* d_Z, double* d_X, void* stream) {
  if (M < 1 || My < 1 || !d_Z || !d_X) return DICH_ERR_ARG;
  if (!aligned8(d_X) || ((uintptr_t)d_Z & 15u) != 0) return DICH_ERR_ARG;
  if (!is_device_ptr(d_Z) || !is_device_ptr(d_X)) return DICH_ERR_ARG;
  const int64_t grid = ((My + 1) / 2 + kPostPairs - 1) / kPostPairs;
  if (grid > INT32_MAX) return DICH_ERR_UNSUPPORTED;
  k_dst_post<<<(unsigned)grid, 256, 0, (cudaStream_t)stream>>>(M, My, (const double2*)d_Z, d_X);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DICH_OK : cuda_fail(e);
}

}  // extern "C"
