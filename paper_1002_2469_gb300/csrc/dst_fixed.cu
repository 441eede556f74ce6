// dst_fixed.cu -- the Poisson driver's orthonormal DST-I (length M along the first axis of an [M, My]
// array) in 64-bit fixed point, for N = M + 1 a power of two from 512 to 4096.
//
// In FP64 the transform is bound by the FP64 pipe (2 operations per clock and SM): an FFT of two columns
// of 4095 rows needs 2.5e5 of them, 765 us of library time for 4095 columns, ten times the time its
// data takes to move.  Here the columns are words in their own units (block floating point): additions
// and products by twiddles go to the integer pipes, FP64 only converts and scales the results.
//   1. the array is transposed, columns become rows;
//   2. one CTA of N / 16 threads per pair of rows: y_k = s_k (a_k + a_{N-k}) + (a_k - a_{N-k}) / 2
//      (s_k = sin(pi k / N)), the pair's FFT z = y + i y' in shared memory (16 bytes a point, 16 points a
//      thread and pass, radices 16, 16 and N / 256 = 2 to 16), the split of both rows' spectra and the running sums
//      of the odd outputs (dst.cu has the formulas);
//   3. the result is transposed back.
// A word of the input is below 2^56; each pass's words are shifted back below 2^59 as far as its largest
// needs (radix 16 grows a component at most 16 sqrt(2)-fold, and every product by a twiddle is halved),
// so the unit stays within a few bits of the data: about 2^-55 of the largest spectrum value, where the
// FP64 transform's rounding errors are about 2^-53 of the spectrum's rms each.
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/dichotomy.h"
#include "fixed.cuh"
#include "planner.cuh"
#include "window.cuh"

namespace dich {

struct cw {
  u64 r, i;   // two's complement
};
__device__ __forceinline__ cw operator+(cw a, cw b) { return cw{a.r + b.r, a.i + b.i}; }
__device__ __forceinline__ cw operator-(cw a, cw b) { return cw{a.r - b.r, a.i - b.i}; }
__device__ __forceinline__ u64 asr(u64 x, int s) { return (u64)((long long)x >> s); }
// Truncations are kept free of bias on average: the odd outputs are running sums over half the spectrum,
// which add up a mean error of a unit per point to N / 2 units.  A product truncates 1.25 units on
// average (1 + half its factor's low word), a halving a quarter: where half a unit is due a bit `par` that
// varies over the points without a pattern (a pattern's mean error would gather at one frequency) adds
// it or not, constants take the nearest whole number.
// x c for a signed word and 0 <= c < 1 (c a multiple of 2^-64), acc added
__device__ __forceinline__ u64 smul(u64 x, u64 c, unsigned acc) {
  return fx_mul(x ^ (1ull << 63), (unsigned)(c >> 32), (unsigned)c, (u64)acc - (c >> 1));
}
// x w / 2 for w = (2 C - 1) + i (2 S - 1), C and S even
__device__ __forceinline__ cw cmul_half(cw x, u64 C, u64 S, unsigned par) {
  const u64 a = x.r ^ (1ull << 63), b = x.i ^ (1ull << 63);
  const u64 hc = C >> 1, hs = S >> 1;
  const u64 re = fx_mul(a, C, hs - hc - asr(x.r - x.i + par, 1)) - fx_mul(b, S, 0ull);
  const u64 im = fx_mul(a, S, (2ull + par) - hs - hc - asr(x.r + x.i + (1u - par), 1)) + fx_mul(b, C, 0ull);
  return cw{re, im};
}
__device__ __forceinline__ cw mul_mi(cw a) { return cw{a.i, 0ull - a.r}; }   // a (-i)

// forward DFTs (exp(-2 pi i / R)) of x[0], x[st], ... in place, natural order
template <int R>
__device__ __forceinline__ void dft(cw* x);
template <>
__device__ __forceinline__ void dft<1>(cw*) {}
template <>
__device__ __forceinline__ void dft<2>(cw* x) {
  const cw a = x[0], b = x[1];
  x[0] = a + b;
  x[1] = a - b;
}
template <>
__device__ __forceinline__ void dft<4>(cw* x) {
  const cw a = x[0] + x[2], b = x[0] - x[2], c = x[1] + x[3], d = mul_mi(x[1] - x[3]);
  x[0] = a + c;
  x[1] = b + d;
  x[2] = a - c;
  x[3] = b - d;
}
constexpr u64 kSqrtHalf = 0xB504F333F9DE6484ull;   // sqrt(1/2) 2^64
constexpr u64 kCos8 = 0xEC835E79946A3145ull;       // cos(pi / 8) 2^64
constexpr u64 kSin8 = 0x61F78A9ABAA58B47ull;       // sin(pi / 8) 2^64
// x exp(-i pi / 4), x exp(-3 i pi / 4)
__device__ __forceinline__ cw rot1(cw x) { return cw{smul(x.r + x.i, kSqrtHalf, 1), smul(x.i - x.r, kSqrtHalf, 2)}; }
__device__ __forceinline__ cw rot3(cw x) { return cw{smul(x.i - x.r, kSqrtHalf, 2), 0ull - smul(x.r + x.i, kSqrtHalf, 1)}; }
// x (c - i s) for 0 <= c, s < 1
__device__ __forceinline__ cw rotcs(cw x, u64 c, u64 s) {
  return cw{smul(x.r, c, 1) + smul(x.i, s, 1), smul(x.i, c, 1) - smul(x.r, s, 1)};
}
template <>
__device__ __forceinline__ void dft<8>(cw* x) {
  cw e[4] = {x[0], x[2], x[4], x[6]}, o[4] = {x[1], x[3], x[5], x[7]};
  dft<4>(e);
  dft<4>(o);
  o[1] = rot1(o[1]);
  o[2] = mul_mi(o[2]);
  o[3] = rot3(o[3]);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    x[k] = e[k] + o[k];
    x[k + 4] = e[k] - o[k];
  }
}
template <>
__device__ __forceinline__ void dft<16>(cw* x) {
  // 4 x 4: columns n2 = 0..3 over n1, twiddles W16^(n2 k1), rows
  cw y[4][4];
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
    cw t[4] = {x[n2], x[n2 + 4], x[n2 + 8], x[n2 + 12]};
    dft<4>(t);
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) y[k1][n2] = t[k1];
  }
  y[1][1] = rotcs(y[1][1], kCos8, kSin8);              // W^1
  y[1][2] = rot1(y[1][2]);                             // W^2
  y[1][3] = rotcs(y[1][3], kSin8, kCos8);              // W^3
  y[2][1] = rot1(y[2][1]);                             // W^2
  y[2][2] = mul_mi(y[2][2]);                           // W^4
  y[2][3] = rot3(y[2][3]);                             // W^6
  y[3][1] = rotcs(y[3][1], kSin8, kCos8);              // W^3
  y[3][2] = rot3(y[3][2]);                             // W^6
  {                                                    // W^9 = -W^1
    const cw t = rotcs(y[3][3], kCos8, kSin8);
    y[3][3] = cw{0ull - t.r, 0ull - t.i};
  }
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    dft<4>(y[k1]);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) x[k1 + 4 * k2] = y[k1][k2];
  }
}

// bits above 2^59 of the largest component seen (m: the OR of the components' magnitudes' high words),
// over the CTA; one barrier.  sh: 32 words per parity of use
template <int T>
__device__ __forceinline__ int cta_shift(unsigned m, unsigned* sh, int limit) {
  m = __reduce_or_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  unsigned all = 0u;
#pragma unroll
  for (int w = 0; w < T / 32; ++w) all |= sh[w];
  return max(0, 32 - __clz((int)all) - (limit - 32));
}

// points of the pair in shared memory: one 16-byte slot of padding per 16
__device__ __forceinline__ int at(int i) { return i + (i >> 4); }

// one pass: sub-transforms of length L become length L R; T = N / 16 threads, 16 points each
template <int N, int L, int R>
__device__ __forceinline__ void pass(cw* z, const ulonglong2* tw, int shift, unsigned& mag) {
  constexpr int T = N / 16, B = 16 / R;
  cw x[B][R];
  // the shift rounds: half of its unit, or one less (par)
  const unsigned odd = shift ? 1u : 0u;
  const u64 half = (1ull << shift >> 1) - odd;
#pragma unroll
  for (int b = 0; b < B; ++b) {
    const int j = threadIdx.x + b * T, k = j % L;
    const unsigned bits = ((unsigned)(j + L) * 2654435761u) >> 12;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      cw v = z[at(j + q * (N / R))];
      if (L > 1) {
        const unsigned par = bits >> q & 1u, par2 = bits >> (q + 4) & 1u;
        v = cw{asr(v.r + half + (par & odd), shift), asr(v.i + half + (par2 & odd), shift)};
        if (q == 0) {
          v = cw{asr(v.r + par2, 1), asr(v.i + par, 1)};
        } else {
          const ulonglong2 w = __ldg(tw + k * q * (N / (L * R)));
          v = cmul_half(v, w.x, w.y, par);
        }
      }
      x[b][q] = v;
    }
    dft<R>(x[b]);
  }
  __syncthreads();   // every point has been read
  mag = 0u;
#pragma unroll
  for (int b = 0; b < B; ++b) {
    const int j = threadIdx.x + b * T, k = j % L;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const cw v = x[b][q];
      z[at((j - k) * R + k + q * L)] = v;
      const int hr = (int)(v.r >> 32), hi = (int)(v.i >> 32);
      mag |= (unsigned)(hr ^ (hr >> 31)) | (unsigned)(hi ^ (hi >> 31));
    }
  }
}

// the sign bit of a row: multiplicative hashing twice, the high bits folded into the low ones between
__device__ __forceinline__ unsigned row_sign(unsigned r) {
  unsigned h = (r + 1u) * 2654435761u;
  h = (h ^ (h >> 15)) * 2654435761u;
  return h & 0x80000000u;
}

// rows 2p, 2p + 1 of w (N doubles each, the first M used) replaced by their transforms times scale.
// tab: N twiddles ((cos + 1) / 2, (1 - sin) / 2) of angles 2 pi m / N, then s_k, k = 0 .. N / 2 (words)
template <int N>
__global__ void __launch_bounds__(N / 16, 512 / (N / 16)) k_dst_fixed(double* w, const ulonglong2* tw, double scale) {
  constexpr int T = N / 16, NW = T / 32, LOGN = (N == 4096) ? 12 : (N == 2048) ? 11 : (N == 1024) ? 10 : 9;
  extern __shared__ __align__(16) unsigned char smem[];
  cw* z = reinterpret_cast<cw*>(smem);
  u64* sums = reinterpret_cast<u64*>(z + at(N));                 // 2 NW
  unsigned* sh = reinterpret_cast<unsigned*>(sums + 2 * NW);     // 4 NW
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  double* r0 = w + (int64_t)blockIdx.x * 2 * N;
  double* r1 = r0 + N;
  const u64* sine = reinterpret_cast<const u64*>(tw + N);

  // ---------------------------------------------------------------- rows -> words -> y
  // thread t: k = 1 + t + i T and N - k, i = 0..7 (k = N / 2 is its own mirror image)
  // What bias the products and shifts keep is the same in every row of one scale, and a solve along the
  // rows' index would add it up over them: each row is negated or not, without a pattern, on its way
  // in and out.
  const unsigned neg0 = row_sign(2u * blockIdx.x), neg1 = row_sign(2u * blockIdx.x + 1u);
  auto flip = [](double a, unsigned g) { return __hiloint2double(__double2hiint(a) ^ (int)g, __double2loint(a)); };
  double a0[8], b0[8], a1[8], b1[8];
  unsigned m0 = 0u, m1 = 0u;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = 1 + tid + i * T;
    a0[i] = flip(r0[k - 1], neg0);
    b0[i] = flip(r0[N - k - 1], neg0);
    a1[i] = flip(r1[k - 1], neg1);
    b1[i] = flip(r1[N - k - 1], neg1);
    m0 = __vimax3_u32(m0, (unsigned)__double2hiint(a0[i]) & 0x7FFFFFFFu, (unsigned)__double2hiint(b0[i]) & 0x7FFFFFFFu);
    m1 = __vimax3_u32(m1, (unsigned)__double2hiint(a1[i]) & 0x7FFFFFFFu, (unsigned)__double2hiint(b1[i]) & 0x7FFFFFFFu);
  }
  m0 = __reduce_max_sync(0xffffffffu, m0);
  m1 = __reduce_max_sync(0xffffffffu, m1);
  if (lane == 0) {
    sh[2 * NW + wid] = m0;
    sh[3 * NW + wid] = m1;
  }
  __syncthreads();
#pragma unroll
  for (int v = 0; v < NW; ++v) {
    m0 = max(m0, sh[2 * NW + v]);
    m1 = max(m1, sh[3 * NW + v]);
  }
  const int e0 = (int)(m0 >> 20), e1 = (int)(m1 >> 20);
  // rows near the lower end of the FP64 range move up first (exactly), so that zeros convert to zero
  const int up0 = e0 < 128 ? 600 : 0, up1 = e1 < 128 ? 600 : 0;
  if (up0)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      a0[i] *= pow2i(600);
      b0[i] *= pow2i(600);
    }
  if (up1)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      a1[i] *= pow2i(600);
      b1[i] *= pow2i(600);
    }
  // |a| 2^sc < 2^56 (e = 0: subnormal, below 2^-1022)
  const int sc0 = 56 - (e0 + up0 + (e0 == 0) - 1022), sc1 = 56 - (e1 + up1 + (e1 == 0) - 1022);
  const unsigned sb0 = (unsigned)(1086 - sc0), sb1 = (unsigned)(1086 - sc1);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = 1 + tid + i * T;
    const u64 s = sine[k];
    auto fold = [&](double a, double b, unsigned sb, u64& y, u64& ym) {
      const u64 x = fx_from_f64_alu(a, sb, 0ull), v = fx_from_f64_alu(b, sb, 0ull);
      const u64 m = smul(x + v, s, ((unsigned)k * 2654435761u) >> 30 ? 1 : 2), d = asr(x - v, 1);
      y = m + d;
      ym = m - d;
    };
    cw y, ym;
    fold(a0[i], b0[i], sb0, y.r, ym.r);
    fold(a1[i], b1[i], sb1, y.i, ym.i);
    z[at(k)] = y;
    if (k != N / 2) z[at(N - k)] = ym;
  }
  if (tid == 0) z[0] = cw{0ull, 0ull};
  __syncthreads();

  // ---------------------------------------------------------------- FFT
  unsigned mag;
  int units = 0;   // right shifts so far (the words' unit is 2^units times the input's)
  pass<N, 1, 16>(z, tw, 0, mag);
  int s = cta_shift<T>(mag, sh, 59);   // (its barrier also orders the points)
  units += s + 1;
  pass<N, 16, 16>(z, tw, s, mag);
  s = cta_shift<T>(mag, sh + NW, 58);   // one bit more of room: the spectra below add two points
  units += s + 1;
  pass<N, 256, N / 256>(z, tw, s, mag);
  __syncthreads();

  // ---------------------------------------------------------------- spectra of both rows, running sums
  // 2 |X_K| <= 2 N 2^56 in the input's unit: below 2^62 after this shift.  The running sums keep 96 bits
  // until then (a shifted point's rounding would add up along them).
  const int s2 = max(0, LOGN - 5 - units);
  units += s2;
  struct sum96 {
    u64 l;
    int h;
  };
  auto add = [](sum96 a, sum96 b) {
    sum96 c;
    c.l = a.l + b.l;
    c.h = a.h + b.h + (c.l < a.l ? 1 : 0);
    return c;
  };
  auto wide = [](u64 v) { return sum96{v, (int)(v >> 32) >> 31}; };
  auto narrow = [s2](sum96 a) { return s2 ? (a.l >> s2) | ((u64)(long long)a.h << (64 - s2)) : a.l; };
  u64 c0[8], c1[8], d0[8], d1[8];
  sum96 t0{0ull, 0}, t1{0ull, 0};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = 8 * tid + i;
    const cw q = z[at(m)], r = m ? z[at(N - m)] : cw{0ull, 0ull};   // m = 0: C_0 / 2 = Re Z_0
    c0[i] = q.r + r.r;
    c1[i] = q.i + r.i;
    d0[i] = asr(r.i - q.i, s2);
    d1[i] = asr(q.r - r.r, s2);
    t0 = add(t0, wide(c0[i]));
    t1 = add(t1, wide(c1[i]));
  }
  const sum96 own0 = t0, own1 = t1;
  auto up = [](sum96 a, int d) {
    return sum96{__shfl_up_sync(0xffffffffu, a.l, d), __shfl_up_sync(0xffffffffu, a.h, d)};
  };
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const sum96 y0 = up(t0, d), y1 = up(t1, d);
    if (lane >= d) {
      t0 = add(t0, y0);
      t1 = add(t1, y1);
    }
  }
  if (lane == 31) {
    sums[wid] = t0.l;
    sums[NW + wid] = t1.l;
    sh[2 * NW + wid] = (unsigned)t0.h;
    sh[3 * NW + wid] = (unsigned)t1.h;
  }
  auto sub = [](sum96 a, sum96 b) {
    sum96 c;
    c.l = a.l - b.l;
    c.h = a.h - b.h - (a.l < b.l ? 1 : 0);
    return c;
  };
  t0 = sub(t0, own0);
  t1 = sub(t1, own1);
  __syncthreads();   // (and every point has been read)
  for (int v = 0; v < wid; ++v) {
    t0 = add(t0, sum96{sums[v], (int)sh[2 * NW + v]});
    t1 = add(t1, sum96{sums[NW + v], (int)sh[3 * NW + v]});
  }
  // words to FP64 by one conversion and one product (two where the unit is near the ends of the range)
  const int k0 = units - sc0 - up0, k1 = units - sc1 - up1;
  const int h0 = k0 / 2, h1 = k1 / 2;
  const bool plain = abs(k0) < 900 && abs(k1) < 900;
  const double f0 = flip(plain ? scale * pow2i(k0) : scale * pow2i(h0), neg0);
  const double f1 = flip(plain ? scale * pow2i(k1) : scale * pow2i(h1), neg1);
  const double g0 = pow2i(k0 - h0), g1 = pow2i(k1 - h1);
  double* o0 = reinterpret_cast<double*>(z);
  // X_{2m}, X_{2m+1} of row 0 at o0, of row 1 behind it; one 16-byte slot of padding per 16 pairs
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = 8 * tid + i;
    t0 = add(t0, wide(c0[i]));
    t1 = add(t1, wide(c1[i]));
    double2 x0 = make_double2(__ll2double_rn((long long)d0[i]) * f0, __ll2double_rn((long long)narrow(t0)) * f0);
    double2 x1 = make_double2(__ll2double_rn((long long)d1[i]) * f1, __ll2double_rn((long long)narrow(t1)) * f1);
    if (!plain) {
      x0 = make_double2(x0.x * g0, x0.y * g0);
      x1 = make_double2(x1.x * g1, x1.y * g1);
    }
    reinterpret_cast<double2*>(o0)[at(m)] = x0;
    reinterpret_cast<double2*>(o0)[at(N / 2 + m)] = x1;
  }
  __syncthreads();
  const double bad = __hiloint2double(0x7FF80000, 0);   // a row with Inf or NaN: every output is NaN
#pragma unroll 4
  for (int j = tid; j < N / 2; j += T) {
    double2 x0 = reinterpret_cast<const double2*>(o0)[at(j)], x1 = reinterpret_cast<const double2*>(o0)[at(N / 2 + j)];
    if (m0 == 0u) x0 = make_double2(0.0, 0.0);   // a row of zeros: nothing of the other row's rounding
    if (m1 == 0u) x1 = make_double2(0.0, 0.0);
    if (e0 == 2047) x0 = make_double2(bad, bad);
    if (e1 == 2047) x1 = make_double2(bad, bad);
    // X_K at index K (index 0 is unused): whole 16-byte stores
    reinterpret_cast<double2*>(r0)[j] = x0;
    reinterpret_cast<double2*>(r1)[j] = x1;
  }
}

// ---------------------------------------------------------------- transposes (64 x 32 tiles)
// out[c ldo + r + oshift] = in[r ldi + c + ishift], r < R, c < C
__global__ void __launch_bounds__(256) k_transpose(const double* in, int64_t ldi, int ishift, double* out, int64_t ldo,
                                                   int oshift, int64_t R, int64_t C) {
  __shared__ double t[32][65];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int64_t tc = (C + 63) / 64, r0 = blockIdx.x / tc * 32, c0 = blockIdx.x % tc * 64;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = (threadIdx.x >> 6) + 4 * i, c = threadIdx.x & 63;
    if (r0 + r < R && c0 + c < C) t[r][c] = __ldcs(in + (r0 + r) * ldi + c0 + c + ishift);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = threadIdx.x & 31, c = (threadIdx.x >> 5) + 8 * i;
    if (r0 + r < R && c0 + c < C) out[(c0 + c) * ldo + r0 + r + oshift] = t[r][c];
  }
}

template <typename K, typename... Args>
static cudaError_t launch_after(K kernel, int64_t grid, int threads, size_t smem, cudaStream_t st, Args... args) {
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute a[1];
  a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = a;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int N>
static cudaError_t launch_fixed(int64_t pairs, double* w, const ulonglong2* tw, double scale, cudaStream_t st) {
  constexpr int T = N / 16, NW = T / 32;
  const size_t smem = sizeof(cw) * (size_t)(N + N / 16) + 8 * 2 * NW + 4 * 4 * NW;
  return launch_after(k_dst_fixed<N>, pairs, T, smem, st, w, tw, scale);
}

}  // namespace dich

using namespace dich;
using namespace dich::plan;

extern "C" int dichotomy_dst(int64_t M, int64_t My, const double* d_a, const void* d_table, double scale,
                             double* d_work, double* d_X, void* stream) {
  const int64_t N = M + 1;
  if (My < 1 || (N != 512 && N != 1024 && N != 2048 && N != 4096)) return DICH_ERR_ARG;
  if (!d_a || !d_table || !d_work || !d_X || !aligned8(d_a) || !aligned8(d_X)) return DICH_ERR_ARG;
  if ((((uintptr_t)d_table | (uintptr_t)d_work) & 15u) != 0) return DICH_ERR_ARG;
  if (!is_device_ptr(d_a) || !is_device_ptr(d_table) || !is_device_ptr(d_work) || !is_device_ptr(d_X)) return DICH_ERR_ARG;
  const int64_t pairs = (My + 1) / 2;
  const int64_t t1 = ((M + 31) / 32) * ((My + 63) / 64), t2 = ((My + 31) / 32) * ((M + 63) / 64);
  if (pairs > INT32_MAX || t1 > INT32_MAX || t2 > INT32_MAX) return DICH_ERR_UNSUPPORTED;
  cudaStream_t st = (cudaStream_t)stream;
  // a row of the work array holds a_1 .. a_M (and one unused element); afterwards X_K at index K
  cudaError_t e = cudaSuccess;
  if (My & 1) e = cudaMemsetAsync(d_work + My * N, 0, sizeof(double) * (size_t)N, st);   // the last pair's second row
  if (e == cudaSuccess) e = launch_after(k_transpose, t1, 256, 0, st, d_a, My, 0, d_work, N, 0, M, My);
  const ulonglong2* tw = (const ulonglong2*)d_table;
  if (e == cudaSuccess) {
    switch (N) {
      case 512: e = launch_fixed<512>(pairs, d_work, tw, scale, st); break;
      case 1024: e = launch_fixed<1024>(pairs, d_work, tw, scale, st); break;
      case 2048: e = launch_fixed<2048>(pairs, d_work, tw, scale, st); break;
      default: e = launch_fixed<4096>(pairs, d_work, tw, scale, st); break;
    }
  }
  if (e == cudaSuccess) e = launch_after(k_transpose, t2, 256, 0, st, d_work, N, 1, d_X, My, 0, My, M);
  return e == cudaSuccess ? DICH_OK : cuda_fail(e);
}
