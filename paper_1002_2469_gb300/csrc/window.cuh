// window.cuh -- the Dichotomy window kernel (sm_103a).
//
// One CTA of NT threads handles a window of up to NT consecutive blocks of one system;
// thread b owns window block b.  Per window:
//   1. the window's rows of F (contiguous in HBM) are copied into shared memory with
//      8-byte cp.async copies, every thread issuing all of its copies before waiting, into
//      a transposed layout (row i of all blocks side by side, stride NT+1 doubles, so the
//      per-thread sweeps below read conflict-free);
//   2. local sweeps (a1): every thread runs the two first-order recurrences of its block
//      (u_i = f_i + rs u_{i-1}, X_i = u_i + ib X_{i+1}, xp_i = g X_i) in place, giving the
//      block ends alpha, omega of T_n^-1 F_m and then beta^{L,R}_m of eq. 16 through the
//      2x2 map M;
//   3. the dichotomy tree (a2): eq. 15 as two affine scans (prefix A, suffix B) -- five
//      warp-shuffle levels, then one shared-memory level across warps -- and the
//      first/last values x_s, x_e of every block (eq. 18);
//   4. the basis correction (a3): x = xp + (x_{s-1} - xp(-1)) v + x_{e+1} w, applied only
//      where the spikes v, w exceed the truncation threshold, and a contiguous,
//      coalesced store of the own rows.
// Windows of a long system overlap by halo blocks on each side whose coupling into the
// own blocks has decayed below the truncation threshold (2^-64 for FP64 plans, 2^-56 for
// MIXED ones, whose float-float values hold about 48 bits); on the
// general path the window instead takes the first/last values from a global scan (the FP64
// form's beta pass leaves xp in x and its apply pass starts from there, without new sweeps).
//
// This file holds the FP64 form's tree and what both window kernels share; the FP64 form's kernel (one
// block per thread) is in window_f64.cuh, the MIXED form's in window_mixed.cuh.
#pragma once

#include "dich_internal.cuh"

namespace dich {

struct WinArgs {
  const SysPlan* plans;   // plan records (device)
  const double* tabs;     // table buffer (device)
  const Item* items;      // batched: one item per CTA; nullptr: single system, one window per CTA
  const double* F;        // right-hand sides
  double* x;              // solutions
  unsigned* status;       // device status word
  const double* iface;    // MODE_APPLY: (x_s, x_e) per block
  double* beta;           // MODE_BETA: (beta^L, beta^R) per block
  const double* xf;       // adjoint: forward solution (gradient sums), else nullptr
  double* part;           // adjoint: per-CTA partial sums [3 per CTA]
  int32_t mode;
  int32_t check_finite;
  int32_t n_smem;         // shared-memory rows (>= largest block size in the launch)
  int32_t sys_offset;     // added to the item's system index (adjoint twin records)
  int64_t ldf, ldx;       // series: right-hand side blockIdx.y starts at F + y ldf, its solution at x + y ldx
  int64_t win0;           // single system: the launch's windows are win0 + [0, gridDim.x)
  int32_t reg_path;       // F and x are device memory: windows of the register path's shape may take it
                          // (2: also those with a shorter last block)
};

// shared memory bytes for a window kernel of width NT and n_smem rows
__host__ __device__ inline size_t window_smem_bytes(int NT, int n_smem) {
  const size_t nw = (size_t)(NT / 32);
  return sizeof(double) * ((size_t)n_smem * (size_t)(NT + 1) + 4 * (size_t)n_smem + 4 * (size_t)NT + 4 * nw + 8);
}

__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// 2^k as a double for |k| <= 1000 (bit construction)
__device__ __forceinline__ double pow2i(int k) { return __hiloint2double((1023 + k) << 20, 0); }

// a warp's three sums: lanes 0-7 return the sum of x, 8-15 that of y, 16-23 that of z (6 additions
// instead of the 15 of three shuffle trees)
__device__ __forceinline__ double warp_sum3(double x, double y, double z, int lane) {
  const bool up = lane & 16, odd = lane & 8;
  double k0 = up ? z : x, k1 = up ? 0.0 : y;
  k0 += __shfl_xor_sync(0xffffffffu, up ? x : z, 16);
  k1 += __shfl_xor_sync(0xffffffffu, up ? y : 0.0, 16);
  double v = (odd ? k1 : k0) + __shfl_xor_sync(0xffffffffu, odd ? k0 : k1, 8);
#pragma unroll
  for (int d = 4; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// barrier over the first NT threads of a CTA of NTF threads
template <int NT, int NTF = NT>
__device__ __forceinline__ void sync_first() {
  if constexpr (NTF == NT)
    __syncthreads();
  else
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}

// The dichotomy tree of one FP64 window (a2): eq. 15 as two affine scans over the window's blocks
// (prefix maps A -> a A + b beta^R left to right, suffix maps B -> c B + d beta^L right to left),
// five warp-shuffle levels and one shared-memory level, then the first/last values of every
// block (eq. 18) in sxs/sxe and the neighbours' values each block needs: XL = x_{s-1}, XR = x_{e+1}.
// bc: the block's coefficient record; zero coupling enters at both window ends.
template <int NT, int NTF = NT>
__device__ __forceinline__ void tree_f64(const double* bc, bool act, double bL, double bR, int64_t mb, int64_t P,
                                         int nwin, int tid, double* swa, double* sxs, double* sxe, double& XL,
                                         double& XR) {
  constexpr int NW = NT / 32;
  const int lane = tid & 31, wid = tid >> 5;
  double pa = act ? bc[BC_A] : 1.0;
  double pb = act ? bc[BC_B] * bR : 0.0;
  double qa = act ? bc[BC_C] : 1.0;
  double qb = act ? bc[BC_D] * bL : 0.0;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const double ya = __shfl_up_sync(0xffffffffu, pa, d), yb = __shfl_up_sync(0xffffffffu, pb, d);
    const double za = __shfl_down_sync(0xffffffffu, qa, d), zb = __shfl_down_sync(0xffffffffu, qb, d);
    if (lane >= d) {
      pb = fma(pa, yb, pb);
      pa = pa * ya;
    }
    if (lane + d < 32) {
      qb = fma(qa, zb, qb);
      qa = qa * za;
    }
  }
  if (lane == 31) {
    swa[wid] = pa;
    swa[NW + wid] = pb;
  }
  if (lane == 0) {
    swa[2 * NW + wid] = qa;
    swa[3 * NW + wid] = qb;
  }
  // previous lane's inclusive prefix, next lane's inclusive suffix
  double ea = __shfl_up_sync(0xffffffffu, pa, 1), eb = __shfl_up_sync(0xffffffffu, pb, 1);
  double fa = __shfl_down_sync(0xffffffffu, qa, 1), fb = __shfl_down_sync(0xffffffffu, qb, 1);
  if (lane == 0) {
    ea = 1.0;
    eb = 0.0;
  }
  if (lane == 31) {
    fa = 1.0;
    fb = 0.0;
  }
  sync_first<NT, NTF>();
  double Aw = 0.0, Bw = 0.0;  // zero coupling enters at both window ends
  for (int w = 0; w < wid; ++w) Aw = fma(swa[w], Aw, swa[NW + w]);
  for (int w = NW - 1; w > wid; --w) Bw = fma(swa[2 * NW + w], Bw, swa[3 * NW + w]);
  const double Am = fma(ea, Aw, eb);
  const double Bm = fma(fa, Bw, fb);
  sxs[tid] = fma(bc[BC_TL], Bm, bL) + Am;            // x_s (eq. 18)
  sxe[tid] = fma(bc[BC_TR], Am, bR + Bm);            // x_e
  sync_first<NT, NTF>();
  if (act) {
    if (!(mb == 0 || tid == 0)) XL = sxe[tid - 1];
    if (!(mb == P - 1 || tid + 1 >= nwin)) XR = sxs[tid + 1];
  }
}

// the window of a CTA: own blocks [m0, m0 + nown) of system `pp`, hl / hr halo blocks
struct Window {
  const SysPlan* pp;
  int64_t m0;
  int nown, hl, hr;
};
__device__ __forceinline__ Window window_of(const WinArgs& A) {
  Window w;
  int sys = 0;
  w.m0 = 0;
  w.nown = 0;
  if (A.items) {
    const Item it = A.items[blockIdx.x];
    sys = it.sys;
    w.m0 = it.m0;
    w.nown = it.n_own;
  }
  sys += A.sys_offset;
  w.pp = A.plans + sys;
  const int64_t P = w.pp->P;
  if (!A.items) {
    w.nown = w.pp->own;
    w.m0 = ((int64_t)blockIdx.x + A.win0) * w.nown;
    if (w.m0 + w.nown > P) w.nown = (int)(P - w.m0);
  }
  w.hl = w.hr = 0;
  if (A.mode == MODE_FULL) {
    w.hl = (int)min((int64_t)w.pp->hl, w.m0);
    w.hr = (int)min((int64_t)w.pp->hr, P - w.m0 - w.nown);
  }
  return w;
}

}  // namespace dich
