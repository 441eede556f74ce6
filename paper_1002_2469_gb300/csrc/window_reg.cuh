// window_reg.cuh -- the register-resident path of the MIXED window kernel (16-row blocks).
//
// A window of 16-row blocks (forward: the system's last block may be shorter) whose launch asks for the
// full solve (MODE_FULL) is solved with a thread's pair of blocks (2 x 16 unknowns) kept in registers
// from the load to the store:
//   - the window's rows of F arrive by 16-byte cp.async copies (8-byte ones where F is not 16-byte
//     aligned), consecutive threads copying consecutive elements, into shared-memory slots of 272
//     bytes, one per thread (its two blocks, 256 contiguous bytes, plus 16 bytes of padding, so that
//     the per-thread 16-byte reads of eight consecutive threads fall in eight different bank groups);
//   - the exponent range of the window (its power-of-two scale), the split into float-float, the
//     two constant-coefficient recurrences (a1), the block-end quantities, beta (eq. 16) and the
//     dichotomy tree (a2, shared with the shared-memory path), the spike correction of eq. 7 (a3)
//     and the join back to FP64 all work on registers: no shared-memory round trip per row;
//   - the output scale g = -1/q is folded into the join: the backward recurrence leaves X with
//     x = g X, the spike correction works in units of X (its coefficients times 1/g = -q), and each
//     output is one FP64 FMA, g * hi + (g * lo), with the window scale undone in the exponent bits;
//   - the solution goes back through the same shared-memory slots, and the window's own (non-halo)
//     rows leave with coalesced stores.
// Windows of any other shape and the general path's passes take the shared-memory path of
// window_mixed.cuh.  Included by window_mixed.cuh after the tree (tree2, Recs2).
#pragma once
#include <type_traits>
#include "ff.cuh"
#include "slots.cuh"
#include "window.cuh"

namespace dich {

struct Recs2;

// the middle record's float-float entries a window copies to shared memory at its start (the
// per-system tables of a batch are then read once per CTA, not at first touch inside the tree): the
// block-coefficient record, the four beta coefficients and the 66 pair-map powers
constexpr int kMidRec = 0, kMidK = 10, kMidPow = 14, kMidEntries = 80;

// shared memory of the register path for NT threads: the pair slots, the two spike tables (and those of
// the thread that holds a shorter last block), the
// warp-boundary first/last values, the scan scratch, the exponent maxima (of the right-hand side
// and, for the adjoint, of the forward solution) and the middle record's entries
__host__ __device__ inline size_t window_reg_smem_bytes(int NT) {
  const size_t nw = (size_t)(NT / 32);
  return (size_t)NT * kRegPairBytes + 4 * 16 * (size_t)kRegRows + 8 * 2 * nw + 8 * 4 * nw + 4 * 4 * nw +
         8 * (size_t)kMidEntries;
}

// a float's bits rebuilt as an FP64 bit pattern with the exponent rebias k (fast windows, ff.cuh)
__device__ __forceinline__ double f32_as_f64(float f, unsigned k) {
  const unsigned b = __float_as_uint(f);
  return __hiloint2double((int)((((unsigned)((int)b >> 3)) & 0x8FFFFFFFu) + k), (int)(b << 29));
}
// the same without the rebias: exactly f * 2^-896 (zeros and subnormal floats included)
__device__ __forceinline__ double f32_as_f64_unbiased(float f) {
  const unsigned b = __float_as_uint(f);
  return __hiloint2double((int)(((unsigned)((int)b >> 3)) & 0x8FFFFFFFu), (int)(b << 29));
}

// The dichotomy tree (a2) of a window whose blocks all carry the middle record -- every block at
// least kl blocks from the system's start and kr from its end, where the ratios of eq. 15-18 are the
// same constants for every block (the Toeplitz saving of Sec. 3.1).  Same scans and first/last
// values as tree2, with uniform coefficients: a thread's pair of blocks composes to the prefix map
// A -> a^2 A + b (a beta^R_0 + beta^R_1) and the suffix map B -> c^2 B + d (c beta^L_1 + beta^L_0),
// level d of the warp scans multiplies by (a^2)^d, (c^2)^d from the plan's power table ((a^2)^t then
// (c^2)^t, t = 0..32, staged in shared memory with the record), and only the plan's `lev` levels run.  A warp's totals enter the
// following warps through (a^2)^32 (prefix) and (c^2)^32 (suffix); lane t of a warp receives the
// prefix of the warps before it times (a^2)^t and the suffix of the warps after it times (c^2)^(31-t).
template <int NT>
__device__ __forceinline__ void tree_mid(const float2* tf, int rm, int pw, const SysPlan* pp, int nwin, int tid,
                                         const ff2& bL, const ff2& bR, ffv* swv, ffv* sbd, ffv& XL0, ffv& XR0,
                                         ffv& XL1, ffv& XR1) {
  // tf + rm: the middle block-coefficient record, tf + pw: the pair-map powers
  constexpr int NW = NT / 32;
  const int lane = tid & 31, wid = tid >> 5;
  const int b0 = 2 * tid, b1 = b0 + 1;
  auto ld = [&](int at) { return ff_of(tf[at]); };
  const ffv a = ld(rm + BC_A), b = ld(rm + BC_B), c = ld(rm + BC_C), d = ld(rm + BC_D);
  const ff2 ac = ff2_pair(a, c);
  // lane x: the prefix (b beta^R of both blocks), lane y: the suffix (d beta^L of both blocks)
  const ff2 pbv = ff2_mul(ff2_bcast(b), bR), qbv = ff2_mul(ff2_bcast(d), bL);
  // composite maps of the pair: prefix a pb_0 + pb_1, suffix c qb_1 + qb_0
  const ff2 p0 = ff2{make_float2(pbv.h.x, qbv.h.y), make_float2(pbv.l.x, qbv.l.y)};   // (pb_0, qb_1)
  const ff2 p1 = ff2{make_float2(pbv.h.y, qbv.h.x), make_float2(pbv.l.y, qbv.l.x)};   // (pb_1, qb_0)
  ff2 Tv = ff2_fma(ac, p0, p1);
  const int lev = pp->lev;
  const bool cheap = pp->tcheap != 0;
  if (cheap) {
    // every level multiplies by at most 2^-24: the product of the leading parts, added to the low
    // part by one FMA, carries the level's term to within about 2^-46 of the larger of the two
    // values (the two dropped cross products, 2^-48 each, and the FMA's rounding); one
    // renormalisation after the levels
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      if (k >= lev) break;
      const int dd = 1 << k;
      const float2 M = make_float2(tf[pw + dd].x, tf[pw + 33 + dd].x);
      const float yh = __shfl_up_sync(0xffffffffu, Tv.h.x, dd);
      const float zh = __shfl_down_sync(0xffffffffu, Tv.h.y, dd);
      Tv.l = fma2(M, make_float2(lane >= dd ? yh : 0.f, lane + dd < 32 ? zh : 0.f), Tv.l);
    }
    Tv = ff2_renorm(Tv);
  } else {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      if (k >= lev) break;
      const int dd = 1 << k;
      const ff2 M = ff2_pair(ld(pw + dd), ld(pw + 33 + dd));
      const float yh = __shfl_up_sync(0xffffffffu, Tv.h.x, dd), yl = __shfl_up_sync(0xffffffffu, Tv.l.x, dd);
      const float zh = __shfl_down_sync(0xffffffffu, Tv.h.y, dd), zl = __shfl_down_sync(0xffffffffu, Tv.l.y, dd);
      const bool up = lane >= dd, dn = lane + dd < 32;
      const ff2 Y{make_float2(up ? yh : 0.f, dn ? zh : 0.f), make_float2(up ? yl : 0.f, dn ? zl : 0.f)};
      Tv = ff2_fma(M, Y, Tv);
    }
  }
  if (lane == 31) swv[wid] = ff2_x(Tv);
  if (lane == 0) swv[NW + wid] = ff2_y(Tv);
  // inclusive values of the neighbouring lanes (the prefix entering the pair, the suffix beyond it)
  float eh = __shfl_up_sync(0xffffffffu, Tv.h.x, 1), el = __shfl_up_sync(0xffffffffu, Tv.l.x, 1);
  float fh = __shfl_down_sync(0xffffffffu, Tv.h.y, 1), fl = __shfl_down_sync(0xffffffffu, Tv.l.y, 1);
  if (lane == 0) eh = el = 0.f;
  if (lane == 31) fh = fl = 0.f;
  __syncthreads();
  ffv Aw = ff_zero(), Bw = ff_zero();   // zero coupling enters at both window ends
  const ffv a32 = ld(pw + 32), c32 = ld(pw + 33 + 32);
  if (lev < 5) {   // couplings reach fewer than 2^(lev+1) <= 32 blocks: only the neighbouring warps'
    if (wid > 0) Aw = swv[wid - 1];
    if (wid < NW - 1) Bw = swv[NW + wid + 1];
  } else {
    for (int w = 0; w < wid; ++w) Aw = ff_fma(a32, Aw, swv[w]);
    for (int w = NW - 1; w > wid; --w) Bw = ff_fma(c32, Bw, swv[NW + w]);
  }
  ff2 E;
  if (cheap) {
    // lane 0 of the prefix and lane 31 of the suffix take the other warps' value with factor 1 and
    // no neighbour value: exactly (Aw, Bw); every other lane's factor is at most 2^-24
    const float mx = tf[pw + lane].x, my = tf[pw + 33 + (31 - lane)].x;
    E = ff2_renorm(ff2{make_float2(lane == 0 ? Aw.h : eh, lane == 31 ? Bw.h : fh),
                       make_float2(lane == 0 ? Aw.l : __fmaf_rn(mx, Aw.h, el),
                                   lane == 31 ? Bw.l : __fmaf_rn(my, Bw.h, fl))});
  } else {
    E = ff2_fma(ff2_pair(ld(pw + lane), ld(pw + 33 + (31 - lane))), ff2_pair(Aw, Bw),
                ff2{make_float2(eh, fh), make_float2(el, fl)});
  }
  // (A entering block 1, B beyond block 0)
  const ff2 G = ff2_fma(ac, E, p0);
  const ff2 Av{make_float2(E.h.x, G.h.x), make_float2(E.l.x, G.l.x)};   // (A_0, A_1)
  const ff2 Bv{make_float2(G.h.y, E.h.y), make_float2(G.l.y, E.l.y)};   // (B_0, B_1)
  // first/last values of both blocks (eq. 18)
  const ff2 xs = ff2_add(ff2_fma(ff2_bcast(ld(rm + BC_TL)), Bv, bL), Av);
  const ff2 xe = ff2_fma(ff2_bcast(ld(rm + BC_TR)), Av, ff2_add(bR, Bv));
  ffv xe_prev, xs_next;
  pair_neighbours<NT>(xs, xe, tid, sbd, xe_prev, xs_next);
  if (b0 > 0) XL0 = xe_prev;
  XR0 = ff2_y(xs);
  XL1 = ff2_x(xe);
  if (b1 + 1 < nwin) XR1 = xs_next;
}

// a CTA's place among the gradient partials: its window's index (single systems run the last window
// first), or its item's
__device__ __forceinline__ unsigned part_of(const WinArgs& A) {
  return A.items ? blockIdx.x : gridDim.x - 1 - blockIdx.x;
}

// ADJ: the adjoint (a5) -- A.F is w, the plan the transposed one, A.x receives lambda, and the
// gradient sums -(sum lambda_r x_{r-1}, sum lambda_r x_r, sum lambda_r x_{r+1}) over the window's own
// rows go to A.part (three per CTA).  The forward solution x (A.xf) comes into the pair slots by a
// second copy as soon as w has moved to registers, and is read back row by row as lambda is
// written over it.
template <int NT, bool ADJ, bool RAGK>
__device__ __forceinline__ void window_reg(const WinArgs& A, const SysPlan* pp, const double* tab, int64_t P,
                                           int64_t wlo, int nwin, int hl, int nown, int64_t row_lo, int len,
                                           unsigned char* smem) {
  constexpr int NW = NT / 32;
  constexpr int R = kRegRows;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  unsigned char* mine = smem + (size_t)tid * kRegPairBytes;
  float4* tv4 = reinterpret_cast<float4*>(smem + (size_t)NT * kRegPairBytes);   // spikes, both lanes
  float4* tw4 = tv4 + R;
  float4* rv4 = tw4 + R;                                                         // the shorter last block's thread
  float4* rw4 = rv4 + R;
  ffv* sbd = reinterpret_cast<ffv*>(rw4 + R);                                   // 2 NW warp-boundary values
  ffv* swv = sbd + 2 * NW;                                                       // 4 NW scan scratch
  unsigned* sexp = reinterpret_cast<unsigned*>(swv + 4 * NW);                    // 2 NW exponent maxima
  unsigned* sexpx = sexp + 2 * NW;                                               // the same for x
  float2* mt = reinterpret_cast<float2*>(sexpx + 2 * NW);                        // middle record entries

  const int b0 = 2 * tid, b1 = b0 + 1;
  const bool act0 = b0 < nwin, act1 = b1 < nwin;
  const int64_t mb0 = wlo + b0, mb1 = wlo + b1;
  const bool last0 = act0 && (mb0 == P - 1), last1 = act1 && (mb1 == P - 1);
  const double* src = A.F + (int64_t)blockIdx.y * A.ldf + pp->off + row_lo;
  double* dst = A.x + (int64_t)blockIdx.y * A.ldx + pp->off + row_lo;

  const bool al_src = (reinterpret_cast<uintptr_t>(src) & 15u) == 0u, al_dst = (reinterpret_cast<uintptr_t>(dst) & 15u) == 0u;
  // ---------------------------------------------------------------- F -> the pair slots (async)
  slots_load(smem, src, len, al_src, lane, wid);
  if constexpr (!ADJ) {   // (the adjoint, at four CTAs per SM, reads them from the tables: measured faster)
    const float2* tf = reinterpret_cast<const float2*>(tab);
    for (int i = tid; i < kMidEntries; i += NT) {
      const int64_t at = (i < kMidK) ? pp->o_bcmf + i : (i < kMidPow ? pp->o_kmf + (i - kMidK) : pp->o_midf + (i - kMidPow));
      mt[i] = tf[at];
    }
  }
  if (tid < R) {   // spike tables with both lanes filled and zeros past the truncation lengths
    const float2* tf = reinterpret_cast<const float2*>(tab);
    const float2 v = (tid < pp->Lv) ? tf[pp->o_vf + tid] : make_float2(0.f, 0.f);
    const float2 w = (tid < pp->Lw) ? tf[pp->o_wf + tid] : make_float2(0.f, 0.f);
    tv4[tid] = make_float4(v.x, v.x, v.y, v.y);
    tw4[tid] = make_float4(w.x, w.x, w.y, w.y);
  }
  // RAGK: a last block of fewer rows (forward only): its thread takes spike tables of its own, the last block's
  // spikes in that block's lane (zero past its rows) beside the full blocks' in the other
  const bool rag = RAGK && len < nwin * R;
  const int nl = R - (nwin * R - len);                 // the last block's rows
  const bool ragt = rag && (last0 || last1);           // this thread holds it
  if (rag && tid < R) {
    const float2* tf = reinterpret_cast<const float2*>(tab);
    const bool lastx = (nwin & 1) != 0;                // its lane
    const float2 v = (tid < pp->Lv) ? tf[pp->o_vf + tid] : make_float2(0.f, 0.f);
    const float2 w = (tid < pp->Lw) ? tf[pp->o_wf + tid] : make_float2(0.f, 0.f);
    // row R - 1 - tid of the block (rw4's index): nl - 1 - row from its end
    const float2 vl = (tid < nl) ? tf[pp->o_vlf + tid] : make_float2(0.f, 0.f);
    const int back = nl - 1 - (R - 1 - tid);
    const float2 wl = (back >= 0) ? tf[pp->o_wlf + back] : make_float2(0.f, 0.f);
    rv4[tid] = lastx ? make_float4(vl.x, v.x, vl.y, v.y) : make_float4(v.x, vl.x, v.y, vl.y);
    rw4[tid] = lastx ? make_float4(wl.x, w.x, wl.y, w.y) : make_float4(w.x, wl.x, w.y, wl.y);
  }
  cp_async_wait_all();
  __syncwarp();   // (the tables staged above are read after the exponent range's barrier)
  if (rag && ragt) {   // rows past the system's end: a value of the block (for the exponent range), zeroed below
    double* col = reinterpret_cast<double*>(mine + (last1 ? 8 * R : 0));
    for (int i = nl; i < R; ++i) col[i] = col[0];
  }

  // ---------------------------------------------------------------- the pair in registers
  // a[k] = rows 2k, 2k+1 of block 2t; b[k] the same of block 2t+1.  The slot part of an inactive
  // block (past the window's end) holds stale values: they are read without a branch, kept out of
  // the exponent range below, and what they become is never stored (the tree takes zero block
  // values for inactive blocks)
  double2 a[R / 2], b[R / 2];
#pragma unroll
  for (int k = 0; k < R / 2; ++k) {
    a[k] = *reinterpret_cast<const double2*>(mine + 16 * k);
    b[k] = *reinterpret_cast<const double2*>(mine + 8 * R + 16 * k);
  }

  // window scale (largest |F| near 2^16, an exact power of two) and the fast criterion: the
  // largest and smallest FP64 high words with the sign cleared, over the active blocks
  int wscale;
  bool fast, flush;   // flush: fast conversions with the window's far-smaller values set to zero
  unsigned hlo;
  {
    unsigned hmax0 = 0u, hmin0 = 0xFFFFFFFFu, hmax1 = 0u, hmin1 = 0xFFFFFFFFu;
#pragma unroll
    for (int k = 0; k < R / 2; ++k) {
      const unsigned u = (unsigned)__double2hiint(a[k].x) & 0x7FFFFFFFu, v = (unsigned)__double2hiint(a[k].y) & 0x7FFFFFFFu;
      hmax0 = __vimax3_u32(hmax0, u, v);
      hmin0 = __vimin3_u32(hmin0, u, v);
      const unsigned y = (unsigned)__double2hiint(b[k].x) & 0x7FFFFFFFu, z = (unsigned)__double2hiint(b[k].y) & 0x7FFFFFFFu;
      hmax1 = __vimax3_u32(hmax1, y, z);
      hmin1 = __vimin3_u32(hmin1, y, z);
    }
    unsigned hmax = max(act0 ? hmax0 : 0u, act1 ? hmax1 : 0u);
    unsigned hmin = min(act0 ? hmin0 : 0xFFFFFFFFu, act1 ? hmin1 : 0xFFFFFFFFu);
    hmax = __reduce_max_sync(0xffffffffu, hmax);
    hmin = __reduce_min_sync(0xffffffffu, hmin);
    if (lane == 0) {
      sexp[wid] = hmax;
      sexp[NW + wid] = hmin;
    }
    __syncthreads();
    hmax = sexp[0];
    hmin = sexp[NW];
#pragma unroll
    for (int w = 1; w < NW; ++w) {
      hmax = max(hmax, sexp[w]);
      hmin = min(hmin, sexp[NW + w]);
    }
    const int emax = (int)(hmax >> 20), emin = (int)(hmin >> 20);
    wscale = (emax == 2047) ? 0 : ((emax == 0) ? 1000 : max(-1000, min(1000, (1023 + 16) - emax)));
    fast = (emin >= 1) && (emax >= 239) && (emax <= 1935) && (emax - emin <= 119);
    flush = !fast && (emax >= 239) && (emax <= 1935);
    hlo = (unsigned)(emax - 119) << 20;
  }
  if constexpr (ADJ) {
    // every thread's slot is in its registers (the barrier of the exponent range): the slots now take
    // the forward solution x
    const double* xsrc = A.xf + pp->off + row_lo;
    slots_load(smem, xsrc, nwin * R, (reinterpret_cast<uintptr_t>(xsrc) & 15u) == 0u, lane, wid);
  }

  // fast windows: the FP64 multiplier of the join, G = g 2^(896 - wscale), folds the rebias of the
  // leading part into the FMA when its exponent stays in range (|F| up to about 2^80 at |g| <= 2^60)
  const int ghw = __double2hiint(pp->g);
  const bool gfold = ((ghw >> 20) & 0x7FF) + 896 - wscale <= 2046;
  const double G = __hiloint2double((int)((unsigned)ghw + ((unsigned)(896 - wscale) << 20)), __double2loint(pp->g));
  auto body = [&](auto fast_, auto gfold_, auto flush_, auto rag_) {
    constexpr bool RAG = decltype(rag_)::value;   // the window holds a shorter last block
    constexpr bool FAST = decltype(fast_)::value;
    constexpr bool GFOLD = decltype(gfold_)::value;
    constexpr bool FLUSH = decltype(flush_)::value;
    const FastK fk = fast_k(wscale);
    float2 H[R], L[R];   // (block 2t, block 2t+1) of row i: hi and lo parts
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const double d0 = (i & 1) ? a[i / 2].y : a[i / 2].x;
      const double d1 = (i & 1) ? b[i / 2].y : b[i / 2].x;
      if (FAST && FLUSH) {
        split_fast_flush(d0, fk, hlo, H[i].x, L[i].x);
        split_fast_flush(d1, fk, hlo, H[i].y, L[i].y);
      } else if (FAST) {
        split_fast(d0, fk, H[i].x, L[i].x);
        split_fast(d1, fk, H[i].y, L[i].y);
      } else {
        split_sc(d0, wscale, H[i].x, L[i].x);
        split_sc(d1, wscale, H[i].y, L[i].y);
      }
    }

    // ------------------------------------------------------------ local recurrences (a1)
    {  // u_i = f_i + rs u_{i-1}, u_{-1} = 0
      const float2 rh = f2(pp->rs_h), rl = f2(pp->rs_l);
      float2 uh = f2(0.f), ul = f2(0.f);
#pragma unroll
      for (int i = 0; i < R; ++i) {
        ff_axpy2(H[i], L[i], rh, rl, uh, ul, uh, ul);
        H[i] = uh;
        L[i] = ul;
      }
    }
    if (RAG && ragt) {   // past the system's end u = 0, so that X = 0 reaches its last row
#pragma unroll
      for (int i = 0; i < R; ++i) {
        if (last0 && i >= nl) H[i].x = L[i].x = 0.f;
        if (last1 && i >= nl) H[i].y = L[i].y = 0.f;
      }
    }
    {  // X_i = u_i + ib X_{i+1}, X_R = 0   (the particular solution is xp = g X)
      const float2 bh = f2(pp->ib_h), bl = f2(pp->ib_l);
      float2 xh = f2(0.f), xl = f2(0.f);
#pragma unroll
      for (int i = R - 1; i >= 0; --i) {
        ff_axpy2(H[i], L[i], bh, bl, xh, xl, xh, xl);
        H[i] = xh;
        L[i] = xl;
      }
    }

    // ------------------------------------------------------------ beta (eq. 16), tree (a2)
    // in units of X (x = g X; the maps of eq. 15 are linear, so the tree runs in any unit):
    // beta^L / g = K1 X_0 + K2 X_{n-1}, beta^R / g = K3 X_0 + K4 X_{n-1} (the block's beta record: the
    // 2x2 map M of eq. 16 applied to alpha / g = X_0 - ib v_0 X_0, omega / g = X_{n-1} - ib v_{n-1} X_0)
    const ff2 zero2{f2(0.f), f2(0.f)};
    const ff2 X0 = ff2_make(H[0], L[0]);
    float2 Xeh = H[R - 1], Xel = L[R - 1];
    if (RAG && ragt) {
#pragma unroll
      for (int i = 0; i < R; ++i)
        if (i == nl - 1) {
          if (last0) {
            Xeh.x = H[i].x;
            Xel.x = L[i].x;
          } else {
            Xeh.y = H[i].y;
            Xel.y = L[i].y;
          }
        }
    }
    const ff2 Xe = ff2_make(Xeh, Xel);
    // forward solve: the slot is idle until the output, so the 64 data registers wait there while
    // the tree runs.  Layout: the packed hi pair of row i (both blocks) at 8 i, the lo pair at
    // 8 R + 8 i, as the packed instructions take them; the output rows 2k, 2k+1 of block 2t go to
    // 16 k and those of block 2t+1 to 8 R + 16 k, the places of the pairs of rows 2k, 2k+1, which
    // are read back just before.
    if constexpr (!ADJ) {
#pragma unroll
      for (int k = 0; k < R / 2; ++k) {
        *reinterpret_cast<float4*>(mine + 16 * k) = make_float4(H[2 * k].x, H[2 * k].y, H[2 * k + 1].x, H[2 * k + 1].y);
        *reinterpret_cast<float4*>(mine + 8 * R + 16 * k) = make_float4(L[2 * k].x, L[2 * k].y, L[2 * k + 1].x, L[2 * k + 1].y);
      }
    }
    const float2* tf = reinterpret_cast<const float2*>(tab);
    // every block of the window carries the middle record: uniform coefficients (tree_mid)
    const bool mid = (nwin == 2 * NT) && (wlo >= pp->kl) && (wlo + nwin <= P - pp->kr);
    ff2 bL, bR;
    ffv XL0 = ff_zero(), XR0 = ff_zero(), XL1 = ff_zero(), XR1 = ff_zero();
    if (mid) {
      // the middle record's entries: staged in shared memory (forward) or in the plan's tables (adjoint)
      const float2* me = ADJ ? tf : mt;
      const int rm = ADJ ? pp->o_bcmf : kMidRec, pw = ADJ ? pp->o_midf : kMidPow, km = ADJ ? pp->o_kmf : kMidK;
      const ffv k1 = ff_of(me[km]), k2 = ff_of(me[km + 1]), k3 = ff_of(me[km + 2]), k4 = ff_of(me[km + 3]);
      bL = ff2_fma(ff2_bcast(k2), Xe, ff2_mul(ff2_bcast(k1), X0));
      bR = ff2_fma(ff2_bcast(k4), Xe, ff2_mul(ff2_bcast(k3), X0));
      tree_mid<NT>(me, rm, pw, pp, nwin, tid, bL, bR, swv, sbd, XL0, XR0, XL1, XR1);
    } else {
      const Recs2 bc2 = recs2(pp, tab, P, act0, act1, mb0, mb1);
      bL = ff2_sel(act0, act1, ff2_fma(bc2.k(1), Xe, ff2_mul(bc2.k(0), X0)), zero2);
      bR = ff2_sel(act0, act1, ff2_fma(bc2.k(3), Xe, ff2_mul(bc2.k(2), X0)), zero2);
      tree2<NT>(bc2, act0, act1, mb0, mb1, P, nwin, tid, bL, bR, swv, sbd, XL0, XR0, XL1, XR1, pp->lev);
    }

    // the next kernel of the stream may begin its launch (it waits for this grid to complete)
    asm volatile("griddepcontrol.launch_dependents;");

    // ------------------------------------------------------------ correction (a3), join, store
    const bool own0 = act0 && b0 >= hl && b0 < hl + nown;
    const bool own1 = act1 && b1 >= hl && b1 < hl + nown;
    const bool anyown = own0 || own1;
    // x = xp + (x_{s-1} - xp(-1)) v + x_{e+1} w, in units of X (x = g X; the tree's first/last values
    // are in those units already): the coefficients are X_{s-1} - ib X_0 and X_{e+1}
    const ff2 ibx = ff2_mul(ff2_bcast(ffv{pp->ib_h, pp->ib_l}), X0);
    const ff2 cL = ff2_sub(ff2_pair(XL0, XL1), ibx);
    const ff2 cR = ff2_pair(XR0, XR1);
    const float2 gh = f2(pp->g_h), glo = f2(pp->g_l);
    const double gd = pp->g;
    const float4* sv4 = (RAG && ragt) ? rv4 : tv4;
    const float4* sw4 = (RAG && ragt) ? rw4 : tw4;

    // the adjoint: x in the slots, its own power-of-two scale, the neighbours' boundary rows
    int xsc = 0;
    bool xfast = false;
    double xlb = 0.0, xrb = 0.0;
    if constexpr (ADJ) {
      cp_async_wait_all();
      __syncthreads();
      unsigned hmax = 0u, hmin = 0xFFFFFFFFu;
#pragma unroll
      for (int k = 0; k < R / 2; ++k) {
        if (act0) {
          const uint4 q = *reinterpret_cast<const uint4*>(mine + 16 * k);
          hmax = __vimax3_u32(hmax, q.y & 0x7FFFFFFFu, q.w & 0x7FFFFFFFu);
          hmin = __vimin3_u32(hmin, q.y & 0x7FFFFFFFu, q.w & 0x7FFFFFFFu);
        }
        if (act1) {
          const uint4 q = *reinterpret_cast<const uint4*>(mine + 8 * R + 16 * k);
          hmax = __vimax3_u32(hmax, q.y & 0x7FFFFFFFu, q.w & 0x7FFFFFFFu);
          hmin = __vimin3_u32(hmin, q.y & 0x7FFFFFFFu, q.w & 0x7FFFFFFFu);
        }
      }
      hmax = __reduce_max_sync(0xffffffffu, hmax);
      hmin = __reduce_min_sync(0xffffffffu, hmin);
      if (lane == 0) {
        sexpx[wid] = hmax;
        sexpx[NW + wid] = hmin;
      }
      // rows beyond the window's loaded blocks are the system's ends there (x = 0), or belong to halo
      // blocks, which contribute no sums
      if (act0 && b0 > 0) xlb = *reinterpret_cast<const double*>(mine - kRegPairBytes + 8 * (2 * R - 1));
      if (b1 + 1 < nwin) xrb = *reinterpret_cast<const double*>(mine + kRegPairBytes);
      __syncthreads();   // every thread holds its neighbours' rows before any slot takes lambda
      hmax = sexpx[0];
      hmin = sexpx[NW];
#pragma unroll
      for (int w = 1; w < NW; ++w) {
        hmax = max(hmax, sexpx[w]);
        hmin = min(hmin, sexpx[NW + w]);
      }
      const int emax = (int)(hmax >> 20), emin = (int)(hmin >> 20);
      xsc = (emax == 2047) ? 0 : ((emax == 0) ? 1000 : max(-1000, min(1000, (1023 + 16) - emax)));
      xfast = (emin >= 1) && (emax >= 239) && (emax <= 1935) && (emax - emin <= 119);
    }
    // the store loop in two instantiations: float-float gradient sums (x fast) or FP64 sums, so
    // that neither keeps the other's accumulators live through the unrolled rows
    auto store_loop = [&](auto xf_) {
    constexpr bool XF = decltype(xf_)::value;
    const FastK fkx = fast_k(xsc);
    // the gradient sums of the thread's rows, lane x block 2t, lane y block 2t+1: float-float
    // (units 2^(wscale + xscale) / g) in windows whose x is fast, else FP64
    float2 smh = f2(0.f), sml = f2(0.f), s0h = f2(0.f), s0l = f2(0.f), sph = f2(0.f), spl = f2(0.f);
    double dm0 = 0.0, dm1 = 0.0, d00 = 0.0, d01 = 0.0, dp0 = 0.0, dp1 = 0.0;
    // x rows as float-float pairs (lane x block 2t, lane y block 2t+1).  In a fast x window every value
    // of the active blocks is normal; only the markers of the system's ends (x_{-1} = x_N = 0) can be
    // zero, and Z says where they may occur: they become (0, 0)
    auto xsplit = [&](double u0, double u1, float2& hh, float2& ll, bool Z) {
      split_fast(u0, fkx, hh.x, ll.x);
      split_fast(u1, fkx, hh.y, ll.y);
      if (Z) {
        if ((__double2hiint(u0) & 0x7FF00000) == 0) hh.x = ll.x = 0.f;
        if ((__double2hiint(u1) & 0x7FF00000) == 0) hh.y = ll.y = 0.f;
      }
    };
    float2 xph = f2(0.f), xpl = f2(0.f), xch = f2(0.f), xcl = f2(0.f);   // x_{r-1}, x_r split
    double2 xa{0.0, 0.0}, xb{0.0, 0.0};   // x rows 2k, 2k+1 of both blocks (pair k)
    double x0e = 0.0, x1s = 0.0;          // block 2t's last row, block 2t+1's first row
    double2 xprev{0.0, 0.0};              // x of the row before the current pair, both lanes
    if constexpr (ADJ) {
      if (act0) xa = *reinterpret_cast<const double2*>(mine);
      if (act1) xb = *reinterpret_cast<const double2*>(mine + 8 * R);
      if (act0) x0e = *reinterpret_cast<const double*>(mine + 8 * (R - 1));
      x1s = xb.x;
      xprev = make_double2(xlb, x0e);
      if constexpr (XF) {
        xsplit(xprev.x, xprev.y, xph, xpl, true);
        xsplit(xa.x, xb.x, xch, xcl, false);
      }
    }

    // the forward solve reads its rows back from the slot, so its loop need not be unrolled all the
    // way (half the code: measured 2.8% faster, the instruction cache then missing less); the
    // adjoint's rows are in registers
    constexpr int KUNROLL = ADJ ? R / 2 : 4;
    if (ADJ || anyown)   // forward: the halo's rows are not wanted
#pragma unroll KUNROLL
    for (int k = 0; k < R / 2; ++k) {
      double o0[2], o1[2];
      double2 na{0.0, 0.0}, nb2{0.0, 0.0};   // the next pair (x of rows 2k+2, 2k+3), read before the
      if constexpr (ADJ) {                   // slot's rows 2k, 2k+1 take lambda
        if (k + 1 < R / 2) {
          if (act0) na = *reinterpret_cast<const double2*>(mine + 16 * (k + 1));
          if (act1) nb2 = *reinterpret_cast<const double2*>(mine + 8 * R + 16 * (k + 1));
        }
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int i = 2 * k + j;
        float2 xh, xl;
        if constexpr (ADJ) {
          xh = H[i];
          xl = L[i];
        } else {   // back from the slot (stored before the tree)
          xh = *reinterpret_cast<const float2*>(mine + 8 * i);
          xl = *reinterpret_cast<const float2*>(mine + 8 * R + 8 * i);
        }
        if (anyown) {
          const float4 v = sv4[i], w = sw4[R - 1 - i];
          ff_fma_acc2(cL.h, cL.l, make_float2(v.x, v.y), make_float2(v.z, v.w), xh, xl);
          ff_fma_acc2(cR.h, cR.l, make_float2(w.x, w.y), make_float2(w.z, w.w), xh, xl);
        }
        if (FAST && GFOLD) {
          // x = g (hi + lo) 2^-wscale = G (hi 2^-896) + (g lo) 2^-wscale: both parts rebuilt as FP64
          // bit patterns (the leading one without rebias), one FMA
          const float2 lg = mul2(xl, gh);
          o0[j] = fma(f32_as_f64_unbiased(xh.x), G, f32_as_f64(lg.x, fk.join));
          o1[j] = fma(f32_as_f64_unbiased(xh.y), G, f32_as_f64(lg.y, fk.join));
        } else if (FAST) {
          const float2 lg = mul2(xl, gh);
          o0[j] = fma(f32_as_f64(xh.x, fk.join), gd, f32_as_f64(lg.x, fk.join));
          o1[j] = fma(f32_as_f64(xh.y, fk.join), gd, f32_as_f64(lg.y, fk.join));
        } else {
          float2 yh, yl;
          ff_mul2(gh, glo, xh, xl, yh, yl);
          o0[j] = join_dadd(yh.x, yl.x, wscale);
          o1[j] = join_dadd(yh.y, yl.y, wscale);
        }
        if constexpr (ADJ) {
          // x_{r-1}, x_r, x_{r+1} of row i in both blocks
          const double2 xc = (j == 0) ? make_double2(xa.x, xb.x) : make_double2(xa.y, xb.y);
          double2 xn;
          if (j == 0)
            xn = make_double2(xa.y, xb.y);
          else if (k + 1 < R / 2)
            xn = make_double2(na.x, nb2.x);
          else
            xn = make_double2(x1s, xrb);
          if constexpr (XF) {
            float2 nh, nl;
            xsplit(xn.x, xn.y, nh, nl, i == R - 1);
            ff_fma_acc2(xh, xl, xph, xpl, smh, sml);
            ff_fma_acc2(xh, xl, xch, xcl, s0h, s0l);
            ff_fma_acc2(xh, xl, nh, nl, sph, spl);
            xph = xch;
            xpl = xcl;
            xch = nh;
            xcl = nl;
          } else {
            dm0 = fma(o0[j], xprev.x, dm0);
            dm1 = fma(o1[j], xprev.y, dm1);
            d00 = fma(o0[j], xc.x, d00);
            d01 = fma(o1[j], xc.y, d01);
            dp0 = fma(o0[j], xn.x, dp0);
            dp1 = fma(o1[j], xn.y, dp1);
          }
          xprev = xc;
        }
      }
      if (anyown) {
        *reinterpret_cast<double2*>(mine + 16 * k) = make_double2(o0[0], o0[1]);
        *reinterpret_cast<double2*>(mine + 8 * R + 16 * k) = make_double2(o1[0], o1[1]);
      }
      if constexpr (ADJ) {
        xa = na;
        xb = nb2;
      }
    }
    __syncwarp();   // the warp's rows of x are in its slots
    slots_store(smem, dst, hl * R, min(len, (hl + nown) * R), al_dst, lane, wid);
    if constexpr (ADJ) {
      // the CTA's three sums: the thread's own lanes, the warp, the CTA (fixed order), one join
      __syncthreads();   // the scan scratch takes the per-warp sums
      if constexpr (XF) {
        auto lanes = [&](float2 h, float2 l) {
          const ffv a0 = own0 ? ffv{h.x, l.x} : ff_zero(), a1 = own1 ? ffv{h.y, l.y} : ff_zero();
          return ff_add(a0, a1);
        };
        ffv a3[3] = {lanes(smh, sml), lanes(s0h, s0l), lanes(sph, spl)};
#pragma unroll
        for (int d = 16; d > 0; d >>= 1)
#pragma unroll
          for (int q = 0; q < 3; ++q) a3[q] = ff_add(a3[q], ff_shfl_down(a3[q], d));
        if (lane == 0)
#pragma unroll
          for (int q = 0; q < 3; ++q) swv[q * NW + wid] = a3[q];
        __syncthreads();
        if (tid < 3) {
          ffv sum = ff_zero();
          for (int w = 0; w < NW; ++w) sum = ff_add(sum, swv[tid * NW + w]);
          // lambda = g X 2^-wscale, x = x' 2^-xscale
          A.part[3 * (size_t)part_of(A) + tid] = join_dadd(sum.h, sum.l, xsc) * pow2i(-wscale) * gd;
        }
      } else {
        double a3[3] = {(own0 ? dm0 : 0.0) + (own1 ? dm1 : 0.0), (own0 ? d00 : 0.0) + (own1 ? d01 : 0.0),
                        (own0 ? dp0 : 0.0) + (own1 ? dp1 : 0.0)};
#pragma unroll
        for (int d = 16; d > 0; d >>= 1)
#pragma unroll
          for (int q = 0; q < 3; ++q) a3[q] += __shfl_down_sync(0xffffffffu, a3[q], d);
        double* sred = reinterpret_cast<double*>(swv);
        if (lane == 0)
#pragma unroll
          for (int q = 0; q < 3; ++q) sred[q * NW + wid] = a3[q];
        __syncthreads();
        if (tid < 3) {
          double sum = 0.0;
          for (int w = 0; w < NW; ++w) sum += sred[tid * NW + w];
          A.part[3 * (size_t)part_of(A) + tid] = sum;
        }
      }
    }
    };
    if (!ADJ || xfast)
      store_loop(std::true_type());
    else
      store_loop(std::false_type());
  };
  const std::true_type yes;
  const std::false_type no;
  auto ragged = [&] {   // its own instantiations: the tests on rows would cost the others registers
    if constexpr (RAGK) {
      if (fast && gfold)
        body(yes, yes, no, yes);
      else if (flush && gfold)
        body(yes, yes, yes, yes);
      else
        body(no, no, no, yes);
    }
  };
  if (rag) {
    ragged();
  } else if (fast && gfold) {
    body(yes, yes, no, no);
  } else if (flush && gfold) {
    body(yes, yes, yes, no);
  } else if (fast) {
    body(yes, no, no, no);
  } else {
    body(no, no, no, no);
  }
}

}  // namespace dich
