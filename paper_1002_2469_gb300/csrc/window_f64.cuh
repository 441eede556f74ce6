// window_f64.cuh -- the FP64 form's window kernel: one window per CTA, in 64-bit fixed point where its
// values suit it (window_fix.cuh), else in FP64 (window.cuh).
//
// NT: the plan's window width in blocks (threads of the FP64 sweeps).  NTF: threads of the CTA, 32 rows
// each in the fixed-point form, at least NT; 0 (NT threads) for launches without that form: fix_threads
// gives 0, the general path's passes, plans without a fixed-point table.
#pragma once
#include "window_fix.cuh"

namespace dich {

template <int NT, int NTF>
__global__ void __launch_bounds__(NTF ? NTF : NT, NTF ? 768 / (NTF ? NTF : NT) : 0) k_window(const WinArgs A) {
  extern __shared__ __align__(16) double sm[];
  // launched with programmatic stream serialization: this grid may start while the previous
  // kernel of the stream finishes; nothing is read or written before that kernel has completed
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const Window win = window_of(A);
  const SysPlan* pp = win.pp;
  const int64_t P = pp->P, m0 = win.m0;
  const int hl = win.hl, nown = win.nown, hr = win.hr;
  if constexpr (NTF != 0) {
    const int64_t rlo = (m0 - hl) * (int64_t)pp->n;
    const int flen = (int)min((int64_t)(hl + nown + hr) * pp->n, pp->N - rlo);
    if (pp->o_fix != 0 && flen <= kFixRows * NTF) {
      if (window_fix<NTF>(A, pp, A.tabs + pp->tab, rlo, flen, hl * pp->n, min(flen, (hl + nown) * pp->n),
                          reinterpret_cast<unsigned char*>(sm)))
        return;
      __syncthreads();   // every thread is done with the shared memory the FP64 form reuses
    }
  }
  constexpr int NW = NT / 32;
  constexpr int LD = NT + 1;
  constexpr int LT = NTF ? NTF : NT;              // threads that load (after fixed point declined, all of them)
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int ns = A.n_smem;
  double* S = sm;
  double* tv = S + (size_t)ns * LD;
  double* tw = tv + ns;
  double* tvl = tw + ns;
  double* twl = tvl + ns;
  double* sxs = twl + ns;
  double* sxe = sxs + NT;
  double* scl = sxe + NT;
  double* scr = scl + NT;
  double* swa = scr + NT;                         // 4 * NW scan scratch

  const int64_t wlo = m0 - hl;
  const int nwin = hl + nown + hr;
  const int n = pp->n, nlast = pp->nlast;
  const int Lv = pp->Lv, Lw = pp->Lw;
  const int64_t off = pp->off;
  const double* tab = A.tabs + pp->tab;
  const bool has_last = (wlo + nwin == P);
  const int64_t row_lo = wlo * (int64_t)n;                   // first row of the window
  const int len = nwin * n - (has_last ? (n - nlast) : 0);  // rows in the window

  // ---------------------------------------------------------------- F -> smem (transposed, async)
  // (MODE_APPLY: the block solutions y the beta pass left in x, instead of F)
  {
    const double* src = (A.mode == MODE_APPLY) ? (A.x + (int64_t)blockIdx.y * A.ldx + off + row_lo)
                                               : (A.F + (int64_t)blockIdx.y * A.ldf + off + row_lo);
    int b = tid / n, i = tid - (tid / n) * n;
    const int db = LT / n, di = LT - (LT / n) * n;
    for (int j = tid; j < len; j += LT) {
      cp_async8(&S[i * LD + b], src + j);
      i += di;
      b += db;
      if (i >= n) {
        i -= n;
        ++b;
      }
    }
  }
  // tables -> smem (overlaps the copies in flight)
  for (int i = tid; i < Lv; i += LT) tv[i] = tab[pp->o_v + i];
  for (int i = tid; i < Lw; i += LT) tw[i] = tab[pp->o_w + i];
  if (has_last)
    for (int i = tid; i < nlast; i += LT) {
      tvl[i] = tab[pp->o_vl + i];
      twl[i] = tab[pp->o_wl + i];
    }
  cp_async_wait_all();
  __syncthreads();
  if (LT > NT && threadIdx.x >= NT) return;   // the barriers below count the first NT threads

  // ---------------------------------------------------------------- local sweeps (a1)
  const bool act = tid < nwin;
  const int64_t mb = wlo + tid;
  const bool lastb = act && (mb == P - 1);
  const int nbk = lastb ? nlast : n;
  double xm1 = 0.0, alpha = 0.0, omega = 0.0;
  if (act && A.mode == MODE_APPLY) {
    xm1 = pp->ib * S[tid];   // xp(-1) = g ib X_0 = ib y_0
  } else if (act) {
    const double rs = pp->rs, ib = pp->ib, g = pp->g;
    double* col = S + tid;
    double u = 0.0;
    int i = 0;
    for (; i + 4 <= nbk; i += 4) {
      const double f0 = col[(i)*LD], f1 = col[(i + 1) * LD], f2 = col[(i + 2) * LD], f3 = col[(i + 3) * LD];
      const double u0 = fma(rs, u, f0);
      const double u1 = fma(rs, u0, f1);
      const double u2 = fma(rs, u1, f2);
      const double u3 = fma(rs, u2, f3);
      col[(i)*LD] = u0;
      col[(i + 1) * LD] = u1;
      col[(i + 2) * LD] = u2;
      col[(i + 3) * LD] = u3;
      u = u3;
    }
    for (; i < nbk; ++i) {
      u = fma(rs, u, col[i * LD]);
      col[i * LD] = u;
    }
    double X = 0.0;
    i = nbk - 1;
    for (; i - 3 >= 0; i -= 4) {
      const double a0 = col[(i)*LD], a1 = col[(i - 1) * LD], a2 = col[(i - 2) * LD], a3 = col[(i - 3) * LD];
      const double X0 = fma(ib, X, a0);
      const double X1 = fma(ib, X0, a1);
      const double X2 = fma(ib, X1, a2);
      const double X3 = fma(ib, X2, a3);
      col[(i)*LD] = g * X0;
      col[(i - 1) * LD] = g * X1;
      col[(i - 2) * LD] = g * X2;
      col[(i - 3) * LD] = g * X3;
      X = X3;
    }
    for (; i >= 0; --i) {
      X = fma(ib, X, col[i * LD]);
      col[i * LD] = g * X;
    }
    const double v0 = lastb ? pp->v0l : pp->v0;
    const double vend = lastb ? pp->vendl : pp->vend;
    const double xm = g * ib * X;
    xm1 = xm;
    alpha = col[0] - xm * v0;
    omega = col[(nbk - 1) * LD] - xm * vend;
  }

  // ---------------------------------------------------------------- beta (eq. 16)
  int64_t rec = pp->o_bcm;
  if (act) {
    if (mb < pp->kl)
      rec = pp->o_bcl + mb * kBC;
    else if (mb >= P - pp->kr)
      rec = pp->o_bcr + (mb - (P - pp->kr)) * kBC;
  }
  const double* bc = tab + rec;
  const double bL = act ? fma(bc[BC_M00], alpha, bc[BC_M01] * omega) : 0.0;
  const double bR = act ? fma(bc[BC_M10], alpha, bc[BC_M11] * omega) : 0.0;

  if (A.mode == MODE_BETA) {  // general path: beta and the block solutions y leave the window
    if (act) {
      A.beta[2 * (pp->gboff + mb)] = bL;
      A.beta[2 * (pp->gboff + mb) + 1] = bR;
    }
    sync_first<NT, NTF ? NTF : NT>();
    double* dst = A.x + (int64_t)blockIdx.y * A.ldx + off + row_lo;
    int b = tid / n, i = tid - (tid / n) * n;
    const int db = NT / n, di = NT - (NT / n) * n;
    for (int j = tid; j < len; j += NT) {
      dst[j] = S[i * LD + b];
      i += di;
      b += db;
      if (i >= n) {
        i -= n;
        ++b;
      }
    }
    return;
  }

  double XL = 0.0, XR = 0.0;
  if (A.mode == MODE_FULL) {
    tree_f64<NT, NTF ? NTF : NT>(bc, act, bL, bR, mb, P, nwin, tid, swa, sxs, sxe, XL, XR);
  } else {  // MODE_APPLY: first/last values of the neighbours from the global scan
    if (act) {
      XL = (mb == 0) ? 0.0 : A.iface[2 * (pp->gboff + mb - 1) + 1];
      XR = (mb == P - 1) ? 0.0 : A.iface[2 * (pp->gboff + mb + 1)];
    }
  }
  // correction coefficients of the block spikes (a3): x = xp + cL v + cR w
  scl[tid] = XL - xm1;
  scr[tid] = XR;
  sync_first<NT, NTF ? NTF : NT>();

  // the next kernel of the stream may begin its launch (it waits for this grid to complete)
  asm volatile("griddepcontrol.launch_dependents;");
  // ---------------------------------------------------------------- correction + store (a3)
  const bool adj = (A.xf != nullptr);
  double g0 = 0.0, gm = 0.0, gp = 0.0;
  unsigned bad = 0u;
  const int64_t N = pp->N;
  {
    const int jlo = hl * n;
    const int jhi = min(len, (hl + nown) * n);
    double* dst = A.x + (int64_t)blockIdx.y * A.ldx + off + row_lo;
    int b = (jlo + tid) / n, i = (jlo + tid) - ((jlo + tid) / n) * n;
    const int db = NT / n, di = NT - (NT / n) * n;
    for (int j = jlo + tid; j < jhi; j += NT) {
      const bool lb = has_last && (b == nwin - 1);
      const int nb = lb ? nlast : n;
      const int lv = lb ? nlast : Lv, lw = lb ? nlast : Lw;
      const int jr = nb - 1 - i;
      double dv = S[i * LD + b];
      if (i < lv) dv = fma(scl[b], (lb ? tvl : tv)[i], dv);
      if (jr < lw) dv = fma(scr[b], (lb ? twl : tw)[jr], dv);
      __stcs(dst + j, dv);
      if (A.check_finite && !isfinite(dv)) bad = 1u;
      if (adj) {
        const int64_t r = row_lo + j;
        const double* xr = A.xf + off + r;
        g0 = fma(dv, xr[0], g0);
        if (r > 0) gm = fma(dv, xr[-1], gm);
        if (r + 1 < N) gp = fma(dv, xr[1], gp);
      }
      i += di;
      b += db;
      if (i >= n) {
        i -= n;
        ++b;
      }
    }
  }
  if (bad) atomicOr(A.status, (unsigned)ST_NONFINITE);
  if (adj) {
    // CTA sum of the three gradient partials in a fixed order
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      g0 += __shfl_down_sync(0xffffffffu, g0, d);
      gm += __shfl_down_sync(0xffffffffu, gm, d);
      gp += __shfl_down_sync(0xffffffffu, gp, d);
    }
    sync_first<NT, NTF ? NTF : NT>();
    if (lane == 0) {
      swa[wid] = gm;
      swa[NW + wid] = g0;
      swa[2 * NW + wid] = gp;
    }
    sync_first<NT, NTF ? NTF : NT>();
    if (tid < 3) {
      double s = 0.0;
      for (int w = 0; w < NW; ++w) s += swa[tid * NW + w];
      A.part[3 * (size_t)blockIdx.x + tid] = s;
    }
  }
}

}  // namespace dich
