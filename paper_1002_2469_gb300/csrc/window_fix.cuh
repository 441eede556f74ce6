// window_fix.cuh -- FP64-form windows in 64-bit fixed point (32 rows per thread, integer pipes).
//
// What bounds the FP64 form is the FP64 pipe: 2 operations per clock per SM, 64 clocks of latency,
// against five operations per unknown.  In a window whose right-hand side spans a narrow exponent
// range the same recurrences run as 64-bit fixed-point numbers on the integer pipes: a product by a
// constant below 1 is one IMAD.WIDE and two IMAD.HI (9.6 such products per clock per SM measured,
// about 30 clocks of latency), and only the conversions back to FP64 (and half of those from it)
// take the FP64 pipe.  The words carry more bits than FP64 mantissas do, so the results are closer to
// the exact solution than the FP64 recurrences' (rms error 4.7e-17 against 1.2e-16 of the solution's
// rms on the headline system); the path is taken only where that holds (fix_table in api.cu, and
// the window's own tests).
//
// The method, on a window of rows 0..len-1 (T = -q (1 - rs E^-1)(1 - ib E), x = g X):
//   u_i = f_i + rs u_{i-1},   X_i = u_i + ib X_{i+1}.
// With rs, ib of one sign s, s^i u_i and s^i X_i obey the same recurrences with R = |rs|, B = |ib|
// (the right-hand side's and the solution's odd rows change sign).  Words are unsigned: u is held as
// u + a and X as X + 2^63, a = 2^63 (1 - B); then u's word recurrence is W' = (F + K) + R W with
// K = a (1 - R), and X's is Y' = W + B Y': no further constants, every term non-negative, and nothing
// exceeds 64 bits while |F| < 2^hb <= K (|u| <= max|F| / (1 - R), |X| <= max|F| / ((1 - R)(1 - B))).
//   1. every thread runs W over its two 16-row halves from zero words (two independent chains);
//   2. the word entering each thread, Uin, is a scan over the threads with powers R^(32 d) (the
//      window's first row gets u = 0, i.e. the word a), cut where R^(32 d) < 2^-64;
//   3. Y over each half from zero: Y_i = W_i + R^(i+1) Uin + B Y_{i+1};
//   4. Xin, the word beyond each thread, by the mirrored scan (the window's end gets X = 0);
//   5. x_i = g (Y_i + B^(16-i) Xin - 2^63), converted and scaled by the window's power of two.
// The products of steps 2 and 4 add back the unit that fx_mul drops on average (a weak system's
// recurrences would sum it up to hundreds of units); the offset that the rows' products leave is the same
// everywhere and comes off with the output product's constant (FX_KG, fix_table in api.cu).
// The right end of the system (x_N = 0) is step 4 itself.  At its left end step 2's u_{-1} = 0 belongs
// to the system extended to the left with zero right-hand side, whose x_{-1} is g ib X_0; the
// homogeneous solution that removes it is X_i -= X_0 B R^(i+1) (x_{-1} = 0 exactly, up to
// (R B)^(N - i) R^(i+1) <= R^N, below 2^-64 by fix_table in api.cu).
//
// Scale.  Words resolve every row to the same absolute unit, FP64 relative to the values around it.  So a
// window is taken in one power of two for all its words only if no row of its own lies too far below
// that: the level of a row is the largest |F| of the rows around it, each weakened by the decay of the
// coupling over their distance (R per row from the left, B from the right; a lower bound of
// |T^-1| |F| there, which the FP64 recurrences' errors are relative to), and every level has to
// reach 2^-lv of the power of two (random right-hand sides do; FX_LVL, fix_table in api.cu).
// A thread sees its own rows and four on both sides (fix_levels).  Where |F| varies more but smoothly -- from
// one block of 32 rows to the next by at most `step` binades, 4 to 8 and at most half the decay of the couplings
// over a block: the spectra and profiles of smooth sources -- every thread takes the largest exponent of its own
// and its two neighbours' blocks; its levels are held to that, its unit lies at most kFixSlope binades from the
// next thread's, and the scans of steps 2 and 4 move signed words between scales.  (What reaches a thread from
// k + 1 blocks away is then below R^(16 k) <= 2^(-4 k) of its own range: 16/15 into u and again into X, for
// which K has room or a bit is kept, FX_SPARE.)  Anything else (zero stretches, isolated values, Inf and NaN) is
// solved in FP64, which resolves a solution's tails relative to themselves.
// (Such a window pays for the copy and the test on top: 33554467 rows with a zero stretch in every window 456 us,
// in FP64 windows alone 441; 1000003 rows, fewer than two windows an SM, 21.9 and 19.6.)  A window of zeros is its
// own solution: 33554467 zeros 88 us, solved in FP64 454.
//
// Layout: one 272-byte slot per thread (slots.cuh) (F, W, Y and x in turn, in place); loops
// unrolled by two row pairs of both halves.
#pragma once
#include <type_traits>
#include "fixed.cuh"
#include "slots.cuh"

namespace dich {

constexpr int kFixRows = 32;     // rows per thread
constexpr int kFixHalf = 16;
// a plan's fixed-point table (64-bit words, at SysPlan::o_fix): fractions are multiples of 2^-64
enum FixIdx {
  FX_R = 0, FX_B, FX_G,          // R, B, |g| 2^-gk in [1/2, 1)
  FX_K, FX_A, FX_KG,             // K (with the products' mean truncation), a, constant of the output product
  FX_HB, FX_GK, FX_FLAGS,        // hb, gk, FIX_* bits
  FX_LEVR, FX_LEVB,              // scan levels: R^(32 2^lev) (B^...) below 2^-64, at most 5
  FX_STEP,                       // binades neighbouring blocks of a varying window may differ by (0: none)
  FX_DR, FX_DB, FX_LVL,          // decay per row (R, B) and lowest level below the unit, in 1/16 binades
  FX_SPARE,                      // headroom (bits, 0 or 1) of a window of varying scale
  FX_P = 16,                     // R^(i+1), i = 0..15
  FX_Q = FX_P + kFixHalf,        // B^(16-i), i = 0..15
  // powers R^(32 t) = m 2^-64 2^-k with m >= 2^63, t = 0..32 (entry 0 unused): the m, then the k, four
  // 16-bit numbers to a word; and B^(32 t)
  FX_RM = FX_Q + kFixHalf,
  FX_RX = FX_RM + 33,
  FX_BM = FX_RX + 9,
  FX_BX = FX_BM + 33,
  FX_WORDS = FX_BX + 9
};
enum FixFlags { FIX_ALT = 1, FIX_NEG = 2, FIX_GUARD = 4 };   // s = -1; g < 0; high gain (step 4's test)

constexpr int kFixSmemWords = 2 * kFixHalf + 2 * 33;   // tables staged in shared memory
// binades from a thread's unit to the next in a window of varying scale: the words that come from the next
// thread have its unit's errors
constexpr int kFixSlope = 2;
// a high-gain system's window must reach 2^-kFixGuard of the words' bound
constexpr int kFixGuard = 8;

// threads of a CTA that tries the fixed-point form on windows of NT blocks of n rows: 32 rows per thread
// in one of the compiled widths (at least NT, which the FP64 form needs), 0 where it is not used.
// It is used where the window's rows, 32 to a thread, need at least NT threads: blocks of 16 rows and more in
// 64-thread windows, of more than 16 in 128- and 256-thread ones.  Shorter blocks are the planner's (or the
// caller's) choice for systems that cannot fill the chip, where the sweeps' latency counts: there the FP64
// sweeps over them are the shorter chain (113 systems of 4096 rows in 256-thread windows of 16-row blocks,
// beside 3983 MIXED ones: 104.7 us for the batch, 106.2 with this form).
// Windows longer than 8192 rows would exceed 256 threads.
__host__ __device__ inline int fix_threads(int NT, int n) {
  const int64_t rows = (int64_t)NT * n;
  const int w = rows <= 2048 ? 64 : (rows <= 4096 ? 128 : 256);
  return (rows < 1024 || rows > 8192 || w < NT) ? 0 : w;
}

__host__ __device__ inline size_t window_fix_smem_bytes(int NTF) {
  const size_t nw = (size_t)(NTF / 32);
  return (size_t)NTF * kRegPairBytes + 8 * (size_t)kFixSmemWords + 8 * 3 * nw + 16 + 8 * 8 * nw + 4 * 2 * nw + 2 * (size_t)NTF;
}

// s r, s a signed word and r = m 2^-64 2^-x, into a unit 2^(sh - x) times as large (sh >= 0)
__device__ __forceinline__ u64 fx_move(u64 s, u64 m, int sh) {
  const long long z = (long long)fx_mul(s ^ (1ull << 63), m, 1ull - (m >> 1));
  return (u64)(z >> min(sh, 63));
}
// a signed word in a unit 2^sh times as large
__device__ __forceinline__ u64 fx_rescale(u64 s, int sh) {
  return sh >= 0 ? (u64)((long long)s >> min(sh, 63)) : s << -sh;
}

// K + d 2^sc by shifts (fx_from_f64_alu, fixed.cuh) ...
// ... or by the FP64 pipe's conversion (scadd = (sc << 20), plus the sign bit to negate): the two share
// the rows, which balances the pipes (measured 255 G unknowns/s, all-integer 257, all-FP64 225)
__device__ __forceinline__ u64 fx_from_f64_cvt(double d, unsigned scadd, u64 K) {
  return (u64)__double2ll_rn(__hiloint2double((int)((unsigned)__double2hiint(d) + scadd), __double2loint(d))) + K;
}
// a word with the output constant already taken off (two's complement) to FP64; ek: exponent and sign
// to add.  The lowest bit is set so that the exponent addition never meets a zero.
__device__ __forceinline__ double fx_to_f64(u64 z, unsigned ek) {
  const double d = __ll2double_rn((long long)(z | 1ull));
  return __hiloint2double((int)((unsigned)__double2hiint(d) + ek), __double2loint(d));
}

// The largest and the lowest level of a thread's rows (nv of them; lowest: of those whose slot it stores), in
// 1/16 binades: the upper 15 bits of |F|, at most 0.15 binades below the logarithm; dr, db: decays per row,
// edge: lane 0's four rows before the warp's and lane 31's behind them, the nearest first.  Two rows to
// a register (i and 16 + i): the chains over both halves in one instruction.
__device__ __forceinline__ void fix_levels(const unsigned char* mine, int nv, bool own, int dr, int db,
                                           const double* edge, int lane, int& largest, int& lowest) {
  constexpr int H = kFixHalf;
  constexpr unsigned kNone = 0x7FFF7FFFu;
  unsigned h[H], top = 0u, low = kNone;
  if (nv == kFixRows) {
#pragma unroll
    for (int k = 0; k < H / 2; ++k) {
      const uint4 v = *reinterpret_cast<const uint4*>(mine + 16 * k);
      const uint4 w = *reinterpret_cast<const uint4*>(mine + 8 * H + 16 * k);
      h[2 * k] = __byte_perm(v.y, w.y, 0x7632) & kNone;
      h[2 * k + 1] = __byte_perm(v.w, w.w, 0x7632) & kNone;
      top = __vimax3_s16x2(top, h[2 * k], h[2 * k + 1]);
    }
  } else {
    const unsigned* mw = reinterpret_cast<const unsigned*>(mine) + 1;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      h[i] = __byte_perm(i < nv ? mw[2 * i] : 0u, H + i < nv ? mw[2 * (H + i)] : 0u, 0x7632) & kNone;
      top = __vmaxs2(top, h[i]);
    }
  }
  const unsigned mr = __byte_perm(0u - (unsigned)dr, 0u, 0x1010), mb = __byte_perm(0u - (unsigned)db, 0u, 0x1010);
  unsigned l = 0u, r = 0u;   // what the last four rows of each half reach to the right, the first four to the left
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    l = __viaddmax_s16x2(l, mr, h[H - 4 + i]);
    r = __viaddmax_s16x2(r, mb, h[3 - i]);
  }
  unsigned pl = __shfl_up_sync(0xffffffffu, l, 1), pr = __shfl_down_sync(0xffffffffu, r, 1);
  if (lane == 0 || lane == 31) {
    const unsigned* ew = reinterpret_cast<const unsigned*>(edge + (lane ? 4 : 0)) + 1;
    const int d = lane ? db : dr;
    int c = 0;
#pragma unroll
    for (int k = 3; k >= 0; --k) c = __viaddmax_s32(c, -d, (int)((ew[2 * k] & 0x7FFFFFFFu) >> 16));
    if (lane == 0) pl = (unsigned)c << 16;
    if (lane == 31) pr = (unsigned)c;
  }
  l = __byte_perm(pl, l, 0x5432);   // what reaches the halves' first rows from the left
  r = __byte_perm(r, pr, 0x5432);   // and their last rows from the right
#pragma unroll
  for (int i = 0; i < H; ++i) h[i] = l = __viaddmax_s16x2(l, mr, h[i]);
  if (nv == kFixRows) {
#pragma unroll
    for (int i = H - 1; i > 0; i -= 2) {
      const unsigned u = __viaddmax_s16x2(r, mb, h[i]);
      r = __viaddmax_s16x2(u, mb, h[i - 1]);
      low = __vimin3_s16x2(low, u, r);
    }
  } else {
#pragma unroll
    for (int i = H - 1; i >= 0; --i) {   // (past the last row: no value, no level to keep)
      const unsigned live = (i < nv ? 0xFFFFu : 0u) | (H + i < nv ? 0xFFFF0000u : 0u);
      r = __viaddmax_s16x2(r, mb, h[i]) & live;
      low = __vmins2(low, r | (kNone & ~live));
    }
  }
  largest = max(top & 0xFFFFu, top >> 16);
  lowest = own ? min(low & 0xFFFFu, low >> 16) : 0x7FFF;
}

// The window's rows [row_lo, row_lo + len) of a system (own rows [j0, j1) of them), len <= 32 NTF.
// Returns false, with every thread of the CTA past a barrier and nothing stored, where the window's
// values do not suit fixed point: the caller then solves it in FP64.
template <int NTF>
__device__ __forceinline__ bool window_fix(const WinArgs& A, const SysPlan* pp, const double* tab, int64_t row_lo,
                                           int len, int j0, int j1, unsigned char* smem) {
  constexpr int NW = NTF / 32;
  constexpr int H = kFixHalf;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  unsigned char* mine = smem + (size_t)tid * kRegPairBytes;
  u64* tp = reinterpret_cast<u64*>(smem + (size_t)NTF * kRegPairBytes);
  u64* tq = tp + H;
  u64* tR = tq + H;
  u64* tB = tR + 33;
  u64* sw = tB + 33;                                         // 3 NW
  u64* sx0 = sw + 3 * NW;                                    // the system's first row (2 entries)
  double* sedge = reinterpret_cast<double*>(sx0 + 2);        // 8 NW: rows past the warps' edges
  int* sexp = reinterpret_cast<int*>(sedge + 8 * NW);        // 2 NW
  short* sblk = reinterpret_cast<short*>(sexp + 2 * NW);     // NTF: exponents of the threads' blocks
  const u64* fx = reinterpret_cast<const u64*>(tab) + pp->o_fix;
  const double* src = A.F + (int64_t)blockIdx.y * A.ldf + pp->off + row_lo;
  double* dst = A.x + (int64_t)blockIdx.y * A.ldx + pp->off + row_lo;

  slots_load(smem, src, len, (reinterpret_cast<uintptr_t>(src) & 15u) == 0u, lane, wid);
  if (lane < 8) {   // four rows on either side of the warp's, the nearest first
    const int j = lane < 4 ? wid * kWarpRows - 1 - lane : (wid + 1) * kWarpRows + lane - 4;
    if (j >= 0 && j < len)
      cp_async8(sedge + 8 * wid + lane, src + j);
    else
      sedge[8 * wid + lane] = 0.0;
  }
  const short* rx = reinterpret_cast<const short*>(fx + FX_RX);
  const short* bx = reinterpret_cast<const short*>(fx + FX_BX);
  for (int i = tid; i < 2 * kFixHalf; i += NTF) tp[i] = fx[FX_P + i];
  for (int i = tid; i < 33; i += NTF) {   // the powers as plain fractions
    tR[i] = rx[i] > 63 ? 0ull : fx[FX_RM + i] >> rx[i];
    tB[i] = bx[i] > 63 ? 0ull : fx[FX_BM + i] >> bx[i];
  }
  cp_async_wait_all();
  __syncwarp();

  // ---------------------------------------------------------------- the window's exponent range
  const int nv = max(0, min(kFixRows, len - kFixRows * tid));   // the thread's rows
  const bool own = kFixRows * tid < j1 && kFixRows * (tid + 1) > j0;   // it stores some of them
  const int dr = (int)fx[FX_DR], db = (int)fx[FX_DB];
  int hmax, lvl;   // largest and lowest level of the thread's rows
  fix_levels(mine, nv, own, dr, db, sedge + 8 * wid, lane, hmax, lvl);
  const int eown = hmax >> 4;
  sblk[tid] = (short)eown;
  hmax = __reduce_max_sync(0xffffffffu, hmax);
  int lmin = __reduce_min_sync(0xffffffffu, lvl);
  if (lane == 0) {
    sexp[wid] = hmax;
    sexp[NW + wid] = lmin;
  }
  __syncthreads();
  hmax = sexp[0];
  lmin = sexp[NW];
#pragma unroll
  for (int w = 1; w < NW; ++w) {
    hmax = max(hmax, sexp[w]);
    lmin = min(lmin, sexp[NW + w]);
  }
  const int emax = hmax >> 4, lv = (int)fx[FX_LVL], spare = (int)fx[FX_SPARE];
  const int hb = (int)fx[FX_HB];
  const int tlast = (len - 1) / kFixRows;   // the last thread with rows
  if (hmax == 0 && A.xf == nullptr) {   // nothing but zeros (or values near the lower end of the FP64 range)?
    unsigned any = 0u;
    for (int i = 0; i < nv; ++i) {
      const uint2 v = *reinterpret_cast<const uint2*>(mine + 8 * i);
      any |= v.x | (v.y & 0x7FFFFFFFu);
    }
    if (!__syncthreads_or((int)any)) {   // the slots hold the solution
      slots_store(smem, dst, j0, j1, (reinterpret_cast<uintptr_t>(dst) & 15u) == 0u, lane, wid);
      return true;
    }
  }
  // one scale, |F| 2^sc < 2^hb <= K, for a window of normal finite values with sc >= 0 (zeros convert
  // exactly then); else each thread's own
  if (emax < 192 || emax > 1020 + hb) return false;
  const bool var = lmin < ((emax + 1) << 4) - lv;
  int e = emax;
  if (var) {
    const int step = (int)fx[FX_STEP];
    const int el = (tid > 0 && nv > 0) ? sblk[tid - 1] : eown, er = (tid < tlast) ? sblk[tid + 1] : eown;
    const int ell = (tid > 1 && nv > 0) ? sblk[tid - 2] : el, err = (tid + 1 < tlast) ? sblk[tid + 2] : er;
    e = max(eown, max(el, er));
    const bool ok = nv == 0 || (eown >= 192 && abs(eown - el) <= step && abs(eown - er) <= step &&
                                max(ell, err) <= e + kFixSlope && lvl >= ((e + 1 + spare) << 4) - lv);
    if (!__syncthreads_and(step > 0 && ok)) return false;
    sblk[tid] = (short)e;   // (read after the next barrier)
  }
  const int sc = hb - (e - 1022) - (var ? spare : 0);
  const u64 K = fx[FX_K], a0 = fx[FX_A];
  const unsigned flags = (unsigned)fx[FX_FLAGS];
  const unsigned alt = (flags & FIX_ALT) ? 0x80000000u : 0u;

  // ---------------------------------------------------------------- 1. forward words of both halves
  u64 E1 = 0, E2 = 0;
  {
    const unsigned rh = (unsigned)(fx[FX_R] >> 32), rl = (unsigned)fx[FX_R];
    const unsigned sb = 1086u - (unsigned)sc, sodd = ((unsigned)sc << 20) + alt;
#pragma unroll 4
    for (int k = 0; k < H / 2; ++k) {
      const double2 f = *reinterpret_cast<const double2*>(mine + 16 * k);
      const double2 h = *reinterpret_cast<const double2*>(mine + 8 * H + 16 * k);
      ulonglong2 w, v;
      w.x = fx_mul(E1, rh, rl, fx_from_f64_alu(f.x, sb, K));
      v.x = fx_mul(E2, rh, rl, fx_from_f64_alu(h.x, sb, K));
      w.y = fx_mul(w.x, rh, rl, fx_from_f64_cvt(f.y, sodd, K));
      v.y = fx_mul(v.x, rh, rl, fx_from_f64_cvt(h.y, sodd, K));
      E1 = w.y;
      E2 = v.y;
      *reinterpret_cast<ulonglong2*>(mine + 16 * k) = w;
      *reinterpret_cast<ulonglong2*>(mine + 8 * H + 16 * k) = v;
    }
  }
  // ---------------------------------------------------------------- 2. the words entering the threads
  const u64 R16 = tp[H - 1], B16 = tq[0];
  u64 Uin;
  const int levr = (int)fx[FX_LEVR], levb = (int)fx[FX_LEVB];
  if (!var) {
    u64 E = fx_mul(E1, R16, E2 + 1);
    if (tid == 0) E = fx_mul(a0, tR[1], E + 1);
    for (int k = 0; k < levr; ++k) {
      const int d = 1 << k;
      const u64 y = __shfl_up_sync(0xffffffffu, E, d);
      E = fx_mul(lane < d ? 0ull : y, tR[d], E + (lane < d ? 0u : 1u));
    }
    if (lane == 31) sw[wid] = E;
    Uin = __shfl_up_sync(0xffffffffu, E, 1);
    if (lane == 0) Uin = 0;
    __syncthreads();
    if (wid > 0) {
      u64 C = sw[wid - 1];
      if (levr >= 5) {   // couplings may span several warps
        C = sw[0];
        for (int w = 1; w < wid; ++w) C = fx_mul(C, tR[32], sw[w] + 1);
      }
      Uin = (lane == 0) ? C : fx_mul(C, tR[lane], Uin + 1);
    } else if (lane == 0) {
      Uin = a0;
    }
  } else {
    // signed words, each in its thread's unit; R <= 2^-1/4 here, so that 16 blocks away nothing is left
    u64 S = fx_mul(E1, R16, E2 + 1) - (a0 - fx_mul(a0, tR[1], 1ull));
    const int lev = min(4, levr + 1);
    for (int k = 0; k < lev; ++k) {
      const int d = 1 << k;
      const u64 y = __shfl_up_sync(0xffffffffu, S, d);
      const int ey = __shfl_up_sync(0xffffffffu, e, d);
      if (lane >= d) S += fx_move(y, fx[FX_RM + d], rx[d] + e - ey);
    }
    if (lane == 31) sw[wid] = S;
    __syncthreads();
    u64 C = 0;
    int eC = e;
    if (wid > 0) {
      C = sw[wid - 1];
      eC = sblk[32 * wid - 1];
      S += fx_move(C, fx[FX_RM + lane + 1], rx[lane + 1] + e - eC);
    }
    const u64 y = __shfl_up_sync(0xffffffffu, S, 1);
    const int ey = __shfl_up_sync(0xffffffffu, e, 1);
    Uin = a0 + (lane == 0 ? fx_rescale(C, e - eC) : fx_rescale(y, e - ey));
  }
  // ---------------------------------------------------------------- 3. backward words
  const u64 Uin2 = fx_mul(Uin, R16, E1 + 1);
  u64 Y1 = 0, Y2 = 0;
  {
    const unsigned bh = (unsigned)(fx[FX_B] >> 32), bl = (unsigned)fx[FX_B];
    const unsigned uh = (unsigned)(Uin >> 32), ul = (unsigned)Uin, vh = (unsigned)(Uin2 >> 32), vl = (unsigned)Uin2;
    // GUARD: the system's last rows lie in this thread; beyond them u = 0 (the word a), so that X = 0
    // reaches row N unchanged
    auto sweep = [&](auto guard_) {
      constexpr bool GUARD = decltype(guard_)::value;
#pragma unroll 4
      for (int k = H / 2 - 1; k >= 0; --k) {
        ulonglong2 w = *reinterpret_cast<const ulonglong2*>(mine + 16 * k);
        ulonglong2 v = *reinterpret_cast<const ulonglong2*>(mine + 8 * H + 16 * k);
        const ulonglong2 p = *reinterpret_cast<const ulonglong2*>(tp + 2 * k);
        auto u = [&](int i, u64 t) { return (GUARD && i >= nv) ? a0 : t; };
        w.y = Y1 = fx_mul(Y1, bh, bl, u(2 * k + 1, fx_mul(p.y, uh, ul, w.y)));
        v.y = Y2 = fx_mul(Y2, bh, bl, u(H + 2 * k + 1, fx_mul(p.y, vh, vl, v.y)));
        w.x = Y1 = fx_mul(Y1, bh, bl, u(2 * k, fx_mul(p.x, uh, ul, w.x)));
        v.x = Y2 = fx_mul(Y2, bh, bl, u(H + 2 * k, fx_mul(p.x, vh, vl, v.x)));
        *reinterpret_cast<ulonglong2*>(mine + 16 * k) = w;
        *reinterpret_cast<ulonglong2*>(mine + 8 * H + 16 * k) = v;
      }
    };
    if (nv == kFixRows)
      sweep(std::false_type());
    else if (nv > 0)
      sweep(std::true_type());
  }
  // ---------------------------------------------------------------- 4. the words beyond the threads
  u64 Xin, E0;   // E0: the thread's first word, complete
  {
    const u64 loc = fx_mul(Y2, B16, Y1 + 1);
    if (!var) {
      u64 E = (nv == 0) ? 0ull : loc;
      if (tid == tlast) E = fx_mul(1ull << 63, tB[1], E + 1);
      for (int k = 0; k < levb; ++k) {
        const int d = 1 << k;
        const u64 y = __shfl_down_sync(0xffffffffu, E, d);
        E = fx_mul(lane + d > 31 ? 0ull : y, tB[d], E + (lane + d > 31 ? 0u : 1u));
      }
      if (lane == 0) sw[NW + wid] = E;
      Xin = __shfl_down_sync(0xffffffffu, E, 1);
      if (lane == 31) Xin = 0;
      __syncthreads();
      if (wid < NW - 1) {
        u64 C = sw[NW + wid + 1];
        if (levb >= 5) {
          C = sw[2 * NW - 1];
          for (int w = NW - 2; w > wid; --w) C = fx_mul(C, tB[32], sw[NW + w] + 1);
        }
        Xin = (lane == 31) ? C : fx_mul(C, tB[31 - lane], Xin + 1);
      }
    } else {
      u64 S = loc - ((1ull << 63) - fx_mul(1ull << 63, tB[1], 1ull));
      if (nv == 0) S = 0;
      const int lev = min(4, levb + 1);
      for (int k = 0; k < lev; ++k) {
        const int d = 1 << k;
        const u64 y = __shfl_down_sync(0xffffffffu, S, d);
        const int ey = __shfl_down_sync(0xffffffffu, e, d);
        if (lane + d <= 31) S += fx_move(y, fx[FX_BM + d], bx[d] + e - ey);
      }
      if (lane == 0) sw[NW + wid] = S;
      __syncthreads();
      u64 C = 0;
      int eC = e;
      if (wid < NW - 1) {
        C = sw[NW + wid + 1];
        eC = sblk[32 * (wid + 1)];
        S += fx_move(C, fx[FX_BM + 32 - lane], bx[32 - lane] + e - eC);
      }
      const u64 y = __shfl_down_sync(0xffffffffu, S, 1);
      const int ey = __shfl_down_sync(0xffffffffu, e, 1);
      Xin = (1ull << 63) + (lane == 31 ? fx_rescale(C, e - eC) : fx_rescale(y, e - ey));
    }
    if (tid >= tlast) Xin = 1ull << 63;
    E0 = fx_mul(Xin, tB[1], loc + 1);
  }
  if (flags & FIX_GUARD) {
    // high gain: the words' unit is set by the largest possible |X|; a window whose solution stays far
    // below that would keep fewer bits than FP64 does
    const u64 m = (E0 >> 63) ? E0 - (1ull << 63) : (1ull << 63) - E0;
    if (!__syncthreads_or(nv > 0 && (m >> (63 - kFixGuard)) != 0)) return false;
  }
  // the next kernel of the stream may begin its launch (it waits for this grid to complete)
  asm volatile("griddepcontrol.launch_dependents;");

  if (row_lo == 0) {
    // the system's first rows: X_i -= X_0 B R^(i+1)
    if (tid == 0) sx0[0] = E0;
    __syncthreads();
    const u64 x0 = sx0[0];
    const bool neg = (x0 >> 63) == 0;
    u64 c = neg ? (1ull << 63) - x0 : x0 - (1ull << 63);
    c = fx_mul(c, fx[FX_B], 0ull);
    if (!var) {
      for (int t = 0; t < (tid >> 5); ++t) c = fx_mul(c, tR[32], 0ull);
      if (lane) c = fx_mul(c, tR[lane], 0ull);
    } else if (tid > 32) {
      c = 0;
    } else if (tid > 0) {   // from the first thread's unit into this one's
      const int sh = rx[tid] + e - sblk[0];
      c = sh > 63 ? 0ull : fx_mul(c, fx[FX_RM + tid], 0ull) >> sh;
    }
    if (c > 2 && nv > 0) {
      const u64 c2 = fx_mul(c, R16, 0ull);
      const unsigned ch = (unsigned)(c >> 32), cl = (unsigned)c, dh = (unsigned)(c2 >> 32), dl = (unsigned)c2;
      const u64 sg = neg ? 0ull : ~0ull;   // two's complement of the correction to subtract it
#pragma unroll 4
      for (int k = 0; k < H / 2; ++k) {
        ulonglong2 w = *reinterpret_cast<const ulonglong2*>(mine + 16 * k);
        ulonglong2 v = *reinterpret_cast<const ulonglong2*>(mine + 8 * H + 16 * k);
        const ulonglong2 p = *reinterpret_cast<const ulonglong2*>(tp + 2 * k);
        w.x += (fx_mul(p.x, ch, cl, 0ull) ^ sg) - sg;
        w.y += (fx_mul(p.y, ch, cl, 0ull) ^ sg) - sg;
        v.x += (fx_mul(p.x, dh, dl, 0ull) ^ sg) - sg;
        v.y += (fx_mul(p.y, dh, dl, 0ull) ^ sg) - sg;
        *reinterpret_cast<ulonglong2*>(mine + 16 * k) = w;
        *reinterpret_cast<ulonglong2*>(mine + 8 * H + 16 * k) = v;
      }
    }
  }

  // ---------------------------------------------------------------- 5. the solution, own rows out
  if (own) {
    const u64 X1 = fx_mul(Xin, B16, Y2 + 1);
    const unsigned xh = (unsigned)(X1 >> 32), xl = (unsigned)X1, yh = (unsigned)(Xin >> 32), yl = (unsigned)Xin;
    const unsigned gh = (unsigned)(fx[FX_G] >> 32), gl = (unsigned)fx[FX_G];
    const u64 kg = fx[FX_KG];
    const unsigned eke = ((unsigned)((int)fx[FX_GK] - sc) << 20) + ((flags & FIX_NEG) ? 0x80000000u : 0u), eko = eke + alt;
#pragma unroll 4
    for (int k = 0; k < H / 2; ++k) {
      const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(mine + 16 * k);
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(mine + 8 * H + 16 * k);
      const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(tq + 2 * k);
      const u64 z0 = fx_mul(fx_mul(q.x, xh, xl, w.x), gh, gl, kg), z1 = fx_mul(fx_mul(q.y, xh, xl, w.y), gh, gl, kg);
      const u64 s0 = fx_mul(fx_mul(q.x, yh, yl, v.x), gh, gl, kg), s1 = fx_mul(fx_mul(q.y, yh, yl, v.y), gh, gl, kg);
      *reinterpret_cast<double2*>(mine + 16 * k) = make_double2(fx_to_f64(z0, eke), fx_to_f64(z1, eko));
      *reinterpret_cast<double2*>(mine + 8 * H + 16 * k) = make_double2(fx_to_f64(s0, eke), fx_to_f64(s1, eko));
    }
  }
  __syncwarp();
  const bool al_dst = (reinterpret_cast<uintptr_t>(dst) & 15u) == 0u;
  if (A.xf == nullptr) {
    slots_store(smem, dst, j0, j1, al_dst, lane, wid);
    return true;
  }
  // the adjoint (a5): the gradient sums over the own rows, in FP64, beside the store
  double g0 = 0.0, gm = 0.0, gp = 0.0;
  {
    const int r0 = max(j0 - wid * kWarpRows, 0), r1 = min(j1 - wid * kWarpRows, kWarpRows);
    const int64_t N = pp->N, rw = row_lo + wid * kWarpRows;
    const double* xf = A.xf + pp->off + rw;
    double* dw = dst + wid * kWarpRows;
    const unsigned char* sl = smem + (size_t)wid * 32 * kRegPairBytes + lane * 8;
#pragma unroll 4
    for (int j = lane + (r0 & ~31); j < r1; j += 32) {
      if (j < r0) continue;
      const double dv = *reinterpret_cast<const double*>(sl + (j >> 5) * kRegPairBytes);
      const int64_t r = rw + j;
      __stcs(dw + j, dv);
      g0 = fma(dv, xf[j], g0);
      gm = fma(dv, r > 0 ? xf[j - 1] : 0.0, gm);
      gp = fma(dv, r + 1 < N ? xf[j + 1] : 0.0, gp);
    }
  }
  g0 = warp_sum3(gm, g0, gp, lane);
  double* sred = reinterpret_cast<double*>(sw);
  __syncthreads();
  if ((lane & 7) == 0 && lane < 24) sred[(lane >> 3) * NW + wid] = g0;
  __syncthreads();
  if (tid < 3) {
    double s = 0.0;
    for (int w = 0; w < NW; ++w) s += sred[tid * NW + w];
    A.part[3 * (size_t)blockIdx.x + tid] = s;
  }
  return true;
}

}  // namespace dich
