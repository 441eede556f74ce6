// fixed.cuh -- 64-bit fixed-point words on the integer pipes: the products and conversions shared by the
// fixed-point form of FP64 windows (window_fix.cuh) and the sine transform (dst_fixed.cu).
#pragma once

namespace dich {

typedef unsigned long long u64;

// acc + x r 2^-64, truncated (1.25 units below on average, at most 3)
__device__ __forceinline__ u64 fx_mul(u64 x, unsigned rh, unsigned rl, u64 acc) {
  const unsigned xh = (unsigned)(x >> 32), xl = (unsigned)x;
  const u64 p = (u64)xh * rh + acc;
  return p + (u64)__umulhi(xl, rh) + (u64)__umulhi(xh, rl);
}
__device__ __forceinline__ u64 fx_mul(u64 x, u64 r, u64 acc) { return fx_mul(x, (unsigned)(r >> 32), (unsigned)r, acc); }

// K + d 2^sc by shifts on the integer pipe (sb = 1086 - sc; smaller values shift out to zero)
__device__ __forceinline__ u64 fx_from_f64_alu(double d, unsigned sb, u64 K) {
  const unsigned hw = (unsigned)__double2hiint(d), lw = (unsigned)__double2loint(d);
  const unsigned sh = sb - ((hw >> 20) & 0x7FFu);
  const unsigned mh = __funnelshift_l(lw, hw, 11) | 0x80000000u, ml = lw << 11;
  u64 v;
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(((u64)mh << 32) | ml), "r"(sh));
  const int m = (int)hw >> 31;
  v ^= (u64)(long long)m;
  return v + K + (u64)(hw >> 31);
}

}  // namespace dich
