// slots.cuh -- a window's rows in shared memory, one padded slot of 32 rows per thread (the register path
// of the MIXED form, window_reg.cuh, and the fixed-point form of FP64 windows, window_fix.cuh).
//
// A slot is 256 contiguous bytes of the vector plus 16 bytes of padding, so that the per-thread
// 16-byte reads of eight consecutive threads fall in eight different bank groups.
// The copies in and out are coalesced over a warp, not one bulk copy (cp.async.bulk) per thread: a
// bulk copy is issued once per warp instruction, so 32 different ones per warp run as a loop over the
// lanes, about 12 instructions per lane and copy (measured on an otherwise empty window kernel: 26
// instructions per unknown with per-thread bulk copies, 12 with these).
#pragma once
#include "window.cuh"

namespace dich {

constexpr int kRegRows = 16;                            // block size of the register path
constexpr int kRegPairBytes = 2 * kRegRows * 8 + 16;    // a thread's two blocks + 16 bytes of padding

// ---------------------------------------------------------------- window rows <-> pair slots
// rows [0, rows) of `src` (rows of the window in order, 32 per slot) into the slots; al16: `src` is
// 16-byte aligned.  Waits are the caller's (cp_async_wait_all,
// then __syncwarp)
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
// Each warp copies the rows of its own 32 slots (1024 rows, contiguous in memory), so that no CTA
// barrier stands between a copy and the rows' use.
constexpr int kWarpRows = 32 * 2 * kRegRows;
__device__ __forceinline__ void slots_load(unsigned char* slots, const double* src, int rows, bool al16, int lane,
                                           int wid) {
  rows = min(rows - wid * kWarpRows, kWarpRows);   // rows of this warp's slots (none: zero or negative)
  src += wid * kWarpRows;
  slots += (size_t)wid * 32 * kRegPairBytes;
  if (al16) {
    unsigned char* d = slots + (lane >> 4) * kRegPairBytes + (lane & 15) * 16;
    const double* g = src + 2 * lane;
    if (rows == kWarpRows) {   // every address one base plus a constant
#pragma unroll
      for (int k = 0; k < kRegRows; ++k) cp_async16(d + k * 2 * kRegPairBytes, g + k * 64);
    } else {
      for (int k = 0; 2 * lane + k * 64 < rows; ++k) {
        if (2 * lane + k * 64 + 1 < rows)
          cp_async16(d + k * 2 * kRegPairBytes, g + k * 64);
        else   // an odd last row: nothing past it is read
          cp_async8(d + k * 2 * kRegPairBytes, g + k * 64);
      }
    }
  } else {
    unsigned char* d = slots + lane * 8;
    const double* g = src + lane;
#pragma unroll 8
    for (int k = 0; lane + k * 32 < rows; ++k) cp_async8(d + k * kRegPairBytes, g + k * 32);
  }
}
// rows [r0, r1) of the window's slots, as far as they lie in the warp's own slots, to dst[r0 .. r1); al16: `dst` is 16-byte aligned
__device__ __forceinline__ void slots_store(const unsigned char* slots, double* dst, int r0, int r1, bool al16,
                                            int lane, int wid) {
  dst += wid * kWarpRows;
  slots += (size_t)wid * 32 * kRegPairBytes;
  r0 = max(r0 - wid * kWarpRows, 0);
  r1 = min(r1 - wid * kWarpRows, kWarpRows);
  if (al16) {
    const int c = (lane & 15) * 16;
    if (r0 == 0 && r1 == kWarpRows) {   // every address one base plus a constant
      const unsigned char* d = slots + (lane >> 4) * kRegPairBytes + c;
      double2* g = reinterpret_cast<double2*>(dst) + lane;
#pragma unroll 8
      for (int k = 0; k < kRegRows; ++k) __stcs(g + k * 32, *reinterpret_cast<const double2*>(d + k * 2 * kRegPairBytes));
      return;
    }
#pragma unroll 2
    for (int j = 2 * lane + (r0 & ~63); j < r1; j += 64) {
      const double2 v = *reinterpret_cast<const double2*>(slots + (j >> 5) * kRegPairBytes + c);
      if (j >= r0 && j + 1 < r1) {
        __stcs(reinterpret_cast<double2*>(dst + j), v);
      } else {   // odd ends of the range
        if (j >= r0) __stcs(dst + j, v.x);
        if (j + 1 >= r0 && j + 1 < r1) __stcs(dst + j + 1, v.y);
      }
    }
  } else {
#pragma unroll 4
    for (int j = lane + (r0 & ~31); j < r1; j += 32)
      if (j >= r0) __stcs(dst + j, *reinterpret_cast<const double*>(slots + (j >> 5) * kRegPairBytes + lane * 8));
  }
}

}  // namespace dich
