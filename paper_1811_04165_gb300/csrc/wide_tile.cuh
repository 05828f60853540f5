// The wide register tile shared by the pre-summed pass and step two: 8 trials x 7
// words (14 samples, two 16-bit lanes per word) per thread, and 8-bit counts.
//
// Keeping int32 sums beside the 16-bit lanes takes three registers per word; the
// counts take half a register: a fold moves the lanes' multiples of kWideCount
// (4096) into 8-bit fields, the four samples of two words to a register, and
// leaves the remainders in the lanes.  Sums up to 255 * 4096 + 65535 are exact, and
// with at most kWideFolds folds no lane's count passes 255, whatever it adds up.
#pragma once

#include <cstdint>

#include "sps_internal.h"
#include "tma.cuh"

namespace sps {

constexpr int kWideTrials = 8;  // trials per thread
constexpr int kWideWords = 7;   // words per thread and trial
constexpr int kWideTime = 64 * kWideWords;  // samples of a warp

// lds_row (tma.cuh) into `w` only where `load` is set (uniform over the warp); otherwise
// `w` keeps its words.
template <int NW, int M = 0>
__device__ __forceinline__ void lds_row_if(bool load, uint32_t addr, uint32_t (&w)[NW]) {
  if constexpr (M < NW) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.shared.u32 %0, [%1+%3];\n\t}"
                 : "+r"(w[M])
                 : "r"(addr), "r"((uint32_t)load), "n"(M * 128));
    lds_row_if<NW, M + 1>(load, addr, w);
  }
}

// The lanes' multiples of kWideCount move to the counts.
template <int ND, int NW>
__device__ __forceinline__ void wide_fold(uint32_t (&lanes)[ND][NW], uint32_t (&cnt)[ND * NW / 2]) {
#pragma unroll
  for (int k = 0; k < ND * NW / 2; k++) {
    uint32_t& x = lanes[2 * k / NW][2 * k % NW];
    uint32_t& y = lanes[(2 * k + 1) / NW][(2 * k + 1) % NW];
    cnt[k] += ((x >> 12) & 0x000F000Fu) + (((y >> 12) & 0x000F000Fu) << 8);
    x &= 0x0FFF0FFFu;
    y &= 0x0FFF0FFFu;
  }
}

// The two sums of word m of trial r.
template <int ND, int NW>
__device__ __forceinline__ int2 wide_sum(const uint32_t (&lanes)[ND][NW], const uint32_t (&cnt)[ND * NW / 2], int r,
                                         int m) {
  const uint32_t c = cnt[(r * NW + m) / 2] >> (8 * ((r * NW + m) & 1));
  return make_int2((int32_t)((lanes[r][m] & 0xFFFFu) + (c & 0xFFu) * kWideCount),
                   (int32_t)((lanes[r][m] >> 16) + ((c >> 16) & 0xFFu) * kWideCount));
}

}  // namespace sps
