// lane_profile.cuh -- the int8 query profile of kernels whose lanes own
// consecutive query rows (lane_kernel.cuh, noalloc.cu).
//
// Profile of 32 lanes with PR rows each (PW bytes: PR in whole words),
// code-major:
//   rows [VB * v, VB * v + VB) of lane l against code c at
//   c * 32 * PW + v * 32 * VB + l * VB,   VB = bytes per load,
// so the lanes of a quarter- or half-warp read distinct banks whatever codes
// they read.
#pragma once

#include "device_common.cuh"

namespace swgb {

constexpr int LANE_ROWS_MAX = 32;
constexpr int SM_ROW = 28;  // bytes per row of the matrix copy: 25 scores, in whole words

// 4 x 4 byte transpose: word b of the result holds byte b of a, b, c, d
__device__ __forceinline__ uint4 transpose4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  const uint32_t ab0 = prmt(a, b, 0x5140u), ab1 = prmt(a, b, 0x7362u);
  const uint32_t cd0 = prmt(c, d, 0x5140u), cd1 = prmt(c, d, 0x7362u);
  return make_uint4(prmt(ab0, cd0, 0x5410u), prmt(ab0, cd0, 0x7632u), prmt(ab1, cd1, 0x5410u),
                    prmt(ab1, cd1, 0x7632u));
}

// A lane's PR rows may be cut into NQ quarters (halves) of PR / NQ rows, each one
// column behind the one above: NQ independent chains of cells per step, for a
// warp that has its scheduler (nearly) to itself, at NQ times the ramp.
template <int PR, int NQ>
struct LaneShape {
  static constexpr int R = PR / NQ;  // rows per quarter
  static constexpr int RW = (R + 3) / 4;  // their profile words
  static constexpr int PW = 4 * RW * NQ;  // profile bytes per lane and code
  static_assert(R % (NQ == 1 ? 2 : 4) == 0 && PW <= LANE_ROWS_MAX, "pairs of rows, at most 32");
  static constexpr int VB = RW % 4 == 0 ? 16 : RW % 2 == 0 ? 8 : 4;  // bytes per profile load
  static constexpr int UNROLL = 4;                                  // steps per loop body
  static constexpr bool AHEAD = PR <= 24;  // registers allow the next step's profile words
};

// The profile of rows [row0 + li * PR, ...) of query residues qr[0, m)
// for lanes li = l % lg.  Four rows and four codes at a time: one word of four
// scores per row, transposed into one word of four rows per code.
// Warp `first` of `warps` takes every warps-th row quad.
template <int PR, int NQ>
__device__ __forceinline__ void lane_profile_rows(uint8_t* prof, const uint8_t* sm,
                                                  const uint8_t* __restrict__ qr, int m, int row0,
                                                  int lg, int first, int warps) {
  constexpr int VB = LaneShape<PR, NQ>::VB, PW = LaneShape<PR, NQ>::PW;
  const int l = threadIdx.x & 31;
  // (of PR = 4 k + 2 rows, the last word's upper half is the next lane's rows
  // and is not used)
  for (int rq = first; rq < PW / 4; rq += warps) {
    const int r0 = row0 + (l & (lg - 1)) * PR + 4 * rq;
    const uint8_t* s[4];
#pragma unroll
    for (int b = 0; b < 4; b++) s[b] = sm + (r0 + b < m ? min((int)qr[r0 + b], PAD_CODE) : PAD_CODE) * SM_ROW;
    uint8_t* dst = prof + (4 * rq / VB) * 32 * VB + l * VB + (4 * rq) % VB;
#pragma unroll
    for (int cq = 0; cq < SM_ROW / 4; cq++) {
      const uint4 w = transpose4(*(const uint32_t*)(s[0] + 4 * cq), *(const uint32_t*)(s[1] + 4 * cq),
                                 *(const uint32_t*)(s[2] + 4 * cq), *(const uint32_t*)(s[3] + 4 * cq));
      const uint32_t v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int b = 0; b < 4; b++)
        if (4 * cq + b < NCODES) *(uint32_t*)(dst + (4 * cq + b) * 32 * PW) = v[b];
    }
  }
}

}  // namespace swgb
