// device_common.cuh -- device helpers shared by the alignment kernels of
// libswgb: lane_kernel.cu, inter_kernel.cu, inter2q_kernel.cu, pair2q_kernel.cu, intra_kernel.cu,
// align_kernel.cu, plain_kernel.cu.
//
// Every kernel computes Eq. 1-3 of arxiv 2309.09609 (Section II-B) in the
// shared-gap form
//
//   h = max(hdiag + SM(q_i, d_j), E(i,j), F(i,j), 0)          (Eq. 1)
//   t = h - Go
//   E(i,j+1) = max(E(i,j) - Ge, t)                             (Eq. 2, next column)
//   F(i+1,j) = max(F(i,j) - Ge, t)                             (Eq. 3, next row)
//   S = max(S, h)
//
// which reorders Algorithm 1 so that H - Go is computed once per cell and E
// and F are produced one step ahead (the paper's future work, Section VI,
// names instruction reordering and narrower integers; the packed kernels do
// both).
//
// Threads wait on one another only at __syncwarp and at barriers of a block or
// of a cluster; the only other interaction between blocks is an atomic work
// counter, so nothing can spin.
#pragma once

#include <stdint.h>

#include "swgb_internal.h"

namespace swgb {

constexpr unsigned FULL = 0xffffffffu;
constexpr int MATRIX_SMEM = 640;  // 25 x 25 int8, rounded up to 16 bytes

__device__ __forceinline__ uint32_t pack2(int v) {
  return ((uint32_t)(uint16_t)(int16_t)v) * 0x00010001u;
}

// prmt with sign replication: result = (sext(a.byte k), sext(b.byte k)) as s16x2
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}
// selector for byte k: nibbles (low to high) k, 8|k, 4+k, 8|(4+k)
__device__ __forceinline__ constexpr uint32_t sext_pair_sel(int k) {
  return (uint32_t)(k | ((8 | k) << 4) | ((4 + k) << 8) | ((12 + k) << 12));
}

__device__ __forceinline__ uint4 ldg_nc(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// 16-byte asynchronous global -> shared copy (L2 only), and its group fences.
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem_src) : "memory");
}
// The same, or zeros and nothing read (bytes 16 or 0).
__device__ __forceinline__ void cp_async16_or_zeros(void* smem_dst, const void* gmem_src,
                                                    int bytes) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s), "l"(gmem_src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---- score output ------------------------------------------------------------
__device__ __forceinline__ void emit_score(const DbView& db, const SearchParams* __restrict__ P,
                                           int q, int s, int score) {
  const int orig = db.perm[s];
  if (orig >= 0) P->scores[(int64_t)q * db.n + orig] = score;
}

// S of each subject of a pair (the halves of smax): recorded, or flagged for the
// int32 recompute when it may have saturated.
__device__ __forceinline__ void emit_pair(const DbView& db, const SearchParams* __restrict__ P,
                                          SearchState* st, const Scratch& scr, int q, int pair,
                                          uint32_t smax) {
#pragma unroll
  for (int half = 0; half < 2; half++) {
    const int sidx = 2 * pair + half;
    const int orig = db.perm[sidx];
    if (orig < 0) continue;
    const int s = (int)(int16_t)(half ? (smax >> 16) : (smax & 0xffffu));
    if (s >= P->sat_threshold) {
      const unsigned long long k = atomicAdd(&st->n_flags, 1ull);
      if ((int64_t)k < scr.flag_capacity)
        scr.flags[k] = make_int2(q, sidx);
      else  // the list is full: mark the pair for the host's next recompute round
        P->scores[(int64_t)q * db.n + orig] = FLAG_SENTINEL;
    } else {
      P->scores[(int64_t)q * db.n + orig] = s;
    }
  }
}

// SM into shared memory (every thread of the block takes part; the caller syncs)
__device__ __forceinline__ void load_matrix(int8_t* sm, const SearchParams* __restrict__ P) {
  for (int i = threadIdx.x; i < NCODES * NCODES; i += blockDim.x) sm[i] = P->sm[i];
}

// int8 profile of one lane's R query rows [i0, i0 + R) of a pass, for every
// code c: byte r of the R-byte row at prof + (c * 32 + lane) * R is
// SM(q[i0 + r], c), and PAD_SCORE past the end of the query.
template <int R>
__device__ __forceinline__ void lane_profile(uint8_t* prof, const int8_t* __restrict__ sm,
                                             const uint8_t* __restrict__ qr, int m, int i0,
                                             int lane) {
  static_assert(R % 8 == 0, "rows per lane must be a multiple of 8");
  int qc[R];
#pragma unroll
  for (int r = 0; r < R; r++) qc[r] = (i0 + r < m) ? (int)qr[i0 + r] : -1;
  for (int c = 0; c < NCODES; c++) {
    uint32_t wv[R / 4];
#pragma unroll
    for (int w = 0; w < R / 4; w++) {
      uint32_t acc = 0;
#pragma unroll
      for (int b = 0; b < 4; b++) {
        const int r = w * 4 + b;
        const int v = qc[r] >= 0 ? (int)sm[qc[r] * NCODES + c] : PAD_SCORE;
        acc |= ((uint32_t)(uint8_t)(int8_t)v) << (8 * b);
      }
      wv[w] = acc;
    }
    uint8_t* dst = prof + (c * 32 + lane) * R;
    if constexpr (R % 16 == 0) {
#pragma unroll
      for (int w = 0; w < R / 4; w += 4)
        *(uint4*)(dst + 4 * w) = make_uint4(wv[w], wv[w + 1], wv[w + 2], wv[w + 3]);
    } else {
#pragma unroll
      for (int w = 0; w < R / 4; w += 2) *(uint2*)(dst + 4 * w) = make_uint2(wv[w], wv[w + 1]);
    }
  }
}

// The lane's profile words along its columns, loaded ahead of the cells: the
// code of column j + 2 and the words of column j + 1 while column j is scored
// (columns past either end read the first or last code, for lanes that skip
// them).
template <int TI>
struct IntraFeed {
  const uint8_t* d;     // the subject's codes
  const uint8_t* prof;  // the lane's profile rows, 32 * TI bytes per code
  int n, code;
  uint32_t next[TI / 4];

  __device__ __forceinline__ int at(int j) const {
    return d[min(max(j, 0), n - 1)];
  }
  __device__ __forceinline__ void words() {
    const uint8_t* lp = prof + code * 32 * TI;
    static_assert(TI == 8 || TI == 16, "rows per lane");
    if constexpr (TI == 8) {
      const uint2 v = *(const uint2*)lp;
      next[0] = v.x, next[1] = v.y;
    } else {
      const uint4 v = *(const uint4*)lp;
      next[0] = v.x, next[1] = v.y, next[2] = v.z, next[3] = v.w;
    }
  }
  __device__ __forceinline__ void start(int j) {  // the next column is j
    code = at(j);
    words();
    code = at(j + 1);
  }
  __device__ __forceinline__ void step(uint32_t (&pw)[TI / 4], int j) {  // column j's words
#pragma unroll
    for (int k = 0; k < TI / 4; k++) pw[k] = next[k];
    words();
    code = at(j + 2);
  }
};

// ---- packed 16-bit cells (two cells per 32-bit word) -------------------------
//
// Each half of a word is one cell's H, E or F as a signed 16-bit integer.  The
// update is bound by the ALU pipe, which runs every 16x2 maximum; the FMA pipe
// runs the 16x2 additions (VIADD) beside it.  So the two additions that need
// no maximum with them go to the FMA pipe, and four maxima per word remain:
//
//   x = hdiag + SM             16x2 add          FMA pipe
//   h = max(x, e, f)           VIMNMX3           ALU pipe    (Eq. 1)
//   t = h - Go                 16x2 subtract     FMA pipe
//   e = max(e - Ge, t, 0)      VIADDMNMX.RELU    ALU pipe    (Eq. 2, next column)
//   f = max(f - Ge, t)         VIADDMNMX         ALU pipe    (Eq. 3, next row)
//   s = max(s, x, x')          VIMNMX3           ALU pipe, once per two words
//
// i.e. 3.5 ALU and 2 FMA operations per word.
//   * Eq. 1's zero term: e is held at 0 or above, which the update gives at no
//     cost, so h >= 0.  An E or F below 0 never reaches an H (each H is at
//     least 0, and a chain only falls from there), so flooring E, or starting
//     E and F at 0 instead of -Go, changes no H.
//   * S is the maximum of x instead of h: a positive H that exceeds its
//     neighbours' came by the diagonal (E and F lie below the H they opened
//     from), so the largest x is the largest H.  It also gives x a second
//     use; with h in its place the compiler folds the addition back into a
//     VIADDMNMX on the ALU pipe.
// In a loop of independent cells, 1,024 threads per SM, that measured 7.9
// cycles per word and scheduler, against 9.3 for the same cell with values
// biased by Go (zero term as a constant in the VIMNMX3, hdiag + SM inside a
// VIADDMNMX: 4.5 ALU and 1 FMA operations).  In the search kernels: 20 queries
// of 144-5,478 residues x 100,000 subjects 169.0 -> 149.2 ms, 96 queries of
// 50-2,000 x 100,000 480.4 -> 422.8 ms, one query of 375 x 570,000 16.4 -> 14.9.
//
// Range: E >= 0, F >= -Go, x >= -128 and E - Ge, F - Ge >= -(Go + Ge) stay
// inside 16 bits, and H does as long as H <= 32767.  H grows by at most
// max(SM) along a diagonal and every cell before the first overflow is exact,
// so a pair whose S reaches SearchParams::sat_threshold, which lies below
// 32767 - max(SM), is recomputed in int32 and any other S is exact.  The two
// halves never mix: every operation works half by half.

// The packed words of the gap penalties: GO2 = (Go, Go), NGE2 = (-Ge, -Ge).
// Gap class G > 0 fixes them at compile time for a common setting, so they
// enter the instructions as immediates instead of registers (7.9 against 8.6
// cycles per word in the loop above); G = 0 reads them from the parameter
// block.  The classes are listed in swgb_internal.h (gap_class).
template <int G>
__device__ __forceinline__ void gap_words(const SearchParams* __restrict__ P, uint32_t& GO2,
                                          uint32_t& NGE2) {
  if constexpr (G == 0) {
    GO2 = pack2(P->go);
    NGE2 = pack2(-P->ge);
  } else {
    GO2 = ((uint32_t)(uint16_t)GapClass<G>::GO) * 0x00010001u;
    NGE2 = ((uint32_t)(uint16_t)(int16_t)(-GapClass<G>::GE)) * 0x00010001u;
  }
}

// One packed cell update: returns H and gives x = hdiag + SM for S; updates E
// of the next column in e and F of the next row in f.
__device__ __forceinline__ uint32_t packed_cell(uint32_t hd, uint32_t w, uint32_t& e, uint32_t& f,
                                                uint32_t& x, uint32_t GO2, uint32_t NGE2) {
  x = __vadd2(hd, w);
  const uint32_t h = __vimax3_s16x2(x, e, f);
  const uint32_t t = __vsub2(h, GO2);
  e = __viaddmax_s16x2_relu(e, NGE2, t);
  f = __viaddmax_s16x2(f, NGE2, t);
  return h;
}

// 32-bit multiply-add, kept on the FMA pipe for address arithmetic and exact
// selections (a product by 0 or 1).
__device__ __forceinline__ uint32_t imad(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}

}  // namespace swgb
