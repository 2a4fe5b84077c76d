// align_kernel.cu -- optimal local alignments with traceback (sw_align).
//
// The score kernels return S only.  For selected pairs this file also
// recovers the alignment behind S, by the traceback of Section II-B.  A team of
// W warps takes a pair:
//
//   * forward: the int32 warp wavefront of Eq. 1-3 (lane k owns AT query rows of
//     a 32*AT-row pass, (H, F) borders by __shfl_up_sync).  Every cell stores
//     four bits -- where H came from, and whether E of the next column and F
//     of the next row open a gap here -- and the team keeps the cell holding S.
//     The passes go round-robin to the team's warps on the stage schedule of
//     the int32 recompute (intra_kernel.cu): pass p starts ALAG stages of 16
//     steps after pass p - 1, a stage ends at the team's barrier, each warp
//     writes the bottom rows of its passes to its own border row and reads
//     those of the warp before;
//   * traceback, by the team's first warp: 32 cells of the path at a time.
//     Along the diagonal the lanes read the bits of the next 32 cells at once
//     and a ballot gives the length of the run; in a gap they read along the
//     row or the column.
//
// Which of several optimal alignments is returned:
//   1. it ends at the first cell (i, j) in row-major order whose H equals S;
//   2. walking back in state H: the diagonal term first, then E, then F,
//      whichever equals H;
//   3. in a gap state the gap opens from H when that reaches the gap's
//      value, else it extends;
//   4. the walk ends with the diagonal step into a cell whose H is 0.
// Transcript, first column to last: 'M' (query and subject residue), 'I'
// (query residue against a gap), 'D' (subject residue against a gap).
//
// Bound by latency: a call has few pairs, so what counts is a pair's chain of
// steps and not the chip's rate.  Hence the bits come off the chain (a subtract
// whose sign a funnel shift collects, four per cell, combined once per lane), the best cell is looked for only in steps whose largest H reaches the
// lane's best, codes and profile words are loaded ahead, and teams are as
// large as the call leaves room for.  Measured, kernel time: 20 pairs of 400
// residues, the longest 662 x 1,236, 1.23 -> 0.34 ms (forward 0.90, walk 0.33
// before); 500 such pairs, the longest subject 3,343, 4.9 -> 0.97 ms.
#include <algorithm>

#include "lane_profile.cuh"

namespace swgb {

constexpr int ASTAGE = 16;  // steps of a stage
constexpr int ALAG = 4;     // stages between the starts of consecutive passes

// A team of W warps, AT query rows per lane: as many warps as there is room
// for and few rows for a call of few pairs, whose steps are then short; a block
// is a team, or four teams of one warp.  The bits of a lane's rows at one step
// are one word.
template <int W>
struct AlignShape {
  static constexpr int AT = W == 16 ? 4 : 8;
  static constexpr int ROWS = 32 * AT;  // rows per pass
  static constexpr int PROFILE = NCODES * 32 * AT;
  static constexpr int TEAMS = W == 1 ? 4 : 1;
  static constexpr int WARPS = W * TEAMS;
};
template <int AT> struct AlignWord;
template <> struct AlignWord<4> { typedef uint16_t type; };
template <> struct AlignWord<8> { typedef uint32_t type; };

// Word (pass p, step t, lane k) holds the cells of the lane's AT rows at
// column t - k: four fields of AT bits, with row r at bit AT - 1 - r of each.
// Fields 0 and 1 tell the source of H (where it is not 0): (1, 0) diagonal,
// (0, 1) E, (0, 0) F; field 2: E of the next column opens here; field 3: F
// of the next row opens here.
__device__ __forceinline__ int64_t bits_word(int n, int p, int t, int lane) {
  return ((int64_t)p * (n + 31) + t) * 32 + lane;
}

__device__ __forceinline__ bool end_before(int v, int i, int j, int bv, int bi, int bj) {
  return v > bv || (v == bv && (i < bi || (i == bi && j < bj)));
}

// acc shifted left by one, with the sign of x (1 when negative) as its last bit
__device__ __forceinline__ uint32_t push_sign(uint32_t acc, int x) {
  return __funnelshift_l((uint32_t)x, acc, 1);
}

struct AlignBest {
  int v, i, j;  // H, 1-based row and column
  __device__ __forceinline__ void take(int v2, int i2, int j2) {
    if (end_before(v2, i2, j2, v, i, j)) {
      v = v2;
      i = i2;
      j = j2;
    }
  }
};

// The forward pass of one pair on the team's W warps; `warp` is this warp's
// place in the team.  Returns the lane's best cell.
template <int W, typename Word, typename Barrier>
__device__ __forceinline__ AlignBest align_forward(const DbView& db,
                                                   const SearchParams* __restrict__ P,
                                                   const AlignItem& it, uint8_t* prof,
                                                   const uint8_t* sm, int lane, int warp,
                                                   Word* bits, int2* border,
                                                   Barrier barrier) {
  constexpr int AT = AlignShape<W>::AT, AROWS = AlignShape<W>::ROWS;
  const int go = P->go, ge = P->ge;
  const int m = P->qlen[it.q];
  const int n = db.clen[it.s];
  const uint8_t* __restrict__ qr = P->qres + P->qoff[it.q];
  const uint8_t* __restrict__ d = db.cont + db.coff[it.s];
  int2* own = border + it.border_off + (int64_t)warp * n;
  const int2* src = border + it.border_off + (int64_t)((warp + W - 1) % W) * n;
  const int npass = n > 0 ? (m + AROWS - 1) / AROWS : 0;
  const int spass = (n + 31 + ASTAGE - 1) / ASTAGE;
  const int period = max(spass, ALAG * W);
  const int nstages =
      npass > 0 ? ((npass - 1) / W) * period + ((npass - 1) % W) * ALAG + spass : 0;
  const int2 top = make_int2(0, -go);
  AlignBest best{0, INT32_MAX, INT32_MAX};
  int H[AT], E[AT], hdiag = 0, out_h = 0, out_f = -go;
  int p = 0;
  int2 bcur = top, bnext = top;
  for (int g = 0; g < nstages; g++) {
    const int rel = g - warp * ALAG;
    int k = -1;
    if (rel >= 0) {
      const int r = rel / period;
      const int kk = rel - r * period;
      if (kk < spass && warp + r * W < npass) {
        k = kk;
        p = warp + r * W;
      }
    }
    if (k >= 0) {  // warp-uniform
      if (k == 0) {
        __syncwarp();
        lane_profile_rows<AT, 1>(prof, sm, qr, m, p * AROWS, 32, 0, 1);
        __syncwarp();
#pragma unroll
        for (int r = 0; r < AT; r++) H[r] = E[r] = 0;
        hdiag = 0;
        out_h = 0;
        out_f = -go;
        bcur = (p > 0 && lane < min(ASTAGE, n)) ? src[lane] : top;
      } else {
        bcur = bnext;
      }
      const int jn = ASTAGE * (k + 1) + lane;
      bnext = (p > 0 && lane < ASTAGE && jn < n) ? src[jn] : top;
      const bool last_pass = (p == npass - 1);
      const int row0 = p * AROWS + lane * AT;  // 0-based row of this lane's first row
      const int t0 = ASTAGE * k;
      const int tend = min(t0 + ASTAGE, n + 31);
      IntraFeed<AT, true> feed{d, prof + lane * AT, n};
      feed.start(t0 - lane);
#pragma unroll 4
      for (int t = t0; t < tend; t++) {
        uint32_t pw[AT / 4];
        feed.step(pw, t - lane);
        int in_h = __shfl_up_sync(FULL, out_h, 1);
        int in_f = __shfl_up_sync(FULL, out_f, 1);
        const int bh = __shfl_sync(FULL, bcur.x, t - t0);
        const int bf = __shfl_sync(FULL, bcur.y, t - t0);
        if (lane == 0) {
          in_h = bh;
          in_f = bf;
        }
        // columns left and right of the subject hold the padding code: their
        // cells leave H and E at 0 before it, and are not looked at after it
        const int j = t - lane;
        int hd = hdiag, f = in_f, top_h = 0;
        hdiag = in_h;
        // signs: H above the diagonal term, above E; H - Go below the next E,
        // below the next F
        uint32_t sa = 0, sb = 0, se = 0, sf = 0;
#pragma unroll
        for (int r = 0; r < AT; r++) {
          const int e = E[r];  // floored at 0: only cells with E > 0 matter to the walk
          const int x = __dp4a((int)pw[r / 4], 1 << (8 * (r & 3)), hd);
          const int h = __vimax3_s32(x, e, f);                  // Eq. 1
          hd = H[r];
          H[r] = h;
          const int tt = h - go;
          E[r] = __viaddmax_s32_relu(e, -ge, tt);               // Eq. 2, next column
          f = __viaddmax_s32(f, -ge, tt);                       // Eq. 3, next row
          sa = push_sign(sa, x - h);
          sb = push_sign(sb, e - h);
          se = push_sign(se, tt - E[r]);
          sf = push_sign(sf, tt - f);
          top_h = max(top_h, h);
        }
        out_h = H[AT - 1];
        out_f = f;
        constexpr uint32_t F = (1u << AT) - 1;
        bits[bits_word(n, p, t, lane)] =
            (Word)((~sa & F) | (~sb & sa & F) << AT | (~se & F) << 2 * AT | (~sf & F) << 3 * AT);
        if (top_h >= best.v && top_h > 0 && j < n) {
#pragma unroll
          for (int r = 0; r < AT; r++)
            if (H[r] > 0 && row0 + r < m) best.take(H[r], row0 + r + 1, j + 1);
        }
        if (lane == 31 && !last_pass && j >= 0 && j < n) own[j] = make_int2(out_h, out_f);
      }
    }
    barrier();
  }
  // the first cell in row-major order holding the largest H of the warp
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int v = __shfl_xor_sync(FULL, best.v, o), i = __shfl_xor_sync(FULL, best.i, o),
              j = __shfl_xor_sync(FULL, best.j, o);
    best.take(v, i, j);
  }
  return best;
}

// The walk back from `best`, on one warp.  v is H (or E or F) of the current
// cell, which the matrix and the penalties give step by step.
template <int W, typename Word>
__device__ __forceinline__ void align_traceback(const DbView& db,
                                                const SearchParams* __restrict__ P,
                                                const AlignItem& it, const AlignBest& best,
                                                const uint8_t* sm, int lane, const Word* bits,
                                                uint8_t* ops, AlignOut* out) {
  constexpr int AT = AlignShape<W>::AT, AROWS = AlignShape<W>::ROWS;
  const int m = P->qlen[it.q];
  const int n = db.clen[it.s];
  const int go = P->go, ge = P->ge;
  const uint8_t* __restrict__ qr = P->qres + P->qoff[it.q];
  const uint8_t* __restrict__ d = db.cont + db.coff[it.s];
  int64_t pos = it.ops_end;  // the transcript is written backwards, ending here
  int i = best.i, j = best.j, v = best.v, state = 0;  // 0: H, 1: E, 2: F
  // a cell's bits, field f at bit f * AT; cells off the matrix open any gap
  auto cell = [&](int ci, int cj) -> uint32_t {
    if (ci < 1 || cj < 1) return 1u << 2 * AT | 1u << 3 * AT;
    const int row = ci - 1, l = row % AROWS / AT;
    return (uint32_t)bits[bits_word(n, row / AROWS, cj - 1 + l, l)] >> (AT - 1 - row % AT);
  };
  // every round takes at least one column or changes the state; the bound only
  // guards against a broken bit matrix
  for (int64_t guard = 0; v > 0 && guard < 2 * ((int64_t)m + n) + 2; guard++) {
    int run;
    uint8_t op;
    if (state == 0) {
      const int ci = i - lane, cj = j - lane;
      const uint32_t w = cell(ci, cj);
      // H after this cell's diagonal step, while the run lasts
      int h = ci >= 1 && cj >= 1 ? (int)(int8_t)sm[qr[ci - 1] * SM_ROW + d[cj - 1]] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(FULL, h, o);
        if (lane >= o) h += x;
      }
      h = v - h;
      const uint32_t other = __ballot_sync(FULL, !(w & 1u)), zero = __ballot_sync(FULL, h == 0);
      const int first = other ? __ffs(other) - 1 : 32;  // not from the diagonal
      const int end = zero ? __ffs(zero) : 33;          // columns to the cell whose H is 0
      run = min(first, end);
      op = 'M';
      if (run > 0) v = __shfl_sync(FULL, h, run - 1);
      if (first < 32) state = __shfl_sync(FULL, w >> AT & 1u, first) ? 1 : 2;
      if (lane < run) ops[pos - 1 - lane] = op;
      pos -= run;
      i -= run;
      j -= run;
    } else {
      const uint32_t w = state == 1 ? cell(i, j - 1 - lane) >> 2 * AT : cell(i - 1 - lane, j) >> 3 * AT;
      const uint32_t opens = __ballot_sync(FULL, w & 1u);
      run = opens ? __ffs(opens) : 32;
      op = state == 1 ? 'D' : 'I';
      if (lane < run) ops[pos - 1 - lane] = op;
      pos -= run;
      (state == 1 ? j : i) -= run;
      v += opens ? (run - 1) * ge + go : run * ge;
      if (opens) state = 0;
    }
  }
  if (lane == 0) {
    AlignOut r{};
    r.score = best.v;
    if (best.v > 0) {
      r.i_end = best.i;
      r.j_end = best.j;
      r.q_begin = i;
      r.s_begin = j;
    }
    r.n_ops = (int32_t)(it.ops_end - pos);
    r.ops_offset = pos;
    *out = r;
  }
}

template <int W>
__global__ void __launch_bounds__(AlignShape<W>::WARPS * 32)
align_kernel(DbView db, const SearchParams* __restrict__ P, const AlignItem* __restrict__ items,
             int n_items, uint8_t* bits, int2* border, AlignOut* out, uint8_t* ops) {
  constexpr int TEAMS = AlignShape<W>::TEAMS;
  typedef typename AlignWord<AlignShape<W>::AT>::type Word;
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ __align__(16) uint8_t sm[NCODES * SM_ROW];
  __shared__ AlignBest red[W];
  for (int i = threadIdx.x; i < NCODES * SM_ROW; i += blockDim.x)
    sm[i] = i % SM_ROW < NCODES ? (uint8_t)P->sm[i / SM_ROW * NCODES + i % SM_ROW] : 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, warp = wib % W;
  uint8_t* prof = smem + wib * AlignShape<W>::PROFILE;
  // uniform over the team
  for (int k = blockIdx.x * TEAMS + wib / W; k < n_items; k += gridDim.x * TEAMS) {
    const AlignItem it = items[k];
    Word* words = (Word*)(bits + it.bits_off);
    AlignBest best = align_forward<W>(db, P, it, prof, sm, lane, warp, words, border, []() {
      if constexpr (W > 1) __syncthreads();
      else __syncwarp();
    });
    if constexpr (W > 1) {
      if (lane == 0) red[warp] = best;
      __syncthreads();
      if (warp == 0)
        for (int w = 1; w < W; w++) best.take(red[w].v, red[w].i, red[w].j);
    }
    if (warp == 0) align_traceback<W>(db, P, it, best, sm, lane, words, ops, out + k);
    if constexpr (W > 1) __syncthreads();  // red is rewritten by the next pair
  }
}

// 16 warps to a pair while there are SMs for every pair, 4 while those teams
// (near enough) fit the chip at once, then one.
int align_team(int n_pairs, int sms) { return n_pairs <= sms ? 16 : n_pairs <= 16 * sms ? 4 : 1; }

template <int W>
static cudaError_t launch_team(int sms, const DbView& db, const SearchParams* params,
                               const AlignItem* items, int n_items, uint8_t* bits, int2* border,
                               AlignOut* out, uint8_t* ops, cudaStream_t stream) {
  const int smem = AlignShape<W>::WARPS * AlignShape<W>::PROFILE;
  cudaError_t e =
      cudaFuncSetAttribute(align_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int teams = AlignShape<W>::TEAMS;
  cudaGetLastError();  // a stale error must not be read as this launch's
  align_kernel<W><<<std::min((n_items + teams - 1) / teams, std::max(sms, 1) * 16),
                    AlignShape<W>::WARPS * 32, smem, stream>>>(db, params, items, n_items, bits,
                                                              border, out, ops);
  return cudaGetLastError();
}

cudaError_t launch_align(int team, int sms, const DbView& db, const SearchParams* params,
                         const AlignItem* items, int n_items, uint8_t* bits, int2* border,
                         AlignOut* out, uint8_t* ops, cudaStream_t stream) {
  if (n_items <= 0) return cudaSuccess;
  auto launch = team == 16 ? launch_team<16> : team == 4 ? launch_team<4> : launch_team<1>;
  return launch(sms, db, params, items, n_items, bits, border, out, ops, stream);
}

int64_t align_bits_bytes(int team, int32_t m, int32_t n) {
  if (m <= 0 || n <= 0) return 0;
  const int at = team == 16 ? AlignShape<16>::AT : AlignShape<4>::AT;
  return (int64_t)((m + 32 * at - 1) / (32 * at)) * (n + 31) * 32 * (at / 2);
}

}  // namespace swgb
