// align_kernel.cu -- optimal local alignments with traceback (sw_align).
//
// The score kernels return S only.  For selected pairs this file also
// recovers the alignment behind S, by the traceback of Section II-B.  A team of
// W warps takes a pair:
//
//   * forward: the int32 warp wavefront of Eq. 1-3 (lane k owns AT query rows of
//     a 32*AT-row pass, (H, F) borders by one rotation).  Every cell stores
//     its H, in 16 bits, where no score of the call can exceed them and the
//     call's cells are few; otherwise four bits -- where H came from, and
//     whether E of the next column and F of the next row open a gap here.  The
//     team keeps the cell holding S.
//     The passes go round-robin to the team's warps on the stage schedule of
//     the int32 recompute (intra_kernel.cu): pass p starts ALAG stages of 16
//     steps after pass p - 1, a stage ends at the team's barrier, each warp
//     writes the bottom rows of its passes to its own border row and reads
//     those of the warp before;
//   * traceback, by the team's first warp: 32 cells of the path at a time.
//     Along the diagonal the lanes read the next 32 cells at once and a ballot
//     gives the length of the run; in a gap they read along the row or the
//     column.  From stored H, a cell came by the diagonal if the one above and
//     left and the matrix add up to it, else by E if some cell to its left
//     does with the gap between them (the nearest one; E may only fall along
//     the row, so any such cell proves it), else by F.
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
// steps, one warp's instructions and their latencies, and not the chip's rate
// (a step of four rows takes 200 cycles: 62 issues, 72 of fixed latency, 37 of
// loads).  Hence stored H, which costs the forward pass half a permute per
// cell; F of the next row from max(x, e), one operation per row on the chain;
// the largest H of each row as one key with its step, without a branch (the
// search for the best cell within the step, taken by some lane in most steps,
// was half of the time); codes and border rows staged in shared memory, and
// teams as large as the call leaves room for.  Where bits are stored, a subtract
// whose sign a funnel shift collects makes each, off the chain.  Measured,
// kernel time, 20 pairs of 400 residues, the longest 662 x 1,236: 1.23 ms with
// one warp to a pair, 0.34 with teams, 0.11 with all of this; 500 such pairs,
// the longest subject 3,343: 4.9 -> 0.97 -> 0.35 ms.  Calls with bits: 40 pairs
// of 6,000 x 6,000 6.8 -> 6.3 ms, 600 of 3,000 x 3,000 7.1 -> 6.8.
#include <algorithm>

#include "lane_profile.cuh"

namespace swgb {

constexpr int ASTAGE = 16;  // steps of a stage
constexpr int ALAG = 4;     // stages between the starts of consecutive passes

__host__ __device__ __forceinline__ int align_stages(int n) { return (n + 31 + ASTAGE - 1) / ASTAGE; }

// H and F of a pass's last row at one column, for the lane or the pass below:
// one word where 16 bits hold them (F is at least -Go).
template <bool KEEP_H> struct AlignEdge;
template <> struct AlignEdge<true> {
  uint32_t v;
  __device__ __forceinline__ AlignEdge() {}
  __device__ __forceinline__ AlignEdge(int h, int f) : v(prmt(h, f, 0x5410u)) {}
  __device__ __forceinline__ int h() const { return v & 0xffffu; }
  __device__ __forceinline__ int f() const { return (int)v >> 16; }
  __device__ __forceinline__ AlignEdge from(int lane) const {
    AlignEdge e;
    e.v = __shfl_sync(FULL, v, lane);
    return e;
  }
};
template <> struct AlignEdge<false> {
  int2 v;
  __device__ __forceinline__ AlignEdge() {}
  __device__ __forceinline__ AlignEdge(int h, int f) : v(make_int2(h, f)) {}
  __device__ __forceinline__ int h() const { return v.x; }
  __device__ __forceinline__ int f() const { return v.y; }
  __device__ __forceinline__ AlignEdge from(int lane) const {
    return AlignEdge(__shfl_sync(FULL, v.x, lane), __shfl_sync(FULL, v.y, lane));
  }
};

// What a warp's stage reads step by step, written at its start: of the last 64
// columns the offset of their code's profile rows, twice over so that a lane's
// columns of a stage are contiguous, and the border row's edges.
template <bool KEEP_H>
struct __align__(16) AlignFeed {
  uint16_t code[128];
  AlignEdge<KEEP_H> edge[ASTAGE];
};

// A team of W warps, AT query rows per lane: as many warps as there is room
// for and few rows for a call of few pairs, whose steps are then short; a block
// is a team, or four teams of one warp.  The cells of a lane's rows at one step
// are one word.  Teams of four take eight rows with bits, whose calls are large
// (600 pairs of 3,000 x 3,000: 6.8 ms, 7.2 with four).
template <int W, bool KEEP_H>
struct AlignShape {
  static constexpr int AT = W == 16 || (W == 4 && KEEP_H) ? 4 : 8;
  static constexpr int ROWS = 32 * AT;  // rows per pass
  static constexpr int PROFILE = NCODES * 32 * AT;
  static constexpr int TEAMS = W == 1 ? 4 : 1;
  static constexpr int WARPS = W * TEAMS;
};
template <int AT, bool KEEP_H> struct AlignWord;
template <> struct AlignWord<4, false> { typedef uint16_t type; };
template <> struct AlignWord<8, false> { typedef uint32_t type; };
template <> struct AlignWord<4, true> { typedef uint2 type; };
template <> struct AlignWord<8, true> { typedef uint4 type; };

// Word (pass p, step t, lane k) holds the cells of the lane's AT rows at
// column t - k: their H, 16 bits each, first row lowest (KEEP_H), or four
// fields of AT bits, with row r at bit AT - 1 - r of each.  A pass runs whole
// stages of steps.
// Fields 0 and 1 tell the source of H (where it is not 0): (1, 0) diagonal,
// (0, 1) E, (0, 0) F; field 2: E of the next column opens here; field 3: F
// of the next row opens here.
__device__ __forceinline__ int64_t bits_word(int n, int p, int t, int lane) {
  return ((int64_t)p * align_stages(n) * ASTAGE + t) * 32 + lane;
}

__device__ __forceinline__ bool end_before(int v, int i, int j, int bv, int bi, int bj) {
  return v > bv || (v == bv && (i < bi || (i == bi && j < bj)));
}

// Edges of a border row: a pass's steps, and 31 columns that it does not reach.
__host__ __device__ __forceinline__ int64_t align_border_row(int n) {
  return (int64_t)align_stages(n) * ASTAGE + 32;
}

// The lane's profile words of one code, its rows at lp.
template <int AT>
__device__ __forceinline__ void lane_words(uint32_t (&w)[AT / 4], const uint8_t* lp) {
  if constexpr (AT == 8) {
    const uint2 v = *(const uint2*)lp;
    w[0] = v.x, w[1] = v.y;
  } else {
    w[0] = *(const uint32_t*)lp;
  }
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
//
// Lane k scores column t - k at step t.  A step's edge goes one lane down, and
// from the pass above to lane 0, in one rotation: lane 31 sends the border
// row's.  The border row holds the pass's edges by step, column j's at j + 31.
template <int W, bool KEEP_H, typename Word, typename Barrier>
__device__ __forceinline__ AlignBest align_forward(const DbView& db,
                                                   const SearchParams* __restrict__ P,
                                                   const AlignItem& it, uint8_t* prof,
                                                   const uint8_t* sm, int lane, int warp,
                                                   Word* bits, AlignEdge<KEEP_H>* border,
                                                   AlignFeed<KEEP_H>& feed, Barrier barrier) {
  typedef AlignEdge<KEEP_H> Edge;
  constexpr int AT = AlignShape<W, KEEP_H>::AT, AROWS = AlignShape<W, KEEP_H>::ROWS;
  const int go = P->go, ge = P->ge;
  const int m = P->qlen[it.q];
  const int n = db.clen[it.s];
  const uint8_t* __restrict__ qr = P->qres + P->qoff[it.q];
  const uint8_t* __restrict__ d = db.cont + db.coff[it.s];
  const int64_t row = align_border_row(n);
  Edge* own = border + it.border_off + warp * row;
  const Edge* src = border + it.border_off + (warp + W - 1) % W * row;
  const int npass = n > 0 ? (m + AROWS - 1) / AROWS : 0;
  const int spass = align_stages(n);
  const int period = max(spass, ALAG * W);
  const int nstages =
      npass > 0 ? ((npass - 1) / W) * period + ((npass - 1) % W) * ALAG + spass : 0;
  const Edge top(0, -go);
  const int from = (lane + 31) & 31;
  const uint8_t* pl = prof + lane * AT;
  AlignBest best{0, INT32_MAX, INT32_MAX};
  // Largest H of each row of the pass and the first step that held it, one key
  // where 16 bits hold both.
  int rv[AT], rt[AT];
  int H[AT], E[AT], hdiag = 0;
  Edge out = top, edge_next = top;
  // the code and the edge that this lane, one of the first ASTAGE, brings to the next stage
  int code_next = PAD_CODE;
  auto fetch = [&](int p, int k) {
    const int j = ASTAGE * k + lane;
    code_next = j < n ? d[j] : PAD_CODE;
    if (p > 0) edge_next = src[j + 31];
  };
  int p = 0;
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
        for (int r = 0; r < AT; r++) H[r] = E[r] = rv[r] = rt[r] = 0;
        hdiag = 0;
        out = top;
        feed.code[32 + lane] = feed.code[96 + lane] = PAD_CODE * 32 * AT;  // columns -32..-1
        edge_next = top;
        if (lane < ASTAGE) fetch(p, 0);
      }
      const bool last_pass = (p == npass - 1);
      const int t0 = ASTAGE * k;
      const bool keep_border = !last_pass && lane == 31;
      Word* wp = bits + bits_word(n, p, t0, lane);
      if (lane < ASTAGE) {
        const int i = (t0 + lane) & 63;
        feed.code[i] = feed.code[i + 64] = code_next * (32 * AT);
        feed.edge[lane] = edge_next;
        if (k + 1 < spass) fetch(p, k + 1);
      }
      __syncwarp();
      const uint16_t* code = feed.code + ((t0 - lane) & 63);
      uint32_t next[AT / 4];
      lane_words<AT>(next, pl + code[0]);
#pragma unroll
      for (int u = 0; u < ASTAGE; u++) {
        const int t = t0 + u;
        uint32_t pw[AT / 4];
#pragma unroll
        for (int r = 0; r < AT / 4; r++) pw[r] = next[r];
        if (u + 1 < ASTAGE) lane_words<AT>(next, pl + code[u + 1]);
        const Edge in = (lane == 31 ? feed.edge[u] : out).from(from);
        // Cells before the subject leave H and E at 0.  Those past it or past
        // the query hold no more than one before them in row-major order.
        int hd = hdiag, f = in.f();
        hdiag = in.h();
        // signs: H above the diagonal term, above E; H - Go below the next E,
        // below the next F
        uint32_t sa = 0, sb = 0, se = 0, sf = 0;
#pragma unroll
        for (int r = 0; r < AT; r++) {
          const int e = E[r];  // floored at 0: only cells with E > 0 matter to the walk
          const int x = __dp4a((int)pw[r / 4], 1 << (8 * (r & 3)), hd);
          const int y = max(x, e), h = max(y, f);               // Eq. 1
          hd = H[r];
          H[r] = h;
          const int tt = h - go;
          E[r] = __viaddmax_s32_relu(e, -ge, tt);               // Eq. 2, next column
          f = __viaddmax_s32(f, -ge, y - go);                   // Eq. 3, next row: Go >= Ge
          if constexpr (KEEP_H) {
            rv[r] = max(rv[r], h * 65536 + (0xffff - t));
          } else {
            sa = push_sign(sa, x - h);
            sb = push_sign(sb, e - h);
            se = push_sign(se, tt - E[r]);
            sf = push_sign(sf, tt - f);
            rt[r] = h > rv[r] ? t : rt[r];
            rv[r] = max(rv[r], h);
          }
        }
        out = Edge(H[AT - 1], f);
        constexpr uint32_t F = (1u << AT) - 1;
        if constexpr (!KEEP_H)
          wp[32 * u] = (Word)((~sa & F) | (~sb & sa & F) << AT | (~se & F) << 2 * AT |
                              (~sf & F) << 3 * AT);
        else if constexpr (AT == 4)
          wp[32 * u] = make_uint2(prmt(H[0], H[1], 0x5410u), prmt(H[2], H[3], 0x5410u));
        else
          wp[32 * u] = make_uint4(prmt(H[0], H[1], 0x5410u), prmt(H[2], H[3], 0x5410u),
                                  prmt(H[4], H[5], 0x5410u), prmt(H[6], H[7], 0x5410u));
        if (keep_border) own[t] = out;
      }
      if (k == spass - 1) {
        if (!last_pass && lane < 31) own[ASTAGE * spass + lane] = top;  // of columns not reached
#pragma unroll
        for (int r = 0; r < AT; r++) {
          const int v = KEEP_H ? rv[r] >> 16 : rv[r], t = KEEP_H ? 0xffff - (rv[r] & 0xffff) : rt[r];
          if (v > 0) best.take(v, p * AROWS + lane * AT + r + 1, t - lane + 1);
        }
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

__device__ __forceinline__ void align_write(const AlignItem& it, const AlignBest& best, int lane,
                                            int i, int j, int64_t pos, AlignOut* out) {
  if (lane != 0) return;
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

// The walk back from `best` over stored H, on one warp.  v is H of the current
// cell.
template <int W>
__device__ __forceinline__ void align_traceback_h(const DbView& db,
                                                  const SearchParams* __restrict__ P,
                                                  const AlignItem& it, const AlignBest& best,
                                                  const uint8_t* sm, int lane, const uint16_t* hs,
                                                  uint8_t* ops, AlignOut* out) {
  constexpr int AT = AlignShape<W, true>::AT, AROWS = AlignShape<W, true>::ROWS;
  const int m = P->qlen[it.q];
  const int n = db.clen[it.s];
  const int go = P->go, ge = P->ge;
  const uint8_t* __restrict__ qr = P->qres + P->qoff[it.q];
  const uint8_t* __restrict__ d = db.cont + db.coff[it.s];
  int64_t pos = it.ops_end;  // the transcript is written backwards, ending here
  int i = best.i, j = best.j, v = best.v;
  auto cell = [&](int ci, int cj) -> int {  // H, 0 on row and column 0 and beyond
    if (ci < 1 || cj < 1) return 0;
    const int row = ci - 1, l = row % AROWS / AT;
    return hs[bits_word(n, row / AROWS, cj - 1 + l, l) * AT + row % AT];
  };
  // The nearest cell k >= 1 to the left in the row (up in the column) with H =
  // v + Go + (k - 1) Ge, or 0; no H exceeds best.v.  128 cells at a time.
  auto opening = [&](bool left) -> int {
    const int room = best.v - v - go;
    if (room < 0) return 0;
    const int cells = (left ? j : i) - 1;
    const int last = ge > 0 ? min(cells, room / ge + 1) : cells;
    for (int k0 = 1; k0 <= last; k0 += 128) {
      int h[4];
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int k = k0 + 32 * u + lane;
        h[u] = k <= last ? cell(left ? i : i - k, left ? j - k : j) : -1;
      }
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const int k = k0 + 32 * u + lane;
        const unsigned hit = __ballot_sync(FULL, k <= last && h[u] == v + go + (k - 1) * ge);
        if (hit) return k0 + 32 * u + __ffs(hit) - 1;
      }
    }
    return 0;
  };
  // every round takes at least one column; the bound only guards against
  // broken cells
  for (int64_t guard = 0; v > 0 && guard < 2 * ((int64_t)m + n) + 2; guard++) {
    const int ci = i - lane, cj = j - lane;
    const bool in = ci >= 1 && cj >= 1;
    const int h = cell(ci, cj);
    int next = __shfl_down_sync(FULL, h, 1);  // the cell above and left
    const int beyond = lane == 31 ? cell(ci - 1, cj - 1) : 0;
    if (lane == 31) next = beyond;
    const int w = in ? (int)(int8_t)sm[qr[ci - 1] * SM_ROW + d[cj - 1]] : 0;
    const uint32_t other = __ballot_sync(FULL, !in || next + w != h);
    const uint32_t zero = __ballot_sync(FULL, next == 0);
    const int first = other ? __ffs(other) - 1 : 32;  // not from the diagonal
    const int end = zero ? __ffs(zero) : 33;          // columns to the cell whose H is 0
    const int run = min(first, end);
    if (lane < run) ops[pos - 1 - lane] = 'M';
    if (run > 0) v = __shfl_sync(FULL, next, run - 1);
    pos -= run;
    i -= run;
    j -= run;
    if (v == 0 || first == 32) continue;
    // a gap ends in this cell
    int k = opening(true);
    const bool left = k > 0;
    if (!left) k = opening(false);
    if (k == 0) break;  // broken cells
    for (int u = lane; u < k; u += 32) ops[pos - 1 - u] = left ? 'D' : 'I';
    pos -= k;
    (left ? j : i) -= k;
    v += go + (k - 1) * ge;
  }
  align_write(it, best, lane, i, j, pos, out);
}

// The walk back from `best` over stored bits, on one warp.  v is H (or E or F)
// of the current cell, which the matrix and the penalties give step by step.
template <int W, typename Word>
__device__ __forceinline__ void align_traceback(const DbView& db,
                                                const SearchParams* __restrict__ P,
                                                const AlignItem& it, const AlignBest& best,
                                                const uint8_t* sm, int lane, const Word* bits,
                                                uint8_t* ops, AlignOut* out) {
  constexpr int AT = AlignShape<W, false>::AT, AROWS = AlignShape<W, false>::ROWS;
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
  align_write(it, best, lane, i, j, pos, out);
}

template <int W, bool KEEP_H>
__global__ void __launch_bounds__(AlignShape<W, KEEP_H>::WARPS * 32)
align_kernel(DbView db, const SearchParams* __restrict__ P, const AlignItem* __restrict__ items,
             int n_items, uint8_t* bits, int2* border, AlignOut* out, uint8_t* ops) {
  constexpr int TEAMS = AlignShape<W, KEEP_H>::TEAMS;
  typedef typename AlignWord<AlignShape<W, KEEP_H>::AT, KEEP_H>::type Word;
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ __align__(16) uint8_t sm[NCODES * SM_ROW];
  __shared__ AlignFeed<KEEP_H> feed[AlignShape<W, KEEP_H>::WARPS];
  __shared__ AlignBest red[W];
  for (int i = threadIdx.x; i < NCODES * SM_ROW; i += blockDim.x)
    sm[i] = i % SM_ROW < NCODES ? (uint8_t)P->sm[i / SM_ROW * NCODES + i % SM_ROW] : 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, warp = wib % W;
  uint8_t* prof = smem + wib * AlignShape<W, KEEP_H>::PROFILE;
  // uniform over the team
  for (int k = blockIdx.x * TEAMS + wib / W; k < n_items; k += gridDim.x * TEAMS) {
    const AlignItem it = items[k];
    Word* words = (Word*)(bits + it.bits_off);
    AlignBest best = align_forward<W, KEEP_H>(db, P, it, prof, sm, lane, warp, words,
                                              (AlignEdge<KEEP_H>*)border, feed[wib], []() {
      if constexpr (W > 1) __syncthreads();
      else __syncwarp();
    });
    if constexpr (W > 1) {
      if (lane == 0) red[warp] = best;
      __syncthreads();
      if (warp == 0)
        for (int w = 1; w < W; w++) best.take(red[w].v, red[w].i, red[w].j);
    }
    if (warp == 0) {
      if constexpr (KEEP_H)
        align_traceback_h<W>(db, P, it, best, sm, lane, (const uint16_t*)words, ops, out + k);
      else
        align_traceback<W>(db, P, it, best, sm, lane, words, ops, out + k);
    }
    if constexpr (W > 1) __syncthreads();  // red is rewritten by the next pair
  }
}

// 16 warps to a pair while there are SMs for every pair, 4 while those teams
// (near enough) fit the chip at once, then one.
int align_team(int n_pairs, int sms) { return n_pairs <= sms ? 16 : n_pairs <= 16 * sms ? 4 : 1; }

template <int W, bool KEEP_H>
static cudaError_t launch_team(int sms, const DbView& db, const SearchParams* params,
                               const AlignItem* items, int n_items, uint8_t* bits, int2* border,
                               AlignOut* out, uint8_t* ops, cudaStream_t stream) {
  const int smem = AlignShape<W, KEEP_H>::WARPS * AlignShape<W, KEEP_H>::PROFILE;
  cudaError_t e =
      cudaFuncSetAttribute(align_kernel<W, KEEP_H>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           smem);
  if (e != cudaSuccess) return e;
  const int teams = AlignShape<W, KEEP_H>::TEAMS;
  cudaGetLastError();  // a stale error must not be read as this launch's
  const int blocks = std::min((n_items + teams - 1) / teams, std::max(sms, 1) * 16);
  align_kernel<W, KEEP_H><<<blocks, AlignShape<W, KEEP_H>::WARPS * 32, smem, stream>>>(
      db, params, items, n_items, bits, border, out, ops);
  return cudaGetLastError();
}

cudaError_t launch_align(int team, bool keep_h, int sms, const DbView& db, const SearchParams* params,
                         const AlignItem* items, int n_items, uint8_t* bits, int2* border,
                         AlignOut* out, uint8_t* ops, cudaStream_t stream) {
  if (n_items <= 0) return cudaSuccess;
  auto launch = keep_h ? team == 16 ? launch_team<16, true> : team == 4 ? launch_team<4, true>
                                                                        : launch_team<1, true>
                       : team == 16 ? launch_team<16, false> : team == 4 ? launch_team<4, false>
                                                                         : launch_team<1, false>;
  return launch(sms, db, params, items, n_items, bits, border, out, ops, stream);
}

int64_t align_border_ints(int team, int32_t n) { return n > 0 ? team * align_border_row(n) : 0; }

int64_t align_bits_bytes(int team, bool keep_h, int32_t m, int32_t n) {
  if (m <= 0 || n <= 0) return 0;
  const int at = team == 16 ? AlignShape<16, true>::AT
                 : team == 4 ? (keep_h ? AlignShape<4, true>::AT : AlignShape<4, false>::AT)
                             : AlignShape<1, true>::AT;
  return (int64_t)((m + 32 * at - 1) / (32 * at)) * align_stages(n) * ASTAGE * 32 *
         (keep_h ? 2 * at : at / 2);
}

}  // namespace swgb
