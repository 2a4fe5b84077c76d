// lane_kernel.cuh -- packed 16-bit scores of (query, subject pair) items on
// groups of 8, 16 or 32 lanes.
//
// A lane group scores two subjects, adjacent in length order, as the two
// halves of every word.  Lane k of the group owns PR consecutive query rows in
// registers and updates column t - k at step t, one whole column of its rows;
// it takes the (H, F) border of the row above from lane k - 1 by shuffle
// (Section II-B: intra-task parallelism with neighbour border exchange).  A
// query of up to LG x PR rows needs no border memory at all; a longer one runs
// in passes of 32 x PR rows whose border row goes through this warp's scratch.
//
// Why lane groups: one warp that sweeps 64 subjects with 32 rows in each lane
// has the lowest cost per column, but its item takes (query / 32 rows) x
// (subject columns) x 32 rows one after the other, and a search with few
// queries has too few of those items for 152 SMs and ends on the longest one.
// With a group per subject pair an item is 8 to 32 times shorter, so a search
// of some thousand subjects already fills the chip, and the ends of a large
// one are short.  What the group costs is the ramp, LG - 1 steps per subject
// pair, and two shuffles, two residue loads and the profile loads per step of
// PR words.  Measured on one GB300 (wall time of the search):
//   1 query of 144 x 2,000 subjects      1.27 -> 0.12 ms
//   1 query of 375 x 20,000              6.04 -> 0.46 ms
//   1 query of 375 x 570,000             15.4 -> 10.9 ms
//   7 queries of 140-600 x 40,000        15.0 ->  6.5 ms
// (before: a warp per 64 subjects, and a warp per subject pair above 1,500
// residues.)  For many subjects of a few tens of residues the ramp is most of an
// item, and a warp per 64 of them is the faster one (inter_kernel.cu).
//
// An item that would outlast the search (a long subject in a small search, a
// long query against few subjects) is cut further: into chains, the query's
// passes on the four warps of a block, each a few stages behind the one above
// (4 queries x 500 subjects, all of 5,000-35,000 residues: 323 ms with the
// passes one after the other, 165 with chains of 8 rows per lane and 156 of 16,
// whose step overhead is spread over twice the words); and each lane's rows
// into halves one column apart, two independent chains of cells for a warp
// alone on its scheduler (1 query of 144 x 2,000: 0.100 -> 0.081 ms of kernel
// time).  Chains of 32 rows measured 188 ms: their profiles leave room for 8
// warps per SM, too few.
// The kernel is bound by the ALU pipe: 4.5 operations per word (packed_cell
// and the merge of the two subjects' profile bytes).
//
// Rows per lane come in steps of 2 where a group holds the whole query, of 4 in
// passes: 3 queries of 66 residues x 549,000 subjects 11.8 ms with steps of 4
// throughout, 10.1 so (80 rows swept instead of 96); 7 queries of 140-600 x
// 40,000 6.75 and 6.5.  Passes in steps of 2 as well measured 1 to 3% less for
// those and 3% more for the rest, by the size of the kernel.
//
// Columns left and right of a subject hold the padding code, whose score of
// -64 leaves H = E = 0 before the first column and raises no S after the last,
// so no step tests its column.  The lanes of a warp walk in step; the items of
// a block's warps are neighbours in length order and share one query profile.
#pragma once

#include "lane_profile.cuh"

namespace swgb {

// Dynamic shared memory: one residue ring per warp, then the block's query
// profile (lane_profile.cuh; for chained passes, one per warp).  Ring: per
// group two blocks of 8 * LG columns, as the byte
// offsets (code x 32 * PW) of the two subjects' profile rows, 16 bits each;
// the first 8 columns are repeated after the last, so 8 steps need one wrap.
constexpr int LANE_PROFILE = NCODES * 32 * LANE_ROWS_MAX;
constexpr int LANE_RING = 4 * (2 * 256 + 32);  // bytes per warp: 2 * 8 * 32 columns and the repeats
constexpr int LANE_RINGS = LANE_WARPS * LANE_RING;
constexpr int LANE_SMEM = LANE_RINGS + LANE_PROFILE;
constexpr int LANE_SMEM_WIDE = LANE_RINGS + LANE_WARPS * LANE_PROFILE / 2;  // chains of 16 rows
constexpr int EDGE_STAGE = 32;  // steps of a stage: a chain's block barriers lie between
constexpr int EDGE_PAD = 64;    // a border row holds column j at EDGE_PAD + j
// Stages between the starts of a chain's consecutive passes of `full` rows per
// lane (4, or 8 and 16 in halves).
__host__ __device__ __forceinline__ constexpr int chain_lag(int full) { return full == 4 ? 3 : 4; }
// Stages of a pass of pr rows per lane over n columns.
__host__ __device__ __forceinline__ constexpr int chain_stages(int pr, int n) {
  return (n + (pr == 4 ? 31 : 63) + EDGE_STAGE - 1) / EDGE_STAGE;
}
// A warp's stage of border columns, and what its last steps read ahead.
struct LaneEdge {
  uint2 col[EDGE_STAGE + 4];
};

// Profile words of one column of a quarter: four rows to a word, per subject.
template <int PR, int NQ>
struct LaneWords {
  static constexpr int RW = LaneShape<PR, NQ>::RW, VB = LaneShape<PR, NQ>::VB;
  uint32_t a[RW], b[RW];

  // pa, pb: the lane's profile rows of the two codes; q: the quarter
  __device__ __forceinline__ void load(const uint8_t* pa, const uint8_t* pb, int q) {
#pragma unroll
    for (int v = 0; v < 4 * RW / VB; v++) {
      const int o = (q * (4 * RW / VB) + v) * 32 * VB;
      if constexpr (VB == 16) {
        const uint4 x = *(const uint4*)(pa + o), y = *(const uint4*)(pb + o);
        a[4 * v] = x.x, a[4 * v + 1] = x.y, a[4 * v + 2] = x.z, a[4 * v + 3] = x.w;
        b[4 * v] = y.x, b[4 * v + 1] = y.y, b[4 * v + 2] = y.z, b[4 * v + 3] = y.w;
      } else if constexpr (VB == 8) {
        const uint2 x = *(const uint2*)(pa + o), y = *(const uint2*)(pb + o);
        a[2 * v] = x.x, a[2 * v + 1] = x.y;
        b[2 * v] = y.x, b[2 * v + 1] = y.y;
      } else {
        a[v] = *(const uint32_t*)(pa + o);
        b[v] = *(const uint32_t*)(pb + o);
      }
    }
  }
};

// One column of quarter q's rows; hd: H above and left of its first row, f: F
// of its first row, then of the row below its last.
template <int PR, int NQ>
__device__ __forceinline__ void lane_column(uint32_t (&H)[PR], uint32_t (&E)[PR], int q,
                                            uint32_t& smax, uint32_t hd, uint32_t& f,
                                            const LaneWords<PR, NQ>& w, uint32_t GO2,
                                            uint32_t NGE2) {
  constexpr int R = LaneShape<PR, NQ>::R;
  uint32_t xp = 0;
#pragma unroll
  for (int i = 0; i < R; i++) {
    const int r = q * R + i;
    uint32_t x;
    const uint32_t h = packed_cell(hd, prmt(w.a[i / 4], w.b[i / 4], sext_pair_sel(i & 3)), E[r], f,
                                   x, GO2, NGE2);
    hd = H[r];
    H[r] = h;
    if (i & 1)
      smax = __vimax3_s16x2(smax, xp, x);
    else
      xp = x;
  }
}

// How a pass meets the one before: alone (the whole query), one after the
// other on one warp, or chained, on another warp of the block.
enum { ALONE = 0, SERIAL = 1, CHAINED = 2 };

// All warps of the block have finished the stage.  The warps of a chain meet
// here from different places of the code, so it is a barrier of its own.
__device__ __forceinline__ void chain_barrier() {
  asm volatile("bar.sync 1, %0;" ::"n"(LANE_WARPS * 32) : "memory");
}

// One pass of the lane's rows over its group's subject pair.  n: columns of
// the warp's longest subject (uniform over the warp); src: the pair's first
// 16-byte chunk of 8 + 8 residues, one every 512 bytes, `chunks` of them.
// Quarter q of lane k updates column t - NQ k - q at step t; it takes what the
// quarter above (the last one of lane k - 1 for q = 0) left at step t - 1.
// With several passes LG is 32, hb_in holds the border row below the pass
// before (unless this is the first) and hb_out takes this pass's (unless it is
// the last): lane 31 writes column j at step j + 32 NQ - 1.  The steps go by
// stages of EDGE_STAGE columns, which the warp fetches a stage ahead and keeps
// in `edge`; a column goes to lane 0 in the rotation that takes the lanes'
// edges one lane down, as lane 31's.  SERIAL: hb_in and hb_out are one row.
// CHAINED: after every stage the block's warps meet at a barrier, and the pass
// before, on another warp, is chain_lag stages ahead: the columns up to 32 k +
// 63 that stage k fetches were written by that pass's step 32 k + 62 + 32 NQ at
// the latest, in its stage k + 1 + NQ, which ended before this stage began.
// (With each step fetching its own border column 4 steps ahead and testing it,
// a chain's step took 124 cycles for 4 rows on a scheduler of its own and 279
// with four warps, 143 and 437 for 8 rows; now 118 and 261, 123 and 409.)
template <int PR, int NQ, int MODE>
__device__ __forceinline__ void lane_sweep(const uint8_t* prof, uint8_t* ring, int lane, int lg,
                                           int n, const uint4* src, int chunks, LaneEdge* edge,
                                           const uint2* hb_in, uint2* hb_out, bool first, bool last, uint32_t& smax,
                                           uint32_t GO2, uint32_t NGE2) {
  constexpr bool PASSES = MODE != ALONE;
  constexpr int U = LaneShape<PR, NQ>::UNROLL;
  constexpr bool AHEAD = LaneShape<PR, NQ>::AHEAD;
  constexpr uint32_t CODE = 32 * LaneShape<PR, NQ>::PW;  // bytes between the profile rows of two codes
  const int li = lane & (lg - 1);
  const int cols = 8 * lg;  // columns per ring block
  // this group's ring: 2 * cols columns and the repeats, 4 bytes each; the
  // gap to the next group's keeps the groups' reads on distinct banks
  uint8_t* gr = ring + (lane / lg) * 4 * (2 * cols + (lg == 8 ? 8 : 16));
  const uint32_t not0 = li == 0 ? 0u : 1u;
  const uint8_t* pl = prof + lane * LaneShape<PR, NQ>::VB;
  uint32_t H[PR], E[PR];
#pragma unroll
  for (int r = 0; r < PR; r++) H[r] = E[r] = 0u;  // H(i, 0) = 0; any E(i, 1) <= 0 will do
  // per quarter: H below its rows one and two steps back, F one step back,
  // and the profile rows of its column's codes
  uint32_t hdiag = 0u, h1[NQ], h2[NQ], f1[NQ];
  const uint8_t *pa[NQ], *pb[NQ];
#pragma unroll
  for (int q = 0; q < NQ; q++) {
    h1[q] = h2[q] = f1[q] = 0u;
    pa[q] = pb[q] = pl + PAD_CODE * CODE;
  }
  const uint4 pad = make_uint4(0x18181818u, 0x18181818u, 0x18181818u, 0x18181818u);
  static_assert(PAD_CODE == 0x18, "the padding chunk");
  // this lane's 8 columns of a ring block
  auto store = [&](int slot, const uint4& v) {
    uint32_t w[8];
#pragma unroll
    for (int c = 0; c < 8; c++) {
      const uint32_t a = prmt(c < 4 ? v.x : v.y, 0u, 0x4440u + (c & 3));
      const uint32_t b = prmt(c < 4 ? v.z : v.w, 0u, 0x4440u + (c & 3));
      w[c] = imad(a, CODE, imad(b, CODE << 16, 0u));
    }
    const uint4 lo = make_uint4(w[0], w[1], w[2], w[3]), hi = make_uint4(w[4], w[5], w[6], w[7]);
    uint4* dst = (uint4*)(gr + 4 * (slot * cols + 8 * li));
    dst[0] = lo;
    dst[1] = hi;
    if (slot == 0 && li == 0) {
      dst = (uint4*)(gr + 4 * 2 * cols);
      dst[0] = lo;
      dst[1] = hi;
    }
  };
  auto load = [&](int b) {
    const int c = b * lg + li;
    return c < chunks ? ldg_nc(src + (int64_t)c * 32) : pad;
  };
  __syncwarp();
  store(1, pad);  // the columns left of the first
  uint4 next = load(0);
  const int steps = n + NQ * lg - 1;
  const uint32_t mask = (uint32_t)(4 * (2 * cols - 1));
  const int span = PASSES ? EDGE_STAGE : cols;
  // columns past the end are zeros, like those above the first pass
  auto border = [&](int c) {
    return !first && c < n ? hb_in[EDGE_PAD + c] : make_uint2(0u, 0u);
  };
  uint2 edge_next;
  if constexpr (PASSES) edge_next = border(lane);
  const int from = (lane + 31) & 31;
  const bool keep = lane == 31 && !last;
  int b = 0;
  for (int t0 = 0; t0 < steps; t0 += span) {
    if (!PASSES || (t0 & (cols - 1)) == 0) {
      __syncwarp();
      store(b & 1, next);
      next = load(++b);
      __syncwarp();
    }
    const int tend = min(t0 + span, steps);
    uint2 bq[U];  // the border of columns t .. t + U - 1
    if constexpr (PASSES) {
      static_assert(U <= 4, "columns read ahead");
      __syncwarp();
      edge->col[lane] = edge_next;
      edge_next = border(t0 + EDGE_STAGE + lane);
      __syncwarp();
#pragma unroll
      for (int u = 0; u < U; u++) bq[u] = edge->col[u];
    }
    // the profile words of step t are loaded one step ahead; the last step of
    // a ring block reads whatever code the slot holds, and is read again here
    LaneWords<PR, NQ> w[NQ];
    auto fetch = [&](const uint8_t* rp) {
      const uint8_t *a = pl + *(const uint16_t*)rp, *b = pl + *(const uint16_t*)(rp + 2);
      w[0].load(a, b, 0);
#pragma unroll
      for (int q = 1; q < NQ; q++) w[q].load(pa[q - 1], pb[q - 1], q);
    };
    if constexpr (AHEAD) fetch(gr + ((uint32_t)(4 * (t0 - NQ * li)) & mask));
#pragma unroll 1
    for (int t = t0; t < tend; t += U) {
      const uint8_t* rp = gr + ((uint32_t)(4 * (t - NQ * li)) & mask);
#pragma unroll
      for (int u = 0; u < U; u++) {
        // the row above: lane k - 1's bottom row, H = F = 0 above the matrix
        uint32_t in_h, in_f;
        if constexpr (PASSES) {
          in_h = __shfl_sync(FULL, lane == 31 ? bq[u].x : h1[NQ - 1], from);
          in_f = __shfl_sync(FULL, lane == 31 ? bq[u].y : f1[NQ - 1], from);
          bq[u] = edge->col[t - t0 + u + U];
        } else {
          in_h = imad(__shfl_up_sync(FULL, h1[NQ - 1], 1, lg), not0, 0u);
          in_f = imad(__shfl_up_sync(FULL, f1[NQ - 1], 1, lg), not0, 0u);
        }
        if constexpr (!AHEAD) fetch(rp + 4 * u);
        LaneWords<PR, NQ> now[NQ];
#pragma unroll
        for (int q = 0; q < NQ; q++) now[q] = w[q];
#pragma unroll
        for (int q = NQ - 1; q > 0; q--) {
          pa[q] = pa[q - 1];
          pb[q] = pb[q - 1];
        }
        if constexpr (NQ > 1) {
          pa[0] = pl + *(const uint16_t*)(rp + 4 * u);
          pb[0] = pl + *(const uint16_t*)(rp + 4 * u + 2);
        }
        if constexpr (AHEAD) fetch(rp + 4 * (u + 1));
        uint32_t nh[NQ], nf[NQ];
#pragma unroll
        for (int q = 0; q < NQ; q++) {
          nf[q] = q == 0 ? in_f : f1[q - 1];
          lane_column<PR, NQ>(H, E, q, smax, q == 0 ? hdiag : h2[q - 1], nf[q], now[q], GO2, NGE2);
          nh[q] = H[(q + 1) * (PR / NQ) - 1];
        }
        hdiag = in_h;
#pragma unroll
        for (int q = 0; q < NQ; q++) {
          h2[q] = h1[q];
          h1[q] = nh[q];
          f1[q] = nf[q];
        }
        if constexpr (PASSES) {
          if (keep) hb_out[EDGE_PAD - (32 * NQ - 1) + t + u] = make_uint2(h1[NQ - 1], f1[NQ - 1]);
        }
      }
    }
    if constexpr (MODE == CHAINED) chain_barrier();
  }
}

// One warp's share of a block item: where its pairs lie.
struct LanePlace {
  int lg, n;         // lanes per group; columns of the warp's longest subject
  const uint4* src;  // this group's subject pair in the interleaved layout
  int chunks;
  LaneEdge* edge;    // the warp's
  uint2* hb;         // the warp's border row
};

// One pass, the rows [row0, row0 + lg x PR) of the query.  `build`: the block
// does not hold this profile yet (uniform over the block).
template <int PR, int NQ, int G>
__device__ __forceinline__ void lane_pass(const SearchParams* __restrict__ P, uint8_t* smem,
                                          const uint8_t* sm, const uint8_t* __restrict__ qr, int m,
                                          int row0, bool build, const LanePlace& at, int pass,
                                          int passes, uint32_t& smax) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint8_t *ring = smem + wib * LANE_RING, *prof = smem + LANE_RINGS;
  uint32_t GO2, NGE2;  // (Go, Go), (-Ge, -Ge)
  gap_words<G>(P, GO2, NGE2);
  if (build) {
    __syncthreads();  // every warp is done with the profile before
    lane_profile_rows<PR, NQ>(prof, sm, qr, m, row0, at.lg, wib, LANE_WARPS);
    __syncthreads();
  }
  if (at.n == 0) return;  // uniform over the warp
  if (passes == 1)
    lane_sweep<PR, NQ, ALONE>(prof, ring, lane, at.lg, at.n, at.src, at.chunks, nullptr, nullptr,
                              nullptr, true, true, smax, GO2, NGE2);
  else if constexpr (NQ == 1 && PR % 4 == 0)  // as the planner cuts a query of several passes
    lane_sweep<PR, 1, SERIAL>(prof, ring, lane, 32, at.n, at.src, at.chunks, at.edge, at.hb,
                              at.hb, pass == 0, pass == passes - 1, smax, GO2, NGE2);
}

// One pass of a chain, on this warp, with a profile of its own.
template <int PR, int NQ, int G>
__device__ __forceinline__ void chain_pass(const SearchParams* __restrict__ P, uint8_t* smem,
                                           const uint8_t* sm, const uint8_t* __restrict__ qr, int m,
                                           int row0, int slice, const LanePlace& at,
                                           const uint2* hb_in, bool first, bool last,
                                           uint32_t& smax) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint8_t *ring = smem + wib * LANE_RING, *prof = smem + LANE_RINGS + wib * slice;
  uint32_t GO2, NGE2;
  gap_words<G>(P, GO2, NGE2);
  __syncwarp();
  lane_profile_rows<PR, NQ>(prof, sm, qr, m, row0, 32, 0, 1);
  __syncwarp();
  lane_sweep<PR, NQ, CHAINED>(prof, ring, lane, 32, at.n, at.src, at.chunks, at.edge, hb_in, at.hb,
                              first, last, smax, GO2, NGE2);
}

// A chain: one subject pair on the whole block, for items that would take too
// long on one warp.  Warp w takes the passes w, w + LANE_WARPS, ...; pass p
// starts at stage (p / W) * period + (p % W) * lag with period the larger of a
// pass's stages and W * lag (lag = chain_lag), so consecutive passes are at least
// lag stages apart, and a warp's next pass starts after its previous one ends
// and at least W * lag stages after it started, when the pass that
// read the border row it will overwrite is further on.  Every warp meets the
// same number of barriers.
template <int G>
__device__ __forceinline__ void lane_chain(const DbView& db, const SearchParams* __restrict__ P,
                                           SearchState* st, const Scratch& scr, uint8_t* smem,
                                           const uint8_t* sm, uint32_t* red, const LaneSeg& sg,
                                           LaneEdge* edge, int unit) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int pair = sg.pair0 + unit;
  uint2* rows = scr.pair_border +
                (scr.lane_row0 + (int64_t)blockIdx.x * LANE_WARPS) * scr.pair_stride;
  LanePlace at;
  at.lg = 32;
  at.n = db.clen[2 * pair];
  at.src = (const uint4*)(db.inter + db.goff[pair / 32]) + (pair & 31);
  at.chunks = db.glen[pair / 32] / CHUNK;
  at.edge = edge + wib;
  at.hb = rows + wib * scr.pair_stride;
  const uint2* hb_in = rows + (wib + LANE_WARPS - 1) % LANE_WARPS * scr.pair_stride;
  const int m = P->qlen[sg.q];
  const uint8_t* __restrict__ qr = P->qres + P->qoff[sg.q];
  // stages of a pass of `full` rows (one of fewer steps waits out the rest)
  const int lag = chain_lag(sg.full), spass = chain_stages(sg.full, at.n);
  const int period = max(spass, LANE_WARPS * lag);
  const int end = (sg.passes - 1) / LANE_WARPS * period + (sg.passes - 1) % LANE_WARPS * lag + spass;
  uint32_t smax = 0u;
  if (at.n > 0) {  // uniform over the block
    int g = 0;
    for (int p = wib; p < sg.passes; p += LANE_WARPS) {
      for (const int start = p / LANE_WARPS * period + p % LANE_WARPS * lag; g < start; g++)
        chain_barrier();
      const bool last = p == sg.passes - 1;
      const int heads = sg.passes - sg.tail, slice = NCODES * 32 * sg.full;
      const int pr = p < heads ? sg.full : sg.pr;
      const int row0 = 32 * (p < heads ? p * sg.full : heads * sg.full + (p - heads) * sg.pr);
      switch (pr) {  // uniform over the warp
        case 4: chain_pass<4, 1, G>(P, smem, sm, qr, m, row0, slice, at, hb_in, p == 0, last, smax); break;
        case 8: chain_pass<8, 2, G>(P, smem, sm, qr, m, row0, slice, at, hb_in, p == 0, last, smax); break;
        default: chain_pass<16, 2, G>(P, smem, sm, qr, m, row0, slice, at, hb_in, p == 0, last, smax); break;
      }
      g += chain_stages(pr, at.n);
    }
    for (; g < end; g++) chain_barrier();
  }
  for (int o = 16; o > 0; o >>= 1) smax = __vmaxs2(smax, __shfl_xor_sync(FULL, smax, o));
  if (lane == 0) red[wib] = smax;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < LANE_WARPS; w++) smax = __vmaxs2(smax, red[w]);
    emit_pair(db, P, st, scr, sg.q, pair, smax);
  }
}

// One block item: LANE_WARPS x 32 / lg subject pairs of one segment.
// `cached` is the segment whose (single-pass) profile the block holds, or -1.
template <int G>
__device__ __forceinline__ void lane_item(const DbView& db, const SearchParams* __restrict__ P,
                                          SearchState* st, const Scratch& scr, uint8_t* smem,
                                          const uint8_t* sm, const LaneSeg& sg, int seg,
                                          int& cached, LaneEdge* edge, int unit) {
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  LanePlace at;
  at.lg = sg.lg;
  const int first = sg.pair0 + (unit * LANE_WARPS + wib) * (32 / sg.lg);  // the warp's first pair
  const int pair = first + lane / sg.lg;
  const bool has = pair < sg.pair1;
  at.n = first < sg.pair1 ? db.clen[2 * first] : 0;
  const int grp = (has ? pair : 0) / 32;
  at.src = (const uint4*)(db.inter + db.goff[grp]) + (pair & 31);
  at.chunks = has ? db.glen[grp] / CHUNK : 0;
  at.edge = edge + wib;
  at.hb = scr.pair_border +
          (scr.lane_row0 + (int64_t)blockIdx.x * LANE_WARPS + wib) * scr.pair_stride;
  const int m = P->qlen[sg.q];
  const uint8_t* __restrict__ qr = P->qres + P->qoff[sg.q];
  uint32_t smax = 0u;
  for (int p = 0; p < sg.passes; p++) {
    // every pass but the last has 32 rows per lane
    const int pr = p < sg.passes - 1 ? LANE_ROWS_MAX : sg.pr;
    const int row0 = p * 32 * LANE_ROWS_MAX;
    const bool build = sg.passes > 1 || cached != seg;
    switch (sg.halves ? -pr : pr) {  // uniform over the block
      case 4: lane_pass<4, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 6: lane_pass<6, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 8: lane_pass<8, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 10: lane_pass<10, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 12: lane_pass<12, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 14: lane_pass<14, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 16: lane_pass<16, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 18: lane_pass<18, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 20: lane_pass<20, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 22: lane_pass<22, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 24: lane_pass<24, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 26: lane_pass<26, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 28: lane_pass<28, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 30: lane_pass<30, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case -8: lane_pass<8, 2, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case -16: lane_pass<16, 2, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case -24: lane_pass<24, 2, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      default: lane_pass<32, 1, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
    }
  }
  cached = sg.passes > 1 ? -1 : seg;
  for (int o = sg.lg >> 1; o > 0; o >>= 1) smax = __vmaxs2(smax, __shfl_xor_sync(FULL, smax, o));
  if (has && (lane & (sg.lg - 1)) == 0) emit_pair(db, P, st, scr, sg.q, pair, smax);
}

template <int G>
__global__ void __launch_bounds__(LANE_WARPS * 32, 4)
lane_kernel(DbView db, const SearchParams* __restrict__ P, SearchState* st, Scratch scr) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ __align__(16) uint8_t sm[NCODES * SM_ROW];
  __shared__ unsigned long long s_item;
  __shared__ LaneEdge edge[LANE_WARPS];
  __shared__ uint32_t red[LANE_WARPS];
  const long long total = P->n_lane_items;
  for (int i = threadIdx.x; i < NCODES * SM_ROW; i += blockDim.x)
    sm[i] = i % SM_ROW < NCODES ? (uint8_t)P->sm[i / SM_ROW * NCODES + i % SM_ROW] : 0;
  const LaneSeg* __restrict__ segs = P->lane_segs;
  const int nseg = P->n_lane_segs;
  int cached = -1;
  __syncthreads();
  // The first item of a block is its index: consecutive blocks start on
  // different SMs, so a search of few items uses every SM (taken from the
  // counter, they all went to the blocks of the SMs that started first).
  for (long long it = blockIdx.x; it < total;) {  // uniform over the block
    int lo = 0, hi = nseg - 1;  // the last segment whose first item is at most `it`
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (segs[mid].first <= it)
        lo = mid;
      else
        hi = mid - 1;
    }
    const LaneSeg sg = segs[lo];
    if (sg.chain) {
      __syncthreads();  // every warp is done with the profile before
      lane_chain<G>(db, P, st, scr, smem, sm, red, sg, edge, (int)(it - sg.first));
      cached = -1;
    } else {
      lane_item<G>(db, P, st, scr, smem, sm, sg, lo, cached, edge, (int)(it - sg.first));
    }
    __syncthreads();  // the item before is read by all, and its chain is done
    if (threadIdx.x == 0) s_item = gridDim.x + atomicAdd(&st->lane_work, 1ull);
    __syncthreads();
    it = (long long)s_item;
  }
}

}  // namespace swgb
