// lane_kernel.cu -- packed 16-bit scores of (query, subject pair) items on
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
//   1 query of 375 x 20,000              6.04 -> 0.58 ms
//   1 query of 375 x 570,000             15.4 -> 10.9 ms
//   7 queries of 400 x 40,000            15.0 ->  7.3 ms
// (before: a warp per 64 subjects, and a warp per subject pair above 1,500
// residues.)
// The kernel is bound by the ALU pipe: 4.5 operations per word (packed_cell
// and the merge of the two subjects' profile bytes).
//
// Columns left and right of a subject hold the padding code, whose score of
// -64 leaves H = E = 0 before the first column and raises no S after the last,
// so no step tests its column.  The lanes of a warp walk in step; the items of
// a block's warps are neighbours in length order and share one query profile.
#include "device_common.cuh"

namespace swgb {

constexpr int LANE_ROWS_MAX = 32;
constexpr int SM_ROW = 28;  // bytes per row of the matrix copy: 25 scores, in whole words

// Dynamic shared memory: the block's query profile, then one residue ring per
// warp.  Profile of the 32 lanes' rows, int8, code-major:
//   rows [VB * v, VB * v + VB) of lane l against code c at
//   c * 32 * PR + v * 32 * VB + l * VB,   VB = bytes per load,
// so the lanes of a quarter- or half-warp read distinct banks whatever codes
// they read.  Ring: per group two blocks of 8 * LG columns, as the byte
// offsets (code x 32 * PR) of the two subjects' profile rows, 16 bits each;
// the first 8 columns are repeated after the last, so 8 steps need one wrap.
constexpr int LANE_PROFILE = NCODES * 32 * LANE_ROWS_MAX;
constexpr int LANE_RING = 4 * (2 * 256 + 32);  // bytes per warp: 2 * 8 * 32 columns and the repeats
constexpr int LANE_SMEM = LANE_PROFILE + LANE_WARPS * LANE_RING;

// 4 x 4 byte transpose: word b of the result holds byte b of a, b, c, d
__device__ __forceinline__ uint4 transpose4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  const uint32_t ab0 = prmt(a, b, 0x5140u), ab1 = prmt(a, b, 0x7362u);
  const uint32_t cd0 = prmt(c, d, 0x5140u), cd1 = prmt(c, d, 0x7362u);
  return make_uint4(prmt(ab0, cd0, 0x5410u), prmt(ab0, cd0, 0x7632u), prmt(ab1, cd1, 0x5410u),
                    prmt(ab1, cd1, 0x7632u));
}

template <int PR>
struct LaneShape {
  static_assert(PR % 4 == 0 && PR <= LANE_ROWS_MAX, "whole 4-row words, at most 32 rows");
  static constexpr int VB = PR % 16 == 0 ? 16 : PR % 8 == 0 ? 8 : 4;  // bytes per profile load
  static constexpr int UNROLL = PR >= 24 ? 2 : 4;                     // steps per loop body
  static constexpr bool AHEAD = PR <= 24;  // registers allow the next step's profile words
};

// The block's profile of rows [row0 + li * PR, ...) of query residues qr[0, m)
// for lanes li = l % lg.  Four rows and four codes at a time: one word of four
// scores per row, transposed into one word of four rows per code.
template <int PR>
__device__ __forceinline__ void lane_block_profile(uint8_t* prof, const uint8_t* sm,
                                                   const uint8_t* __restrict__ qr, int m, int row0,
                                                   int lg) {
  constexpr int VB = LaneShape<PR>::VB;
  const int l = threadIdx.x & 31;
  for (int rq = threadIdx.x >> 5; rq < PR / 4; rq += LANE_WARPS) {
    const int r0 = row0 + (l & (lg - 1)) * PR + 4 * rq;
    const uint8_t* s[4];
#pragma unroll
    for (int b = 0; b < 4; b++) s[b] = sm + (r0 + b < m ? (int)qr[r0 + b] : PAD_CODE) * SM_ROW;
    uint8_t* dst = prof + (4 * rq / VB) * 32 * VB + l * VB + (4 * rq) % VB;
#pragma unroll
    for (int cq = 0; cq < SM_ROW / 4; cq++) {
      const uint4 w = transpose4(*(const uint32_t*)(s[0] + 4 * cq), *(const uint32_t*)(s[1] + 4 * cq),
                                 *(const uint32_t*)(s[2] + 4 * cq), *(const uint32_t*)(s[3] + 4 * cq));
      const uint32_t v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int b = 0; b < 4; b++)
        if (4 * cq + b < NCODES) *(uint32_t*)(dst + (4 * cq + b) * 32 * PR) = v[b];
    }
  }
}

// The lane's profile words of one column: four rows to a word, per subject.
template <int PR>
struct LaneWords {
  uint32_t a[PR / 4], b[PR / 4];
};

template <int PR>
__device__ __forceinline__ void lane_words(LaneWords<PR>& w, const uint8_t* pa, const uint8_t* pb) {
  constexpr int VB = LaneShape<PR>::VB;
#pragma unroll
  for (int v = 0; v < PR / VB; v++) {
    if constexpr (VB == 16) {
      const uint4 x = *(const uint4*)(pa + v * 32 * VB), y = *(const uint4*)(pb + v * 32 * VB);
      w.a[4 * v] = x.x, w.a[4 * v + 1] = x.y, w.a[4 * v + 2] = x.z, w.a[4 * v + 3] = x.w;
      w.b[4 * v] = y.x, w.b[4 * v + 1] = y.y, w.b[4 * v + 2] = y.z, w.b[4 * v + 3] = y.w;
    } else if constexpr (VB == 8) {
      const uint2 x = *(const uint2*)(pa + v * 32 * VB), y = *(const uint2*)(pb + v * 32 * VB);
      w.a[2 * v] = x.x, w.a[2 * v + 1] = x.y;
      w.b[2 * v] = y.x, w.b[2 * v + 1] = y.y;
    } else {
      w.a[v] = *(const uint32_t*)(pa + v * 32 * VB);
      w.b[v] = *(const uint32_t*)(pb + v * 32 * VB);
    }
  }
}

// One column of the lane's PR rows.
template <int PR>
__device__ __forceinline__ void lane_column(uint32_t (&H)[PR], uint32_t (&E)[PR], uint32_t& smax,
                                            uint32_t hd, uint32_t& f, const LaneWords<PR>& w,
                                            uint32_t GO2, uint32_t NGE2) {
  uint32_t xp = 0;
#pragma unroll
  for (int r = 0; r < PR; r++) {
    uint32_t x;
    const uint32_t h = packed_cell(hd, prmt(w.a[r / 4], w.b[r / 4], sext_pair_sel(r & 3)), E[r], f,
                                   x, GO2, NGE2);
    hd = H[r];
    H[r] = h;
    if (r & 1)
      smax = __vimax3_s16x2(smax, xp, x);
    else
      xp = x;
  }
}

// One pass of the lane's rows over its group's subject pair.  n: columns of
// the warp's longest subject (uniform over the warp); src: the pair's first
// 16-byte chunk of 8 + 8 residues, one every 512 bytes, `chunks` of them.
// PASSES: the query has more rows than one pass (LG is 32 then): hb holds the
// border row below the pass before (unless this is the first) and takes this
// pass's (unless it is the last): lane 0 reads column j at step j - U, lane 31
// rewrites it at step j + 31.
template <int PR, bool PASSES>
__device__ __forceinline__ void lane_sweep(const uint8_t* prof, uint8_t* ring, int lane, int lg,
                                           int n, const uint4* src, int chunks, uint2* hb,
                                           bool first, bool last, uint32_t& smax, uint32_t GO2,
                                           uint32_t NGE2) {
  constexpr int U = LaneShape<PR>::UNROLL;
  constexpr bool AHEAD = LaneShape<PR>::AHEAD;
  constexpr uint32_t CODE = 32 * PR;  // bytes between the profile rows of two codes
  const int li = lane & (lg - 1);
  const int cols = 8 * lg;  // columns per ring block
  // this group's ring: 2 * cols columns and the repeats, 4 bytes each; the
  // gap to the next group's keeps the groups' reads on distinct banks
  uint8_t* gr = ring + (lane / lg) * 4 * (2 * cols + (lg == 8 ? 8 : 16));
  const uint32_t not0 = li == 0 ? 0u : 1u;
  const uint8_t* pl = prof + lane * LaneShape<PR>::VB;
  uint32_t H[PR], E[PR];
#pragma unroll
  for (int r = 0; r < PR; r++) H[r] = E[r] = 0u;  // H(i, 0) = 0; any E(i, 1) <= 0 will do
  uint32_t hdiag = 0u, out_h = 0u, out_f = 0u;
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
  const int steps = n + lg - 1;
  const uint32_t mask = (uint32_t)(4 * (2 * cols - 1));
  int b = 0;
  for (int t0 = 0; t0 < steps; t0 += cols, b++) {
    __syncwarp();
    store(b & 1, next);
    next = load(b + 1);
    __syncwarp();
    const int tend = min(t0 + cols, steps);
    uint2 bq[U];  // the border of columns t .. t + U - 1
    if constexpr (PASSES) {
#pragma unroll
      for (int u = 0; u < U; u++) bq[u] = hb[min(t0 + u, n - 1)];
    }
    // the profile words of step t are loaded one step ahead; the last step of
    // a ring block reads whatever code the slot holds, and is read again here
    LaneWords<PR> w;
    auto fetch = [&](const uint8_t* rp) {
      lane_words<PR>(w, pl + *(const uint16_t*)rp, pl + *(const uint16_t*)(rp + 2));
    };
    if constexpr (AHEAD) fetch(gr + ((uint32_t)(4 * (t0 - li)) & mask));
#pragma unroll 1
    for (int t = t0; t < tend; t += U) {
      const uint8_t* rp = gr + ((uint32_t)(4 * (t - li)) & mask);
#pragma unroll
      for (int u = 0; u < U; u++) {
        // the row above: lane k - 1's bottom row, H = F = 0 above the matrix
        uint32_t in_h = imad(__shfl_up_sync(FULL, out_h, 1, lg), not0, 0u);
        uint32_t in_f = imad(__shfl_up_sync(FULL, out_f, 1, lg), not0, 0u);
        if constexpr (PASSES) {
          const uint2 bv = bq[u];
          bq[u] = hb[min(t + u + U, n - 1)];
          if (li == 0 && !first) {
            in_h = bv.x;
            in_f = bv.y;
          }
        }
        if constexpr (!AHEAD) fetch(rp + 4 * u);
        const LaneWords<PR> now = w;
        if constexpr (AHEAD) fetch(rp + 4 * (u + 1));
        uint32_t f = in_f;
        lane_column<PR>(H, E, smax, hdiag, f, now, GO2, NGE2);
        hdiag = in_h;
        out_h = H[PR - 1];
        out_f = f;
        if constexpr (PASSES) {
          const int j = t + u - 31;
          if (lane == 31 && !last && j >= 0 && j < n) hb[j] = make_uint2(out_h, out_f);
        }
      }
    }
  }
}

// S of each subject of the group's pair: recorded, or flagged for the int32
// recompute when it may have saturated.
__device__ __forceinline__ void lane_emit(const DbView& db, const SearchParams* __restrict__ P,
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

// One warp's share of a block item: where its pairs lie.
struct LanePlace {
  int lg, n;         // lanes per group; columns of the warp's longest subject
  const uint4* src;  // this group's subject pair in the interleaved layout
  int chunks;
  uint2* hb;         // the warp's border row
};

// One pass, the rows [row0, row0 + lg x PR) of the query.  `build`: the block
// does not hold this profile yet (uniform over the block).
template <int PR, int G>
__device__ __forceinline__ void lane_pass(const SearchParams* __restrict__ P, uint8_t* smem,
                                          const uint8_t* sm, const uint8_t* __restrict__ qr, int m,
                                          int row0, bool build, const LanePlace& at, int pass,
                                          int passes, uint32_t& smax) {
  uint8_t* ring = smem + LANE_PROFILE + (threadIdx.x >> 5) * LANE_RING;
  const int lane = threadIdx.x & 31;
  uint32_t GO2, NGE2;  // (Go, Go), (-Ge, -Ge)
  gap_words<G>(P, GO2, NGE2);
  if (build) {
    __syncthreads();  // every warp is done with the profile before
    lane_block_profile<PR>(smem, sm, qr, m, row0, at.lg);
    __syncthreads();
  }
  if (at.n == 0) return;  // uniform over the warp
  if (passes == 1)
    lane_sweep<PR, false>(smem, ring, lane, at.lg, at.n, at.src, at.chunks, nullptr, true, true,
                          smax, GO2, NGE2);
  else
    lane_sweep<PR, true>(smem, ring, lane, 32, at.n, at.src, at.chunks, at.hb, pass == 0,
                         pass == passes - 1, smax, GO2, NGE2);
}

// One block item: LANE_WARPS x 32 / lg subject pairs of one segment.
// `cached` is the segment whose (single-pass) profile the block holds, or -1.
template <int G>
__device__ __forceinline__ void lane_item(const DbView& db, const SearchParams* __restrict__ P,
                                          SearchState* st, const Scratch& scr, uint8_t* smem,
                                          const uint8_t* sm, const LaneSeg& sg, int seg,
                                          int& cached, int unit) {
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
    switch (pr) {  // uniform over the block
      case 4: lane_pass<4, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 8: lane_pass<8, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 12: lane_pass<12, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 16: lane_pass<16, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 20: lane_pass<20, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 24: lane_pass<24, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      case 28: lane_pass<28, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
      default: lane_pass<32, G>(P, smem, sm, qr, m, row0, build, at, p, sg.passes, smax); break;
    }
  }
  cached = sg.passes > 1 ? -1 : seg;
  for (int o = sg.lg >> 1; o > 0; o >>= 1) smax = __vmaxs2(smax, __shfl_xor_sync(FULL, smax, o));
  if (has && (lane & (sg.lg - 1)) == 0) lane_emit(db, P, st, scr, sg.q, pair, smax);
}

template <int G>
__global__ void __launch_bounds__(LANE_WARPS * 32, 4)
lane_kernel(DbView db, const SearchParams* __restrict__ P, SearchState* st, Scratch scr) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ __align__(16) uint8_t sm[NCODES * SM_ROW];
  __shared__ unsigned long long s_item;
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
    lane_item<G>(db, P, st, scr, smem, sm, sg, lo, cached, (int)(it - sg.first));
    __syncthreads();  // the item before is read by all
    if (threadIdx.x == 0) s_item = gridDim.x + atomicAdd(&st->lane_work, 1ull);
    __syncthreads();
    it = (long long)s_item;
  }
}

typedef void (*LaneKernel)(DbView, const SearchParams*, SearchState*, Scratch);

static LaneKernel pick_lane(int gclass) {
  return gclass == 1 ? lane_kernel<1> : gclass == 2 ? lane_kernel<2> : lane_kernel<0>;
}

int lane_blocks_per_sm() {
  for (int g = 0; g < GAP_CLASSES; g++) {  // every variant the plan may launch
    if (cudaFuncSetAttribute(pick_lane(g), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             LANE_SMEM) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
  }
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pick_lane(0), LANE_WARPS * 32,
                                                    (size_t)LANE_SMEM) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return nb;
}

cudaError_t launch_lanes(int gclass, int blocks, const DbView& db, const SearchParams* params,
                         SearchState* state, const Scratch& scr, cudaStream_t stream) {
  cudaGetLastError();  // a stale error must not be read as this launch's
  pick_lane(gclass)<<<blocks, LANE_WARPS * 32, LANE_SMEM, stream>>>(db, params, state, scr);
  return cudaGetLastError();
}

}  // namespace swgb
