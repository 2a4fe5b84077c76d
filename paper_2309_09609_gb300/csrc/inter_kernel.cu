// inter_kernel.cu -- the inter-task kernel of libswgb with two subjects per
// 32-bit word.
//
// Item = (query, group of 64 length-sorted subjects).  Each lane owns two
// subjects, the two 16-bit halves of every word, and 32 query rows held in
// registers; it sweeps the group's columns strip by strip (Section II-B:
// inter-task parallelism, one matrix per processing element).  One persistent
// launch takes the items from an atomic counter, longest groups first.
//
// It is for subjects that are short beside a lane group's ramp (lane_kernel.cuh:
// 8 to 32 steps per subject pair), which it does not have: its lanes share
// their columns, not their rows.  The ALU pipe bounds both, at 4.5 operations per
// word.  Where subjects are longer, or the items too few to fill the chip, the
// lane groups are faster; plan_groups in api.cu estimates which.  Measured, one
// query against 570,000 subjects, with the lane groups and with this kernel:
//   3,000 residues x subjects of 5-15     11.1 ms  3.4 ms
//   1,000 x 20-40                          4.9     2.8
//   3,000 x 50-70                         23.3    14.9
#include "device_common.cuh"

namespace swgb {

constexpr int I_ROWS = 32;   // query rows per strip
constexpr int I_COLS = CHUNK;  // columns of a wavefront: one chunk
constexpr int I_RING = 3;    // chunks in flight per warp
constexpr int I_WARPS = 8;   // per block, one block per SM

// A warp's shared memory.  The strip profile, int8, replicated 8 times so that
// the 8 lanes of a quarter-warp read 16-byte rows of any residue codes from 8
// distinct bank groups:
//   byte (c, half h, copy p, row r) at ((c * 2 + h) * 8 + p) * 16 + (r - 16 h)
// Then the cp.async staging ring: per chunk, the 4 border vectors (one per
// column pair) and the residue vector of every lane.
constexpr int I_HALVES = I_ROWS / 16;
constexpr int I_BORDERS = NCODES * 8 * I_ROWS;          // I_RING x 4 x 32 x 16 bytes
constexpr int I_RESIDUES = I_BORDERS + I_RING * 4 * 512;  // I_RING x 32 x 16 bytes
constexpr int I_SLICE = I_RESIDUES + I_RING * 512;

// Word w (0..3) of a profile vector.
__device__ __forceinline__ uint32_t word_of(const uint4& v, int w) {
  return w == 0 ? v.x : w == 1 ? v.y : w == 2 ? v.z : v.w;
}

// A chunk's eight columns as one wavefront: at step k column c updates row
// k - c, so up to eight cell updates of a step are independent.  Hp[r] / E[r]
// hold H / E of the previous column on entry and of the eighth on exit; b[q] /
// o[q] hold (H, F) of columns 2q and 2q + 1 above / at the bottom of the strip.
// Each column holds only the 16-row half of its profile rows that it is in.
__device__ __forceinline__ void inter_chunk(uint32_t (&Hp)[I_ROWS], uint32_t (&E)[I_ROWS],
                                            uint32_t& hdiag, uint32_t& smax, const uint8_t* slice,
                                            int p16, const uint4& rr, const uint4 (&b)[4],
                                            uint4 (&o)[4], uint32_t GO2, uint32_t NGE2) {
  constexpr int T = I_ROWS, W = I_COLS;
  uint32_t ca[W], cb[W];
#pragma unroll
  for (int c = 0; c < W; c++) {
    ca[c] = ((c < 4 ? rr.x : rr.y) >> (8 * (c & 3))) & 0xffu;
    cb[c] = ((c < 4 ? rr.z : rr.w) >> (8 * (c & 3))) & 0xffu;
  }
  uint4 pa[W], pb[W];
  uint32_t htop[W], f[W], last[W], last2[W], bottom[W];
#pragma unroll
  for (int q = 0; q < 4; q++) {
    htop[2 * q] = b[q].x;
    f[2 * q] = b[q].y;
    htop[2 * q + 1] = b[q].z;
    f[2 * q + 1] = b[q].w;
  }
#pragma unroll
  for (int c = 0; c < W; c++) last[c] = last2[c] = bottom[c] = 0u;
  uint32_t hd0 = hdiag;  // column 0's diagonal: previous column, previous row
  hdiag = htop[W - 1];
#pragma unroll
  for (int k = 0; k < T + W - 1; k++) {
    uint32_t out[W], x[W];
#pragma unroll
    for (int c = 0; c < W; c++) {
      out[c] = x[c] = 0u;
      const int r = k - c;
      if (r < 0 || r >= T) continue;
      if ((r & 15) == 0) {  // this column enters a new half of its profile rows
        pa[c] = *(const uint4*)(slice + (ca[c] * I_HALVES + (r >> 4)) * 128 + p16);
        pb[c] = *(const uint4*)(slice + (cb[c] * I_HALVES + (r >> 4)) * 128 + p16);
      }
      uint32_t hd;
      if (c == 0) {
        hd = hd0;
        hd0 = Hp[r];
      } else {
        hd = r == 0 ? htop[c - 1] : last2[c - 1];  // H of column c - 1, row r - 1
      }
      const int w = (r >> 2) & 3;
      uint32_t e = E[r];
      out[c] = packed_cell(hd, prmt(word_of(pa[c], w), word_of(pb[c], w), sext_pair_sel(r & 3)), e,
                           f[c], x[c], GO2, NGE2);
      E[r] = e;
      if (c == W - 1) Hp[r] = out[c];
      if (r == T - 1) bottom[c] = out[c];
    }
    // S over this step's cells (pairs through a three-input max)
    const int lo = k - (T - 1) > 0 ? k - (T - 1) : 0;
    const int hi = k < W - 1 ? k : W - 1;
    int c = lo;
    for (; c + 1 <= hi; c += 2) smax = __vimax3_s16x2(smax, x[c], x[c + 1]);
    if (c == hi) smax = __vmaxs2(smax, x[c]);
#pragma unroll
    for (int c2 = 0; c2 < W; c2++) {
      last2[c2] = last[c2];
      last[c2] = out[c2];
    }
  }
#pragma unroll
  for (int q = 0; q < 4; q++) o[q] = make_uint4(bottom[2 * q], f[2 * q], bottom[2 * q + 1], f[2 * q + 1]);
}

// Query q against group g on one warp.
template <int G>
__device__ void inter_item(const DbView& db, const SearchParams* __restrict__ P, SearchState* st,
                           const int8_t* __restrict__ sm, uint8_t* slice, int lane,
                           int64_t warp_id, const Scratch& scr, int q, int g) {
  constexpr int T = I_ROWS;
  const int L = db.glen[g];  // multiple of CHUNK
  const int m = P->qlen[q];
  const uint8_t* __restrict__ qr = P->qres + P->qoff[q];
  const uint4* __restrict__ res = (const uint4*)(db.inter + db.goff[g]) + lane;
  uint4* bd = scr.inter_border + warp_id * scr.inter_stride_vec + lane;
  uint32_t GO2, NGE2;  // (Go, Go), (-Ge, -Ge)
  gap_words<G>(P, GO2, NGE2);
  const int p16 = (lane & 7) * 16;
  const int nstrips = L > 0 ? (m + T - 1) / T : 0;
  const int nch = L / CHUNK;
  uint4* bring = (uint4*)(slice + I_BORDERS) + lane;   // [slot][pair][lane]
  uint4* rring = (uint4*)(slice + I_RESIDUES) + lane;  // [slot][lane]
  uint32_t smax = 0u;
  for (int s = 0; s < nstrips; s++) {
    __syncwarp();
    if (lane < NCODES) {  // code c = lane: T bytes, written to all 8 copies
      const int i0 = s * T;
      uint32_t wv[T / 4];
#pragma unroll
      for (int w = 0; w < T / 4; w++) {
        uint32_t acc = 0;
#pragma unroll
        for (int b = 0; b < 4; b++) {
          const int i = i0 + w * 4 + b;
          const int v = i < m ? (int)sm[(int)qr[i] * NCODES + lane] : PAD_SCORE;
          acc |= ((uint32_t)(uint8_t)(int8_t)v) << (8 * b);
        }
        wv[w] = acc;
      }
#pragma unroll
      for (int h = 0; h < I_HALVES; h++) {
        const uint4 v = make_uint4(wv[4 * h], wv[4 * h + 1], wv[4 * h + 2], wv[4 * h + 3]);
#pragma unroll
        for (int p = 0; p < 8; p++)  // copies in a lane-rotated order: fewer bank conflicts
          *(uint4*)(slice + ((lane * I_HALVES + h) * 8 + ((p + lane) & 7)) * 16) = v;
      }
    }
    __syncwarp();
    uint32_t Hp[T], E[T];
#pragma unroll
    for (int r = 0; r < T; r++) Hp[r] = E[r] = 0u;  // H(i, 0) = 0; any E(i, 1) <= 0 will do
    uint32_t hdiag = 0u;
    const bool last = (s == nstrips - 1);
    // Staging ring of I_RING chunks, copied with cp.async I_RING - 1 chunks ahead
    // (commit group c = chunk c).  A slot is refilled only after the registers
    // read from it were consumed.  The first strip's border, H = F = 0 above
    // the matrix, is filled in without a read (copied chunk by chunk from one
    // word in global memory, every warp of the chip asked one slice of L2 for
    // it: one query of 375 x 200,000 subjects of 250-350 took 5.8 ms, now 3.5).
    const int bytes = s == 0 ? 0 : 16;
    auto stage = [&](int j) {
#pragma unroll
      for (int k = 0; k < 4; k++)
        cp_async16_or_zeros(bring + ((j % I_RING) * 4 + k) * 32, bd + (j * 4 + k) * 32, bytes);
      cp_async16(rring + (j % I_RING) * 32, res + j * 32);
    };
#pragma unroll
    for (int j = 0; j < I_RING - 1; j++) {
      if (j < nch) stage(j);
      cp_async_commit();
    }
#pragma unroll 1
    for (int c = 0; c < nch; c++) {
      if (c + I_RING - 1 < nch) stage(c + I_RING - 1);
      cp_async_commit();
      cp_async_wait<I_RING - 1>();  // chunk c has landed
      const int slot = c % I_RING;
      const uint4 rr = rring[slot * 32];
      const uint4 bv[4] = {bring[(slot * 4 + 0) * 32], bring[(slot * 4 + 1) * 32],
                           bring[(slot * 4 + 2) * 32], bring[(slot * 4 + 3) * 32]};
      uint4 ov[4];
      inter_chunk(Hp, E, hdiag, smax, slice, p16, rr, bv, ov, GO2, NGE2);
      if (!last) {
#pragma unroll
        for (int k = 0; k < 4; k++) bd[(c * 4 + k) * 32] = ov[k];
      }
    }
    cp_async_wait<0>();
  }
  emit_pair(db, P, st, scr, q, g * (GROUP / 2) + lane, smax);
}

template <int G>
__global__ void __launch_bounds__(I_WARPS * 32, 1)
inter_kernel(DbView db, const SearchParams* __restrict__ P, SearchState* st, Scratch scr) {
  extern __shared__ __align__(16) uint8_t smem[];
  int8_t* sm = (int8_t*)smem;
  load_matrix(sm, P);
  __syncthreads();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint8_t* slice = smem + MATRIX_SMEM + wib * I_SLICE;
  const int64_t warp_id = (int64_t)blockIdx.x * I_WARPS + wib;
  const int nq = P->nq;
  const int64_t total = P->n_inter_items;
  if (nq <= 0 || total <= 0) return;  // uniform over the grid
  for (;;) {
    unsigned long long it = 0;
    if (lane == 0) it = atomicAdd(&st->inter_work, 1ull);
    it = __shfl_sync(FULL, it, 0);
    if ((int64_t)it >= total) break;
    const int g = P->g_first + (int)((int64_t)it / nq);
    inter_item<G>(db, P, st, sm, slice, lane, warp_id, scr, P->qorder[(int64_t)it % nq], g);
  }
}

typedef void (*InterKernel)(DbView, const SearchParams*, SearchState*, Scratch);

static InterKernel pick_inter(int gclass) {
  return gclass == 1 ? inter_kernel<1> : gclass == 2 ? inter_kernel<2> : inter_kernel<0>;
}

constexpr int I_SMEM = MATRIX_SMEM + I_WARPS * I_SLICE;

int inter_warps() { return I_WARPS; }

int inter_blocks_per_sm() {
  for (int g = 0; g < GAP_CLASSES; g++) {  // every variant the plan may launch
    if (cudaFuncSetAttribute(pick_inter(g), cudaFuncAttributeMaxDynamicSharedMemorySize, I_SMEM) !=
        cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
  }
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pick_inter(0), I_WARPS * 32, I_SMEM) !=
      cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return nb;
}

cudaError_t launch_inter(int gclass, int blocks, const DbView& db, const SearchParams* params,
                         SearchState* state, const Scratch& scr, cudaStream_t stream) {
  cudaGetLastError();  // a stale error must not be read as this launch's
  pick_inter(gclass)<<<blocks, I_WARPS * 32, I_SMEM, stream>>>(db, params, state, scr);
  return cudaGetLastError();
}

}  // namespace swgb
