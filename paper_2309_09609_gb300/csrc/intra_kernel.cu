// intra_kernel.cu -- the int32 intra-task kernel of libswgb: exact scores of
// the pairs that the packed 16-bit kernels cannot score.
//
// The warp wavefront of Section II-B (intra-task parallelism with neighbour
// border exchange) in int32: lane k owns TI query rows of a 32*TI-row pass and
// sweeps the subject one step behind lane k-1, which hands it the (H, F)
// border of its last row through __shfl_up_sync.  The bottom row of a pass is
// the top border of the next one and goes through a per-warp scratch row.
//
// One launch does two kinds of work, of which a search has only one:
//   * int32 intra-task items (query, subject), one warp each -- every subject
//     when the packed path is off (forced, or gaps too large for 16 bits);
//   * the pairs flagged by the packed kernels (16-bit score at the saturation
//     threshold), one block each: the passes of the query are dealt round-robin
//     to the block's warps, pass p starting LAG stages of 32 steps after pass
//     p - 1, so a flagged pair of two 35,000-residue sequences runs on sixteen
//     warps instead of one.  Stages end at __syncthreads, which orders each
//     border write before its read and each read before the next overwrite.
//
// Few flagged pairs leave most SMs idle that way, and the search waits for the
// longest.  They are therefore scored by recompute_kernel where that ends
// first: the same schedule over the 128 warps of a cluster of sixteen blocks,
// with the cluster's barrier between the stages.  Many pairs fill the chip one
// block each, and a query of few passes leaves most blocks of a cluster idle,
// which takes its pairs in turn (recompute_in_clusters).  Two pairs of 35,000 x
// 26,620 residues took 68 ms on a block each, 15.9 on clusters of eight blocks
// of 16 warps, 11.6 on clusters of sixteen of 8 (two warps to a scheduler) and
// 9.7 with the codes and profile words loaded ahead of their columns.
#include <cooperative_groups.h>

#include "device_common.cuh"

namespace swgb {

template <int TI>
struct IntraSlice {
  static constexpr int BYTES = NCODES * 32 * TI;  // lane_profile<TI> of one pass
};

constexpr int LAG = 3;  // stages between the starts of consecutive passes (block items)

// The TI cells of one lane at one column: (in_h, in_f) are H and F of the row
// above the lane's first row at this column; pw are the lane's profile words
// of the column's residue.  Eq. 1-3 in the shared-gap form, int32.
template <int TI>
__device__ __forceinline__ void intra_cells(int (&Hp)[TI], int (&E)[TI], int& hdiag, int& out_h,
                                            int& out_f, int& S, int in_h, int in_f,
                                            const uint32_t (&pw)[TI / 4], int go, int ge) {
  int hd = hdiag, xp = 0;
  hdiag = in_h;
  int f = in_f;
#pragma unroll
  for (int r = 0; r < TI; r++) {
    // as packed_cell: E >= 0 stands for the zero term, S from the diagonal term
    // (one DP4A picks row r's score from its profile word and adds it)
    const int x = __dp4a((int)pw[r / 4], 1 << (8 * (r & 3)), hd);
    const int h = __vimax3_s32(x, E[r], f);  // Eq. 1
    hd = Hp[r];
    Hp[r] = h;
    const int tt = h - go;
    E[r] = __viaddmax_s32_relu(E[r], -ge, tt);  // Eq. 2, next column
    f = __viaddmax_s32(f, -ge, tt);             // Eq. 3, next row
    if (r & 1)
      S = __vimax3_s32(S, xp, x);
    else
      xp = x;
  }
  out_h = Hp[TI - 1];
  out_f = f;
}

template <int TI>
__device__ __forceinline__ void intra_start(int (&Hp)[TI], int (&E)[TI], int& hdiag, int& out_h,
                                            int& out_f, int go) {
#pragma unroll
  for (int r = 0; r < TI; r++) {
    Hp[r] = 0;  // H(i, 0)
    E[r] = 0;   // any E(i, 1) <= 0 gives the same H
  }
  hdiag = 0;
  out_h = 0;
  out_f = -go;
}

// One (query, subject) pair on one warp, all passes in order.
template <int TI>
__device__ void intra_warp_item(const DbView& db, const SearchParams* __restrict__ P,
                                const int8_t* __restrict__ sm, uint8_t* slice, int lane,
                                int2* hb, int q, int s) {
  const int n = db.clen[s];
  const int m = P->qlen[q];
  const uint8_t* __restrict__ d = db.cont + db.coff[s];
  const uint8_t* __restrict__ qr = P->qres + P->qoff[q];
  const int go = P->go, ge = P->ge;
  constexpr int ROWS = 32 * TI;
  const int npass = (m + ROWS - 1) / ROWS;
  int S = 0;
  for (int p = 0; p < npass && n > 0; p++) {
    __syncwarp();
    lane_profile<TI>(slice, sm, qr, m, p * ROWS + lane * TI, lane);
    __syncwarp();
    int Hp[TI], E[TI], hdiag, out_h, out_f;
    intra_start<TI>(Hp, E, hdiag, out_h, out_f, go);
    const bool last_pass = (p == npass - 1);
    const int steps = n + 31;
    IntraFeed<TI> feed{d, slice + lane * TI, n};
    feed.start(-lane);
    for (int t = 0; t < steps; t++) {
      uint32_t pw[TI / 4];
      feed.step(pw, t - lane);
      int in_h = __shfl_up_sync(FULL, out_h, 1);
      int in_f = __shfl_up_sync(FULL, out_f, 1);
      const int j = t - lane;
      if (lane == 0) {
        if (p > 0 && j < n) {
          const int2 v = hb[j];
          in_h = v.x;
          in_f = v.y;
        } else {
          in_h = 0;    // H(0, j)
          in_f = -go;  // F(1, j)
        }
      }
      if (j >= 0 && j < n) {
        intra_cells<TI>(Hp, E, hdiag, out_h, out_f, S, in_h, in_f, pw, go, ge);
        if (lane == 31 && !last_pass) hb[j] = make_int2(out_h, out_f);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) S = max(S, __shfl_xor_sync(FULL, S, o));
  if (lane == 0) emit_score(db, P, q, s, S);
}

// Stages of a pair's passes on W warps.
template <int TI>
__device__ __forceinline__ int pair_stages(int m, int n, int W) {
  const int npass = n > 0 ? (m + 32 * TI - 1) / (32 * TI) : 0;
  const int spass = (n + 31 + 31) / 32;  // of one pass (n + 31 steps)
  if (npass == 0) return 0;
  return (npass - 1) / W * max(spass, LAG * W) + (npass - 1) % W * LAG + spass;
}

// One (query, subject) pair on the W warps of a block, or of a cluster of
// blocks.  Pass p runs on warp p % W and starts at stage (p / W) * period +
// (p % W) * LAG, with period = max(stages of a pass, LAG * W): consecutive
// passes are LAG stages apart, and a warp's next pass starts after its
// previous one ends.  Lane 0 of pass p at column j needs the bottom row of pass
// p - 1 at column j, written by that pass at its step j + 31, i.e. at most two
// of its stages after the stage holding its step j; LAG = 3 leaves one stage in
// between, in which the warp fetches the next 32 border values with one
// coalesced load.  own: this warp's border row, src: that of the warp before;
// they go through L2, where the other blocks of a cluster see them.  Returns
// the block's maximum in thread 0.
template <int TI, int W, int BLOCK_WARPS, typename Barrier>
__device__ int intra_block_item(const DbView& db, const SearchParams* __restrict__ P,
                                const int8_t* __restrict__ sm, uint8_t* slice, int lane, int wib,
                                int warp, int2* own, const int2* src, int* red, int q, int s,
                                Barrier barrier) {
  constexpr int ROWS = 32 * TI;
  const int n = db.clen[s];
  const int m = P->qlen[q];
  const uint8_t* __restrict__ d = db.cont + db.coff[s];
  const uint8_t* __restrict__ qr = P->qres + P->qoff[q];
  const int go = P->go, ge = P->ge;
  const int npass = n > 0 ? (m + ROWS - 1) / ROWS : 0;
  const int spass = (n + 31 + 31) / 32;  // stages of one pass (n + 31 steps)
  const int period = max(spass, LAG * W);
  const int nstages = pair_stages<TI>(m, n, W);
  const int2 top = make_int2(0, -go);                   // (H(0, j), F(1, j))
  int S = 0;
  int Hp[TI], E[TI], hdiag = 0, out_h = 0, out_f = -go;
  int p = 0;
  int2 bcur = top, bnext = top;  // border of columns 32k + lane and 32(k + 1) + lane
  for (int g = 0; g < nstages; g++) {
    const int rel = g - warp * LAG;
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
        lane_profile<TI>(slice, sm, qr, m, p * ROWS + lane * TI, lane);
        __syncwarp();
        intra_start<TI>(Hp, E, hdiag, out_h, out_f, go);
        bcur = (p > 0 && lane < n) ? __ldcg(src + lane) : top;
      } else {
        bcur = bnext;
      }
      const int jn = 32 * (k + 1) + lane;
      bnext = (p > 0 && jn < n) ? __ldcg(src + jn) : top;
      const bool last_pass = (p == npass - 1);
      const int t0 = 32 * k;
      const int tend = min(t0 + 32, n + 31);
      IntraFeed<TI> feed{d, slice + lane * TI, n};
      feed.start(t0 - lane);
#pragma unroll 4
      for (int t = t0; t < tend; t++) {
        uint32_t pw[TI / 4];
        feed.step(pw, t - lane);
        int in_h = __shfl_up_sync(FULL, out_h, 1);
        int in_f = __shfl_up_sync(FULL, out_f, 1);
        const int bh = __shfl_sync(FULL, bcur.x, t - t0);
        const int bf = __shfl_sync(FULL, bcur.y, t - t0);
        if (lane == 0) {
          in_h = bh;
          in_f = bf;
        }
        const int j = t - lane;
        if (j >= 0 && j < n) {
          intra_cells<TI>(Hp, E, hdiag, out_h, out_f, S, in_h, in_f, pw, go, ge);
          if (lane == 31 && !last_pass) __stcg(own + j, make_int2(out_h, out_f));
        }
      }
    }
    barrier();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) S = max(S, __shfl_xor_sync(FULL, S, o));
  if (lane == 0) red[wib] = S;
  __syncthreads();
  int best = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < BLOCK_WARPS; w++) best = max(best, red[w]);
  return best;
}

// Whether the flagged pairs go to clusters (`clusters` 0: never): if the stages of
// the cluster that has most end before those of the longest pair on a block.
// Every warp of either kernel gets the same answer from the same list.
// Measured, microseconds a stage: 8.0 on a block of 16 busy warps, 6.4 on a
// cluster, 8.6 where its SMs hold a second one's blocks (8 pairs at a time, with
// 9 clusters); here in fifths.  Milliseconds for pairs of 3,100 residues, of 8,000 and of 16,000,
// with clusters and without: 4 pairs 0.84 and 0.94, 2.2 and 4.4, 4.4 and 16.7; 10
// pairs 1.79 and 0.94, 4.7 and 4.4, 9.5 and 16.7; 36 pairs 4.2 and 0.95, 11.6 and
// 4.4, 23.3 and 16.8 (all of which had gone to clusters).
template <int TI>
__device__ __forceinline__ bool recompute_in_clusters(const DbView& db,
                                                      const SearchParams* __restrict__ P,
                                                      const Scratch& scr, unsigned long long flagged,
                                                      unsigned clusters) {
  if (flagged == 0 || flagged > (unsigned long long)RECOMPUTE_PER_CLUSTER * clusters) return false;
  long long most = 0, block = 0;
  for (unsigned c = threadIdx.x & 31; c < clusters; c += 32) {
    long long mine = 0;
    for (unsigned it = c; it < (unsigned)flagged; it += clusters) {
      const int2 fl = scr.flags[it];
      const int m = P->qlen[fl.x], n = db.clen[fl.y];
      const unsigned left = (unsigned)flagged - (it - c);  // pairs of this turn and the next ones
      mine += (long long)pair_stages<TI>(m, n, RECOMPUTE_CLUSTER * RECOMPUTE_WARPS) *
              (4 * left > 3 * clusters ? 43 : 32);
      block = max(block, 40ll * pair_stages<TI>(m, n, INTRA_WARPS));
    }
    most = max(most, mine);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    most = max(most, __shfl_xor_sync(FULL, most, o));
    block = max(block, __shfl_xor_sync(FULL, block, o));
  }
  return most < block;
}

template <int TI>
__global__ void __launch_bounds__(INTRA_WARPS * 32)
intra_kernel(DbView db, const SearchParams* __restrict__ P, SearchState* st, Scratch scr,
             unsigned clusters) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ unsigned long long s_item;
  __shared__ int red[INTRA_WARPS];
  int8_t* sm = (int8_t*)smem;
  load_matrix(sm, P);
  __syncthreads();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint8_t* slice = smem + MATRIX_SMEM + wib * IntraSlice<TI>::BYTES;
  const int64_t warp0 = (int64_t)blockIdx.x * INTRA_WARPS;
  int2* border = scr.intra_border + warp0 * scr.intra_stride;
  const int nq = P->nq;
  if (nq <= 0) return;  // uniform over the grid
  // int32 intra-task items, one warp each (longest subjects first)
  const int64_t n_items = P->n_intra_items;
  for (;;) {
    unsigned long long it = 0;
    if (lane == 0) it = atomicAdd(&st->intra_work, 1ull);
    it = __shfl_sync(FULL, it, 0);
    if ((int64_t)it >= n_items) break;
    const int s = (int)((int64_t)it / nq);
    const int q = P->qorder[(int64_t)it % nq];
    intra_warp_item<TI>(db, P, sm, slice, lane, border + wib * scr.intra_stride, q, s);
  }
  __syncthreads();
  // flagged pairs, one block each
  const unsigned long long nf = *(volatile unsigned long long*)&st->n_flags;
  const unsigned long long total =
      nf < (unsigned long long)scr.flag_capacity ? nf : (unsigned long long)scr.flag_capacity;
  if (total == 0 || recompute_in_clusters<TI>(db, P, scr, total, clusters)) return;  // recompute_kernel
  const int64_t stride = scr.intra_stride;
  for (;;) {
    if (threadIdx.x == 0) s_item = atomicAdd(&st->recompute, 1ull);
    __syncthreads();
    const unsigned long long it = s_item;
    __syncthreads();  // every thread has read s_item before thread 0 rewrites it
    if (it >= total) break;
    const int2 fl = scr.flags[it];
    const int best = intra_block_item<TI, INTRA_WARPS, INTRA_WARPS>(
        db, P, sm, slice, lane, wib, wib, border + wib * stride,
        border + (wib + INTRA_WARPS - 1) % INTRA_WARPS * stride, red, fl.x, fl.y,
        []() { __syncthreads(); });
    if (threadIdx.x == 0) emit_score(db, P, fl.x, fl.y, best);
  }
}

// Few flagged pairs, one cluster each: cluster c takes the pairs c, c +
// clusters, ...  Every block of a cluster runs the same stages.
template <int TI>
__global__ void __cluster_dims__(RECOMPUTE_CLUSTER) __launch_bounds__(RECOMPUTE_WARPS * 32)
recompute_kernel(DbView db, const SearchParams* __restrict__ P, SearchState* st, Scratch scr,
                 unsigned clusters) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ int red[RECOMPUTE_WARPS];
  __shared__ int block_best;
  const unsigned long long nf = *(volatile unsigned long long*)&st->n_flags;
  const unsigned long long total =
      nf < (unsigned long long)scr.flag_capacity ? nf : (unsigned long long)scr.flag_capacity;
  if (!recompute_in_clusters<TI>(db, P, scr, total, clusters)) return;  // uniform over the grid
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  constexpr int W = RECOMPUTE_CLUSTER * RECOMPUTE_WARPS;
  int8_t* sm = (int8_t*)smem;
  load_matrix(sm, P);
  __syncthreads();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int rank = (int)cluster.block_rank(), warp = rank * RECOMPUTE_WARPS + wib;
  uint8_t* slice = smem + MATRIX_SMEM + wib * IntraSlice<TI>::BYTES;
  // the cluster's border rows, one per warp
  int2* rows = scr.intra_border + ((int64_t)blockIdx.x - rank) * RECOMPUTE_WARPS * scr.intra_stride;
  int2* own = rows + warp * scr.intra_stride;
  const int2* src = rows + (warp + W - 1) % W * scr.intra_stride;
  for (unsigned long long it = blockIdx.x / RECOMPUTE_CLUSTER; it < total; it += clusters) {
    const int2 fl = scr.flags[it];
    const int best = intra_block_item<TI, W, RECOMPUTE_WARPS>(db, P, sm, slice, lane, wib, warp, own, src, red, fl.x,
                                             fl.y, [&]() { cluster.sync(); });
    if (threadIdx.x == 0) block_best = best;
    cluster.sync();
    if (rank == 0 && threadIdx.x == 0) {
      int score = best;
      for (int r = 1; r < RECOMPUTE_CLUSTER; r++)
        score = max(score, *cluster.map_shared_rank(&block_best, r));
      emit_score(db, P, fl.x, fl.y, score);
    }
    cluster.sync();  // block_best is read, and no block leaves before that
  }
}

// Pairs marked FLAG_SENTINEL by a packed kernel whose flag list was full:
// each (query, sorted subject) slot is read once, grid-stride, and every
// marked pair is counted and, while there is room, listed.
__global__ void collect_kernel(DbView db, const SearchParams* __restrict__ P, SearchState* st,
                               Scratch scr) {
  const int64_t slots = (int64_t)db.groups * GROUP;
  const int64_t total = (int64_t)P->nq * slots;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int q = (int)(i / slots);
    const int s = (int)(i - (int64_t)q * slots);
    const int orig = db.perm[s];
    if (orig < 0 || P->scores[(int64_t)q * db.n + orig] != FLAG_SENTINEL) continue;
    const unsigned long long k = atomicAdd(&st->n_flags, 1ull);
    if ((int64_t)k < scr.flag_capacity) scr.flags[k] = make_int2(q, s);
  }
}

cudaError_t launch_collect(int blocks, const DbView& db, const SearchParams* params,
                           SearchState* state, const Scratch& scr, cudaStream_t stream) {
  cudaGetLastError();  // a stale error must not be read as this launch's
  collect_kernel<<<blocks, 256, 0, stream>>>(db, params, state, scr);
  return cudaGetLastError();
}

typedef void (*IntraKernel)(DbView, const SearchParams*, SearchState*, Scratch, unsigned);

static IntraKernel pick_intra(int rows) {
  if (rows == 8) return intra_kernel<8>;
  if (rows == 16) return intra_kernel<16>;
  return nullptr;
}

static IntraKernel pick_recompute(int rows) {
  return rows == 8 ? recompute_kernel<8> : recompute_kernel<16>;
}

static size_t slices_bytes(int rows, int warps) {
  const int slice = rows == 8 ? IntraSlice<8>::BYTES : IntraSlice<16>::BYTES;
  return (size_t)MATRIX_SMEM + (size_t)warps * slice;
}

static size_t recompute_smem_bytes(int rows) { return slices_bytes(rows, RECOMPUTE_WARPS); }

size_t intra_smem_bytes(int rows) { return slices_bytes(rows, INTRA_WARPS); }

int intra_blocks_per_sm(int rows) {
  IntraKernel k = pick_intra(rows);
  if (!k) return 0;
  const size_t smem = intra_smem_bytes(rows);
  int nb = 0;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, INTRA_WARPS * 32, smem) !=
          cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return nb;
}

int recompute_clusters(int rows, int blocks) {
  const int most = blocks / RECOMPUTE_CLUSTER;
  if (most < 1) return 0;
  IntraKernel k = pick_recompute(rows);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(RECOMPUTE_CLUSTER);
  cfg.blockDim = dim3(RECOMPUTE_WARPS * 32);
  cfg.dynamicSmemBytes = recompute_smem_bytes(rows);
  cudaLaunchAttribute shape{};
  shape.id = cudaLaunchAttributeClusterDimension;
  shape.val.clusterDim.x = RECOMPUTE_CLUSTER;
  shape.val.clusterDim.y = shape.val.clusterDim.z = 1;
  cfg.attrs = &shape;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)cfg.dynamicSmemBytes) != cudaSuccess ||
      cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n < most ? n : most;
}

cudaError_t launch_intra(const KernelConfig& kc, int clusters, bool items, const DbView& db,
                         const SearchParams* params, SearchState* state, const Scratch& scr,
                         cudaStream_t stream) {
  IntraKernel k = pick_intra(kc.variant);
  if (!k) return cudaErrorInvalidValue;
  cudaGetLastError();  // a stale error must not be read as this launch's
  if (!items && clusters > 0) {  // flagged pairs: few of them, or many
    pick_recompute(kc.variant)<<<clusters * RECOMPUTE_CLUSTER, RECOMPUTE_WARPS * 32,
                                 recompute_smem_bytes(kc.variant), stream>>>(
        db, params, state, scr, (unsigned)clusters);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  k<<<kc.blocks, INTRA_WARPS * 32, kc.smem, stream>>>(db, params, state, scr, (unsigned)clusters);
  return cudaGetLastError();
}

}  // namespace swgb
