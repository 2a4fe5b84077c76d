// noalloc.cu -- sw_search_pairs_noalloc: exact scores without allocating memory.
//
// Every other search entry point allocates device memory (a database, a plan,
// scratch for the kernels).  Some callers cannot allow that: a host framework
// that owns every device allocation through its own pool, a service that
// must not allocate once it is serving (so memory use stays fixed and no call
// can fail with out-of-memory), or code that is not permitted to call
// cudaMalloc at all.  This entry point takes the caller's device buffers for
// inputs and outputs and keeps its scratch -- (H, F) border rows for 512 blocks,
// a work counter and a status word -- in the file-scope array below, whose
// size is fixed at build time.  Every GPU that loads the library holds that
// array until the process exits.
//
// The kernel scores each pair on one warp, in int32: lane k owns PR consecutive
// query rows, takes the (H, F) border of the row above from lane k - 1 by
// shuffle and walks one column a step, as in lane_kernel.cuh.  PR follows the
// query's length, so a query of up to 1,024 residues needs no border memory.
// A block takes a query and a few subjects, builds one profile in shared
// memory for its warps, and they share the subjects out as they finish.
//
// A longer query, and a query of over 256 residues against a subject of over
// 1,024, goes first and as a chain: passes of 256 rows on the block's four
// warps, each two stages of 64 columns behind the one above, borders through
// rings in shared memory, and from the fourth warp to the first one's next pass
// through a row of the array.  One warp would take 1.2 ms for 1,024 x 4,096.
//
// Bound by the ALU pipe at 3.5 operations per cell: one DP4A adds a row's
// score, picked from the four in a profile word, to the diagonal (a PRMT and an
// add took the ALU pipe twice; in a loop of independent cells 7.9 cycles per
// warp and scheduler, against 9.1 for the earlier update).  16 queries of 400 x
// 2,000 subjects: 12.5 -> 2.2 ms, 2.8 without the chains (before: 512 warps on the
// whole chip, 256-row passes through the border rows, codes loaded at the step
// that used them).  Rows per lane come in steps of 2: 2.05 -> 1.96 ms and 2.23 ->
// 2.13 against steps of 4.
#include <mutex>

#include "lane_profile.cuh"

namespace swgb {
namespace {

constexpr int NA_MAX_LEN = 4096;         // longest subject accepted
constexpr int NA_WARPS = 4;              // warps per block
constexpr int NA_ROWS = 512;             // border rows: blocks that may run chains
constexpr int NA_HEADER = 32;            // int2 slots (256 bytes) for the counters and status
constexpr size_t NA_SCRATCH = NA_HEADER + (size_t)NA_ROWS * NA_MAX_LEN;  // int2: ~16 MiB
constexpr int NA_ALONE = 32 * LANE_ROWS_MAX;  // longest query on one warp
constexpr int NA_CHAIN_PR = 8;                // rows per lane in a chain
constexpr int NA_CHAIN_PASS = 32 * NA_CHAIN_PR;
constexpr int NA_CHAIN_LEN = 1024;            // longest subject that is not one
constexpr int NA_STAGE = 64;                  // steps between a chain's barriers
constexpr int NA_LAG = 2;                     // stages between consecutive passes
constexpr int NA_EDGE = 256;                  // columns of a border ring
constexpr int NA_COLS = 256;                 // columns per ring block: 8 per lane
constexpr unsigned NA_BAD_LENGTH = 1u, NA_BAD_CODE = 2u;

// The scratch of sw_search_pairs_noalloc.  In host code this name is only a
// stand-in for the device array: its device address comes from
// cudaGetSymbolAddress, once per device (see scratch_for_current_device).
static __device__ __align__(256) int2 g_noalloc_scratch[NA_SCRATCH];

struct NaMatrix {
  int8_t sm[NCODES * NCODES];  // SM(query code, subject code), PAD row/column = PAD_SCORE
};

struct NaArgs {
  const uint8_t *qres, *sres;
  const int64_t *qoff, *soff;
  const int32_t *qlen, *slen;
  int32_t* scores;
  int nq, ns, go, ge;
  // subjects per block item: of the chains, and of the other pairs, whose
  // items are large for the subjects [0, split) and small, and last, for the
  // rest: a block's warps share a large one out evenly, and small ones end
  // the call evenly
  int chain, large, small, split;
};

// The warps of a chain meet here from different places of the code.
__device__ __forceinline__ void na_chain_barrier() {
  asm volatile("bar.sync 1, %0;" ::"n"(NA_WARPS * 32) : "memory");
}

// Where a chain's pass takes the border row above it and leaves its own: rings
// of NA_EDGE columns, or a whole row (mask -1).  A ring's reader is NA_LAG
// stages behind its writer, which is then at most 64 * 2 + 32 columns ahead.
struct NaEdges {
  const int2* in;
  int2* out;
  int in_mask, out_mask;
  bool first, last;
};

// One pass of a pair, on a warp: n > 0 columns, the lane's PR rows of the
// profile; bad is set when a subject code is outside the alphabet.  CHAIN: the
// passes of the pair run on the block's warps, which meet at a barrier every
// NA_STAGE steps.
template <int PR, bool CHAIN>
__device__ __forceinline__ void na_sweep(const uint8_t* prof, uint16_t* ring, int lane, int n,
                                         const uint8_t* __restrict__ d, const NaEdges& ed, int& S,
                                         int& bad, int go, int ge) {
  using Shape = LaneShape<PR, 1>;
  constexpr int VB = Shape::VB, U = Shape::UNROLL, PW = Shape::PW;
  const uint8_t* pl = prof + lane * VB;
  const int not0 = lane == 0 ? 0 : 1;
  int H[PR], E[PR];
#pragma unroll
  for (int r = 0; r < PR; r++) H[r] = E[r] = 0;  // H(i, 0) = 0; any E(i, 1) <= 0 will do
  int hdiag = 0, out_h = 0, out_f = 0;
  // this lane's 8 codes of ring block b, padding past the subject's end and
  // for a code outside the alphabet
  auto load = [&](int b) {
    uint32_t w[2] = {0u, 0u};
    const int c = b * NA_COLS + 8 * lane;
#pragma unroll
    for (int i = 0; i < 8; i++) {
      int code = PAD_CODE;
      if (c + i < n) {
        code = d[c + i];
        if (code >= ALPHA) {
          code = PAD_CODE;
          bad = 1;
        }
      }
      w[i / 4] |= (uint32_t)code << (8 * (i % 4));
    }
    return make_uint2(w[0], w[1]);
  };
  // as the byte offsets of the codes' profile rows; the first 8 columns are
  // repeated after the last
  auto store = [&](int slot, const uint2 v) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const uint32_t x = i < 2 ? v.x : v.y;
      w[i] = ((x >> (16 * (i & 1))) & 0xffu) * (32 * PW) +
             (((x >> (16 * (i & 1) + 8)) & 0xffu) * (32 * PW) << 16);
    }
    const uint4 o = make_uint4(w[0], w[1], w[2], w[3]);
    *(uint4*)(ring + slot * NA_COLS + 8 * lane) = o;
    if (slot == 0 && lane == 0) *(uint4*)(ring + 2 * NA_COLS) = o;
  };
  __syncwarp();
  store(1, make_uint2(0x18181818u, 0x18181818u));  // the columns left of the first
  uint2 next = load(0);
  const int steps = n + 31;
  int b = 0;
  constexpr int SPAN = CHAIN ? NA_STAGE : NA_COLS;
  for (int t0 = 0; t0 < steps; t0 += SPAN) {
    if (!CHAIN || t0 % NA_COLS == 0) {
      __syncwarp();
      store(b & 1, next);
      next = load(++b);
      __syncwarp();
    }
    const int tend = min(t0 + SPAN, steps);
    int2 bq[U];  // the border of columns t .. t + U - 1
    if constexpr (CHAIN) {
#pragma unroll
      for (int u = 0; u < U; u++) bq[u] = ed.in[min(t0 + u, n - 1) & ed.in_mask];
    }
#pragma unroll 1
    for (int t = t0; t < tend; t += U) {
      const uint16_t* rp = ring + ((t - lane) & (2 * NA_COLS - 1));
#pragma unroll
      for (int u = 0; u < U; u++) {
        int in_h = __shfl_up_sync(FULL, out_h, 1) * not0;  // H = F = 0 above the matrix
        int in_f = __shfl_up_sync(FULL, out_f, 1) * not0;
        if constexpr (CHAIN) {
          const int2 bv = bq[u];
          bq[u] = ed.in[min(t + u + U, min(tend, n) - 1) & ed.in_mask];
          if (lane == 0 && !ed.first) {
            in_h = bv.x;
            in_f = bv.y;
          }
        }
        const uint8_t* pp = pl + rp[u];
        uint32_t w[PW / 4];
#pragma unroll
        for (int v = 0; v < PW / VB; v++) {
          if constexpr (VB == 16) {
            const uint4 x = *(const uint4*)(pp + v * 32 * VB);
            w[4 * v] = x.x, w[4 * v + 1] = x.y, w[4 * v + 2] = x.z, w[4 * v + 3] = x.w;
          } else if constexpr (VB == 8) {
            const uint2 x = *(const uint2*)(pp + v * 32 * VB);
            w[2 * v] = x.x, w[2 * v + 1] = x.y;
          } else {
            w[v] = *(const uint32_t*)(pp + v * 32 * VB);
          }
        }
        int hd = hdiag, f = in_f, xp = 0;
#pragma unroll
        for (int r = 0; r < PR; r++) {
          // the update of packed_cell in int32; DP4A adds the row's byte to hd
          const int x = __dp4a((int)w[r / 4], 1 << (8 * (r & 3)), hd);
          const int h = __vimax3_s32(x, E[r], f);
          hd = H[r];
          H[r] = h;
          const int tt = h - go;
          E[r] = __viaddmax_s32_relu(E[r], -ge, tt);
          f = __viaddmax_s32(f, -ge, tt);
          if (r & 1)
            S = __vimax3_s32(S, xp, x);
          else
            xp = x;
        }
        hdiag = in_h;
        out_h = H[PR - 1];
        out_f = f;
        if constexpr (CHAIN) {
          const int j = t + u - 31;
          if (lane == 31 && !ed.last && j >= 0 && j < n)
            ed.out[j & ed.out_mask] = make_int2(out_h, out_f);
        }
      }
    }
    if constexpr (CHAIN) na_chain_barrier();
  }
}

__device__ __forceinline__ void na_alone(int pr, const uint8_t* prof, uint16_t* ring, int lane,
                                         int n, const uint8_t* d, int& S, int& bad, int go,
                                         int ge) {
  const NaEdges none{nullptr, nullptr, 0, 0, true, true};
  switch (pr) {  // uniform over the block
    case 4: na_sweep<4, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 6: na_sweep<6, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 8: na_sweep<8, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 10: na_sweep<10, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 12: na_sweep<12, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 14: na_sweep<14, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 16: na_sweep<16, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 18: na_sweep<18, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 20: na_sweep<20, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 22: na_sweep<22, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 24: na_sweep<24, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 26: na_sweep<26, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 28: na_sweep<28, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    case 30: na_sweep<30, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
    default: na_sweep<32, false>(prof, ring, lane, n, d, none, S, bad, go, ge); break;
  }
}

// The profile of a query of up to 32 * pr rows, by the whole block.
__device__ __forceinline__ void na_profile(int pr, uint8_t* prof, const uint8_t* sm,
                                           const uint8_t* qr, int m, int wib) {
  switch (pr) {
    case 4: lane_profile_rows<4, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 6: lane_profile_rows<6, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 8: lane_profile_rows<8, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 10: lane_profile_rows<10, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 12: lane_profile_rows<12, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 14: lane_profile_rows<14, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 16: lane_profile_rows<16, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 18: lane_profile_rows<18, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 20: lane_profile_rows<20, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 22: lane_profile_rows<22, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 24: lane_profile_rows<24, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 26: lane_profile_rows<26, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 28: lane_profile_rows<28, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    case 30: lane_profile_rows<30, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
    default: lane_profile_rows<32, 1>(prof, sm, qr, m, 0, 32, wib, NA_WARPS); break;
  }
}

__device__ __forceinline__ int na_warp_max(int S) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) S = max(S, __shfl_xor_sync(FULL, S, o));
  return S;
}

// Pairs that run as chains.
__device__ __forceinline__ bool na_is_chain(int m, int n) {
  return m > NA_ALONE || (m > NA_CHAIN_PASS && n > NA_CHAIN_LEN);
}

// One pair on the block's warps, n > 0.  Pass p runs on warp p % NA_WARPS from
// stage (p / W) * period + (p % W) * NA_LAG on, with a period that leaves a
// ring's reader time to finish before its writer's next pass.  Returns this
// lane's S; every warp meets the same number of barriers.
__device__ __forceinline__ int na_chain(uint8_t* prof, uint16_t* ring, int2 (*edges)[NA_EDGE],
                                        int2* row, const uint8_t* sm, const uint8_t* qr, int m,
                                        const uint8_t* d, int n, int lane, int wib, int& bad,
                                        int go, int ge) {
  constexpr int W = NA_WARPS;
  const int passes = (m + NA_CHAIN_PASS - 1) / NA_CHAIN_PASS;
  const int spass = (n + 31 + NA_STAGE - 1) / NA_STAGE;
  const int period = max(spass + NA_LAG, W * NA_LAG);
  const int end = (passes - 1) / W * period + (passes - 1) % W * NA_LAG + spass;
  uint8_t* mine = prof + wib * NCODES * NA_CHAIN_PASS;
  NaEdges ed;
  ed.in = wib == 0 ? row : edges[wib - 1];
  ed.in_mask = wib == 0 ? -1 : NA_EDGE - 1;
  ed.out = wib == W - 1 ? row : edges[wib];
  ed.out_mask = wib == W - 1 ? -1 : NA_EDGE - 1;
  int S = 0, g = 0;
  for (int p = wib; p < passes; p += W) {
    for (const int start = p / W * period + p % W * NA_LAG; g < start; g++) na_chain_barrier();
    ed.first = p == 0;
    ed.last = p == passes - 1;
    __syncwarp();
    lane_profile_rows<NA_CHAIN_PR, 1>(mine, sm, qr, m, p * NA_CHAIN_PASS, 32, 0, 1);
    __syncwarp();
    na_sweep<NA_CHAIN_PR, true>(mine, ring, lane, n, d, ed, S, bad, go, ge);
    g += spass;
  }
  for (; g < end; g++) na_chain_barrier();
  return S;
}

__global__ void __launch_bounds__(NA_WARPS * 32, 4)
noalloc_kernel(NaArgs a, NaMatrix mat, int2* scratch) {
  __shared__ __align__(16) uint8_t prof[NCODES * 32 * LANE_ROWS_MAX];
  __shared__ __align__(16) uint16_t ring_all[NA_WARPS][2 * NA_COLS + 8];
  __shared__ __align__(16) int2 edges[NA_WARPS - 1][NA_EDGE];
  __shared__ __align__(16) uint8_t sm[NCODES * SM_ROW];
  __shared__ unsigned long long s_item;
  __shared__ int s_subject, s_qbad, red_s[NA_WARPS], red_bad[NA_WARPS];
  for (int i = threadIdx.x; i < NCODES * SM_ROW; i += blockDim.x)
    sm[i] = i % SM_ROW < NCODES ? (uint8_t)mat.sm[i / SM_ROW * NCODES + i % SM_ROW] : 0;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint16_t* ring = ring_all[wib];
  unsigned int* status = (unsigned int*)(scratch + 1);
  const int n_large = a.split / a.large, n_small = (a.ns - a.split + a.small - 1) / a.small;
  const int n_chain = (a.ns - 1) / a.chain + 1;  // items per query
  const bool rows = blockIdx.x < NA_ROWS;
  int2* row = scratch + NA_HEADER + (size_t)(rows ? blockIdx.x : 0) * NA_MAX_LEN;
  // round 0: the chains, on the blocks with a border row; round 1: the other
  // pairs, and the refused ones, on all blocks
  for (int round = rows ? 0 : 1; round < 2; round++) {
    unsigned long long* counter = (unsigned long long*)scratch + (round == 0 ? 0 : 2);
    const long long total = (long long)a.nq * (round == 0 ? n_chain : n_large + n_small);
    int checked = -1, cached = -1;  // the query scanned for bad codes, and that of the profile
    // a block's first item is its index, so few items spread over the SMs
    const unsigned starters = round == 0 ? min(gridDim.x, (unsigned)NA_ROWS) : gridDim.x;
    for (bool start = true;; start = false) {
      __syncthreads();  // the item before is done with the shared words
      if (threadIdx.x == 0) {
        s_item = start ? blockIdx.x : starters + atomicAdd(counter, 1ull);
        s_subject = 0;
      }
      __syncthreads();
      const long long it = (long long)s_item;
      if (it >= total) break;  // uniform over the block
      int q, s0, cnt;
      if (round == 0) {
        q = (int)(it / n_chain), s0 = (int)(it % n_chain) * a.chain;
        cnt = min(a.chain, a.ns - s0);
      } else if (it < (long long)a.nq * n_large) {
        q = (int)(it / n_large), s0 = (int)(it % n_large) * a.large;
        cnt = a.large;
      } else {
        const long long i = it - (long long)a.nq * n_large;
        q = (int)(i / n_small), s0 = a.split + (int)(i % n_small) * a.small;
        cnt = min(a.small, a.ns - s0);
      }
      const int m = a.qlen[q];
      // a negative length, or residues to read from a NULL buffer
      const bool q_ok = m >= 0 && (m == 0 || a.qres);
      if (round == 0 && (!q_ok || m <= NA_CHAIN_PASS)) continue;  // no chain with this query
      const uint8_t* qr = a.qres + (q_ok && m > 0 ? a.qoff[q] : 0);
      const int pr = max(4, (min(m, NA_ALONE) + 63) / 64 * 2);  // of a query on one warp
      // a subject length that may be scored
      auto valid = [&](int n) { return q_ok && n >= 0 && n <= NA_MAX_LEN && (n == 0 || a.sres); };
      if (q_ok && m > 0 && checked != q) {
        if (threadIdx.x == 0) s_qbad = 0;
        __syncthreads();
        int bad = 0;
        for (int i = threadIdx.x; i < m; i += blockDim.x) bad |= qr[i] >= ALPHA;
        if (bad) s_qbad = 1;  // every writer writes 1
        __syncthreads();
        checked = q;
      }
      const bool qbad = q_ok && m > 0 && s_qbad;
      if (round == 0) {
        for (int k0 = 0; k0 < cnt; k0 += 32) {
          const int nk = k0 + lane < cnt ? a.slen[s0 + k0 + lane] : -1;
          unsigned todo = __ballot_sync(FULL, nk > 0 && valid(nk) && na_is_chain(m, nk));
          for (; todo; todo &= todo - 1) {  // uniform over the block
            const int k = __ffs(todo) - 1, s = s0 + k0 + k;
            const int n = __shfl_sync(FULL, nk, k);
            int bad = 0;
            const int S = na_warp_max(na_chain(prof, ring, edges, row, sm, qr, m,
                                               a.sres + a.soff[s], n, lane, wib, bad, a.go, a.ge));
            bad = __any_sync(FULL, bad);
            if (lane == 0) {
              red_s[wib] = S;
              red_bad[wib] = bad;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
              int best = red_s[0];
              for (int w = 1; w < NA_WARPS; w++) {
                best = max(best, red_s[w]);
                bad |= red_bad[w];
              }
              // a code outside the alphabet on either side: no score
              if (bad || qbad)
                atomicOr(status, NA_BAD_CODE);
              else
                a.scores[(long long)q * a.ns + s] = best;
            }
            __syncthreads();  // the next pair rewrites the shared words
          }
        }
        continue;
      }
      if (q_ok && m > 0 && m <= NA_ALONE && cached != q) {
        na_profile(pr, prof, sm, qr, m, wib);
        cached = q;
        __syncthreads();
      }
      // the warps take the chunk's subjects one by one
      for (;;) {
        int k = 0;
        if (lane == 0) k = atomicAdd(&s_subject, 1);
        k = __shfl_sync(FULL, k, 0);
        if (k >= cnt) break;
        const int s = s0 + k, n = a.slen[s];
        if (!valid(n)) {  // refused, with nothing read or written
          if (lane == 0) atomicOr(status, NA_BAD_LENGTH);
          continue;
        }
        if (n > 0 && na_is_chain(m, n)) continue;  // scored in round 0
        int S = 0, bad = 0;
        if (m > 0 && n > 0) {
          na_alone(pr, prof, ring, lane, n, a.sres + a.soff[s], S, bad, a.go, a.ge);
          // a code outside the alphabet on either side: the pair gets no score
          bad = __any_sync(FULL, bad) || qbad;
          S = na_warp_max(S);
        }
        if (lane == 0) {
          if (bad)
            atomicOr(status, NA_BAD_CODE);
          else
            a.scores[(long long)q * a.ns + s] = S;
        }
      }
    }
  }
}

// True when p is device memory of device `dev` (or managed memory), which a
// kernel launched on `dev` may read and write.
bool on_device(const void* p, int dev) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (a.type == cudaMemoryTypeManaged) return true;
  return a.type == cudaMemoryTypeDevice && a.device == dev;
}

struct NaDevice {
  int2* scratch;
  int blocks;  // grid: resident blocks of the whole device
};
std::mutex g_na_lock;
NaDevice g_na[64] = {};

// Device address of g_noalloc_scratch on the current device and the grid for
// it, looked up once per device (cudaGetSymbolAddress needs that device
// current).
sw_status scratch_for_current_device(NaDevice* out) {
  int dev = 0;
  CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return sw_set_error(SW_EINVAL, "device ordinal %d out of range", dev);
  std::lock_guard<std::mutex> g(g_na_lock);
  if (!g_na[dev].scratch) {
    int sms = 0, bps = 0;
    CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, noalloc_kernel, NA_WARPS * 32, 0));
    int2* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress((void**)&p, g_noalloc_scratch);
    if (e != cudaSuccess) return sw_set_cuda_error(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
    g_na[dev] = {p, sms * (bps > 0 ? bps : 1)};
  }
  *out = g_na[dev];
  return SW_OK;
}

}  // namespace
}  // namespace swgb

using namespace swgb;

extern "C" sw_status sw_search_pairs_noalloc(const uint8_t* queries, const int64_t* q_offsets,
                                             const int32_t* q_lengths, int32_t n_queries,
                                             const uint8_t* subjects, const int64_t* s_offsets,
                                             const int32_t* s_lengths, int32_t n_subjects,
                                             int32_t gap_open, int32_t gap_extend,
                                             const int8_t* matrix, int32_t* scores,
                                             void* stream) {
  sw_clear_error();
  if (n_queries < 0 || n_subjects < 0)
    return sw_set_error(SW_EINVAL, "sw_search_pairs_noalloc: negative count");
  if (gap_open < 0 || gap_extend < 0 || gap_open > 100000000 || gap_extend > 100000000)
    return sw_set_error(SW_EINVAL, "sw_search_pairs_noalloc: gap penalties must be in [0, 1e8]");
  if (n_queries == 0 || n_subjects == 0) return SW_OK;
  // the residue buffers may be NULL when every length on that side is 0
  // (the kernel refuses to read a NULL buffer); the others are always read
  if (!q_offsets || !q_lengths || !s_offsets || !s_lengths || !scores)
    return sw_set_error(SW_EINVAL, "sw_search_pairs_noalloc: NULL buffer");
  int cur = 0;
  CUDA_TRY(cudaGetDevice(&cur));
  const void* bufs[7] = {queries, q_offsets, q_lengths, subjects, s_offsets, s_lengths, scores};
  static const char* names[7] = {"queries", "q_offsets", "q_lengths", "subjects",
                                 "s_offsets", "s_lengths", "scores"};
  for (int i = 0; i < 7; i++) {
    if (!bufs[i]) continue;
    if (!on_device(bufs[i], cur))
      return sw_set_error(SW_EINVAL, "sw_search_pairs_noalloc: %s is not device memory of the "
                          "current device (%d)", names[i], cur);
  }
  NaMatrix mat;
  int8_t m[ALPHA * ALPHA];
  if (matrix)
    for (int i = 0; i < ALPHA * ALPHA; i++) m[i] = matrix[i];
  else
    sw_default_matrix(m);
  for (int a = 0; a < NCODES; a++)
    for (int b = 0; b < NCODES; b++)
      mat.sm[a * NCODES + b] = (a < ALPHA && b < ALPHA) ? m[a * ALPHA + b] : (int8_t)PAD_SCORE;
  NaDevice na;
  sw_status st = scratch_for_current_device(&na);
  if (st != SW_OK) return st;
  int2* scratch = na.scratch;
  cudaStream_t s = (cudaStream_t)stream;
  // the counters and the status word must start at zero on every call
  CUDA_TRY(cudaMemsetAsync(scratch, 0, NA_HEADER * sizeof(int2), s));
  NaArgs a{queries, subjects, q_offsets, s_offsets, q_lengths, s_lengths, scores, n_queries,
           n_subjects, gap_open + gap_extend, gap_extend, 0, 0, 0, 0};
  // large items for three quarters of the subjects, at least four to a block;
  // small ones of a subject per warp
  const int64_t pairs = (int64_t)n_queries * n_subjects;
  auto items = [&](int64_t per_block, int lo, int hi) {
    const int64_t c = pairs / (per_block * na.blocks);
    return (int)(c < lo ? lo : c > hi ? hi : c);
  };
  a.chain = items(64, 1, 32);
  a.small = items(64, NA_WARPS, 16);
  a.large = items(4, NA_WARPS, 64);
  a.split = (int)((int64_t)n_subjects * 3 / 4 / a.large) * a.large;
  noalloc_kernel<<<na.blocks, NA_WARPS * 32, 0, s>>>(a, mat, scratch);
  CUDA_TRY(cudaGetLastError());
  unsigned int status = 0;
  CUDA_TRY(cudaMemcpyAsync(&status, scratch + 1, sizeof status, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  if (status & NA_BAD_LENGTH)
    return sw_set_error(SW_EINVAL, "sw_search_pairs_noalloc: a length is negative or a subject "
                        "is longer than %d residues; those pairs were not scored", NA_MAX_LEN);
  if (status & NA_BAD_CODE)
    return sw_set_error(SW_EINVAL, "sw_search_pairs_noalloc: residue code >= 24 in the input");
  return SW_OK;
}
