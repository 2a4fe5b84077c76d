// noalloc.cu -- sw_search_pairs_noalloc: exact scores without allocating memory.
//
// Every other search entry point allocates device memory (a database, a plan,
// scratch for the kernels).  Some callers cannot allow that: a host framework
// that owns every device allocation through its own pool, a service that
// must not allocate once it is serving (so memory use stays fixed and no call
// can fail with out-of-memory), or code that is not permitted to call
// cudaMalloc at all.  This entry point takes the caller's device buffers for
// inputs and outputs and keeps its scratch -- one (H, F) border row per warp,
// a work counter and a status word -- in the file-scope array below, whose
// size is fixed at build time.  Every GPU that loads the library holds that
// array until the process exits.
//
// The kernel scores each pair on one warp, in int32: lane k owns PR consecutive
// query rows, takes the (H, F) border of the row above from lane k - 1 by
// shuffle and walks one column a step, as in lane_kernel.cuh.  PR follows the
// query's length, so a query of up to 1,024 residues needs no border memory
// and any number of warps may run; a longer one goes in passes of 1,024 rows
// whose border rows lie in the array, on the blocks that have rows there.  A
// block takes a query and a few subjects, builds one profile in shared memory
// for its warps, and they share the subjects out as they finish.
//
// Bound by the ALU pipe at 3.5 operations per cell: one DP4A adds a row's
// score, picked from the four in a profile word, to the diagonal (a PRMT and an
// add took the ALU pipe twice; in a loop of independent cells 7.9 cycles per
// warp and scheduler, against 9.1 for the earlier update).  16 queries of 400 x
// 2,000 subjects: 12.5 -> 2.5 ms (before: 512 warps on the whole chip, 256-row passes
// through the border rows, codes loaded at the step that used them).
#include <mutex>

#include "lane_profile.cuh"

namespace swgb {
namespace {

constexpr int NA_MAX_LEN = 4096;         // longest subject accepted
constexpr int NA_WARPS = 4;              // warps per block
constexpr int NA_ROW_BLOCKS = 128;       // blocks with border rows
constexpr int NA_HEADER = 32;            // int2 slots (256 bytes) for the counters and status
constexpr size_t NA_SCRATCH =
    NA_HEADER + (size_t)NA_ROW_BLOCKS * NA_WARPS * NA_MAX_LEN;  // int2: ~16 MiB
constexpr int NA_PASS = 32 * LANE_ROWS_MAX;  // query rows of a pass
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
  int chunk;  // subjects per block item
};

// One pass of a pair, on a warp: n > 0 columns, the lane's PR rows of the
// profile.  hb: the border row of a query of several passes (PASSES), as in
// lane_sweep; bad is set when a subject code is outside the alphabet.
template <int PR, bool PASSES>
__device__ __forceinline__ void na_sweep(const uint8_t* prof, uint16_t* ring, int lane, int n,
                                         const uint8_t* __restrict__ d, int2* hb, bool first,
                                         bool last, int& S, int& bad, int go, int ge) {
  using Shape = LaneShape<PR, 1>;
  constexpr int VB = Shape::VB, U = Shape::UNROLL;
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
      w[i] = ((x >> (16 * (i & 1))) & 0xffu) * (32 * PR) +
             (((x >> (16 * (i & 1) + 8)) & 0xffu) * (32 * PR) << 16);
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
  for (int t0 = 0; t0 < steps; t0 += NA_COLS) {
    __syncwarp();
    store(b & 1, next);
    next = load(++b);
    __syncwarp();
    const int tend = min(t0 + NA_COLS, steps);
    int2 bq[U];  // the border of columns t .. t + U - 1
    if constexpr (PASSES) {
#pragma unroll
      for (int u = 0; u < U; u++) bq[u] = hb[min(t0 + u, n - 1)];
    }
#pragma unroll 1
    for (int t = t0; t < tend; t += U) {
      const uint16_t* rp = ring + ((t - lane) & (2 * NA_COLS - 1));
#pragma unroll
      for (int u = 0; u < U; u++) {
        int in_h = __shfl_up_sync(FULL, out_h, 1) * not0;  // H = F = 0 above the matrix
        int in_f = __shfl_up_sync(FULL, out_f, 1) * not0;
        if constexpr (PASSES) {
          const int2 bv = bq[u];
          bq[u] = hb[min(t + u + U, n - 1)];
          if (lane == 0 && !first) {
            in_h = bv.x;
            in_f = bv.y;
          }
        }
        const uint8_t* pp = pl + rp[u];
        uint32_t w[PR / 4];
#pragma unroll
        for (int v = 0; v < PR / VB; v++) {
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
        if constexpr (PASSES) {
          const int j = t + u - 31;
          if (lane == 31 && !last && j >= 0 && j < n) hb[j] = make_int2(out_h, out_f);
        }
      }
    }
  }
}

template <bool PASSES>
__device__ __forceinline__ void na_pass(int pr, const uint8_t* prof, uint16_t* ring, int lane,
                                        int n, const uint8_t* d, int2* hb, bool first, bool last,
                                        int& S, int& bad, int go, int ge) {
  switch (pr) {  // uniform over the block
    case 4: na_sweep<4, PASSES>(prof, ring, lane, n, d, hb, first, last, S, bad, go, ge); break;
    case 8: na_sweep<8, PASSES>(prof, ring, lane, n, d, hb, first, last, S, bad, go, ge); break;
    case 12: na_sweep<12, PASSES>(prof, ring, lane, n, d, hb, first, last, S, bad, go, ge); break;
    case 16: na_sweep<16, PASSES>(prof, ring, lane, n, d, hb, first, last, S, bad, go, ge); break;
    case 20: na_sweep<20, PASSES>(prof, ring, lane, n, d, hb, first, last, S, bad, go, ge); break;
    case 24: na_sweep<24, PASSES>(prof, ring, lane, n, d, hb, first, last, S, bad, go, ge); break;
    case 28: na_sweep<28, PASSES>(prof, ring, lane, n, d, hb, first, last, S, bad, go, ge); break;
    default: na_sweep<32, PASSES>(prof, ring, lane, n, d, hb, first, last, S, bad, go, ge); break;
  }
}

// The profile of rows [row0, row0 + 32 * pr), by the whole block.
__device__ __forceinline__ void na_profile(int pr, uint8_t* prof, const uint8_t* sm,
                                           const uint8_t* qr, int m, int row0, int wib) {
  switch (pr) {
    case 4: lane_profile_rows<4, 1>(prof, sm, qr, m, row0, 32, wib, NA_WARPS); break;
    case 8: lane_profile_rows<8, 1>(prof, sm, qr, m, row0, 32, wib, NA_WARPS); break;
    case 12: lane_profile_rows<12, 1>(prof, sm, qr, m, row0, 32, wib, NA_WARPS); break;
    case 16: lane_profile_rows<16, 1>(prof, sm, qr, m, row0, 32, wib, NA_WARPS); break;
    case 20: lane_profile_rows<20, 1>(prof, sm, qr, m, row0, 32, wib, NA_WARPS); break;
    case 24: lane_profile_rows<24, 1>(prof, sm, qr, m, row0, 32, wib, NA_WARPS); break;
    case 28: lane_profile_rows<28, 1>(prof, sm, qr, m, row0, 32, wib, NA_WARPS); break;
    default: lane_profile_rows<32, 1>(prof, sm, qr, m, row0, 32, wib, NA_WARPS); break;
  }
}

__device__ __forceinline__ int na_warp_max(int S) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) S = max(S, __shfl_xor_sync(FULL, S, o));
  return S;
}

__global__ void __launch_bounds__(NA_WARPS * 32, 4)
noalloc_kernel(NaArgs a, NaMatrix mat, int2* scratch) {
  __shared__ __align__(16) uint8_t prof[NCODES * 32 * LANE_ROWS_MAX];
  __shared__ __align__(16) uint16_t ring_all[NA_WARPS][2 * NA_COLS + 8];
  __shared__ __align__(16) uint8_t sm[NCODES * SM_ROW];
  __shared__ unsigned long long s_item;
  __shared__ int s_subject, s_qbad;
  for (int i = threadIdx.x; i < NCODES * SM_ROW; i += blockDim.x)
    sm[i] = i % SM_ROW < NCODES ? (uint8_t)mat.sm[i / SM_ROW * NCODES + i % SM_ROW] : 0;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint16_t* ring = ring_all[wib];
  unsigned int* status = (unsigned int*)(scratch + 1);
  const int chunks = (a.ns - 1) / a.chunk + 1;  // per query
  const long long total = (long long)a.nq * chunks;
  const bool rows = blockIdx.x < NA_ROW_BLOCKS;
  int2* hb = scratch + NA_HEADER + (size_t)(rows ? blockIdx.x * NA_WARPS + wib : 0) * NA_MAX_LEN;
  // round 0: the queries of several passes, on the blocks with border rows;
  // round 1: the others, on all blocks
  for (int round = rows ? 0 : 1; round < 2; round++) {
    unsigned long long* counter = (unsigned long long*)scratch + (round == 0 ? 0 : 2);
    int cached = -1;  // the query whose single-pass profile the block holds
    // a block's first item is its index, so few items spread over the SMs
    const unsigned starters = round == 0 ? min(gridDim.x, (unsigned)NA_ROW_BLOCKS) : gridDim.x;
    for (bool start = true;; start = false) {
      __syncthreads();  // the item before is done with the shared words
      if (threadIdx.x == 0) {
        s_item = start ? blockIdx.x : starters + atomicAdd(counter, 1ull);
        s_subject = 0;
      }
      __syncthreads();
      const long long it = (long long)s_item;
      if (it >= total) break;  // uniform over the block
      const int q = (int)(it / chunks), s0 = (int)(it % chunks) * a.chunk;
      const int cnt = min(a.chunk, a.ns - s0);
      const int m = a.qlen[q];
      if ((m > NA_PASS) != (round == 0)) continue;
      // a negative length, or residues to read from a NULL buffer
      const bool q_ok = m >= 0 && (m == 0 || a.qres);
      const uint8_t* qr = a.qres + (q_ok && m > 0 ? a.qoff[q] : 0);
      const int passes = q_ok && m > 0 ? (m + NA_PASS - 1) / NA_PASS : 0;
      const int last_rows = m - (passes - 1) * NA_PASS;
      const int pr = max(1, ((last_rows + 31) / 32 + 3) / 4) * 4;  // of the last pass
      if (passes > 0 && cached != q) {
        if (threadIdx.x == 0) s_qbad = 0;
        __syncthreads();
        int bad = 0;
        for (int i = threadIdx.x; i < m; i += blockDim.x) bad |= qr[i] >= ALPHA;
        if (bad) s_qbad = 1;  // every writer writes 1
        if (passes == 1) {
          na_profile(pr, prof, sm, qr, m, 0, wib);
          cached = q;
        }
        __syncthreads();
      }
      const bool qbad = passes > 0 && s_qbad;
      // the warps take the chunk's subjects one by one; with several passes, in
      // step, since they share each pass's profile
      for (int k = wib;; k += NA_WARPS) {
        if (passes <= 1) {
          if (lane == 0) k = atomicAdd(&s_subject, 1);
          k = __shfl_sync(FULL, k, 0);
          if (k >= cnt) break;
        } else if (k - wib >= cnt) {
          break;  // uniform over the block
        }
        const int s = s0 + min(k, cnt - 1);
        const int n = a.slen[s];
        // refused, with nothing read or written: a bad length on either side
        const bool ok = k < cnt && q_ok && n >= 0 && n <= NA_MAX_LEN && (n == 0 || a.sres);
        if (k < cnt && !ok && lane == 0) atomicOr(status, NA_BAD_LENGTH);
        const uint8_t* d = a.sres + (ok && n > 0 ? a.soff[s] : 0);
        int S = 0, bad = 0;
        if (passes == 1) {
          if (ok && n > 0)
            na_pass<false>(pr, prof, ring, lane, n, d, nullptr, true, true, S, bad, a.go, a.ge);
        } else {
          for (int p = 0; p < passes; p++) {
            const int rows_p = p < passes - 1 ? LANE_ROWS_MAX : pr;
            __syncthreads();  // every warp is done with the profile before
            na_profile(rows_p, prof, sm, qr, m, p * NA_PASS, wib);
            __syncthreads();
            if (ok && n > 0)
              na_pass<true>(rows_p, prof, ring, lane, n, d, hb, p == 0, p == passes - 1, S, bad,
                            a.go, a.ge);
          }
        }
        if (!ok) continue;
        // a code outside the alphabet on either side: the pair gets no score
        bad = __any_sync(FULL, bad) || (qbad && n > 0);
        S = na_warp_max(S);
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
           n_subjects, gap_open + gap_extend, gap_extend, 0};
  // subjects per block item: about eight items per block, and between one
  // subject per warp and 64 (a profile is built per item)
  const int64_t per = (int64_t)n_queries * n_subjects / ((int64_t)na.blocks * 8);
  a.chunk = (int)(per < NA_WARPS ? NA_WARPS : per > 64 ? 64 : (per + NA_WARPS - 1) / NA_WARPS * NA_WARPS);
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
