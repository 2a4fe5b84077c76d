// swgb_internal.h -- types and helpers shared by the CUDA translation units
// of libswgb.  Nothing here is part of the public ABI (include/swgb.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/swgb.h"

namespace swgb {

// ---- alphabet and layout constants ------------------------------------------
constexpr int ALPHA = 24;        // BLOSUM62 symbols A R N D C Q E G H I L K M F P S T W Y V B Z X *
constexpr int PAD_CODE = 24;     // trailing padding residue (never in user input)
constexpr int NCODES = 25;       // ALPHA + PAD
constexpr int PAD_SCORE = -64;   // SM against PAD: trailing cells scoring <= 0 leave S unchanged
constexpr int GROUP = 64;        // subjects per inter-task group (32 lanes x 2 packed subjects)
constexpr int CHUNK = 8;         // residues per subject per interleaved chunk
constexpr int CHUNK_BYTES = GROUP * CHUNK;  // 512 bytes: one chunk of a whole group
constexpr int S16_LIMIT = 32767;
// Score written for a saturated pair that found the flag list full; no
// exact score is negative, so a later pass can find the pair by it.
constexpr int32_t FLAG_SENTINEL = -1;
// Default capacity of a plan's flag list (saturated pairs per search round).
constexpr int64_t DEFAULT_FLAG_CAPACITY = 1 << 20;

// ---- error reporting ----------------------------------------------------------
sw_status sw_set_error(sw_status st, const char* fmt, ...);
sw_status sw_set_cuda_error(cudaError_t err, const char* where);
void sw_clear_error();

#define CUDA_TRY(call)                                                       \
  do {                                                                       \
    cudaError_t _e = (call);                                                 \
    if (_e != cudaSuccess) return ::swgb::sw_set_cuda_error(_e, #call);      \
  } while (0)

// ---- device-resident database view (passed by value to kernels) -------------
struct DbView {
  const uint8_t* inter;  // interleaved groups: [group][chunk][lane][2 subjects][8 residues]
  const int64_t* goff;   // [G] byte offset of each group in `inter`
  const int32_t* glen;   // [G] group length padded to a multiple of CHUNK
  const uint8_t* cont;   // all subjects, sorted by length (descending), contiguous
  const int64_t* coff;   // [N] offset of sorted subject s in `cont`
  const int32_t* clen;   // [N] length of sorted subject s
  const int32_t* perm;   // [G * GROUP] sorted index -> caller index, -1 for padding slots
  int64_t n;             // subjects
  int32_t groups;        // G
  int32_t max_len;       // longest subject
};

// ---- work of the lane-group kernel (lane_kernel.cu) ---------------------------
// One segment: a query against the subject pairs [pair0, pair1) of the length
// order, on groups of lg lanes with pr rows each.  A query of several passes
// has lg = 32, `full` rows per lane (32, less only in a chain) in every pass
// but the last `tail` (1, more only in a chain), and pr in those.  chain: the
// passes of a pair run on the warps of a block, one behind the other, instead
// of one after the other on a warp.
// halves: each lane's rows in two halves, one column apart (a query of one pass).
struct LaneSeg {
  long long first;  // its first block item
  int32_t q, lg, pr, passes, tail, full, chain, halves;
  int32_t pair0, pair1;
};

// ---- per-search parameters, read by the kernels from device memory ----------
// Kept in device memory (not kernel arguments) so that one captured CUDA graph
// serves every batch: a new search only rewrites this block.  Aligned to 16
// bytes: at 8 the lane groups' kernel is compiled to a slower one (5 queries of 74 x
// 546 subjects of 3,100: 0.47 ms of kernel time, then 0.50).
struct alignas(16) SearchParams {
  const uint8_t* qres;    // concatenated query codes
  const int64_t* qoff;    // [nq]
  const int32_t* qlen;    // [nq]
  const int32_t* qorder;  // [nq] query indices, longest first
  int32_t* scores;        // [nq x N] caller order
  // two queries per word (inter2q_kernel.cu): the strip table, per strip
  // (query of half 0, its first row | end bit 31, query of half 1, its first
  // row | end bit 31), query -1 for an empty half; and per stream pair its
  // first strip and strip count
  const int4* strips;
  const int2* spairs;
  int64_t n_inter2_items; // stream pairs x 2 x inter groups (0: it does not run)
  int64_t n_inter_items;  // (query, inter group) items of inter_kernel.cu (0: it does not run)
  // two queries per word for the long subjects (pair2q_kernel.cu): a strip
  // table of 32-row strips and its stream pairs, in the same format
  const int4* strips2;
  const int2* spairs2;
  int64_t n_pair2_items;  // stream pairs x groups of PAIR2_GROUP long subjects (0: the lane groups score them)
  const LaneSeg* lane_segs;  // lane-group kernel: its segments ...
  int64_t n_lane_items;      // ... and block items (0: it does not run)
  int64_t n_intra_items;  // n_long x nq  (int32 intra-task items, when the packed path is off)
  int32_t nq;
  int32_t n_lane_segs;
  int32_t n_spairs;       // stream pairs of the two-query kernel
  int32_t n_spairs2;      // stream pairs of the two-query intra-task kernel
  int32_t n_long;         // sorted subjects [0, n_long) go to the intra-task kernels
  int32_t g_first;        // first inter-task group (n_long / GROUP)
  int32_t go;             // Go = gap_open + gap_extend  (Eq. 2-3)
  int32_t ge;             // Ge = gap_extend
  int32_t sat_threshold;  // packed path: S >= this (32767 - max SM - Go) is recomputed in int32
  int8_t sm[NCODES * NCODES];  // SM(query code, subject code), PAD row/column = PAD_SCORE
};

// ---- per-search device state (zeroed before each search) --------------------
struct SearchState {
  unsigned long long n_flags;     // saturated pairs appended to the flag list
  unsigned long long recompute;   // next flagged pair (int32 intra-task kernel, per block)
  unsigned long long intra_work;  // next int32 intra-task item (per warp)
  unsigned long long work2;       // next work item (two-query inter-task kernel)
  unsigned long long inter_work;  // next work item (two-subject inter-task kernel)
  unsigned long long lane_work;   // next block item (lane-group kernel)
  unsigned long long pair2_work;  // next work item (two-query intra-task kernel, per block)
  unsigned int status;            // reserved: error bits raised on the device
  unsigned int pad;
};

// ---- scratch handed to the kernels --------------------------------------------
struct Scratch {
  uint4* inter_border;        // per warp: [chunk][4][lane] uint4 (H,F words of 2 columns)
  int64_t inter_stride_vec;   // uint4 per warp
  int2* intra_border;         // per warp: [column] (H, F) int32
  int64_t intra_stride;       // int2 per warp
  int2* flags;                // saturated pairs: (query index, sorted subject index)
  int64_t flag_capacity;
  uint2* pair_border;         // lane-group and two-query intra-task kernels, per warp:
                              // [column] (H, F) words of the pass border
  int64_t lane_row0;          // the lane-group kernel's first row
  int64_t pair_stride;        // uint2 per warp
};

// ---- gap classes ------------------------------------------------------------------
// The packed kernels are compiled for two common gap settings with the
// penalties as compile-time constants, besides the general form that reads
// them at run time:
//   class 1: gap_open 10, gap_extend 2 (Go = 12, Ge = 2), the paper's "10/2";
//   class 2: gap_open 11, gap_extend 1 (Go = 12, Ge = 1), BLAST's default.
template <int G> struct GapClass;
template <> struct GapClass<1> { static constexpr int GO = 12, GE = 2; };
template <> struct GapClass<2> { static constexpr int GO = 12, GE = 1; };
constexpr int GAP_CLASSES = 3;
inline int gap_class(int go, int ge) {
  if (go == GapClass<1>::GO && ge == GapClass<1>::GE) return 1;
  if (go == GapClass<2>::GO && ge == GapClass<2>::GE) return 2;
  return 0;
}

// ---- kernel launchers -----------------------------------------------------------
struct KernelConfig {
  int variant;     // inter: packed rows per strip (16/24/32); intra: int32 rows per lane (8/16)
  int warps;       // warps per block
  int blocks;      // grid size
  size_t smem;     // dynamic shared memory per block
};

// Inter-task kernel with two queries per word (inter2q_kernel.cu), 16, 24 or
// 32 rows per strip.
size_t inter2q_smem_bytes(int rows, int warps);
int inter2q_warps(int rows);  // warps per block (one block per SM)
int inter2q_blocks_per_sm(int rows, int warps);  // resident blocks per SM, 0 if none
cudaError_t launch_inter2q(const KernelConfig& kc, int gclass, const DbView& db,
                           const SearchParams* params, SearchState* state, const Scratch& scr,
                           cudaStream_t stream);

// Inter-task kernel with two subjects per word (inter_kernel.cu), for short
// subjects.  Scratch: one inter_border row per warp.
int inter_warps();  // warps per block
int inter_blocks_per_sm();
cudaError_t launch_inter(int gclass, int blocks, const DbView& db, const SearchParams* params,
                         SearchState* state, const Scratch& scr, cudaStream_t stream);

// Int32 intra-task kernel (intra_kernel.cu): int32 items one warp each, then
// flagged pairs one block each.  Scratch: one border row per warp.
constexpr int INTRA_WARPS = 16;  // warps per block
size_t intra_smem_bytes(int rows);
int intra_blocks_per_sm(int rows);
// Clusters of RECOMPUTE_CLUSTER blocks that fit the device at once (0: none, or
// no room for one), at most blocks / RECOMPUTE_CLUSTER.
int recompute_clusters(int rows, int blocks);
// items: int32 items, which leave no flagged pairs; otherwise the flagged pairs,
// on `clusters` clusters (0: none, a block each) or a block each
cudaError_t launch_intra(const KernelConfig& kc, int clusters, bool items, const DbView& db,
                         const SearchParams* params, SearchState* state, const Scratch& scr,
                         cudaStream_t stream);
constexpr int RECOMPUTE_CLUSTER = 16;     // blocks per cluster
constexpr int RECOMPUTE_WARPS = 8;        // warps per block
constexpr int RECOMPUTE_PER_CLUSTER = 4;  // at most so many flagged pairs per cluster

// Flag-list overflow (intra_kernel.cu): appends every pair whose score in
// P->scores is FLAG_SENTINEL to the flag list (up to its capacity, counting
// all of them in state->n_flags), for a further round of the int32 kernel.
cudaError_t launch_collect(int blocks, const DbView& db, const SearchParams* params,
                           SearchState* state, const Scratch& scr, cudaStream_t stream);

// Lane-group kernel, two subjects per word (lane_kernel.cu).  Scratch: one
// pair_border row per warp.
constexpr int LANE_WARPS = 4;  // warps per block
// wide: with the shared memory for chains of more than 8 rows per lane (fewer
// blocks per SM)
int lane_blocks_per_sm(bool wide);
cudaError_t launch_lanes(int gclass, bool wide, int blocks, const DbView& db,
                         const SearchParams* params, SearchState* state, const Scratch& scr,
                         cudaStream_t stream);

// Packed intra-task kernel with two queries per word, long subjects
// (pair2q_kernel.cu): one block of pair2q_warps() warps per SM, one subject
// per warp, 32-row strips; scratch: the pair_border rows [0, blocks x warps).
constexpr int PAIR2_STRIP = 32;  // rows per strip of its strip table
constexpr int PAIR2_GROUP = 12;  // subjects per item (the warps of a block)
int pair2q_warps();
size_t pair2q_smem_bytes();
int pair2q_blocks_per_sm();
cudaError_t launch_pair2q(int gclass, int blocks, const DbView& db, const SearchParams* params,
                          SearchState* state, const Scratch& scr, cudaStream_t stream);
// Plain int32 baseline (Algorithm 1 per cell), one query per launch (plain_kernel.cu).
int plain_blocks_per_sm();
cudaError_t launch_plain(int blocks, const DbView& db, const SearchParams* params, int query,
                         int2* border, const int64_t* border_off, cudaStream_t stream);

// Optimal local alignments with traceback (align_kernel.cu).
struct AlignItem {
  int32_t q;          // query index (SearchParams::qres / qoff / qlen)
  int32_t s;          // sorted subject index
  int64_t bits_off;   // first byte of this pair's direction bits
  int64_t border_off; // first int2 of this pair's pass-border row
  int64_t ops_end;    // the transcript ends just before this byte of the ops buffer
};
struct AlignOut {
  int32_t score;
  int32_t i_end, j_end;      // 1-based cell of the score (0 when it is 0)
  int32_t q_begin, s_begin;  // 0-based first aligned residues
  int32_t n_ops;
  int64_t ops_offset;        // the transcript occupies [ops_offset, ops_offset + n_ops)
};
// int2 of an n-column pair's border rows, one per warp of the team
int64_t align_border_ints(int team, int32_t n);
// bytes of an m x n pair's cells: H in 16 bits (keep_h) or 4 direction bits
int64_t align_bits_bytes(int team, bool keep_h, int32_t m, int32_t n);
// Warps to a pair (each with a border row of the subject's length) for a call
// of n_pairs.
int align_team(int n_pairs, int sms);
cudaError_t launch_align(int team, bool keep_h, int sms, const DbView& db, const SearchParams* params,
                         const AlignItem* items, int n_items, uint8_t* bits, int2* border,
                         AlignOut* out, uint8_t* ops, cudaStream_t stream);

// Integer-pipe microbenchmark (intpeak.cu).
int intpeak_run(int op, int blocks_per_sm, int threads, int iters, double* lane_ops_per_clk_sm,
                double* clock_mhz, double* seconds);

}  // namespace swgb
