// api.cu -- host side of libswgb: the C ABI of include/swgb.h.
//
//   * sw_db_create: sorts subjects by length and builds the two device
//     layouts (interleaved groups of 64 for the inter-task kernels and the
//     lane groups, contiguous for the others); the split of the database by
//     length into a short (inter-task) and long (intra-task) part follows
//     Section III-A.
//   * sw_plan_*: a reusable search context.  Its device memory is allocated
//     once (the host-order scores buffer at the first search that needs it);
//     per search one block is copied (parameters, zeroed counters, queries and
//     work tables) and the kernels it needs are launched, several of them
//     from a CUDA graph (one per gap class and set of kernels).  A flag-list
//     overflow is recomputed in further rounds after that.
//   * sw_search: through a plan kept by the database.
//   * sw_search_plain: the int32 baseline, one kernel launch per query.
//   * sw_align: optimal alignments with traceback of selected pairs.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <memory>
#include <mutex>
#include <new>
#include <numeric>
#include <thread>
#include <vector>

#include "swgb_internal.h"

using namespace swgb;

// ---- errors ---------------------------------------------------------------------
namespace swgb {
static thread_local char g_err[512] = "";

sw_status sw_set_error(sw_status st, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof g_err, fmt, ap);
  va_end(ap);
  return st;
}

sw_status sw_set_cuda_error(cudaError_t err, const char* where) {
  cudaGetLastError();  // clear a sticky launch error so the context stays usable
  return sw_set_error(err == cudaErrorMemoryAllocation ? SW_ENOMEM : SW_ECUDA, "%s: %s", where,
                      cudaGetErrorString(err));
}

void sw_clear_error() { g_err[0] = 0; }
}  // namespace swgb

extern "C" const char* sw_last_error(void) { return g_err; }

// ---- alphabet and BLOSUM62 ------------------------------------------------------
static const char kAlphabet[] = "ARNDCQEGHILKMFPSTWYVBZX*";
static constexpr int kCodeX = 22;

extern "C" sw_status sw_encode(const char* text, int64_t n, uint8_t* out) {
  if (n < 0 || (n > 0 && (!text || !out))) return sw_set_error(SW_EINVAL, "sw_encode: bad arguments");
  int8_t table[256];
  for (int i = 0; i < 256; i++) table[i] = kCodeX;
  for (int c = 0; c < ALPHA; c++) {
    const unsigned char u = (unsigned char)kAlphabet[c];
    table[u] = (int8_t)c;
    if (u >= 'A' && u <= 'Z') table[u - 'A' + 'a'] = (int8_t)c;
  }
  for (int64_t i = 0; i < n; i++) out[i] = (uint8_t)table[(unsigned char)text[i]];
  return SW_OK;
}

// BLOSUM62 (Henikoff & Henikoff 1992), NCBI table in the order of kAlphabet.
// The paper searches with BLOSUM62 (Section IV-A) without printing it.
static const int8_t kBlosum62[ALPHA * ALPHA] = {
    4,  -1, -2, -2, 0,  -1, -1, 0,  -2, -1, -1, -1, -1, -2, -1, 1,  0,  -3, -2, 0,  -2, -1, 0,  -4,
    -1, 5,  0,  -2, -3, 1,  0,  -2, 0,  -3, -2, 2,  -1, -3, -2, -1, -1, -3, -2, -3, -1, 0,  -1, -4,
    -2, 0,  6,  1,  -3, 0,  0,  0,  1,  -3, -3, 0,  -2, -3, -2, 1,  0,  -4, -2, -3, 3,  0,  -1, -4,
    -2, -2, 1,  6,  -3, 0,  2,  -1, -1, -3, -4, -1, -3, -3, -1, 0,  -1, -4, -3, -3, 4,  1,  -1, -4,
    0,  -3, -3, -3, 9,  -3, -4, -3, -3, -1, -1, -3, -1, -2, -3, -1, -1, -2, -2, -1, -3, -3, -2, -4,
    -1, 1,  0,  0,  -3, 5,  2,  -2, 0,  -3, -2, 1,  0,  -3, -1, 0,  -1, -2, -1, -2, 0,  3,  -1, -4,
    -1, 0,  0,  2,  -4, 2,  5,  -2, 0,  -3, -3, 1,  -2, -3, -1, 0,  -1, -3, -2, -2, 1,  4,  -1, -4,
    0,  -2, 0,  -1, -3, -2, -2, 6,  -2, -4, -4, -2, -3, -3, -2, 0,  -2, -2, -3, -3, -1, -2, -1, -4,
    -2, 0,  1,  -1, -3, 0,  0,  -2, 8,  -3, -3, -1, -2, -1, -2, -1, -2, -2, 2,  -3, 0,  0,  -1, -4,
    -1, -3, -3, -3, -1, -3, -3, -4, -3, 4,  2,  -3, 1,  0,  -3, -2, -1, -3, -1, 3,  -3, -3, -1, -4,
    -1, -2, -3, -4, -1, -2, -3, -4, -3, 2,  4,  -2, 2,  0,  -3, -2, -1, -2, -1, 1,  -4, -3, -1, -4,
    -1, 2,  0,  -1, -3, 1,  1,  -2, -1, -3, -2, 5,  -1, -3, -1, 0,  -1, -3, -2, -2, 0,  1,  -1, -4,
    -1, -1, -2, -3, -1, 0,  -2, -3, -2, 1,  2,  -1, 5,  0,  -2, -1, -1, -1, -1, 1,  -3, -1, -1, -4,
    -2, -3, -3, -3, -2, -3, -3, -3, -1, 0,  0,  -3, 0,  6,  -4, -2, -2, 1,  3,  -1, -3, -3, -1, -4,
    -1, -2, -2, -1, -3, -1, -1, -2, -2, -3, -3, -1, -2, -4, 7,  -1, -1, -4, -3, -2, -2, -1, -2, -4,
    1,  -1, 1,  0,  -1, 0,  0,  0,  -1, -2, -2, 0,  -1, -2, -1, 4,  1,  -3, -2, -2, 0,  0,  0,  -4,
    0,  -1, 0,  -1, -1, -1, -1, -2, -2, -1, -1, -1, -1, -2, -1, 1,  5,  -2, -2, 0,  -1, -1, 0,  -4,
    -3, -3, -4, -4, -2, -2, -3, -2, -2, -3, -2, -3, -1, 1,  -4, -3, -2, 11, 2,  -3, -4, -3, -2, -4,
    -2, -2, -2, -3, -2, -1, -2, -3, 2,  -1, -1, -2, -1, 3,  -3, -2, -2, 2,  7,  -1, -3, -2, -1, -4,
    0,  -3, -3, -3, -1, -2, -2, -3, -3, 3,  1,  -2, 1,  -1, -2, -2, 0,  -3, -1, 4,  -3, -2, -1, -4,
    -2, -1, 3,  4,  -3, 0,  1,  -1, 0,  -3, -4, 0,  -3, -3, -2, 0,  -1, -4, -3, -3, 4,  1,  -1, -4,
    -1, 0,  0,  1,  -3, 3,  4,  -2, 0,  -3, -3, 1,  -1, -3, -1, 0,  -1, -3, -2, -2, 1,  4,  -1, -4,
    0,  -1, -1, -1, -2, -1, -1, -1, -1, -1, -1, -1, -1, -1, -2, 0,  0,  -2, -1, -1, -1, -1, -1, -4,
    -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, -4, 1,
};

extern "C" void sw_default_matrix(int8_t* out) {
  if (out) memcpy(out, kBlosum62, sizeof kBlosum62);
}

extern "C" void sw_options_default(sw_options* opt) {
  if (!opt) return;
  opt->rows_per_thread = 32;
  opt->warps_per_block = 8;
  opt->long_cutoff = 1500;
  opt->intra_rows = 8;
  opt->use_graph = 1;
  opt->force_int32 = 0;
  opt->auto_cutoff = 0;
  opt->wide_min_len = 0;
  opt->wide_min_subject = 4096;
  opt->inter_columns = 8;
  opt->overlap_kernels = 0;
  opt->two_query = 1;
  opt->two_query_rows = 32;
  opt->two_query_pairs = 0;
  opt->flag_capacity = 0;
  opt->two_query_long = 1;
}

// ---- small helpers ----------------------------------------------------------------
// Host-side fault injection for tests: with SWGB_FAULT=alloc the device
// allocations of sw_db_create and sw_plan_create report out-of-memory, with
// SWGB_FAULT=copy the first copy of a search reports a failed copy, and with
// SWGB_FAULT=clusters a plan is made as on a device that has no room for a
// cluster of the recompute, so these paths run without a device fault.  Read
// at every call; unset, it changes nothing.
static bool injected_fault(const char* what) {
  const char* f = getenv("SWGB_FAULT");
  return f && strcmp(f, what) == 0;
}

static bool is_device_ptr(const void* p) {
  if (!p) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

template <typename T>
static cudaError_t dalloc(T** p, size_t count) {
  *p = nullptr;
  if (count == 0) count = 1;
  return cudaMalloc((void**)p, count * sizeof(T));
}

static int parallel_threads() {
  unsigned h = std::thread::hardware_concurrency();
  return (int)std::max(1u, std::min(h, 32u));
}

template <typename F>
static void parallel_for(int64_t n, F f) {
  const int nt = (int)std::min<int64_t>(parallel_threads(), std::max<int64_t>(n, 1));
  if (nt <= 1) {
    for (int64_t i = 0; i < n; i++) f(i);
    return;
  }
  std::atomic<int64_t> next(0);
  std::vector<std::thread> th;
  for (int t = 0; t < nt; t++)
    th.emplace_back([&]() {
      for (;;) {
        const int64_t lo = next.fetch_add(64);
        if (lo >= n) break;
        const int64_t hi = std::min(n, lo + 64);
        for (int64_t i = lo; i < hi; i++) f(i);
      }
    });
  for (auto& x : th) x.join();
}

// ---- database -----------------------------------------------------------------------
static void plan_free(sw_plan* p);

// Buffers of sw_align calls, grown to the largest call so far up to the keep
// limits: device memory, and pinned memory for what goes up and comes back.
struct AlignBuffers {
  uint8_t* dev = nullptr;
  uint8_t* pinned = nullptr;
  size_t dev_bytes = 0, pinned_bytes = 0;

  cudaError_t reserve(size_t dev_need, size_t pinned_need) {
    cudaError_t e = cudaSuccess;
    if (dev_bytes < dev_need) {
      cudaFree(dev);
      dev_bytes = 0;
      e = cudaMalloc((void**)&dev, dev_need);
      if (e == cudaSuccess) dev_bytes = dev_need;
      else dev = nullptr;
    }
    if (e == cudaSuccess && pinned_bytes < pinned_need) {
      cudaFreeHost(pinned);
      pinned_bytes = 0;
      e = cudaMallocHost((void**)&pinned, pinned_need);
      if (e == cudaSuccess) pinned_bytes = pinned_need;
      else pinned = nullptr;
    }
    return e;
  }
  // gives back what exceeds the limits (0: everything)
  void trim(size_t dev_keep, size_t pinned_keep) {
    if (dev_bytes > dev_keep) {
      cudaFree(dev);
      dev = nullptr;
      dev_bytes = 0;
    }
    if (pinned_bytes > pinned_keep) {
      cudaFreeHost(pinned);
      pinned = nullptr;
      pinned_bytes = 0;
    }
  }
};

struct sw_db {
  int device = 0;
  DbView view{};
  std::vector<int32_t> glen_h;   // padded group lengths (host copy)
  std::vector<int64_t> gcol_h;   // [G + 1] padded columns of groups [0, g)
  std::vector<int32_t> clen_h;   // sorted lengths (host copy)
  std::vector<int64_t> cres_h;   // [N + 1] residues of sorted subjects [0, s)
  std::vector<int32_t> sorted_of_h;  // caller index -> sorted index
  int64_t residues = 0;
  // owned device buffers
  uint8_t* inter = nullptr;
  int64_t* goff = nullptr;
  int32_t* glen = nullptr;
  uint8_t* cont = nullptr;
  int64_t* coff = nullptr;
  int32_t* clen = nullptr;
  int32_t* perm = nullptr;
  // the plan behind sw_search, kept between calls (guarded by oneshot_mu)
  sw_plan* oneshot = nullptr;
  std::mutex oneshot_mu;
  // sw_align's buffers between calls; a call that finds them in use by another
  // thread takes its own
  AlignBuffers align;
  std::mutex align_mu;
};

static void db_free(sw_db* db) {
  if (!db) return;
  plan_free(db->oneshot);
  int cur = 0;
  cudaGetDevice(&cur);
  cudaSetDevice(db->device);
  cudaFree(db->inter);
  cudaFree(db->goff);
  cudaFree(db->glen);
  cudaFree(db->cont);
  cudaFree(db->coff);
  cudaFree(db->clen);
  cudaFree(db->perm);
  db->align.trim(0, 0);
  cudaSetDevice(cur);
  cudaGetLastError();  // a failed free or device switch leaves no stale error
  delete db;
}

// Device memory for a call or a plan of the database.  What sw_align keeps for
// its next call gives way to it.
template <typename T>
static cudaError_t db_alloc(sw_db* db, T** p, size_t count) {
  cudaError_t e = dalloc(p, count);
  if (e != cudaErrorMemoryAllocation) return e;
  std::unique_lock<std::mutex> kept(db->align_mu, std::try_to_lock);
  if (!kept.owns_lock() || !db->align.dev) return e;  // in use, or nothing there
  cudaGetLastError();
  db->align.trim(0, SIZE_MAX);
  return dalloc(p, count);
}

extern "C" sw_status sw_db_create(const uint8_t* residues, const int32_t* lengths,
                                  int64_t n_subjects, int device, sw_db** out) {
  sw_clear_error();
  if (!out) return sw_set_error(SW_EINVAL, "sw_db_create: out is NULL");
  *out = nullptr;
  if (n_subjects < 0 || n_subjects > (int64_t)INT32_MAX - GROUP)
    return sw_set_error(SW_EINVAL, "sw_db_create: n_subjects %lld out of range", (long long)n_subjects);
  if (n_subjects > 0 && !lengths) return sw_set_error(SW_EINVAL, "sw_db_create: lengths is NULL");
  const int64_t N = n_subjects;
  std::vector<int64_t> off(N);
  int64_t total = 0;
  int32_t max_len = 0;
  for (int64_t i = 0; i < N; i++) {
    if (lengths[i] < 0) return sw_set_error(SW_EINVAL, "sw_db_create: length[%lld] < 0", (long long)i);
    off[i] = total;
    total += lengths[i];
    max_len = std::max(max_len, lengths[i]);
  }
  if (total > 0 && !residues) return sw_set_error(SW_EINVAL, "sw_db_create: residues is NULL");
  for (int64_t i = 0; i < total; i++)
    if (residues[i] >= ALPHA)
      return sw_set_error(SW_EINVAL, "sw_db_create: residue code %d at %lld (codes are 0..23)",
                          (int)residues[i], (long long)i);
  CUDA_TRY(cudaSetDevice(device));

  // sort by length, longest first (stable: ties keep caller order)
  std::vector<int32_t> order(N);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(),
                   [&](int32_t a, int32_t b) { return lengths[a] > lengths[b]; });
  const int32_t G = (int32_t)((N + GROUP - 1) / GROUP);
  std::vector<int32_t> glen(G), clen(N), perm((size_t)G * GROUP, -1);
  std::vector<int64_t> goff(G), coff(N);
  int64_t inter_bytes = 0, c = 0;
  for (int32_t g = 0; g < G; g++) {
    const int32_t L = lengths[order[(size_t)g * GROUP]];  // the group's longest
    glen[g] = (L + CHUNK - 1) / CHUNK * CHUNK;
    goff[g] = inter_bytes;
    inter_bytes += (int64_t)glen[g] * GROUP;
  }
  for (int64_t s = 0; s < N; s++) {
    perm[s] = order[s];
    clen[s] = lengths[order[s]];
    coff[s] = c;
    c += clen[s];
  }
  std::vector<uint8_t> inter((size_t)std::max<int64_t>(inter_bytes, 1)), cont((size_t)std::max<int64_t>(total, 1));
  parallel_for(G, [&](int64_t g) {
    uint8_t* base = inter.data() + goff[g];
    const int32_t L = glen[g];
    for (int k = 0; k < GROUP; k++) {
      const int64_t s = g * GROUP + k;
      const uint8_t* src = s < N ? residues + off[order[s]] : nullptr;
      const int32_t len = s < N ? lengths[order[s]] : 0;
      uint8_t* dst = base + (k >> 1) * 16 + (k & 1) * 8;
      for (int32_t j = 0; j < L; j++)
        dst[(int64_t)(j / CHUNK) * CHUNK_BYTES + (j % CHUNK)] = j < len ? src[j] : (uint8_t)PAD_CODE;
    }
  });
  parallel_for(N, [&](int64_t s) {
    if (clen[s]) memcpy(cont.data() + coff[s], residues + off[order[s]], (size_t)clen[s]);
  });

  sw_db* db = new sw_db();
  db->device = device;
  db->residues = total;
  cudaError_t e = injected_fault("alloc") ? cudaErrorMemoryAllocation : cudaSuccess;
#define DB_ALLOC_COPY(dst, src, count)                                                     \
  if (e == cudaSuccess) e = dalloc(&db->dst, (count));                                     \
  if (e == cudaSuccess && (count) > 0)                                                     \
    e = cudaMemcpy(db->dst, (src), sizeof(*db->dst) * (size_t)(count), cudaMemcpyHostToDevice);
  DB_ALLOC_COPY(inter, inter.data(), inter_bytes);
  DB_ALLOC_COPY(goff, goff.data(), G);
  DB_ALLOC_COPY(glen, glen.data(), G);
  DB_ALLOC_COPY(cont, cont.data(), total);
  DB_ALLOC_COPY(coff, coff.data(), N);
  DB_ALLOC_COPY(clen, clen.data(), N);
  DB_ALLOC_COPY(perm, perm.data(), (int64_t)G * GROUP);
#undef DB_ALLOC_COPY
  if (e != cudaSuccess) {
    sw_status st = sw_set_cuda_error(e, "sw_db_create: device upload");
    db_free(db);
    return st;
  }
  db->view.inter = db->inter;
  db->view.goff = db->goff;
  db->view.glen = db->glen;
  db->view.cont = db->cont;
  db->view.coff = db->coff;
  db->view.clen = db->clen;
  db->view.perm = db->perm;
  db->view.n = N;
  db->view.groups = G;
  db->view.max_len = max_len;
  db->gcol_h.assign((size_t)G + 1, 0);
  for (int32_t g = 0; g < G; g++) db->gcol_h[g + 1] = db->gcol_h[g] + glen[g];
  db->glen_h = std::move(glen);
  db->cres_h.assign((size_t)N + 1, 0);
  for (int64_t s = 0; s < N; s++) db->cres_h[s + 1] = db->cres_h[s] + clen[s];
  db->clen_h = std::move(clen);
  db->sorted_of_h.resize((size_t)N);
  for (int64_t s2 = 0; s2 < N; s2++) db->sorted_of_h[order[s2]] = (int32_t)s2;
  *out = db;
  return SW_OK;
}

extern "C" void sw_db_destroy(sw_db* db) { db_free(db); }
extern "C" int64_t sw_db_subjects(const sw_db* db) { return db ? db->view.n : 0; }
extern "C" int64_t sw_db_residues(const sw_db* db) { return db ? db->residues : 0; }
extern "C" int32_t sw_db_max_length(const sw_db* db) { return db ? db->view.max_len : 0; }

// ---- query batch validation and parameter block ------------------------------------
struct HostBatch {
  std::vector<uint8_t> res_copy;  // only when the caller's queries live on the device
  std::vector<int32_t> len;
  std::vector<int64_t> off;
  std::vector<int32_t> order;
  const uint8_t* res = nullptr;   // host view of the residues
  int64_t total = 0;
  bool res_on_device = false;
};

static sw_status read_batch(const uint8_t* queries, const int32_t* q_lengths, int32_t nq,
                            HostBatch& hb) {
  if (nq < 0) return sw_set_error(SW_EINVAL, "n_queries < 0");
  if (nq > 0 && !q_lengths) return sw_set_error(SW_EINVAL, "q_lengths is NULL");
  hb.len.resize(nq);
  if (nq > 0) {
    if (is_device_ptr(q_lengths)) {
      CUDA_TRY(cudaMemcpy(hb.len.data(), q_lengths, sizeof(int32_t) * nq, cudaMemcpyDeviceToHost));
    } else {
      memcpy(hb.len.data(), q_lengths, sizeof(int32_t) * nq);
    }
  }
  hb.off.resize(nq);
  hb.total = 0;
  for (int32_t i = 0; i < nq; i++) {
    if (hb.len[i] < 0) return sw_set_error(SW_EINVAL, "q_lengths[%d] < 0", i);
    hb.off[i] = hb.total;
    hb.total += hb.len[i];
  }
  if (hb.total > 0 && !queries) return sw_set_error(SW_EINVAL, "queries is NULL");
  hb.res_on_device = hb.total > 0 && is_device_ptr(queries);
  if (hb.res_on_device) {
    hb.res_copy.resize(hb.total);
    CUDA_TRY(cudaMemcpy(hb.res_copy.data(), queries, hb.total, cudaMemcpyDeviceToHost));
    hb.res = hb.res_copy.data();
  } else {
    hb.res = queries;
  }
  for (int64_t i = 0; i < hb.total; i++)
    if (hb.res[i] >= ALPHA)
      return sw_set_error(SW_EINVAL, "query residue code %d at %lld (codes are 0..23)",
                          (int)hb.res[i], (long long)i);
  hb.order.resize(nq);
  std::iota(hb.order.begin(), hb.order.end(), 0);
  std::stable_sort(hb.order.begin(), hb.order.end(),
                   [&](int32_t a, int32_t b) { return hb.len[a] > hb.len[b]; });
  return SW_OK;
}

// Largest gap penalty sum kept on the packed 16-bit path: E and F stay
// >= -(Go + Ge) >= -32768 there.
static constexpr int kPackedMaxGap = 16384;
// Searches smaller than this many cells skip the load-balancing cutoff.
static constexpr double kAutoCutoffMinCells = 1e10;
static constexpr int kMaxGap = 100000000;

// *max_sm: the largest matrix entry (optional).
static sw_status fill_scoring(SearchParams& P, int32_t gap_open, int32_t gap_extend,
                              const int8_t* matrix, bool* packed_ok, int* max_sm = nullptr) {
  if (gap_open < 0 || gap_extend < 0 || gap_open > kMaxGap || gap_extend > kMaxGap)
    return sw_set_error(SW_EINVAL, "gap penalties must be in [0, %d]", kMaxGap);
  int8_t m[ALPHA * ALPHA];
  if (matrix) {
    if (is_device_ptr(matrix)) {
      CUDA_TRY(cudaMemcpy(m, matrix, sizeof m, cudaMemcpyDeviceToHost));
    } else {
      memcpy(m, matrix, sizeof m);
    }
  } else {
    memcpy(m, kBlosum62, sizeof m);
  }
  int maxsm = 0;
  for (int a = 0; a < NCODES; a++)
    for (int b = 0; b < NCODES; b++)
      P.sm[a * NCODES + b] = (a < ALPHA && b < ALPHA) ? m[a * ALPHA + b] : (int8_t)PAD_SCORE;
  for (int i = 0; i < ALPHA * ALPHA; i++) maxsm = std::max(maxsm, (int)m[i]);
  P.go = gap_open + gap_extend;
  P.ge = gap_extend;
  P.sat_threshold = S16_LIMIT - maxsm - P.go;
  *packed_ok = (P.go + P.ge) <= kPackedMaxGap;
  if (max_sm) *max_sm = maxsm;
  return SW_OK;
}

// ---- plan ---------------------------------------------------------------------------------
// segments of the lane-group kernel per query: at most one per shape in a
// large batch, more in a batch of few queries, and two in one of so many that
// no item is long beside the search
constexpr int MAX_SEGS = 8, MAX_SEGS_FEW = 24, MAX_SEGS_MANY = 2;
constexpr int FEW_QUERIES = 32, MANY_QUERIES = 4096;
static constexpr int max_segs(int32_t nq) {
  return nq <= FEW_QUERIES ? MAX_SEGS_FEW : nq <= MANY_QUERIES ? MAX_SEGS : MAX_SEGS_MANY;
}
// the most segments of any batch of up to max_queries queries
static constexpr size_t seg_capacity(int32_t max_queries) {
  const size_t few = (size_t)MAX_SEGS_FEW * std::min(max_queries, FEW_QUERIES);
  const size_t large = (size_t)MAX_SEGS * std::min(max_queries, MANY_QUERIES);
  return std::max(std::max(few, large), (size_t)MAX_SEGS_MANY * max_queries);
}

// An array of a size known once, its elements not initialised: what is never
// used of a plan of large capacity costs no page.
template <typename T>
struct Table {
  std::unique_ptr<T[]> items;
  size_t count = 0;
  bool reserve(size_t n) {
    items.reset(n <= (size_t)PTRDIFF_MAX / sizeof(T) ? new (std::nothrow) T[n] : nullptr);
    count = items ? n : 0;
    return items != nullptr;
  }
  size_t size() const { return count; }
  T* data() const { return items.get(); }
  T& operator[](size_t i) const { return items[i]; }
};

// The upload block: parameters, state, then the tables, each on a 16-byte boundary.
static constexpr size_t block_align(size_t bytes) { return (bytes + 15) & ~(size_t)15; }
static constexpr size_t BLOCK_HEADER = block_align(sizeof(SearchParams)) + block_align(sizeof(SearchState));

// The kernels of one search (bits of sw_plan::kernels): the two-query kernel
// or the lane groups for the long subjects, the lane groups (for the short
// subjects, or for all in one launch) or one of the inter-task kernels for the
// short ones, and the int32 kernel.
// K_WIDE: the lane groups are launched with room for chains of 16 rows.
enum { K_PAIR2 = 1, K_LANES_LONG = 2, K_LANES = 4, K_INTER2 = 8, K_INTER = 16, K_INT32 = 32,
       K_WIDE = 64, K_SETS = 128 };

struct sw_plan {
  sw_db* db = nullptr;
  int device = 0;           // the database's device, kept for plan_free
  sw_options opt{};
  KernelConfig kc2{};       // inter-task kernel, two queries per word
  KernelConfig ikc{};       // int32 intra-task kernel
  int32_t clusters = 0;     // clusters of its recompute of few flagged pairs
  int32_t max_queries = 0;
  int64_t max_residues = 0;
  int32_t g_first = 0;      // first inter-task group under the cutoff
  int32_t sms = 1;
  int32_t pair2_blocks = 0;   // grid of pair2q_kernel
  int32_t inter_blocks = 0;   // grid of inter_kernel
  int32_t lane_blocks[2] = {0, 0};  // grid of lane_kernel: as it is, and wide
  // One device block and its pinned image hold what a search uploads, in one
  // copy: the parameter block, the zeroed state, and the tables that follow
  // (the query arrays, the lane-group segments, the stream pairs, the strip
  // table, the residues), packed back to back.
  uint8_t* block = nullptr;
  uint8_t* block_h = nullptr;
  size_t block_bytes = 0;
  SearchParams* params = nullptr;   // in block
  SearchState* state = nullptr;     // in block
  SearchState* state_h = nullptr;   // pinned: the state a search left
  // the tables while a search is planned
  Table<int4> strips;               // strip tables of the two-query kernels
  Table<int2> spairs;               // their stream pairs
  Table<LaneSeg> segs;
  int32_t* scores_dev = nullptr;  // used when the caller's scores live on the host:
                                  // allocated by the first such search
  cudaStream_t stream = nullptr;  // the stream of the search in flight
  Scratch scr{};
  // graphs, one per gap class (the packed kernels are compiled per class) and
  // set of kernels
  cudaGraphExec_t graphs[GAP_CLASSES][K_SETS] = {};
  int gclass = 0;   // gap class of the search being staged ...
  int kernels = 0;  // ... and its kernels
  int lane_grid = 0;
  cudaEvent_t done = nullptr;
  // before the long subjects' kernel, before and after the short subjects'
  // kernel, after the recompute
  cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
  // overlap_kernels: the short subjects' kernel on a stream of its own
  cudaStream_t side = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
  cudaEvent_t ev_join = nullptr;  // overlap: after both
  double long_share = 0;  // the long subjects' share of the cells (one launch for all)
  bool in_flight = false;
  sw_stats stats{};
  sw_stats pending{};
};

static void plan_free(sw_plan* p) {
  if (!p) return;
  int cur = 0;
  cudaGetDevice(&cur);
  // the plan's own device: its database may already be gone (a garbage
  // collector can finalize the two in either order)
  cudaSetDevice(p->device);
  for (auto& c : p->graphs)
    for (auto& g : c)
      if (g) cudaGraphExecDestroy(g);
  if (p->done) cudaEventDestroy(p->done);
  for (auto& e : p->ev)
    if (e) cudaEventDestroy(e);
  if (p->fork) cudaEventDestroy(p->fork);
  if (p->join) cudaEventDestroy(p->join);
  if (p->ev_join) cudaEventDestroy(p->ev_join);
  if (p->side) cudaStreamDestroy(p->side);
  cudaFree(p->block);
  cudaFree(p->scores_dev);
  cudaFree(p->scr.inter_border);
  cudaFree(p->scr.intra_border);
  cudaFree(p->scr.flags);
  cudaFree(p->scr.pair_border);
  cudaFreeHost(p->block_h);
  cudaFreeHost(p->state_h);
  cudaSetDevice(cur);
  cudaGetLastError();  // a failed free or device switch leaves no stale error
  delete p;
}

extern "C" sw_status sw_plan_create(sw_db* db, int32_t max_queries, int64_t max_query_residues,
                                    const sw_options* opt, sw_plan** out) {
  sw_clear_error();
  if (!out) return sw_set_error(SW_EINVAL, "sw_plan_create: out is NULL");
  *out = nullptr;
  if (!db) return sw_set_error(SW_EINVAL, "sw_plan_create: db is NULL");
  if (max_queries < 1 || max_query_residues < 0)
    return sw_set_error(SW_EINVAL, "sw_plan_create: bad capacity");
  sw_options o;
  sw_options_default(&o);
  if (opt) o = *opt;
  if (o.rows_per_thread != 16 && o.rows_per_thread != 32)
    return sw_set_error(SW_EINVAL, "rows_per_thread must be 16 or 32");
  if (o.intra_rows != 8 && o.intra_rows != 16)
    return sw_set_error(SW_EINVAL, "intra_rows must be 8 or 16");
  if (o.warps_per_block < 1 || o.warps_per_block > 8)
    return sw_set_error(SW_EINVAL, "warps_per_block must be 1..8");
  if (o.long_cutoff < 0) return sw_set_error(SW_EINVAL, "long_cutoff < 0");
  if (o.inter_columns != 4 && o.inter_columns != 8)
    return sw_set_error(SW_EINVAL, "inter_columns must be 4 or 8");
  if (o.wide_min_len < 0 || o.wide_min_subject < 0)
    return sw_set_error(SW_EINVAL, "wide_min_len and wide_min_subject must be >= 0");
  if (o.flag_capacity < 0) return sw_set_error(SW_EINVAL, "flag_capacity < 0");
  if (o.two_query < 0 || o.two_query > 2) return sw_set_error(SW_EINVAL, "two_query must be 0, 1 or 2");
  if (o.two_query_rows != 16 && o.two_query_rows != 24 && o.two_query_rows != 32)
    return sw_set_error(SW_EINVAL, "two_query_rows must be 16, 24 or 32");
  if (o.two_query_pairs < 0) return sw_set_error(SW_EINVAL, "two_query_pairs < 0");
  if (o.two_query_long < 0 || o.two_query_long > 2)
    return sw_set_error(SW_EINVAL, "two_query_long must be 0, 1 or 2");
  CUDA_TRY(cudaSetDevice(db->device));

  sw_plan* p = new (std::nothrow) sw_plan();
  if (!p) return sw_set_error(SW_ENOMEM, "sw_plan_create: out of host memory");
  p->db = db;
  p->device = db->device;
  p->opt = o;
  p->max_queries = max_queries;
  p->max_residues = max_query_residues;
  const DbView& v = db->view;
  // groups whose longest subject exceeds the cutoff go to the intra-task kernel
  int32_t gf = 0;
  if (o.force_int32) {
    gf = v.groups;
  } else {
    while (gf < v.groups && db->glen_h[gf] > o.long_cutoff) gf++;
  }
  p->g_first = gf;
  const int32_t L_inter = gf < v.groups ? db->glen_h[gf] : 0;

  int dev_sms = 0;
  cudaDeviceGetAttribute(&dev_sms, cudaDevAttrMultiProcessorCount, db->device);
  p->sms = dev_sms;
  // the two-query kernel: one block per SM, as many warps as its shared memory allows
  const int warps2 = inter2q_warps(o.two_query_rows);
  const int bps2 = inter2q_blocks_per_sm(o.two_query_rows, warps2);
  if (bps2 < 1) {
    plan_free(p);
    return sw_set_error(SW_ECUDA, "two-query inter-task kernel cannot launch (rows %d)",
                        o.two_query_rows);
  }
  p->kc2.variant = o.two_query_rows;
  p->kc2.warps = warps2;
  p->kc2.blocks = dev_sms * bps2;
  p->kc2.smem = inter2q_smem_bytes(o.two_query_rows, warps2);
  const int ibps = inter_blocks_per_sm();
  if (ibps < 1) {
    plan_free(p);
    return sw_set_error(SW_ECUDA, "inter-task kernel cannot launch");
  }
  p->inter_blocks = dev_sms * ibps;
  // border rows of the inter-task kernels, of which a search launches one
  const int64_t W = std::max((int64_t)p->kc2.blocks * p->kc2.warps,
                             (int64_t)p->inter_blocks * inter_warps());
  // one block of INTRA_WARPS per SM: enough for the int32 items, and the
  // border scratch (one subject-length row per warp) stays bounded
  if (intra_blocks_per_sm(o.intra_rows) < 1) {
    plan_free(p);
    return sw_set_error(SW_ECUDA, "int32 intra-task kernel cannot launch (rows %d)", o.intra_rows);
  }
  p->ikc.variant = o.intra_rows;
  p->ikc.warps = INTRA_WARPS;
  p->ikc.blocks = dev_sms;
  p->ikc.smem = intra_smem_bytes(o.intra_rows);
  p->clusters = injected_fault("clusters") ? 0 : recompute_clusters(o.intra_rows, p->ikc.blocks);
  const int64_t WI = (int64_t)p->ikc.blocks * INTRA_WARPS;
  for (int wide = 0; wide < 2; wide++) {
    const int lbps = lane_blocks_per_sm(wide != 0);
    if (lbps < 1) {
      plan_free(p);
      return sw_set_error(SW_ECUDA, "lane-group kernel cannot launch");
    }
    p->lane_blocks[wide] = dev_sms * lbps;
  }
  const int p2bps = pair2q_blocks_per_sm();
  if (p2bps < 1) {
    plan_free(p);
    return sw_set_error(SW_ECUDA, "two-query packed intra-task kernel cannot launch");
  }
  p->pair2_blocks = dev_sms * p2bps;
  // border rows of the two-query intra-task kernel and of the lane-group
  // kernel, which share them unless overlap_kernels runs them side by side
  const int64_t rows2 = (int64_t)p->pair2_blocks * pair2q_warps();
  const int64_t rowsl = (int64_t)std::max(p->lane_blocks[0], p->lane_blocks[1]) * LANE_WARPS;
  const int64_t WP = o.overlap_kernels ? rows2 + rowsl : std::max(rows2, rowsl);
  p->scr.lane_row0 = o.overlap_kernels ? rows2 : 0;

  cudaError_t e = injected_fault("alloc") ? cudaErrorMemoryAllocation : cudaSuccess;
  p->scr.inter_stride_vec = (int64_t)(L_inter / CHUNK) * 4 * 32;
  p->scr.intra_stride = std::max(v.max_len, 1);
  // (the lane kernel's rows start 64 columns before the first and end 4 after
  // the last; the two-query pair kernel loads its border 4 columns ahead)
  p->scr.pair_stride = std::max(v.max_len, 1) + 72;
  p->scr.flag_capacity = o.flag_capacity > 0
                            ? (int64_t)o.flag_capacity
                            : std::min<int64_t>((int64_t)max_queries * std::max<int64_t>(v.n, 1),
                                                DEFAULT_FLAG_CAPACITY);
  // strips of the two tables (the inter-task kernel's, at least 16 rows per
  // strip, and the intra-task kernel's, 32): every query padded to whole
  // strips (at least one), and as many empty halves at most; stream pairs:
  // one per two queries at most, per table
  if (!p->strips.reserve(2 * ((size_t)max_query_residues / 16 + 2 * (size_t)max_queries) + 16) ||
      !p->spairs.reserve(2 * ((size_t)max_queries / 2 + 1)) ||
      !p->segs.reserve(seg_capacity(max_queries))) {
    plan_free(p);
    return sw_set_error(SW_ENOMEM, "sw_plan_create: out of host memory for %d queries of %lld residues",
                        max_queries, (long long)max_query_residues);
  }
  p->block_bytes = BLOCK_HEADER + block_align((size_t)max_queries * sizeof(int64_t)) +
                   2 * block_align((size_t)max_queries * sizeof(int32_t)) +
                   block_align(p->segs.size() * sizeof(LaneSeg)) +
                   block_align(p->spairs.size() * sizeof(int2)) +
                   block_align(p->strips.size() * sizeof(int4)) +
                   block_align((size_t)std::max<int64_t>(max_query_residues, 1));
  if (e == cudaSuccess) e = db_alloc(db, &p->scr.pair_border, (size_t)(WP * p->scr.pair_stride));
  if (e == cudaSuccess) e = db_alloc(db, &p->block, p->block_bytes);
  if (e == cudaSuccess) e = db_alloc(db, &p->scr.inter_border, (size_t)(W * std::max<int64_t>(p->scr.inter_stride_vec, 1)));
  if (e == cudaSuccess) e = db_alloc(db, &p->scr.intra_border, (size_t)(WI * p->scr.intra_stride));
  if (e == cudaSuccess) e = db_alloc(db, &p->scr.flags, (size_t)p->scr.flag_capacity);
  if (e == cudaSuccess) e = cudaMallocHost((void**)&p->block_h, p->block_bytes);
  if (e == cudaSuccess) e = cudaMallocHost((void**)&p->state_h, sizeof(SearchState));
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->done, cudaEventDisableTiming);
  for (auto& ev : p->ev)
    if (e == cudaSuccess) e = cudaEventCreate(&ev);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->join, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&p->side, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreate(&p->ev_join);
  if (e != cudaSuccess) {
    sw_status st = sw_set_cuda_error(e, "sw_plan_create: allocation");
    plan_free(p);
    return st;
  }
  p->params = (SearchParams*)p->block;
  p->state = (SearchState*)(p->block + block_align(sizeof(SearchParams)));
  memset(p->block_h, 0, BLOCK_HEADER);
  memset(p->state_h, 0, sizeof(SearchState));
  *out = p;
  return SW_OK;
}

extern "C" void sw_plan_destroy(sw_plan* plan) {
  if (plan && plan->in_flight) cudaEventSynchronize(plan->done);
  plan_free(plan);
}

// The device work of one search, after the upload of its parameters and
// zeroed counters: the kernel of the long subjects, that of the short ones
// (or the lane-group kernel for both) and the int32 intra-task kernel
// (saturated pairs, or everything when the packed path is off) -- those of
// p->kernels, in launches of their own.  Events around the kernels give their
// device time on the launching stream.  Under stream capture an event record
// only orders the capture unless it carries cudaEventRecordExternal, which
// makes it a real event-record node of the graph; outside capture that flag
// is illegal.
static cudaError_t record(cudaEvent_t ev, cudaStream_t s, bool capturing) {
  return capturing ? cudaEventRecordWithFlags(ev, s, cudaEventRecordExternal)
                   : cudaEventRecord(ev, s);
}

static cudaError_t enqueue_kernels(sw_plan* p, cudaStream_t s, bool capturing) {
  const int gc = p->gclass, set = p->kernels;
  const DbView& v = p->db->view;
  // with a kernel for the long subjects and one for the short ones,
  // overlap_kernels issues the latter on a second stream: one of its blocks
  // needs a whole SM's shared memory, so it starts on an SM when the blocks
  // there run out of work, and no SM idles in their tails
  const bool is_long = set & (K_PAIR2 | K_LANES_LONG), is_short = set & (K_LANES | K_INTER2 | K_INTER);
  const bool overlap = p->opt.overlap_kernels && is_long && is_short, wide = set & K_WIDE;
  cudaError_t e = record(p->ev[0], s, capturing);
  if (e == cudaSuccess && overlap) e = cudaEventRecord(p->fork, s);
  if (e == cudaSuccess && (set & K_PAIR2))
    e = launch_pair2q(gc, p->pair2_blocks, v, p->params, p->state, p->scr, s);
  if (e == cudaSuccess && (set & K_LANES_LONG))
    e = launch_lanes(gc, wide, p->lane_grid, v, p->params, p->state, p->scr, s);
  cudaStream_t s2 = s;
  if (overlap) {
    s2 = p->side;
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s2, p->fork, 0);
  }
  if (e == cudaSuccess && is_long && is_short) e = record(p->ev[1], s, capturing);
  if (e == cudaSuccess && (set & K_LANES))
    e = launch_lanes(gc, wide, p->lane_grid, v, p->params, p->state, p->scr, s2);
  if (e == cudaSuccess && (set & K_INTER2))
    e = launch_inter2q(p->kc2, gc, v, p->params, p->state, p->scr, s2);
  if (e == cudaSuccess && (set & K_INTER))
    e = launch_inter(gc, p->inter_blocks, v, p->params, p->state, p->scr, s2);
  if (e == cudaSuccess) e = record(p->ev[2], s2, capturing);
  if (overlap) {
    if (e == cudaSuccess) e = cudaEventRecord(p->join, s2);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, p->join, 0);
    if (e == cudaSuccess) e = record(p->ev_join, s, capturing);
  }
  if (set & K_INT32) {
    if (e == cudaSuccess) e = launch_intra(p->ikc, p->clusters, (set & ~K_INT32) == 0, v, p->params, p->state, p->scr, s);
    if (e == cudaSuccess) e = record(p->ev[3], s, capturing);
  }
  return e;
}

static cudaError_t run_kernels(sw_plan* p, cudaStream_t s) {
  // one kernel is launched as it is, on a grid of its size
  const int launches = p->kernels & ~K_WIDE;
  const bool single = (launches & (launches - 1)) == 0;
  if (!p->opt.use_graph || single) return enqueue_kernels(p, s, false);
  p->lane_grid = p->lane_blocks[(p->kernels & K_WIDE) != 0];  // a graph serves searches of any size
  cudaGraphExec_t& graph = p->graphs[p->gclass][p->kernels];
  if (!graph) {
    cudaStream_t cs;
    cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    cudaGraph_t g = nullptr;
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      cudaError_t e2 = enqueue_kernels(p, cs, true);
      e = cudaStreamEndCapture(cs, &g);
      if (e2 != cudaSuccess) e = e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&graph, g, 0);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cs);
    if (e != cudaSuccess) {
      graph = nullptr;
      return e;
    }
  }
  return cudaGraphLaunch(graph, s);
}

// Splits the queries of one stream pair between its two streams so that the
// longer stream is as short as the strip counts allow: an exact subset sum
// over the pair's queries (reachable sums as bit sets, one per prefix of the
// queries, then a walk back from the largest sum not above half the total).
// Dealing longest first leaves the two streams of a pair up to a query's
// length apart; this closes the gap.  Pairs of more than 64 queries keep the
// dealt split (with many short queries it is already even).
static void balance_pair(std::vector<int32_t>& a, std::vector<int32_t>& b, int64_t& la,
                         int64_t& lb, const std::vector<int64_t>& strips_of) {
  std::vector<int32_t> all(a);
  all.insert(all.end(), b.begin(), b.end());
  const size_t n = all.size();
  const int64_t S = la + lb, H = S / 2;
  if (n < 2 || n > 64 || std::max(la, lb) == S - H) return;
  const size_t W = (size_t)(H / 64 + 1);
  const uint64_t top_mask = (H % 64 == 63) ? ~0ull : ((2ull << (H % 64)) - 1);
  std::vector<uint64_t> reach((n + 1) * W, 0);
  reach[0] = 1;  // the empty set sums to 0
  for (size_t i = 0; i < n; i++) {
    const uint64_t* src = &reach[i * W];
    uint64_t* dst = &reach[(i + 1) * W];
    const int64_t sh = strips_of[all[i]];
    const size_t ws = (size_t)(sh / 64);
    const int bs = (int)(sh % 64);
    for (size_t w = 0; w < W; w++) {
      uint64_t v = src[w];
      if (w >= ws) {
        v |= src[w - ws] << bs;
        if (bs && w > ws) v |= src[w - ws - 1] >> (64 - bs);
      }
      dst[w] = v;
    }
    dst[W - 1] &= top_mask;  // sums above H are not kept
  }
  const uint64_t* fin = &reach[n * W];
  int64_t t = H;
  while (t > 0 && !((fin[t / 64] >> (t % 64)) & 1)) t--;
  if (S - t >= std::max(la, lb)) return;
  std::vector<int32_t> taken, rest;
  int64_t r = t;
  for (size_t i = n; i-- > 0;) {
    const uint64_t* prev = &reach[i * W];
    if ((prev[r / 64] >> (r % 64)) & 1) {
      rest.push_back(all[i]);  // the sum r is reachable without query i
    } else {
      taken.push_back(all[i]);
      r -= strips_of[all[i]];
    }
  }
  a.assign(rest.rbegin(), rest.rend());
  b.assign(taken.rbegin(), taken.rend());
  la = S - t;
  lb = t;
}

// Query streams for two queries per word (inter2q_kernel.cu and
// pair2q_kernel.cu): deals the batch's queries to 2K streams, longest first,
// each to the stream with the fewest strips so far (each query padded to
// whole strips of T rows, at least one), pairs streams 2k and 2k + 1 and
// balances each pair's two streams (balance_pair).
// Unless fixed_K > 0, K is the power of two, at most nq / 2, for which the
// search is expected to end first.  Fewer, longer streams pad less (a stream
// pair is as long as its longer stream, in units of `unit` strips, and the
// fewer queries a pair holds the less evenly its two streams split), but an
// item is as long as its stream pair: the longest one -- the longest column
// set (len_max) against the longest pair -- takes `len_max x strips`, and the
// whole search len_sum columns against every pair over `workers`.  Items run
// longest first, so a longest item well within the search costs little: kTail
// of its length (20 queries of 144-5,478 x 100,000 subjects took 126.3, 129.4
// and 135.9 ms with 2, 4 and 8 pairs, 96 of 50-2,000 402, 395 and 395 with 2, 4
// and 8).  Writes the strip table (per strip: the query of each half, its
// first row | end bit 31; query -1 for an empty half) to tab and per stream
// pair (first strip, counted from first_strip, strips) to pairs.  Returns K, or
// 0 when the table would exceed cap strips; *n_strips is the table's length.
static int32_t deal_streams(const HostBatch& hb, int32_t nq, int T, int32_t fixed_K,
                            double workers, int unit, double len_max, double len_sum,
                            int4* tab, int2* pairs, int64_t first_strip, int64_t cap,
                            int64_t* n_strips) {
  *n_strips = 0;
  std::vector<int64_t> strips_of((size_t)nq);
  for (int32_t i = 0; i < nq; i++) strips_of[i] = std::max<int64_t>(1, (hb.len[i] + T - 1) / T);
  std::vector<std::vector<int32_t>> streams;
  std::vector<int64_t> load;
  // the streams as a heap, the shortest (of equals the first) on top
  std::vector<std::pair<int64_t, int32_t>> heap;
  auto deal = [&](int32_t K) {
    streams.resize((size_t)2 * K);
    for (auto& s : streams) s.clear();
    load.assign((size_t)2 * K, 0);
    heap.resize((size_t)2 * K);
    for (int32_t t = 0; t < 2 * K; t++) heap[(size_t)t] = {0, t};
    for (int32_t i = 0; i < nq; i++) {
      const int32_t q = hb.order[i];
      std::pop_heap(heap.begin(), heap.end(), std::greater<>());
      auto& top = heap.back();
      streams[(size_t)top.second].push_back(q);
      top.first += strips_of[q];
      load[(size_t)top.second] = top.first;
      std::push_heap(heap.begin(), heap.end(), std::greater<>());
    }
    for (int32_t k = 0; k < K; k++)
      balance_pair(streams[2 * k], streams[2 * k + 1], load[2 * k], load[2 * k + 1], strips_of);
  };
  auto pair_strips = [&](int32_t k) { return std::max(load[2 * k], load[2 * k + 1]); };
  constexpr double kTail = 0.045;
  int32_t K = fixed_K > 0 ? std::min(fixed_K, nq / 2) : 1;
  if (fixed_K == 0) {
    double best = 1e300;
    for (int32_t k2 = 1; k2 <= nq / 2; k2 *= 2) {
      deal(k2);
      int64_t smax = 0, ssum = 0;
      for (int32_t k = 0; k < k2; k++) {
        const int64_t S = (pair_strips(k) + unit - 1) / unit * unit;
        smax = std::max(smax, S);
        ssum += S;
      }
      const double all = len_sum * (double)ssum / workers, longest = len_max * (double)smax;
      const double t = std::max(all, longest) + kTail * std::min(all, longest);
      if (t < best) {
        best = t;
        K = k2;
      }
      if (longest < 0.2 * all) break;  // more pairs only pad more
    }
  }
  deal(K);
  int64_t total = 0;
  for (int32_t k = 0; k < K; k++) total += pair_strips(k);
  if (total > cap) return 0;
  int64_t at = 0;
  for (int32_t k = 0; k < K; k++) {
    const int64_t S = pair_strips(k);
    pairs[k] = make_int2((int32_t)(first_strip + at), (int32_t)S);
    // each half walks its stream: query index, first row, end bit
    int4* t4 = tab + at;
    for (int half = 0; half < 2; half++) {
      const std::vector<int32_t>& st = streams[2 * k + half];
      size_t qi = 0;
      int64_t row = 0;
      for (int64_t s = 0; s < S; s++) {
        int32_t q = -1, first = 0;
        if (qi < st.size()) {
          q = st[qi];
          first = (int32_t)row;
          row += T;
          if (row >= (int64_t)strips_of[q] * T) {  // this query's last strip
            first |= (int32_t)0x80000000u;
            ++qi;
            row = 0;
          }
        }
        if (half == 0) {
          t4[s].x = q;
          t4[s].y = first;
        } else {
          t4[s].z = q;
          t4[s].w = first;
        }
      }
    }
    at += S;
  }
  *n_strips = at;
  return K;
}

// The fewest strips that stream pairs of these queries can have, in all and in the
// longest pair.
struct StreamFloor {
  int64_t strips, longest;
};
static StreamFloor stream_floor(const HostBatch& hb, int32_t nq, int T) {
  StreamFloor f{0, 0};
  for (int32_t i = 0; i < nq; i++) {
    const int64_t s = std::max<int64_t>(1, (hb.len[i] + T - 1) / T);
    f.strips += s;
    f.longest = std::max(f.longest, s);
  }
  f.strips = (f.strips + 1) / 2;
  return f;
}

// The short subjects' two-query layout (inter2q_kernel.cu): items are
// (stream pair, half of a 64-subject group), the workers its warps.  Returns
// the number of stream pairs, and in *cycles what the layout is expected to
// take, in SM cycles: the larger of kQ2WordCycles per word row and scheduler
// and the longest item, whose warp shares its scheduler with one other, and a
// part of the smaller for the search's end (the larger alone took this kernel
// for 3 queries of 400 x 222,000: 27.3 ms, the lane groups 20.1; 5 of 400 x
// 71,000: 11.4 and 9.1).  Returns 0, without dealing, when no deal could take
// less than `limit` (14 queries took longer to deal than to score against 4
// subjects).  A strip costs kQ2StripCycles beside its words, for its profile and
// its ends: 20 queries of 375 x 570,000 subjects of 5-15 residues take 11.9 ms,
// of which the words alone would be 6.5.  (2 to 20 queries of 300-2,000 x 20,000
// to 570,000 subjects: within 8% of the time measured.)
static constexpr double kQ2WordCycles = 9.0, kQ2ItemCycles = 16.5, kQ2StripCycles = 3000;
static int32_t plan_streams(sw_plan* p, const HostBatch& hb, int32_t nq, int32_t g_first,
                            double limit, int64_t* n_strips, double* cycles) {
  const int T = p->kc2.variant;
  const DbView& v = p->db->view;
  *n_strips = 0;
  const double glen_sum = (double)(p->db->gcol_h[v.groups] - p->db->gcol_h[g_first]);
  const double glen_max = g_first < v.groups ? p->db->glen_h[g_first] : 0.0;
  // scheduler cycles of a strip of every half group, and those of the longest
  // group's on a warp
  const double strip = 2 * (kQ2WordCycles * T * glen_sum + kQ2StripCycles * (v.groups - g_first)) /
                       (4.0 * p->sms);
  const double item_strip = kQ2ItemCycles * T * glen_max + 2 * kQ2StripCycles;
  auto end_of = [](double all, double item) {  // as for the lane groups
    return std::max(all, item) + 0.2 * std::min(all, item);
  };
  const StreamFloor least = stream_floor(hb, nq, T);
  if (end_of((double)least.strips * strip, (double)least.longest * item_strip) >= limit) return 0;
  const int32_t K = deal_streams(hb, nq, T, p->opt.two_query_pairs,
                                 (double)p->kc2.blocks * p->kc2.warps, 1, glen_max, 2 * glen_sum,
                                 p->strips.data(), p->spairs.data(), 0,
                                 (int64_t)p->strips.size(), n_strips);
  int64_t longest = 0;
  for (int32_t k = 0; k < K; k++) longest = std::max<int64_t>(longest, p->spairs[(size_t)k].y);
  *cycles = end_of((double)*n_strips * strip, (double)longest * item_strip);
  // Items of about one length end in whole rounds: of the first r W + 1 some warp
  // takes r + 1 (32 queries of 12,234 x 3,345 subjects of 89, 1.4 items per warp:
  // 21.8 ms, two subjects per word 19.3).
  const int64_t W = (int64_t)p->kc2.blocks * p->kc2.warps;
  for (int64_t r = 1; r < 8 && K > 0 && r * W < (int64_t)K * 2 * (v.groups - g_first); r++) {
    const double L = p->db->glen_h[(size_t)(g_first + r * W / K / 2)];
    *cycles = std::max(*cycles, (double)(r + 1) * (double)*n_strips / K *
                                    (kQ2ItemCycles * T * L + 2 * kQ2StripCycles));
  }
  return K;
}

// The long subjects' two-query layout (pair2q_kernel.cu), its table placed
// after the short subjects' (first_strip, first_pair): items are (stream
// pair, group of PAIR2_GROUP long subjects), the workers its blocks.  Returns the
// number of stream pairs, and in *cycles what the layout is expected to take:
// the passes' steps of 32 words, three warps to a scheduler, over as many
// rounds of blocks as the items need, or the longest item.
static constexpr double kP2WordCycles = 8.9;
static int32_t plan_streams_long(sw_plan* p, const HostBatch& hb, int32_t nq, int64_t n_long,
                                 int64_t first_strip, int32_t first_pair, double limit,
                                 int64_t* n_strips, double* cycles) {
  *n_strips = 0;
  if (nq < 2 || n_long <= 0) return 0;
  const int32_t* clen = p->db->clen_h.data();
  double len_sum = 0;
  for (int64_t s = 0; s < n_long; s += PAIR2_GROUP) len_sum += clen[s];
  const double groups = (double)((n_long + PAIR2_GROUP - 1) / PAIR2_GROUP);
  const double step = 3 * 32 * kP2WordCycles;  // cycles per step of a block's three warps
  const double all_steps = step * (len_sum + 127 * groups), item_steps = step * ((double)clen[0] + 127);
  const StreamFloor least = stream_floor(hb, nq, PAIR2_STRIP);
  if (std::max((double)((least.strips + 31) / 32) * all_steps / p->sms,
               (double)((least.longest + 31) / 32) * item_steps) >= limit)
    return 0;
  const int32_t K = deal_streams(hb, nq, PAIR2_STRIP, p->opt.two_query_pairs,
                                 (double)p->pair2_blocks, 32, clen[0],
                                 len_sum, p->strips.data() + first_strip,
                                 p->spairs.data() + first_pair, first_strip,
                                 (int64_t)p->strips.size() - first_strip, n_strips);
  double total = 0, longest = 0;
  for (int32_t k = 0; k < K; k++) {
    const double passes = (double)((p->spairs[(size_t)(first_pair + k)].y + 31) / 32);
    total += passes * all_steps;
    longest = std::max(longest, passes * item_steps);
  }
  *cycles = std::max(total / p->sms, longest);
  return K;
}

// The short subjects on the two-subject inter-task kernel (inter_kernel.cu):
// items are (query, group of 64), the workers its warps, two to a scheduler.
// Returns what it is expected to take, in SM cycles, as plan_streams does.
// Fitted to 1 to 20 queries of 144-5,478 residues x 100,000 to 570,000 subjects of
// 5-15 to 250-350 residues: within 8% of the time measured above 0.4 ms.
static constexpr double kIWordCycles = 10.5, kIStripCycles = 1000, kIItemCycles = 18;
static double plan_groups(const sw_plan* p, const HostBatch& hb, int32_t nq, int32_t g_first) {
  const sw_db* db = p->db;
  const int32_t G = db->view.groups;
  double strips = 0;
  for (int32_t i = 0; i < nq; i++) strips += (hb.len[i] + 31) / 32;
  const double longest = (double)((hb.len[hb.order[0]] + 31) / 32);
  const double all = strips * (kIWordCycles * 32 * (double)(db->gcol_h[G] - db->gcol_h[g_first]) +
                               kIStripCycles * (G - g_first)) / (4.0 * p->sms);
  const double item = longest * (kIItemCycles * 32 * db->glen_h[g_first] + 2 * kIStripCycles);
  return std::max(all, item) + 0.2 * std::min(all, item);
}

// The lane-group kernel's segments (lane_kernel.cu) for the subject pairs
// [pair0, pair1): per query up to one per shape.  A shape costs, per subject
// pair, (columns + ramp) steps of every pass on LG / 32 of a warp.  The cheapest
// shape is used, except where one item of it would take longer than `tail` of
// the whole search: those subjects (a prefix, longest first) go to a shape
// with shorter items, a larger group, halves or a chain.
// Measured cycles of a step with PR rows per lane: of a scheduler with four
// warps, 98, 185, 273 and 366 for 8, 16, 24 and 32 rows, 94 and 262 for 8 and
// 24 rows in halves, 65 and 102 for 4 and 8 rows in a chain; of a warp alone,
// 158, 284, 403 and 559, in halves 108 and 280, in a chain 118 and 123.
struct LaneCand {
  int lg, pr, passes, full, chain, halves;
  int tail = 1;  // passes of pr rows at the end, the others of `full`
  int ramp() const { return halves ? 2 * lg : lg; }
  double busy(int rows) const {  // scheduler cycles of a step
    return ((halves ? 10.5 : 11.1) * rows + 9) * (chain ? 1.1 : 1.0);
  }
  double alone(int rows) const {  // cycles of a step on a scheduler of its own
    return (halves ? 10.7 * rows + 22 : 16.0 * rows + 30) + (chain ? 18 : 0);
  }
  // scheduler cycles of one step of every pass
  double thr() const { return (passes - tail) * busy(full) + tail * busy(pr); }
  // cycles of the passes over n columns when `share` warps share a scheduler
  double item(double n, double share) const {
    if (!chain)
      return (n + ramp()) * std::max((passes - 1) * alone(full) + alone(pr), share * thr());
    const double step = std::max(alone(full), share * busy(full));
    const double lag = full == 4 ? 3 : 4;
    const double stages = (n + ramp()) / 32 + 1, period = std::max(stages, LANE_WARPS * lag);
    if (tail > 1)
      return ((passes - tail) / LANE_WARPS * period * step +
              ((tail - 1) * lag + stages) * std::max(alone(pr), share * busy(pr))) * 32;
    return ((passes - 1) / LANE_WARPS * period + (passes - 1) % LANE_WARPS * lag + stages) * 32 * step;
  }
};

// A block item costs kLaneItemCycles on each of its schedulers beside its steps,
// which counts where subjects are short (185 queries of 71 x 31,600 subjects of 11,
// 183,000 items: 2.05 ms, estimated at 1.33 without this term, 1.79 with it).
static constexpr double kLaneItemCycles = 800;

// The shapes for a query of m residues: 8, 16 and 32 lanes; 32 lanes in halves;
// chains of 4 to 16 rows per lane (16 only with the wide launch).
static constexpr int MAX_SHAPES = 12;
static int lane_candidates(int32_t m, bool wide, LaneCand* c) {
  int n = 0;
  auto fit = [](int rows, int step) { return std::max(step, (rows + step - 1) / step * step); };
  for (int lg = 8; lg <= 32; lg *= 2) {
    const int passes = lg == 32 ? std::max(1, (m + 1023) / 1024) : 1;
    const int rows = (m - (passes - 1) * 1024 + lg - 1) / lg;  // per lane, last pass
    if (rows <= 32) c[n++] = LaneCand{lg, std::max(4, fit(rows, passes > 1 ? 4 : 2)), passes, 32, 0, 0};
  }
  if (m <= 24 * 32) c[n++] = LaneCand{32, fit((m + 31) / 32, 8), 1, 32, 0, 1};
  for (int full : {4, 8, 16}) {
    if (m <= 32 * full || (full > 8 && !wide)) continue;  // one pass; no room for the profiles
    const int passes = (m + 32 * full - 1) / (32 * full);
    if (passes > LANE_WARPS && (full < 8 || (wide && full < 16))) continue;  // a larger one has fewer
    int pr = fit((m - (passes - 1) * 32 * full + 31) / 32, 4);
    while (pr & (pr - 1)) pr += 4;  // chains come in 4, 8 and 16 rows
    c[n++] = LaneCand{32, pr, passes, full, 1, full > 4};
    // The passes after the last whole round of the block's warps leave some of
    // them idle: the same rows as up to a round of passes of fewer rows each.
    const int heads = m / (32 * full * LANE_WARPS) * LANE_WARPS, rest = m - heads * 32 * full;
    if (heads == 0 || rest == 0) continue;
    pr = 4;
    while (32 * pr * LANE_WARPS < rest) pr *= 2;
    const int tail = (rest + 32 * pr - 1) / (32 * pr);
    if (pr < full && tail > 1) c[n++] = LaneCand{32, pr, heads + tail, full, 1, 1, tail};
  }
  return n;
}

// What the lane groups take for these subject pairs at the least: the cheapest
// shapes, with every scheduler busy to the end.
static double lanes_floor(const sw_plan* p, const HostBatch& hb, int32_t nq, int64_t pair0,
                          int64_t pair1) {
  const sw_db* db = p->db;
  const double cols =
      0.5 * (double)(db->cres_h[std::min(db->view.n, 2 * pair1)] - db->cres_h[2 * pair0]);
  double cycles = 0;
  for (int32_t i = 0; i < nq; i++) {
    const int32_t m = hb.len[i], lg = m <= 256 ? 8 : m <= 512 ? 16 : 32;
    cycles += 11.1 / 32 * m * (cols + (double)(pair1 - pair0) * lg) +
              (double)(pair1 - pair0) * lg / 32 * kLaneItemCycles;
  }
  return cycles / (4.0 * p->sms);
}

// The segments for the subject pairs [pair0, pair1), without and with wide
// chains: the ones expected to end the search soonest.  *cycles is that time,
// *wide tells whether they need the wide launch.  The length order is cut at
// pair0 + 0, 1, 2, 4, 8, ...; a piece takes the cheapest shape whose item is at
// most `tail` of the search for its longest pair, or the shape with the
// shortest item, and a few values of `tail` are tried (one for a large batch,
// whose items are short beside the search).  Items start in the order of their
// expected time.  Two rules measured: the times judged beside a full chip as
// well (4 queries of 10,000-37,000 residues x 500 subjects of up to 35,000,
// where passes one after the other looked short beside the few warps that they
// are: 201 -> 140 ms), and the pieces of a few queries as segments of their own
// (7 queries of 140-600 x 40,000, whose shorter subjects no longer start before
// another query's long ones: 7.2 -> 6.75 ms).
static int64_t plan_lanes(sw_plan* p, const HostBatch& hb, int32_t nq, int64_t pair0, int64_t pair1,
                          int32_t* n_segs, double* cycles, bool* wide) {
  *n_segs = 0;
  *cycles = 0;
  *wide = false;
  if (nq <= 0 || pair0 >= pair1) return 0;
  const sw_db* db = p->db;
  const int64_t N = db->view.n;
  int64_t cut[66];
  int cuts = 0;
  for (int64_t at = 0; at < pair1 - pair0; at = at ? 2 * at : 1) cut[cuts++] = pair0 + at;
  cut[cuts] = pair1;
  double cols[65], len[65], all_cols = 0;  // columns of each piece, its longest subject
  for (int i = 0; i < cuts; i++) {
    cols[i] = 0.5 * (double)(db->cres_h[std::min(N, 2 * cut[i + 1])] - db->cres_h[2 * cut[i]]);
    len[i] = (double)db->clen_h[(size_t)(2 * cut[i])];
    all_cols += cols[i];
  }
  const double npairs = (double)(pair1 - pair0), sched = 4.0 * p->sms;
  // scheduler cycles, and warps, of a shape on `n` pairs of `c` columns
  auto cost = [](const LaneCand& x, double c, double n) {
    return x.thr() * x.lg / 32 * (c + n * x.ramp());
  };
  auto warps_of = [](const LaneCand& x, double n) {
    return n * (x.chain ? std::min(x.passes, LANE_WARPS) : x.lg / 32.0);
  };
  struct Query {
    int32_t m, n;  // its length, how many there are
    LaneCand c[MAX_SHAPES];
    int nc;
  };
  struct Piece {
    LaneCand c;
    LaneSeg s;
    double t;
  };
  // queries of one length, neighbours in the order, are planned once
  std::vector<Query> qs;
  std::vector<int32_t> kind((size_t)nq);
  for (int32_t i = 0; i < nq; i++) {
    const int32_t m = hb.len[hb.order[i]];
    if (i == 0 || m != qs.back().m) qs.push_back(Query{m, 0});
    qs.back().n++;
    kind[(size_t)i] = (int32_t)qs.size() - 1;
  }
  std::vector<double> times;
  std::vector<Piece> pieces, best_pieces;
  double best = 1e300, best_total = 0;
  const bool large = nq > FEW_QUERIES;
  for (int w = 0; w < (!large && hb.len[hb.order[0]] > 512 ? 2 : 1); w++) {
    const double resident = (double)p->lane_blocks[w] * LANE_WARPS / sched;
    auto share_of = [&](double warps) { return std::min(resident, std::max(1.0, warps / sched)); };
    double total = 0, warps = 0;
    for (Query& q : qs) {
      q.nc = lane_candidates(q.m, w != 0, q.c);
      std::sort(q.c, q.c + q.nc, [&](const LaneCand& a, const LaneCand& b) {
        return cost(a, all_cols, npairs) < cost(b, all_cols, npairs);
      });
      total += q.n * cost(q.c[0], all_cols, npairs);
      warps += q.n * warps_of(q.c[0], npairs);
    }
    const double t_all = total / sched;
    // an item's time is judged beside as many warps as the cheapest shapes
    // have, and beside as many as there is room for: shorter items are more
    const double shares[2] = {share_of(warps), resident};
    for (int f = 0; f < (!large && shares[0] < 0.9 * resident ? 2 : 1); f++) {
      const double share = shares[f];
      // the time of an item of each shape on each piece
      times.resize(qs.size() * cuts * MAX_SHAPES);
      for (size_t i = 0; i < qs.size(); i++)
        for (int k = 0; k < cuts; k++)
          for (int c = 0; c < qs[i].nc; c++)
            times[(i * cuts + k) * MAX_SHAPES + c] = qs[i].c[c].item(len[k], share);
      for (double tail : {1e9, 1.2, 0.8, 0.5, 0.35}) {
        if (large && tail != 0.5) continue;
        pieces.clear();
        total = warps = 0;
        for (int32_t i = 0; i < nq; i++) {
          const size_t qk = (size_t)kind[(size_t)i];
          const Query& q = qs[qk];
          int last = -1;
          size_t first = pieces.size();
          for (int k = 0; k < cuts; k++) {
            const double* t = &times[(qk * cuts + k) * MAX_SHAPES];
            int c = 0;
            while (c < q.nc && t[c] > tail * t_all) c++;
            if (c == q.nc) c = (int)(std::min_element(t, t + q.nc) - t);
            const bool room = pieces.size() - first < (size_t)max_segs(nq);
            if (c != last && last >= 0 && !room) c = last;
            const LaneCand& x = q.c[c];
            // of a few queries, much shorter subjects are a segment of their own,
            // which may come after the longer items of other queries
            if (c == last && (large || !room || len[k] > 0.6 * pieces.back().t)) {
              pieces.back().s.pair1 = (int32_t)cut[k + 1];
            } else {
              const LaneSeg sg{0, hb.order[i], x.lg, x.pr, x.passes, x.tail, x.full, x.chain, x.halves,
                               (int32_t)cut[k], (int32_t)cut[k + 1]};
              pieces.push_back({x, sg, len[k]});
            }
            last = c;
            total += cost(x, cols[k], (double)(cut[k + 1] - cut[k]));
            warps += warps_of(x, (double)(cut[k + 1] - cut[k]));
          }
        }
        double longest = 0;
        for (size_t i = pieces.size(); i-- > 0;) {
          Piece& x = pieces[i];
          x.t = x.c.item(x.t, share_of(warps));
          longest = std::max(longest, x.t);
          // a query's longest subjects go first, however short their shape's items
          if (i + 1 < pieces.size() && pieces[i + 1].s.q == x.s.q) x.t = std::max(x.t, pieces[i + 1].t);
        }
        // the longest item starts first, beside the rest of the work; fewer
        // warps on a scheduler (wide) hide less latency
        const double t = (std::max(longest, total / sched) + 0.2 * std::min(longest, total / sched)) *
                         (w ? 1.05 : 1.0);
        // of equals the later one, whose items are shorter, for the same work
        if (t < 0.999 * best || (t < 1.004 * best && total < 1.01 * best_total)) {
          best = std::min(best, t);
          best_total = total;
          best_pieces = pieces;
          *wide = w != 0;
        }
        if (longest < 0.3 * total / sched) break;  // shorter items cannot help
      }
    }
  }
  std::stable_sort(best_pieces.begin(), best_pieces.end(),
                   [](const Piece& a, const Piece& b) { return a.t > b.t; });
  int64_t items = 0, on_warps = 0;  // all, and those that are no chains
  for (size_t i = 0; i < best_pieces.size(); i++) {
    LaneSeg& sg = p->segs[i];
    sg = best_pieces[i].s;
    sg.first = items;
    const int64_t per = sg.chain ? 1 : LANE_WARPS * 32 / sg.lg;
    const int64_t n = (sg.pair1 - sg.pair0 + per - 1) / per;
    items += n;
    if (!sg.chain) on_warps += n;
  }
  *cycles = best + kLaneItemCycles * 4 * (double)on_warps / sched;
  *n_segs = (int32_t)best_pieces.size();
  return items;
}

// The stream layout alone, for a given number of stream pairs (host only).
extern "C" sw_status sw_query_streams(const int32_t* q_lengths, int32_t n_queries, int32_t rows,
                                      int32_t n_pairs, int32_t* strips, int64_t strip_capacity,
                                      int32_t* pairs, int64_t* n_strips) {
  sw_clear_error();
  if (rows != 16 && rows != 24 && rows != 32)
    return sw_set_error(SW_EINVAL, "rows must be 16, 24 or 32");
  if (n_queries < 2 || n_pairs < 1 || n_pairs > n_queries / 2)
    return sw_set_error(SW_EINVAL, "n_pairs must be 1..n_queries/2 (n_queries %d)", n_queries);
  if (!q_lengths || !strips || !pairs || !n_strips || strip_capacity < 0)
    return sw_set_error(SW_EINVAL, "sw_query_streams: NULL buffer or negative capacity");
  HostBatch hb;
  hb.len.assign(q_lengths, q_lengths + n_queries);
  for (int32_t i = 0; i < n_queries; i++)
    if (hb.len[i] < 0) return sw_set_error(SW_EINVAL, "q_lengths[%d] < 0", i);
  hb.order.resize(n_queries);
  std::iota(hb.order.begin(), hb.order.end(), 0);
  std::stable_sort(hb.order.begin(), hb.order.end(),
                   [&](int32_t a, int32_t b) { return hb.len[a] > hb.len[b]; });
  // built in aligned storage, then copied: the caller's buffers need only
  // int32 alignment
  int64_t bound = 0;  // the table is at most every query's strips long
  for (int32_t i = 0; i < n_queries; i++) bound += std::max<int64_t>(1, (hb.len[i] + rows - 1) / rows);
  std::vector<int4> tab((size_t)std::min(strip_capacity, bound));
  std::vector<int2> pr((size_t)n_pairs);
  const int32_t K = deal_streams(hb, n_queries, rows, n_pairs, 1.0, 1, 0.0, 0.0, tab.data(),
                                 pr.data(), 0, strip_capacity, n_strips);
  if (K == 0) return sw_set_error(SW_EBUSY, "the strip table exceeds %lld strips",
                                  (long long)strip_capacity);
  memcpy(strips, tab.data(), sizeof(int4) * (size_t)*n_strips);
  memcpy(pairs, pr.data(), sizeof(int2) * (size_t)K);
  return SW_OK;
}

// Stages a batch into the plan and enqueues everything up to (not including)
// the copy of the scores to a host buffer.
static sw_status plan_enqueue(sw_plan* p, const HostBatch& hb, int32_t nq, int32_t gap_open,
                              int32_t gap_extend, const int8_t* matrix, int32_t* scores_dev,
                              cudaStream_t s) {
  if (nq > p->max_queries || hb.total > p->max_residues)
    return sw_set_error(SW_EBUSY, "batch (%d queries, %lld residues) exceeds the plan (%d, %lld)",
                        nq, (long long)hb.total, p->max_queries, (long long)p->max_residues);
  SearchParams& P = *(SearchParams*)p->block_h;
  bool packed_ok = true;
  int max_sm = 0;
  sw_status st = fill_scoring(P, gap_open, gap_extend, matrix, &packed_ok, &max_sm);
  if (st != SW_OK) return st;
  const DbView& v = p->db->view;
  // packed: the 16-bit kernels score every pair; otherwise (penalties too
  // large for 16 bits, or forced) every pair goes to the int32 intra-task code
  const bool packed = packed_ok && !p->opt.force_int32;
  int32_t gf = packed ? p->g_first : v.groups;
  const double total_cells = (double)hb.total * (double)p->db->residues;
  if (packed && p->opt.auto_cutoff && total_cells >= kAutoCutoffMinCells) {
    // Load balance: a (query, group) item is 64 subjects x the group length x
    // the query length.  Groups whose largest item exceeds a quarter of one
    // warp's share of the search go to the intra-task kernel instead, where
    // each subject is its own item.  Groups are sorted longest first.  Small
    // searches (a few milliseconds) are left alone.
    const double warps = (double)p->kc2.blocks * p->kc2.warps;
    const double share = total_cells / warps;
    const int32_t mmax = hb.len[hb.order[0]];
    while (gf < v.groups && (double)GROUP * p->db->glen_h[gf] * mmax > 0.25 * share) gf++;
  }
  const int64_t n_long = std::min<int64_t>(v.n, (int64_t)gf * GROUP);
  P.scores = scores_dev;
  P.nq = nq;
  P.n_long = (int32_t)n_long;
  P.g_first = gf;
  P.n_intra_items = packed ? 0 : n_long * nq;
  P.n_spairs = P.n_spairs2 = 0;
  P.n_inter_items = P.n_inter2_items = P.n_pair2_items = P.n_lane_items = 0;
  P.n_lane_segs = 0;
  int64_t n_strips = 0, n_strips2 = 0;
  int kernels = 0;
  double long_share = 0;
  if (packed && nq > 0 && v.n > 0) {
    // Each part of the subjects -- the long ones, above the cutoff, and the
    // short ones -- goes to a two-query kernel or to the lane groups, whichever
    // is expected to finish it first (options two_query and two_query_long: 0
    // never two queries, 2 always with two or more queries).  Short subjects go
    // to the two-subject inter-task kernel where it is expected to beat both, the
    // lane groups by a tenth: theirs may be one launch for all subjects, whose
    // end is shorter than that of two.
    const int64_t npairs = (v.n + 1) / 2, long_pairs = std::min(npairs, (n_long + 1) / 2);
    const bool has_long = n_long > 0, has_short = gf < v.groups;
    double t2 = 0;
    bool two = false, two_long = false, wide = false, groups = false;
    // the lane groups' segments for a range of subject pairs, planned once while
    // the range stays the same
    int32_t n_segs = 0;
    int64_t lane_items = 0, planned0 = -1, planned1 = -1;
    double tl = 0;
    auto lanes = [&](int64_t pair0, int64_t pair1) {
      if (pair0 != planned0 || pair1 != planned1)
        lane_items = plan_lanes(p, hb, nq, pair0, pair1, &n_segs, &tl, &wide);
      planned0 = pair0;
      planned1 = pair1;
      return tl;
    };
    if (has_short) {
      const bool may = nq >= 2 && p->opt.two_query > 0;
      int32_t K = 0;
      if (may && p->opt.two_query == 2) {
        K = plan_streams(p, hb, nq, gf, 1e300, &n_strips, &t2);
        two = K > 0;
      }
      if (!two) {
        const double t1 = plan_groups(p, hb, nq, gf);
        groups = t1 < 0.95 * lanes_floor(p, hb, nq, long_pairs, npairs);
        const double t = may || groups ? lanes(long_pairs, npairs) : 0;
        if (may && p->opt.two_query == 1) K = plan_streams(p, hb, nq, gf, t, &n_strips, &t2);
        two = K > 0 && t2 < t && !(groups && t1 < t2);
        groups = groups && !two && t1 < 0.9 * t;
      }
      if (two) {
        P.n_spairs = K;
        P.n_inter2_items = (int64_t)K * 2 * (v.groups - gf);
      } else {
        n_strips = 0;
      }
    }
    if (has_long && nq >= 2 && p->opt.two_query_long > 0) {
      const double t = p->opt.two_query_long == 1 ? lanes(0, long_pairs) : 1e300;
      const int32_t K2 =
          plan_streams_long(p, hb, nq, n_long, n_strips, P.n_spairs, t, &n_strips2, &t2);
      two_long = K2 > 0 && t2 < t;
      if (two_long) {
        P.n_spairs2 = K2;
        P.n_pair2_items = (int64_t)K2 * ((n_long + PAIR2_GROUP - 1) / PAIR2_GROUP);
        kernels |= K_PAIR2;
      } else {
        n_strips2 = 0;
      }
    }
    const bool lanes_long = has_long && !two_long, lanes_short = has_short && !two && !groups;
    if (lanes_long || lanes_short) {
      lanes(lanes_long ? 0 : long_pairs, lanes_short ? npairs : long_pairs);
      P.n_lane_items = lane_items;
      P.n_lane_segs = n_segs;
      p->lane_grid = (int)std::min<int64_t>(P.n_lane_items, p->lane_blocks[wide]);
      kernels |= (lanes_short ? K_LANES : K_LANES_LONG) | (wide ? K_WIDE : 0);
      if (lanes_long && lanes_short && p->db->residues > 0)
        long_share = (double)p->db->cres_h[n_long] / (double)p->db->residues;
    }
    if (two) kernels |= K_INTER2;
    if (groups) {
      P.n_inter_items = (int64_t)(v.groups - gf) * nq;
      kernels |= K_INTER;
    }
    // no score above max_sm per aligned column: without one at the recompute
    // threshold the int32 kernel has nothing to do
    const int64_t longest = hb.len[hb.order[0]];
    if (max_sm * std::min<int64_t>(longest, v.max_len) >= P.sat_threshold) kernels |= K_INT32;
  } else if (nq > 0 && v.n > 0) {
    kernels = K_INT32;
  }
  // the upload block: parameters, zeroed state, tables
  size_t at = BLOCK_HEADER;
  auto put = [&](const void* src, size_t bytes) {
    uint8_t* dev = p->block + at;
    if (bytes) memcpy(p->block_h + at, src, bytes);
    at += block_align(bytes);
    return dev;
  };
  P.qoff = (const int64_t*)put(hb.off.data(), sizeof(int64_t) * nq);
  P.qlen = (const int32_t*)put(hb.len.data(), sizeof(int32_t) * nq);
  P.qorder = (const int32_t*)put(hb.order.data(), sizeof(int32_t) * nq);
  P.lane_segs = (const LaneSeg*)put(p->segs.data(), sizeof(LaneSeg) * P.n_lane_segs);
  P.spairs = (const int2*)put(p->spairs.data(), sizeof(int2) * (P.n_spairs + P.n_spairs2));
  P.spairs2 = P.spairs + P.n_spairs;
  P.strips = P.strips2 = (const int4*)put(p->strips.data(), sizeof(int4) * (n_strips + n_strips2));
  P.qres = put(hb.res, (size_t)hb.total);
  if (injected_fault("copy"))
    return sw_set_cuda_error(cudaErrorInvalidValue, "query upload (injected fault)");
  CUDA_TRY(cudaMemcpyAsync(p->block, p->block_h, at, cudaMemcpyHostToDevice, s));
  p->stream = s;
  p->gclass = gap_class(P.go, P.ge);
  p->kernels = kernels;
  p->long_share = long_share;
  if (kernels) CUDA_TRY(run_kernels(p, s));
  memset(p->state_h, 0, sizeof(SearchState));
  if (kernels & K_INT32)
    CUDA_TRY(cudaMemcpyAsync(p->state_h, p->state, sizeof(SearchState), cudaMemcpyDeviceToHost, s));
  p->pending = sw_stats{};
  int64_t qsum = hb.total;
  p->pending.cells = qsum * p->db->residues;
  p->pending.inter_items = packed && P.n_spairs == 0 ? (int64_t)(v.groups - gf) * nq : 0;
  p->pending.inter2_items = P.n_inter2_items;
  p->pending.pair2_items = P.n_pair2_items;
  p->pending.intra_items = n_long * nq;  // (query, long subject) pairs, packed or int32
  p->pending.inter_cells = qsum * (p->db->residues - p->db->cres_h[n_long]);
  for (int k = kernels & ~K_WIDE; k; k &= k - 1) p->pending.kernels_launched++;
  if ((kernels & K_INT32) && kernels != K_INT32 && p->clusters > 0)
    p->pending.kernels_launched++;  // both recomputes
  return SW_OK;
}

static void finish_stats(sw_plan* p) {
  p->stats = p->pending;
  const int set = p->kernels;
  const bool is_long = set & (K_PAIR2 | K_LANES_LONG), is_short = set & (K_LANES | K_INTER2 | K_INTER);
  const bool both = is_long && is_short;
  // with overlap_kernels the kernels of both parts start at ev[0]
  const bool ov = p->opt.overlap_kernels != 0 && both;
  auto between = [&](cudaEvent_t a, cudaEvent_t b) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, a, b) != cudaSuccess) {
      cudaGetLastError();
      ms = -1.f;
    }
    return ms;
  };
  if (both) {
    p->stats.pair_ms = between(p->ev[0], p->ev[1]);
    p->stats.search_ms = between(ov ? p->ev[0] : p->ev[1], p->ev[2]);
  } else if (is_long) {
    p->stats.pair_ms = between(p->ev[0], p->ev[2]);
  } else if (is_short) {
    // one launch for all subjects: its time split by their cells
    const float ms = between(p->ev[0], p->ev[2]);
    p->stats.pair_ms = (float)p->long_share * ms;
    p->stats.search_ms = ms - p->stats.pair_ms;
  }
  if (set & K_INT32) p->stats.recompute_ms = between(ov ? p->ev_join : p->ev[2], p->ev[3]);
  p->stats.recomputed_pairs = (int64_t)p->state_h->n_flags;
  p->in_flight = false;
}

// More saturated pairs than the flag list holds: the packed kernels wrote
// FLAG_SENTINEL for those that found it full.  Each round collects the
// marked pairs into the list (counting all of them) and recomputes the
// listed ones in int32, whose exact scores replace the marks; the round in
// which every marked pair fits the list is the last.  Runs after the search
// has completed, synchronously on its stream.
static cudaError_t overflow_rounds(sw_plan* p, int32_t* rounds) {
  *rounds = 0;
  cudaStream_t s = p->stream;
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->db->device);
  unsigned long long nf = p->state_h->n_flags;
  while (nf > (unsigned long long)p->scr.flag_capacity) {
    cudaError_t e = cudaMemsetAsync(p->state, 0, sizeof(SearchState), s);
    if (e == cudaSuccess) e = launch_collect(4 * std::max(sms, 1), p->db->view, p->params, p->state, p->scr, s);
    if (e == cudaSuccess) e = launch_intra(p->ikc, p->clusters, false, p->db->view, p->params, p->state, p->scr, s);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(p->state_h, p->state, sizeof(SearchState), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    nf = p->state_h->n_flags;
    ++*rounds;
  }
  return cudaSuccess;
}

// Statistics, then any overflow rounds, of a search that has completed.
static sw_status complete_search(sw_plan* p) {
  finish_stats(p);
  cudaError_t e = overflow_rounds(p, &p->stats.overflow_rounds);
  if (e != cudaSuccess) return sw_set_cuda_error(e, "recompute of the flag-list overflow");
  return SW_OK;
}

extern "C" sw_status sw_plan_search(sw_plan* plan, const uint8_t* queries, const int32_t* q_lengths,
                                    int32_t n_queries, int32_t gap_open, int32_t gap_extend,
                                    const int8_t* matrix, int32_t* scores, void* stream) {
  sw_clear_error();
  if (!plan) return sw_set_error(SW_EINVAL, "plan is NULL");
  if (plan->in_flight) return sw_set_error(SW_EBUSY, "plan has a search in flight");
  CUDA_TRY(cudaSetDevice(plan->db->device));
  HostBatch hb;
  sw_status st = read_batch(queries, q_lengths, n_queries, hb);
  if (st != SW_OK) return st;
  const int64_t N = plan->db->view.n;
  if (n_queries > 0 && N > 0 && !scores) return sw_set_error(SW_EINVAL, "scores is NULL");
  cudaStream_t s = (cudaStream_t)stream;
  const bool dev_out = is_device_ptr(scores);
  if (!dev_out && !plan->scores_dev) {
    // scores for a host buffer are staged on the device: the first such
    // search allocates the plan's staging buffer
    cudaError_t ea = injected_fault("alloc") ? cudaErrorMemoryAllocation
                                             : db_alloc(plan->db, &plan->scores_dev,
                                                        (size_t)plan->max_queries * std::max<int64_t>(N, 1));
    if (ea != cudaSuccess) {
      plan->scores_dev = nullptr;
      return sw_set_cuda_error(ea, "sw_plan_search: host-order scores buffer");
    }
  }
  int32_t* target = dev_out ? scores : plan->scores_dev;
  st = plan_enqueue(plan, hb, n_queries, gap_open, gap_extend, matrix, target, s);
  if (st != SW_OK) return st;
  plan->in_flight = true;
  const size_t out_bytes = sizeof(int32_t) * (size_t)n_queries * (size_t)N;
  if (!dev_out && out_bytes > 0)
    CUDA_TRY(cudaMemcpyAsync(scores, plan->scores_dev, out_bytes, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaEventRecord(plan->done, s));
  cudaError_t e = cudaEventSynchronize(plan->done);
  if (e != cudaSuccess) {
    finish_stats(plan);
    return sw_set_cuda_error(e, "sw_plan_search");
  }
  st = complete_search(plan);
  if (st != SW_OK) return st;
  if (plan->stats.overflow_rounds > 0 && !dev_out && out_bytes > 0) {
    // the copy above predates the overflow rounds' scores
    CUDA_TRY(cudaMemcpyAsync(scores, plan->scores_dev, out_bytes, cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
  }
  CUDA_TRY(cudaGetLastError());
  return SW_OK;
}

extern "C" sw_status sw_plan_search_async(sw_plan* plan, const uint8_t* queries,
                                          const int32_t* q_lengths, int32_t n_queries,
                                          int32_t gap_open, int32_t gap_extend,
                                          const int8_t* matrix, int32_t* scores, void* stream) {
  sw_clear_error();
  if (!plan) return sw_set_error(SW_EINVAL, "plan is NULL");
  if (plan->in_flight) return sw_set_error(SW_EBUSY, "plan has a search in flight");
  CUDA_TRY(cudaSetDevice(plan->db->device));
  HostBatch hb;
  sw_status st = read_batch(queries, q_lengths, n_queries, hb);
  if (st != SW_OK) return st;
  if (n_queries > 0 && plan->db->view.n > 0 && !is_device_ptr(scores))
    return sw_set_error(SW_EINVAL, "sw_plan_search_async needs device scores");
  cudaStream_t s = (cudaStream_t)stream;
  st = plan_enqueue(plan, hb, n_queries, gap_open, gap_extend, matrix, scores, s);
  if (st != SW_OK) return st;
  CUDA_TRY(cudaEventRecord(plan->done, s));
  plan->in_flight = true;
  return SW_OK;
}

extern "C" sw_status sw_plan_wait(sw_plan* plan, int32_t timeout_ms) {
  if (!plan) return sw_set_error(SW_EINVAL, "plan is NULL");
  if (!plan->in_flight) return SW_OK;
  const auto t0 = std::chrono::steady_clock::now();
  for (;;) {
    cudaError_t e = cudaEventQuery(plan->done);
    if (e == cudaSuccess) return complete_search(plan);
    if (e != cudaErrorNotReady) {
      plan->in_flight = false;
      return sw_set_cuda_error(e, "sw_plan_wait");
    }
    if (timeout_ms >= 0) {
      const double ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
      if (ms >= timeout_ms) return sw_set_error(SW_ETIMEDOUT, "search still running after %d ms", timeout_ms);
    }
    std::this_thread::sleep_for(std::chrono::microseconds(50));
  }
}

extern "C" sw_status sw_plan_stats(const sw_plan* plan, sw_stats* out) {
  if (!plan || !out) return sw_set_error(SW_EINVAL, "NULL argument");
  *out = plan->stats;
  return SW_OK;
}

extern "C" sw_status sw_search(sw_db* db, const uint8_t* queries, const int32_t* q_lengths,
                               int32_t n_queries, int32_t gap_open, int32_t gap_extend,
                               const int8_t* matrix, int32_t* scores, void* stream) {
  sw_clear_error();
  if (!db) return sw_set_error(SW_EINVAL, "db is NULL");
  CUDA_TRY(cudaSetDevice(db->device));
  HostBatch hb;
  sw_status st = read_batch(queries, q_lengths, n_queries, hb);
  if (st != SW_OK) return st;
  std::lock_guard<std::mutex> guard(db->oneshot_mu);
  sw_plan*& plan = db->oneshot;
  int32_t want_q = std::max(n_queries, 1);
  int64_t want_res = hb.total;
  if (plan && (plan->max_queries < want_q || plan->max_residues < want_res)) {
    want_q = std::max(want_q, plan->max_queries);
    want_res = std::max(want_res, plan->max_residues);
    plan_free(plan);
    plan = nullptr;
  }
  if (!plan) {
    sw_options o;
    sw_options_default(&o);
    st = sw_plan_create(db, want_q, want_res, &o, &plan);
    if (st != SW_OK) {
      plan = nullptr;
      return st;
    }
  }
  return sw_plan_search(plan, queries, q_lengths, n_queries, gap_open, gap_extend, matrix, scores,
                        stream);
}

// ---- plain baseline ----------------------------------------------------------------------
extern "C" sw_status sw_search_plain(sw_db* db, const uint8_t* queries, const int32_t* q_lengths,
                                     int32_t n_queries, int32_t gap_open, int32_t gap_extend,
                                     const int8_t* matrix, int32_t* scores, void* stream) {
  sw_clear_error();
  if (!db) return sw_set_error(SW_EINVAL, "db is NULL");
  CUDA_TRY(cudaSetDevice(db->device));
  HostBatch hb;
  sw_status st = read_batch(queries, q_lengths, n_queries, hb);
  if (st != SW_OK) return st;
  const DbView& v = db->view;
  const int64_t N = v.n;
  if (n_queries > 0 && N > 0 && !scores) return sw_set_error(SW_EINVAL, "scores is NULL");
  SearchParams P;
  memset(&P, 0, sizeof P);
  bool packed_ok;
  st = fill_scoring(P, gap_open, gap_extend, matrix, &packed_ok);
  if (st != SW_OK) return st;
  if (n_queries == 0 || N == 0) return SW_OK;
  cudaStream_t s = (cudaStream_t)stream;
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, db->device);
  const int bps = std::max(1, std::min(plain_blocks_per_sm(), 8));
  const int grid = (int)std::min<int64_t>((int64_t)sms * bps, v.groups);
  std::vector<int64_t> boff(grid);
  int64_t btotal = 0;
  for (int b = 0; b < grid; b++) {
    boff[b] = btotal;
    btotal += (int64_t)db->glen_h[b] * GROUP;  // a block's first group is its longest
  }
  const bool dev_out = is_device_ptr(scores);
  uint8_t* qres = nullptr;
  int64_t *qoff = nullptr, *boff_d = nullptr;
  int32_t *qlen = nullptr, *sc = nullptr;
  int2* border = nullptr;
  SearchParams* Pd = nullptr;
  cudaError_t e = db_alloc(db, &qres, hb.total);
  if (e == cudaSuccess) e = db_alloc(db, &qoff, n_queries);
  if (e == cudaSuccess) e = db_alloc(db, &qlen, n_queries);
  if (e == cudaSuccess) e = db_alloc(db, &boff_d, grid);
  if (e == cudaSuccess) e = db_alloc(db, &border, btotal);
  if (e == cudaSuccess) e = db_alloc(db, &Pd, 1);
  if (e == cudaSuccess && !dev_out) e = db_alloc(db, &sc, (size_t)n_queries * N);
  if (e == cudaSuccess && hb.total > 0)
    e = cudaMemcpyAsync(qres, hb.res, hb.total, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(qoff, hb.off.data(), sizeof(int64_t) * n_queries, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(qlen, hb.len.data(), sizeof(int32_t) * n_queries, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(boff_d, boff.data(), sizeof(int64_t) * grid, cudaMemcpyHostToDevice, s);
  P.qres = qres;
  P.qoff = qoff;
  P.qlen = qlen;
  P.scores = dev_out ? scores : sc;
  P.nq = n_queries;
  if (e == cudaSuccess) e = cudaMemcpyAsync(Pd, &P, sizeof P, cudaMemcpyHostToDevice, s);
  for (int32_t q = 0; q < n_queries && e == cudaSuccess; q++)
    e = launch_plain(grid, v, Pd, q, border, boff_d, s);
  if (e == cudaSuccess && !dev_out)
    e = cudaMemcpyAsync(scores, sc, sizeof(int32_t) * (size_t)n_queries * N, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(qres);
  cudaFree(qoff);
  cudaFree(qlen);
  cudaFree(boff_d);
  cudaFree(border);
  cudaFree(Pd);
  cudaFree(sc);
  if (e != cudaSuccess) return sw_set_cuda_error(e, "sw_search_plain");
  return SW_OK;
}

// ---- optimal alignments with traceback ------------------------------------------------------
// Largest buffer of cells of one chunk of pairs (bytes).
static constexpr int64_t kAlignChunkBytes = 8ll << 30;
// A call's cells with H kept, at most (bytes, two to a cell): larger calls are
// bound by the chip's rate, where four bits cost no more (20 pairs of 5,000 x
// 5,000, just below: 5.0 ms with bits, 4.1 with H).
static constexpr int64_t kAlignKeepH = 1ll << 30;
static constexpr int32_t kAlignKeepHColumns = 65000;  // a cell's step in 16 bits
// What a database keeps of a call's buffers, at most.
static constexpr size_t kAlignKeepDevice = 512u << 20, kAlignKeepPinned = 16u << 20;

extern "C" sw_status sw_align(sw_db* db, const uint8_t* queries, const int32_t* q_lengths,
                              int32_t n_queries, const int32_t* pair_query,
                              const int64_t* pair_subject, int32_t n_pairs, int32_t gap_open,
                              int32_t gap_extend, const int8_t* matrix, sw_alignment* out,
                              uint8_t* ops, int64_t ops_capacity, void* stream) {
  sw_clear_error();
  if (!db) return sw_set_error(SW_EINVAL, "db is NULL");
  if (n_pairs < 0) return sw_set_error(SW_EINVAL, "n_pairs < 0");
  if (n_pairs > 0 && (!pair_query || !pair_subject || !out))
    return sw_set_error(SW_EINVAL, "pair_query, pair_subject or out is NULL");
  CUDA_TRY(cudaSetDevice(db->device));
  HostBatch hb;
  sw_status st = read_batch(queries, q_lengths, n_queries, hb);
  if (st != SW_OK) return st;
  SearchParams P;
  memset(&P, 0, sizeof P);
  bool packed_ok;
  int max_sm = 0;
  st = fill_scoring(P, gap_open, gap_extend, matrix, &packed_ok, &max_sm);
  if (st != SW_OK) return st;
  const int64_t N = db->view.n;
  // per pair: sorted subject, sizes, and its transcript slot
  std::vector<AlignItem> items((size_t)n_pairs);
  std::vector<int64_t> slot((size_t)n_pairs + 1, 0);
  for (int32_t k = 0; k < n_pairs; k++) {
    const int32_t q = pair_query[k];
    const int64_t sub = pair_subject[k];
    if (q < 0 || q >= n_queries)
      return sw_set_error(SW_EINVAL, "pair_query[%d] = %d is not a query index", k, q);
    if (sub < 0 || sub >= N)
      return sw_set_error(SW_EINVAL, "pair_subject[%d] = %lld is not a subject index", k,
                          (long long)sub);
    const int32_t s = db->sorted_of_h[(size_t)sub];
    items[k].q = q;
    items[k].s = s;
    slot[k + 1] = slot[k] + hb.len[q] + db->clen_h[s];
  }
  if (n_pairs > 0 && slot[n_pairs] > 0 && (!ops || ops_capacity < slot[n_pairs]))
    return sw_set_error(SW_EINVAL, "ops needs %lld bytes, has %lld", (long long)slot[n_pairs],
                        (long long)ops_capacity);
  if (n_pairs == 0) return SW_OK;
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, db->device);
  const int team = align_team(n_pairs, sms);  // warps to a pair
  // H of every cell is kept where 16 bits hold it and the cells are few, else
  // four direction bits
  bool keep_h = P.go <= INT16_MAX;
  int64_t cell_bytes = 0;
  for (int32_t k = 0; k < n_pairs && keep_h; k++) {
    const int32_t m = hb.len[items[k].q], n = db->clen_h[items[k].s];
    cell_bytes += align_bits_bytes(team, true, m, n);
    keep_h = cell_bytes <= kAlignKeepH && (int64_t)max_sm * std::min(m, n) <= INT16_MAX &&
             n <= kAlignKeepHColumns;
  }
  // chunks of pairs whose cells fit kAlignChunkBytes (one pair may exceed it alone)
  std::vector<int32_t> chunk_begin;
  int64_t max_words = 0, max_border = 0;
  auto chunk = [&]() {
    chunk_begin.assign(1, 0);
    max_words = max_border = 0;
    int64_t words = 0, border = 0;
    for (int32_t k = 0; k < n_pairs; k++) {
      const int64_t w = align_bits_bytes(team, keep_h, hb.len[items[k].q], db->clen_h[items[k].s]);
      if (k > chunk_begin.back() && words + w > kAlignChunkBytes) {
        chunk_begin.push_back(k);
        words = border = 0;
      }
      items[k].bits_off = words;
      items[k].border_off = border;
      items[k].ops_end = slot[k + 1];
      words += w;
      border += align_border_ints(team, db->clen_h[items[k].s]);
      max_words = std::max(max_words, words);
      max_border = std::max(max_border, border);
    }
    chunk_begin.push_back(n_pairs);
  };
  chunk();
  cudaStream_t cs = (cudaStream_t)stream;
  // One device buffer: what goes up (parameters, items, the query arrays) in
  // one copy, what comes back (records, transcripts) in one copy, the border
  // rows and the cells.
  const size_t up_items = block_align(sizeof(SearchParams));
  const size_t up_qoff = up_items + block_align(sizeof(AlignItem) * (size_t)n_pairs);
  const size_t up_qlen = up_qoff + block_align(sizeof(int64_t) * (size_t)n_queries);
  const size_t up_qres = up_qlen + block_align(sizeof(int32_t) * (size_t)n_queries);
  const size_t up_bytes = up_qres + block_align((size_t)hb.total);
  const size_t ops_at = block_align(sizeof(AlignOut) * (size_t)n_pairs);
  const size_t back_bytes = ops_at + block_align((size_t)slot[n_pairs]);
  const size_t at_out = up_bytes, at_border = at_out + back_bytes;
  size_t at_bits = 0;
  auto dev_bytes = [&]() {
    at_bits = at_border + block_align(sizeof(int2) * (size_t)max_border);
    return at_bits + (size_t)std::max<int64_t>(max_words, 1);
  };
  std::unique_lock<std::mutex> kept(db->align_mu, std::try_to_lock);
  AlignBuffers own;
  AlignBuffers& buf = kept.owns_lock() ? db->align : own;
  // Each way through pinned memory while the database keeps that much of it; a
  // larger call uploads from where its arrays lie and reads back into pageable
  // memory (5 pairs of 50,000 queries, 20 MB of residues: 9.0 ms through memory
  // pinned for the call, 7.1 so).
  const bool pin_up = up_bytes <= kAlignKeepPinned, pin_back = back_bytes <= kAlignKeepPinned;
  std::unique_ptr<uint8_t[]> pageable;
  if (!pin_back) {
    pageable.reset(new (std::nothrow) uint8_t[back_bytes]);
    if (!pageable) return sw_set_error(SW_ENOMEM, "sw_align: out of host memory");
  }
  const size_t pin_bytes = std::max(pin_up ? up_bytes : 0, pin_back ? back_bytes : 0);
  cudaError_t e = buf.reserve(dev_bytes(), pin_bytes);
  if (e == cudaErrorMemoryAllocation && keep_h) {
    cudaGetLastError();  // no room for H of every cell: a quarter of that for bits
    keep_h = false;
    chunk();
    e = buf.reserve(dev_bytes(), pin_bytes);
  }
  uint8_t* host = pin_back ? buf.pinned : pageable.get();
  if (e == cudaSuccess) {
    P.qoff = (const int64_t*)(buf.dev + up_qoff);
    P.qlen = (const int32_t*)(buf.dev + up_qlen);
    P.qres = buf.dev + up_qres;
    P.nq = n_queries;
    auto put = [&](size_t at, const void* src, size_t bytes) {
      if (bytes == 0 || e != cudaSuccess) return;
      if (pin_up)
        memcpy(buf.pinned + at, src, bytes);
      else
        e = cudaMemcpyAsync(buf.dev + at, src, bytes, cudaMemcpyHostToDevice, cs);
    };
    put(0, &P, sizeof P);
    put(up_items, items.data(), sizeof(AlignItem) * (size_t)n_pairs);
    put(up_qoff, hb.off.data(), sizeof(int64_t) * (size_t)n_queries);
    put(up_qlen, hb.len.data(), sizeof(int32_t) * (size_t)n_queries);
    put(up_qres, hb.res, (size_t)hb.total);
    if (pin_up) e = cudaMemcpyAsync(buf.dev, buf.pinned, up_bytes, cudaMemcpyHostToDevice, cs);
  }
  const AlignItem* items_d = (const AlignItem*)(buf.dev + up_items);
  AlignOut* out_d = (AlignOut*)(buf.dev + at_out);
  for (size_t c = 0; c + 1 < chunk_begin.size() && e == cudaSuccess; c++) {
    const int32_t k0 = chunk_begin[c], nk = chunk_begin[c + 1] - k0;
    e = launch_align(team, keep_h, sms, db->view, (const SearchParams*)buf.dev, items_d + k0, nk,
                     buf.dev + at_bits, (int2*)(buf.dev + at_border), out_d + k0,
                     buf.dev + at_out + ops_at, cs);
    // the next chunk reuses the cells: its kernel runs after this one's on the stream
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(host, buf.dev + at_out, back_bytes, cudaMemcpyDeviceToHost, cs);
  if (e == cudaSuccess)
    e = cudaStreamSynchronize(cs);
  else
    cudaStreamSynchronize(cs);  // nothing queued may outlive the buffers
  if (e == cudaSuccess) {
    const AlignOut* res = (const AlignOut*)host;
    for (int32_t k = 0; k < n_pairs; k++) {
      const AlignOut& r = res[k];
      out[k].score = r.score;
      out[k].q_begin = r.q_begin;
      out[k].q_end = r.score > 0 ? r.i_end : 0;
      out[k].s_begin = r.s_begin;
      out[k].s_end = r.score > 0 ? r.j_end : 0;
      out[k].n_ops = r.n_ops;
      out[k].ops_offset = r.ops_offset;
      if (r.n_ops > 0) memcpy(ops + r.ops_offset, host + ops_at + r.ops_offset, (size_t)r.n_ops);
    }
  }
  buf.trim(kept.owns_lock() ? kAlignKeepDevice : 0, kept.owns_lock() ? kAlignKeepPinned : 0);
  if (e != cudaSuccess) return sw_set_cuda_error(e, "sw_align");
  return SW_OK;
}

// ---- microbenchmark ----------------------------------------------------------------------
extern "C" sw_status sw_intpeak(int32_t op, int32_t blocks_per_sm, int32_t threads, int32_t iters,
                                double* out) {
  sw_clear_error();
  if (!out) return sw_set_error(SW_EINVAL, "out is NULL");
  int rc = intpeak_run(op, blocks_per_sm, threads, iters, &out[0], &out[1], &out[2]);
  if (rc == SW_EINVAL) return sw_set_error(SW_EINVAL, "sw_intpeak: bad arguments");
  return (sw_status)rc;
}
