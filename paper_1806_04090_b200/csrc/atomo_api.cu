// C ABI of the library (see include/atomo.h): argument checks, payload layout, workspace
// carving and kernel sequencing.  No arithmetic of the method lives here.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "atomo_kernels.cuh"

using namespace atomo;

// Descriptor tables of a call (layer descriptors, tile lists, tensor maps, header templates) live in a device buffer
// of their own and are uploaded only when they differ from what that buffer already holds: a training loop calls
// with the same pointers and shapes every step, so in steady state a call issues no host-to-device copy at all (a
// copy of a few KB would otherwise queue behind whatever the application has on the copy engine, e.g. the next
// step's inputs).
struct TableCache {
  uint8_t* d = nullptr; size_t cap = 0;        // device buffer
  uint8_t* h = nullptr; size_t hcap = 0;       // pinned staging buffer of the last upload
  std::vector<uint8_t> last;                   // what the device buffer holds
  cudaEvent_t ev = nullptr; bool ev_pending = false;
  cudaStream_t last_stream = nullptr;
};

// A few caches side by side, found by a key over the caller's pointers and shapes: an application that alternates
// between a few sets of buffers (double-buffered gradients, several payloads in flight) still uploads nothing in
// steady state.  The key only picks the way; whether an upload is needed is decided on the table bytes themselves.
struct TableWays {
  static constexpr int kWays = 8;
  TableCache way[kWays];
  uint64_t key[kWays] = {};
  uint64_t used[kWays] = {};                   // 0 = never used, else the tick of the last use
  uint64_t tick = 0;
};

struct atomo_ctx {
  int device = 0;
  TableWays tab_sp, tab_avg;
  int64_t table_uploads = 0, table_reuses = 0;
  uint8_t* ws = nullptr;
  size_t ws_bytes = 0;
  int64_t ws_limit = -1;             // most that the workspace may grow to (-1: no limit)
  uint32_t* h_flag = nullptr;        // pinned: convergence flag / state mirror
  EwLqPart* h_lq = nullptr;          // pinned: results of the l_q sums, written by the GPU
  uint32_t* ew_words = nullptr;      // device: barrier counters of the entry-wise encode (zero between launches), the ticket of the l_q sums
  // stage timers: one set of events per API call, a ring of kEvRing sets (a set is read out -- its call is long
  // finished by then -- before it is used again), sums since profiling was switched on
  static constexpr int kEvRing = 32;
  cudaEvent_t ev[kEvRing][ATOMO_N_STAGES][2] = {};
  bool ev_used[kEvRing][ATOMO_N_STAGES] = {};
  int ev_cur = 0;
  int64_t launches[ATOMO_N_STAGES] = {};
  double acc_ms[ATOMO_N_STAGES] = {};
  int64_t acc_launches[ATOMO_N_STAGES] = {};
  int64_t acc_calls = 0;
  bool profiling = false;
  bool configured = false;
  int max_sweeps = 40;
  float tol = 3e-7f;
  int eig_mode = 1;                  // 1: Cholesky factor + Jacobi on its rows; 0: Jacobi on [A | I]
  int refine_min_short = 2048;       // layers with at least this short side get the sigma refinement pass
  bool tc_gram = true;               // Gram matrix on tcgen05 where the layer's layout allows it
  bool tc_ok = false;                // tensor-map entry point found
  // work beside the call's stream, which forks it and joins it again inside the call: a stream per priority that calls came with, since a
  // caller's work must not wait for less urgent work of others on its side stream
  std::vector<std::pair<int, cudaStream_t>> sides;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  int eig_scheme = 3;                // eigen-solve: 0 = Jacobi, one launch per step, 1 = persistent (cooperative), 2 = clusters first, 3 = tridiagonal route first
  int tri_clusters = -1;             // co-resident clusters of the tridiagonal reduction (-1 = not asked yet, 0 = unavailable)
  int tri_big_ok = -1;               // two-stage tridiagonal reduction for short sides above 512 (-1 = not asked yet)
  int band_capacity[2][13];          // co-resident CTAs of its first stage, by instance and ceil(log2(short side)) (-1 = not asked yet)
  int chase_capacity[5] = {-1, -1, -1, -1, -1};   // clusters of its second stage side by side, by log2(CTAs)
  int band_limit = -1, chase_limit = -1;          // at most that many of either, whatever the queries say (-1: no limit)
  int tri_big_ctas = 0;              // CTAs per layer of that reduction: 0 = chosen per batch, else 1, 2, 4, 8 or 16
  int eig_scheme_used = -1;          // what the last spectral encode actually ran
  int ew_format = ATOMO_EW_EXPLICIT; // payload format of entry-wise encodes
  int ew_launch = 0;                 // 0: one cooperative kernel per vector where it fits one wave; 1: always solve + sample/pack kernels
  std::vector<EwState*> ew_last_state;   // per vector of the last entry-wise encode: its state record (device) ...
  std::vector<int> ew_last_chunks;       // ... and its chunks in the one-kernel form (0: the two-kernel form ran)
  int64_t ew_sat_cap = 0;            // compact format: capacity of the saturated list
  int cluster_capacity[16] = {-1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1};   // by log2(rp_max), -1 = not asked yet
  std::string err;
  atomo_ctx() { for (auto& f : band_capacity) for (int& c : f) c = -1; }
};

namespace {

struct Arena {
  uint8_t* base; size_t off = 0;
  explicit Arena(uint8_t* b) : base(b) {}
  template <typename T> T* take(size_t count) {
    off = (off + 255) & ~size_t(255);
    T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
    off += count * sizeof(T);
    return p;
  }
};

int fail_cuda(atomo_ctx* ctx, cudaError_t e, const char* what) {
  ctx->err = std::string(what) + ": " + cudaGetErrorString(e);
  return ATOMO_ERR_CUDA;
}
constexpr int kLqResults = 64;                                 // vectors per round of the l_q sums
constexpr int kEwBarrierWords = kEwBatch * kEwBarrierStride;
constexpr int kEwWords = kEwBarrierWords + 32;
#define CK(call)                                                            \
  do {                                                                      \
    cudaError_t e__ = (call);                                               \
    if (e__ != cudaSuccess) return fail_cuda(ctx, e__, #call);              \
  } while (0)

// FNV-1a over a block of bytes, chained through h
uint64_t table_key(uint64_t h, const void* data, size_t bytes) {
  const uint8_t* b = static_cast<const uint8_t*>(data);
  for (size_t i = 0; i < bytes; ++i) { h ^= b[i]; h *= 1099511628211ull; }
  return h;
}
constexpr uint64_t kKeySeed = 1469598103934665603ull;

// the way that served this key last, else a way never used, else the one unused for longest
TableCache& table_pick(TableWays& tw, uint64_t key) {
  int pick = -1;
  for (int i = 0; i < TableWays::kWays; ++i) if (tw.used[i] && tw.key[i] == key) { pick = i; break; }
  if (pick < 0) {
    pick = 0;
    for (int i = 1; i < TableWays::kWays; ++i) if (tw.used[i] < tw.used[pick]) pick = i;
  }
  tw.key[pick] = key; tw.used[pick] = ++tw.tick;
  return tw.way[pick];
}
void table_free(TableCache& tc);
void table_free(TableWays& tw) { for (auto& w : tw.way) table_free(w); }

// device buffer of at least `bytes` for a table cache (growing it forgets the cached contents)
int table_reserve(atomo_ctx* ctx, TableCache& tc, size_t bytes) {
  if (bytes <= tc.cap) return ATOMO_OK;
  CK(cudaDeviceSynchronize());
  if (tc.d) CK(cudaFree(tc.d));
  tc.d = nullptr; tc.cap = 0; tc.last.clear();
  const size_t want = bytes + bytes / 4 + 4096;
  CK(cudaMalloc(&tc.d, want));
  tc.cap = want;
  return ATOMO_OK;
}

// makes the device buffer hold host[0 .. bytes): nothing to do if it already does
int table_commit(atomo_ctx* ctx, TableCache& tc, const uint8_t* host, size_t bytes, cudaStream_t st) {
  if (tc.ev == nullptr) CK(cudaEventCreateWithFlags(&tc.ev, cudaEventDisableTiming));
  if (tc.last.size() == bytes && std::memcmp(tc.last.data(), host, bytes) == 0) {
    if (st != tc.last_stream && tc.ev_pending) CK(cudaStreamWaitEvent(st, tc.ev, 0));   // the upload ran on another stream
    ++ctx->table_reuses;
    return ATOMO_OK;
  }
  if (tc.ev_pending) { CK(cudaEventSynchronize(tc.ev)); tc.ev_pending = false; }          // the staging buffer is free again
  if (tc.last_stream != st && tc.last_stream != nullptr) CK(cudaStreamSynchronize(tc.last_stream));   // readers of the old tables
  if (bytes > tc.hcap) {
    if (tc.h) CK(cudaFreeHost(tc.h));
    tc.h = nullptr; tc.hcap = 0;
    CK(cudaMallocHost(&tc.h, bytes + bytes / 4 + 4096));
    tc.hcap = bytes + bytes / 4 + 4096;
  }
  std::memcpy(tc.h, host, bytes);
  CK(cudaMemcpyAsync(tc.d, tc.h, bytes, cudaMemcpyHostToDevice, st));
  CK(cudaEventRecord(tc.ev, st));
  tc.ev_pending = true;
  tc.last.assign(host, host + bytes);
  tc.last_stream = st;
  ++ctx->table_uploads;
  return ATOMO_OK;
}

void table_free(TableCache& tc) {
  if (tc.d) cudaFree(tc.d);
  if (tc.h) cudaFreeHost(tc.h);
  if (tc.ev) cudaEventDestroy(tc.ev);
  tc = TableCache();
}

// optional: the caller can do with less, so that a workspace that does not fit beside what is allocated already is not even tried
// (freeing the old one first, and waiting for the device, on every such call)
int ensure_ws(atomo_ctx* ctx, size_t bytes, bool optional = false) {
  if (bytes <= ctx->ws_bytes) return ATOMO_OK;
  const size_t limit = ctx->ws_limit < 0 ? SIZE_MAX : (size_t)ctx->ws_limit;
  size_t free_bytes = 0, all_bytes = 0;
  if (bytes > limit || (optional && cudaMemGetInfo(&free_bytes, &all_bytes) == cudaSuccess && bytes > free_bytes + ctx->ws_bytes)) {
    ctx->err = "no room for a workspace of " + std::to_string(bytes) + " bytes";
    return ATOMO_ERR_CUDA;
  }
  if (ctx->ws) { CK(cudaDeviceSynchronize()); CK(cudaFree(ctx->ws)); ctx->ws = nullptr; ctx->ws_bytes = 0; }
  size_t want = std::min(bytes + bytes / 8 + (1 << 20), limit);
  cudaError_t e = cudaMalloc(&ctx->ws, want);
  if (e == cudaErrorMemoryAllocation && want > bytes) {        // without the spare part, then
    cudaGetLastError();
    e = cudaMalloc(&ctx->ws, want = bytes);
  }
  if (e != cudaSuccess) { cudaGetLastError(); ctx->ws = nullptr; return fail_cuda(ctx, e, "cudaMalloc(workspace)"); }
  ctx->ws_bytes = want;
  return ATOMO_OK;
}

void stage_begin(atomo_ctx* ctx, int stage, cudaStream_t st) {
  if (!ctx->profiling) return;
  cudaEventRecord(ctx->ev[ctx->ev_cur][stage][0], st);
  ctx->ev_used[ctx->ev_cur][stage] = true;
}
void stage_end(atomo_ctx* ctx, int stage, cudaStream_t st, int64_t n_launch) {
  ctx->launches[stage] += n_launch;
  ctx->acc_launches[stage] += n_launch;
  if (!ctx->profiling) return;
  cudaEventRecord(ctx->ev[ctx->ev_cur][stage][1], st);
}
// adds the times of one event set to the sums and frees the set (waits for its events: only the newest sets can
// still be running)
void stage_harvest(atomo_ctx* ctx, int slot) {
  for (int i = 0; i < ATOMO_N_STAGES; ++i) {
    if (!ctx->ev_used[slot][i]) continue;
    float ms = 0.0f;
    if (cudaEventSynchronize(ctx->ev[slot][i][1]) == cudaSuccess &&
        cudaEventElapsedTime(&ms, ctx->ev[slot][i][0], ctx->ev[slot][i][1]) == cudaSuccess)
      ctx->acc_ms[i] += (double)ms;
    ctx->ev_used[slot][i] = false;
  }
}
// a new API call: the next event set of the ring
void stage_reset(atomo_ctx* ctx) {
  for (int i = 0; i < ATOMO_N_STAGES; ++i) ctx->launches[i] = 0;
  ++ctx->acc_calls;
  if (!ctx->profiling) return;
  ctx->ev_cur = (ctx->ev_cur + 1) % atomo_ctx::kEvRing;
  stage_harvest(ctx, ctx->ev_cur);
}

int next_pow2_at_least(int x, int lo) { int p = lo; while (p < x) p <<= 1; return p; }

struct SpLayout {                 // payload offsets of one spectral layer
  uint32_t kc; uint64_t off_idx, off_coef, off_short, off_long;
};

uint64_t layout_spectral(const int32_t* rows, const int32_t* cols, int n_layers, int32_t k_cap,
                         std::vector<SpLayout>* out) {
  uint64_t off = sizeof(atomo_payload_header) + (uint64_t)n_layers * sizeof(atomo_layer_header);
  for (int l = 0; l < n_layers; ++l) {
    const int64_t r = std::min(rows[l], cols[l]), L = std::max(rows[l], cols[l]);
    const uint32_t kc = (uint32_t)std::min<int64_t>(k_cap, r);
    SpLayout lo;
    lo.kc = kc;
    off = align_up(off, 16); lo.off_idx = off; off += (uint64_t)kc * 4;
    off = align_up(off, 16); lo.off_coef = off; off += (uint64_t)kc * 4;
    off = align_up(off, 16); lo.off_short = off; off += (uint64_t)kc * r * 4;
    off = align_up(off, 16); lo.off_long = off; off += (uint64_t)kc * L * 4;
    if (out) out->push_back(lo);
  }
  return align_up(off, 16);
}

struct EwLayout { uint32_t kc, sc; uint64_t off_idx, off_val, off_tiles, off_sat; };

// explicit: idx u32[kc], val f32[kc], tile table.  compact: entries u16[kc], saturated values f32[sc], tile table,
// saturated indices u32[sc] (sc = the saturated list's capacity, clamped to n).
uint64_t layout_entrywise(const int64_t* n, int n_vecs, int64_t k_cap, bool compact, int64_t sat_cap,
                          std::vector<EwLayout>* out) {
  uint64_t off = sizeof(atomo_payload_header) + (uint64_t)n_vecs * sizeof(atomo_layer_header);
  for (int l = 0; l < n_vecs; ++l) {
    const uint32_t kc = (uint32_t)std::min<int64_t>(k_cap, n[l]);
    EwLayout lo{};
    lo.kc = kc;
    lo.sc = compact ? (uint32_t)std::min<int64_t>(sat_cap, n[l]) : 0u;
    off = align_up(off, 16); lo.off_idx = off; off += (uint64_t)kc * (compact ? 2 : 4);
    off = align_up(off, 16); lo.off_val = off; off += (uint64_t)(compact ? lo.sc : kc) * 4;
    off = align_up(off, 16); lo.off_tiles = off; off += ((uint64_t)(n[l] + ATOMO_EW_TILE - 1) / ATOMO_EW_TILE + 1) * 4;
    off = align_up(off, 16); lo.off_sat = off; off += (uint64_t)lo.sc * 4;
    if (out) out->push_back(lo);
  }
  return align_up(off, 16);
}

// The vectors of an entry-wise decode in launches of up to kEwBatch of them (one tile per CTA); returns their number
template <typename F>
int for_each_ew_decode(const uint8_t* payload, const int64_t* cols, float* const* out, int n_layers, F launch) {
  const int tile = ew_tile_elems();
  auto fill = [&](auto& B, int first, int count) {
    uint32_t tiles = 0;
    for (int i = 0; i < count; ++i) {
      B.v[i] = EwDecode{out[first + i], cols[first + i], first + i, tiles};
      tiles += (uint32_t)((cols[first + i] + tile - 1) / tile);
    }
    B.n = count; B.payload = payload;
    launch(B, tiles);
  };
  int n_launch = 0;
  for (int l = 0; l < n_layers; ++n_launch) {
    // a vector has fewer than 2^20 tiles, so a batch stays far below the grid limit
    const int count = std::min(n_layers - l, kEwBatch);
    if (count == 1) { EwDecodeBatch<1> B{}; fill(B, l, 1); } else { EwDecodeBatch<kEwBatch> B{}; fill(B, l, count); }
    l += count;
  }
  return n_launch;
}

// What the occupancy queries say of the two-stage reduction, asked for once per context: CTAs of the band reduction that are
// resident together (layers of at most r rows), clusters of the bulge chase that run side by side
int band_room(atomo_ctx* ctx, int form, int r) {
  int lg = 0;
  while ((1 << lg) < r) ++lg;
  int& known = ctx->band_capacity[form][lg];
  if (known < 0) known = sp_band_capacity(form, 1 << lg);
  return ctx->band_limit >= 0 ? std::min(known, ctx->band_limit) : known;
}
int chase_room(atomo_ctx* ctx, int ctas) {
  int lg = 0;
  while ((1 << lg) < ctas) ++lg;
  int& known = ctx->chase_capacity[lg];
  if (known < 0) known = sp_chase_capacity(ctas);
  return ctx->chase_limit >= 0 && ctas > 1 ? std::min(known, ctx->chase_limit) : known;
}
// Layers of up to 512 rows that the TF32 kernel cannot take: integer Gram kernel, or FMA kernel.  `narrow`: how many of them in the call have
// up to 64 rows (one tile of either kernel).  The integer kernel costs two or three launches more and a CTA of 10 us per tile, the FMA kernel a walk
// along the long side on one CTA up to 512 columns, on several from there.  A whole encode, FMA | integer, us:
//   one layer: 17 x 193 95 | 99, 64 x 257 163 | 163, 17 x 321 103 | 99, 128 x 321 268 | 259, 17 x 513 119 | 98; tall 321 x 180 375 | 380, 401 x 128 274 | 268,
//   401 x 64 170 | 172, 449 x 64 174 | 173
//   20 layers: 48 x 257 149 | 153, 48 x 353 157 | 154; 50: 17 x 401 117 | 122, 17 x 513 133 | 123, 64 x 513 201 | 190
//   100 layers: 128 x 321 774 | 769, 33 x 449 190 | 205, 33 x 513 216 | 212, 17 x 1201 180 | 208, 17 x 2401 204 | 208; tall 801 x 64 340 | 332,
//   1601 x 64 415 | 431
//   200 layers (the host's part of the call bounds the narrow ones): 33 x 801 334 | 362, 64 x 801 487 | 498, 64 x 1201 540 | 536, 17 x 2401 331 | 371,
//   33 x 2401 463 | 406, 17 x 5001 489 | 376; 600: 17 x 2401 986 | 1068, 64 x 801 1234 | 1275, 64 x 2401 1602 | 1525
// beside: other layers of the call take the integer kernel, so that a few short ones cost it next to nothing, and the FMA kernel a launch of its own
// (116 x 261 beside 789 x 1195 and 512 x 513, Gram stage: 147 | 125).  The longest keep the FMA kernel's bounded number of parts.
bool i8_small(int r, int L, bool tall, int narrow, bool beside) {
  if (r <= 16 || L > 1 << 16) return false;
  if (beside && narrow <= 32) return L >= 192;
  if (r > 64) return L >= (tall ? 400 : 320);
  if (narrow <= 32) return L >= (tall ? 448 : 320);
  if (narrow <= (r > 32 ? 128 : 64)) return L >= 512;
  return r * L >= 1 << 16;
}
// digits of the integer Gram kernel, as many bytes as their gradients: layers whose own exceed kI8Bytes take the other kernels; the others' are
// made and used in groups of layers, one behind the other in the same kI8Group bytes (96 layers of 1024 x 4096, two groups: 24 waves of CTAs as in one)
constexpr int64_t kI8Bytes = (int64_t)1 << 33, kI8Group = (int64_t)1 << 30;
constexpr int64_t kI8Elements = (int64_t)1 << 26;             // elements from which layers of 513 .. 1024 rows take the integer Gram kernel
int chase_class(int r) { return r <= 1024 ? 1024 : r <= 2048 ? 2048 : 4096; }   // short sides that share a form of the chase

// the context's side stream with the priority of st
int side_stream(atomo_ctx* ctx, cudaStream_t st, cudaStream_t* out) {
  int priority = 0;
  CK(cudaStreamGetPriority(st, &priority));
  for (auto& q : ctx->sides) if (q.first == priority) { *out = q.second; return ATOMO_OK; }
  cudaStream_t s = nullptr;
  CK(cudaStreamCreateWithPriority(&s, cudaStreamNonBlocking, priority));
  ctx->sides.emplace_back(priority, s);
  *out = s;
  return ATOMO_OK;
}

bool bad_budget(double s) { return !(s > 0.0) || !std::isfinite(s); }

}  // namespace

extern "C" {

int atomo_create(atomo_ctx** out, int device) {
  if (!out || device < 0) return ATOMO_ERR_INVALID_ARG;
  atomo_ctx* ctx = new atomo_ctx();
  ctx->device = device;
  *out = ctx;
  CK(cudaSetDevice(device));
  CK(cudaMallocHost(&ctx->h_flag, 256));
  CK(cudaMallocHost(&ctx->h_lq, kLqResults * sizeof(EwLqPart)));
  CK(cudaMalloc(&ctx->ew_words, kEwWords * sizeof(uint32_t)));
  CK(cudaMemset(ctx->ew_words, 0, kEwWords * sizeof(uint32_t)));
  for (int r = 0; r < atomo_ctx::kEvRing; ++r)
    for (int i = 0; i < ATOMO_N_STAGES; ++i) { CK(cudaEventCreate(&ctx->ev[r][i][0])); CK(cudaEventCreate(&ctx->ev[r][i][1])); }
  int e = sp_configure();
  if (e == 0) e = ew_configure();
  if (e != 0) return fail_cuda(ctx, (cudaError_t)e, "cudaFuncSetAttribute(max dynamic shared memory)");
  ctx->tc_ok = sp_tc_configure() == 0;
  CK(cudaEventCreateWithFlags(&ctx->ev_fork, cudaEventDisableTiming));
  CK(cudaEventCreateWithFlags(&ctx->ev_join, cudaEventDisableTiming));
  ctx->configured = true;
  return ATOMO_OK;
}

int atomo_destroy(atomo_ctx* ctx) {
  if (!ctx) return ATOMO_ERR_INVALID_ARG;
  cudaSetDevice(ctx->device);
  cudaDeviceSynchronize();
  for (auto& q : ctx->sides) cudaStreamDestroy(q.second);
  if (ctx->ev_fork) cudaEventDestroy(ctx->ev_fork);
  if (ctx->ev_join) cudaEventDestroy(ctx->ev_join);
  if (ctx->ws) cudaFree(ctx->ws);
  if (ctx->ew_words) cudaFree(ctx->ew_words);
  table_free(ctx->tab_sp); table_free(ctx->tab_avg);
  if (ctx->h_flag) cudaFreeHost(ctx->h_flag);
  if (ctx->h_lq) cudaFreeHost(ctx->h_lq);
  for (int r = 0; r < atomo_ctx::kEvRing; ++r)
    for (int i = 0; i < ATOMO_N_STAGES; ++i) for (int j = 0; j < 2; ++j) if (ctx->ev[r][i][j]) cudaEventDestroy(ctx->ev[r][i][j]);
  delete ctx;
  return ATOMO_OK;
}

const char* atomo_last_cuda_error(atomo_ctx* ctx) { return ctx ? ctx->err.c_str() : "null context"; }

int64_t atomo_payload_bytes_spectral(const int32_t* rows, const int32_t* cols, int32_t n_layers, int32_t k_cap) {
  if (!rows || !cols || n_layers <= 0 || k_cap <= 0) return -1;
  for (int l = 0; l < n_layers; ++l) if (rows[l] <= 0 || cols[l] <= 0) return -1;
  return (int64_t)layout_spectral(rows, cols, n_layers, k_cap, nullptr);
}

int64_t atomo_payload_bytes_entrywise(const int64_t* n, int32_t n_vecs, int64_t k_cap) {
  if (!n || n_vecs <= 0 || k_cap <= 0) return -1;
  for (int l = 0; l < n_vecs; ++l) if (n[l] <= 0 || n[l] >= (int64_t(1) << 32)) return -1;
  return (int64_t)layout_entrywise(n, n_vecs, k_cap, false, 0, nullptr);
}

int64_t atomo_payload_bytes_entrywise_compact(const int64_t* n, int32_t n_vecs, int64_t k_cap, int64_t sat_cap) {
  if (!n || n_vecs <= 0 || k_cap <= 0 || sat_cap < 0) return -1;
  for (int l = 0; l < n_vecs; ++l) if (n[l] <= 0 || n[l] >= (int64_t(1) << 32)) return -1;
  return (int64_t)layout_entrywise(n, n_vecs, k_cap, true, sat_cap, nullptr);
}

int atomo_set_entrywise_format(atomo_ctx* ctx, int32_t format, int64_t sat_cap) {
  if (!ctx || (format != ATOMO_EW_EXPLICIT && format != ATOMO_EW_COMPACT)) return ATOMO_ERR_INVALID_ARG;
  if (format == ATOMO_EW_COMPACT && sat_cap < 0) return ATOMO_ERR_INVALID_ARG;
  ctx->ew_format = format;
  ctx->ew_sat_cap = format == ATOMO_EW_COMPACT ? sat_cap : 0;
  return ATOMO_OK;
}

int atomo_set_profiling(atomo_ctx* ctx, int enabled) {
  if (!ctx) return ATOMO_ERR_INVALID_ARG;
  CK(cudaSetDevice(ctx->device));
  // switching on starts the sums afresh; event sets still in flight are read out first
  for (int r = 0; r < atomo_ctx::kEvRing; ++r) stage_harvest(ctx, r);
  if (enabled) {
    for (int i = 0; i < ATOMO_N_STAGES; ++i) { ctx->acc_ms[i] = 0.0; ctx->acc_launches[i] = 0; }
    ctx->acc_calls = 0;
  }
  ctx->profiling = enabled != 0;
  return ATOMO_OK;
}

int atomo_get_stage_totals(atomo_ctx* ctx, double* ms, int64_t* launches, int64_t* calls) {
  if (!ctx) return ATOMO_ERR_INVALID_ARG;
  CK(cudaSetDevice(ctx->device));
  // everything recorded so far is added up (this waits for the newest calls' events); the current set stays in use
  // for get_stage_times, so its times are read without freeing it
  for (int r = 0; r < atomo_ctx::kEvRing; ++r) if (r != ctx->ev_cur) stage_harvest(ctx, r);
  for (int i = 0; i < ATOMO_N_STAGES; ++i) {
    double cur = 0.0;
    if (ctx->profiling && ctx->ev_used[ctx->ev_cur][i]) {
      float t = 0.0f;
      CK(cudaEventSynchronize(ctx->ev[ctx->ev_cur][i][1]));
      CK(cudaEventElapsedTime(&t, ctx->ev[ctx->ev_cur][i][0], ctx->ev[ctx->ev_cur][i][1]));
      cur = (double)t;
    }
    if (ms) ms[i] = ctx->acc_ms[i] + cur;
    if (launches) launches[i] = ctx->acc_launches[i];
  }
  if (calls) *calls = ctx->acc_calls;
  return ATOMO_OK;
}

int atomo_get_stage_times(atomo_ctx* ctx, float* ms, int64_t* launches) {
  if (!ctx) return ATOMO_ERR_INVALID_ARG;
  CK(cudaSetDevice(ctx->device));
  for (int i = 0; i < ATOMO_N_STAGES; ++i) {
    if (launches) launches[i] = ctx->launches[i];
    if (!ms) continue;
    ms[i] = 0.0f;
    if (ctx->profiling && ctx->ev_used[ctx->ev_cur][i]) {
      CK(cudaEventSynchronize(ctx->ev[ctx->ev_cur][i][1]));
      CK(cudaEventElapsedTime(&ms[i], ctx->ev[ctx->ev_cur][i][0], ctx->ev[ctx->ev_cur][i][1]));
    }
  }
  return ATOMO_OK;
}

int atomo_set_eig_params(atomo_ctx* ctx, int32_t max_sweeps, float tol) {
  if (!ctx || max_sweeps < 1 || max_sweeps > 1000 || !(tol > 0.0f) || !(tol < 1.0f)) return ATOMO_ERR_INVALID_ARG;
  ctx->max_sweeps = max_sweeps;
  ctx->tol = tol;
  return ATOMO_OK;
}

int atomo_last_eig_scheme(atomo_ctx* ctx) { return ctx ? ctx->eig_scheme_used : -1; }

int atomo_get_table_uploads(atomo_ctx* ctx, int64_t* uploads, int64_t* reuses) {
  if (!ctx) return ATOMO_ERR_INVALID_ARG;
  if (uploads) *uploads = ctx->table_uploads;
  if (reuses) *reuses = ctx->table_reuses;
  return ATOMO_OK;
}

int atomo_set_persistent_eig(atomo_ctx* ctx, int32_t enabled) {
  if (!ctx || enabled < 0 || enabled > 3) return ATOMO_ERR_INVALID_ARG;
  ctx->eig_scheme = enabled;
  return ATOMO_OK;
}

int atomo_set_tridiag_ctas(atomo_ctx* ctx, int32_t ctas_per_layer) {
  if (!ctx) return ATOMO_ERR_INVALID_ARG;
  if (ctas_per_layer != 0 && ctas_per_layer != 1 && ctas_per_layer != 2 && ctas_per_layer != 4 && ctas_per_layer != 8 &&
      ctas_per_layer != 16)
    return ATOMO_ERR_INVALID_ARG;
  ctx->tri_big_ctas = ctas_per_layer;
  return ATOMO_OK;
}

int atomo_limit_tridiag_route(atomo_ctx* ctx, int32_t band_ctas, int32_t chase_clusters) {
  if (!ctx || band_ctas < -1 || chase_clusters < -1) return ATOMO_ERR_INVALID_ARG;
  ctx->band_limit = band_ctas;
  ctx->chase_limit = chase_clusters;
  return ATOMO_OK;
}

int atomo_limit_workspace(atomo_ctx* ctx, int64_t bytes) {
  if (!ctx || bytes < -1) return ATOMO_ERR_INVALID_ARG;
  ctx->ws_limit = bytes;
  return ATOMO_OK;
}

int atomo_set_gram_path(atomo_ctx* ctx, int32_t tensor_cores) {
  if (!ctx) return ATOMO_ERR_INVALID_ARG;
  ctx->tc_gram = tensor_cores != 0;
  return ATOMO_OK;
}

int atomo_set_sigma_refinement(atomo_ctx* ctx, int32_t min_short_side) {
  if (!ctx || min_short_side < 0) return ATOMO_ERR_INVALID_ARG;
  ctx->refine_min_short = min_short_side;
  return ATOMO_OK;
}

int atomo_set_eig_mode(atomo_ctx* ctx, int32_t mode) {
  if (!ctx || (mode != 0 && mode != 1)) return ATOMO_ERR_INVALID_ARG;
  ctx->eig_mode = mode;
  return ATOMO_OK;
}

// ==================================================================================================
// use_digits: whether layers may take the integer Gram kernel; comes back false, with nothing launched, if there is no room for their digits
static int encode_spectral_with(atomo_ctx* ctx, const atomo_mat* layers, int32_t n_layers, double s, uint64_t seed,
                                uint64_t step, int32_t k_cap, void* payload, int64_t capacity_bytes,
                                const atomo_debug* dbg, void* stream, const float* const* given_sigma,
                                const float* const* given_short, bool& use_digits) {
  const bool given = given_sigma != nullptr;                   // the decomposition comes from the caller: S1 is skipped
  if (!ctx || !layers || n_layers <= 0 || k_cap <= 0 || !payload) return ATOMO_ERR_INVALID_ARG;
  if (bad_budget(s)) return ATOMO_ERR_BUDGET;
  if ((reinterpret_cast<uintptr_t>(payload) & 15u) != 0) return ATOMO_ERR_INVALID_ARG;
  std::vector<int32_t> rows(n_layers), cols(n_layers);
  for (int l = 0; l < n_layers; ++l) {
    const atomo_mat& m = layers[l];
    if (!m.data || m.rows <= 0 || m.cols <= 0 || m.ld < m.cols) return ATOMO_ERR_INVALID_ARG;
    if (std::min(m.rows, m.cols) > kSmemRowsMaxRp) return ATOMO_ERR_INVALID_ARG;
    rows[l] = m.rows; cols[l] = m.cols;
  }
  std::vector<SpLayout> lay;
  const uint64_t total = layout_spectral(rows.data(), cols.data(), n_layers, k_cap, &lay);
  if ((int64_t)total > capacity_bytes) return ATOMO_ERR_CAPACITY;
  CK(cudaSetDevice(ctx->device));
  cudaStream_t st = (cudaStream_t)stream;
  const int max_sweeps = ctx->max_sweeps;
  uint8_t* pay = static_cast<uint8_t*>(payload);
  atomo_layer_header* d_hdr = reinterpret_cast<atomo_layer_header*>(pay + sizeof(atomo_payload_header));

  // ---- host descriptors, tiles, workspace carving (two passes: size, then pointers) ----
  std::vector<SpLayer> L(n_layers);
  std::vector<int> tc_layers, i8_layers;
  std::vector<int64_t> i8_at;                                // where a layer's digits start in its group's
  std::vector<TileRef> gram_tiles, gram_parts, block_pairs, bp_tiles, chol_ctas, refine_tiles, tc_tiles, i8_prep, i8_tiles;
  const int map_bytes = sp_tc_map_bytes();
  std::vector<uint8_t> maps_blob((size_t)n_layers * map_bytes, 0);
  int chol_panels = 0;
  // groups of layers that take the integer Gram kernel, by position in i8_layers; what the largest group's digits take
  struct I8Group { int first, count, prep, n_rows, n_prep, tiles, n_tiles; };
  std::vector<I8Group> i8_groups;
  int64_t i8_bytes = 0, i8_room = 0;
  int64_t mid_elements = 0;                                  // of the layers with a short side of 513 .. 1024
  int narrow = 0;
  bool beside = false;                                       // see i8_small()
  for (int l = 0; l < n_layers; ++l) {
    const atomo_mat& m = layers[l];
    const int r = std::min(m.rows, m.cols);
    if (r > 512 && r <= 1024) mid_elements += (int64_t)m.rows * m.cols;
    if (r > 16 && r <= 64 && !sp_tc_eligible(m.data, m.rows, m.cols, m.ld)) ++narrow;
  }
  auto tf32 = [&](const atomo_mat& m, bool fits) {
    const int r = std::min(m.rows, m.cols);
    return (r <= 512 || (r <= 1024 && (mid_elements < kI8Elements || !fits))) && sp_tc_eligible(m.data, m.rows, m.cols, m.ld);
  };
  for (int l = 0; l < n_layers && !beside; ++l) {
    const atomo_mat& m = layers[l];
    const int r = std::min(m.rows, m.cols);
    beside = !tf32(m, true) && (r > 512 || i8_small(r, std::max(m.rows, m.cols), m.rows > m.cols, narrow, false));
  }
  int row_floats_max = 0, steps_max = 0, r_max = 0, rp_max = 0, r_max_tall = 0, k_cap_max = 1;
  for (int l = 0; l < n_layers; ++l) {
    SpLayer& d = L[l];
    const atomo_mat& m = layers[l];
    d.G = m.data; d.rows = m.rows; d.cols = m.cols; d.ld = m.ld;
    d.tall = m.rows > m.cols;
    d.r = std::min(m.rows, m.cols); d.L = std::max(m.rows, m.cols);
    d.rp = next_pow2_at_least(d.r, 32);
    d.acc = ctx->eig_mode == 0 ? 1 : 0;
    d.ldx = d.acc ? 2 * d.rp : d.rp;
    if (d.acc && d.ldx > 1024) return ATOMO_ERR_INVALID_ARG;   // route 0 holds rows of 2 rp floats: short side <= 512
    d.B = d.ldx <= 1024 ? 16 : (d.ldx == 2048 ? 8 : 4);          // a rotation is shared by 1, 2 or 4 warps
    d.nb = d.rp / d.B;
    d.layer = (uint32_t)l; d.k_cap = lay[l].kc;
    k_cap_max = std::max(k_cap_max, (int)d.k_cap);
    r_max = std::max(r_max, d.r); rp_max = std::max(rp_max, d.rp);
    const int gt = (d.r + 63) / 64;
    d.tc = 0; d.gram_split = 1;
    d.fma_split = given ? 1 : sp_gram_split(d.r, d.L);
    d.gram_part_len = sp_gram_part(d.r, d.L);
    const int64_t digits = 4 * (int64_t)d.r * sp_i8_pitch(d.L);
    const bool digits_fit = use_digits && digits <= kI8Bytes;
    // The TF32 kernel's fp32 accumulation truncates, which perturbs sum(sigma) -- and with it the largest p_i -- by a few
    // 1e-6 at a short side of 1024 and more above (measured 6e-6 at 4096): layers with a short side above 1024 take the integer
    // kernel, and below those that the TF32 kernel cannot take (i8_small), or of 513 to 1024 rows all where they are many (TF32 |
    // integer, us: 20 layers of 1000 x 1200 241 | 259, one of 1024 x 4096 51 | 64, 40 of 520 x 8000 1081 | 767, 96 of 1024 x 4096 2818 | 2185)
    if (ctx->tc_gram && ctx->tc_ok && !d.acc && tf32(m, digits_fit)) {
      d.tc = 1;
      if (sp_tc_make_map(maps_blob.data() + (size_t)l * map_bytes, d.G, d.rows, d.cols, d.ld) != 0) return ATOMO_ERR_INVALID_ARG;
      tc_layers.push_back(l);
    } else if (ctx->tc_gram && ctx->tc_ok && !d.acc && !given && digits_fit && (d.r > 512 || i8_small(d.r, d.L, d.tall, narrow, beside))) {
      d.tc = 2;
      if (i8_groups.empty() || i8_bytes + digits > kI8Group) { i8_groups.push_back({(int)i8_layers.size(), 0, 0, 0, 0, 0, 0}); i8_bytes = 0; }
      ++i8_groups.back().count;
      i8_at.push_back(i8_bytes);
      i8_bytes += (digits + 255) / 256 * 256;
      i8_room = std::max(i8_room, i8_bytes);
      i8_layers.push_back(l);
    } else {
      for (int a = 0; a < gt; ++a) for (int b = a; b < gt; ++b) for (int c = 0; c < d.fma_split; ++c) (d.r > 1024 ? gram_tiles : gram_parts).push_back({l, a, b, c});
    }
    for (int p = 0; p < d.nb / 2; ++p) block_pairs.push_back({l, p, 0, 0});
    row_floats_max = std::max(row_floats_max, d.ldx); steps_max = std::max(steps_max, d.nb - 1);
    if (!d.acc && d.rp > 1024) {
      const int per = sp_cholesky_big_rows_per_cta();
      for (int c = 0; c < (d.rp + per - 1) / per; ++c) chol_ctas.push_back({l, c, 0, 0});
      chol_panels = std::max(chol_panels, (d.r + 31) / 32);
    }
    d.bp_tiles = d.tall ? (d.L + sp_bp_rows_per_tile() - 1) / sp_bp_rows_per_tile()
                        : (d.L + sp_bp_cols_per_tile() - 1) / sp_bp_cols_per_tile();
    {   // row chunks of the wide back-projection: 64 rows each, fewer and longer when k_cap makes the partials large
      const int64_t per_chunk = (int64_t)d.k_cap * d.L * (int64_t)sizeof(float);
      const int unit = sp_bp_chunk_rows();
      const int want = (d.r + unit - 1) / unit;
      const int fit = (int)std::max<int64_t>(1, ((int64_t)32 << 20) / per_chunk);
      const int chunks = d.tall ? 1 : std::min(want, fit);
      d.bp_chunk_rows = ((d.r + chunks - 1) / chunks + unit - 1) / unit * unit;
      d.bp_chunks = d.tall ? 1 : (d.r + d.bp_chunk_rows - 1) / d.bp_chunk_rows;
    }
    for (int t = 0; t < d.bp_tiles; ++t) for (int c = 0; c < d.bp_chunks; ++c) bp_tiles.push_back({l, t, c, 0});
    if (d.tall) r_max_tall = std::max(r_max_tall, d.r);
    d.refine = d.r >= ctx->refine_min_short ? 1 : 0;
    d.refine_tiles = (d.L + 63) / 64;
    if (d.refine)
      for (int a = 0; a < gt; ++a) for (int b = 0; b < d.refine_tiles; ++b) refine_tiles.push_back({l, a, b, 0});
  }
  gram_tiles.insert(gram_tiles.end(), gram_parts.begin(), gram_parts.end());   // (an instance of the kernel each)
  // Tridiagonal routes first: eigenvalues of every atom from T = Q^T A Q, vectors for the kept atoms only -- in the
  // registers of a cluster for short sides up to 512, in two stages with A in global memory above (no per-atom refinement,
  // no request for the whole short-side basis).  Otherwise the Jacobi routes, the cluster form first.
  bool tri_form = !given && ctx->eig_scheme == 3 && ctx->eig_mode != 0 && !(dbg && dbg->short_vecs);
  bool any_small = false, any_big = false;
  for (int l = 0; l < n_layers && tri_form; ++l) (L[l].rp <= sp_tridiag_max_rp() ? any_small : any_big) = true;
  if (tri_form && any_small) {
    if (ctx->tri_clusters < 0) ctx->tri_clusters = sp_configure_tridiag();
    if (ctx->tri_clusters < 1) tri_form = false;
  }
  if (tri_form && any_big) {
    if (ctx->tri_big_ok < 0) ctx->tri_big_ok = (sp_configure_band() == 0 && sp_configure_eigvec_big() == 0 && sp_configure_bisect() == 0) ? 1 : 0;
    if (ctx->tri_big_ok < 1 || r_max > sp_band_max_r()) tri_form = false;
  }
  // the large layers, largest first; a GPU that cannot hold a CTA of their band reduction or a cluster of their chase takes the
  // Jacobi routes
  std::vector<int> big_layers;
  int band_form = 0;
  if (tri_form && any_big) {
    int64_t strips = 0;
    for (int l = 0; l < n_layers; ++l) if (L[l].rp > sp_tridiag_max_rp()) { big_layers.push_back(l); strips += sp_band_strips(L[l].r); }
    std::stable_sort(big_layers.begin(), big_layers.end(), [&](int a, int b) { return L[a].r > L[b].r; });
    band_form = sp_band_form(r_max, strips);
    bool can = band_room(ctx, band_form, r_max) >= 1;
    for (int l : big_layers) { const int few = sp_chase_ctas(chase_class(L[l].r), 1, 0); can &= chase_room(ctx, few) >= 1; }
    if (!can) { tri_form = false; big_layers.clear(); }
  }
  for (int l = 0; l < n_layers; ++l) {
    L[l].tri = !tri_form ? 0 : (L[l].rp <= sp_tridiag_max_rp() ? 1 : 2);
    if (L[l].tri) { L[l].refine = 0; }
  }
  if (tri_form) refine_tiles.clear();
  bool cluster_form = !given && !tri_form && ctx->eig_scheme >= 2 && ctx->eig_mode != 0;
  for (int l = 0; l < n_layers && cluster_form; ++l) cluster_form = L[l].nb / 2 <= sp_jacobi_cluster_ctas() && L[l].rp <= sp_jacobi_cluster_max_rp();
  if (cluster_form) {
    int lg = 0;
    while ((1 << lg) < rp_max) ++lg;
    if (ctx->cluster_capacity[lg] < 0) ctx->cluster_capacity[lg] = sp_jacobi_cluster_capacity(rp_max);
    if (ctx->cluster_capacity[lg] < 1) cluster_form = false;
  }
  for (int l = 0; l < n_layers; ++l) L[l].lam_ready = (cluster_form || tri_form || given) ? 1 : 0;
  if (given) { for (int l = 0; l < n_layers; ++l) L[l].refine = 0; refine_tiles.clear(); }
  // tensor-core Gram tiles: while the batch has fewer CTAs than the GPU has SMs, the K range of a layer's tiles is split into parts of
  // at most `most` stages (TF32: 32 columns each, 16 at least; integers: 64 columns, 8 at least), the smallest `most` with which the
  // parts of all layers are resident together.  (Doubling the longest layer's split as long as it fitted left one of the ResNet-18
  // set's four largest layers with twice the others' stages: 83 -> 63 us.)
  {
    int sms = 148, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    auto tiles_of = [&](int l) { const int tt = (L[l].r + sp_tc_tile() - 1) / sp_tc_tile(); return (int64_t)tt * (tt + 1) / 2; };
    auto split = [&](const std::vector<int>& which, int least, auto stages_of, auto min_of) {
      auto parts = [&](int l, int most) { return std::max(min_of(l), std::max(1, std::min((stages_of(l) + most - 1) / most, stages_of(l) / least))); };
      int lo = least, hi = least;                              // (more stages per part: never more parts)
      for (int l : which) hi = std::max(hi, stages_of(l));
      while (lo < hi) {
        const int mid = (lo + hi) / 2;
        int64_t total = 0;
        for (int l : which) total += tiles_of(l) * parts(l, mid);
        if (total <= sms) hi = mid; else lo = mid + 1;
      }
      for (int l : which) L[l].gram_split = parts(l, lo);
    };
    split(tc_layers, 16, [&](int l) { return (L[l].L + 31) / 32; }, [](int) { return 1; });
    for (I8Group& g : i8_groups) {
      const std::vector<int> which(i8_layers.begin() + g.first, i8_layers.begin() + g.first + g.count);
      split(which, 8, [&](int l) { return sp_i8_stages(L[l].L); }, [&](int l) { return sp_i8_min_split(L[l].L); });
      int64_t i8_row_count = 0;                              // (rows per CTA of the digits' kernel: one after the other, eight CTAs per SM)
      for (int l : which) if (sp_i8_by_rows(L[l].L, L[l].tall)) i8_row_count += L[l].r;
      const int row_step = (int)std::min<int64_t>(16, std::max<int64_t>(1, i8_row_count / (8 * sms)));
      std::vector<TileRef> two_pass;
      g.prep = (int)i8_prep.size(); g.tiles = (int)i8_tiles.size();
      for (int l : which) {
        const int tt = (L[l].r + sp_tc_tile() - 1) / sp_tc_tile();
        for (int a = 0; a < tt; ++a) for (int b = a; b < tt; ++b)
          for (int c = 0; c < L[l].gram_split; ++c) i8_tiles.push_back({l, a, b, c});
        int na = 0, nb = 0;
        sp_i8_prep_tiles(L[l].r, L[l].L, L[l].tall, &na, &nb);
        if (sp_i8_by_rows(L[l].L, L[l].tall)) for (int a = 0; a < na; a += row_step) i8_prep.push_back({l, a, 0, row_step});
        else for (int a = 0; a < na; ++a) for (int b = 0; b < nb; ++b) two_pass.push_back({l, a, b, 0});
      }
      g.n_rows = (int)i8_prep.size() - g.prep;
      i8_prep.insert(i8_prep.end(), two_pass.begin(), two_pass.end());
      g.n_prep = (int)i8_prep.size() - g.prep; g.n_tiles = (int)i8_tiles.size() - g.tiles;
    }
    for (int l : tc_layers) {
      const int tt = (L[l].r + sp_tc_tile() - 1) / sp_tc_tile();
      for (int a = 0; a < tt; ++a) for (int b = a; b < tt; ++b)
        for (int c = 0; c < L[l].gram_split; ++c) tc_tiles.push_back({l, a, b, c});
    }
  }
  // cluster tables of the eigen stage: small tridiagonal layers packed into 16-CTA clusters, largest first (a layer
  // takes rp / 32 consecutive ranks of one cluster); or, on the Jacobi cluster route, the block pairs of every layer
  std::vector<ClusterCta> ctas;
  int n_clusters = 0, rp_max_small = 32;
  if (tri_form) {
    const int per = sp_tridiag_cluster_ctas();
    std::vector<int> order;
    for (int l = 0; l < n_layers; ++l) if (L[l].tri == 1) { order.push_back(l); rp_max_small = std::max(rp_max_small, L[l].rp); }
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return L[a].rp > L[b].rp; });
    std::vector<int> used;
    for (int l : order) {
      const int nc = sp_tridiag_ctas_of(L[l].rp);
      size_t c = 0;
      while (c < used.size() && used[c] + nc > per) ++c;
      if (c == used.size()) { used.push_back(0); ctas.resize(ctas.size() + per, ClusterCta{-1, 0, 0, 0}); }
      for (int sl = 0; sl < nc; ++sl) ctas[c * per + used[c] + sl] = ClusterCta{l, sl, used[c], nc};
      used[c] += nc;
    }
    n_clusters = (int)used.size();
  } else if (cluster_form) {
    const int per = sp_jacobi_cluster_ctas();
    std::vector<int> order(n_layers);
    for (int l = 0; l < n_layers; ++l) order[l] = l;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return L[a].nb > L[b].nb; });
    std::vector<int> used;                                 // slots taken in each cluster (first fit, largest first)
    for (int l : order) {
      const int need_slots = L[l].nb / 2;
      size_t c = 0;
      while (c < used.size() && used[c] + need_slots > per) ++c;
      if (c == used.size()) { used.push_back(0); ctas.resize(ctas.size() + per, ClusterCta{-1, 0, 0, 0}); }
      for (int sl = 0; sl < need_slots; ++sl) ctas[c * per + used[c] + sl] = ClusterCta{l, sl, used[c], 0};
      used[c] += need_slots;
    }
    n_clusters = (int)used.size();
  }
  // two-stage reduction of the large layers, largest first: CTAs of the first stage dealt in proportion to the work (r^3); a
  // launch holds as many as are resident together (they wait for one another), further layers take another launch
  struct BandRun { int first, count, form, r_max; };
  std::vector<BandRun> band_runs;
  std::vector<ClusterCta> band_ctas;
  if (tri_form && any_big) {
    for (size_t i = 0; i < big_layers.size();) {
      const int rm = L[big_layers[i]].r, room = band_room(ctx, band_form, rm);   // (at least what the largest layer was given above)
      const int fixed = ctx->tri_big_ctas;                           // CTAs per layer asked for (0: chosen here)
      size_t n = 0;
      int used = 0;
      double work = 0.0;
      while (i + n < big_layers.size()) {
        const int want = fixed > 0 ? std::min({fixed, sp_band_strips(L[big_layers[i + n]].r), room}) : 1;
        if (used + want > room) break;
        used += want;
        const double rr = L[big_layers[i + n]].r;
        work += rr * rr * rr;
        ++n;
      }
      // (a strip's columns are dealt to CTAs as well: four warps' worth of a strip are enough for one)
      const int band_spread = std::max(1, sp_band_parts(band_form) / 4);
      std::vector<int> g(n);
      int total = 0;
      for (size_t q = 0; q < n; ++q) {
        const double rr = L[big_layers[i + q]].r;
        const int strips = sp_band_strips(L[big_layers[i + q]].r);
        g[q] = fixed > 0 ? std::min({fixed, strips, room}) : std::max(1, std::min(strips * band_spread, (int)(room * (rr * rr * rr / work))));
        total += g[q];
      }
      for (size_t q = n; total > room; q = q > 1 ? q - 1 : n) if (g[q - 1] > 1) { --g[q - 1]; --total; }   // the minimum of one each went over
      BandRun run{(int)band_ctas.size(), 0, band_form, rm};
      for (size_t q = 0; q < n; ++q) for (int c = 0; c < g[q]; ++c) band_ctas.push_back(ClusterCta{big_layers[i + q], c, 0, g[q]});
      run.count = (int)band_ctas.size() - run.first;
      band_runs.push_back(run);
      i += n;
    }
  }
  // the tables go to the table cache (device buffer tab_sp, host mirror `tables` with the same offsets), everything
  // the kernels write to the workspace
  SpLayer* d_layers = nullptr; TileRef *d_gram = nullptr, *d_pairs = nullptr, *d_bp = nullptr, *d_chol = nullptr, *d_ref = nullptr, *d_tc = nullptr, *d_i8_prep = nullptr, *d_i8 = nullptr;
  uint8_t* d_maps = nullptr;
  uint32_t *d_flag = nullptr, *d_coarse = nullptr;
  ClusterCta* d_ctas = nullptr;
  int* d_big = nullptr;
  ClusterCta* d_band = nullptr;
  const float** d_given = nullptr;
  atomo_layer_header* d_hdr_tmpl = nullptr;
  std::vector<uint8_t> tables;
  size_t table_bytes = 0;
  uint64_t tkey = table_key(kKeySeed, layers, (size_t)n_layers * sizeof(atomo_mat));
  tkey = table_key(tkey, &payload, sizeof(payload));
  tkey = table_key(tkey, &k_cap, sizeof(k_cap));
  if (given) { tkey = table_key(tkey, given_sigma, (size_t)n_layers * sizeof(float*)); tkey = table_key(tkey, given_short, (size_t)n_layers * sizeof(float*)); }
  TableCache& tab = table_pick(ctx->tab_sp, tkey);
  for (int pass = 0; pass < 2; ++pass) {
    Arena T(pass ? tab.d : nullptr);
    d_layers = T.take<SpLayer>(n_layers);
    d_gram = T.take<TileRef>(gram_tiles.size());
    d_pairs = T.take<TileRef>(block_pairs.size());
    d_bp = T.take<TileRef>(bp_tiles.size());
    d_chol = T.take<TileRef>(chol_ctas.size());
    d_ref = T.take<TileRef>(refine_tiles.size());
    d_tc = T.take<TileRef>(tc_tiles.size());
    d_i8_prep = T.take<TileRef>(i8_prep.size());
    d_i8 = T.take<TileRef>(i8_tiles.size());
    d_maps = T.take<uint8_t>(maps_blob.size());
    d_ctas = T.take<ClusterCta>(ctas.size());
    d_big = T.take<int>(big_layers.size());
    d_band = T.take<ClusterCta>(band_ctas.size());
    d_given = T.take<const float*>(given ? (size_t)2 * n_layers : 0);
    d_hdr_tmpl = T.take<atomo_layer_header>(n_layers);
    table_bytes = T.off + 256;
    if (pass == 0) { const int rc = table_reserve(ctx, tab, table_bytes); if (rc != ATOMO_OK) return rc; }
  }
  tables.assign(table_bytes, 0);
  auto put = [&](const void* dev_ptr, const void* src, size_t bytes) {
    if (bytes) std::memcpy(tables.data() + (reinterpret_cast<const uint8_t*>(dev_ptr) - tab.d), src, bytes);
  };
  uint8_t* zero_beg = nullptr; size_t zero_bytes = 0;
  size_t need = 0;
  for (int pass = 0; pass < 2; ++pass) {
    Arena A(pass ? ctx->ws : nullptr);
    d_flag = A.take<uint32_t>(4);
    int8_t* const digits = A.take<int8_t>((size_t)i8_room);
    for (size_t q = 0; q < i8_layers.size(); ++q) L[i8_layers[q]].i8_dig = digits + i8_at[q];
    size_t dbg_atoms = 0, dbg_words = 0, dbg_sq = 0;
    for (int l = 0; l < n_layers; ++l) {
      SpLayer& d = L[l];
      d.lam = A.take<float>(d.rp);
      d.perm = A.take<int>(d.r);
      float* sig_ws = A.take<float>(d.r);
      float* prob_ws = A.take<float>(d.r);
      uint32_t* mask_ws = A.take<uint32_t>((d.r + 31) / 32);
      d.sigma = (dbg && dbg->sigma) ? dbg->sigma + dbg_atoms : sig_ws;
      d.prob = (dbg && dbg->prob) ? dbg->prob + dbg_atoms : prob_ws;
      d.mask_words = (dbg && dbg->mask_words) ? dbg->mask_words + dbg_words : mask_ws;
      d.dbg_short = (dbg && dbg->short_vecs) ? dbg->short_vecs + dbg_sq : nullptr;
      dbg_atoms += d.r; dbg_words += (d.r + 31) / 32; dbg_sq += (size_t)d.r * d.r;
      d.p_sel = A.take<float>(d.k_cap);
      d.bp_part = A.take<float>((size_t)d.bp_chunks * d.k_cap * d.L);
      d.scale = A.take<float>(1);
      {
        const int tt = (d.r + sp_tc_tile() - 1) / sp_tc_tile();
        d.gram_part = A.take<float>(d.tc == 1 && d.gram_split > 1
                                        ? (size_t)tt * (tt + 1) / 2 * d.gram_split * sp_tc_tile() * sp_tc_tile() : 0);
      }
      d.gram_sums = A.take<double>(d.tc == 1 ? 0 : (size_t)std::max(sp_gram_sums(d.r, d.fma_split), d.tc == 2 ? sp_i8_sums(d.r, d.gram_split) : 0));
      d.i8_ld = sp_i8_pitch(d.L);
      d.td_d = A.take<double>(d.tri ? d.rp : 0); d.td_e = A.take<double>(d.tri ? d.rp : 0);
      d.lam64 = A.take<double>(d.tri ? d.rp : 0);
      d.td_ldv = (d.r + 3) / 4 * 4;
      d.td_V = A.take<float>(d.tri ? (size_t)d.r * d.td_ldv : 0);
      d.tb_z = A.take<double>(d.tri ? (size_t)d.k_cap * d.rp : 0);
      d.close_work = A.take<double>(d.tri ? (size_t)kCloseWork * d.rp : 0);
      d.close_flag = A.take<uint32_t>(d.tri ? d.k_cap : 0);
      {
        const size_t on = d.tri == 2 ? 1 : 0, rows = (size_t)sp_band_strips(d.r) * 64;
        d.bd_UW = A.take<float>(on * rows * 2 * kBandWidth);
        d.bd_X = A.take<float>(on * rows * kBandWidth);
        d.bd_part = A.take<double>(on * sp_band_parts(band_form) * rows * kBandWidth);
        d.bd_S = A.take<double>(on * 3 * 128);
        d.bd_G = A.take<double>(on * rows / 32 * 36);
        d.bd_band = A.take<double>(on * d.r * (kBandWidth + 1));
        d.bd_T = A.take<double>(on * sp_band_steps(d.r) * kBandWidth * kBandWidth);
        d.bd_V2 = A.take<double>(on * d.r * sp_chase_row(d.r));
      }
      d.chol_dd = A.take<float>(32 * 32 + 32);
      d.row_inv = A.take<float>(d.rp);
      d.refine_partials = A.take<float>(d.refine ? (size_t)d.refine_tiles * d.rp : 0);
      d.hdr = d_hdr + l;
      d.idx = reinterpret_cast<uint32_t*>(pay + lay[l].off_idx);
      d.coef = reinterpret_cast<float*>(pay + lay[l].off_coef);
      d.shortv = reinterpret_cast<float*>(pay + lay[l].off_short);
      d.longv = reinterpret_cast<float*>(pay + lay[l].off_long);
    }
    // zero-filled region: rotation counters and the X matrices
    uint8_t* zb = reinterpret_cast<uint8_t*>(A.take<uint32_t>(0));
    size_t z0 = A.off;
    for (int l = 0; l < n_layers; ++l) { L[l].rot_count = A.take<uint32_t>(max_sweeps); L[l].step_bar = A.take<uint32_t>(1); L[l].vec_ticket = A.take<uint32_t>(2); L[l].bd_bar = A.take<uint32_t>(1); }
    for (int l = 0; l < n_layers; ++l) {
      const int tt = (L[l].r + sp_tc_tile() - 1) / sp_tc_tile();
      const int tf = (L[l].r + 63) / 64;
      L[l].gram_ticket = A.take<uint32_t>(L[l].gram_split > 1 ? (size_t)(tt * (tt + 1) / 2) : 0);
      L[l].fma_ticket = A.take<uint32_t>(L[l].tc != 1 && L[l].fma_split > 1 ? (size_t)(tf * (tf + 1) / 2) : 0);
    }
    for (int l = 0; l < n_layers; ++l) {
      L[l].i8_max = A.take<uint32_t>(L[l].tc == 2 ? (size_t)L[l].r : 0);
      L[l].i8_stat = A.take<I8Stat>(L[l].tc == 2 ? (size_t)L[l].r : 0);
    }
    d_coarse = A.take<uint32_t>(1);
    for (int l = 0; l < n_layers; ++l) L[l].X = A.take<float>(L[l].tri ? 0 : (size_t)L[l].rp * L[l].ldx);
    zero_beg = zb; zero_bytes = A.off - z0;
    for (int l = 0; l < n_layers; ++l) {
      SpLayer& d = L[l];
      if (d.acc) { d.A = d.X; d.lda = d.ldx; }
      else if (d.tri == 2) { d.lda = (int64_t)sp_band_strips(d.r) * 64; d.A = A.take<float>((size_t)d.r * d.lda); }   // whole strips
      else { d.A = A.take<float>((size_t)d.r * d.r); d.lda = d.r; }
    }
    need = A.off + 256;
    if (pass == 0) {
      const int rc = ensure_ws(ctx, need, i8_room > 0);
      if (rc != ATOMO_OK) { use_digits = i8_room == 0; return rc; }
    }
  }

  stage_reset(ctx);
  // ---- tables (uploaded only if they changed since the last call), headers, zero-filled regions ----
  atomo_payload_header gh{};
  gh.magic = ATOMO_MAGIC; gh.version = ATOMO_VERSION; gh.kind = ATOMO_KIND_SPECTRAL; gh.n_layers = (uint32_t)n_layers;
  gh.total_bytes = total; gh.seed = seed; gh.step = step; gh.s = s;
  {
    std::vector<atomo_layer_header> tmpl(n_layers);
    for (int l = 0; l < n_layers; ++l) {
      atomo_layer_header h{};
      h.rows = rows[l]; h.cols = cols[l]; h.k_cap = lay[l].kc; h.k = 0; h.status = ATOMO_OK;
      h.off_idx = lay[l].off_idx; h.off_val = lay[l].off_coef; h.off_short = lay[l].off_short; h.off_long = lay[l].off_long;
      tmpl[l] = h;
    }
    put(d_hdr_tmpl, tmpl.data(), tmpl.size() * sizeof(atomo_layer_header));
  }
  for (int l : i8_layers)
    if (sp_i8_make_map(maps_blob.data() + (size_t)l * map_bytes, L[l].i8_dig, L[l].r, L[l].L, L[l].i8_ld) != 0) return ATOMO_ERR_INVALID_ARG;
  put(d_layers, L.data(), L.size() * sizeof(SpLayer));
  put(d_gram, gram_tiles.data(), gram_tiles.size() * sizeof(TileRef));
  put(d_pairs, block_pairs.data(), block_pairs.size() * sizeof(TileRef));
  put(d_bp, bp_tiles.data(), bp_tiles.size() * sizeof(TileRef));
  put(d_chol, chol_ctas.data(), chol_ctas.size() * sizeof(TileRef));
  put(d_ref, refine_tiles.data(), refine_tiles.size() * sizeof(TileRef));
  put(d_tc, tc_tiles.data(), tc_tiles.size() * sizeof(TileRef));
  put(d_i8_prep, i8_prep.data(), i8_prep.size() * sizeof(TileRef));
  put(d_i8, i8_tiles.data(), i8_tiles.size() * sizeof(TileRef));
  put(d_maps, maps_blob.data(), maps_blob.size());
  put(d_ctas, ctas.data(), ctas.size() * sizeof(ClusterCta));
  put(d_big, big_layers.data(), big_layers.size() * sizeof(int));
  put(d_band, band_ctas.data(), band_ctas.size() * sizeof(ClusterCta));
  if (given) {
    std::vector<const float*> ptrs(2 * (size_t)n_layers);
    for (int l = 0; l < n_layers; ++l) { ptrs[l] = given_sigma[l]; ptrs[n_layers + l] = given_short[l]; }
    put(d_given, ptrs.data(), ptrs.size() * sizeof(const float*));
  }
  { const int rc = table_commit(ctx, tab, tables.data(), table_bytes, st); if (rc != ATOMO_OK) return rc; }
  launch_sp_begin(pay, gh, d_hdr_tmpl, n_layers, d_flag, st);          // payload header, layer headers, flags
  CK(cudaMemsetAsync(zero_beg, 0, zero_bytes, st));

  // ---- S1: Gram matrix, scaling ----
  stage_begin(ctx, ATOMO_STAGE_GRAM, st);
  if (given) {
    // singular values and short-side vectors as given: squared into the eigenvalue slots, vectors into the rows of X
    launch_sp_load_svd(d_layers, n_layers, d_given, d_given + n_layers, st);
  } else {
  if (ctx->eig_mode == 0) launch_sp_init(d_layers, n_layers, nullptr, 0, st);   // the identity half of [A | I]
  launch_sp_gram(d_layers, d_gram, (int)gram_tiles.size(), (int)gram_parts.size(), st);
  launch_sp_gram_tc(d_layers, d_maps, d_tc, (int)tc_tiles.size(), d_flag + 1, st);
  for (const I8Group& g : i8_groups) launch_sp_gram_i8(d_layers, d_maps, d_i8_prep + g.prep, g.n_rows, g.n_prep, d_i8 + g.tiles, g.n_tiles, d_flag + 1, d_coarse, st);
  if (!i8_layers.empty()) launch_sp_gram_coarse(d_layers, n_layers, d_coarse, st);
  launch_sp_scale(d_layers, n_layers, r_max, st);
  }
  if (!given && ctx->eig_mode != 0 && !tri_form) {
    const int ec = launch_sp_cholesky(d_layers, n_layers, rp_max, st);
    if (ec != 0) return fail_cuda(ctx, (cudaError_t)ec, "cudaLaunchKernelEx(cholesky)");
    const int e = launch_sp_cholesky_big(d_layers, d_chol, (int)chol_ctas.size(), chol_panels, st);
    if (e != 0) return fail_cuda(ctx, (cudaError_t)e, "cudaLaunchCooperativeKernel(cholesky)");
  }
  const bool fma_large = gram_tiles.size() > gram_parts.size();
  int i8_launches = i8_groups.empty() ? 0 : 1;
  for (const I8Group& g : i8_groups) i8_launches += 1 + (g.n_rows > 0 ? 1 : 0) + (g.n_prep > g.n_rows ? 2 : 0);
  stage_end(ctx, ATOMO_STAGE_GRAM, st, given ? 1 : 2 + (fma_large ? 1 : 0) + (gram_parts.empty() ? 0 : 1) + (tc_tiles.empty() ? 0 : 1) +
                                           i8_launches);
  CK(cudaGetLastError());

  // ---- S1: eigen-solver; the host reads a convergence flag once per sweep of the largest layer ----
  stage_begin(ctx, ATOMO_STAGE_EIG, st);
  int t_done = 0;
  int64_t n_eig_launch = 0;
  bool flags_pending = false;
  // Persistent form: the block pairs of a group of whole layers are co-resident (one CTA per SM) and solve their
  // layers in one cooperative launch.  A batch larger than the GPU is cut into such groups, launched one after
  // the other; a single layer with more block pairs than the GPU holds CTAs falls back to one launch per step.
  cudaStream_t side = nullptr;
  if (tri_form && any_small && any_big) { const int rc = side_stream(ctx, st, &side); if (rc != ATOMO_OK) return rc; }
  if (tri_form) {
    // small layers beside larger ones: their reduction (0.5 to 0.7 ms on up to 96 SMs) runs on a stream of the context's own next to the
    // chase, which leaves most of the GPU idle; the call's stream waits for it before the eigenvalues
    const bool beside = n_clusters > 0 && any_big;
    if (n_clusters > 0 && !beside) {
      const int e = launch_sp_tridiag(d_layers, d_ctas, n_clusters, d_flag + 1, st);
      if (e != 0) return fail_cuda(ctx, (cudaError_t)e, "cudaLaunchKernelEx(tridiagonal reduction)");
      ++n_eig_launch;
    }
    for (const BandRun& b : band_runs) {                             // larger layers: to a band, then to tridiagonal form
      const int e = launch_sp_band(d_layers, d_band + b.first, b.count, b.form, b.r_max, d_flag + 1, st);
      if (e != 0) return fail_cuda(ctx, (cudaError_t)e, "cudaLaunchCooperativeKernel(band reduction)");
      ++n_eig_launch;
    }
    if (beside) CK(cudaEventRecord(ctx->ev_fork, st));
    int chase_err = 0;
    for (size_t i = 0, n; i < big_layers.size() && chase_err == 0; i += n) {   // (sorted: layers of one class are neighbours)
      const int of = chase_class(L[big_layers[i]].r);
      n = 1;
      while (i + n < big_layers.size() && chase_class(L[big_layers[i + n]].r) == of) ++n;
      const int c = sp_chase_ctas(of, (int)n, of > 1024 ? chase_room(ctx, of / 256) : 0);
      chase_err = launch_sp_chase(d_layers, d_big + i, (int)n, c, st);
      ++n_eig_launch;
    }
    if (beside) {                                                    // (behind the chase in the order of launches: the longer one first)
      CK(cudaStreamWaitEvent(side, ctx->ev_fork, 0));
      const int e = launch_sp_tridiag(d_layers, d_ctas, n_clusters, d_flag + 1, side);
      CK(cudaEventRecord(ctx->ev_join, side));
      CK(cudaStreamWaitEvent(st, ctx->ev_join, 0));
      if (e != 0) return fail_cuda(ctx, (cudaError_t)e, "cudaLaunchKernelEx(tridiagonal reduction)");
      ++n_eig_launch;
    }
    if (chase_err != 0) return fail_cuda(ctx, (cudaError_t)chase_err, "cudaLaunchKernelEx(bulge chase)");
    // the eigenvalues are timed with the sampling stage.  No host wait on this route: a bounded wait of
    // the Gram kernel that ran out is reported by the sampling kernel in every layer's status word
    // (ATOMO_ERR_TIMEOUT, nothing kept)
  }
  if (cluster_form) {
    const int e = launch_sp_jacobi_cluster(d_layers, d_ctas, n_clusters, rp_max, max_sweeps, ctx->tol, st);
    if (e != 0) return fail_cuda(ctx, (cudaError_t)e, "cudaLaunchKernelEx(jacobi clusters)");
    launch_sp_check(d_layers, n_layers, steps_max * max_sweeps, max_sweeps, d_flag, st);
    n_eig_launch = 2;
    CK(cudaMemsetAsync(d_flag + 2, 0, 2 * sizeof(uint32_t), st));
    CK(cudaMemcpyAsync(ctx->h_flag, d_flag, 4 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    flags_pending = true;                                  // read at the end of the call, after everything is enqueued
  }
  const int capacity = (!given && !cluster_form && !tri_form && ctx->eig_scheme >= 1) ? sp_jacobi_persistent_capacity(row_floats_max) : 0;
  int max_layer_pairs = 0;
  for (int l = 0; l < n_layers; ++l) max_layer_pairs = std::max(max_layer_pairs, L[l].nb / 2);
  const bool persistent = capacity > 0 && max_layer_pairs <= capacity;
  if (!given) ctx->eig_scheme_used = tri_form ? 3 : cluster_form ? 2 : (persistent ? 1 : 0);
  if (cluster_form || tri_form || given) {
    // done above
  } else if (persistent) {
    // d_flag[2] is raised if a step barrier gave up, d_flag[3] receives the steps executed
    CK(cudaMemsetAsync(d_flag + 2, 0, 2 * sizeof(uint32_t), st));
    const int t_max = steps_max * max_sweeps;
    size_t first = 0;                                     // block_pairs is ordered by layer
    while (first < block_pairs.size()) {
      size_t last = first;
      while (last < block_pairs.size()) {
        const int l = block_pairs[last].layer;
        const size_t layer_pairs = (size_t)L[l].nb / 2;
        if (last + layer_pairs - first > (size_t)capacity) break;
        last += layer_pairs;
      }
      const int e = launch_sp_jacobi_persistent(d_layers, d_pairs + first, (int)(last - first), row_floats_max, max_sweeps,
                                                ctx->tol, d_flag + 2, st);
      if (e != 0) return fail_cuda(ctx, (cudaError_t)e, "cudaLaunchCooperativeKernel(jacobi)");
      ++n_eig_launch;
      first = last;
    }
    launch_sp_check(d_layers, n_layers, t_max, max_sweeps, d_flag, st);
    ++n_eig_launch;
    CK(cudaMemcpyAsync(ctx->h_flag, d_flag, 4 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    flags_pending = true;                                  // read at the end of the call, after everything is enqueued
  } else
  for (int it = 0; it < max_sweeps; ++it) {
    for (int j = 0; j < steps_max; ++j, ++t_done, ++n_eig_launch)
      launch_sp_jacobi_step(d_layers, d_pairs, (int)block_pairs.size(), row_floats_max, t_done, max_sweeps, ctx->tol, st);
    launch_sp_check(d_layers, n_layers, t_done, max_sweeps, d_flag, st);
    CK(cudaMemcpyAsync(ctx->h_flag, d_flag, 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (ctx->h_flag[1] != 0) { ctx->err = "a bounded wait in the tensor-core Gram kernel ran out"; return ATOMO_ERR_TIMEOUT; }
    if (ctx->h_flag[0]) break;
  }
  stage_end(ctx, ATOMO_STAGE_EIG, st, n_eig_launch);

  // ---- S2-S4: (refined singular values,) probabilities, draws, compaction ----
  stage_begin(ctx, ATOMO_STAGE_SAMPLE, st);
  if (tri_form) {                                                   // all eigenvalues of the tridiagonal matrices
    int64_t n_eig = 0;
    for (int l = 0; l < n_layers; ++l) n_eig += L[l].r;
    launch_sp_bisect(d_layers, n_layers, r_max, n_eig, st);
  }
  launch_sp_refine(d_layers, n_layers, d_ref, (int)refine_tiles.size(), st);
  const PhiloxKey key{(uint32_t)seed, (uint32_t)(seed >> 32)};
  launch_sp_finalize_sample(d_layers, n_layers, s, key, kind_step_word(ATOMO_KIND_SPECTRAL, step), max_sweeps,
                            tri_form ? d_flag + 1 : nullptr, st);
  stage_end(ctx, ATOMO_STAGE_SAMPLE, st, tri_form ? 2 : 1);

  // ---- S4: long-side vectors of the kept atoms ----
  stage_begin(ctx, ATOMO_STAGE_BACKPROJECT, st);
  if (tri_form) {                                                   // short-side vectors of the kept atoms
    if (any_small && any_big) {                                     // both kinds side by side, as their reductions
      CK(cudaEventRecord(ctx->ev_fork, st));
      CK(cudaStreamWaitEvent(side, ctx->ev_fork, 0));
      launch_sp_eigvec(d_layers, n_layers, rp_max_small, side);
      CK(cudaEventRecord(ctx->ev_join, side));
    } else if (any_small) launch_sp_eigvec(d_layers, n_layers, rp_max_small, st);
    int rps = 0;
    for (int l : big_layers) rps |= L[l].rp <= 1024 ? 1 : L[l].rp <= 2048 ? 2 : 4;
    launch_sp_eigvec_big(d_layers, d_big, (int)big_layers.size(), rps, s, st);
    if (any_small && any_big) CK(cudaStreamWaitEvent(st, ctx->ev_join, 0));
  }
  launch_sp_backproject(d_layers, d_bp, (int)bp_tiles.size(), std::max(r_max_tall, 1), st);
  launch_sp_finish_atoms(d_layers, n_layers, k_cap_max, st);
  stage_end(ctx, ATOMO_STAGE_BACKPROJECT, st, tri_form ? 2 + (any_small ? 1 : 0) + (any_big ? 1 : 0) : 2);
  CK(cudaGetLastError());
  if (flags_pending) {
    // the one host wait of the persistent forms: the kernels' bounded waits report here
    CK(cudaStreamSynchronize(st));
    if (ctx->h_flag[1] != 0) { ctx->err = "a bounded wait in the tensor-core Gram kernel ran out"; return ATOMO_ERR_TIMEOUT; }
    if (ctx->h_flag[2] != 0) { ctx->err = "a step barrier of the persistent eigen-solve ran out of polls"; return ATOMO_ERR_TIMEOUT; }
  }
  return ATOMO_OK;
}

static int encode_spectral_impl(atomo_ctx* ctx, const atomo_mat* layers, int32_t n_layers, double s, uint64_t seed,
                                uint64_t step, int32_t k_cap, void* payload, int64_t capacity_bytes,
                                const atomo_debug* dbg, void* stream, const float* const* given_sigma,
                                const float* const* given_short) {
  bool use_digits = true;
  const int rc = encode_spectral_with(ctx, layers, n_layers, s, seed, step, k_cap, payload, capacity_bytes, dbg, stream, given_sigma, given_short, use_digits);
  if (use_digits) return rc;
  // beside a nearly full GPU: the Gram kernels that need no digits
  return encode_spectral_with(ctx, layers, n_layers, s, seed, step, k_cap, payload, capacity_bytes, dbg, stream, given_sigma, given_short, use_digits);
}

int atomo_encode_spectral(atomo_ctx* ctx, const atomo_mat* layers, int32_t n_layers, double s, uint64_t seed,
                          uint64_t step, int32_t k_cap, void* payload, int64_t capacity_bytes,
                          const atomo_debug* dbg, void* stream) {
  return encode_spectral_impl(ctx, layers, n_layers, s, seed, step, k_cap, payload, capacity_bytes, dbg, stream, nullptr, nullptr);
}

int atomo_encode_spectral_from_svd(atomo_ctx* ctx, const atomo_mat* layers, int32_t n_layers,
                                   const float* const* sigma, const float* const* short_vecs, double s, uint64_t seed,
                                   uint64_t step, int32_t k_cap, void* payload, int64_t capacity_bytes,
                                   const atomo_debug* dbg, void* stream) {
  if (!sigma || !short_vecs || n_layers <= 0) return ATOMO_ERR_INVALID_ARG;
  for (int l = 0; l < n_layers; ++l) if (!sigma[l] || !short_vecs[l]) return ATOMO_ERR_INVALID_ARG;
  return encode_spectral_impl(ctx, layers, n_layers, s, seed, step, k_cap, payload, capacity_bytes, dbg, stream, sigma, short_vecs);
}

// ==================================================================================================
int atomo_encode_entrywise(atomo_ctx* ctx, const atomo_vec* vecs, int32_t n_vecs, double s, uint64_t seed,
                           uint64_t step, int64_t k_cap, void* payload, int64_t capacity_bytes,
                           const atomo_debug* dbg, void* stream) {
  if (!ctx || !vecs || n_vecs <= 0 || k_cap <= 0 || !payload) return ATOMO_ERR_INVALID_ARG;
  if (bad_budget(s)) return ATOMO_ERR_BUDGET;
  if ((reinterpret_cast<uintptr_t>(payload) & 15u) != 0) return ATOMO_ERR_INVALID_ARG;
  std::vector<int64_t> ns(n_vecs);
  for (int l = 0; l < n_vecs; ++l) {
    if (!vecs[l].data || vecs[l].n <= 0 || vecs[l].n >= (int64_t(1) << 32)) return ATOMO_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(vecs[l].data) & 3u) != 0) return ATOMO_ERR_INVALID_ARG;
    ns[l] = vecs[l].n;
  }
  std::vector<EwLayout> lay;
  const bool compact = ctx->ew_format == ATOMO_EW_COMPACT;
  const uint64_t total = layout_entrywise(ns.data(), n_vecs, k_cap, compact, ctx->ew_sat_cap, &lay);
  if ((int64_t)total > capacity_bytes) return ATOMO_ERR_CAPACITY;
  CK(cudaSetDevice(ctx->device));
  cudaStream_t st = (cudaStream_t)stream;
  stage_reset(ctx);
  uint8_t* pay = static_cast<uint8_t*>(payload);
  atomo_layer_header* d_hdr = reinterpret_cast<atomo_layer_header*>(pay + sizeof(atomo_payload_header));
  const int tile = ew_tile_elems();

  // Launches: runs of consecutive vectors (at most kEwBatch, their chunks one wave of resident CTAs) go through one
  // launch of the one-kernel form; a vector too long for that takes the two-kernel form on its own.
  struct Run { int first, count, solve_ctas; bool list; };       // solve_ctas > 0: two-kernel form
  std::vector<Run> runs;
  std::vector<EwVec> V(n_vecs);
  const bool want_list = ctx->ew_launch == 0 && !(dbg && dbg->prob);   // asking for the probabilities means a second read
  for (int l = 0; l < n_vecs; ++l) {
    EwVec& v = V[l];
    v = EwVec{};
    v.g = vecs[l].data; v.n = vecs[l].n; v.n_tiles = (v.n + tile - 1) / tile;
    v.pay = pay; v.hdr = d_hdr + l;
    v.off_idx = lay[l].off_idx; v.off_val = lay[l].off_val; v.off_tiles = lay[l].off_tiles; v.off_sat = lay[l].off_sat;
    v.layer = (uint32_t)l; v.k_cap = lay[l].kc; v.sat_cap = lay[l].sc; v.compact = compact ? 1 : 0;
  }
  auto two_kernels = [&](int l) {
    const int ctas = ew_solve_ctas(V[l].n_tiles);
    V[l].n_ctas = std::max(ctas, ew_pack_ctas(V[l].n_tiles));    // what the workspace has to hold
    V[l].candidates = 0;
    return ctas;
  };
  for (int l = 0; l < n_vecs;) {
    int count = ctx->ew_launch == 1 ? 0 : std::min(n_vecs - l, kEwBatch);
    bool list = want_list;
    for (; count > 0; --count) {
      if (list && ew_plan(&V[l], count, true) > 0) break;
      if (ew_plan(&V[l], count, false) > 0) { list = false; break; }   // longer chunks fit without the list's slots
    }
    if (count == 0) {
      const int ctas = two_kernels(l);
      if (ctas <= 0) return fail_cuda(ctx, cudaGetLastError(), "occupancy query for the cooperative solve");
      runs.push_back({l, 1, ctas, false});
      ++l;
      continue;
    }
    if (list) {
      list = false;
      for (int i = l; i < l + count; ++i) {
        V[i].candidates = V[i].n_tiles > V[i].n_ctas && ew_list_pays(V[i].n, V[i].n_tiles, V[i].n_ctas, s) ? 1 : 0;
        list |= V[i].candidates != 0;
      }
      if (!list && ew_plan(&V[l], count, false) == 0) return fail_cuda(ctx, cudaErrorInvalidConfiguration, "entry-wise launch plan");
    }
    runs.push_back({l, count, 0, list});
    l += count;
  }
  for (int pass = 0; pass < 2; ++pass) {
    Arena A(pass ? ctx->ws : nullptr);
    size_t dbg_atoms = 0, dbg_words = 0;
    for (int l = 0; l < n_vecs; ++l) {
      EwVec& v = V[l];
      const int64_t n_words = (v.n + 31) / 32;
      const bool want_mask = dbg && dbg->mask_words;           // the mask words leave the kernel only when asked for
      v.n_words = want_mask ? n_words : 0;
      v.mask_words = want_mask ? dbg->mask_words + dbg_words : nullptr;
      v.prob_out = (dbg && dbg->prob) ? dbg->prob + dbg_atoms : nullptr;
      dbg_atoms += v.n; dbg_words += n_words;
      v.partials = A.take<EwPartial>((size_t)3 * v.n_ctas);
      v.state = A.take<EwState>(1);
      v.chunk_status = A.take<uint64_t>((size_t)std::max(v.n_ctas, ew_pack_ctas(v.n_tiles)));
      v.ticket = A.take<uint32_t>(1);
    }
    if (pass == 0) { const int rc = ensure_ws(ctx, A.off + 256); if (rc != ATOMO_OK) return rc; }
  }

  EwBegin begin{};
  begin.on = 1;
  atomo_payload_header& gh = begin.gh;
  gh.magic = ATOMO_MAGIC; gh.version = ATOMO_VERSION; gh.kind = ATOMO_KIND_ENTRYWISE; gh.n_layers = (uint32_t)n_vecs;
  gh.total_bytes = total; gh.seed = seed; gh.step = step; gh.s = s;
  gh.ew_format = (uint64_t)ctx->ew_format; gh.ew_sat_cap = compact ? (uint64_t)ctx->ew_sat_cap : 0;
  auto fill = [&](auto& B, int first, int count) {
    for (int i = 0; i < count; ++i) { B.v[i] = V[first + i]; B.v[i].barrier = ctx->ew_words + i * kEwBarrierStride; }
    B.n = count; B.s = s; B.key = philox_round_keys(PhiloxKey{(uint32_t)seed, (uint32_t)(seed >> 32)});
    B.kind_step = kind_step_word(ATOMO_KIND_ENTRYWISE, step);
    B.begin = begin; B.begin.on = first == 0 ? 1 : 0;
  };
  auto solve = [&](int l, int solve_ctas) {
    EwBatch<1> B{};
    fill(B, l, 1);
    return launch_ew_solve(B, solve_ctas, ew_pack_ctas(V[l].n_tiles), st);
  };
  auto sample_pack = [&](int l) {
    EwBatch<1> B{};
    fill(B, l, 1);
    return launch_ew_sample_pack(B, ew_pack_ctas(V[l].n_tiles), st);
  };
  ctx->ew_last_state.resize(n_vecs); ctx->ew_last_chunks.resize(n_vecs);
  for (int l = 0; l < n_vecs; ++l) { ctx->ew_last_state[l] = V[l].state; ctx->ew_last_chunks[l] = V[l].n_ctas; }
  // the probabilities of the vectors that take two kernels are a stage of their own; all other encoding is timed as packing
  int64_t n_launch = 0, n_solve = 0;
  for (const Run& r : runs) n_solve += r.solve_ctas > 0 ? 1 : 0;
  if (n_solve > 0) {
    stage_begin(ctx, ATOMO_STAGE_EW_REDUCE, st);
    for (const Run& r : runs) {
      if (r.solve_ctas == 0) continue;
      const int e = solve(r.first, r.solve_ctas);
      if (e != 0) return fail_cuda(ctx, (cudaError_t)e, "cudaLaunchCooperativeKernel(entry-wise solve)");
      ctx->ew_last_chunks[r.first] = 0;
    }
    stage_end(ctx, ATOMO_STAGE_EW_REDUCE, st, n_solve);
  }
  stage_begin(ctx, ATOMO_STAGE_EW_PACK, st);
  for (const Run& r : runs) {
    int e = 0;
    if (r.solve_ctas > 0) {
      e = sample_pack(r.first);
      ++n_launch;
    } else {
      if (r.count == 1) { EwBatch<1> B{}; fill(B, r.first, 1); e = launch_ew_encode(B, r.list, st); }
      else { EwBatch<kEwBatch> B{}; fill(B, r.first, r.count); e = launch_ew_encode(B, r.list, st); }
      ++n_launch;
      if (e == (int)cudaErrorCooperativeLaunchTooLarge) {
        // fewer CTAs fit the GPU at once than the occupancy query promised: the two-kernel form, vector by vector
        cudaGetLastError();
        e = 0;
        for (int l = r.first; l < r.first + r.count && e == 0; ++l) {
          V[l].candidates = 0;
          const int ctas = std::min(ew_solve_ctas(V[l].n_tiles), V[l].n_ctas);   // the workspace was carved for that many
          e = ctas > 0 ? solve(l, ctas) : (int)cudaErrorCooperativeLaunchTooLarge;
          if (e == 0) e = sample_pack(l);
          ctx->ew_last_chunks[l] = 0;
          n_launch += 2;
        }
      }
    }
    if (e != 0) return fail_cuda(ctx, (cudaError_t)e, "launch of the entry-wise encode");
  }
  stage_end(ctx, ATOMO_STAGE_EW_PACK, st, n_launch);
  CK(cudaGetLastError());
  return ATOMO_OK;
}

int atomo_get_entrywise_list_chunks(atomo_ctx* ctx, int32_t vec, uint32_t* from_list, uint32_t* chunks) {
  if (!ctx || vec < 0 || vec >= (int32_t)ctx->ew_last_state.size()) return ATOMO_ERR_INVALID_ARG;
  CK(cudaSetDevice(ctx->device));
  CK(cudaDeviceSynchronize());
  uint32_t n = 0;
  if (ctx->ew_last_chunks[vec] > 0)
    CK(cudaMemcpy(&n, &ctx->ew_last_state[vec]->list_chunks, sizeof(n), cudaMemcpyDeviceToHost));
  if (from_list) *from_list = n;
  if (chunks) *chunks = (uint32_t)ctx->ew_last_chunks[vec];
  return ATOMO_OK;
}

// ==================================================================================================
int atomo_set_entrywise_launch(atomo_ctx* ctx, int32_t two_kernels) {
  if (!ctx || two_kernels < 0 || two_kernels > 2) return ATOMO_ERR_INVALID_ARG;
  ctx->ew_launch = two_kernels;
  return ATOMO_OK;
}

int atomo_lq_budget(atomo_ctx* ctx, const atomo_vec* vecs, int32_t n_vecs, double q, double* s_out, void* stream) {
  if (!ctx || !vecs || n_vecs <= 0 || !s_out || !(q >= 1.0)) return ATOMO_ERR_INVALID_ARG;
  for (int l = 0; l < n_vecs; ++l) {
    if (!vecs[l].data || vecs[l].n <= 0) return ATOMO_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(vecs[l].data) & 3u) != 0) return ATOMO_ERR_INVALID_ARG;
  }
  CK(cudaSetDevice(ctx->device));
  cudaStream_t st = (cudaStream_t)stream;
  const int max_ctas = 148 * 8;
  EwLqPart* d_part = nullptr;
  for (int pass = 0; pass < 2; ++pass) {
    Arena A(pass ? ctx->ws : nullptr);
    d_part = A.take<EwLqPart>(max_ctas);
    if (pass == 0) { const int rc = ensure_ws(ctx, A.off + 256); if (rc != ATOMO_OK) return rc; }
  }
  uint32_t* const ticket = ctx->ew_words + kEwBarrierWords;
  // the sums of up to kLqResults vectors arrive in pinned memory; one wait for all of them
  for (int l0 = 0; l0 < n_vecs; l0 += kLqResults) {
    const int n = std::min(n_vecs - l0, kLqResults);
    for (int i = 0; i < n; ++i) launch_ew_lq(vecs[l0 + i].data, vecs[l0 + i].n, 0, q, 0.0, d_part, ticket, ctx->h_lq + i, max_ctas, st);
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(st));
    bool more = false;
    std::vector<double> l1(n), amax(n);
    for (int i = 0; i < n; ++i) {
      const EwLqPart r = ctx->h_lq[i];
      l1[i] = r.sum; amax[i] = r.amax;
      double& out = s_out[l0 + i];
      if (!(r.amax <= 3.0e38) || !(r.sum == r.sum)) { out = std::nan(""); l1[i] = -1.0; }
      else if (r.amax == 0.0) { out = 0.0; l1[i] = -1.0; }
      else if (std::isinf(q)) out = r.sum / r.amax;
      else if (q == 1.0) out = 1.0;
      else if (q == 2.0) out = r.sum / std::sqrt(r.sq);
      else { launch_ew_lq(vecs[l0 + i].data, vecs[l0 + i].n, 1, q, 1.0 / r.amax, d_part, ticket, ctx->h_lq + i, max_ctas, st); more = true; continue; }
      l1[i] = -1.0;
    }
    if (!more) continue;
    CK(cudaGetLastError());
    CK(cudaStreamSynchronize(st));
    for (int i = 0; i < n; ++i)
      if (l1[i] >= 0.0) s_out[l0 + i] = l1[i] / (amax[i] * std::pow(ctx->h_lq[i].sum, 1.0 / q));
  }
  return ATOMO_OK;
}

// ==================================================================================================
int atomo_decode(atomo_ctx* ctx, int32_t kind, const void* payload, const int64_t* rows, const int64_t* cols,
                 float* const* out, int32_t n_layers, void* stream) {
  if (!ctx || !payload || !rows || !cols || !out || n_layers <= 0) return ATOMO_ERR_INVALID_ARG;
  if (kind != ATOMO_KIND_SPECTRAL && kind != ATOMO_KIND_ENTRYWISE) return ATOMO_ERR_INVALID_ARG;
  for (int l = 0; l < n_layers; ++l) if (!out[l] || rows[l] <= 0 || cols[l] <= 0) return ATOMO_ERR_INVALID_ARG;
  CK(cudaSetDevice(ctx->device));
  cudaStream_t st = (cudaStream_t)stream;
  stage_reset(ctx);
  const uint8_t* pay = static_cast<const uint8_t*>(payload);
  stage_begin(ctx, ATOMO_STAGE_DECODE, st);
  if (kind == ATOMO_KIND_ENTRYWISE) {
    for (int l = 0; l < n_layers; ++l) if (rows[l] != 1) return ATOMO_ERR_INVALID_ARG;
    const int n_launch = for_each_ew_decode(pay, cols, out, n_layers, [&](const auto& B, uint32_t tiles) { launch_ew_decode(B, tiles, st); });
    stage_end(ctx, ATOMO_STAGE_DECODE, st, n_launch);
  } else {
    ++ctx->table_reuses;                                           // counted as a call with nothing to upload: the layers travel as kernel arguments
    const int n_launch = launch_sp_decode(pay, nullptr, 1, rows, cols, out, n_layers, st);
    stage_end(ctx, ATOMO_STAGE_DECODE, st, n_launch);
  }
  CK(cudaGetLastError());
  return ATOMO_OK;
}

// ==================================================================================================
int atomo_decode_average(atomo_ctx* ctx, int32_t kind, const void* const* payloads, int32_t n_payloads,
                         const int64_t* rows, const int64_t* cols, float* const* out, int32_t n_layers, void* stream) {
  if (!ctx || !payloads || n_payloads <= 0 || !rows || !cols || !out || n_layers <= 0) return ATOMO_ERR_INVALID_ARG;
  if (kind != ATOMO_KIND_SPECTRAL && kind != ATOMO_KIND_ENTRYWISE) return ATOMO_ERR_INVALID_ARG;
  for (int p = 0; p < n_payloads; ++p) if (!payloads[p]) return ATOMO_ERR_INVALID_ARG;
  for (int l = 0; l < n_layers; ++l) {
    if (!out[l] || rows[l] <= 0 || cols[l] <= 0) return ATOMO_ERR_INVALID_ARG;
    if (kind == ATOMO_KIND_ENTRYWISE && rows[l] != 1) return ATOMO_ERR_INVALID_ARG;
  }
  CK(cudaSetDevice(ctx->device));
  cudaStream_t st = (cudaStream_t)stream;
  stage_reset(ctx);
  const uint8_t** d_pay = nullptr;
  size_t tb = 0;
  TableCache& tab = table_pick(ctx->tab_avg, table_key(kKeySeed, payloads, (size_t)n_payloads * sizeof(void*)));
  for (int pass = 0; pass < 2; ++pass) {
    Arena T(pass ? tab.d : nullptr);
    d_pay = T.take<const uint8_t*>(n_payloads);
    tb = T.off + 256;
    if (pass == 0) { const int rc = table_reserve(ctx, tab, tb); if (rc != ATOMO_OK) return rc; }
  }
  {
    std::vector<uint8_t> tables(tb, 0);
    std::memcpy(tables.data() + (reinterpret_cast<uint8_t*>(d_pay) - tab.d), payloads, (size_t)n_payloads * sizeof(void*));
    const int rc = table_commit(ctx, tab, tables.data(), tb, st);
    if (rc != ATOMO_OK) return rc;
  }
  stage_begin(ctx, ATOMO_STAGE_DECODE, st);
  if (kind == ATOMO_KIND_SPECTRAL) {
    const int n_launch = launch_sp_decode(nullptr, d_pay, n_payloads, rows, cols, out, n_layers, st);
    stage_end(ctx, ATOMO_STAGE_DECODE, st, n_launch);
  } else {
    const int n_launch = for_each_ew_decode(nullptr, cols, out, n_layers, [&](const auto& B, uint32_t n_tiles) {
      launch_ew_decode_average(B, n_tiles, d_pay, n_payloads, st);
    });
    stage_end(ctx, ATOMO_STAGE_DECODE, st, n_launch);
  }
  CK(cudaGetLastError());
  return ATOMO_OK;
}

// ==================================================================================================
int atomo_payload_read_headers(atomo_ctx* ctx, const void* payload, int32_t n_layers, atomo_payload_header* hdr,
                               atomo_layer_header* layers, void* stream) {
  if (!ctx || !payload || n_layers <= 0) return ATOMO_ERR_INVALID_ARG;
  CK(cudaSetDevice(ctx->device));
  cudaStream_t st = (cudaStream_t)stream;
  const uint8_t* pay = static_cast<const uint8_t*>(payload);
  if (hdr) CK(cudaMemcpyAsync(hdr, pay, sizeof(*hdr), cudaMemcpyDeviceToHost, st));
  if (layers)
    CK(cudaMemcpyAsync(layers, pay + sizeof(atomo_payload_header), (size_t)n_layers * sizeof(atomo_layer_header),
                       cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  return ATOMO_OK;
}

int atomo_payload_status(atomo_ctx* ctx, const void* payload, int32_t n_layers, int32_t* worst, int32_t* first_bad_layer,
                         void* stream) {
  if (!ctx || !payload || n_layers <= 0) return ATOMO_ERR_INVALID_ARG;
  std::vector<atomo_layer_header> h(n_layers);
  const int rc = atomo_payload_read_headers(ctx, payload, n_layers, nullptr, h.data(), stream);
  if (rc != ATOMO_OK) return rc;
  int32_t w = ATOMO_OK, first = -1;
  for (int l = 0; l < n_layers; ++l)
    if (h[l].status != ATOMO_OK && first < 0) { w = (int32_t)h[l].status; first = l; }
  if (worst) *worst = w;
  if (first_bad_layer) *first_bad_layer = first;
  return ATOMO_OK;
}

}  // extern "C"
