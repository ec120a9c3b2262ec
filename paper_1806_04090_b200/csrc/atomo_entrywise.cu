// Entry-wise ATOMO on flat gradients: atoms e_i, lambda_i = g_i (Section 3 of the paper; the
// QSGD / TernGrad family of Section 4 are the budgets s = ||g||_1/||g||_2 and ||g||_1/||g||_inf).
//
//   ew_encode (cooperative)    : all vectors of a call (up to kEwBatch) in one launch; a CTA owns a chunk of consecutive
//                                tiles of one vector.
//     pass 1                     ||g||_1 (fp64 accumulation), ||g||_inf, non-finite scan; then the water-filling form
//                                of Algorithm 1 -- every atom with |g_i| (s - n_s) > sum_{unsaturated} |g_j| gets
//                                p = 1; repeated until no new atom saturates (zero rounds when g is s-balanced,
//                                Lemma 3).  The CTAs of a vector meet at a barrier of their own.
//     pass 2                     p_i = |g_i| (s-n_s)/T, Philox word, keep decision -> code bytes in shared memory; the
//                                counts of the earlier chunks are added (one bounded wait, no chain); ordered
//                                compaction from the code bytes: idx ascending, val = g_i / p_i; the last chunk writes
//                                k, the capacity check and the header.  Compact format (the ternary form of Section 4):
//                                a kept atom with p < 1 weighs sign(g_i) c, so it travels as a 16-bit entry (index
//                                inside its tile, sign bit); the atoms with p = 1 keep (idx, val) in a list of their own
//   ew_solve + ew_sample_pack  : the same two passes as two kernels, for vectors whose code bytes do not fit the shared
//                                memory of one wave of resident CTAs
//   ew_decode                  : a tile is put together in shared memory and leaves as one bulk copy, either format
#include <algorithm>
#include <type_traits>

#include "atomo_kernels.cuh"

namespace atomo {

namespace {

// One CTA per SM: the warps of an SM share one chunk.  (Four CTAs of 256 threads with a chunk each took as long as the
// slowest of them: the scheduler favours the oldest warps, so that of four equal chunks on an SM the first was done after 104 us
// and the last, by then alone with eight warps, after 200.)
constexpr int kEwThreads = 1024;
constexpr int kEwWarps = kEwThreads / kWarp;
constexpr int kEwTile = ATOMO_EW_TILE;        // elements per tile
constexpr int kEwUnits = 8;                   // units per tile: what a warp takes at a time, 16 atoms per lane
// The keep decisions of a block of four atoms (one Philox call) are a byte: K_j in bit j, S_j in bit 4 + j.
// (K, S) = (1, sign bit of g): kept with p < 1; (0, 1): kept with p = 1 (saturated); (0, 0): not kept.
constexpr int kEwBlocks = kEwTile / 4;        // blocks (code bytes) per tile
constexpr int kEwPrefixes = kEwTile / 32;     // list form: prefix words per tile
constexpr int kEwRegTiles = kEwWarps / kEwUnits;   // chunks of at most this many tiles stay in registers: a unit per warp
constexpr int kEwBig = 8;                     // a thread's entries of the list of runs with atoms that may saturate
constexpr int kEwStage = 256;                 // kept atoms per staging window (one per warp) of the compaction
constexpr uint32_t kEwPollLimit = 1u << 22;   // polls of a bounded wait (with a sleep between them)
constexpr uint64_t kFlagReady = 1ull << 63;

__device__ __forceinline__ float4 load4(const float* __restrict__ g, int64_t i, int64_t n, bool aligned) {
  if (aligned && i + 3 < n) return __ldg(reinterpret_cast<const float4*>(g + i));
  float4 v;
  v.x = (i + 0 < n) ? __ldg(g + i + 0) : 0.0f;
  v.y = (i + 1 < n) ? __ldg(g + i + 1) : 0.0f;
  v.z = (i + 2 < n) ? __ldg(g + i + 2) : 0.0f;
  v.w = (i + 3 < n) ? __ldg(g + i + 3) : 0.0f;
  return v;
}

// The chunk of a CTA: n_my tiles of the vector from tile0 on, elements [beg, end)
struct EwChunk {
  int64_t tile0, beg, end;
  int n_my, n_full, n_units;    // n_full: tiles that lie inside the vector and can be read with 16-byte loads
  uint32_t index;               // position among the vector's chunks
  bool aligned;
};
__device__ __forceinline__ EwChunk ew_chunk(const EwVec& v, uint32_t index) {
  EwChunk c;
  const int64_t q = v.n_tiles / v.n_ctas, rem = v.n_tiles % v.n_ctas;    // the first `rem` chunks have q + 1 tiles
  c.index = index;
  c.tile0 = (int64_t)index * q + min((int64_t)index, rem);
  c.n_my = (int)(q + ((int64_t)index < rem ? 1 : 0));
  c.beg = c.tile0 * kEwTile;
  c.end = min(v.n, c.beg + (int64_t)c.n_my * kEwTile);
  c.aligned = (reinterpret_cast<uintptr_t>(v.g) & 15u) == 0;
  c.n_full = c.aligned ? (int)((c.end - c.beg) / kEwTile) : 0;
  c.n_units = c.n_my * kEwUnits;
  return c;
}
// number of a lane's first float4 of a unit inside the chunk; its other three are 256 apart
__device__ __forceinline__ uint32_t ew_unit_block(int unit) {
  return (uint32_t)(unit / kEwUnits) * kEwBlocks + (uint32_t)(unit % kEwUnits) * kWarp + threadIdx.x % kWarp;
}
// float4 number u = 0 .. 3 of a lane's 16 atoms of a unit; zeros past the end
__device__ __forceinline__ float4 ew_load_unit(const EwVec& v, const EwChunk& c, int unit, int u) {
  const int64_t i = c.beg + 4 * (int64_t)ew_unit_block(unit) + 1024 * u;
  if (unit / kEwUnits < c.n_full) return __ldg(reinterpret_cast<const float4*>(v.g + i));
  return i < c.end ? load4(v.g, i, c.end, c.aligned) : make_float4(0.f, 0.f, 0.f, 0.f);
}
__device__ __forceinline__ void ew_load_unit(const EwVec& v, const EwChunk& c, int unit, float4 (&x)[4]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) x[u] = unit >= 0 && unit < c.n_units ? ew_load_unit(v, c, unit, u) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// f(blk, x) for the four blocks (blk: number inside the chunk) and end(blk) with the first one's for every unit of the chunk,
// each warp its own in ascending order.  kAhead units' loads are on their way: a float4's registers are loaded again as soon
// as it has been used.  Two where the work per unit is small and the pass is bound by HBM; one where it is bound by
// instruction issue (a second set of registers spilled), and there a barrier every few rounds keeps the warps abreast: left
// alone the oldest ones run ahead and the last ones end alone.
template <int kAhead, typename F, typename E>
__device__ __forceinline__ void ew_for_units(const EwVec& v, const EwChunk& c, float4 (&x)[kAhead][4], F f, E end) {
  constexpr int kStep = kEwWarps / kEwUnits * kEwBlocks;   // blocks from a warp's unit to its next
  const int n = c.n_units, n_full = c.n_full * kEwUnits;
  int unit = (int)(threadIdx.x / kWarp);
  uint32_t blk = ew_unit_block(unit);
  const float4* src = reinterpret_cast<const float4*>(v.g + c.beg) + blk + kAhead * kStep;
  for (int u0 = 0, round = 0; u0 < n; u0 += kAhead * kEwWarps, ++round) {
#pragma unroll
    for (int h = 0; h < kAhead; ++h) {
      if (unit < n) {
        const int next = unit + kAhead * kEwWarps;
        if (next < n_full) {
#pragma unroll
          for (int u = 0; u < 4; ++u) { f(blk + (uint32_t)(256 * u), x[h][u]); x[h][u] = __ldg(src + 256 * u); }
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u) { f(blk + (uint32_t)(256 * u), x[h][u]); if (next < n) x[h][u] = ew_load_unit(v, c, next, u); }
        }
        end(blk);
      }
      unit += kEwWarps; blk += kStep; src += kStep;
    }
    if (kAhead == 1 && (round & 3) == 3) __syncthreads();
  }
}
template <int kAhead>
__device__ __forceinline__ void ew_load_ahead(const EwVec& v, const EwChunk& c, float4 (&x)[kAhead][4]) {
#pragma unroll
  for (int h = 0; h < kAhead; ++h) ew_load_unit(v, c, (int)(threadIdx.x / kWarp) + h * kEwWarps, x[h]);
}

struct EwAcc { double sum; float amax; uint32_t cnt; };

struct EwShared {                 // static shared memory of the encode and solve kernels
  double sum[kEwWarps];
  float mx[kEwWarps], est[kEwWarps];
  uint32_t cnt[kEwWarps];
  unsigned long long scan[kEwWarps], before[kEwWarps];
  uint32_t big[kEwWarps];       // runs on the warps' lists, closed up
  uint32_t big_over, stop, fail, next_unit;
};

// block reduction in a fixed order, result valid in every thread
__device__ __forceinline__ EwAcc ew_block_reduce(EwAcc a, EwShared& sh) {
  const int w = threadIdx.x / kWarp, l = threadIdx.x % kWarp;
  a.sum = warp_sum(a.sum); a.amax = warp_max(a.amax); a.cnt = __reduce_add_sync(0xffffffffu, a.cnt);
  __syncthreads();
  if (l == 0) { sh.sum[w] = a.sum; sh.mx[w] = a.amax; sh.cnt[w] = a.cnt; }
  __syncthreads();
  return EwAcc{warp_sum(sh.sum[l]), warp_max(sh.mx[l]), __reduce_add_sync(0xffffffffu, sh.cnt[l])};
}
// sum of one float per thread, valid in every thread
__device__ __forceinline__ float ew_block_sum(float x, EwShared& sh) {
  x = warp_sum(x);
  if (threadIdx.x % kWarp == 0) sh.est[threadIdx.x / kWarp] = x;
  __syncthreads();
  return warp_sum(sh.est[threadIdx.x % kWarp]);
}

// Barrier among the CTAs of one vector (all resident: cooperative launch).  `target` is the number of arrivals since
// the counter was zeroed; the wait is bounded and a wait that runs out is reported in the layer's status word.
__device__ __forceinline__ void ew_barrier(const EwVec& v, uint32_t target, EwShared& sh) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(v.barrier, 1u);
    uint32_t polls = 0;
    while (*(volatile uint32_t*)v.barrier < target) {
      if (++polls > kEwPollLimit) { sh.fail = 1u; break; }
      __nanosleep(20);
    }
    __threadfence();
  }
  __syncthreads();
}
// ---- pass 1 -------------------------------------------------------------------------------------------------------
// Sums in short fp32 runs (16 terms per lane and unit), then fp64.  amax ignores NaN (and the sum keeps it), so "some
// entry is NaN" is "the sum is NaN" and "some entry is infinite" is "amax is infinite": no test per entry.
__device__ __forceinline__ float max4(const float4& x) {
  return fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w)));
}
__device__ __forceinline__ void ew_sums(const float4& x, float& fsum, float& amax) {
  fsum += fabsf(x.x); fsum += fabsf(x.y); fsum += fabsf(x.z); fsum += fabsf(x.w);
  amax = fmaxf(amax, max4(x));
}
// the warps' first units (x): sum of |g| over them, scaled to the vector
__device__ __forceinline__ double ew_estimate_l1(const EwVec& v, const EwChunk& c, const float4 (&x)[4], EwShared& sh) {
  float ts = 0.0f, m = 0.0f;
#pragma unroll
  for (int u = 0; u < 4; ++u) ew_sums(x[u], ts, m);
  ts = ew_block_sum(ts, sh);
  const double seen = (double)min((int64_t)kEwRegTiles * kEwTile, c.end - c.beg);
  return (double)ts * (double)v.n / seen;
}
// Runs (a lane's 16 atoms of a unit) with an atom above a lower bound of the saturation threshold, listed during pass 1 so
// that the water-filling rounds read those alone and not the whole vector (a round over 100 million elements costs 65 us,
// the listed runs of 100 M Laplace entries at s = 10 % are 0.5 % of it).  The bound is 0.8 l1_est / s with l1_est the sum over
// the chunk's first tiles scaled to the vector; the rounds lower the threshold a little (there: by half a per cent).  A round
// forms the listed runs anew without the saturated atoms, exactly as a round over the whole chunk would.
// Every thread lists its own runs in slots of its own and the warps close them up before the first round, so that the sums have a
// fixed order; a thread without a slot left sends the rounds to memory (a chunk of up to 32 tiles has a slot for every run).
// (One list of the CTA, filled through an atomic counter and dealt to the threads by position, gave fp64 sums that depended on
// which warp came first.  25 M elements at 13 %: 94.6 us with it, 96.9 so, 99.0 where a round goes through a thread's own slots; a
// list per warp, placed by ballot, doubled the spills of this pass: 100 M elements at 10 % 341 -> 358 us, so 342.)
constexpr uint32_t kEwClosed = 0xFFFFFFFFu;
struct EwBigList {
  uint32_t* run;                // [kEwBig][kEwThreads] the runs' first blocks inside the chunk, shared memory
  uint32_t n;                   // this thread's; kEwClosed: closed up
  float lo;                     // runs with an atom above lo are listed; inf: no list
  double rest;                  // this thread's sum over the runs not listed
};

// pass 1 with that list; the caller has zeroed sh.big_over
__device__ __forceinline__ EwAcc ew_pass_big(const EwVec& v, const EwChunk& c, const double s, EwBigList& B, EwShared& sh) {
  double sum = 0.0, rest = 0.0;
  float amax = 0.0f;
  uint32_t at = threadIdx.x;
  float4 x[2][4];
  ew_load_ahead(v, c, x);
  {
    const float lo = (float)(0.8 * ew_estimate_l1(v, c, x[0], sh) / s);
    // a zero or non-finite estimate, or a budget that keeps every atom (threshold 0): no list
    B.lo = (lo > 0.0f && s < (double)v.n) ? lo : __int_as_float(0x7f800000);
  }
  float fsum = 0.0f, m = 0.0f;
  ew_for_units(v, c, x, [&](uint32_t, const float4& y) { ew_sums(y, fsum, m); }, [&](uint32_t blk) {
    amax = fmaxf(amax, m);
    sum += (double)fsum;
    if (!(m > B.lo)) rest += (double)fsum;
    else if (at < (uint32_t)(kEwBig * kEwThreads)) { B.run[at] = blk; at += kEwThreads; }
    else sh.big_over = 1u;
    fsum = 0.0f; m = 0.0f;
  });
  B.rest = rest;
  B.n = at / kEwThreads;
  return EwAcc{sum, amax, 0u};
}
// one water-filling round over the chunk: unsaturated sum and saturated count at threshold theta, from memory
__device__ __forceinline__ void ew_round_sums(const float4& x, const float theta, float& fsum, uint32_t& cnt) {
  const float a[4] = {fabsf(x.x), fabsf(x.y), fabsf(x.z), fabsf(x.w)};
#pragma unroll
  for (int j = 0; j < 4; ++j) { if (a[j] > theta) ++cnt; else fsum += a[j]; }
}
__device__ __forceinline__ EwAcc ew_round_memory(const EwVec& v, const EwChunk& c, const float theta) {
  EwAcc acc{0.0, 0.0f, 0u};
  float4 x[2][4];
  ew_load_ahead(v, c, x);
  float fsum = 0.0f;
  ew_for_units(v, c, x, [&](uint32_t, const float4& y) { ew_round_sums(y, theta, fsum, acc.cnt); }, [&](uint32_t) { acc.sum += (double)fsum; fsum = 0.0f; });
  return acc;
}
// The warp's lists in place, row by row, without the gaps (an entry never moves past one that is still to be read): entry p of the
// warp is in row p / 32, column p % 32 of its part.  Returns their number.
__device__ __forceinline__ uint32_t ew_close_up(uint32_t* const mine, const uint32_t n_mine, const int lane) {
  const uint32_t rows = __reduce_max_sync(0xffffffffu, n_mine);
  uint32_t total = 0;
  for (uint32_t e = 0; e < rows; ++e) {
    const bool have = e < n_mine;
    const uint32_t b = have ? mine[e * kEwThreads + lane] : 0u, votes = __ballot_sync(0xffffffffu, have);
    const uint32_t p = total + __popc(votes & ((1u << lane) - 1u));
    __syncwarp();
    if (have) mine[(p >> 5) * kEwThreads + (p & 31u)] = b;
    total += __popc(votes);
  }
  __syncwarp();
  return total;
}
// ... and from the list, where it holds every run with an atom above theta: run i of all the warps' lists one after the other goes to
// thread i (mod the CTA).  Called by every thread of the CTA.
__device__ __forceinline__ EwAcc ew_round_list(const EwVec& v, const EwChunk& c, EwBigList& B, const float theta, EwShared& sh) {
  EwAcc acc{B.rest, 0.0f, 0u};
  const int w = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
  if (B.n != kEwClosed) {
    const uint32_t n = ew_close_up(B.run + w * kWarp, B.n, lane);
    if (lane == 0) sh.big[w] = n;
    B.n = kEwClosed;
    __syncthreads();
  }
  uint32_t upto = sh.big[lane];                            // lane: runs of the warps up to this one
#pragma unroll
  for (int q = 1; q < kWarp; q <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, upto, q); if (lane >= q) upto += t; }
  const uint32_t total = __shfl_sync(0xffffffffu, upto, kWarp - 1);
  for (uint32_t i0 = w * kWarp; i0 < total; i0 += kEwThreads) {
    const uint32_t i = i0 + lane;
    int of = 0;                                            // the warp whose list holds it
#pragma unroll
    for (int q = kWarp / 2; q > 0; q >>= 1) if (__shfl_sync(0xffffffffu, upto, of + q - 1) <= i) of += q;
    const uint32_t before = __shfl_sync(0xffffffffu, upto, max(of - 1, 0)), e = i - (of > 0 ? before : 0u);
    if (i >= total) continue;
    const int64_t base = c.beg + 4 * (int64_t)B.run[(e >> 5) * kEwThreads + of * kWarp + (e & 31u)];
    float4 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t at = base + (int64_t)u * 1024;
      x[u] = at < c.end ? load4(v.g, at, c.end, c.aligned) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float fsum = 0.0f;
#pragma unroll
    for (int u = 0; u < 4; ++u) ew_round_sums(x[u], theta, fsum, acc.cnt);
    acc.sum += (double)fsum;
  }
  return acc;
}

// ---- pass 1 with a list of candidates (small budgets) ----------------------------------------------------------------
// The keep decision of an atom needs ||g||_1, which only the end of the first pass knows; but the Philox word of an
// atom depends on its index alone.  So the first pass already draws the words and lists the few blocks of four atoms
// (one Philox call) that can still hold a kept one: an atom is kept (Eq. 2 with p < 1) iff word < floor(|g| scale 2^32),
// and the pass tests word <= |g| M with M = 1.25 scale_est 2^32, where scale_est comes from the sum over the chunk's
// first tiles, scaled to the vector's length.  The test of a block is one fused multiply-add per atom (its sign is exact),
// a maximum and one predicated store; a thread keeps its blocks in slots of its own, so the list needs neither atomics
// nor votes.  After the barrier the true scale is known.  If M >= scale 2^32 (1 + 2^-22) (the slack covers the
// rounding of the decision's product), the vector is s-balanced (no atom with p = 1) and no thread ran out of slots,
// the list covers every kept atom of the chunk and the exact decision is taken on its blocks alone (their words are
// drawn and their entries read again, mostly from the L2): the chunk is read once.  Otherwise the CTA reads its chunk
// a second time.  Either way the decision is the same integer comparison on the same operands, so the payload does not
// depend on which way a chunk went.
// Bound: instruction issue (Philox4x32-10 is 40 of about 75 instructions per four atoms).  Listing single atoms with
// their values, two stores and a test each, took 171 instructions per four atoms and 38 us for the pass over 25.6 M
// elements.
constexpr int kEwCandPerThread = 16;             // list entries per thread; 1.25 s (atoms per thread) / n are expected
constexpr int kEwCandBytes = (kEwCandPerThread + 1) * kEwThreads * 4;   // one more row takes what does not fit (never read)
struct EwCands {
  uint32_t* blk;      // [kEwCandPerThread + 1][kEwThreads] Philox blocks
  float m32;          // the multiplier M the list was made with (0: no list)
  uint32_t addr;      // shared-memory address of this thread's next slot: rows of kEwThreads 4-byte entries
  uint32_t addr0;     // ... of its first slot
};
__device__ __forceinline__ uint32_t ew_cand_count(const EwCands& C) { return (C.addr - C.addr0) / (4u * kEwThreads); }

// one block (blk: its Philox block, atom / 4); entries past the chunk's end are zeros, which are listed only where the word is
// zero (and the exact decision drops them)
__device__ __forceinline__ void ew_cand_block(const float4& x, const uint32_t blk, const uint32_t layer,
                                              const PhiloxRoundKeys& key, const uint32_t kind_step, EwCands& C) {
  const float m32 = C.m32;
  const uint32_t spill = C.addr0 + (uint32_t)(kEwCandPerThread * kEwThreads * 4);   // this thread's slot in the extra row
  const uint4 wd = philox4x32_10(make_uint4(blk, 0u, layer, kind_step), key);
  const float d0 = fmaf(fabsf(x.x), m32, -__uint2float_rz(wd.x)), d1 = fmaf(fabsf(x.y), m32, -__uint2float_rz(wd.y));
  const float d2 = fmaf(fabsf(x.z), m32, -__uint2float_rz(wd.z)), d3 = fmaf(fabsf(x.w), m32, -__uint2float_rz(wd.w));
  const float d = fmaxf(fmaxf(d0, d1), fmaxf(d2, d3));
  const uint32_t o = min(C.addr, spill);
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ge.f32 p, %2, 0f00000000;\n\t"
      "@p st.shared.u32 [%1], %3;\n\t"
      "@p add.u32 %0, %0, %4;\n\t}"
      : "+r"(C.addr)
      : "r"(o), "f"(d), "r"(blk), "n"(kEwThreads * 4)
      : "memory");
}

__device__ __forceinline__ EwAcc ew_pass_cand(const EwVec& v, const EwChunk& c, const double s, const PhiloxRoundKeys& key,
                                              const uint32_t kind_step, EwCands& C, EwShared& sh) {
  double sum = 0.0;
  float amax = 0.0f;
  float4 x[1][4];
  ew_load_ahead(v, c, x);
  {
    // M = 1.25 (s / l1_est) 2^32.  A zero or non-finite estimate gives inf or NaN: the threads' lists overflow or stay
    // empty and the check after the barrier sends the chunk the other way
    const float m32 = (float)(1.25 * s * 4294967296.0 / ew_estimate_l1(v, c, x[0], sh));
    C.m32 = m32 > 0.0f ? m32 : 0.0f;
  }
  const uint32_t blk_beg = (uint32_t)(c.beg >> 2);
  float fsum = 0.0f;
  ew_for_units(v, c, x, [&](uint32_t blk, const float4& y) {
    ew_sums(y, fsum, amax);
    ew_cand_block(y, blk_beg + blk, v.layer, key, kind_step, C);
  }, [&](uint32_t) {
    sum += (double)fsum;
    fsum = 0.0f;
    if (C.addr > C.addr0 + (uint32_t)(kEwCandPerThread * kEwThreads * 4)) {   // no slot left: this chunk will be read twice
      sh.stop = 1u;
      C.m32 = -1.0f;                                       // nothing more to list
    }
  });
  return EwAcc{sum, amax, 0u};
}

// ---- the solve --------------------------------------------------------------------------------------------------------
// what the probability solve leaves for the sampling pass (every CTA of the vector computes the same values)
struct EwSolved { double T0; float scale, theta, c, amax; uint32_t n_sat, rounds; bool nonfinite; };

// `first`: this thread's part of pass 1; `round(theta)`: this thread's part of a water-filling round over the chunk
template <typename Round>
__device__ __forceinline__ EwSolved ew_solve(const EwVec& v, const EwChunk& c, const double s, const EwAcc& first, Round round, EwShared& sh) {
  const int nb = v.n_ctas;
  uint32_t arrivals = 0;
  // every chunk's partial sums out, those of all chunks in; each CTA adds them in the same order
  auto exchange = [&](EwAcc mine, int buf) {
    mine = ew_block_reduce(mine, sh);
    if (nb == 1) return mine;
    EwPartial* const part = v.partials + (size_t)buf * nb;
    if (threadIdx.x == 0) part[c.index] = EwPartial{mine.sum, mine.amax, mine.cnt};
    arrivals += (uint32_t)nb;
    ew_barrier(v, arrivals, sh);
    EwAcc tot{0.0, 0.0f, 0u};
    for (int i = threadIdx.x; i < nb; i += kEwThreads) {
      static_assert(sizeof(EwPartial) == 16, "one 16-byte load");
      const int4 raw = __ldcg(reinterpret_cast<const int4*>(part + i));
      tot.sum += __hiloint2double(raw.y, raw.x); tot.amax = fmaxf(tot.amax, __int_as_float(raw.z)); tot.cnt += (uint32_t)raw.w;
    }
    return ew_block_reduce(tot, sh);
  };
  EwAcc tot = exchange(first, 0);
  const double T0 = tot.sum;
  const float amax = tot.amax;
  const bool nonfinite = !(T0 == T0) || !(amax <= 3.402823466e38f);     // an entry is NaN or infinite
  double T = T0, s_cur = s;
  uint32_t n_sat = 0, rounds = 0;
  // atoms with |g| > theta are unbalanced (Definition 1) for the current (T, s_cur); Lemma 3: none if
  // s <= ||g||_1 / ||g||_inf.  The comparison is made in fp32 everywhere so that every kernel agrees on
  // which atoms are saturated.  A budget of n or more keeps every non-zero atom: threshold 0 at once.
  float theta = s >= (double)v.n ? 0.0f : (float)(T0 / s);
  bool done = nonfinite || !(amax > theta);
  while (!done && rounds < kEwMaxRounds) {
    // buffers alternate: a chunk may still read the previous exchange while others write this one
    tot = exchange(round(theta), (int)(rounds & 1) + 1);
    ++rounds;
    if (tot.cnt == n_sat) { done = true; }             // no new saturated atom: (T, s_cur) stand
    else {
      n_sat = tot.cnt; T = tot.sum; s_cur = s - (double)n_sat;
      const float th = (T > 0.0 && s_cur > 0.0) ? (float)(T / s_cur) : 0.0f;
      theta = fminf(theta, th);
    }
  }
  const bool live = T > 0.0 && s_cur > 0.0 && !nonfinite;
  EwSolved r;
  r.T0 = T0; r.theta = theta; r.n_sat = n_sat; r.rounds = rounds; r.nonfinite = nonfinite; r.amax = amax;
  r.scale = live ? (float)(s_cur / T) : 0.0f;            // p_i = |g_i| * scale
  r.c = live ? (float)(T / s_cur) : 0.0f;                // weight of kept unsaturated atoms
  return r;
}
// what the vector's barrier counts in a solve: every CTA once per exchange
__device__ __forceinline__ uint32_t ew_arrivals(const EwVec& v, const EwSolved& S) { return v.n_ctas > 1 ? (uint32_t)v.n_ctas * (1u + S.rounds) : 0u; }
__device__ __forceinline__ void ew_store_state(const EwVec& v, const EwSolved& S) {
  EwState* st = v.state;
  st->T0 = S.T0; st->theta = S.theta; st->amax = S.amax; st->n_sat = S.n_sat; st->rounds = S.rounds;
  st->nonfinite = S.nonfinite ? 1u : 0u; st->scale = S.scale; st->c = S.c;
}

// ---- the keep decisions -------------------------------------------------------------------------------------------------
// p = 1 on the saturated set, min(|g| scale, 1) elsewhere; keep iff p >= 1 or word < floor(p 2^32).  t = |g| scale32 is the
// same product times 2^32 (exact).  word < floor(t) is word <= t - 1 in whole numbers, and rz(word) <= rd(t - 1) in fp32 says
// exactly that: below 2^24 both sides are exact (t is a multiple of its last place, at most 1); above, rd(t - 1) is the
// largest fp32 number below t, and rz(word) is below t iff word is.  (The conversion of t to an integer would go through
// the pipe that converts 16 numbers per clock: 46 us for 100 M atoms.)
struct EwDecide { float scale, scale32, theta, below_one; bool dead; };   // atoms with |g| < below_one have p < 1
__device__ __forceinline__ EwDecide ew_decide_of(const EwSolved& S) {
  EwDecide d;
  d.scale = S.scale; d.scale32 = S.scale * 4294967296.0f; d.theta = S.theta; d.dead = S.nonfinite;
  // |g| scale is below 1 by more than the rounding of the product, and |g| below theta.  (The fast path also wants a kept
  // atom's entry to be a normal number: t >= 1 means |g| >= 1 / scale32.)
  d.below_one = d.scale32 > 0.0f && d.scale32 < 1.0e27f && !d.dead ? fminf(d.theta, 0.999f / S.scale) : 0.0f;
  return d;
}
// code byte of a block, any case; i: index of its first atom
__device__ __noinline__ uint32_t ew_code_any(const float4 x, const uint4 wd, const EwDecide d, const int64_t i, const int64_t end) {
  const float g[4] = {x.x, x.y, x.z, x.w};
  const uint32_t ww[4] = {wd.x, wd.y, wd.z, wd.w};
  uint32_t code = 0;
  for (int j = 0; j < 4; ++j) {
    const float a = fabsf(g[j]), t = a * d.scale32;
    const bool sat = a > d.theta;
    if (d.dead || i + j >= end || !(sat || t >= 4294967296.0f || __uint2float_rz(ww[j]) <= __fadd_rd(t, -1.0f))) continue;
    if (!sat) code |= 1u << j;
    if (sat || __float_as_int(g[j]) < 0) code |= 16u << j;
  }
  return code;
}
// ... where every |g| of the block is below below_one and inside the chunk.  What bounds pass 2 is the pipe for logic, compares
// and votes (half the rate of multiply-adds, and the rounds of Philox need it for 20 instructions per block), so the byte is
// put together by multiply-adds: saturated to [0, 1] they are the indicators of "kept" and "negative", and the sum at 2^23
// has the byte as its last bits.  (A compare and a vote per bit: 143 instructions per block, 65 of them in that pipe.)
__device__ __forceinline__ uint32_t ew_code_plain(const float4& x, const uint4& wd, const EwDecide& d) {
  const float g[4] = {x.x, x.y, x.z, x.w};
  const uint32_t ww[4] = {wd.x, wd.y, wd.z, wd.w};
  float acc = 8388608.0f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float over = __fsub_rn(__fadd_rd(__fmul_rn(fabsf(g[j]), d.scale32), -1.0f), __uint2float_rz(ww[j]));   // kept iff >= 0; else at most -2^-24
    const float kept = __saturatef(fmaf(over, 1.152921504606846976e18f, 1.0f));
    const float neg = __saturatef(g[j] * -8.507059173023462e37f);                     // (of a kept atom: |g| >= 2^-90)
    acc = fmaf(kept, fmaf(neg, (float)(16 << j), (float)(1 << j)), acc);
  }
  return __float_as_uint(acc) & 255u;
}
__device__ __forceinline__ uint4 ew_block_words(const EwVec& v, const EwChunk& c, const int unit, const int u, const PhiloxRoundKeys& key,
                                                const uint32_t kind_step) {
  // block of 4 atoms = atom >> 2 < 2^30 (n < 2^32): the high counter word is zero
  return philox4x32_10(make_uint4((uint32_t)(c.beg >> 2) + ew_unit_block(unit) + (uint32_t)(256 * u), 0u, v.layer, kind_step), key);
}
__device__ __forceinline__ void ew_block_decide(const EwChunk& c, const int unit, const int u, const float4& x, const uint4& wd, const EwDecide& d, uint8_t* code) {
  const uint32_t blk = ew_unit_block(unit) + (uint32_t)(256 * u);
  const bool plain = unit / kEwUnits < c.n_full && max4(x) < d.below_one;      // almost always
  code[blk] = (uint8_t)(plain ? ew_code_plain(x, wd, d) : ew_code_any(x, wd, d, c.beg + 4 * (int64_t)blk, c.end));
}
// the probabilities (debug output)
__device__ __forceinline__ void ew_block_prob(const EwVec& v, const EwChunk& c, const int unit, const int u, const float4& x, const EwDecide& d) {
  const int64_t i = c.beg + 4 * (int64_t)ew_unit_block(unit) + 1024 * u;
  const float a[4] = {fabsf(x.x), fabsf(x.y), fabsf(x.z), fabsf(x.w)};
  for (int j = 0; j < 4 && i + j < c.end; ++j)
    v.prob_out[i + j] = d.dead ? 0.0f : ((a[j] > d.theta) ? 1.0f : fminf(a[j] * d.scale, 1.0f));
}
// pass 2 over the chunk, read (again) from memory.  The warps take the units as they become free, from the chunk's last to its
// first: pass 1 read them in ascending order just before, so the end of the chunk is what the L2 still holds.
__device__ __forceinline__ void ew_decide_memory(const EwVec& v, const EwChunk& c, const EwDecide& d, const PhiloxRoundKeys& key,
                                                 const uint32_t kind_step, EwShared& sh, uint8_t* code) {
  const int lane = threadIdx.x % kWarp;
  if (threadIdx.x == 0) sh.next_unit = 0u;
  __syncthreads();
  auto take = [&]() -> int {                               // next unit, or a negative number
    uint32_t t = 0;
    if (lane == 0) t = atomicAdd(&sh.next_unit, 1u);
    return c.n_units - 1 - (int)__shfl_sync(0xffffffffu, t, 0);
  };
  float4 x[4];
  int unit = take();
  ew_load_unit(v, c, unit, x);
  const uint32_t blk_beg = (uint32_t)(c.beg >> 2);
  while (unit >= 0) {
    const int next = take();
    const uint32_t blk = ew_unit_block(unit);
    if (unit / kEwUnits < c.n_full && next / kEwUnits < c.n_full && next >= 0 && v.prob_out == nullptr) {
      const float4* const src = reinterpret_cast<const float4*>(v.g + c.beg) + ew_unit_block(next);
      float m = 0.0f;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint4 wd = philox4x32_10(make_uint4(blk_beg + blk + (uint32_t)(256 * u), 0u, v.layer, kind_step), key);
        code[blk + (uint32_t)(256 * u)] = (uint8_t)ew_code_plain(x[u], wd, d);
        m = fmaxf(m, max4(x[u]));
        x[u] = __ldg(src + 256 * u);
      }
      if (!(m < d.below_one)) {                            // rare: a lane's blocks again, with the tests for p = 1
        for (int u = 0; u < 4; ++u) {
          const float4 y = ew_load_unit(v, c, unit, u);
          const uint4 wd = philox4x32_10(make_uint4(blk_beg + blk + (uint32_t)(256 * u), 0u, v.layer, kind_step), key);
          code[blk + (uint32_t)(256 * u)] = (uint8_t)ew_code_any(y, wd, d, c.beg + 4 * (int64_t)(blk + 256 * u), c.end);
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        ew_block_decide(c, unit, u, x[u], ew_block_words(v, c, unit, u, key, kind_step), d, code);
        if (v.prob_out != nullptr) ew_block_prob(v, c, unit, u, x[u], d);
        if (next >= 0) x[u] = ew_load_unit(v, c, next, u);
      }
    }
    unit = next;
  }
}
// pass 2 on the candidate blocks alone; the code bytes start at zero.  A warp first closes up its lanes' lists, so that every lane
// decides on the same number of blocks: the fullest lane has three times the average.  What was decided on a block goes back to its place: code byte << 24 | block inside
// the chunk.  Returns the warp's number of blocks.
__device__ __forceinline__ uint32_t ew_decide_list(const EwVec& v, const EwChunk& c, const EwDecide& d, const PhiloxRoundKeys& key,
                                                   const uint32_t kind_step, const EwCands& C, uint8_t* __restrict__ code) {
  const int lane = threadIdx.x % kWarp;
  uint32_t* const mine = C.blk + (threadIdx.x - lane);     // entry p of the warp: row p / 32, column p % 32
  const uint32_t blk_beg = (uint32_t)(c.beg >> 2), total = ew_close_up(mine, ew_cand_count(C), lane);
  for (uint32_t e0 = lane; e0 < total; e0 += 4 * kWarp) {
    uint32_t b[4];
    float4 x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {                          // four blocks' entries in flight
      const uint32_t e = e0 + q * kWarp;
      b[q] = e < total ? mine[(e >> 5) * kEwThreads + lane] : 0xFFFFFFFFu;
      if (b[q] != 0xFFFFFFFFu) x[q] = load4(v.g, 4 * (int64_t)b[q], c.end, c.aligned);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (b[q] == 0xFFFFFFFFu) break;
      const uint4 wd = philox4x32_10(make_uint4(b[q], 0u, v.layer, kind_step), key);
      const uint32_t local = b[q] - blk_beg;
      const uint32_t said = max4(x[q]) < d.below_one ? ew_code_plain(x[q], wd, d) : ew_code_any(x[q], wd, d, 4 * (int64_t)b[q], c.end);
      if (said) atomicOr(reinterpret_cast<uint32_t*>(code) + (local >> 2), said << (8u * (local & 3u)));
      mine[((e0 + q * kWarp) >> 5) * kEwThreads + lane] = (said << 24) | local;
    }
  }
  return total;
}

// ---- counts of the earlier chunks, ordered compaction, headers -----------------------------------------------------------
struct EwLists {                  // where a chunk's kept atoms go
  uint32_t* idx; float* val; uint16_t* ent; uint32_t* sat_idx; uint32_t* table;
  bool compact;
  // position in the entry list (explicit: every kept atom; compact: those with p < 1) for counts as below
  __device__ __forceinline__ uint64_t list_of(unsigned long long x) const { return compact ? (x & 0xFFFFFFFFull) - (x >> 32) : x & 0xFFFFFFFFull; }
};
__device__ __forceinline__ EwLists ew_lists(const EwVec& v) {
  EwLists o;
  o.idx = reinterpret_cast<uint32_t*>(v.pay + v.off_idx); o.ent = reinterpret_cast<uint16_t*>(v.pay + v.off_idx);
  o.val = reinterpret_cast<float*>(v.pay + v.off_val); o.table = reinterpret_cast<uint32_t*>(v.pay + v.off_tiles);
  o.sat_idx = reinterpret_cast<uint32_t*>(v.pay + v.off_sat);
  o.compact = v.compact != 0;
  return o;
}
// The chunk's counts (kept atoms, saturated ones in bits 32 ..) go out; the CTA then waits (bounded) until every earlier chunk of
// the vector has published and adds their counts -- all chunks of a wave finish their decisions together, so nobody waits
// on a chain.  Returns the counts before this chunk.  The last chunk writes k, the capacity check and the layer header; a
// wait that runs out raises ATOMO_ERR_TIMEOUT.  Every thread of the CTA passes the same `total`.
//
// One-kernel form: that CTA also leaves the vector's barrier counter at zero.  Every CTA has published, so nobody looks at the barrier
// any more, and `arrivals` is what it must have counted.  So every launch finds a zero, whatever the host launched before it, in
// a replayed graph too; a counter that was not zero (after a wait that ran out) shows as ATOMO_ERR_TIMEOUT, once.  (Counting the
// CTAs out with an atomic each at their ends: 1.5 M elements 24.6 us instead of 23.9.)
__device__ __forceinline__ unsigned long long ew_publish(const EwVec& v, const EwChunk& c, const EwSolved& S, const uint32_t arrivals, const EwLists& o,
                                                         const unsigned long long total, EwShared& sh) {
  const int tid = threadIdx.x, lane = tid % kWarp, w = tid / kWarp;
  unsigned long long base = 0;
  if (v.n_ctas > 1) {
    if (tid == 0) *(volatile unsigned long long*)(v.chunk_status + c.index) = kFlagReady | total;
    unsigned long long before = 0;
    for (uint32_t ci = tid; ci < c.index; ci += kEwThreads) {
      unsigned long long sv;
      uint32_t polls = 0;
      for (;;) {
        sv = *(volatile const unsigned long long*)(v.chunk_status + ci);
        if ((sv & kFlagReady) || ++polls > kEwPollLimit) break;
        __nanosleep(40);
      }
      if (!(sv & kFlagReady)) sh.fail = 1u;
      before += sv & ~kFlagReady;                          // totals < 2^32 in all: the two fields never mix
    }
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) before += __shfl_xor_sync(0xffffffffu, before, q);
    if (lane == 0) sh.before[w] = before;
    __syncthreads();
    base = sh.before[lane];
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) base += __shfl_xor_sync(0xffffffffu, base, q);
  }
  if (tid == 0) {
    if (sh.fail) raise_status(v.hdr, ATOMO_ERR_TIMEOUT);
    if (c.tile0 + c.n_my == v.n_tiles) {                   // the last chunk knows k: capacity check, layer header
      atomo_layer_header* h = v.hdr;
      const unsigned long long all = base + total;
      const uint64_t k = all & 0xFFFFFFFFull, k_sat = all >> 32, k_list = o.list_of(all);
      uint32_t seen, status;                               // (both loads on their way before either is looked at)
      asm volatile("ld.volatile.global.u32 %0, [%2];\n\tld.volatile.global.u32 %1, [%3];" : "=&r"(seen), "=r"(status) : "l"(v.barrier), "l"(&h->status) : "memory");
      if (arrivals > 0) *(volatile uint32_t*)v.barrier = 0u;
      h->n_sat = S.n_sat; h->c = S.c; h->l1 = S.T0; h->sweeps = S.rounds;
      uint32_t bad = ATOMO_OK;
      if (sh.fail || (arrivals > 0 && seen != arrivals)) bad = ATOMO_ERR_TIMEOUT;
      else if (S.nonfinite) bad = ATOMO_ERR_NONFINITE;
      else if (k_list > (uint64_t)v.k_cap || (o.compact && k_sat > (uint64_t)v.sat_cap)) bad = ATOMO_ERR_CAPACITY;
      if (bad != ATOMO_OK) raise_status(h, bad);
      const bool ok = bad == ATOMO_OK && status == ATOMO_OK;
      h->k = ok ? (uint32_t)k : 0u;
      if (o.compact) h->n_sat = ok ? (uint32_t)k_sat : 0u; // the length of the saturated list
      o.table[v.n_tiles] = ok ? (uint32_t)k_list : 0u;
    }
  }
  return base;
}
// the low nibbles of eight code bytes as 32 bits in the order of the atoms
__device__ __forceinline__ uint32_t ew_nibbles(uint32_t lo, uint32_t hi) {
  lo &= 0x0F0F0F0Fu; hi &= 0x0F0F0F0Fu;
  lo = (lo | (lo >> 4)) & 0x00FF00FFu; hi = (hi | (hi >> 4)) & 0x00FF00FFu;
  return __byte_perm(lo, hi, 0x6420);
}
// K and S bits of 32 consecutive atoms: word `at` of the chunk
__device__ __forceinline__ void ew_word(const uint8_t* __restrict__ code, const int at, uint32_t& kk, uint32_t& ss) {
  const uint2 b = reinterpret_cast<const uint2*>(code)[at];
  kk = ew_nibbles(b.x, b.y); ss = ew_nibbles(b.x >> 4, b.y >> 4);
}
// debug output: the kept atoms as a plain bit mask
__device__ __forceinline__ void ew_mask_out(const EwVec& v, const EwChunk& c, const uint8_t* __restrict__ code) {
  for (int wi = threadIdx.x; wi < c.n_my * (kEwTile / 32); wi += kEwThreads) {
    const int64_t widx = c.tile0 * (kEwTile / 32) + wi;
    uint32_t kk, ss;
    ew_word(code, wi, kk, ss);
    if (widx < v.n_words) v.mask_words[widx] = kk | ss;
  }
}

// Compaction of the decisions taken on the list: a scan over the counts of 32 atoms each, then every kept atom finds its own
// place from the prefix and the bits before it, and stores its entry directly.  `n_blocks`: what ew_decide_list returned;
// pref: kEwPrefixes words per tile of the chunk.
__device__ __forceinline__ void ew_pack_list(const EwVec& v, const EwChunk& c, const EwSolved& S, const uint32_t arrivals, const EwCands& C, const uint32_t n_blocks,
                                             const uint8_t* __restrict__ code, uint32_t* __restrict__ pref, EwShared& sh) {
  const int tid = threadIdx.x, lane = tid % kWarp, w = tid / kWarp;
  const EwLists o = ew_lists(v);
  const int n = c.n_my * kEwPrefixes, per = (n + kEwThreads - 1) / kEwThreads;   // consecutive words per thread
  const int g0 = min(tid * per, n), g1 = min(g0 + per, n);
  auto count = [&](int at) -> uint32_t {                   // no atom has p = 1: the K bits alone
    const uint2 b = reinterpret_cast<const uint2*>(code)[at];
    return (uint32_t)(__popc(b.x & 0x0F0F0F0Fu) + __popc(b.y & 0x0F0F0F0Fu));
  };
  uint32_t cnt = 0;
  for (int at = g0; at < g1; ++at) { pref[at] = cnt; cnt += count(at); }
  uint32_t inc = cnt;
#pragma unroll
  for (int q = 1; q < 32; q <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, q); if (lane >= q) inc += t; }
  if (lane == 31) sh.cnt[w] = inc;
  __syncthreads();
  const uint32_t part = sh.cnt[lane];
  const uint32_t total = __reduce_add_sync(0xffffffffu, part);
  const uint32_t before = __reduce_add_sync(0xffffffffu, lane < w ? part : 0u) + inc - cnt;
  for (int at = g0; at < g1; ++at) pref[at] += before;
  const uint64_t base = ew_publish(v, c, S, arrivals, o, total, sh);
  __syncthreads();                                         // pref is complete
  if (v.n_words > 0) ew_mask_out(v, c, code);
  for (int t = tid; t < c.n_my; t += kEwThreads) o.table[c.tile0 + t] = (uint32_t)min(base + pref[t * kEwPrefixes], (uint64_t)0xFFFFFFFFull);
  const uint32_t* const mine = C.blk + (tid - lane);
  const float cw = S.c;
  for (uint32_t e = lane; e < n_blocks; e += kWarp) {
    const uint32_t said = mine[(e >> 5) * kEwThreads + lane];
    uint32_t nib = (said >> 24) & 15u;
    if (nib == 0) continue;
    const uint32_t b = said & 0xFFFFFFu, byte = b & 7u;
    const uint2 eight = reinterpret_cast<const uint2*>(code)[b >> 3];
    const uint32_t below = (1u << (8u * (byte & 3u))) - 1u;    // the earlier bytes of the block's own word
    const uint32_t lo = eight.x & 0x0F0F0F0Fu & (byte < 4u ? below : 0xFFFFFFFFu), hi = eight.y & 0x0F0F0F0Fu & (byte < 4u ? 0u : below);
    uint64_t pos = base + pref[b >> 3] + (uint32_t)(__popc(lo) + __popc(hi));
    const uint32_t i0 = (uint32_t)(c.beg + 4 * (int64_t)b);
    for (; nib; nib &= nib - 1, ++pos) {
      const uint32_t j = (uint32_t)(__ffs(nib) - 1), neg = (said >> (28 + j)) & 1u;
      if (pos >= (uint64_t)v.k_cap) continue;
      // the value of a kept atom with p < 1 is sign(g) c
      if (o.compact) o.ent[pos] = (uint16_t)(((i0 + j) & (uint32_t)(kEwTile - 1)) | (neg << 15));
      else { o.idx[pos] = i0 + j; o.val[pos] = neg ? -cw : cw; }
    }
  }
}

// Compaction of the code bytes.  A warp takes a run of strips of 1024 atoms, 32 consecutive atoms per lane; a scan over the
// lanes gives every lane its place in the lists, the kept atoms are put into the warp's window in shared memory in order and
// the window leaves with coalesced stores (direct 4-byte stores from every thread's own run cost an L2 request each).  A
// strip with more kept atoms than the window holds is written 32 atoms at a time, an atom per lane.  The signs in the code
// bytes make a second read of the kept atoms' values unnecessary, except for saturated ones.
__device__ __forceinline__ void ew_pack(const EwVec& v, const EwChunk& c, const EwSolved& S, const uint32_t arrivals, const uint8_t* __restrict__ code,
                                        uint32_t* __restrict__ stage, EwShared& sh) {
  const int tid = threadIdx.x, lane = tid % kWarp, w = tid / kWarp;
  const EwLists o = ew_lists(v);
  const bool compact = o.compact;
  const int n_strips = c.n_my * (kEwTile / 1024), u_lo = n_strips * w / kEwWarps, u_hi = n_strips * (w + 1) / kEwWarps;
  unsigned long long mine = 0;                             // kept atoms of the warp's run; saturated ones in bits 32 ..
  for (int u = u_lo; u < u_hi; ++u) {
    uint32_t kk, ss;
    ew_word(code, u * 32 + lane, kk, ss);                  // this lane's 32 atoms of the strip
    mine += ((unsigned long long)__popc(ss & ~kk) << 32) | (unsigned long long)__popc(kk | ss);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  if (lane == 0) sh.scan[w] = mine;
  __syncthreads();
  unsigned long long total = sh.scan[lane], run = lane < w ? total : 0ull;   // of the chunk; of the earlier warps
#pragma unroll
  for (int q = 16; q > 0; q >>= 1) { total += __shfl_xor_sync(0xffffffffu, total, q); run += __shfl_xor_sync(0xffffffffu, run, q); }
  run += ew_publish(v, c, S, arrivals, o, total, sh);
  if (v.n_words > 0) ew_mask_out(v, c, code);
  // the warp's window: atom inside the strip | saturated << 14 | sign << 15
  uint16_t* const win = reinterpret_cast<uint16_t*>(stage) + w * kEwStage;
  const float cw = S.c;
  const uint64_t k_cap = v.k_cap, sat_cap = v.sat_cap;
  for (int u = u_lo; u < u_hi; ++u) {
    uint32_t kk, ss;
    ew_word(code, u * 32 + lane, kk, ss);                  // this lane's 32 atoms of the strip
    const uint32_t sat_bits = ss & ~kk, list_bits = compact ? kk : kk | ss;
    const uint32_t cnt = (uint32_t)__popc(list_bits) | ((uint32_t)__popc(sat_bits) << 16);   // at most 1024 each per strip
    uint32_t inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += t; }
    const uint32_t all = __shfl_sync(0xffffffffu, inc, 31);
    const uint32_t n_list = all & 0xFFFFu, n_sat = all >> 16;
    const uint64_t list0 = o.list_of(run);                   // list position of the strip's first entry
    if (u % (kEwTile / 1024) == 0 && lane == 0) o.table[c.tile0 + u / (kEwTile / 1024)] = (uint32_t)min(list0, (uint64_t)0xFFFFFFFFull);
    const uint32_t atom0 = (uint32_t)((c.tile0 * (kEwTile / 1024) + u) * 1024);
    if (n_list <= (uint32_t)kEwStage) {
      uint32_t pos = (inc - cnt) & 0xFFFFu;
      const uint32_t at0 = 32u * (uint32_t)lane;
      if (n_sat == 0) {
        for (uint32_t left = list_bits; left; left &= left - 1) {
          const uint32_t b = (uint32_t)(__ffs(left) - 1);
          win[pos++] = (uint16_t)((at0 + b) | (((ss >> b) & 1u) << 15));
        }
      } else {
        for (uint32_t left = list_bits; left; left &= left - 1) {
          const uint32_t b = (uint32_t)(__ffs(left) - 1);
          win[pos++] = (uint16_t)((at0 + b) | (((ss >> b) & 1u) << 15) | (((sat_bits >> b) & 1u) << 14));
        }
      }
      __syncwarp();
      for (uint32_t e = lane; e < n_list; e += kWarp) {
        if (list0 + e >= k_cap) continue;
        const uint32_t en = win[e], i = atom0 + (en & 1023u);
        if (compact) { o.ent[list0 + e] = (uint16_t)((i & (uint32_t)(kEwTile - 1)) | (en & 0x8000u)); continue; }
        // kept atom: saturated (p = 1) keeps g; otherwise g / p = sign(g) T / (s - n_s)
        o.idx[list0 + e] = i;
        o.val[list0 + e] = (en & 0x4000u) ? __ldg(v.g + i) : (en & 0x8000u) ? -cw : cw;
      }
      __syncwarp();
    } else {
      uint64_t at = list0;
      for (int t = 0; t < 32; ++t) {
        const bool in = (__shfl_sync(0xffffffffu, list_bits, t) >> lane) & 1u;
        const bool neg = (__shfl_sync(0xffffffffu, ss, t) >> lane) & 1u, sat = (__shfl_sync(0xffffffffu, sat_bits, t) >> lane) & 1u;
        const uint32_t have = __ballot_sync(0xffffffffu, in);
        const uint64_t pos = at + __popc(have & ((1u << lane) - 1u));
        const uint32_t i = atom0 + 32u * (uint32_t)t + (uint32_t)lane;
        if (in && pos < k_cap) {
          if (compact) o.ent[pos] = (uint16_t)((i & (uint32_t)(kEwTile - 1)) | (neg ? 0x8000u : 0u));
          else { o.idx[pos] = i; o.val[pos] = sat ? __ldg(v.g + i) : neg ? -cw : cw; }
        }
        at += __popc(have);
      }
    }
    if (compact && n_sat) {                                // the saturated atoms' own list
      uint64_t at = run >> 32;
      for (int t = 0; t < 32; ++t) {
        const bool in = (__shfl_sync(0xffffffffu, sat_bits, t) >> lane) & 1u;
        const uint32_t have = __ballot_sync(0xffffffffu, in);
        const uint64_t pos = at + __popc(have & ((1u << lane) - 1u));
        const uint32_t i = atom0 + 32u * (uint32_t)t + (uint32_t)lane;
        if (in && pos < sat_cap) { o.sat_idx[pos] = i; o.val[pos] = __ldg(v.g + i); }
        at += __popc(have);
      }
    }
    run += compact ? ((unsigned long long)n_sat << 32) + n_list + n_sat : ((unsigned long long)n_sat << 32) + n_list;
  }
}

// payload header (by the first vector's first CTA) and the layer header as it stands before the counts are known
__device__ __forceinline__ void ew_write_headers(const EwVec& v, const EwBegin& b, const bool first_vec) {
  if (threadIdx.x != 0) return;
  if (b.on && first_vec) *reinterpret_cast<atomo_payload_header*>(v.pay) = b.gh;
  atomo_layer_header h{};
  h.rows = 1; h.cols = v.n; h.k_cap = v.k_cap; h.status = ATOMO_OK;
  h.off_idx = v.off_idx; h.off_val = v.off_val; h.off_short = v.off_tiles; h.off_long = v.compact ? v.off_sat : 0;
  *v.hdr = h;
}

// a value the compiler cannot trace: what is worked out from it after a pass is worked out anew instead of being kept in
// registers (and spilled) through the pass
__device__ __forceinline__ uint32_t ew_opaque(uint32_t x) { asm volatile("" : "+r"(x)); return x; }

template <int N>
__device__ __forceinline__ int ew_vec_of(const EwVec (&vecs)[N], const int n, const int cta) {
  int i = 0;
  if (N > 1) while (i + 1 < n && cta >= vecs[i + 1].cta0) ++i;
  return i;
}

// The one-kernel form.  Dynamic shared memory: [scratch: candidate slots, or list of large atoms, later the staging window]
// [code bytes of the chunk] [list form: prefix words].  A chunk of at most kEwRegTiles tiles keeps its entries in
// registers and draws its words before the barrier: nothing is read twice and no list is kept.
// kForm: what the chunks of the launch are, where they are all of one kind (64 registers hold any one of the kinds, but for the code of
// all of them together a chunk's entries were spilled); kMixed asks each chunk.  Spilled bytes 368 | 76 .. 136 for one vector, 504 | 76
// for several (of different kinds: a network's layers still take the first).  An encode, us, one instance for all | by kind: 100 k elements 14.5 | 13.4, 600 k
// 18.5 | 17.5, 1.5 M 18.8 | 17.3, 30 M at 10 % 75.8 | 72.5; within 3 % of each other: 3 M and 100 M at 10 %, 25.6 M, 60 M and 200 M at 1 % and less.
enum { kMixed, kRegisters, kCandidates, kBigList };
template <int N, int kForm>
__global__ void __launch_bounds__(kEwThreads, 1) ew_encode_kernel(const __grid_constant__ EwBatch<N> B) {
  extern __shared__ __align__(16) uint32_t ew_smem[];
  __shared__ EwShared sh;
  const int tid = threadIdx.x;
  const int vi = ew_vec_of(B.v, B.n, (int)blockIdx.x);
  const EwVec& v = B.v[vi];
  EwChunk c = ew_chunk(v, blockIdx.x - (uint32_t)v.cta0);
  uint32_t* const scratch = ew_smem;
  uint8_t* const code = reinterpret_cast<uint8_t*>(ew_smem + B.scratch_words);
  if (tid == 0) { sh.big_over = 0u; sh.stop = 0u; sh.fail = 0u; }
  if (c.index == 0) {
    ew_write_headers(v, B.begin, vi == 0);
    if (tid == 0) v.state->list_chunks = 0u;               // counted after the barrier
  }
  if (tid == 0) v.chunk_status[c.index] = 0ull;            // ordered before its first use by the barrier after pass 1
  __syncthreads();
  if constexpr (kForm == kMixed || kForm == kRegisters)
  if (kForm == kRegisters || (c.n_my <= kEwRegTiles && v.prob_out == nullptr && !v.candidates)) {
    float4 x[4];
    uint4 wd[4];
    const int unit = tid / kWarp;
    ew_load_unit(v, c, (int)(threadIdx.x / kWarp), x);
#pragma unroll
    for (int u = 0; u < 4; ++u) wd[u] = ew_block_words(v, c, unit, u, B.key, B.kind_step);
    float fsum = 0.0f, amax = 0.0f;
#pragma unroll
    for (int u = 0; u < 4; ++u) ew_sums(x[u], fsum, amax);
    const EwSolved S = ew_solve(v, c, B.s, EwAcc{(double)fsum, amax, 0u}, [&](float theta) {
      EwAcc a{0.0, 0.0f, 0u};
      float f = 0.0f;
#pragma unroll
      for (int u = 0; u < 4; ++u) ew_round_sums(x[u], theta, f, a.cnt);
      a.sum = (double)f;
      return a;
    }, sh);
    if (c.index == 0 && tid == 0) ew_store_state(v, S);
    const EwDecide d = ew_decide_of(S);
    if (unit < c.n_units) {
#pragma unroll
      for (int u = 0; u < 4; ++u) ew_block_decide(c, unit, u, x[u], wd[u], d, code);
    }
    __syncthreads();
    ew_pack(v, c, S, ew_arrivals(v, S), code, scratch, sh);
    return;
  }
  if constexpr (kForm == kMixed || kForm == kCandidates)
  if (kForm == kCandidates || v.candidates) {
    const uint32_t cand0 = (uint32_t)__cvta_generic_to_shared(scratch) + 4u * tid;
    EwCands cands{scratch, 0.0f, cand0, cand0};
    for (int i = tid; i < c.n_my * (kEwBlocks / 16); i += kEwThreads) reinterpret_cast<uint4*>(code)[i] = make_uint4(0u, 0u, 0u, 0u);
    const EwAcc first = ew_pass_cand(v, c, B.s, B.key, B.kind_step, cands, sh);
    c = ew_chunk(v, ew_opaque(blockIdx.x) - (uint32_t)v.cta0);
    const EwSolved S = ew_solve(v, c, B.s, first, [&](float theta) { return ew_round_memory(v, c, theta); }, sh);
    if (c.index == 0 && tid == 0) ew_store_state(v, S);
    const EwDecide d = ew_decide_of(S);
    // the list covers every kept atom of the chunk if it was made with a multiplier that covers the true scale, did not
    // overflow and no atom has p = 1
    bool from_list = cands.m32 > 0.0f && S.n_sat == 0 && !d.dead && S.scale > 0.0f &&
                     cands.m32 >= d.scale32 * (1.0f + 2.384185791015625e-07f);
    from_list = __syncthreads_or(ew_cand_count(cands) > (uint32_t)kEwCandPerThread || sh.stop != 0u ? 1 : 0) == 0 && from_list;
    if (from_list) {
      if (tid == 0) atomicAdd(&v.state->list_chunks, 1u);
      const uint32_t n_blocks = ew_decide_list(v, c, d, B.key, B.kind_step, cands, code);
      __syncthreads();
      ew_pack_list(v, c, S, ew_arrivals(v, S), cands, n_blocks, code, reinterpret_cast<uint32_t*>(code + c.n_my * kEwBlocks), sh);
    } else {
      ew_decide_memory(v, c, d, B.key, B.kind_step, sh, code);
      __syncthreads();
      ew_pack(v, c, S, ew_arrivals(v, S), code, scratch, sh);
    }
    return;
  }
  if constexpr (kForm == kMixed || kForm == kBigList) {
    EwBigList big{scratch, 0u, 0.0f, 0.0};
    const EwAcc first = ew_pass_big(v, c, B.s, big, sh);
    c = ew_chunk(v, ew_opaque(blockIdx.x) - (uint32_t)v.cta0);
    const float lo = big.lo;
    const EwSolved S = ew_solve(v, c, B.s, first, [&](float theta) {
      // (a barrier has passed since the pass)
      return *(volatile uint32_t*)&sh.big_over == 0u && theta >= lo ? ew_round_list(v, c, big, theta, sh) : ew_round_memory(v, c, theta);
    }, sh);
    if (c.index == 0 && tid == 0) ew_store_state(v, S);
    ew_decide_memory(v, c, ew_decide_of(S), B.key, B.kind_step, sh, code);
    __syncthreads();
    ew_pack(v, c, S, ew_arrivals(v, S), code, scratch, sh);
  }
}

// The two-kernel form: the solve leaves its result in the state record; a CTA of the second kernel takes the next chunk of
// consecutive tiles by ticket, so that every chunk it will wait for is already running, however many waves the grid takes.
__global__ void __launch_bounds__(kEwThreads, 1) ew_solve_kernel(const __grid_constant__ EwBatch<1> B, int n_pack_chunks) {
  __shared__ EwShared sh;
  __shared__ uint32_t s_big[kEwBig * kEwThreads];
  const EwVec& v = B.v[0];
  const EwChunk c = ew_chunk(v, blockIdx.x);
  const int tid = threadIdx.x;
  if (tid == 0) { sh.big_over = 0u; sh.stop = 0u; sh.fail = 0u; }
  if (blockIdx.x == 0) {
    ew_write_headers(v, B.begin, true);
    if (tid == 0) { *v.ticket = 0u; v.state->list_chunks = 0u; }
  }
  for (int i = blockIdx.x * kEwThreads + tid; i < n_pack_chunks; i += gridDim.x * kEwThreads) v.chunk_status[i] = 0ull;   // for the second kernel
  __syncthreads();
  EwBigList big{s_big, 0u, 0.0f, 0.0};
  const EwAcc first = ew_pass_big(v, c, B.s, big, sh);
  const float lo = big.lo;
  const EwSolved S = ew_solve(v, c, B.s, first, [&](float theta) {
    return *(volatile uint32_t*)&sh.big_over == 0u && theta >= lo ? ew_round_list(v, c, big, theta, sh) : ew_round_memory(v, c, theta);
  }, sh);
  if (blockIdx.x == 0 && tid == 0) ew_store_state(v, S);
  if (tid == 0 && sh.fail) raise_status(v.hdr, ATOMO_ERR_TIMEOUT);
  // nobody publishes here: the CTAs count themselves out, and the last one leaves both counters at zero
  if (v.n_ctas > 1 && tid == 0 && atomicAdd(v.barrier + 1, 1u) == (uint32_t)v.n_ctas - 1u) { v.barrier[0] = 0u; v.barrier[1] = 0u; }
}

__global__ void __launch_bounds__(kEwThreads, 1) ew_sample_pack_kernel(const __grid_constant__ EwBatch<1> B) {
  extern __shared__ __align__(16) uint32_t ew_smem[];
  __shared__ EwShared sh;
  __shared__ uint32_t s_ticket;
  const EwVec& v = B.v[0];
  const EwState* st = v.state;
  EwSolved S;
  S.T0 = st->T0; S.scale = st->scale; S.theta = st->theta; S.c = st->c; S.n_sat = st->n_sat; S.rounds = st->rounds; S.amax = st->amax;
  S.nonfinite = st->nonfinite != 0;
  if (threadIdx.x == 0) { s_ticket = atomicAdd(v.ticket, 1u); sh.fail = 0u; }
  __syncthreads();
  const EwChunk c = ew_chunk(v, s_ticket);
  uint8_t* const code = reinterpret_cast<uint8_t*>(ew_smem + B.scratch_words);
  ew_decide_memory(v, c, ew_decide_of(S), B.key, B.kind_step, sh, code);
  __syncthreads();
  ew_pack(v, c, S, 0u, code, ew_smem, sh);
}

// ---- decode -------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t lower_bound_u32(const uint32_t* __restrict__ a, uint32_t n, uint64_t key) {
  uint32_t lo = 0, hi = n;
  while (lo < hi) { const uint32_t mid = (lo + hi) >> 1; if ((uint64_t)__ldg(a + mid) < key) lo = mid + 1; else hi = mid; }
  return lo;
}

// What a decoder needs of one vector of a payload; nothing is kept where the header does not fit the shapes
struct EwSource {
  const uint32_t* idx; const uint16_t* ent; const float* val; const uint32_t* table; const uint32_t* sat_idx;
  uint32_t k, n_sat; float c; bool compact, ok;
};
__device__ __forceinline__ EwSource ew_source(const uint8_t* payload, const int layer, const int64_t n) {
  const atomo_payload_header* gh = reinterpret_cast<const atomo_payload_header*>(payload);
  const atomo_layer_header* h = reinterpret_cast<const atomo_layer_header*>(payload + sizeof(atomo_payload_header)) + layer;
  EwSource r;
  r.compact = gh->ew_format == ATOMO_EW_COMPACT;
  const uint32_t sat_cap = r.compact ? (uint32_t)min(gh->ew_sat_cap, (uint64_t)0xFFFFFFFFull) : 0u;
  r.ok = gh->magic == ATOMO_MAGIC && gh->kind == ATOMO_KIND_ENTRYWISE && gh->ew_format <= ATOMO_EW_COMPACT &&
         h->rows == 1 && h->cols == n;
  if (r.compact) r.ok = r.ok && h->n_sat <= h->k && h->n_sat <= sat_cap && h->k - h->n_sat <= h->k_cap;
  else r.ok = r.ok && h->k <= h->k_cap;
  r.n_sat = (r.ok && r.compact) ? h->n_sat : 0u;
  r.k = r.ok ? h->k - r.n_sat : 0u;                        // entries of the idx / entry list
  r.c = h->c;
  r.idx = reinterpret_cast<const uint32_t*>(payload + h->off_idx);
  r.ent = reinterpret_cast<const uint16_t*>(payload + h->off_idx);
  r.val = reinterpret_cast<const float*>(payload + h->off_val);
  r.table = reinterpret_cast<const uint32_t*>(payload + h->off_short);   // list entries before each tile
  r.sat_idx = reinterpret_cast<const uint32_t*>(payload + h->off_long);
  return r;
}
__device__ __forceinline__ void ew_raise_payload(const uint8_t* payload, const int layer) {
  raise_status(reinterpret_cast<atomo_layer_header*>(const_cast<uint8_t*>(payload) + sizeof(atomo_payload_header)) + layer, ATOMO_ERR_PAYLOAD);
}

// A tile from shared memory to the output: one bulk copy where the output allows it (16-byte base), plain stores for the
// rest.  Called by every thread of the CTA after its last write to the tile.
__device__ __forceinline__ void ew_tile_out(float* __restrict__ out, const float* __restrict__ s_tile, const int64_t left, const int threads) {
  const bool bulk = (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
  const int n = (int)min(left, (int64_t)kEwTile), n_bulk = bulk ? n & ~3 : 0;
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && n_bulk > 0) {
    const uint32_t src = (uint32_t)__cvta_generic_to_shared(s_tile);
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(out), "r"(src), "r"(n_bulk * 4) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
  for (int i = n_bulk + threadIdx.x; i < n; i += threads) out[i] = s_tile[i];
  if (threadIdx.x == 0 && n_bulk > 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the tile may go now
}

// One tile per CTA, all vectors of the call in one launch.  Bound: HBM writes.  The tile is zeroed and filled in shared
// memory and leaves as one 16 KB bulk copy, so the L2 sees whole lines only (zero stores followed by the kept values as
// 4-byte stores of their own, behind a barrier, took 21.4 us for 25.6 M elements at 1 % and 106 us for 100 M at 10 %).
// Small CTAs, so that a dozen tiles per SM overlap their chains header -> tile table -> entries.
constexpr int kEwDecThreads = 128;
template <int N>
__global__ void __launch_bounds__(kEwDecThreads) ew_decode_kernel(const __grid_constant__ EwDecodeBatch<N> B) {
  __shared__ __align__(128) float s_tile[kEwTile];
  int vi = 0;
  if (N > 1) while (vi + 1 < B.n && blockIdx.x >= B.v[vi + 1].tile0) ++vi;
  const EwDecode& d = B.v[vi];
  const int64_t tile = blockIdx.x - d.tile0, tile_base = tile * kEwTile, left = d.n - tile_base;
  const int tid = threadIdx.x;
  const EwSource s = ew_source(B.payload, d.layer, d.n);
  if (!s.ok && tile == 0 && tid == 0) ew_raise_payload(B.payload, d.layer);
  uint32_t lo = 0, hi = 0;
  if (s.k) { lo = min(__ldg(s.table + tile), s.k); hi = min(__ldg(s.table + tile + 1), s.k); }
#pragma unroll
  for (int i = 0; i < kEwTile / 4 / kEwDecThreads; ++i) reinterpret_cast<float4*>(s_tile)[tid + i * kEwDecThreads] = make_float4(0.f, 0.f, 0.f, 0.f);
  // the first entries are on their way while the zeros settle
  uint32_t j = lo + tid, i0 = 0;
  float v0 = 0.0f;
  if (j < hi) {
    if (!s.compact) { i0 = __ldg(s.idx + j) - (uint32_t)tile_base; v0 = __ldg(s.val + j); }
    else { const uint32_t e = __ldg(s.ent + j); i0 = e & (uint32_t)(kEwTile - 1); v0 = (e & 0x8000u) ? -s.c : s.c; }
  }
  __syncthreads();
  while (j < hi) {
    if (i0 < (uint32_t)kEwTile) s_tile[i0] = v0;
    j += kEwDecThreads;
    if (j < hi) {
      if (!s.compact) { i0 = __ldg(s.idx + j) - (uint32_t)tile_base; v0 = __ldg(s.val + j); }
      else { const uint32_t e = __ldg(s.ent + j); i0 = e & (uint32_t)(kEwTile - 1); v0 = (e & 0x8000u) ? -s.c : s.c; }
    }
  }
  if (s.n_sat) {                                           // compact: the saturated atoms of this tile (ascending list)
    for (uint32_t q = lower_bound_u32(s.sat_idx, s.n_sat, (uint64_t)tile_base) + tid; q < s.n_sat; q += kEwDecThreads) {
      const int64_t off = (int64_t)__ldg(s.sat_idx + q) - tile_base;
      if (off >= kEwTile) break;
      if (off >= 0) s_tile[off] = __ldg(s.val + q);
    }
  }
  ew_tile_out(d.out + tile_base, s_tile, left, kEwDecThreads);
}

// ---- decode and average ---------------------------------------------------------------------------
// out = (1/P) sum over the payloads (combine step of data-parallel training, Section 2): a tile per CTA in shared memory
// receives payload 0's kept values, then payload 1's, ... (indices are unique inside a payload, so no two threads meet
// between barriers) and leaves once; explicit and compact payloads may be mixed.  Bound: HBM writes.  The payloads'
// headers and table entries are fetched by one thread each, then the entries of all of them, as one sequence of up to
// 2048 at a time, before the first is added: the chain of dependent loads is paid once per tile instead of once per
// payload (88 us for eight payloads of 25.6 M elements at 1 % with a payload at a time).  A window is instantiated for one, two, four or
// eight entries per thread: with eight always, of which two were in use at 1 %, most instructions did nothing (73.6 -> 61.4 us).
constexpr int kAvgThreads = 256, kAvgPer = 8, kAvgPayloads = 64;     // payloads per round: their ranges sit in shared memory
struct AvgSource { const void* idx; const float* val; const uint32_t* sat_idx; uint32_t lo, sat_begin, n_sat, compact; float c; };
template <int N>
__global__ void __launch_bounds__(kAvgThreads) ew_decode_average_kernel(const __grid_constant__ EwDecodeBatch<N> B,
                                                                        const uint8_t* const* __restrict__ payloads,
                                                                        const int n_payloads, const float inv_p) {
  __shared__ __align__(128) float s_tile[kEwTile];
  __shared__ AvgSource s_src[kAvgPayloads];
  __shared__ uint32_t s_begin[kAvgPayloads + 1];             // entries of the earlier payloads of the round
  int vi = 0;
  if (N > 1) while (vi + 1 < B.n && blockIdx.x >= B.v[vi + 1].tile0) ++vi;
  const EwDecode& d = B.v[vi];
  const int64_t tile = blockIdx.x - d.tile0, tile_base = tile * kEwTile, left = d.n - tile_base;
  const int tid = threadIdx.x;
#pragma unroll
  for (int i = 0; i < kEwTile / 4 / kAvgThreads; ++i) reinterpret_cast<float4*>(s_tile)[tid + i * kAvgThreads] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int p0 = 0; p0 < n_payloads; p0 += kAvgPayloads) {
    const int np = min(kAvgPayloads, n_payloads - p0);
    __syncthreads();                                       // the previous round has used the ranges
    if (tid < np) {
      const uint8_t* payload = payloads[p0 + tid];
      const EwSource s = ew_source(payload, d.layer, d.n);
      if (!s.ok && tile == 0) ew_raise_payload(payload, d.layer);
      uint32_t lo = 0, hi = 0;
      if (s.k) { lo = min(__ldg(s.table + tile), s.k); hi = min(__ldg(s.table + tile + 1), s.k); }
      const uint32_t sat0 = s.n_sat ? lower_bound_u32(s.sat_idx, s.n_sat, (uint64_t)tile_base) : 0u;
      s_src[tid] = AvgSource{s.idx, s.val, s.sat_idx, lo, sat0, s.n_sat, s.compact ? 1u : 0u, s.c};
      s_begin[tid + 1] = hi > lo ? hi - lo : 0u;
    }
    __syncthreads();
    if (tid == 0) {
      uint32_t run = 0;
      s_begin[0] = 0;
      for (int p = 0; p < np; ++p) { run += s_begin[p + 1]; s_begin[p + 1] = run; }
    }
    __syncthreads();
    const uint32_t total = s_begin[np];
    int p_next = 0;                                        // payloads before it are complete
    auto add_saturated = [&](int p) {                      // compact: the atoms with p = 1, none of them in the entry list
      const AvgSource& s = s_src[p];
      for (uint32_t q = s.sat_begin + tid; q < s.n_sat; q += kAvgThreads) {
        const int64_t off = (int64_t)__ldg(s.sat_idx + q) - tile_base;
        if (off >= kEwTile) break;
        if (off >= 0) s_tile[off] += __ldg(s.val + q);
      }
    };
    // a window of kPer entries per thread
    auto window = [&](const uint32_t e0, auto per_tag) {
      constexpr int kPer = decltype(per_tag)::value;
      // this thread's entries of the window: element, value, payload
      uint32_t el[kPer]; float vl[kPer]; int pl[kPer];
      int p = 0;
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const uint32_t e = e0 + (uint32_t)(q * kAvgThreads) + tid;
        el[q] = kEwTile; vl[q] = 0.0f; pl[q] = np;
        if (e < total) {
          while (e >= s_begin[p + 1]) ++p;
          const AvgSource& s = s_src[p];
          const uint32_t j = s.lo + (e - s_begin[p]);
          pl[q] = p;
          if (!s.compact) {
            el[q] = __ldg(reinterpret_cast<const uint32_t*>(s.idx) + j) - (uint32_t)tile_base;
            vl[q] = __ldg(s.val + j);
          } else {
            const uint32_t en = __ldg(reinterpret_cast<const uint16_t*>(s.idx) + j);
            el[q] = en & (uint32_t)(kEwTile - 1);
            vl[q] = (en & 0x8000u) ? -s.c : s.c;
          }
        }
      }
      const uint32_t e_end = min(e0 + (uint32_t)(kAvgThreads * kPer), total);
      for (int pp = p_next; pp < np && s_begin[pp] < e_end; ++pp) {     // payload by payload, in array order
#pragma unroll
        for (int q = 0; q < kPer; ++q) if (pl[q] == pp && el[q] < (uint32_t)kEwTile) s_tile[el[q]] += vl[q];
        if (s_begin[pp + 1] <= e_end) { add_saturated(pp); p_next = pp + 1; }
        __syncthreads();
      }
    };
    for (uint32_t e0 = 0; e0 < total; e0 += kAvgThreads * kAvgPer) {   // (uniform: as many entries per thread as the window has)
      const uint32_t left_e = total - e0;
      if (left_e <= kAvgThreads) window(e0, std::integral_constant<int, 1>{});
      else if (left_e <= 2 * kAvgThreads) window(e0, std::integral_constant<int, 2>{});
      else if (left_e <= 4 * kAvgThreads) window(e0, std::integral_constant<int, 4>{});
      else window(e0, std::integral_constant<int, kAvgPer>{});
    }
    for (; p_next < np; ++p_next) if (s_src[p_next].n_sat) { add_saturated(p_next); __syncthreads(); }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kEwTile / 4 / kAvgThreads; ++i) {
    float4& t = reinterpret_cast<float4*>(s_tile)[tid + i * kAvgThreads];
    t = make_float4(t.x * inv_p, t.y * inv_p, t.z * inv_p, t.w * inv_p);
  }
  ew_tile_out(d.out + tile_base, s_tile, left, kAvgThreads);
}

// ---- l_q budget (Section 4: the budget s = ||g||_1 / ||g||_q turns entry-wise ATOMO into QSGD for q = 2 and
//      into TernGrad for q = infinity) --------------------------------------------------------------------
// pass 0: sum |g|, max |g| and sum g^2 (fp64: the squares of fp32 numbers neither overflow nor vanish there, so q = 2 needs
// no scaling and one read of the vector); pass 1 (other finite q > 1): sum (|g| / amax)^q.  fp64 sums, added up by the last
// CTA in a fixed order into host memory.  Bound: HBM (two passes with 4-byte loads and a host-side sum of the CTAs' parts
// took 2 x 85 us for 25.6 M elements, where one read is 16 us).
constexpr int kLqThreads = 256, kLqWarps = kLqThreads / kWarp;
__global__ void __launch_bounds__(kLqThreads) ew_lq_kernel(const float* __restrict__ g, int64_t n, int pass, double q,
                                                           double inv_amax, EwLqPart* __restrict__ part, uint32_t* __restrict__ ticket,
                                                           EwLqPart* __restrict__ result) {
  __shared__ double s_sum[kLqWarps], s_sq[kLqWarps];
  __shared__ float s_max[kLqWarps];
  __shared__ uint32_t s_last;
  const int tid = threadIdx.x, lane = tid % kWarp, w = tid / kWarp;
  const bool aligned = (reinterpret_cast<uintptr_t>(g) & 15u) == 0;
  double sum = 0.0, sq = 0.0;
  float amax = 0.0f;
  auto one = [&](float x) {
    const float a = fabsf(x);
    if (pass == 0) {
      const double d = (double)a;
      sum += d; sq = fma(d, d, sq); amax = fmaxf(amax, a);
      if (!(a <= 3.0e38f)) amax = __int_as_float(0x7f800000);
    } else if (a > 0.0f) sum += pow((double)a * inv_amax, q);
  };
  const int64_t n4 = aligned ? n / 4 : 0, stride = (int64_t)gridDim.x * kLqThreads;
  for (int64_t i = (int64_t)blockIdx.x * kLqThreads + tid; i < n4; i += 4 * stride) {
    float4 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = i + u * stride < n4 ? __ldg(reinterpret_cast<const float4*>(g) + i + u * stride) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 4; ++u) { one(x[u].x); one(x[u].y); one(x[u].z); one(x[u].w); }
  }
  for (int64_t i = 4 * n4 + (int64_t)blockIdx.x * kLqThreads + tid; i < n; i += stride) one(__ldg(g + i));
  auto reduce = [&]() {
    sum = warp_sum(sum); sq = warp_sum(sq); amax = warp_max(amax);
    __syncthreads();
    if (lane == 0) { s_sum[w] = sum; s_sq[w] = sq; s_max[w] = amax; }
    __syncthreads();
    sum = 0.0; sq = 0.0; amax = 0.0f;
    for (int i = 0; i < kLqWarps; ++i) { sum += s_sum[i]; sq += s_sq[i]; amax = fmaxf(amax, s_max[i]); }   // fixed order
  };
  reduce();
  if (tid == 0) {
    part[blockIdx.x] = EwLqPart{sum, sq, (double)amax};
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1 ? 1u : 0u;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  sum = 0.0; sq = 0.0; amax = 0.0f;
  for (int i = tid; i < (int)gridDim.x; i += kLqThreads) {
    sum += __ldcg(&part[i].sum); sq += __ldcg(&part[i].sq); amax = fmaxf(amax, (float)__ldcg(&part[i].amax));
  }
  reduce();
  if (tid == 0) { *ticket = 0u; *result = EwLqPart{sum, sq, (double)amax}; }
}

}  // namespace

// ---- host-side launchers --------------------------------------------------------------------------
void launch_ew_lq(const float* g, int64_t n, int pass, double q, double inv_amax, EwLqPart* part, uint32_t* ticket,
                  EwLqPart* result, int max_ctas, cudaStream_t st) {
  const int ctas = (int)std::max<int64_t>(1, std::min<int64_t>(max_ctas, (n + 16 * kLqThreads - 1) / (16 * kLqThreads)));
  ew_lq_kernel<<<ctas, kLqThreads, 0, st>>>(g, n, pass, q, inv_amax, part, ticket, result);
}

namespace {
int ew_sms() {
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}
// the slots of the candidate list; else the staging windows (or the list of runs with large atoms)
size_t ew_scratch_bytes(bool list) { return list ? (size_t)kEwCandBytes : std::max((size_t)kEwWarps * kEwStage * sizeof(uint16_t), (size_t)kEwBig * kEwThreads * sizeof(uint32_t)); }
static_assert(kEwCandBytes >= kEwWarps * kEwStage * 2 && kEwCandBytes >= kEwBig * kEwThreads * 4, "the scratch area serves in turn");
size_t ew_dyn_bytes(int tiles, bool list) {
  return ew_scratch_bytes(list) + (size_t)tiles * (kEwBlocks + (list ? kEwPrefixes * sizeof(uint32_t) : 0));
}
constexpr size_t kEwMaxDyn = 225 * 1024;            // dynamic shared memory of a CTA (227 KB less the static part)
constexpr int kEwPackTiles = 64;                    // tiles per chunk of the two-kernel form
}  // namespace

int ew_configure() {
  const void* fns[] = {(const void*)ew_encode_kernel<1, kMixed>, (const void*)ew_encode_kernel<1, kRegisters>, (const void*)ew_encode_kernel<1, kCandidates>,
                       (const void*)ew_encode_kernel<1, kBigList>, (const void*)ew_encode_kernel<kEwBatch, kMixed>,
                       (const void*)ew_encode_kernel<kEwBatch, kRegisters>, (const void*)ew_sample_pack_kernel};
  for (const void* f : fns) {
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEwMaxDyn);
    if (e != cudaSuccess) return (int)e;
  }
  for (const void* f : {(const void*)ew_decode_kernel<1>, (const void*)ew_decode_kernel<kEwBatch>, (const void*)ew_decode_average_kernel<1>,
                        (const void*)ew_decode_average_kernel<kEwBatch>}) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return (int)e;
  }
  return 0;
}

// Chunks of equal size (in tiles) over all vectors, as small as one wave of resident CTAs allows: the fewer tiles a CTA
// walks over, the shorter the chain between two barriers.  Sets n_ctas and cta0; 0 if the vectors do not fit one wave.
int ew_plan(EwVec* v, int n_vecs, bool list) {
  const int sms = ew_sms();
  int64_t total = 0;
  for (int i = 0; i < n_vecs; ++i) total += v[i].n_tiles;
  for (int64_t t = std::max<int64_t>(1, total / sms); ew_dyn_bytes((int)std::min<int64_t>(t, 4096), list) <= kEwMaxDyn; ++t) {
    int64_t ctas = 0;
    for (int i = 0; i < n_vecs; ++i) ctas += (v[i].n_tiles + t - 1) / t;
    if (ctas > sms) continue;
    int at = 0;
    for (int i = 0; i < n_vecs; ++i) { v[i].n_ctas = (int)((v[i].n_tiles + t - 1) / t); v[i].cta0 = at; at += v[i].n_ctas; }
    return at;
  }
  return 0;
}
// Whether the candidate list pays for a vector of n elements at budget s in n_ctas chunks.  A thread expects 1.25 s (its
// atoms) / n candidates and has kEwCandPerThread slots: beyond a quarter of them overflows become likely; and with more
// than a quarter of the blocks listed (budgets above 5 % of the length) the decisions on the list cost what the second
// read does.  A chunk that fits the registers needs no list.
bool ew_list_pays(int64_t n, int64_t n_tiles, int n_ctas, double s) {
  const int64_t tiles = (n_tiles + n_ctas - 1) / n_ctas;
  if (tiles <= kEwRegTiles || 1.25 * s * 4.0 > 0.25 * (double)n) return false;
  return 1.25 * s * (double)(tiles * kEwTile) / ((double)n * kEwThreads) <= 0.25 * kEwCandPerThread;
}

template <int N>
int launch_ew_encode(EwBatch<N>& B, bool list, cudaStream_t st) {
  int64_t most = 1;
  int ctas = 0;
  bool waits = false;                                // CTAs that wait for one another have to be resident together
  for (int i = 0; i < B.n; ++i) {
    most = std::max(most, (B.v[i].n_tiles + B.v[i].n_ctas - 1) / B.v[i].n_ctas);
    ctas += B.v[i].n_ctas;
    waits |= B.v[i].n_ctas > 1;
  }
  B.scratch_words = (int)(ew_scratch_bytes(list) / sizeof(uint32_t));
  const size_t smem = ew_dyn_bytes((int)most, list);
  // the instance for what the chunks are (a vector's chunks differ by one tile: those beside the bound may be of two kinds); calls
  // with several vectors are either all short or mixed
  bool all_reg = true, all_cand = true, all_big = true;
  for (int i = 0; i < B.n; ++i) {
    const EwVec& v = B.v[i];
    const bool reg = v.prob_out == nullptr && !v.candidates;   // may keep short chunks in registers
    all_reg &= reg && (v.n_tiles + v.n_ctas - 1) / v.n_ctas <= kEwRegTiles;
    all_cand &= v.candidates != 0;
    all_big &= !v.candidates && (!reg || v.n_tiles / v.n_ctas > kEwRegTiles);
  }
  const void* fn = (const void*)ew_encode_kernel<N, kMixed>;
  if (all_reg) fn = (const void*)ew_encode_kernel<N, kRegisters>;
  else if constexpr (N == 1) { if (all_cand) fn = (const void*)ew_encode_kernel<1, kCandidates>; else if (all_big) fn = (const void*)ew_encode_kernel<1, kBigList>; }
  void* args[] = {&B};
  if (!waits) return (int)cudaLaunchKernel(fn, dim3((unsigned)ctas), dim3(kEwThreads), args, smem, st);
  return (int)cudaLaunchCooperativeKernel(fn, dim3((unsigned)ctas), dim3(kEwThreads), args, smem, st);
}
template int launch_ew_encode<1>(EwBatch<1>&, bool, cudaStream_t);
template int launch_ew_encode<kEwBatch>(EwBatch<kEwBatch>&, bool, cudaStream_t);

int ew_solve_ctas(int64_t n_tiles) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ew_solve_kernel, kEwThreads, 0) != cudaSuccess || per_sm < 1) { cudaGetLastError(); return 0; }
  return (int)std::min<int64_t>(n_tiles, (int64_t)ew_sms() * per_sm);
}
int ew_pack_ctas(int64_t n_tiles) {
  return (int)std::max<int64_t>((n_tiles + kEwPackTiles - 1) / kEwPackTiles, std::min<int64_t>(n_tiles, (int64_t)ew_sms()));
}
// (the two take the same batch, one after the other)
int launch_ew_solve(EwBatch<1>& B, int solve_ctas, int pack_ctas, cudaStream_t st) {
  B.v[0].n_ctas = solve_ctas; B.v[0].cta0 = 0;
  void* args[] = {&B, &pack_ctas};
  return (int)cudaLaunchCooperativeKernel((const void*)ew_solve_kernel, dim3((unsigned)solve_ctas), dim3(kEwThreads), args, 0, st);
}
int launch_ew_sample_pack(EwBatch<1>& B, int pack_ctas, cudaStream_t st) {
  B.v[0].n_ctas = pack_ctas; B.v[0].cta0 = 0;
  B.scratch_words = (int)(ew_scratch_bytes(false) / sizeof(uint32_t));
  const int64_t most = (B.v[0].n_tiles + pack_ctas - 1) / pack_ctas;
  ew_sample_pack_kernel<<<(unsigned)pack_ctas, kEwThreads, ew_dyn_bytes((int)most, false), st>>>(B);
  return (int)cudaGetLastError();
}
template <int N>
void launch_ew_decode(const EwDecodeBatch<N>& B, uint32_t n_tiles, cudaStream_t st) {
  ew_decode_kernel<N><<<n_tiles, kEwDecThreads, 0, st>>>(B);
}
template void launch_ew_decode<1>(const EwDecodeBatch<1>&, uint32_t, cudaStream_t);
template void launch_ew_decode<kEwBatch>(const EwDecodeBatch<kEwBatch>&, uint32_t, cudaStream_t);
template <int N>
void launch_ew_decode_average(const EwDecodeBatch<N>& B, uint32_t n_tiles, const uint8_t* const* d_payloads, int n_payloads, cudaStream_t st) {
  ew_decode_average_kernel<N><<<n_tiles, kAvgThreads, 0, st>>>(B, d_payloads, n_payloads, 1.0f / (float)n_payloads);
}
template void launch_ew_decode_average<1>(const EwDecodeBatch<1>&, uint32_t, const uint8_t* const*, int, cudaStream_t);
template void launch_ew_decode_average<kEwBatch>(const EwDecodeBatch<kEwBatch>&, uint32_t, const uint8_t* const*, int, cudaStream_t);
int ew_tile_elems() { return kEwTile; }

}  // namespace atomo
