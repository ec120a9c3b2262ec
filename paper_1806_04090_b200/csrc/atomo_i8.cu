// Gram matrix of the short side on the 5th-generation tensor cores from 8-bit integers: layers with a short side above 1024, all that the
// TF32 kernel (atomo_tc.cu) cannot take (tall, or rows that do not start on 16-byte boundaries) but for very short or
// narrow ones, and those of 513 to 1024 rows where a call has many elements of them.
//
//   sp_i8_row_kernel    vector i in units of 2^(E_i - 30), 2^E_i above its largest magnitude, rounded to integers, written as four
//                       signed base-256 digits in four planes [digit][i][k], contiguous along the contraction whatever G's layout:
//                       rows of up to 8192 entries, a CTA each, which stay in registers between the maximum and the digits
//   sp_i8_max_kernel, sp_i8_slice_kernel   the same in two passes over G: longer rows, and the columns of tall layers
//   sp_gram_i8_kernel   A_ij = sum over digit pairs (p, q), p + q <= 3, of integer products: ten MMAs (kind::i8) per 32 columns into four
//                       32-bit accumulators, one per weight p + q.  Integer sums are exact; the four sums meet in 64 bits.
//                       Tiles with wide vectors: the other six pairs in a pass ahead, whose sum weight 3 starts from.
//   sp_gram_coarse_kernel (atomo_spectral.cu)   tiles with vectors wider still, from fp32 products over what the integers left
//
// Precision.  A typical sum off the diagonal is s = sqrt(L) times the two vectors' r.m.s. entries; the fp32 FMA kernel's runs of 32 products
// round at 2^-23.8 of it.  Here the pairs left out are 2^-30.8 of s times the two vectors' peaks (2^E over the r.m.s. entry: 4 to 8 for
// Gaussian rows): 2^-26 of s for such rows, as much as the FMA kernel's rounding where the peaks multiply to 128.  Tiles above that
// take all sixteen pairs, 1.6 times the MMAs (two layers of 4096 x 4096 517 us | 837).  What is left then is the rounding of an entry, once, at
// 2^-31 of its vector's largest (entries above a 64th of it not at all).  It falls behind fp32 products where an entry of 2^8
// times the bulk meets another vector's bulk: a vector of which a quarter of the entries (zeros aside) is below 2^(E - 9) gets its
// tiles of 64 from the FMA kernel (6.4 ms for two layers of 4096 rows, as before there were integers; nothing but the launch, 2 us, otherwise).
// Against 64 bits, without the second and third form | with them | FMA kernel, median angle of 48 kept vectors' to the exact ones, 1030 x 4100:
// one entry of 100 per row 5.4e-5 | 1.8e-5 | 1.6e-5, of 1000 2.6e-4 | 1.2e-4 | 1.2e-4, Student t with 2 degrees of freedom 2.2e-5 | 1.5e-5 |
// 1.5e-5, Gaussian 1.3e-5 | 1.3e-5 | 1.4e-5.
// On the diagonal the left-out squares have one sign and would lower every eigenvalue (the nuclear norm of 2000 x 2048 with few strong directions by 5e-6):
// the slicing kernel adds them up, and the diagonal's entries get them back.  Singular values of 2000 x 2048 noise, FMA kernel | this
// one, r.m.s. over six seeds: ||sigma - exact|| / ||sigma|| 5.4e-8 | 5.6e-8, under few strong directions 5.0e-6 | 4.6e-6 (the rounding of A to
// fp32 and the reduction, common to both); 1024 x 4096, TF32 kernel | this one: 1.35e-7 | 2.9e-8.  The TF32 kernel's accumulator
// truncates, which is why the larger layers never took it.
// An accumulator holds parts of up to 32768 columns (at most 49408 per column in magnitude, 2^31 in all).  A tile's columns are split
// over several CTAs while the GPU has SMs left; the parts are integers of up to 2^36 per column, so that up to 131072 columns their sum in fp64 is exact and
// does not depend on the split (the pass ahead rounds its sum to weight 3 once per part: there the last bit of an entry of A may).
// Longer layers' parts are added with fp64 rounding, in their order: 2^-53 of the sum.
//
// One CTA per 128 x 128 tile of the upper triangle, all 512 columns of the tensor memory.
//   warp 0      TMA producer: 64 columns of 128 vectors, four digits (32 KB a side, 64-byte swizzle), no multicast
//   warp 1      allocates TMEM and issues the MMAs from one lane; tcgen05.commit frees a stage
//   warps 2-5   at the end: TMEM -> fp64 -> shared memory -> both triangles of A
// Every mbarrier wait is bounded; a wait that runs out sets an error word and the CTA leaves through the common exit (TMEM is freed).
// Bound: the tensor cores (1430 cycles per stage of 64 columns, 1280 of them twenty MMAs of 128 x 128 x 32), and the last wave of CTAs
// (1056 tiles of two layers of 4096 rows on 148 SMs).  Before (fp32 FMA kernel, or TF32) | now with the digits, us: two layers of
// 4096 x 4096 6390 | 593, nine of 2048 x 2048 3646 | 429, 20 of 1000 x 1201 1174 | 260, 96 of 1024 x 4096 2818 | 2230.  The sums' way out
// of the tensor memory took 31 k cycles per tile with 64-bit integer conversions and a store per entry and row, a third of that now.
// The vectors' ranges and the second group cost 5 % (96 layers: digits 595 -> 645 us, this kernel 1523 -> 1586): the digits' squares and products by __dp4a on the words
// that are written anyway (40 % with integer arithmetic per entry).
#include <algorithm>

#include "atomo_kernels.cuh"
#include "atomo_umma.cuh"

namespace atomo {

namespace {
constexpr int kI8Tile = 128;                       // output tile edge (UMMA M = N = 128)
constexpr int kI8K = 64;                           // columns per stage = one 64-byte swizzle atom
constexpr int kI8Stages = 3;
constexpr int kI8PlaneBytes = kI8Tile * kI8K;      // 8 KB
constexpr int kI8SideBytes = 4 * kI8PlaneBytes;
constexpr int kI8StageBytes = 2 * kI8SideBytes;    // 64 KB
constexpr int kI8Threads = 192;
constexpr int kI8SmemBytes = kI8Stages * kI8StageBytes + 1024 /*alignment slack*/ + 128 /*barriers*/;
constexpr uint32_t kI8TmemCols = 512;              // four 128-column accumulators
constexpr int kI8PartK = 32768;                    // columns that an accumulator holds
// the two preparing kernels' tiles: short x long side
constexpr int kI8WideRows = 16, kI8WideCols = 1024, kI8TallCols = 64, kI8TallRows = 128;
constexpr int kI8RowLen = 8192;                    // longest row that the registers of a CTA hold
// a vector's peak is 2^E over the r.m.s. of its entries: tiles in which a row's and a column's multiply to more than this take all digit pairs
constexpr float kI8WidePeaks = 128.0f;

// exponent with |x| < 2^E for every x up to the magnitude whose bits these are
__device__ __forceinline__ int i8_exponent(uint32_t bits) { return max((int)(bits >> 23), 1) - 126; }
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

// an integer as a double: 2^52 + 2^31 + x has x in its last bits (one addition; the conversions run at a quarter of its rate)
__device__ __forceinline__ double i8_double(int x) { return __hiloint2double(0x43300000, x ^ (int)0x80000000) - 4503601774854144.0; }

// kind::i8: signed 8-bit A and B, 32-bit integer accumulator, both K-major, M = 128, N = 128
constexpr uint32_t kI8Idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kI8Tile >> 3) << 17) | ((uint32_t)(kI8Tile >> 4) << 24);
// K-major operand, 64-byte swizzle: rows of 64 bytes, 8-row groups 512 bytes apart
__device__ __forceinline__ uint64_t i8_smem_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) /*LBO (unused)*/ | (32ull << 32) /*SBO = 512 B*/ |
         (1ull << 46) /*descriptor version*/ | (4ull << 61) /*SWIZZLE_64B*/;
}
__device__ __forceinline__ void i8_mma(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, {%5, %6, %7, %8}, p;\n\t}\n"
      ::"r"(tmem_d), "l"(da), "l"(db), "r"(kI8Idesc), "r"(accumulate), "r"(0u), "r"(0u), "r"(0u), "r"(0u) : "memory");
}
__device__ __forceinline__ void i8_tma_load(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
               ::"r"(dst), "l"(map), "r"(bar), "r"(x), "r"(y), "r"(0) : "memory");
}
}  // namespace

__global__ void __launch_bounds__(256) sp_i8_max_kernel(const SpLayer* __restrict__ layers, const TileRef* __restrict__ tiles) {
  const TileRef ref = tiles[blockIdx.x];
  const SpLayer& L = layers[ref.layer];
  const float* __restrict__ G = L.G;
  const int64_t ld = L.ld;
  const int r = L.r, len = L.L, tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  if (!L.tall) {                                               // a warp per row: two rows of 1024 entries each
    for (int i = ref.a * kI8WideRows + w; i < min(r, (ref.a + 1) * kI8WideRows); i += 8) {
      const float* g = G + (int64_t)i * ld;
      const int k0 = ref.b * kI8WideCols, n = min(len - k0, kI8WideCols);
      uint32_t m = 0;
#pragma unroll 8
      for (int k = lane; k < n; k += 32) m = max(m, __float_as_uint(__ldg(g + k0 + k)) & 0x7fffffffu);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0) atomicMax(L.i8_max + i, m);
    }
  } else {                                                     // a thread per column, every fourth row
    const int i = ref.a * kI8TallCols + tid % kI8TallCols;
    if (i < r) {
      uint32_t m = 0;
#pragma unroll 8
      for (int k = ref.b * kI8TallRows + tid / kI8TallCols; k < min(len, (ref.b + 1) * kI8TallRows); k += 256 / kI8TallCols)
        m = max(m, __float_as_uint(__ldg(G + (int64_t)k * ld + i)) & 0x7fffffffu);
      atomicMax(L.i8_max + i, m);
    }
  }
}

namespace {
// what a thread has seen of a vector (of 32 of its entries at most)
struct I8Seen { int rest = 0, twice = 0, square = 0; uint32_t counts = 0; };
// four neighbouring entries of a vector, as one word per digit
__device__ __forceinline__ void i8_put(const float (&x)[4], uint32_t bits, int8_t* dst, int64_t plane, I8Seen& seen) {
  // 2^(30 - E) in two factors; a vector with an infinity or a NaN gets zeros here and a NaN for its scale later
  const bool finite = bits < 0x7f800000u;
  const int t = 30 - i8_exponent(bits), half = t >> 1;
  const float s1 = finite ? pow2f(half) : 0.0f, s2 = pow2f(t - half), few = finite ? 2097152.0f : 0.0f;
  uint32_t d[4];
  seen.counts += 0x40000u;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const float y = x[u] * s1 * s2;
    d[u] = ((uint32_t)__float2int_rn(y) + 0x00808080u) ^ 0x00808080u;   // |y| <= 2^30 (or NaN, to 0): the bytes are the signed digits
    seen.counts += fabsf(y) < few ? 1u : 0u;
  }
  if (fminf(fminf(fabsf(x[0]), fabsf(x[1])), fminf(fabsf(x[2]), fabsf(x[3]))) == 0.0f) {   // zeros are not counted
#pragma unroll
    for (int u = 0; u < 4; ++u) seen.counts -= x[u] == 0.0f ? (finite ? 0x10001u : 0x10000u) : 0u;
  }
  // 4 x 4 bytes transposed
  const uint32_t a = __byte_perm(d[0], d[1], 0x5140), b = __byte_perm(d[2], d[3], 0x5140);
  const uint32_t c = __byte_perm(d[0], d[1], 0x7362), e = __byte_perm(d[2], d[3], 0x7362);
  const int w3 = (int)__byte_perm(a, b, 0x5410), w2 = (int)__byte_perm(a, b, 0x7632);
  const int w1 = (int)__byte_perm(c, e, 0x5410), w0 = (int)__byte_perm(c, e, 0x7632);
  *reinterpret_cast<int*>(dst + 3 * plane) = w3;
  *reinterpret_cast<int*>(dst + 2 * plane) = w2;
  *reinterpret_cast<int*>(dst + plane) = w1;
  *reinterpret_cast<int*>(dst) = w0;
  seen.rest = __dp4a(w2, w2, seen.rest);
  seen.twice = __dp4a(w1, w3, seen.twice);
  seen.square = __dp4a(w0, w0, seen.square);
}
__device__ __forceinline__ void i8_add(const I8Seen& seen, I8Stat* to, int lane) {   // (integers: the order does not matter)
  const int rest = __reduce_add_sync(0xffffffffu, seen.rest + 2 * seen.twice), square = __reduce_add_sync(0xffffffffu, seen.square);
  const uint32_t counts = __reduce_add_sync(0xffffffffu, seen.counts);
  if (lane == 0) {
    atomicAdd(&to->rest, (unsigned long long)(long long)rest);
    atomicAdd(&to->square, (unsigned long long)square);
    atomicAdd(&to->counts, (unsigned long long)(counts >> 16) << 32 | (counts & 0xffffu));
  }
}
}  // namespace

// VECS: float4 per thread, rows of up to 1024 VECS entries
template <int VECS>
__device__ __forceinline__ void i8_rows(const SpLayer& L, const int i_lo, const int i_hi, uint32_t (*s_max)[8]) {
  const float* __restrict__ G = L.G;
  const int64_t ld = L.ld, pitch = L.i8_ld, plane = pitch * L.r;
  const int len = L.L, tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const bool vec = (ld % 4 == 0) && ((reinterpret_cast<uintptr_t>(G) & 15u) == 0);
  for (int i = i_lo; i < i_hi; ++i) {
    const float* g = G + (int64_t)i * ld;
    float x[VECS][4];
    uint32_t m = 0;
#pragma unroll
    for (int v = 0; v < VECS; ++v) {
      const int k = 4 * (tid + 256 * v);
      if (vec && k + 3 < len) { const float4 q = __ldg(reinterpret_cast<const float4*>(g + k)); x[v][0] = q.x; x[v][1] = q.y; x[v][2] = q.z; x[v][3] = q.w; }
      else {
#pragma unroll
        for (int u = 0; u < 4; ++u) x[v][u] = k + u < len ? __ldg(g + k + u) : 0.0f;
      }
    }
#pragma unroll
    for (int v = 0; v < VECS; ++v)
#pragma unroll
      for (int u = 0; u < 4; ++u) m = max(m, __float_as_uint(x[v][u]) & 0x7fffffffu);
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) s_max[i & 1][w] = m;
    __syncthreads();                                           // (two rows in turn: a barrier lies between a read and the next write)
#pragma unroll
    for (int q = 0; q < 8; ++q) m = max(m, s_max[i & 1][q]);
    if (tid == 0) L.i8_max[i] = m;
    I8Seen seen;
#pragma unroll
    for (int v = 0; v < VECS; ++v) {
      const int k = 4 * (tid + 256 * v);
      if (k < len) i8_put(x[v], m, L.i8_dig + (int64_t)i * pitch + k, plane, seen);
    }
    i8_add(seen, L.i8_stat + i, lane);
  }
}

__global__ void __launch_bounds__(256) sp_i8_row_kernel(const SpLayer* __restrict__ layers, const TileRef* __restrict__ tiles) {
  __shared__ uint32_t s_max[2][8];
  const TileRef ref = tiles[blockIdx.x];
  const SpLayer& L = layers[ref.layer];
  const int i_lo = ref.a, i_hi = min(L.r, ref.a + ref.c);      // (a few rows, one after the other)
  if (L.L <= 2048) i8_rows<2>(L, i_lo, i_hi, s_max);
  else if (L.L <= 4096) i8_rows<4>(L, i_lo, i_hi, s_max);
  else i8_rows<8>(L, i_lo, i_hi, s_max);
}

__global__ void __launch_bounds__(256) sp_i8_slice_kernel(const SpLayer* __restrict__ layers, const TileRef* __restrict__ tiles) {
  __shared__ float s_x[kI8TallRows][kI8TallCols + 1];
  const TileRef ref = tiles[blockIdx.x];
  const SpLayer& L = layers[ref.layer];
  const float* __restrict__ G = L.G;
  const int64_t ld = L.ld, pitch = L.i8_ld, plane = pitch * L.r;
  const int r = L.r, len = L.L, tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  if (!L.tall) {
    const bool vec = (ld % 4 == 0) && ((reinterpret_cast<uintptr_t>(G) & 15u) == 0);
    for (int i = ref.a * kI8WideRows + w; i < min(r, (ref.a + 1) * kI8WideRows); i += 8) {
      const float* g = G + (int64_t)i * ld;
      const uint32_t bits = L.i8_max[i];
      I8Seen seen;
#pragma unroll 4
      for (int k = ref.b * kI8WideCols + 4 * lane; k < min(len, (ref.b + 1) * kI8WideCols); k += 128) {
        float x[4];
        if (vec && k + 3 < len) { const float4 v = __ldg(reinterpret_cast<const float4*>(g + k)); x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w; }
        else {
#pragma unroll
          for (int u = 0; u < 4; ++u) x[u] = k + u < len ? __ldg(g + k + u) : 0.0f;
        }
        i8_put(x, bits, L.i8_dig + (int64_t)i * pitch + k, plane, seen);
      }
      i8_add(seen, L.i8_stat + i, lane);
    }
  } else {
    const int i0 = ref.a * kI8TallCols, k0 = ref.b * kI8TallRows;
#pragma unroll 8
    for (int q = tid; q < kI8TallRows * kI8TallCols; q += 256) {
      const int kk = q / kI8TallCols, ii = q % kI8TallCols;
      s_x[kk][ii] = k0 + kk < len && i0 + ii < r ? __ldg(G + (int64_t)(k0 + kk) * ld + i0 + ii) : 0.0f;
    }
    __syncthreads();
    const int k = k0 + 4 * lane;
    for (int ii = w; ii < min(kI8TallCols, r - i0); ii += 8) {
      const float x[4] = {s_x[4 * lane][ii], s_x[4 * lane + 1][ii], s_x[4 * lane + 2][ii], s_x[4 * lane + 3][ii]};
      I8Seen seen;
      if (k < pitch) i8_put(x, L.i8_max[i0 + ii], L.i8_dig + (int64_t)(i0 + ii) * pitch + k, plane, seen);
      i8_add(seen, L.i8_stat + i0 + ii, lane);
    }
  }
}

__global__ void __launch_bounds__(kI8Threads, 1) sp_gram_i8_kernel(const SpLayer* __restrict__ layers, const CUtensorMap* __restrict__ maps,
                                                                   const TileRef* __restrict__ tiles, uint32_t* __restrict__ err,
                                                                   uint32_t* __restrict__ coarse) {
  extern __shared__ uint8_t i8_smem[];
  __shared__ double s_scale[2][kI8Tile];                       // 2^(E - 18) of the tile's rows and columns
  __shared__ double s_rest[kI8Tile];                           // what a diagonal tile's squares lack
  __shared__ float s_peak[2 * kI8Tile / 32];                   // by 32 rows or columns: largest squared ratio of 2^E to the r.m.s. entry
  const uint32_t base = (smem_u32(i8_smem) + 1023u) & ~1023u;
  uint8_t* base_ptr = i8_smem + (base - smem_u32(i8_smem));
  const uint32_t bars = base + kI8Stages * kI8StageBytes;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (kI8Stages + s); };
  const uint32_t done_bar = bars + 8u * (2 * kI8Stages), low_bar = done_bar + 8u, start_bar = done_bar + 16u;
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(base_ptr + kI8Stages * kI8StageBytes + 8 * (2 * kI8Stages + 3));
  volatile uint32_t* s_abort = s_tmem + 1;
  volatile uint32_t* s_last = s_tmem + 2;
  const TileRef ref = tiles[blockIdx.x];
  const SpLayer& L = layers[ref.layer];
  const CUtensorMap* map = maps + ref.layer;
  const int ti = ref.a, tj = ref.b, r = L.r;
  const bool diag = ti == tj;
  const int all_kb = (L.L + kI8K - 1) / kI8K, n_split = L.gram_split;
  const int kb_lo = (int)((int64_t)all_kb * ref.c / n_split), num_kb = (int)((int64_t)all_kb * (ref.c + 1) / n_split) - kb_lo;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;

  if (tid == 0) {
    for (int s = 0; s < kI8Stages; ++s) { tc_mbar_init(full_bar(s), 1); tc_mbar_init(empty_bar(s), 1); }
    tc_mbar_init(done_bar, 1);
    tc_mbar_init(low_bar, 1);
    tc_mbar_init(start_bar, 128);
    *s_abort = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int q = tid; q < 2 * kI8Tile; q += kI8Threads) {        // (whole warps)
    const int i = (q < kI8Tile ? ti : tj) * kI8Tile + q % kI8Tile;
    const uint32_t bits = i < r ? L.i8_max[i] : 0u;
    const I8Stat st = i < r ? L.i8_stat[i] : I8Stat{0, 0, 0};
    const float peak = st.square ? (float)L.L * 4096.0f / (float)st.square : 0.0f;
    const uint32_t top = __reduce_max_sync(0xffffffffu, __float_as_uint(peak));
    if (lane == 0) s_peak[q / 32] = __uint_as_float(top);
    if (diag && ref.c == 0 && i8_coarse(st)) *coarse = 1u;
    if (q < kI8Tile) s_rest[q] = diag ? (double)(long long)st.rest * (1.0 / 256.0) : 0.0;
    s_scale[q / kI8Tile][q % kI8Tile] = bits < 0x7f800000u ? __hiloint2double((1023 + i8_exponent(bits) - 18) << 20, 0) : __longlong_as_double(0x7ff8000000000000ll);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32((const void*)s_tmem)), "r"(kI8TmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_d = *s_tmem;
  float peak_i = 0.0f, peak_j = 0.0f;
#pragma unroll
  for (int q = 0; q < kI8Tile / 32; ++q) { peak_i = fmaxf(peak_i, s_peak[q]); peak_j = fmaxf(peak_j, s_peak[kI8Tile / 32 + q]); }
  const bool wide = peak_i * peak_j > kI8WidePeaks * kI8WidePeaks;   // (squares; uniform) the pairs p + q >= 4 as well, ahead of the others
  const int all_it = wide ? 2 * num_kb : num_kb;

  int issued = 0;                                              // (thread 0) stages asked for
  if (warp == 0) {
    if (lane == 0) {
      for (int it = 0; it < all_it; ++it) {
        const int s = it % kI8Stages, kb = it < num_kb ? it : it - num_kb;
        if (!tc_mbar_wait(empty_bar(s), ((uint32_t)(it / kI8Stages) & 1u) ^ 1u, s_abort)) break;
        const uint32_t stage = base + s * kI8StageBytes;
        tc_mbar_expect_tx(full_bar(s), diag ? kI8SideBytes : kI8StageBytes);
        i8_tma_load(stage, map, full_bar(s), (kb_lo + kb) * kI8K, ti * kI8Tile);
        if (!diag) i8_tma_load(stage + kI8SideBytes, map, full_bar(s), (kb_lo + kb) * kI8K, tj * kI8Tile);
        issued = it + 1;
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      bool ok = true;
      int it = 0;
      if (wide) {                                              // weights 4, 5, 6 into the accumulators 0, 1, 2
        for (; it < num_kb; ++it) {
          const int s = it % kI8Stages;
          ok = tc_mbar_wait(full_bar(s), (uint32_t)(it / kI8Stages) & 1u, s_abort);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a = base + s * kI8StageBytes, b = diag ? a : a + kI8SideBytes;
#pragma unroll
          for (int k = 0; k < kI8K / 32; ++k) {
#pragma unroll
            for (int p = 1; p < 4; ++p)
#pragma unroll
              for (int q = 4 - p; q < 4; ++q)
                i8_mma(tmem_d + (uint32_t)((p + q - 4) * kI8Tile), i8_smem_desc(a + p * kI8PlaneBytes + k * 32), i8_smem_desc(b + q * kI8PlaneBytes + k * 32),
                       it > 0 || k > 0 || q < 3 ? 1u : 0u);   // (q = 3 comes first for every weight)
          }
          tc_commit(empty_bar(s));
        }
        if (ok) {
          tc_commit(low_bar);
          ok = tc_mbar_wait(start_bar, 0u, s_abort);
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
      }
      for (; ok && it < all_it; ++it) {
        const int s = it % kI8Stages;
        ok = tc_mbar_wait(full_bar(s), (uint32_t)(it / kI8Stages) & 1u, s_abort);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const bool first = it == all_it - num_kb;
        const uint32_t a = base + s * kI8StageBytes, b = diag ? a : a + kI8SideBytes;
#pragma unroll
        for (int k = 0; k < kI8K / 32; ++k) {                  // UMMA K = 32 bytes
#pragma unroll
          for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q + p < 4; ++q)
              i8_mma(tmem_d + (uint32_t)((p + q) * kI8Tile), i8_smem_desc(a + p * kI8PlaneBytes + k * 32), i8_smem_desc(b + q * kI8PlaneBytes + k * 32),
                     !first || k > 0 || p > 0 || (wide && q == 3) ? 1u : 0u);   // (p = 0 comes first for every weight)
        }
        tc_commit(empty_bar(s));
      }
      if (ok) tc_commit(done_bar);
    }
  } else {
    // warp q of the four reads TMEM lanes 32 q .. 32 q + 31 (q = warp % 4)
    const int q = warp % 4, row = 32 * q + lane;
    auto load16 = [&](int (&v)[16], int col) {
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
            "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
          : "r"(tmem_d + ((uint32_t)(32 * q) << 16) + (uint32_t)col) : "memory");
    };
    if (wide) {
      // the sums of the weights 4, 5 and 6 in units of weight 3, rounded once: what that weight's accumulator starts from
      __all_sync(0xffffffffu, tc_mbar_wait(low_bar, 0u, s_abort));
      asm volatile("bar.sync 2, 128;" ::: "memory");
      if (tid == 64) *s_last = *s_abort;                       // (one reading for all: other roles may still give up)
      asm volatile("bar.sync 2, 128;" ::: "memory");
      if (*s_last == 0u) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
        for (int c0 = 0; c0 < kI8Tile; c0 += 16) {
          int v[3][16];
#pragma unroll
          for (int l = 0; l < 3; ++l) load16(v[l], l * kI8Tile + c0);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 16; ++j)
            v[0][j] = (int)(((long long)v[0][j] * 65536 + (long long)v[1][j] * 256 + v[2][j] + (1 << 23)) >> 24);
          asm volatile(
              "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};\n"
              ::"r"(v[0][0]), "r"(v[0][1]), "r"(v[0][2]), "r"(v[0][3]), "r"(v[0][4]), "r"(v[0][5]), "r"(v[0][6]), "r"(v[0][7]),
              "r"(v[0][8]), "r"(v[0][9]), "r"(v[0][10]), "r"(v[0][11]), "r"(v[0][12]), "r"(v[0][13]), "r"(v[0][14]), "r"(v[0][15]),
              "r"(tmem_d + ((uint32_t)(32 * q) << 16) + (uint32_t)(3 * kI8Tile + c0)) : "memory");
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        tc_mbar_arrive(start_bar);
      }
    }
    __all_sync(0xffffffffu, tc_mbar_wait(done_bar, 0u, s_abort));
    // what the four warps do next depends on the abort word alone: it is set before a warp whose wait ran out gets here
    asm volatile("bar.sync 2, 128;" ::: "memory");
    const bool ok = *s_abort == 0u;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int tt = (r + kI8Tile - 1) / kI8Tile, tile_id = ti * tt - ti * (ti - 1) / 2 + (tj - ti);
    double* const parts = L.gram_sums + (int64_t)tile_id * n_split * (kI8Tile * kI8Tile) + row;
    float* const s_tile = reinterpret_cast<float*>(base_ptr);  // (every load has landed, every MMA has read its operands)
    constexpr int kPad = kI8Tile + 4;                          // 16-byte rows
    const double si = s_scale[0][row];
    const int64_t lda = L.lda;
    float* const A = L.A;
    const int gi = ti * kI8Tile + row;                         // this thread's row of the tile
    // sixteen columns of it: into shared memory for the tile itself; the mirror's rows take a warp's lanes side by side
    auto emit = [&](int c0, const double (&sum)[16]) {
      float f[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) f[j] = (float)((sum[j] + (c0 + j == row && !wide ? s_rest[row] : 0.0)) * si * s_scale[1][c0 + j]);
#pragma unroll
      for (int j = 0; j < 16; j += 4) *reinterpret_cast<float4*>(&s_tile[row * kPad + c0 + j]) = make_float4(f[j], f[j + 1], f[j + 2], f[j + 3]);
      if (!diag && gi < r) {
#pragma unroll
        for (int j = 0; j < 16; ++j) { const int gj = tj * kI8Tile + c0 + j; if (gj < r) A[(int64_t)gj * lda + gi] = f[j]; }
      }
    };
    if (ok) {
#pragma unroll 1
      for (int c0 = 0; c0 < kI8Tile; c0 += 16) {
        int v[4][16];
#pragma unroll
        for (int l = 0; l < 4; ++l) load16(v[l], l * kI8Tile + c0);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        double sum[16];
#pragma unroll
        for (int j = 0; j < 16; ++j)                           // below 2^53: exact
          sum[j] = fma(i8_double(v[0][j]), 16777216.0, fma(i8_double(v[1][j]), 65536.0, fma(i8_double(v[2][j]), 256.0, i8_double(v[3][j]))));
        if (n_split > 1) {
#pragma unroll
          for (int j = 0; j < 16; ++j) parts[((int64_t)ref.c * kI8Tile + c0 + j) * kI8Tile] = sum[j];
        } else emit(c0, sum);
      }
    }
    bool write_tile = ok;
    if (ok && n_split > 1) {                                   // the last part to finish adds them up, in order
      __threadfence();
      asm volatile("bar.sync 2, 128;" ::: "memory");
      if (tid == 64) *s_last = atomicAdd(L.gram_ticket + tile_id, 1u) == (uint32_t)(n_split - 1) ? 1u : 0u;
      asm volatile("bar.sync 2, 128;" ::: "memory");
      write_tile = *s_last != 0;
      if (write_tile) {
        __threadfence();
#pragma unroll 1
        for (int c0 = 0; c0 < kI8Tile; c0 += 16) {
          double sum[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) sum[j] = 0.0;
#pragma unroll 4
          for (int sp = 0; sp < n_split; ++sp) {
#pragma unroll
            for (int j = 0; j < 16; ++j) sum[j] += __ldcg(parts + ((int64_t)sp * kI8Tile + c0 + j) * kI8Tile);
          }
          emit(c0, sum);
        }
      }
    }
    if (write_tile) {                                          // uniform over the four warps
      asm volatile("bar.sync 2, 128;" ::: "memory");
      const bool vec = lda % 4 == 0 && (reinterpret_cast<uintptr_t>(A) & 15u) == 0;
      const int gcol = tj * kI8Tile + 4 * lane;
#pragma unroll 4
      for (int rr = warp - 2; rr < kI8Tile; rr += 4) {         // a warp per row
        const int grow = ti * kI8Tile + rr;
        if (grow < r) {
          const float4 f = *reinterpret_cast<const float4*>(&s_tile[rr * kPad + 4 * lane]);
          float* const dst = A + (int64_t)grow * lda + gcol;
          if (vec && gcol + 3 < r) *reinterpret_cast<float4*>(dst) = f;
          else {
            if (gcol < r) dst[0] = f.x;
            if (gcol + 1 < r) dst[1] = f.y;
            if (gcol + 2 < r) dst[2] = f.z;
            if (gcol + 3 < r) dst[3] = f.w;
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*s_abort) {                                              // given up: the copies on their way land first (bounded, too)
    if (tid == 0)
      for (int it = max(0, issued - kI8Stages); it < issued; ++it) tc_mbar_wait(full_bar(it % kI8Stages), (uint32_t)(it / kI8Stages) & 1u, nullptr);
    __syncthreads();
  }
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(kI8TmemCols) : "memory");
  }
  if (tid == 0 && *s_abort) atomicExch(err, (uint32_t)ATOMO_ERR_TIMEOUT);
}

// ---- host side ------------------------------------------------------------------------------------
int sp_i8_configure() {
  if (cudaFuncSetAttribute(sp_gram_i8_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kI8SmemBytes) == cudaSuccess) return 0;
  cudaGetLastError();
  return 1;
}
int64_t sp_i8_pitch(int len) { return ((int64_t)len + 15) / 16 * 16; }
int sp_i8_stages(int len) { return (len + kI8K - 1) / kI8K; }
int sp_i8_min_split(int len) { return (sp_i8_stages(len) + kI8PartK / kI8K - 1) / (kI8PartK / kI8K); }
int64_t sp_i8_sums(int r, int split) {
  const int64_t tt = (r + kI8Tile - 1) / kI8Tile;
  return split > 1 ? tt * (tt + 1) / 2 * split * kI8Tile * kI8Tile : 0;
}
bool sp_i8_by_rows(int len, bool tall) { return !tall && len <= kI8RowLen; }
// tiles of the layer's preparing kernels (by rows: the rows themselves, which the caller groups)
void sp_i8_prep_tiles(int r, int len, bool tall, int* short_tiles, int* long_tiles) {
  const int a = tall ? kI8TallCols : kI8WideRows, b = tall ? kI8TallRows : kI8WideCols;
  *short_tiles = sp_i8_by_rows(len, tall) ? r : (r + a - 1) / a; *long_tiles = sp_i8_by_rows(len, tall) ? 1 : (len + b - 1) / b;
}
// tensor map of the digits [4][r][pitch]: boxes of 64 columns x 128 vectors x 4 digits, 64-byte swizzle, zero fill outside
int sp_i8_make_map(void* out_map /*CUtensorMap, host*/, const int8_t* digits, int r, int len, int64_t pitch) {
  const cuuint64_t dims[3] = {(cuuint64_t)len, (cuuint64_t)r, 4};
  const cuuint64_t strides[2] = {(cuuint64_t)pitch, (cuuint64_t)pitch * r};
  const cuuint32_t box[3] = {(cuuint32_t)kI8K, (cuuint32_t)kI8Tile, 4};
  const cuuint32_t estr[3] = {1, 1, 1};
  return g_encode_tiled(reinterpret_cast<CUtensorMap*>(out_map), CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<int8_t*>(digits), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS ? 0 : 1;
}
void launch_sp_gram_i8(const SpLayer* d_layers, const void* d_maps, const TileRef* d_prep, int n_rows, int n_prep, const TileRef* d_tiles, int n_tiles,
                       uint32_t* d_err, uint32_t* d_coarse, cudaStream_t st) {
  if (n_tiles <= 0) return;
  if (n_rows > 0) sp_i8_row_kernel<<<n_rows, 256, 0, st>>>(d_layers, d_prep);
  if (n_prep > n_rows) {
    sp_i8_max_kernel<<<n_prep - n_rows, 256, 0, st>>>(d_layers, d_prep + n_rows);
    sp_i8_slice_kernel<<<n_prep - n_rows, 256, 0, st>>>(d_layers, d_prep + n_rows);
  }
  sp_gram_i8_kernel<<<n_tiles, kI8Threads, kI8SmemBytes, st>>>(d_layers, reinterpret_cast<const CUtensorMap*>(d_maps), d_tiles, d_err, d_coarse);
}

}  // namespace atomo
