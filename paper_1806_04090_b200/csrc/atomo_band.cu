// Spectral atoms, short sides above 512: reduction of the scaled Gram matrix A (r x r, fp32, in global memory) to a
// tridiagonal T in two stages (the small layers' one-stage reduction in registers: atomo_tridiag.cu).
//
//   sp_band_kernel   A -> band matrix B = Q1^T A Q1 with eight sub-diagonals.  Panels of eight columns: Householder QR of
//                    the panel, then A -= U W^T + W U^T over the trailing block.  The update of a panel and the product of
//                    the updated block with the next panel's reflectors share one pass, so the matrix is read and written
//                    once per eight columns (a one-stage reduction reads it once per column).
//   sp_chase_kernel  B -> T = Q2^T B Q2 by bulge chasing, fp64, the band in shared memory (one CTA per layer up to a short
//                    side of 1024, a cluster above), all sweeps in flight at once.
//
// Then the eigenvalues of T and vectors for the kept atoms only, as on the small route; a vector of T goes
// through the chase's reflectors and then through the panels' (I - U T U^T, the columns of U as rows of td_V) in the vector
// kernels of atomo_tridiag_big.cu.
//
// Precision: the matrix, the panel vectors U and W and the panel itself are fp32; products run in fp32 over 32 terms and are
// added up in fp64; panel dots, scalars and the whole chase are fp64.  Q1 is applied as I - U T U^T with T formed from the
// fp64 dots of the rounded U, so that it is orthogonal whatever the rounding of U.
#include <algorithm>

#include <cooperative_groups.h>

#include "atomo_kernels.cuh"

namespace cg = cooperative_groups;

namespace atomo {

namespace {
constexpr int kBw = kBandWidth;               // columns per panel = sub-diagonals of the band
constexpr int kStrip = 64;                    // rows per strip: two per lane
constexpr uint32_t kBandPollLimit = 1u << 22;
static_assert(kBw == 8, "the operand vectors are two float4");
}  // namespace

// ---- stage 1: dense -> band ---------------------------------------------------------------------------------------------
// Panel k (c = 8 k): columns c .. c+7 below row c+7.  The rows (= columns: A is symmetric) are cut into strips of 64.
// A[j][i] with i in the strip is read as row j, two neighbouring entries per lane (256 bytes per warp), so a lane keeps
// everything of its two rows -- their entries of U and W of the panel before, and their eight sums of the product -- in
// registers and walks over the columns j, whose U, W and new U entries are broadcast from shared memory: 48 multiply-adds per
// 8 bytes read and written and six 16-byte broadcasts, no exchange between lanes.  The columns of a strip are split into PARTS
// tasks, dealt to the warps of all the layer's CTAs in turn (a strip per CTA left half of them idle on average); the parts of a
// sum are added in fp64.  A warp streams its columns through a ring of its own (asynchronous copies of four columns with their
// U and W).  Twelve warps per SM: with sixteen the 128 registers do not hold a task.
// (The sixteen products that update an entry are summed before they are added to it: added one by one they rounded the matrix
// sixteen times per panel, and the singular values of 2000 x 2048 noise were off by 1.6e-7 instead of 5.4e-8.)
// Bound: latency of the walk (with few layers 14 k cycles of a panel's 40 k at 1023 rows, 68 k of 100 k with two layers of 4096; a group
// of four columns takes a lone warp about 1000 cycles, its 200 multiply-adds alone would take 200), and the chain of a panel's small
// steps: own rows and first barrier 8 k, sums of the Gram matrix 2 k, 8 x 8 factorisation 3.5 k, U 2 .. 7 k (conversions), second
// barrier 4 k, T and what follows from it 3.5 k.  Two layers of 4096 rows: 106 (one-stage reduction) -> 49.7 -> 25.8 -> 23.4 ms; 96 of
// 1024: 29.4 -> 13.0 -> 12.7; one of 1023: 2.03 -> 1.71.  The last step is the chain's: with few layers the own rows are shared by all warps
// of a CTA, eight lanes to a row (one warp took 8 k cycles), U^T U is added up like U^T A U instead of by every CTA, T is solved for
// by columns in registers, a column per lane in the factorisation (6.1 k), barriers by release and acquire instead of fences.  Tried and
// dropped: 32 or 64 tasks per strip (two of 4096 rows 26.3 and 32.1 ms, one of 1023 the same and 10 % slower).
// The panel's QR is a Householder QR worked out on 8 x 8 matrices: the reflectors' norms and products follow from the panel's
// Gram matrix (downdated as rows of R split off) and its first eight rows, and below those rows V = X K with an 8 x 8 matrix
// K.  A column whose remainder is below 3e-8 of it is left alone (the fp32 panel has no more digits).  However inexact V is
// for an ill-conditioned panel, Q stays orthogonal: T comes from the actual dots of the rounded U.
// A panel has two barriers among the layer's CTAs:
//   every CTA: Gram matrix and first rows of the panel in, 8 x 8 factorisation (one warp), U = X K for all rows
//   pass:      tasks: update with the panel before, product with this panel's U, U^T A U; U^T U of own rows      -> barrier
//   every CTA: T, T^T (U^T A U) T; own rows: W = (A U) T - 1/2 U T^T (U^T A U) T, entries of the next panel and their Gram
//              matrix                                                                                          -> barrier
// Sums over rows are formed per half strip in an order of their own and added up in that order, U^T A U in multiples of a
// fixed unit, so the result does not depend on G.  With two CTAs per SM, which belong to different layers, one's chains and
// barriers overlap with the other's pass.
namespace {

constexpr int kGroup = 4;                     // columns that travel together through a warp's ring
constexpr int kGroupFloats = kGroup * (kStrip + 16);
// U^T A U is rounded to multiples of 2^-50 (the last place of 4 .. 8) as it is added up: sums below 8 are then exact in any order.
// (A's trace is about one and U's columns are unit vectors, so that no partial sum passes two.)
constexpr double kFix = 6.0;

struct BandShared {
  double T[8][8], S[8][8], Y[8][8], X[8][8];
  double K[8][8], vtop[8][8];     // K scaled to unit vectors; the reflectors' entries in the panel's first eight rows
  double M[36], G[36], sum[16][36];
  double s_part[16][64];          // the warps' parts of U^T A U
  double m_part[16][40];          // ... and of U^T U
  double top[8][8];
  double Wc[8][8], Uc[8][8], Pc[8][8];   // W, U and A U of the next panel's pivot rows
  uint32_t fail;
};

// reduce-scatter of eight doubles over a warp: the lane ends with the sum of value (lane >> 2) & 7
__device__ __forceinline__ double band_scatter8(const double (&v)[8], int lane) {
  double a[4], b[2], c;
  const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
#pragma unroll
  for (int i = 0; i < 4; ++i) { const double keep = h4 ? v[4 + i] : v[i], send = h4 ? v[i] : v[4 + i]; a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16); }
#pragma unroll
  for (int i = 0; i < 2; ++i) { const double keep = h3 ? a[2 + i] : a[i], send = h3 ? a[i] : a[2 + i]; b[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8); }
  { const double keep = h2 ? b[1] : b[0], send = h2 ? b[0] : b[1]; c = keep + __shfl_xor_sync(0xffffffffu, send, 4); }
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  return c;
}
// eight of the 36 dots (lower triangle by rows, number 8 BLK and on) of the columns of a 32 x 8 block, one row (a, b) per lane: the
// lane ends with dot 8 BLK + lane / 4
template <int BLK>
__device__ __forceinline__ double band_dots(const float4 a, const float4 b, int lane) {
  const double d[8] = {(double)a.x, (double)a.y, (double)a.z, (double)a.w, (double)b.x, (double)b.y, (double)b.z, (double)b.w};
  double v[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  int e = 0;
#pragma unroll
  for (int p = 0; p < 8; ++p)
#pragma unroll
    for (int q = 0; q <= p; ++q, ++e) if (e / 8 == BLK) v[e % 8] = d[p] * d[q];
  return band_scatter8(v, lane);
}
// (Out of line, as the 8 x 8 factorisation below: a panel is a walk through the whole kernel, and what runs once per panel should stay small.)
__device__ __noinline__ double band_dots_of(int blk, const float4 a, const float4 b, int lane) {
  switch (blk) {
    case 0: return band_dots<0>(a, b, lane);
    case 1: return band_dots<1>(a, b, lane);
    case 2: return band_dots<2>(a, b, lane);
    case 3: return band_dots<3>(a, b, lane);
    default: return band_dots<4>(a, b, lane);
  }
}
// all 36 of them by one warp, to dst
__device__ __noinline__ void band_gram32(const float4 a, const float4 b, double* __restrict__ dst, int lane) {
  const double x[5] = {band_dots<0>(a, b, lane), band_dots<1>(a, b, lane), band_dots<2>(a, b, lane), band_dots<3>(a, b, lane), band_dots<4>(a, b, lane)};
  if ((lane & 3) == 0) {
#pragma unroll
    for (int blk = 0; blk < 5; ++blk) if (blk * 8 + (lane >> 2) < 36) dst[blk * 8 + (lane >> 2)] = x[blk];
  }
}

// barrier among the layer's CTAs (co-resident: cooperative launch), bounded; a wait that runs out shows as
// ATOMO_ERR_TIMEOUT in the layers' status words
__device__ __forceinline__ void band_barrier(uint32_t* ctr, uint32_t target, BandShared& sh, uint32_t* timeout_flag) {
  __syncthreads();
  if (threadIdx.x == 0) {
    // (release and acquire at device scope; what the block's other threads did is ordered by the block barriers around them)
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
    uint32_t polls = 0, seen;
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(ctr) : "memory");
      if (seen >= target || sh.fail != 0u) break;
      if (++polls > kBandPollLimit) { sh.fail = 1u; *timeout_flag = 1u; }
    }
  }
  __syncwarp();                                              // (without it the polling thread's warp may stay divided past the barrier)
  __syncthreads();
}

// sums of 36 values over `n` blocks of global memory, in an order that depends on THREADS alone; complete after the caller's
// next barrier but one (this function has one inside)
template <int THREADS>
__device__ __forceinline__ void band_sum36(const double* __restrict__ src, int first, int n, double (*part)[36], double* __restrict__ dst) {
  constexpr int kGroups = THREADS / 36 < 16 ? THREADS / 36 : 16;
  const int tid = threadIdx.x, gr = tid / 36, e = tid % 36;
  if (gr < kGroups) {
    double s = 0.0;
#pragma unroll 4
    for (int b = first / kGroups * kGroups + gr; b < n; b += kGroups) if (b >= first) s += __ldcg(src + (int64_t)b * 36 + e);
    part[gr][e] = s;
  }
  __syncthreads();
  if (tid < 36) {
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < kGroups; ++q) s += part[q][tid];
    dst[tid] = s;
  }
}

// Householder QR of the panel on its Gram matrix (lower triangle in sh.G) and first eight rows (sh.top), one warp.  Lane l < 8
// holds column l of the Gram matrix, of the rows and of K (the other lanes do the same on copies), so that what a step needs of
// its own column is in registers and the pivot column's entries arrive while the norm's roots are taken.  Leaves R in sh.top, the unit
// reflectors' entries in the first eight rows in sh.vtop (zero above the diagonal) and K, scaled likewise.
__device__ __noinline__ void band_small_qr(BandShared& sh, const int n_ref, const int lane) {
  __syncwarp();
  const int l = lane & 7;
  double top[8], g[8], k[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    top[i] = sh.top[i][l];
    g[i] = sh.G[i >= l ? i * (i + 1) / 2 + l : l * (l + 1) / 2 + i];
    k[i] = i == l ? 1.0 : 0.0;
  }
  const double orig = sh.G[l * (l + 1) / 2 + l];             // squared norm of column l as given
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const double nx2 = __shfl_sync(0xffffffffu, g[t], t), x0 = __shfl_sync(0xffffffffu, top[t], t), o = __shfl_sync(0xffffffffu, orig, t);
    double x[8], kt[8];                                      // the pivot column's entries below the diagonal, its column of K
#pragma unroll
    for (int i = t + 1; i < 8; ++i) x[i] = __shfl_sync(0xffffffffu, top[i], t);
#pragma unroll
    for (int i = 0; i <= t; ++i) kt[i] = __shfl_sync(0xffffffffu, k[i], t);
    double alpha = x0, beta = 0.0, un = 0.0;
    const bool act = t < n_ref && nx2 > 1.0e-290 && nx2 > 1.0e-15 * o;   // else H = I: a zero column, or no digits left
    if (act) {
      const double nx = nx2 * rsqrt(nx2);
      alpha = -copysign(nx, x0);
      un = rsqrt(2.0 * fma(fabs(x0), nx, nx2));              // 1 / ||v||
      beta = 2.0 * un * un;
    }
    x[t] = x0 - alpha;
    const double gl = l > t ? beta * (g[t] - alpha * top[t]) : 0.0;   // beta v^T x_l
#pragma unroll
    for (int i = t; i < 8; ++i) top[i] = fma(-gl, x[i], top[i]);
#pragma unroll
    for (int i = 0; i <= t; ++i) k[i] = fma(-gl, kt[i], k[i]);
    if (lane == t) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        sh.vtop[i][t] = i < t ? 0.0 : x[i] * un;
        sh.K[i][t] = i <= t ? kt[i] * un : 0.0;
        if (act && i >= t) top[i] = i == t ? alpha : 0.0;
      }
    }
#pragma unroll
    for (int i = t + 1; i < 8; ++i) g[i] = fma(-__shfl_sync(0xffffffffu, top[t], i), top[t], g[i]);   // row t of R leaves the Gram matrix
  }
  if (lane < 8) {
#pragma unroll
    for (int i = 0; i < 8; ++i) sh.top[i][l] = top[i];
  }
}

}  // namespace

// A CTA of THREADS threads, MINB per SM
template <int THREADS, int MINB, int PARTS, int STAGES>
__global__ void __launch_bounds__(THREADS, MINB) sp_band_kernel(const SpLayer* __restrict__ layers, const ClusterCta* __restrict__ ctas,
                                                                uint32_t* __restrict__ timeout_flag) {
  constexpr int kWarps = THREADS / 32;
  constexpr bool kSpread = PARTS >= 16;                      // few layers: a CTA has one or two half strips of its own
  extern __shared__ __align__(16) float band_smem[];
  __shared__ BandShared sh;
  const ClusterCta me = ctas[blockIdx.x];
  const SpLayer& L = layers[me.layer];
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const int r = L.r, g = me.slot, G = me.pad;
  const int n_strips = (r + kStrip - 1) / kStrip;
  float* const A = L.A; const int64_t lda = L.lda; const int ld32 = (int)lda;           // lda is a multiple of the strip: whole strips may be read and written
  float* const gUW = L.bd_UW; float* const gX = L.bd_X;
  double* const gPart = L.bd_part; double* const gS = L.bd_S; double* const gB = L.bd_band;
  double* const gG = L.bd_G;
  float* const gV = L.td_V; const int64_t ldv = L.td_ldv;
  double* const gT = L.bd_T;
  float* const s_u = band_smem;                              // [r][8] this panel's U, by row
  float* const s_ring = band_smem + (size_t)(r + kGroup) * 8; // [warps][STAGES] groups of columns on their way
  if (tid == 0) sh.fail = 0u;
  if (tid < kGroup * 8) s_u[(size_t)r * 8 + tid] = 0.0f;     // rows past the end, of a last group that is not full
  uint32_t arrivals = 0;
  auto own_from = [&](int row) { const int h = row / 32; return h + ((g - h % G) % G + G) % G; };   // this CTA's first half strip, then every G-th
  for (int c = 0; c < r; c += kBw) {
    // ---- own rows: U and W of the panel before out, entries of this panel (columns c .. c+7) and the Gram matrix of those
    // below the band ----
    if constexpr (kSpread) {                                 // eight lanes per row, all warps on the CTA's few half strips
      const int h0 = own_from(c), n_own = h0 < 2 * n_strips ? (2 * n_strips - 1 - h0) / G + 1 : 0;
      float* const s_x = s_ring;                             // [half strips of a round][32][8], the panel's entries (the ring is idle)
      constexpr int kRound = kWarps * STAGES * kGroupFloats / 256;
      for (int n0 = 0; n0 < n_own; n0 += kRound) {
        const int n_now = min(kRound, n_own - n0);
        for (int q = w; q < 8 * n_now; q += kWarps) {        // four rows
          const int t = lane & 7, i = (h0 + (n0 + q / 8) * G) * 32 + q % 8 * 4 + (lane >> 3);
          const bool in = i >= c && i < r;
          float x = in && c + t < r ? __ldcg(A + (int64_t)(c + t) * lda + i) : 0.0f;
          if (c > 0) {
            double part[PARTS];
#pragma unroll
            for (int z = 0; z < PARTS; ++z) part[z] = in ? __ldcg(gPart + ((int64_t)z * n_strips * kStrip + i) * 8 + t) : 0.0;
            double p = 0.0, z = 0.0;                         // the product A U: the parts added in order
#pragma unroll
            for (int q2 = 0; q2 < PARTS; ++q2) p += part[q2];
            const float4* const us = reinterpret_cast<const float4*>(s_u + (size_t)(in ? i : r) * 8);   // (zeros past the end)
            const float4 ua = us[0], ub = us[1];
            const float uu[8] = {ua.x, ua.y, ua.z, ua.w, ub.x, ub.y, ub.z, ub.w};
            // W[i][t] = sum_s P[i][s] T[s][t] - 1/2 sum_s U[i][s] (T^T S T)[s][t]
#pragma unroll
            for (int s = 0; s < 8; ++s) {
              const double ps = __shfl_sync(0xffffffffu, p, (lane & 24) + s);
              if (s <= t) z = fma(ps, sh.T[s][t], z);
              z = fma((double)uu[s], sh.X[s][t], z);
            }
            const float ww = (float)z;
            z = (double)x;
#pragma unroll
            for (int s = 0; s < 8; ++s) z -= fma((double)uu[s], sh.Wc[t][s], (double)__shfl_sync(0xffffffffu, ww, (lane & 24) + s) * sh.Uc[t][s]);
            x = in && c + t < r ? (float)z : 0.0f;
            gUW[(int64_t)i * 16 + t] = in ? s_u[(size_t)i * 8 + t] : 0.0f;
            gUW[(int64_t)i * 16 + 8 + t] = ww;
          }
          gX[(int64_t)i * 8 + t] = x;
          s_x[q * 32 + lane] = i < c + kBw ? 0.0f : x;
        }
        __syncthreads();
        for (int q = w; q < 5 * n_now; q += kWarps) {        // eight of a half strip's dots
          const float4* const src = reinterpret_cast<const float4*>(s_x + (q / 5) * 256 + lane * 8);
          const double x = band_dots_of(q % 5, src[0], src[1], lane);
          const int e = q % 5 * 8 + (lane >> 2);
          if ((lane & 3) == 0 && e < 36) gG[(int64_t)(h0 + (n0 + q / 5) * G) * 36 + e] = x;
        }
        if (n0 + kRound < n_own) __syncthreads();
      }
    } else                                                   // half a strip per warp
    {
      for (int half = own_from(c) + w * G; half < 2 * n_strips; half += kWarps * G) {
        const int i = half * 32 + lane;
        const bool in = i >= c && i < r;
        float x[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = in && c + t < r ? __ldcg(A + (int64_t)(c + t) * lda + i) : 0.0f;
        if (c > 0) {
          float uu[8], ww[8];
          double p[8];                                       // the product A U: the parts added in order
#pragma unroll
          for (int t = 0; t < 8; ++t) p[t] = 0.0;
          const double2* src = reinterpret_cast<const double2*>(gPart + (int64_t)i * 8);
#pragma unroll 4
          for (int part = 0; part < PARTS; ++part, src += (int64_t)n_strips * kStrip * 4) {
#pragma unroll
            for (int t = 0; t < 4; ++t) { const double2 d = in ? __ldcg(src + t) : make_double2(0.0, 0.0); p[2 * t] += d.x; p[2 * t + 1] += d.y; }
          }
#pragma unroll
          for (int t = 0; t < 8; ++t) uu[t] = in ? s_u[(size_t)i * 8 + t] : 0.0f;
          double z[8];                                       // W[i][t] = sum_s P[i][s] T[s][t] - 1/2 sum_s U[i][s] (T^T S T)[s][t]
#pragma unroll
          for (int t = 0; t < 8; ++t) z[t] = 0.0;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
#pragma unroll
            for (int t = 0; t < 8; ++t) { if (q <= t) z[t] = fma(p[q], sh.T[q][t], z[t]); z[t] = fma((double)uu[q], sh.X[q][t], z[t]); }
          }
#pragma unroll
          for (int t = 0; t < 8; ++t) { ww[t] = (float)z[t]; z[t] = (double)x[t]; }
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const double uq = (double)uu[q], wq = (double)ww[q];
#pragma unroll
            for (int t = 0; t < 8; ++t) z[t] -= fma(uq, sh.Wc[t][q], wq * sh.Uc[t][q]);
          }
#pragma unroll
          for (int t = 0; t < 8; ++t) x[t] = in && c + t < r ? (float)z[t] : 0.0f;
          float4* du = reinterpret_cast<float4*>(gUW + (int64_t)i * 16);
          float4* dw = du + 2;
          du[0] = make_float4(uu[0], uu[1], uu[2], uu[3]); du[1] = make_float4(uu[4], uu[5], uu[6], uu[7]);
          dw[0] = make_float4(ww[0], ww[1], ww[2], ww[3]); dw[1] = make_float4(ww[4], ww[5], ww[6], ww[7]);
        }
        float4 lo = make_float4(x[0], x[1], x[2], x[3]), hi = make_float4(x[4], x[5], x[6], x[7]);
        float4* dx = reinterpret_cast<float4*>(gX + (int64_t)i * 8);
        dx[0] = lo; dx[1] = hi;
        if (i < c + kBw) { lo = make_float4(0.f, 0.f, 0.f, 0.f); hi = lo; }
        band_gram32(lo, hi, gG + (int64_t)half * 36, lane);
      }
    }
    // U^T A U and U^T U are added up in one of three sets of 128 words in turn; the next panel's is cleared here: its last readers are
    // past the barrier before this one, its adders wait for the one after it
    double* const s_sum = gS + c / kBw % 3 * 128;
    if (g == 0 && tid < 128) { gS[(c / kBw + 1) % 3 * 128 + tid] = 0.0; if (c == 0) s_sum[tid] = 0.0; }
    arrivals += (uint32_t)G;
    band_barrier(L.bd_bar, arrivals, sh, timeout_flag);
    if (sh.fail) break;
    const int row0 = c + kBw;                                // first row below the band of the panel
    const int m = r - row0;                                  // panel rows
    const int first_strip = row0 / kStrip;
    // ---- diagonal block, QR of the panel (every CTA) ----
    if (g == 0 && tid < kBw * kBw) {
      const int a = tid / kBw, b = tid % kBw;                // entry (c + a, c + b), a >= b
      if (a >= b && c + a < r) gB[(int64_t)(c + b) * (kBw + 1) + a - b] = (double)__ldcg(gX + (int64_t)(c + a) * 8 + b);
    }
    if (m <= 0) break;
    if (tid >= THREADS - 64) {
      const int q = tid - (THREADS - 64), a = q / 8, b = q % 8;
      sh.top[a][b] = row0 + a < r ? (double)__ldcg(gX + (int64_t)(row0 + a) * 8 + b) : 0.0;
    }
    band_sum36<THREADS>(gG, c / 32, 2 * n_strips, sh.sum, sh.G);
    __syncthreads();
    const int n_ref = min(kBw, m - 1);                       // reflectors of this panel: rows row0 + t .. r-1, at least two of them
    if (w == 0) band_small_qr(sh, n_ref, lane);
    __syncthreads();
    for (int i = row0 + tid; i < r; i += THREADS) {
      float u[8];
      if (i < row0 + kBw) {
#pragma unroll
        for (int t = 0; t < 8; ++t) u[t] = (float)sh.vtop[i - row0][t];
      } else {
        const float4 a = __ldcg(reinterpret_cast<const float4*>(gX + (int64_t)i * 8)), b = __ldcg(reinterpret_cast<const float4*>(gX + (int64_t)i * 8) + 1);
        const double x[8] = {(double)a.x, (double)a.y, (double)a.z, (double)a.w, (double)b.x, (double)b.y, (double)b.z, (double)b.w};
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          double z = 0.0;
#pragma unroll
          for (int q = 0; q <= t; ++q) z = fma(x[q], sh.K[q][t], z);
          u[t] = (float)z;
        }
      }
      float4* d = reinterpret_cast<float4*>(s_u + (size_t)i * 8);
      d[0] = make_float4(u[0], u[1], u[2], u[3]); d[1] = make_float4(u[4], u[5], u[6], u[7]);
    }
    // R: rows row0 + a, columns c + t, t >= a
    if (g == 0 && tid < 64) {
      const int a = tid / 8, t = tid % 8;
      if (t >= a && row0 + a < r) gB[(int64_t)(c + t) * (kBw + 1) + kBw + a - t] = sh.top[a][t];
    }
    const bool first = c == 0;
    // ---- pass ----
    const int per = ((m + PARTS - 1) / PARTS + 3) & ~3;      // columns per task, a multiple of the group
    __syncthreads();
    sh.s_part[w][lane] = sh.s_part[w][lane + 32] = 0.0;
    sh.m_part[w][lane] = 0.0;
    if (lane < 8) sh.m_part[w][lane + 32] = 0.0;
    __syncwarp();
    // tasks (strip, part), dealt to the warps of all CTAs
    for (int task = g + w * G; task < (n_strips - first_strip) * PARTS; task += kWarps * G) {
      const int s = first_strip + task / PARTS, part = task % PARTS;
      const int jb = row0 + part * per, je = min(jb + per, r);
      const int i = s * kStrip + 2 * lane;
      double* const dst = gPart + ((int64_t)part * n_strips * kStrip + i) * 8;
      if (jb >= je) {                                        // an empty part
#pragma unroll
        for (int t = 0; t < 16; t += 2) *reinterpret_cast<double2*>(dst + t) = make_double2(0.0, 0.0);
        continue;
      }
      // a group of four columns: 64 entries of A each (16 bytes per lane, half a warp per column), then their U and W
      const uint32_t ring = (uint32_t)__cvta_generic_to_shared(s_ring + (size_t)w * STAGES * kGroupFloats);
      const float* src = A + (int64_t)(jb + lane / 16) * lda + s * kStrip + (lane & 15) * 4;   // the next group to ask for
      const float* const src_uw = gUW + lane * 4;
      const int back = 2 * lane - (lane & 15) * 4 - (lane / 16 + (STAGES - 1) * kGroup) * ld32;   // from there to the group at work
      int stage = 0;
      auto issue = [&](int j) {                              // columns j .. j + 3 into the ring
        if (j < je) {
          const uint32_t d = ring + stage * (kGroupFloats * 4) + lane * 16;
          const int n = je - j;                              // (lanes past the end fill with zeros)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(lane / 16 < n ? src : A), "r"(lane / 16 < n ? 16 : 0) : "memory");
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d + 512), "l"(2 + lane / 16 < n ? src + 2 * ld32 : A),
                       "r"(2 + lane / 16 < n ? 16 : 0) : "memory");
          if (!first && lane < 16)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d + 1024), "l"(src_uw + (lane / 4 < n ? j * 16 : 0)), "r"(lane / 4 < n ? 16 : 0) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory"); // one group per call, empty or not: the counting stays uniform
        src += kGroup * ld32;
        stage = stage == STAGES - 1 ? 0 : stage + 1;
      };
#pragma unroll
      for (int q = 0; q < STAGES - 1; ++q) issue(jb + q * kGroup);
      float up0[8], wp0[8], up1[8], wp1[8];
      double p0[8], p1[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) { up0[t] = wp0[t] = up1[t] = wp1[t] = 0.0f; p0[t] = p1[t] = 0.0; }
      if (!first) {
        const float4* own = reinterpret_cast<const float4*>(gUW + (int64_t)i * 16);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 a = __ldcg(own + h), b = __ldcg(own + 2 + h), d = __ldcg(own + 4 + h), e = __ldcg(own + 6 + h);
          up0[4 * h] = -a.x; up0[4 * h + 1] = -a.y; up0[4 * h + 2] = -a.z; up0[4 * h + 3] = -a.w;
          wp0[4 * h] = -b.x; wp0[4 * h + 1] = -b.y; wp0[4 * h + 2] = -b.z; wp0[4 * h + 3] = -b.w;
          up1[4 * h] = -d.x; up1[4 * h + 1] = -d.y; up1[4 * h + 2] = -d.z; up1[4 * h + 3] = -d.w;
          wp1[4 * h] = -e.x; wp1[4 * h + 1] = -e.y; wp1[4 * h + 2] = -e.z; wp1[4 * h + 3] = -e.w;
        }
      }
      // (two loops, so that the fp64 sums can leave the registers for the inner one: a spill among the 128 registers costs
      // every group a round trip to the L2, there is no L1 left beside the shared memory)
#pragma unroll 1
      for (int j0 = jb; j0 < je; j0 += 32) {                 // fp32 runs of up to 32 columns
        float q0[8], q1[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) q0[t] = q1[t] = 0.0f;
#pragma unroll 1
        for (int j = j0; j < min(je, j0 + 32); j += kGroup) {
          asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
          __syncwarp();                                      // the group has landed for the warp; the stage of the one before is free
          const int at = stage == STAGES - 1 ? 0 : stage + 1;
          float* const ap = const_cast<float*>(src) + back;
          issue(j + (STAGES - 1) * kGroup);
          const float* const st = s_ring + ((size_t)w * STAGES + at) * kGroupFloats;
          const float4* const un = reinterpret_cast<const float4*>(s_u) + (size_t)j * 2;
          // the columns are stored together at the end: a store between them might alias the shared memory for all the
          // compiler knows, so that a column's loads would wait for the column before it
          float2 out[kGroup];
#pragma unroll
          for (int u = 0; u < kGroup; ++u) {                 // one column: update, product
            float2 v = *reinterpret_cast<const float2*>(st + u * kStrip + 2 * lane);
            if (!first) {
              const float4* o = reinterpret_cast<const float4*>(st + kGroup * kStrip + u * 16);
              const float4 cu0 = o[0], cu1 = o[1], cw0 = o[2], cw1 = o[3];
              const float cu[8] = {cu0.x, cu0.y, cu0.z, cu0.w, cu1.x, cu1.y, cu1.z, cu1.w};
              const float cw[8] = {cw0.x, cw0.y, cw0.z, cw0.w, cw1.x, cw1.y, cw1.z, cw1.w};
              // the sixteen products are summed before they meet the entry: one rounding at the entry's scale per panel.  The last
              // reflectors' first: what the first ones take away is the largest where few directions outweigh the rest (with the
              // first ones first sigma of 2000 x 2048 at noise 0.05 was off by 8.1e-6 instead of 3.9e-6); in two chains (one:
              // VGG-11 58.6 ms, two 58.4)
              float dx = up0[7] * cw[7], dy = up1[7] * cw[7], ex = up0[6] * cw[6], ey = up1[6] * cw[6];
              dx = fmaf(wp0[7], cu[7], dx); dy = fmaf(wp1[7], cu[7], dy);
              ex = fmaf(wp0[6], cu[6], ex); ey = fmaf(wp1[6], cu[6], ey);
#pragma unroll
              for (int t = 5; t >= 0; t -= 2) {
                dx = fmaf(up0[t], cw[t], dx); dy = fmaf(up1[t], cw[t], dy);
                dx = fmaf(wp0[t], cu[t], dx); dy = fmaf(wp1[t], cu[t], dy);
                ex = fmaf(up0[t - 1], cw[t - 1], ex); ey = fmaf(up1[t - 1], cw[t - 1], ey);
                ex = fmaf(wp0[t - 1], cu[t - 1], ex); ey = fmaf(wp1[t - 1], cu[t - 1], ey);
              }
              dx += ex; dy += ey;
              v.x += dx; v.y += dy;
            }
            out[u] = v;
            const float4 n0 = un[2 * u], n1 = un[2 * u + 1];
            const float cn[8] = {n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, n1.z, n1.w};
#pragma unroll
            for (int t = 0; t < 8; ++t) { q0[t] = fmaf(v.x, cn[t], q0[t]); q1[t] = fmaf(v.y, cn[t], q1[t]); }
          }
          if (!first) {
#pragma unroll
            for (int u = 0; u < kGroup; ++u) if (j + u < je) *reinterpret_cast<float2*>(ap + u * ld32) = out[u];
          }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) { p0[t] += (double)q0[t]; p1[t] += (double)q1[t]; }
      }
      __syncwarp();                                          // the ring is free for the warp's next task
      // rows outside the trailing block (past the end A holds whatever the workspace held) count as zeros
      const bool in0 = i >= row0 && i < r, in1 = i + 1 >= row0 && i + 1 < r;
#pragma unroll
      for (int t = 0; t < 8; ++t) { if (!in0) p0[t] = 0.0; if (!in1) p1[t] = 0.0; }
#pragma unroll
      for (int t = 0; t < 8; t += 2) {
        *reinterpret_cast<double2*>(dst + t) = make_double2(p0[t], p0[t + 1]);
        *reinterpret_cast<double2*>(dst + 8 + t) = make_double2(p1[t], p1[t + 1]);
      }
#pragma unroll 1
      for (int a = 0; a < 8; ++a) {                          // row a of U^T (A U): this task's rows and columns
        const double ua = in0 ? (double)s_u[(size_t)i * 8 + a] : 0.0, ub = in1 ? (double)s_u[(size_t)(i + 1) * 8 + a] : 0.0;
        double x[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) x[t] = fma(ub, p1[t], fma(ua, p0[t], kFix)) - kFix;
        const double sum = band_scatter8(x, lane);
        if ((lane & 3) == 0) sh.s_part[w][a * 8 + (lane >> 2)] += sum;
      }
    }
    constexpr int kPieces = kSpread ? 5 : 1;                 // U^T U of the own half strips, eight dots at a time or all 36
    for (int q = w; ; q += kWarps) {
      const int half = own_from(row0) + q / kPieces * G;
      if (half >= 2 * n_strips) break;
      const int i = half * 32 + lane;
      const bool in = i >= row0 && i < r;
      const float4* src = reinterpret_cast<const float4*>(s_u + (size_t)(in ? i : r) * 8);
      if (kSpread) {                                         // (in multiples of 2^-50 again)
        const double x = band_dots_of(q % 5, src[0], src[1], lane);
        if ((lane & 3) == 0) sh.m_part[w][q % 5 * 8 + (lane >> 2)] += (x + kFix) - kFix;
      } else {
        band_gram32(src[0], src[1], sh.sum[w], lane);
        __syncwarp();
        for (int e = lane; e < 36; e += 32) sh.m_part[w][e] += (sh.sum[w][e] + kFix) - kFix;
        __syncwarp();
      }
    }
    __syncthreads();
    if (tid < 100) {
      double t = 0.0;
#pragma unroll
      for (int ww = 0; ww < kWarps; ++ww) t += tid < 64 ? sh.s_part[ww][tid] : sh.m_part[ww][tid - 64];
      atomicAdd(s_sum + tid, t);
    }
    arrivals += (uint32_t)G;
    band_barrier(L.bd_bar, arrivals, sh, timeout_flag);
    // ---- T, T^T S T, W of the next panel's pivot rows (every CTA, one warp) ----
    if (tid < 64) sh.S[tid / 8][tid % 8] = __ldcg(s_sum + tid);
    else if (tid < 100) sh.M[tid - 64] = __ldcg(s_sum + tid);
    else if (tid >= THREADS - 64) {                          // the product's next pivot rows
      const int q = tid - (THREADS - 64), i = row0 + q / 8;
      double p = 0.0;
      if (i < r) {
        const double* src = gPart + (int64_t)i * 8 + q % 8;
#pragma unroll
        for (int part = 0; part < PARTS; ++part) p += __ldcg(src + (int64_t)part * n_strips * kStrip * 8);
      }
      sh.Pc[q / 8][q % 8] = p;
    }
    __syncthreads();
    if (w == 0) {
      // T is the inverse of the upper triangle of U^T U with half its diagonal: lane t solves for column t from the diagonal up
      if (lane < 8) {
        double col[8];
#pragma unroll
        for (int q = 7; q >= 0; --q) {
          double z = 0.0;
#pragma unroll
          for (int x = 7; x > q; --x) z = fma(sh.M[x * (x + 1) / 2 + q], col[x], z);
          const double d = sh.M[q * (q + 1) / 2 + q], tau = d > 0.5 ? 2.0 / d : 0.0;
          col[q] = q > lane ? 0.0 : q == lane ? tau : -tau * z;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) sh.T[q][lane] = col[q];
      }
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int a = lane / 8 + 4 * h, b = lane % 8;
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) t = fma(sh.S[a][q], sh.T[q][b], t);
        sh.Y[a][b] = t;
        if (g == 0) gT[(int64_t)(c / kBw) * 64 + a * 8 + b] = sh.T[a][b];   // for the back-transformation, as the reflectors' rows below
      }
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h) {                          // X = -1/2 T^T S T
        const int a = lane / 8 + 4 * h, b = lane % 8;
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) t = fma(sh.T[q][a], sh.Y[q][b], t);
        sh.X[a][b] = -0.5 * t;
      }
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int a = lane / 8 + 4 * h, t = lane % 8, i = row0 + a;
        double z = 0.0;
        if (i < r) {
#pragma unroll
          for (int q = 0; q < 8; ++q) { z = fma(sh.Pc[a][q], sh.T[q][t], z); z = fma((double)s_u[(size_t)i * 8 + q], sh.X[q][t], z); }
        }
        sh.Wc[a][t] = (double)(float)z;
        sh.Uc[a][t] = i < r ? (double)s_u[(size_t)i * 8 + t] : 0.0;
      }
    }
    __syncthreads();
    // the reflectors' rows for the back-transformation (zero above row0 + t)
    for (int s = g; s < n_strips; s += G)
      for (int q = tid; q < kStrip * 8; q += THREADS) {
        const int t = q / kStrip, i = s * kStrip + q % kStrip;
        if (i < r && c + t < r) gV[(int64_t)(c + t) * ldv + i] = i >= row0 + t ? s_u[(size_t)i * 8 + t] : 0.0f;
      }
  }
}

// ---- stage 2: band -> tridiagonal -----------------------------------------------------------------------------------------
// Bulge chasing with reflectors of length eight.  Sweep j brings column j to tridiagonal form: step -1 forms the reflector of
// the column's rows R_0 = j+1 .. j+8; step t = 0, 1, .. applies the reflector of the rows R_t = j+1+8t .. j+8+8t from both sides
// to their diagonal block D and from the right to the block Bn below it (rows R_{t+1}), which this fills, forms the reflector of
// the first column of Bn and applies it to Bn from the left, so that the next step's block starts as the band does.  A step
// therefore touches the columns R_t only, and step t of sweep j+1 needs step t+1 of sweep j and nothing later: sweep j runs step
// tick - 2 j - 1, all active sweeps (one in 15 columns) advance together, separated by a barrier per tick, 2 r ticks in all.
// (With the left product in the step after, each step reached into three blocks and the sweeps had to keep three ticks
// apart, one in 23 columns.)  No flags, no waits.  Measured, before | now: two layers of 4096 rows 14.1 | 8.0 ms, one of 1023 2.12 |
// 1.42, 96 of 1024 3.18 | 2.09; of the first, 4 ms come from the closer sweeps and 2 from the two halves below.
// The band sits in shared memory as fp64, 15 sub-diagonals (eight and the fill) per column, and four more words: a reflector
// waits for its step in those of the block's first two columns, those of the next two carry w between the lanes of D.  A step is
// two independent halves, D and Bn, each taken by four lanes of different warps: what bounds a tick where few sweeps are at work
// is the number of instructions that one warp issues one after the other (about four cycles each).  Lane k holds the rows k and
// k + 4 of its block, products with the reflector from the right are its own, and all addresses are one base plus offsets that
// never change.  (Eight lanes instead of four: half the instructions of a warp, but every vector is handed to twice as many
// lanes, and shared memory bounds a CTA with 1024 columns at work.)  A sweep stays with its lanes.  What lies outside the
// matrix is stored as zeros, lanes without a step work on a dummy block of zeros: no bounds tests.
// Larger short sides are spread over a cluster, down to 256 columns per CTA.  A cluster barrier and the reads of a
// neighbour's memory in every tick took 4.4 us per tick, three times the step itself; so a CTA also keeps copies of the
// columns next to its own, works on them as well, and gets them afresh every kChTicks ticks: its neighbours store them into
// a buffer of its own, two in turn, so that one cluster barrier separates what is stored from what is read.  What it lacks spoils these
// columns from their outer ends inwards: by eight columns a tick from above (a sweep moves down by a block), by seven from
// below (a sweep that misses its predecessor's work spoils its own block, seven columns further up), hence the widths.
namespace {
constexpr int kChLd = 20;                     // doubles per column: 16 of the band and four more; a half-warp's loads of D and Bn meet 16 different banks
constexpr int kChVec = 16;                    // where those start
constexpr int kChTicks = 8;                   // ticks between two exchanges
template <int C, int COLS> struct ChForm {     // CTAs per layer, columns per CTA
  static constexpr int kAbove = C > 1 ? 8 * kChTicks + 8 : 0, kBelow = C > 1 ? 7 * kChTicks + 8 : 16;
  static constexpr int kLocal = kAbove + COLS + kBelow;   // columns in shared memory, then eight of zeros
  static constexpr int kSteps = (kLocal - 3) / 15 + 1;    // sweeps that can be at work on them
  static constexpr int kWarps = (kSteps + 7) / 8;         // of either half
  static_assert(15 * 8 * kWarps >= kLocal - 2, "a sweep is taken up before its first step");
  static constexpr int kThreads = 2 * 32 * kWarps;
  static constexpr int kHalo = C > 1 ? kAbove + kBelow : 0;
  // the neighbours' columns arrive in two buffers in turn where there is room for them
  static constexpr bool kPush = (size_t)(kLocal + kBw + 2 * kHalo) * kChLd * sizeof(double) <= 227 * 1024;
  static constexpr size_t kSmem = (size_t)(kLocal + kBw + (kPush ? 2 * kHalo : 0)) * kChLd * sizeof(double);
};
// sum over the four lanes of a step
__device__ __forceinline__ double ch_sum(double x) {
  x += __shfl_xor_sync(0xffffffffu, x, 1);
  return x + __shfl_xor_sync(0xffffffffu, x, 2);
}
__device__ __forceinline__ double ch_dot(const double (&a)[8], const double (&u)[8]) {
  return (fma(a[0], u[0], a[1] * u[1]) + fma(a[2], u[2], a[3] * u[3])) + (fma(a[4], u[4], a[5] * u[5]) + fma(a[6], u[6], a[7] * u[7]));
}
// eight doubles from the spare words of two neighbouring columns
__device__ __forceinline__ void ch_vec(const double* p, double (&u)[8]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const double2 a = *reinterpret_cast<const double2*>(p + h * kChLd), b = *reinterpret_cast<const double2*>(p + h * kChLd + 2);
    u[4 * h] = a.x; u[4 * h + 1] = a.y; u[4 * h + 2] = b.x; u[4 * h + 3] = b.y;
  }
}
// n double2 from src to dst, either of them perhaps in a neighbour's shared memory
template <int THREADS, int N>
__device__ __forceinline__ void ch_copy(double* dst, const double* src) {
  constexpr int kMine = (N + THREADS - 1) / THREADS;
#pragma unroll 8
  for (int c = 0; c < kMine; ++c) {
    const int q = threadIdx.x + c * THREADS;
    if (q < N) reinterpret_cast<double2*>(dst)[q] = reinterpret_cast<const double2*>(src)[q];
  }
}
}  // namespace

template <int C, int COLS>
__global__ void __launch_bounds__(ChForm<C, COLS>::kThreads, 1) sp_chase_kernel(const SpLayer* __restrict__ layers, const int* __restrict__ list) {
  using F = ChForm<C, COLS>;
  constexpr int kAbove = F::kAbove, kBelow = F::kBelow, kLocal = F::kLocal, kThreads = F::kThreads, kSlots = 8 * F::kWarps;
  extern __shared__ __align__(16) double ch_smem[];
  const SpLayer& L = layers[list[blockIdx.x / C]];
  const int rank = C > 1 ? (int)(blockIdx.x % C) : 0;
  const int tid = threadIdx.x, lane = tid % 32;
  const int r = L.r;
  const double* const gB = L.bd_band;
  const int64_t row = sp_chase_row(r);                       // doubles per sweep in L.bd_V2
  const int col0 = rank * COLS, lo = col0 - kAbove;       // first own column, first column in shared memory
  double* const s_in = ch_smem + (kLocal + kBw) * kChLd;     // [2][kHalo] columns from the neighbours
  double *above = ch_smem, *below = ch_smem;                 // the neighbours' shared memory
  if (C > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    above = cluster.map_shared_rank(ch_smem, max(rank - 1, 0));
    below = cluster.map_shared_rank(ch_smem, min(rank + 1, C - 1));
  }
  for (int q = tid; q < (kLocal + kBw) * kChLd; q += kThreads) {
    const int j = lo + q / kChLd, d = q % kChLd;
    ch_smem[q] = q / kChLd < kLocal && j >= 0 && j < r && d <= kBw && j + d < r ? gB[(int64_t)j * (kBw + 1) + d] : 0.0;
  }
  if (C > 1) cg::this_cluster().sync(); else __syncthreads();
  const bool diag = tid >= kThreads / 2;                     // this warp's half of a step: D, or Bn
  const int k = tid & 3;
  // offsets of the rows k and k + 4 of D from its first diagonal entry (rows of Bn: on + (kChLd - 1) e, four further down)
  int od[2][8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    od[0][e] = e <= k ? (kChLd - 1) * e + k : (kChLd - 1) * k + e;
    od[1][e] = e <= k + 4 ? (kChLd - 1) * e + k + 4 : (kChLd - 1) * (k + 4) + e;
  }
  const int on = kBw + k;
  const int ticks = max(2 * r - 4, 0);                       // (no sweep for r < 3)
  constexpr int kLast = kLocal - kBw - 2;                    // last local start whose columns, and the next block's first two, are all here
  // sweep j's step t = tick - 2 j - 1 starts at row j + 1 + 8 t = 8 tick - 7 - 15 j (step -1: column j, seven further down).
  // Lanes go on with the sweep kSlots further when theirs has left the columns that are here.
  int j = tid % (kThreads / 2) / 4, t = -2 * j - 1, start = -7 - lo - 15 * j;   // (start: local)
  double* to2 = L.bd_V2 + j * row + k / 2 * 64 + k % 2;      // where the sweep's reflectors go: in groups of 32, entries by pairs
  for (int tick = 0; tick < ticks; ++tick) {
    if (C > 1 && tick % kChTicks == 0 && tick > 0) {         // every CTA's own columns are up to date
      cg::cluster_group cluster = cg::this_cluster();
      if (F::kPush) {
        double* const in = s_in + (tick / kChTicks & 1) * (F::kHalo * kChLd);
        const int64_t away = in - ch_smem;
        if (rank > 0) ch_copy<kThreads, kBelow * kChLd / 2>(above + away + kAbove * kChLd, ch_smem + kAbove * kChLd);
        if (rank < C - 1) ch_copy<kThreads, kAbove * kChLd / 2>(below + away, ch_smem + COLS * kChLd);
        cluster.sync();
        if (rank > 0) ch_copy<kThreads, kAbove * kChLd / 2>(ch_smem, in);
        if (rank < C - 1) ch_copy<kThreads, kBelow * kChLd / 2>(ch_smem + (kAbove + COLS) * kChLd, in + kAbove * kChLd);
        __syncthreads();
      } else {
        cluster.sync();
        if (rank > 0) ch_copy<kThreads, kAbove * kChLd / 2>(ch_smem, above + COLS * kChLd);
        if (rank < C - 1) ch_copy<kThreads, kBelow * kChLd / 2>(ch_smem + (kAbove + COLS) * kChLd, below + kAbove * kChLd);
        cluster.sync();                                      // copies taken before anybody goes on
      }
    }
    const bool first = t == -1;
    const bool active = j <= r - 3 && t >= -1 && start <= kLast && (first ? start + 7 : start) >= 0 && start + lo <= r - 2;
    if (diag) {
      if (__any_sync(0xffffffffu, active && !first)) {       // D - u w^T - w u^T, w = 2 (y - s u), y = D u, s = u^T y
        double* const pd = ch_smem + (active && !first ? start : kLocal) * kChLd;
        double* const pu = pd + kChVec;
        double u[8], dd[2][8], we[8];
        ch_vec(pu, u);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int e = 0; e < 8; ++e) dd[h][e] = pd[od[h][e]];
        const double uk[2] = {pu[k], pu[kChLd + k]};         // entries k and k + 4
        const double y[2] = {ch_dot(dd[0], u), ch_dot(dd[1], u)};
        const double s = ch_sum(fma(uk[0], y[0], uk[1] * y[1]));
        const double wk[2] = {2.0 * fma(-s, uk[0], y[0]), 2.0 * fma(-s, uk[1], y[1])};
        pu[2 * kChLd + k] = wk[0]; pu[3 * kChLd + k] = wk[1];
        __syncwarp();
        ch_vec(pu + 2 * kChLd, we);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int e = 0; e < 8; ++e) if (e <= k + 4 * h) pd[od[h][e]] = fma(-u[e], wk[h], fma(-we[e], uk[h], dd[h][e]));
      }
    } else if (__any_sync(0xffffffffu, active)) {
      double* const pd = ch_smem + (active && !first ? start : kLocal) * kChLd;
      double* const pn = pd + on;
      double* const pb = active && first ? ch_smem + (start + 7) * kChLd + 1 + k : pn;   // Bn's first column (step -1: column j)
      double u[8], bn[2][8];
      ch_vec(pd + kChVec, u);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        bn[h][0] = pb[4 * h];
#pragma unroll
        for (int e = 1; e < 8; ++e) bn[h][e] = pn[(kChLd - 1) * e + 4 * h];
      }
      // from the right, and the norm of what is now the first column
      const double p[2] = {-2.0 * ch_dot(bn[0], u), -2.0 * ch_dot(bn[1], u)};
      const double x[2] = {fma(p[0], u[0], bn[0][0]), fma(p[1], u[0], bn[1][0])};
      const double nx2 = ch_sum(fma(x[0], x[0], x[1] * x[1])), x0 = __shfl_sync(0xffffffffu, x[0], lane & 28);
#pragma unroll
      for (int e = 1; e < 8; ++e) { bn[0][e] = fma(p[0], u[e], bn[0][e]); bn[1][e] = fma(p[1], u[e], bn[1][e]); }
      // the next block's reflector (H = I for a zero column, or where it has one row only): v = x - alpha e_0, v^T v / 2 = half
      const bool more = start + lo + kBw <= r - 2, act = nx2 > 1.0e-290 && more;
      const double nx = nx2 * rsqrt(nx2);
      const double alpha = act ? -copysign(nx, x0) : x0;
      const double v[2] = {act ? (k == 0 ? x[0] - alpha : x[0]) : 0.0 * x[0], act ? x[1] : 0.0 * x[1]};
      const double us = act ? rsqrt(2.0 * fma(fabs(x0), nx, nx2)) : 0.0;      // 1 / ||v||
      double z[8];                                           // v^T Bn
#pragma unroll
      for (int e = 1; e < 8; ++e) z[e] = ch_sum(fma(v[0], bn[0][e], v[1] * bn[1][e]));
      const double un[2] = {v[0] * us, v[1] * us};           // entries k and k + 4 of the unit vector
      const double c[2] = {-2.0 * us * un[0], -2.0 * us * un[1]};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        pb[4 * h] = k == 0 && h == 0 ? alpha : 0.0;
#pragma unroll
        for (int e = 1; e < 8; ++e) pn[(kChLd - 1) * e + 4 * h] = fma(z[e], c[h], bn[h][e]);
      }
      if (active) {
        double* const to = ch_smem + (start + kBw) * kChLd + kChVec + k;
        to[0] = un[0]; to[kChLd] = un[1];
        const int own = (first ? start + 7 : start) - kAbove;
        if (more && own >= 0 && own < COLS) {
          double* const to = to2 + (t + 1) / 32 * 256 + (t + 1) % 32 * 2;
          to[0] = un[0]; to[128] = un[1];
        }
      }
    }
    __syncthreads();
    ++t; start += kBw;
    if (start > kLast) { j += kSlots; t -= 2 * kSlots; start -= 15 * kSlots; to2 += kSlots * row; }
  }
  for (int q = tid; q < COLS; q += kThreads) {
    const int jj = col0 + q;
    if (jj < r) { L.td_d[jj] = ch_smem[(size_t)(kAbove + q) * kChLd]; L.td_e[jj] = jj + 1 < r ? ch_smem[(size_t)(kAbove + q) * kChLd + 1] : 0.0; }
  }
  if (C > 1) cg::this_cluster().sync();                      // nobody leaves while a neighbour may still read its memory
}

// ---- host side ----------------------------------------------------------------------------------------------------------------
namespace {
int band_sms() {
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}
// The instances of the band kernel.  Many layers up to 1024 rows: two small CTAs per SM.  Few layers, or larger ones: one CTA of
// twelve warps per SM, a strip's columns in sixteen tasks.  Shared memory: U of the panel and the warps' rings.
struct BandForm { int max_r, threads, per_sm, parts, stages; const void* fn; };
const BandForm kBandForms[] = {
    {1024, 192, 2, 4, 4, (const void*)sp_band_kernel<192, 2, 4, 4>},
    {4096, 384, 1, 16, 4, (const void*)sp_band_kernel<384, 1, 16, 4>},
};
size_t band_smem(const BandForm& f, int r_max) { return ((size_t)(r_max + kGroup) * 8 + (size_t)f.threads / 32 * f.stages * kGroupFloats) * sizeof(float); }
constexpr size_t kChAlone = 120 * 1024;       // more than half an SM's shared memory: a CTA on its own
template <int C, int COLS> int chase_configure() {
  auto* fn = sp_chase_kernel<C, COLS>;
  const size_t smem = std::max(ChForm<C, COLS>::kSmem, C >= 8 ? kChAlone : (size_t)0);   // (the capacity is asked for with that much)
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return 1;
  if (C > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return 1;
  return 0;
}
}  // namespace

int sp_band_max_r() { return 4096; }
int sp_band_strips(int r) { return (r + kStrip - 1) / kStrip; }
int sp_band_steps(int r) { return (r + kBw - 1) / kBw; }
// Which instance a batch takes whose layers have `strips` strips in all and at most r_max rows: one for the whole batch, so that a
// larger layer's chain of panels overlaps with the others' work (both stages in one launch | the layers of up to 1024 rows apart,
// ms: 60 of 700 rows and one of 1100 12.4 | 12.7, 30 of 530 and one of 1100 8.4 | 9.8, 60 of 700 and two of 2000 21.0 | 20.0).
int sp_band_form(int r_max, int64_t strips) { return r_max <= kBandForms[0].max_r && strips > band_sms() ? 0 : 1; }
int sp_band_parts(int form) { return kBandForms[form].parts; }
// CTAs that one launch can hold together (0: not available)
int sp_band_capacity(int form, int r_max) {
  const BandForm& f = kBandForms[form];
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f.fn, f.threads, band_smem(f, r_max)) != cudaSuccess) { cudaGetLastError(); return 0; }
  return band_sms() * std::min(per, f.per_sm);
}

int sp_configure_band() {
  int bad = 0;
  for (const BandForm& f : kBandForms) {
    bad |= cudaFuncSetAttribute(f.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)band_smem(f, f.max_r)) != cudaSuccess;
    bad |= cudaFuncSetAttribute(f.fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess;
  }
  bad |= chase_configure<1, 1024>() | chase_configure<2, 1024>() | chase_configure<4, 1024>() |
         chase_configure<8, 256>() | chase_configure<16, 256>();
  if (bad) cudaGetLastError();
  return bad;
}

int launch_sp_band(const SpLayer* d_layers, const ClusterCta* d_ctas, int n_ctas, int form, int r_max, uint32_t* d_timeout, cudaStream_t st) {
  const BandForm& f = kBandForms[form];
  void* args[] = {&d_layers, &d_ctas, &d_timeout};
  return (int)cudaLaunchCooperativeKernel(f.fn, dim3((unsigned)n_ctas), dim3(f.threads), args, band_smem(f, r_max), st);
}

namespace {
template <int C, int COLS> int chase_launch(const SpLayer* d_layers, const int* d_list, int n, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n * C); cfg.blockDim = dim3(ChForm<C, COLS>::kThreads); cfg.dynamicSmemBytes = ChForm<C, COLS>::kSmem; cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = C > 1 ? 1 : 0;
  return (int)cudaLaunchKernelEx(&cfg, sp_chase_kernel<C, COLS>, d_layers, d_list);
}
}  // namespace
// Clusters of `ctas` CTAs that run side by side with an SM for each CTA (0: not available).  (The instances of 256 columns leave
// room for a second CTA on an SM; asked for as if they did not.)
int sp_chase_capacity(int ctas) {
  if (ctas == 1) return band_sms();
  const bool wide = ctas >= 8;
  const void* fn = ctas == 2 ? (const void*)sp_chase_kernel<2, 1024> : ctas == 4 ? (const void*)sp_chase_kernel<4, 1024>
                 : ctas == 8 ? (const void*)sp_chase_kernel<8, 256> : (const void*)sp_chase_kernel<16, 256>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ctas); cfg.blockDim = dim3(wide ? ChForm<8, 256>::kThreads : ChForm<2, 1024>::kThreads);
  cfg.dynamicSmemBytes = wide ? kChAlone : ChForm<2, 1024>::kSmem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)ctas; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
  return n;
}
// CTAs per layer of the chase for n layers of r rows (up to 1024, 2048 or 4096): 256 columns each while the clusters run side by
// side with an SM per CTA, else 1024 columns.  A whole encode, 256 | 1024 columns, ms: 9 of 2048 rows 25.4 | 26.9, 14 32.7 | 34.2;
// of 4096 rows 1 37.9 | 42.2, 7 100.5 | 104.8 (14 and 7 clusters fit).  Up to 1024 rows a single CTA is faster than a cluster of
// four (the chase of 1023 rows 1.42 | 1.47, of 600 rows 1.01 | 1.12) and leaves the others their SMs.
int sp_chase_ctas(int r, int n, int wide_capacity) {
  const int few = r <= 1024 ? 1 : r <= 2048 ? 2 : 4;
  return few > 1 && n <= wide_capacity ? 4 * few : few;
}
// d_list: n layers that take `ctas` CTAs each
int launch_sp_chase(const SpLayer* d_layers, const int* d_list, int n, int ctas, cudaStream_t st) {
  if (n <= 0) return 0;
  switch (ctas) {
    case 1: return chase_launch<1, 1024>(d_layers, d_list, n, st);
    case 2: return chase_launch<2, 1024>(d_layers, d_list, n, st);
    case 4: return chase_launch<4, 1024>(d_layers, d_list, n, st);
    case 8: return chase_launch<8, 256>(d_layers, d_list, n, st);
    default: return chase_launch<16, 256>(d_layers, d_list, n, st);
  }
}

}  // namespace atomo
