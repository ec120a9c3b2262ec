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
// Then the eigenvalues of T by bisection and vectors for the kept atoms only, as on the small route; a vector of T goes
// through the chase's reflectors (sp_chase_back, used by the vector kernels of atomo_tridiag_big.cu) and then through the
// panels' (unit vectors u, H = I - 2 u u^T, rows of td_V).
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
// Panel k (c = 8 k): columns c .. c+7 below row c+7.  The rows (= columns: A is symmetric) are cut into strips of 64; a
// layer's G CTAs take the strips in turn.  A[j][i] with i in the strip is read as row j, two neighbouring entries per lane
// (256 bytes per warp), so a lane keeps everything of its two rows -- their entries of U and W of the panel before, and
// their eight sums of the product -- in registers and walks over the columns j, whose U, W and new U entries are broadcast
// from shared memory: 48 multiply-adds per 8 bytes read and written and six 16-byte broadcasts, no exchange between lanes.
// The columns of a strip are split into `parts` tasks for the warps; the parts of a sum are added in fp64 in a fixed order
// that depends on neither G nor the batch.
// A panel has two barriers among the layer's CTAs:
//   every CTA: QR of the whole panel (redundant: its entries are exchanged anyway, and the chain of eight column steps is
//              what a panel costs when little of the matrix is left)
//   pass:      own strips: update with the panel before, product with this panel's U; S = U^T A U per strip      -> barrier
//   every CTA: T^T S T; own rows: W = (A U) T - 1/2 U (T^T S T), entries of the next panel                     -> barrier
// With two CTAs per SM, which belong to different layers, one's chains and barriers overlap with the other's pass.
namespace {

struct BandShared {
  double red[2][16][8];           // per warp: parts of the panel's dots (alternating buffers)
  double m[16][36];               // per warp: parts of U^T U
  double T[8][8], S[8][8], Y[8][8], X[8][8];
  float Wc[8][8];                 // W of the next panel's pivot rows
  double piv[2][8];               // entries of the pivot row (alternating buffers)
  double M[36];
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

// barrier among the layer's CTAs (co-resident: cooperative launch), bounded; a wait that runs out shows as
// ATOMO_ERR_TIMEOUT in the layers' status words
__device__ __forceinline__ void band_barrier(uint32_t* ctr, uint32_t target, BandShared& sh, uint32_t* timeout_flag) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1u);
    uint32_t polls = 0;
    while (*(volatile uint32_t*)ctr < target && sh.fail == 0u) {
      if (++polls > kBandPollLimit) { sh.fail = 1u; *timeout_flag = 1u; }
    }
    __threadfence();
  }
  __syncthreads();
}

}  // namespace

// THREADS threads hold RPT panel rows each (as type PT); MINB CTAs per SM
template <int THREADS, int RPT, typename PT, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) sp_band_kernel(const SpLayer* __restrict__ layers, const ClusterCta* __restrict__ ctas,
                                                                const int cap, uint32_t* __restrict__ timeout_flag) {
  constexpr int kWarps = THREADS / 32;
  extern __shared__ __align__(16) float band_smem[];
  __shared__ BandShared sh;
  const ClusterCta me = ctas[blockIdx.x];
  const SpLayer& L = layers[me.layer];
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const int r = L.r, g = me.slot, G = me.pad;
  const int n_strips = (r + kStrip - 1) / kStrip;
  float* const A = L.A; const int64_t lda = L.lda;
  float* const gU = L.bd_U; float* const gW = L.bd_W; float* const gX = L.bd_X;
  double* const gPart = L.bd_part; double* const gP = L.bd_P; double* const gS = L.bd_S; double* const gB = L.bd_band;
  float* const gV = L.td_V; const int64_t ldv = L.td_ldv;
  float* const s_u = band_smem;                              // [r][8] this panel's U, by row
  float* const s_ops = band_smem + (size_t)r * 8;            // [cap][16] U and W of the panel before, columns col0 ..
  if (tid == 0) sh.fail = 0u;
  uint32_t arrivals = 0;
  // the first panel as it stands: entries A[t][i] of the own strips
  for (int s = g; s < n_strips; s += G)
    for (int q = tid; q < kStrip * 8; q += THREADS) {
      const int t = q / kStrip, i = s * kStrip + q % kStrip;
      if (i < r && t < r) gX[(int64_t)t * lda + i] = A[(int64_t)t * lda + i];
    }
  arrivals += (uint32_t)G;
  band_barrier(L.bd_bar, arrivals, sh, timeout_flag);

  for (int c = 0; c < r; c += kBw) {
    const int row0 = c + kBw;                                // first row below the band of the panel
    const int m = r - row0;                                  // panel rows
    // ---- diagonal block, QR of the panel (every CTA) ----
    if (g == 0 && tid < kBw * kBw) {
      const int a = tid / kBw, b = tid % kBw;                // entry (c + a, c + b), a >= b
      if (a >= b && c + a < r) gB[(int64_t)(c + b) * (kBw + 1) + a - b] = (double)__ldcg(gX + (int64_t)b * lda + c + a);
    }
    if (m <= 0) break;
    PT x[RPT][8];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      const int i = row0 + tid + q * THREADS;
#pragma unroll
      for (int t = 0; t < 8; ++t) x[q][t] = i < r ? (PT)__ldcg(gX + (int64_t)t * lda + i) : (PT)0;
    }
    const int n_ref = min(kBw, m - 1);                       // reflectors of this panel: rows row0 + t .. r-1, at least two of them
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      if (t < n_ref) {
        // dots of column t with the columns t .. 7 over the rows row0 + t .. (rows above carry zeros in column t: see below)
        double d[8];
#pragma unroll
        for (int l = 0; l < 8; ++l) {
          d[l] = 0.0;
          if (l >= t) {
            PT acc = (PT)0;
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
              const bool in = q > 0 || tid >= t;
              acc = in ? fma(x[q][t], x[q][l], acc) : acc;
            }
            d[l] = (double)acc;
          }
        }
        const double part = band_scatter8(d, lane);
        if ((lane & 3) == 0) sh.red[t & 1][w][lane >> 2] = part;
        if (tid == t) {
#pragma unroll
          for (int l = 0; l < 8; ++l) sh.piv[t & 1][l] = (double)x[0][l];
        }
        __syncthreads();
        double tot = 0.0;
#pragma unroll
        for (int ww = 0; ww < kWarps / 4; ++ww) tot += sh.red[t & 1][4 * ww + (lane >> 3)][lane & 7];
        tot += __shfl_xor_sync(0xffffffffu, tot, 8);
        tot += __shfl_xor_sync(0xffffffffu, tot, 16);        // lane: the dot with column lane & 7
        const double nx2 = __shfl_sync(0xffffffffu, tot, t), x0 = sh.piv[t & 1][t];
        double alpha = 0.0, beta = 0.0, un = 0.0;
        if (nx2 > 1.0e-290) {                                // below: a zero column (H = I)
          const double nx = nx2 * rsqrt(nx2);
          alpha = -copysign(nx, x0);
          const double half = fma(fabs(x0), nx, nx2);        // v^T v / 2
          un = rsqrt(2.0 * half);
          beta = 2.0 * un * un;
        }
        const double gl = beta * (tot - alpha * sh.piv[t & 1][lane & 7]);    // beta v^T x_l for l = lane & 7
        PT gc[8];
#pragma unroll
        for (int l = 0; l < 8; ++l) gc[l] = l > t ? (PT)__shfl_sync(0xffffffffu, gl, l) : (PT)0;
        const PT al = (PT)alpha, us = (PT)un;
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
          const bool below = q > 0 || tid > t, pivot = q == 0 && tid == t;
          const PT v = below ? x[q][t] : pivot ? x[q][t] - al : (PT)0;
#pragma unroll
          for (int l = 0; l < 8; ++l) if (l > t) x[q][l] = fma(-gc[l], v, x[q][l]);
          const int i = row0 + tid + q * THREADS;
          if (i < r) s_u[(size_t)i * 8 + t] = (float)(v * us);
          if (pivot) x[q][t] = al;
          // (column t of the rows below is not needed any more)
        }
      } else {
#pragma unroll
        for (int q = 0; q < RPT; ++q) { const int i = row0 + tid + q * THREADS; if (i < r) s_u[(size_t)i * 8 + t] = 0.0f; }
      }
    }
    // R: rows row0 + a (held by thread a), columns c + t, t >= a (all columns where no reflector acted)
    if (g == 0 && tid < kBw && row0 + tid < r) {
#pragma unroll
      for (int t = 0; t < 8; ++t) if (t >= tid) gB[(int64_t)(c + t) * (kBw + 1) + row0 + tid - (c + t)] = (double)x[0][t];
    }
    __syncthreads();
    // U^T U of the rounded U, 36 dots; then T (I - U T U^T is the product of the I - tau u u^T with tau = 2 / u^T u)
    {
      double acc[36];
#pragma unroll
      for (int e = 0; e < 36; ++e) acc[e] = 0.0;
      for (int i = row0 + tid; i < r; i += THREADS) {
        const float4 a = *reinterpret_cast<const float4*>(s_u + (size_t)i * 8), b = *reinterpret_cast<const float4*>(s_u + (size_t)i * 8 + 4);
        const double u[8] = {(double)a.x, (double)a.y, (double)a.z, (double)a.w, (double)b.x, (double)b.y, (double)b.z, (double)b.w};
        int e = 0;
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
          for (int q = 0; q <= p; ++q, ++e) acc[e] = fma(u[p], u[q], acc[e]);
      }
#pragma unroll
      for (int e0 = 0; e0 < 36; e0 += 8) {
        double v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = e0 + e < 36 ? acc[e0 + e < 36 ? e0 + e : 0] : 0.0;
        const double sum = band_scatter8(v, lane);
        if ((lane & 3) == 0 && e0 + (lane >> 2) < 36) sh.m[w][e0 + (lane >> 2)] = sum;
      }
      __syncthreads();
      if (w == 0) {
        for (int e = lane; e < 36; e += 32) {
          double s = 0.0;
          for (int ww = 0; ww < kWarps; ++ww) s += sh.m[ww][e];
          sh.M[e] = s;
        }
        __syncwarp();
        // column t of T: tau_t in place t, -tau_t T[0:t, 0:t] M[0:t, t] above
        for (int t = 0; t < 8; ++t) {
          const double mtt = sh.M[t * (t + 1) / 2 + t], tau = mtt > 0.5 ? 2.0 / mtt : 0.0;
          double z = 0.0;
          if (lane < t) for (int q = lane; q < t; ++q) z = fma(sh.T[lane][q], sh.M[t * (t + 1) / 2 + q], z);
          __syncwarp();
          if (lane < 8) sh.T[lane][t] = lane < t ? -tau * z : lane == t ? tau : 0.0;
          __syncwarp();
        }
      }
    }
    // the reflectors' rows for the back-transformation, own strips (zero above row0 + t)
    for (int s = g; s < n_strips; s += G)
      for (int q = tid; q < kStrip * 8; q += THREADS) {
        const int t = q / kStrip, i = s * kStrip + q % kStrip;
        if (i < r && c + t < r) gV[(int64_t)(c + t) * ldv + i] = i >= row0 + t ? s_u[(size_t)i * 8 + t] : 0.0f;
      }
    // ---- pass over the own strips ----
    const bool first = c == 0;
    const int first_strip = row0 / kStrip;
    const int s0 = first_strip + ((g - first_strip % G) % G + G) % G;      // first active strip of this CTA
    const int parts = L.bd_parts;
    const int per = ((m + parts - 1) / parts + 3) & ~3;                    // columns per task, a multiple of 4
    for (int col0 = row0; col0 < r; col0 += cap) {
      const int col1 = min(r, col0 + cap);
      if (!first) {
        __syncthreads();                                     // the block before has been used
        for (int q = tid; q < (col1 - col0) * 4; q += THREADS) {
          const int j = col0 + q / 4, h = q % 4;
          const float4* src = reinterpret_cast<const float4*>((h < 2 ? gU : gW) + (int64_t)j * 8) + (h & 1);
          reinterpret_cast<float4*>(s_ops)[(size_t)(j - col0) * 4 + h] = __ldcg(src);
        }
      }
      __syncthreads();
      // tasks (strip, part) of this block of columns, dealt to the warps; the strips of this CTA are s0, s0 + G, ...
      const int n_own = s0 < n_strips ? (n_strips - 1 - s0) / G + 1 : 0;
      for (int task = w; task < n_own * parts; task += kWarps) {
        const int s = s0 + task / parts * G, part = task % parts;
        const int jb = max(row0 + part * per, col0), je = min(min(row0 + (part + 1) * per, r), col1);
        const int i = s * kStrip + 2 * lane;
        const bool in = i < r;
        double* const dst = gPart + ((int64_t)part * n_strips * kStrip + (int64_t)s * kStrip + 2 * lane) * 8;
        if (jb >= je) {
          if (row0 + part * per >= r && col0 == row0 && in) {      // an empty part
#pragma unroll
            for (int t = 0; t < 16; t += 2) *reinterpret_cast<double2*>(dst + t) = make_double2(0.0, 0.0);
          }
          continue;
        }
        float up0[8], wp0[8], up1[8], wp1[8];
        double p0[8], p1[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) { up0[t] = wp0[t] = up1[t] = wp1[t] = 0.0f; p0[t] = p1[t] = 0.0; }
        if (in && !first) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float4 a = __ldcg(reinterpret_cast<const float4*>(gU + (int64_t)i * 8) + h), b = __ldcg(reinterpret_cast<const float4*>(gW + (int64_t)i * 8) + h);
            const float4 d = __ldcg(reinterpret_cast<const float4*>(gU + (int64_t)i * 8 + 8) + h), e = __ldcg(reinterpret_cast<const float4*>(gW + (int64_t)i * 8 + 8) + h);
            up0[4 * h] = a.x; up0[4 * h + 1] = a.y; up0[4 * h + 2] = a.z; up0[4 * h + 3] = a.w;
            wp0[4 * h] = b.x; wp0[4 * h + 1] = b.y; wp0[4 * h + 2] = b.z; wp0[4 * h + 3] = b.w;
            up1[4 * h] = d.x; up1[4 * h + 1] = d.y; up1[4 * h + 2] = d.z; up1[4 * h + 3] = d.w;
            wp1[4 * h] = e.x; wp1[4 * h + 1] = e.y; wp1[4 * h + 2] = e.z; wp1[4 * h + 3] = e.w;
          }
        }
        if (jb > row0 + part * per && in) {                  // the part began in an earlier block of columns
#pragma unroll
          for (int t = 0; t < 8; t += 2) {
            const double2 a = *reinterpret_cast<const double2*>(dst + t), b = *reinterpret_cast<const double2*>(dst + 8 + t);
            p0[t] = a.x; p0[t + 1] = a.y; p1[t] = b.x; p1[t + 1] = b.y;
          }
        }
        float q0[8], q1[8];                                  // fp32 runs of up to 32 columns
#pragma unroll
        for (int t = 0; t < 8; ++t) q0[t] = q1[t] = 0.0f;
        float* ap = A + (int64_t)jb * lda + i;
        const float4* ops = reinterpret_cast<const float4*>(s_ops) + (size_t)(jb - col0) * 4;
        const float4* un = reinterpret_cast<const float4*>(s_u) + (size_t)jb * 2;
        constexpr int kU = 4;
        float2 a[kU], an[kU];
        auto fetch = [&](float2 (&buf)[kU], int j, const float* p) {
#pragma unroll
          for (int u = 0; u < kU; ++u) buf[u] = in && j + u < je ? *reinterpret_cast<const float2*>(p + (int64_t)u * lda) : make_float2(0.f, 0.f);
        };
        auto columns = [&](float2 (&buf)[kU], int j, float* p) {
#pragma unroll
          for (int u = 0; u < kU; ++u) {
            if (j + u < je) {
              float2 v = buf[u];
              if (!first) {
                const float4 cu0 = ops[4 * u], cu1 = ops[4 * u + 1], cw0 = ops[4 * u + 2], cw1 = ops[4 * u + 3];
                const float cu[8] = {cu0.x, cu0.y, cu0.z, cu0.w, cu1.x, cu1.y, cu1.z, cu1.w};
                const float cw[8] = {cw0.x, cw0.y, cw0.z, cw0.w, cw1.x, cw1.y, cw1.z, cw1.w};
                float d0 = 0.0f, d1 = 0.0f;
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                  d0 = fmaf(up0[t], cw[t], d0); d1 = fmaf(up1[t], cw[t], d1);
                  d0 = fmaf(wp0[t], cu[t], d0); d1 = fmaf(wp1[t], cu[t], d1);
                }
                v.x -= d0; v.y -= d1;
                if (in) *reinterpret_cast<float2*>(p + (int64_t)u * lda) = v;
              }
              const float4 n0 = un[2 * u], n1 = un[2 * u + 1];
              const float cn[8] = {n0.x, n0.y, n0.z, n0.w, n1.x, n1.y, n1.z, n1.w};
#pragma unroll
              for (int t = 0; t < 8; ++t) { q0[t] = fmaf(v.x, cn[t], q0[t]); q1[t] = fmaf(v.y, cn[t], q1[t]); }
            }
          }
        };
        auto flush = [&]() {
#pragma unroll
          for (int t = 0; t < 8; ++t) { p0[t] += (double)q0[t]; p1[t] += (double)q1[t]; q0[t] = q1[t] = 0.0f; }
        };
        fetch(a, jb, ap);
        for (int j = jb, n = 0; j < je; j += 2 * kU, n += 2 * kU) {
          fetch(an, j + kU, ap + (int64_t)kU * lda);
          columns(a, j, ap);
          ops += 4 * kU; un += 2 * kU; ap += (int64_t)kU * lda;
          fetch(a, j + 2 * kU, ap + (int64_t)kU * lda);
          columns(an, j + kU, ap);
          ops += 4 * kU; un += 2 * kU; ap += (int64_t)kU * lda;
          if ((n & 31) == 24) flush();
        }
        flush();
        if (in) {
#pragma unroll
          for (int t = 0; t < 8; t += 2) {
            *reinterpret_cast<double2*>(dst + t) = make_double2(p0[t], p0[t + 1]);
            *reinterpret_cast<double2*>(dst + 8 + t) = make_double2(p1[t], p1[t + 1]);
          }
        }
      }
    }
    __syncthreads();
    // ---- P = A U of the own rows (parts added in order), S = U^T P per strip ----
    for (int s = s0; s < n_strips; s += G) {
      double acc[8];
#pragma unroll
      for (int a = 0; a < 8; ++a) acc[a] = 0.0;
      for (int q = tid; q < kStrip * 8; q += THREADS) {      // lane: row q / 8, column q % 8
        const int i = s * kStrip + q / 8;
        double p = 0.0;
        if (i < r && i >= row0) {
          for (int part = 0; part < parts; ++part) p += gPart[((int64_t)part * n_strips * kStrip + i) * 8 + q % 8];
          gP[(int64_t)i * 8 + q % 8] = p;
#pragma unroll
          for (int a = 0; a < 8; ++a) acc[a] = fma((double)s_u[(size_t)i * 8 + a], p, acc[a]);
        }
      }
#pragma unroll
      for (int a = 0; a < 8; ++a) { acc[a] += __shfl_xor_sync(0xffffffffu, acc[a], 8); acc[a] += __shfl_xor_sync(0xffffffffu, acc[a], 16); }
      double* const part_s = &sh.m[0][0];                    // [warp][64] does not fit: one value of a at a time
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        if (lane < 8) part_s[w * 8 + lane] = acc[a];
        __syncthreads();
        if (tid < 8) {
          double t = 0.0;
          for (int ww = 0; ww < kWarps; ++ww) t += part_s[ww * 8 + tid];
          gS[(int64_t)s * 64 + a * 8 + tid] = t;
        }
        __syncthreads();
      }
    }
    arrivals += (uint32_t)G;
    band_barrier(L.bd_bar, arrivals, sh, timeout_flag);
    // ---- T^T S T; W of the next panel's pivot rows (every CTA) ----
    if (tid < 64) {
      double t = 0.0;
      for (int s = first_strip; s < n_strips; ++s) t += __ldcg(gS + (int64_t)s * 64 + tid);
      sh.S[tid / 8][tid % 8] = t;
    }
    __syncthreads();
    if (tid < 64) {
      const int a = tid / 8, b = tid % 8;
      double t = 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q) t = fma(sh.S[a][q], sh.T[q][b], t);
      sh.Y[a][b] = t;
    }
    __syncthreads();
    if (tid < 64) {
      const int a = tid / 8, b = tid % 8;
      double t = 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q) t = fma(sh.T[q][a], sh.Y[q][b], t);
      sh.X[a][b] = t;
    }
    __syncthreads();
    auto w_of = [&](const double* p, int i, int t) {         // W[i][t] = sum_s P[i][s] T[s][t] - 1/2 sum_s U[i][s] X[s][t]
      double z = 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q) z = fma(p[q], sh.T[q][t], fma(-0.5 * (double)s_u[(size_t)i * 8 + q], sh.X[q][t], z));
      return z;
    };
    if (tid < 64) {
      const int a = tid / 8, i = row0 + a;
      double p[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) p[q] = i < r ? __ldcg(gP + (int64_t)i * 8 + q) : 0.0;
      sh.Wc[a][tid % 8] = i < r ? (float)w_of(p, i, tid % 8) : 0.0f;
    }
    __syncthreads();
    // ---- own rows: U, W out, entries of the next panel ----
    for (int s = s0; s < n_strips; s += G)
      for (int q = tid; q < kStrip * 8; q += THREADS) {      // entry (row, t): rows along the lanes for the panel's rows of A
        const int i = s * kStrip + q % kStrip, t = q / kStrip;
        if (i < row0 || i >= r) {
          if (i < r) { gU[(int64_t)i * 8 + t] = 0.0f; gW[(int64_t)i * 8 + t] = 0.0f; }
          continue;
        }
        double p[8];
#pragma unroll
        for (int h = 0; h < 8; ++h) p[h] = gP[(int64_t)i * 8 + h];
        const float wi = (float)w_of(p, i, t);
        gU[(int64_t)i * 8 + t] = s_u[(size_t)i * 8 + t];
        gW[(int64_t)i * 8 + t] = wi;
      }
    __syncthreads();
    for (int s = s0; s < n_strips; s += G)
      for (int q = tid; q < kStrip * 8; q += THREADS) {
        const int i = s * kStrip + q % kStrip, t = q / kStrip;
        if (i < row0 || i >= r || row0 + t >= r) continue;
        double v = (double)__ldcg(A + (int64_t)(row0 + t) * lda + i);
#pragma unroll
        for (int h = 0; h < 8; ++h)
          v -= fma((double)s_u[(size_t)i * 8 + h], (double)sh.Wc[t][h], (double)gW[(int64_t)i * 8 + h] * (double)s_u[(size_t)(row0 + t) * 8 + h]);
        gX[(int64_t)t * lda + i] = (float)v;
      }
    arrivals += (uint32_t)G;
    band_barrier(L.bd_bar, arrivals, sh, timeout_flag);
    if (sh.fail) break;
  }
}

// ---- stage 2: band -> tridiagonal -----------------------------------------------------------------------------------------
// Bulge chasing with reflectors of length eight.  Sweep j brings column j to tridiagonal form: step 0 reflects the rows
// R_0 = j+1 .. j+8 of column j; applied from both sides this fills the block below (rows R_1, columns R_0), whose first column
// step 1 reflects, and so on down the band (rows R_t = j+1+8t .. j+8+8t).  A step works on three 8 x 8 blocks: rows R_t x
// columns R_{t-1} from the left (step 0: column j), the diagonal block R_t from both sides, rows R_{t+1} x columns R_t from
// the right.  Step t of sweep j+1 needs step t+2 of sweep j, so sweep j runs step tick - 3 j: all active sweeps (one in 23
// columns) advance together, separated by a barrier per tick, 3 r ticks in all.  No flags, no waits.
// The band sits in shared memory as fp64, 15 sub-diagonals (eight and the fill) per column; sixteen lanes take a step (a lane
// holds row l mod 8 and every other column of the blocks), so that a warp advances two sweeps.
// Bound: the latency of a tick (two dependent reductions over eight lanes, two reciprocal square roots, an update), times
// 3 r.  Short sides above 1024 are spread over a cluster, 1024 columns per CTA; only steps at the edge of a CTA's columns
// touch the next CTA's memory, and the barrier per tick is the cluster's.
namespace {
constexpr int kChThreads = 736;               // 46 half-warps: 1024 columns hold at most 45 active sweeps
constexpr int kChCols = 1024;                 // columns per CTA
constexpr int kChLd = 20;                     // doubles per column: 16 in use; 19 between neighbours of a row spreads the banks
}  // namespace

template <int C>
__global__ void __launch_bounds__(kChThreads, 1) sp_chase_kernel(const SpLayer* __restrict__ layers, const int* __restrict__ list) {
  extern __shared__ __align__(16) double ch_smem[];
  const SpLayer& L = layers[list[blockIdx.x / C]];
  const int rank = C > 1 ? (int)(blockIdx.x % C) : 0;
  const int tid = threadIdx.x, lane = tid % 32;
  const int r = L.r;
  const double* const gB = L.bd_band;
  float* const gV2 = L.bd_V2;
  const int ns = (r + kBw - 1) / kBw;                        // steps per sweep that gV2 has room for
  const int col0 = rank * kChCols;
  double* peer[2] = {ch_smem, ch_smem};                      // this CTA's columns, the next one's
  if (C > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    peer[1] = cluster.map_shared_rank(ch_smem, min(rank + 1, C - 1));
  }
  for (int q = tid; q < kChCols * 16; q += kChThreads) {
    const int j = col0 + q / 16, d = q % 16;
    ch_smem[(q / 16) * kChLd + d] = j < r && d <= kBw && j + d < r ? gB[(int64_t)j * (kBw + 1) + d] : 0.0;
  }
  auto sync = [&]() { if (C > 1) cg::this_cluster().sync(); else __syncthreads(); };
  sync();
  // entry (i, j), i >= j, of this CTA's or the next one's columns (zero where it is outside the matrix or the stored diagonals)
  auto at = [&](int i, int j) -> double* {
    const int jl = j - col0;
    double* const base = C > 1 && jl >= kChCols ? peer[1] + (size_t)(jl - kChCols) * kChLd : ch_smem + (size_t)jl * kChLd;
    return base + (i - j);
  };
  const int half = tid / 16, hl = tid % 16, row = hl & 7, par = hl >> 3;   // a lane's columns of a block: par, par + 2, par + 4, par + 6
  const int ticks = 3 * (r - 3) + 1;                         // (no sweep for r < 3)
  for (int tick = 0; tick < ticks; ++tick) {
    // sweep j's step t = tick - 3 j starts at row j + 1 + 8 t = 8 tick + 1 - 23 j; this CTA takes the steps whose first column
    // is one of its own
    const int top = 8 * tick + 1;
    const int hi = col0 + kChCols - 1;                       // last column of this CTA
    const int j_lo = top - kBw > hi ? (top - kBw - hi + 22) / 23 : 0;
    const int j = j_lo + half;
    const int start = top - 23 * j, t = tick - 3 * j;
    const int prev = t > 0 ? start - kBw : j;                // first column of the block to the left
    const bool active = j <= r - 3 && t >= 0 && prev >= col0 && prev <= hi && start <= r - 2;
    if (__any_sync(0xffffffffu, active)) {
      const int i = start + row;                             // this lane's row in R_t; in R_{t+1}: i + 8
      const bool in = active && i < r, in2 = active && i + kBw < r;
      double bl[4], dd[4], bn[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int cq = par + 2 * q;
        bl[q] = in && (t > 0 || cq == 0) ? *at(i, prev + cq) : 0.0;
        const int jc = start + cq;
        dd[q] = in && jc < r ? (i >= jc ? *at(i, jc) : *at(jc, i)) : 0.0;
        bn[q] = in2 && jc < r ? *at(i + kBw, jc) : 0.0;
      }
      // reflector of the first column of the left block (lanes par == 0, q == 0)
      const double xr = __shfl_sync(0xffffffffu, bl[0], (lane & 16) | row);
      double nx2 = xr * xr;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) nx2 += __shfl_xor_sync(0xffffffffu, nx2, o);
      const double x0 = __shfl_sync(0xffffffffu, xr, lane & 16);
      double alpha = 0.0, us = 0.0;
      if (nx2 > 1.0e-290) {
        const double nx = nx2 * rsqrt(nx2);
        alpha = -copysign(nx, x0);
        us = rsqrt(2.0 * fma(fabs(x0), nx, nx2));            // 1 / ||v||
      }
      const double u = (row == 0 ? xr - alpha : xr) * us;    // unit vector; 0 for a zero column (H = I)
      double uc[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) uc[q] = __shfl_sync(0xffffffffu, u, (lane & 16) | (par + 2 * q));
      // y = D u and p = Bn u (rows), z = u^T Bl (columns)
      double y = 0.0, p = 0.0, z[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) { y = fma(dd[q], uc[q], y); p = fma(bn[q], uc[q], p); z[q] = u * bl[q]; }
      y += __shfl_xor_sync(0xffffffffu, y, 8);
      p += __shfl_xor_sync(0xffffffffu, p, 8);
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
#pragma unroll
        for (int q = 0; q < 4; ++q) z[q] += __shfl_xor_sync(0xffffffffu, z[q], o);
      }
      double s = u * y;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const double wr = 2.0 * fma(-s, u, y);                 // D - u w^T - w u^T, w = 2 (y - s u)
      double wc[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) wc[q] = __shfl_sync(0xffffffffu, wr, (lane & 16) | (par + 2 * q));
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int cq = par + 2 * q, jc = start + cq;
        if (in && (t > 0 || cq == 0)) *at(i, prev + cq) = cq == 0 ? (row == 0 ? alpha : 0.0) : fma(-2.0 * u, z[q], bl[q]);
        if (in && jc <= i) *at(i, jc) = fma(-u, wc[q], fma(-wr, uc[q], dd[q]));
        if (in2 && jc < r) *at(i + kBw, jc) = fma(-2.0 * p, uc[q], bn[q]);
      }
      if (active && par == 0) gV2[((int64_t)j * ns + t) * kBw + row] = (float)u;
    }
    sync();
  }
  for (int q = tid; q < kChCols; q += kChThreads) {
    const int j = col0 + q;
    if (j < r) { L.td_d[j] = ch_smem[(size_t)q * kChLd]; L.td_e[j] = j + 1 < r ? ch_smem[(size_t)q * kChLd + 1] : 0.0; }
  }
  if (C > 1) cg::this_cluster().sync();                      // nobody leaves while a neighbour may still reach into its memory
}

// ---- host side ----------------------------------------------------------------------------------------------------------------
namespace {
int band_sms() {
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}
// the instances of the band kernel, by the largest short side of the batch
struct BandForm { int max_r, threads, per_sm, cap; const void* fn; };
const BandForm kBandForms[] = {
    // two CTAs per SM hold U of the panel (32 B per row) and all columns' U and W of the panel before (64 B) twice over
    {1024, 256, 2, 1024, (const void*)sp_band_kernel<256, 4, double, 2>},
    {2048, 512, 1, 1024, (const void*)sp_band_kernel<512, 4, double, 1>},
    {4096, 512, 1, 1024, (const void*)sp_band_kernel<512, 8, float, 1>},
};
const BandForm& band_form(int r_max) { for (const BandForm& f : kBandForms) if (r_max <= f.max_r) return f; return kBandForms[2]; }
size_t band_smem(const BandForm& f, int r_max) { return ((size_t)r_max * 8 + (size_t)std::min(f.cap, r_max) * 16) * sizeof(float); }
size_t chase_smem() { return (size_t)kChCols * kChLd * sizeof(double); }
template <int C> int chase_configure() {
  if (cudaFuncSetAttribute(sp_chase_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)chase_smem()) != cudaSuccess) return 1;
  return 0;
}
}  // namespace

int sp_band_max_r() { return 4096; }
int sp_band_strips(int r) { return (r + kStrip - 1) / kStrip; }
// tasks that a strip's columns are split into: enough for the warps of a CTA that has few strips
int sp_band_parts(int r) { return r <= 1024 ? 4 : 16; }
int sp_band_steps(int r) { return (r + kBw - 1) / kBw; }
// CTAs that one launch can hold together, for a batch of layers of at most r_max rows (0: not available)
int sp_band_capacity(int r_max) {
  const BandForm& f = band_form(r_max);
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
  bad |= chase_configure<1>() | chase_configure<2>() | chase_configure<4>();
  if (bad) cudaGetLastError();
  return bad;
}

int launch_sp_band(const SpLayer* d_layers, const ClusterCta* d_ctas, int n_ctas, int r_max, uint32_t* d_timeout, cudaStream_t st) {
  const BandForm& f = band_form(r_max);
  int cap = std::min(f.cap, r_max);
  void* args[] = {&d_layers, &d_ctas, &cap, &d_timeout};
  return (int)cudaLaunchCooperativeKernel(f.fn, dim3((unsigned)n_ctas), dim3(f.threads), args, band_smem(f, r_max), st);
}

namespace {
template <int C> int chase_launch(const SpLayer* d_layers, const int* d_list, int n, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n * C); cfg.blockDim = dim3(kChThreads); cfg.dynamicSmemBytes = chase_smem(); cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = C > 1 ? 1 : 0;
  return (int)cudaLaunchKernelEx(&cfg, sp_chase_kernel<C>, d_layers, d_list);
}
}  // namespace
int sp_chase_ctas(int r) { return r <= kChCols ? 1 : r <= 2 * kChCols ? 2 : 4; }
// d_list: n layers that take `ctas` CTAs each
int launch_sp_chase(const SpLayer* d_layers, const int* d_list, int n, int ctas, cudaStream_t st) {
  if (n <= 0) return 0;
  switch (ctas) {
    case 1: return chase_launch<1>(d_layers, d_list, n, st);
    case 2: return chase_launch<2>(d_layers, d_list, n, st);
    default: return chase_launch<4>(d_layers, d_list, n, st);
  }
}

}  // namespace atomo
