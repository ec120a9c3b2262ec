// Spectral atoms by the tridiagonal route (Section 5 of the paper asks for the SVD of every layer gradient; only
// the singular VALUES of all atoms enter the probabilities of Eq. 3 / Algorithm 1, and only the few KEPT atoms of
// Eq. 2 need their vectors).  For layers with a short side of at most 512:
//
//   sp_tridiag_cluster_kernel : Householder reduction of the scaled Gram matrix A (r x r) to a symmetric
//                               tridiagonal T = Q^T A Q, in fp64.  A layer's rows sit in blocks of 32 on rp/32 CTAs
//                               of a 16-CTA cluster and stay in registers; per step the product A v and the next
//                               pivot column's ingredients travel through distributed shared memory.  The
//                               reflectors go to global memory as fp32 unit vectors for the back-transformation.
//   sp_bisect_kernel          : all eigenvalues of T from Sturm counts and determinants (division-free three-term
//                               recurrence with power-of-two rescaling).
//   (sp_finalize_sample_kernel sorts, solves Algorithm 1 and draws, as for the other routes)
//   sp_eigvec_kernel          : for the kept atoms only: eigenvector of T by a twisted factorisation with one
//                               Rayleigh-quotient correction, back-transformation u = Q z with the reflectors
//                               (eight at a time, fp32), normalised short-side vector into the payload; kept atoms with
//                               nearly equal eigenvalues are orthogonalised against each other at the end, and where they are
//                               too close for vectors of their own (sp_finalize_sample_kernel), these are there already.
//
// Work per layer: about 2 r^3 fp64 flops for the reduction (full symmetric storage: matrix-vector product and
// rank-two update of the trailing block), about 11 r^2 to 32 r^2 recurrence steps for the eigenvalues, O(r^2) per kept atom.
#include <type_traits>

#include <cooperative_groups.h>

#include "atomo_kernels.cuh"
#include "atomo_twisted.cuh"

namespace cg = cooperative_groups;

namespace atomo {

namespace {

constexpr int kTriCtas = 16;          // CTAs per cluster
constexpr int kTriThreads = 256;
constexpr int kTriWarps = kTriThreads / 32;
constexpr int kTriRows = 32;          // rows of A per CTA, four per warp
constexpr int kTriMaxRp = 512;        // largest padded short side
constexpr int kTriCols = kTriMaxRp / 32;   // columns per lane
constexpr uint32_t kTriWaitLimit = 1u << 18;

}  // namespace

// ---- Householder tridiagonalisation ------------------------------------------------------------------------
// Step k (k = 0 .. r-3) with x = A[k+1.., k]:  alpha = -sign(x_0) ||x||,  v = x - alpha e_1,  beta = 2 / v^T v,
// H = I - beta v v^T;  q = A22 v,  K = beta^2/2 q^T v,  w = beta q - K v,  A22 -= v w^T + w v^T;  d_k = A[k][k],
// e_k = alpha.
// Layout: CTA g of a layer's nc = rp / 32 CTAs holds the rows 32 g .. 32 g + 31, four per warp, in registers for the
// whole reduction; a lane holds the columns lane + 32 (nc-1-m) in slot m, so that the columns still alive are the
// first slots.  The trailing block shrinks from the top left: a step works on the live slots only, and a CTA whose
// rows are all done leaves the exchange.
// A step is a chain of short dependent pieces (the fp64 work of 512 rows is 770 cycles at most, on average half of
// that), so the pieces are few: with q_i the owners also send c_i = A[i][k+1] as it is after update k-1, from which
// every CTA forms the next pivot column x_i = c_i - v_i w_{k+1} - w_i v_{k+1} itself; the update of step k and the
// product of A with that column, its first entry left out, share one pass over the rows, while the norm of the column
// is still being summed up; the reflector's first entry v_0 = x_0 - alpha is added as v_0 A[i][k+2] afterwards.  The
// entries travel as asynchronous stores into the peers' shared memory that count down a barrier there (980 cycles for
// 16 CTAs, against 1660 for stores and a cluster barrier).  Eight warps: every exchange between lanes is paid once
// per warp, and the fp64 chains of two warps per scheduler do not get in each other's way.
// 512 rows: 1408 -> 749 us, 64 rows: 148 -> 75 us (before: sixteen warps of two rows, stores and a cluster barrier, the
// reflector ahead of the pass).
__device__ __forceinline__ uint32_t tri_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t tri_map(uint32_t a, int rank) {
  uint32_t o;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(a), "r"(rank));
  return o;
}
// bounded wait for a phase of a barrier in shared memory; false if it ran out
__device__ __forceinline__ bool tri_wait(uint32_t bar, uint32_t phase) {
  for (uint32_t n = 0; n < kTriWaitLimit; ++n) {
    uint32_t ok;
    asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                 : "=r"(ok) : "r"(bar), "r"(phase) : "memory");
    if (ok) return true;
  }
  return false;
}
// sum of eight doubles in shared memory, the same bits in every thread
__device__ __forceinline__ double tri_sum8(const double* s) {
  const double2* q = reinterpret_cast<const double2*>(s);
  const double2 a = q[0], b = q[1], c = q[2], d = q[3];
  return ((a.x + a.y) + (b.x + b.y)) + ((c.x + c.y) + (d.x + d.y));
}

// an entry of each of the four register rows, slot chosen at run time (uniform over the warp): a jump, not 64 selects
#define TRI_CASE(M) case M: c[0] = row[0][M]; c[1] = row[1][M]; c[2] = row[2][M]; c[3] = row[3][M]; break;
#define TRI_PICK(slot)                                                                                    \
  switch (slot) {                                                                                         \
    TRI_CASE(0) TRI_CASE(1) TRI_CASE(2) TRI_CASE(3) TRI_CASE(4) TRI_CASE(5) TRI_CASE(6) TRI_CASE(7)       \
    TRI_CASE(8) TRI_CASE(9) TRI_CASE(10) TRI_CASE(11) TRI_CASE(12) TRI_CASE(13) TRI_CASE(14)              \
    default: c[0] = row[0][15]; c[1] = row[1][15]; c[2] = row[2][15]; c[3] = row[3][15]; break;           \
  }

__global__ void __launch_bounds__(kTriThreads, 1) sp_tridiag_cluster_kernel(const SpLayer* __restrict__ layers,
                                                                            const ClusterCta* __restrict__ ctas,
                                                                            uint32_t* __restrict__ timeout_flag) {
  static_assert(kTriCols == 16 && kTriWarps == 8 && kTriRows == 4 * kTriWarps, "TRI_PICK lists 16 slots, four rows per warp");
  cg::cluster_group cluster = cg::this_cluster();
  // the vectors' entries start at [32]: a pass over an even number of slots may run into the 32 zeros before them
  __shared__ __align__(16) double2 s_qc[2][kTriMaxRp];        // (q, c) of step k in s_qc[(k + 1) & 1] (written by the row owners)
  __shared__ __align__(16) double s_v[2][32 + kTriMaxRp];     // v of step k, likewise
  __shared__ __align__(16) double s_w[32 + kTriMaxRp];
  __shared__ __align__(16) double s_k[kTriWarps], s_n[kTriWarps];
  __shared__ __align__(16) double s_c2[kTriRows];
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ double s_x0;
  __shared__ uint32_t s_late;                                 // a thread's wait ran out
  const ClusterCta me = ctas[blockIdx.x];
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tri_smem(&s_bar[0])) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tri_smem(&s_bar[1])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_late = 0u;
  }
  for (int i = tid; i < 32 + kTriMaxRp; i += kTriThreads) { s_v[0][i] = s_v[1][i] = s_w[i] = 0.0; }
  for (int i = tid; i < kTriMaxRp; i += kTriThreads) { s_qc[0][i] = s_qc[1][i] = make_double2(0.0, 0.0); }
  cluster.sync();                                             // every CTA of the cluster runs: remote stores may start
  if (me.layer < 0) { cluster.sync(); return; }
  const SpLayer& L = layers[me.layer];
  const int r = L.r, nc = me.pad, g = me.slot, base = me.base_rank;
  // the layer's pointers in registers: a field read through `layers` inside a loop would be a global load each time
  double* const td_d = L.td_d; double* const td_e = L.td_e; float* const td_V = L.td_V;
  const float* const gA = L.A; const int64_t lda = L.lda; const int ldv = L.td_ldv;
  const int my_steps = max(r - 2, 0);
  const int row_lo = 32 * g + 4 * w;                          // this warp's rows
  double row[4][kTriCols];
#pragma unroll
  for (int m = 0; m < kTriCols; ++m) {
    const int j = lane + 32 * (nc - 1 - m);
#pragma unroll
    for (int e = 0; e < 4; ++e) row[e][m] = m < nc && j < r && row_lo + e < r ? (double)gA[(int64_t)(row_lo + e) * lda + j] : 0.0;
  }
  const int jA = tid, jB = tid + kTriThreads;                 // this thread's entries of the vectors
  // step -1: no update, the pivot column is column 0
  if (jA < r) s_qc[0][jA] = make_double2(0.0, (double)gA[jA]);
  if (jB < r) s_qc[0][jB] = make_double2(0.0, (double)gA[jB]);
  __syncthreads();
  double vA = 0.0, vB = 0.0, beta = 0.0, v0 = 0.0;            // v, beta and the first entry of v of step k
  const int e_own = lane >> 3;                                // the row whose sum this lane ends up with
  const bool files = g == (max(r, 1) - 1) >> 5;               // the CTA of the last rows, alive to the end, files T and the reflectors
  const uint32_t dst0 = tri_map(tri_smem(&s_qc[0][row_lo + e_own]), base + min(lane & 7, nc - 1));
  const uint32_t dst1 = tri_map(tri_smem(&s_qc[0][row_lo + e_own]), base + min((lane & 7) + 8, nc - 1));
  const uint32_t bar0 = tri_map(tri_smem(&s_bar[0]), base + min(lane & 7, nc - 1));
  const uint32_t bar1 = tri_map(tri_smem(&s_bar[0]), base + min((lane & 7) + 8, nc - 1));
  for (int k = -1; k < my_steps && 32 * g + 31 >= k + 2; ++k) {
    const int par = (k + 1) & 1, nxt = par ^ 1;
    const int q1 = k + 1, q2 = k + 2;
    const bool last = q1 == my_steps;                         // no reflector follows
    const int g_lo = q2 >> 5;                                 // first CTA, and first block of columns, that is still alive
    // every thread polls, but the CTA gives up as one (below, where the answer is not waited for): a thread that left alone would
    // meet the others in different barriers
    if (k >= 0 && !tri_wait(tri_smem(&s_bar[par]), (uint32_t)(k >> 1) & 1u)) s_late = 1u;
    const double2 qcA = s_qc[par][jA], qcB = s_qc[par][jB];
    const double2 qc1 = s_qc[par][min(q1, kTriMaxRp - 1)];
    // K = beta^2/2 q^T v (v is zero outside the live rows)
    const double part = warp_sum(fma(qcA.x, vA, qcB.x * vB));
    if (lane == 0) s_k[w] = part;
    __syncthreads();
    const double K = 0.5 * beta * beta * tri_sum8(s_k);
    const double w1 = fma(-K, v0, beta * qc1.x);              // w_{k+1}
    const bool inA = jA > q1 && jA < r, inB = jB > q1 && jB < r;
    const double wA = inA ? fma(-K, vA, beta * qcA.x) : 0.0, wB = inB ? fma(-K, vB, beta * qcB.x) : 0.0;
    const double xA = inA ? qcA.y - fma(vA, w1, wA * v0) : 0.0, xB = inB ? qcB.y - fma(vB, w1, wB * v0) : 0.0;
    s_w[32 + jA] = wA; s_w[32 + jB] = wB;
    s_v[nxt][32 + jA] = jA == q2 ? 0.0 : xA; s_v[nxt][32 + jB] = jB == q2 ? 0.0 : xB;
    if (jA == q2) s_x0 = xA;
    if (jB == q2) s_x0 = xB;
    if (files) {
      if (tid == (q1 & (kTriThreads - 1))) td_d[q1] = qc1.y - 2.0 * v0 * w1;
      if (last && r > 1 && tid == ((r - 1) & (kTriThreads - 1))) td_e[r - 2] = r - 1 < kTriThreads ? xA : xB;
    }
    __syncthreads();
    const bool late = s_late != 0u;
    if (tid == 0 && !last) {
      const uint32_t bytes = (uint32_t)(nc - g_lo) * kTriRows * sizeof(double2);
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tri_smem(&s_bar[nxt])), "r"(bytes) : "memory");
    }
    // update of the rows with (v, w), fused with their products with the next v; meanwhile the norm of the next column
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    double nsq = fma(xA, xA, xB * xB);
    auto pass = [&](auto n_tag) {
      constexpr int kN = decltype(n_tag)::value;
      nsq = warp_sum(nsq);
      double vi[4], wi[4];
#pragma unroll
      for (int e = 0; e < 4; e += 2) {
        const double2 v2 = *reinterpret_cast<const double2*>(&s_v[par][32 + row_lo + e]), w2 = *reinterpret_cast<const double2*>(&s_w[32 + row_lo + e]);
        vi[e] = -v2.x; vi[e + 1] = -v2.y; wi[e] = -w2.x; wi[e + 1] = -w2.y;
      }
      const int at = 32 * nc + lane;                          // slot m: [at - 32 m]
#pragma unroll
      for (int m = 0; m < kN; ++m) {
        const double vq = s_v[par][at - 32 * m], wq = s_w[at - 32 * m], vn = s_v[nxt][at - 32 * m];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          row[e][m] = fma(vi[e], wq, fma(wi[e], vq, row[e][m]));
          a[e] = fma(row[e][m], vn, a[e]);
        }
      }
    };
#define TRI_PASS(N) pass(std::integral_constant<int, N>{})
    switch (nc - g_lo) {
      case 0: case 1: TRI_PASS(1); break;
      case 2: TRI_PASS(2); break;
      case 3: case 4: TRI_PASS(4); break;
      case 5: case 6: TRI_PASS(6); break;
      case 7: case 8: TRI_PASS(8); break;
      case 9: case 10: TRI_PASS(10); break;
      case 11: case 12: TRI_PASS(12); break;
      case 13: case 14: TRI_PASS(14); break;
      default: TRI_PASS(16); break;
    }
#undef TRI_PASS
    if (lane == 0) s_n[w] = nsq;
    {                                                         // column k+2 of the rows
      double c[4];
      TRI_PICK(nc - 1 - g_lo)
      if (lane == (q2 & 31)) {
        *reinterpret_cast<double2*>(&s_c2[4 * w]) = make_double2(c[0], c[1]);
        *reinterpret_cast<double2*>(&s_c2[4 * w + 2]) = make_double2(c[2], c[3]);
      }
    }
    __syncthreads();
    const double nx2 = tri_sum8(s_n), x0 = s_x0, c2 = s_c2[4 * w + e_own];
    if (late) { *timeout_flag = 1u; break; }
    if (last) {                                               // order 1 and 2 as they are: only the last diagonal entry is left
      if (r > 1 && (lane & 7) == 0 && row_lo + e_own == r - 1) td_d[r - 1] = c2;
      break;
    }
    // the sums of the four rows over the lanes: lane ends with row lane / 8
    double sum;
    {
      const bool h4 = lane & 16, h3 = lane & 8;
      const double b0 = (h4 ? a[2] : a[0]) + __shfl_xor_sync(0xffffffffu, h4 ? a[0] : a[2], 16);
      const double b1 = (h4 ? a[3] : a[1]) + __shfl_xor_sync(0xffffffffu, h4 ? a[1] : a[3], 16);
      sum = (h3 ? b1 : b0) + __shfl_xor_sync(0xffffffffu, h3 ? b0 : b1, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    // the square root comes from the reciprocal square root; v^T v / 2 = ||x||^2 + |x_0| ||x||
    double alpha = 0.0, half = 0.0;
    v0 = 0.0;
    if (nx2 > 1.0e-140) {                                     // below: treated as a zero column (H = I), of a matrix of trace 1; beta^2 stays finite
      const double nx = nx2 * rsqrt(nx2);
      alpha = -copysign(nx, x0);
      v0 = x0 - alpha;
      half = fma(fabs(x0), nx, nx2);
    }
    // (q, c) of the rows to the CTAs that are alive in the next step; two peers per lane
    {
      const double q = fma(v0, c2, sum);
      const int peer_lo = (q2 + 1) >> 5, t = lane & 7;
      const uint32_t off = nxt * (uint32_t)sizeof(s_qc[0]), offb = nxt * (uint32_t)sizeof(s_bar[0]);
      if (t >= peer_lo && t < nc)
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(dst0 + off), "d"(q), "d"(c2), "r"(bar0 + offb) : "memory");
      if (t + 8 >= peer_lo && t + 8 < nc)
        asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(dst1 + off), "d"(q), "d"(c2), "r"(bar1 + offb) : "memory");
    }
    const double un = half > 0.0 ? rsqrt(2.0 * half) : 0.0;   // 1 / ||v||
    beta = 2.0 * un * un;
    vA = jA == q2 ? v0 : xA; vB = jB == q2 ? v0 : xB;
    if (jA == q2) s_v[nxt][32 + jA] = v0;
    if (jB == q2) s_v[nxt][32 + jB] = v0;
    if (files) {                                              // reflectors as unit vectors (H = I - 2 u u^T): no range trouble in fp32
      if (jA < r) td_V[(int64_t)q1 * ldv + jA] = (float)(vA * un);
      if (jB < r) td_V[(int64_t)q1 * ldv + jB] = (float)(vB * un);
      if (tid == 0) td_e[q1] = alpha;
    }
  }
  cluster.sync();                                             // nobody leaves while a peer may still write here
}
#undef TRI_PICK
#undef TRI_CASE

// ---- eigenvalues of T: Sturm counts -------------------------------------------------------------------------
// count(x) = number of eigenvalues below x = sign changes of p_0 = 1, p_1 = d_0 - x, p_{i+1} = (d_i - x) p_i -
// e_{i-1}^2 p_{i-1}.  The pair (p_i, p_{i-1}) is rescaled by a power of two every 8 steps (ratios and signs keep).  The last
// term, |p_r| = |det(T - x I)| up to a constant factor, comes as val * 2^ex.
struct SturmPoint { double x, val; int cnt, ex; };
// (d + 1 and e2 on 16-byte boundaries, padded with kSturmPad, far above every eigenvalue, and 0 up to eight entries past the end: there
// the step is p <- (pad - x) p, which keeps the sign.)  A step is one multiply-add in the serial chain: the operands of the next eight
// steps are fetched, the sign bits gathered and the power of two taken (from a pair two steps back) beside it.
__device__ __forceinline__ SturmPoint sturm_point(const double* __restrict__ d, const double* __restrict__ e2, int r, double x) {
  double pm = 1.0, p = d[0] - x;
  uint32_t signs = (uint32_t)__double2hiint(p) >> 31;         // the newest in bit 0
  int cnt = (int)signs, shift = 0;
  auto fetch = [&](double (&dd)[8], double (&ee)[8], int i0) {
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      const double2 a = *reinterpret_cast<const double2*>(d + i0 + u), b = *reinterpret_cast<const double2*>(e2 + i0 + u - 1);
      dd[u] = a.x; dd[u + 1] = a.y; ee[u] = b.x; ee[u + 1] = b.y;
    }
  };
  double dd[8], ee[8];
  if (r > 1) fetch(dd, ee, 1);
#pragma unroll 2
  for (int i0 = 1; i0 < r; i0 += 8) {
    double nd[8], ne[8];
    fetch(nd, ne, i0 + 8 < r ? i0 + 8 : i0);
    int top = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double pn = fma(dd[u] - x, p, -ee[u] * pm);
      signs = __funnelshift_l((uint32_t)__double2hiint(pn), signs, 1);
      pm = p; p = pn;
      if (u == 5) top = max(__double2hiint(p) & 0x7fffffff, __double2hiint(pm) & 0x7fffffff) >> 20;
    }
    cnt += __popc((signs ^ (signs >> 1)) & 0xffu);
    const int ex = max(min(top - 1023, 1022), -1022);
    const double sc = __hiloint2double((1023 - ex) << 20, 0);
    p *= sc; pm *= sc; shift += ex;
#pragma unroll
    for (int u = 0; u < 8; ++u) { dd[u] = nd[u]; ee[u] = ne[u]; }
  }
  return SturmPoint{x, fabs(p), cnt, shift};
}
// where the line through the two values crosses zero, as a part of the way from a to b (the values have opposite signs)
__device__ __forceinline__ double sturm_part(const SturmPoint& a, const SturmPoint& b) {
  const int top = max(a.ex, b.ex);
  const double va = a.val * __hiloint2double((1023 + max(a.ex - top, -1022)) << 20, 0), vb = b.val * __hiloint2double((1023 + max(b.ex - top, -1022)) << 20, 0);
  return va / fmax(va + vb, 1.0e-300);
}
__device__ __forceinline__ SturmPoint sturm_from(const SturmPoint& p, int lane) {
  return SturmPoint{__shfl_sync(0xffffffffu, p.x, lane), __shfl_sync(0xffffffffu, p.val, lane), __shfl_sync(0xffffffffu, p.cnt, lane),
                    __shfl_sync(0xffffffffu, p.ex, lane)};
}

constexpr double kSturmPad = 1.0e6;    // diagonal entries past the end (the matrices are scaled to trace <= 1)
constexpr int kBisRounds = 100;        // bound of the loop (halving the brackets alone would take 30)

// A CTA takes THREADS / LANES neighbouring eigenvalues.  Two rounds of THREADS counts bracket them: points over the whole
// spectrum, then over the part that holds the CTA's eigenvalues, so that most brackets hold a single one.  Then two or four lanes per
// eigenvalue: as long as a bracket holds several, it is cut in equal parts; after that the determinant, which the
// counts yield for nothing, says where in the bracket the eigenvalue lies, and the lanes' points are set around that crossing, at a
// distance delta (with four lanes 4 delta as well), a part of the bracket that is squared when the inner
// pair has caught the eigenvalue.  Every bracket is one by the counts: the values only choose
// the points.  Final brackets are below 4e-13 of the spectrum's extent, and the line through their values is exact to about 5e-14
// of it (the midpoint where a bracket still holds several).
// Bound: the serial chain of the recurrence with few eigenvalues (four lanes, 2 + 8 rounds), fp64 with many (two lanes, half the counts).
// Before, with sections without the values (13 rounds of eight counts, 26 of two or 41 of one) and a recurrence that
// waited for its operands | now, us: ResNet-18 set 118 | 74, one 64 x 64 layer 16.7 | 11.1, two layers of 4096 rows 2152 | 985, nine
// of 2048 1022 | 601, 96 of 1024 1724 | 1026.  One lane with a regula falsi took 1035 us on the last: a warp waits for its slowest.
template <int LANES, int THREADS>
__global__ void __launch_bounds__(THREADS) sp_bisect_kernel(const SpLayer* __restrict__ layers, int bis_stride) {
  static_assert(LANES == 2 || LANES == 4, "two lanes per eigenvalue or four");
  constexpr int kPerCta = THREADS / LANES;
  const SpLayer& L = layers[blockIdx.y];
  if (!L.tri) return;
  const int r = L.r;
  const int tid = threadIdx.x, lane = tid % 32;
  const int j0 = (int)blockIdx.x * kPerCta;
  if (j0 >= r) return;
  extern __shared__ __align__(16) double bis_smem[];           // d and e^2, r_max + 8 entries each
  double* const s_d = bis_smem + 1;                            // (entry 1 on a 16-byte boundary)
  double* const s_e2 = bis_smem + bis_stride;
  __shared__ SturmPoint s_pt[THREADS];
  __shared__ double s_lo[THREADS / 32], s_hi[THREADS / 32];
  // Gershgorin interval, widened a little; a NaN or Inf anywhere poisons the result
  double gl = 1.0e300, gu = -1.0e300;
  bool bad = false;
  for (int i = tid; i < r + 8; i += THREADS) {
    const double d = i < r ? L.td_d[i] : kSturmPad, er = i + 1 < r ? L.td_e[i] : 0.0, el = i > 0 && i < r ? L.td_e[i - 1] : 0.0;
    s_d[i] = d;
    s_e2[i] = er * er;
    if (i < r) {
      gl = fmin(gl, d - fabs(el) - fabs(er)); gu = fmax(gu, d + fabs(el) + fabs(er));
      bad |= !finite64(d) || !finite64(er * er);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) { gl = fmin(gl, __shfl_xor_sync(0xffffffffu, gl, o)); gu = fmax(gu, __shfl_xor_sync(0xffffffffu, gu, o)); }
  if (lane == 0) { s_lo[tid / 32] = gl; s_hi[tid / 32] = gu; }
  bad = __syncthreads_or(bad);
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) { gl = fmin(gl, s_lo[w]); gu = fmax(gu, s_hi[w]); }
  const int j = j0 + tid / LANES, jj = min(j, r - 1);         // ascending order; lanes past the end follow the last eigenvalue
  const bool files = tid % LANES == 0 && j < r;
  if (bad) {
    if (files) { L.lam64[j] = __longlong_as_double(0x7ff8000000000000ll); L.lam[j] = __int_as_float(0x7fc00000); }
    return;
  }
  const double pad = 1.0e-14 * fmax(fabs(gl), fabs(gu)) + 1.0e-300;
  gl -= pad; gu += pad;
  const double tol = fmax(4.0e-13 * (gu - gl), 1.0e-15 * fmax(fabs(gl), fabs(gu)));
  SturmPoint lo, hi;
  {
    const double h = (gu - gl) * (1.0 / (THREADS + 1));
    const int cnt = sturm_point(s_d, s_e2, r, fma((double)(tid + 1), h, gl)).cnt;
    const int below = __syncthreads_count(cnt <= j0), upto = __syncthreads_count(cnt <= min(j0 + kPerCta, r) - 1);
    const double a = fma((double)below, h, gl), b = upto == THREADS ? gu : fma((double)(upto + 1), h, gl);
    s_pt[tid] = sturm_point(s_d, s_e2, r, tid == THREADS - 1 ? b : fma((double)tid, (b - a) * (1.0 / (THREADS - 1)), a));
    __syncthreads();
    int first = 0, n = THREADS;                               // points whose count is at most jj come first
    while (n > 0) { const int half = n / 2; if (s_pt[first + half].cnt <= jj) { first += half + 1; n -= half + 1; } else n = half; }
    first = max(1, min(first, THREADS - 1));
    lo = s_pt[first - 1]; hi = s_pt[first];
  }
  double lam = 0.5 * (lo.x + hi.x);
  const int t = lane % LANES, base = lane - t;
  constexpr double kRho = 1.0 / 16.0, kRhoMost = LANES == 4 ? 0.125 : 0.25;
  double rho = kRho;
  bool done = false;
  for (int it = 0; it < kBisRounds; ++it) {
    const double w = hi.x - lo.x;
    const bool single = hi.cnt - lo.cnt == 1;
    const double s = fma(sturm_part(lo, hi), w, lo.x);
    if (!done) lam = single ? s : 0.5 * (lo.x + hi.x);
    done |= w <= tol;
    if (__all_sync(0xffffffffu, done)) break;
    const double delta = fmax(rho * w, 0.45 * tol);
    // the inner point of this lane's side and the outer one, inside the bracket in this order
    const bool left = t < LANES / 2, inner = LANES == 2 || t == 1 || t == 2;
    const double way = left ? s - lo.x : hi.x - s;            // from the crossing to the end on this side
    const double in = way > delta ? delta : 0.999 * way, out = way > 4.0 * delta ? 4.0 * delta : 0.5 * (in + way);
    const double off = inner ? in : out;
    const double x = single ? (left ? s - off : s + off) : fma((double)(t + 1), w * (1.0 / (LANES + 1)), lo.x);
    const SturmPoint p = sturm_point(s_d, s_e2, r, x);
    const int le = __popc(__ballot_sync(0xffffffffu, p.cnt <= jj) >> base & ((1u << LANES) - 1u));   // points not above the eigenvalue
    const SturmPoint a = sturm_from(p, base + max(le - 1, 0)), b = sturm_from(p, base + min(le, LANES - 1));
    if (!done) {
      if (le > 0) lo = a;
      if (le < LANES) hi = b;
      const double now = hi.x - lo.x;
      rho = !single ? kRho : now <= 2.01 * delta ? fmax(rho * rho, 3.8e-6) : LANES == 4 && now <= 3.03 * delta ? rho : fmin(sqrt(rho), kRhoMost);
    }
  }
  if (files) { L.lam64[j] = lam; L.lam[j] = (float)lam; }
}

// ---- vectors of the kept atoms --------------------------------------------------------------------------------
constexpr int kVecThreads = 256;
constexpr int kVecWarps = kVecThreads / 32;
constexpr int kVecCtasPerLayer = 4;   // at most
constexpr int kVecGroup = 8;          // reflectors applied together in the back-transformation
constexpr int kVecStages = 4;         // groups in flight between global and shared memory
constexpr int kVecWork = 3;           // work vectors of the twisted factorisation per warp
constexpr double kSameEig = 1.0e-9;   // scaled units (largest eigenvalue below 1): eigenvalues this close share a subspace

// One warp per kept atom, the atoms dealt to the layer's CTAs in turn.  The reflectors go in groups of eight as I - U T U^T: T is the
// inverse of the triangle that U^T U and a diagonal of 1/2 make (unit reflectors, H = I - 2 u u^T), worked out for all groups by the
// warps that have no vector of T to solve for.  A lane owns columns 4 lane .. 4 lane + 3 of every 128; the groups stream through a ring of
// kVecStages buffers filled by asynchronous copies, a row per warp, kVecStages - 1 groups ahead of use.
// Bound: the serial recurrences of the vector of T, then the chain of a group (dots, sums over the lanes, T, update).  512 rows, three kept
// atoms, four reflectors at a time with their products formed by every warp | now: ResNet-18 set 115 | 84 us
// (170 with the factorisation that waited for its operands), 40 layers of 500 rows 146 | 87, one of 64 rows 18.6 | 14.6.
__global__ void __launch_bounds__(kVecThreads, 1) sp_eigvec_kernel(const SpLayer* __restrict__ layers) {
  static_assert(kVecGroup == 8 && kVecWarps == 8, "a warp copies a row of a group");
  const SpLayer& L = layers[blockIdx.x];
  if (L.tri != 1) return;                                     // larger layers: sp_eigvec_big_kernel
  extern __shared__ __align__(16) unsigned char vec_smem[];
  const int r = L.r, rp = L.rp;
  double* s_d = reinterpret_cast<double*>(vec_smem);          // [rp]
  double* s_e = s_d + rp;                                     // [rp]
  double* s_work = s_e + rp;                                  // [warps][kVecWork][rp]
  float* s_ref = reinterpret_cast<float*>(s_work + (size_t)kVecWarps * kVecWork * rp);   // [kVecStages][kVecGroup][rp] ring of reflector groups
  float* s_t = s_ref + (size_t)kVecStages * kVecGroup * rp;   // [rp / 8][8][8] T of the groups
  __shared__ float s_dots[kVecWarps][32];
  __shared__ int s_next;                                      // groups whose T somebody has taken on
  __shared__ uint32_t s_last;
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const uint32_t k = L.hdr->k, n_ctas = gridDim.y, given = L.vec_ticket[1];
  // the layer's pointers in registers (a field read through `layers` inside a loop is a global load each time)
  const float* const gV = L.td_V; const int ldv = L.td_ldv; const double* const gLam = L.lam64;
  const int* const gPerm = L.perm; const uint32_t* const gIdx = L.idx; float* const gShort = L.shortv;
  const int nref = max(r - 2, 0);
  const int ngroups = (nref + kVecGroup - 1) / kVecGroup;
  constexpr int kQuads = kTriMaxRp / 128;
  if (blockIdx.y < k) {
    for (int i = tid; i < r; i += kVecThreads) { s_d[i] = L.td_d[i]; s_e[i] = i + 1 < r ? L.td_e[i] : 0.0; }
    if (tid == 0) s_next = 0;
    __syncthreads();
  }
  double* wa = s_work + (size_t)w * kVecWork * rp;
  double* wb = wa + rp;
  double* z = wb + rp;
  bool have_t = false;
  for (uint32_t a0 = blockIdx.y; a0 < k; a0 += n_ctas * kVecWarps) {
    const uint32_t a = a0 + n_ctas * w;
    const bool have = a < k;
    float4 zr[kQuads];                                        // z[128 m + 4 lane ..]
#pragma unroll
    for (int m = 0; m < kQuads; ++m) zr[m] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (have) {
      double n2 = 1.0;
      if (given && L.close_flag[a]) {                         // close to another kept atom's eigenvalue: sp_close_vectors has it
        for (int i = lane; i < r; i += 32) z[i] = L.tb_z[(int64_t)a * rp + i];
        __syncwarp();
      } else {
        const int ei = gPerm[gIdx[a]];                        // index of the atom's eigenvalue (ascending order)
        double lambda = gLam[ei];
        const double corr = twisted_vector(s_d, s_e, r, lambda, wa, wb, z, lane, &n2);
        // the vector's error is about |correction| / gap to the nearest other eigenvalue: well-separated atoms are done
        double gap = 1.0e300;
        if (ei > 0) gap = fmin(gap, fabs(lambda - gLam[ei - 1]));
        if (ei + 1 < r) gap = fmin(gap, fabs(gLam[ei + 1] - lambda));
        if (finite64(corr) && !(fabs(corr) <= 1.0e-9 * gap)) {   // one Rayleigh-quotient step, then the vector again
          lambda += corr;
          __syncwarp();
          twisted_vector(s_d, s_e, r, lambda, wa, wb, z, lane, &n2);
        }
      }
      const double inv = n2 > 0.0 ? rsqrt(n2) : 0.0;
#pragma unroll
      for (int m = 0; m < kQuads; ++m) {
        const int i = 128 * m + 4 * lane;
        if (i < r) zr[m] = make_float4((float)(z[i] * inv), i + 1 < r ? (float)(z[i + 1] * inv) : 0.f, i + 2 < r ? (float)(z[i + 2] * inv) : 0.f,
                                       i + 3 < r ? (float)(z[i + 3] * inv) : 0.f);
      }
    }
    if (!have_t) {                                            // T of the groups, whoever is free
      for (;;) {
        int gi = 0;
        if (lane == 0) gi = atomicAdd(&s_next, 1);
        gi = __shfl_sync(0xffffffffu, gi, 0);
        if (gi >= ngroups) break;
        float dots[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) dots[e] = 0.0f;
        for (int m = 8 * gi / 128; 128 * m < r; ++m) {
          float u[8][4];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int kk = 8 * gi + q, i = 128 * m + 4 * lane;
            const float* src = gV + (int64_t)kk * ldv + i;    // (rows of ldv floats, whole float4)
            const float4 v = kk < nref && i < r ? __ldcg(reinterpret_cast<const float4*>(src)) : make_float4(0.f, 0.f, 0.f, 0.f);
            u[q][0] = v.x; u[q][1] = i + 1 < r ? v.y : 0.f; u[q][2] = i + 2 < r ? v.z : 0.f; u[q][3] = i + 3 < r ? v.w : 0.f;
          }
          int e = 0;
#pragma unroll
          for (int x = 1; x < 8; ++x)
#pragma unroll
            for (int q = 0; q < x; ++q, ++e) dots[e] = fmaf(u[x][0], u[q][0], fmaf(u[x][1], u[q][1], fmaf(u[x][2], u[q][2], fmaf(u[x][3], u[q][3], dots[e]))));
        }
        // sums over the lanes: lane ends with pair `lane`
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const bool high = lane & o;
#pragma unroll
          for (int e = 0; e < o; ++e) {
            const float keep = high ? dots[e + o] : dots[e], send = high ? dots[e] : dots[e + o];
            dots[e] = keep + __shfl_xor_sync(0xffffffffu, send, o);
          }
        }
        s_dots[w][lane] = dots[0];
        __syncwarp();
        if (lane < 8) {                                       // column `lane` of T, from the diagonal up
          double col[8];
#pragma unroll
          for (int q = 7; q >= 0; --q) {
            double t = 0.0;
#pragma unroll
            for (int x = 7; x > q; --x) t = fma((double)s_dots[w][x * (x - 1) / 2 + q], col[x], t);
            col[q] = q > lane ? 0.0 : q == lane ? 2.0 : -2.0 * t;
          }
#pragma unroll
          for (int q = 0; q < 8; ++q) s_t[gi * 64 + q * 8 + lane] = (float)col[q];
        }
        __syncwarp();
      }
      have_t = true;
    }
    // u = H_0 H_1 ... H_{r-3} z, the groups from the last to the first, in fp32 (an orthogonal map of a unit vector whose result is
    // stored in fp32 anyway): z -= U (T (U^T z))
    auto issue_group = [&](int gi) {
      if (gi >= 0) {
        const int kk = kVecGroup * gi + w;
        const float* srow = gV + (int64_t)min(kk, max(nref - 1, 0)) * ldv;   // rows start on 16-byte boundaries (ldv is a multiple of 4)
        float* drow = s_ref + ((size_t)(gi % kVecStages) * kVecGroup + w) * rp;
        for (int i = 128 * (8 * gi / 128) + 4 * lane; i < rp; i += 128) {
          const int bytes = kk < nref ? 4 * max(0, min(4, r - i)) : 0;   // the rest of the 16 bytes is filled with zeros
          const uint32_t dst = (uint32_t)__cvta_generic_to_shared(drow + i);
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(bytes ? srow + i : gV), "r"(bytes) : "memory");
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");    // one group per call, empty or not: the counting stays uniform
    };
    for (int st = 0; st < kVecStages - 1; ++st) issue_group(ngroups - 1 - st);
    for (int gi = ngroups - 1; gi >= 0; --gi) {
      asm volatile("cp.async.wait_group %0;" ::"n"(kVecStages - 2) : "memory");
      __syncthreads();                                        // group gi has landed for everybody; the buffer of gi + 1 is free
      issue_group(gi - (kVecStages - 1));
      if (have) {
        const float* const ref = s_ref + (size_t)(gi % kVecStages) * kVecGroup * rp + 4 * lane;
        const float4* const trow = reinterpret_cast<const float4*>(s_t + gi * 64 + (lane >> 2) * 8);
        const float4 t0 = trow[0], t1 = trow[1];
        const int m0 = 8 * gi / 128;                          // (rows of the group are zero before)
        float4 u[8][kQuads];
        float p[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) p[q] = 0.0f;
#pragma unroll
        for (int m = 0; m < kQuads; ++m) {
          if (m >= m0 && 128 * m < rp) {
            const bool in = 128 * m + 4 * lane < rp;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              u[q][m] = in ? *reinterpret_cast<const float4*>(ref + q * rp + 128 * m) : make_float4(0.f, 0.f, 0.f, 0.f);
              p[q] = fmaf(u[q][m].x, zr[m].x, fmaf(u[q][m].y, zr[m].y, fmaf(u[q][m].z, zr[m].z, fmaf(u[q][m].w, zr[m].w, p[q]))));
            }
          }
        }
        // sums over the lanes: lane ends with dot lane / 4
        float sum;
        {
          float b[4], c2[2];
          const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
#pragma unroll
          for (int q = 0; q < 4; ++q) b[q] = (h4 ? p[q + 4] : p[q]) + __shfl_xor_sync(0xffffffffu, h4 ? p[q] : p[q + 4], 16);
#pragma unroll
          for (int q = 0; q < 2; ++q) c2[q] = (h3 ? b[q + 2] : b[q]) + __shfl_xor_sync(0xffffffffu, h3 ? b[q] : b[q + 2], 8);
          sum = (h2 ? c2[1] : c2[0]) + __shfl_xor_sync(0xffffffffu, h2 ? c2[0] : c2[1], 4);
          sum += __shfl_xor_sync(0xffffffffu, sum, 2);
          sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        }
        const float tt[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
        float ca = 0.0f, cb = 0.0f;                           // (T p)_{lane / 4}
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
          ca = fmaf(tt[q], __shfl_sync(0xffffffffu, sum, 4 * q), ca);
          cb = fmaf(tt[q + 1], __shfl_sync(0xffffffffu, sum, 4 * q + 4), cb);
        }
        const float mine = ca + cb;
        float c[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) c[q] = __shfl_sync(0xffffffffu, mine, 4 * q);
#pragma unroll
        for (int m = 0; m < kQuads; ++m) {
          if (m >= m0 && 128 * m < rp) {
            float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              d.x = fmaf(c[q], u[q][m].x, d.x); d.y = fmaf(c[q], u[q][m].y, d.y);
              d.z = fmaf(c[q], u[q][m].z, d.z); d.w = fmaf(c[q], u[q][m].w, d.w);
            }
            zr[m].x -= d.x; zr[m].y -= d.y; zr[m].z -= d.z; zr[m].w -= d.w;
          }
        }
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                          // the ring is free for the next atoms
    if (have) {
      float n2 = 0.0f;
#pragma unroll
      for (int m = 0; m < kQuads; ++m) n2 = fmaf(zr[m].x, zr[m].x, fmaf(zr[m].y, zr[m].y, fmaf(zr[m].z, zr[m].z, fmaf(zr[m].w, zr[m].w, n2))));
      n2 = warp_sum(n2);
      const float inv = n2 > 0.0f ? rsqrtf(n2) : 0.0f;
#pragma unroll
      for (int m = 0; m < kQuads; ++m) {
        const int i = 128 * m + 4 * lane;
        float* const dst = gShort + (int64_t)a * r + i;
        if (i < r) dst[0] = zr[m].x * inv;
        if (i + 1 < r) dst[1] = zr[m].y * inv;
        if (i + 2 < r) dst[2] = zr[m].z * inv;
        if (i + 3 < r) dst[3] = zr[m].w * inv;
      }
    }
  }
  // the last CTA of the layer orthogonalises kept atoms whose eigenvalues nearly coincide (their vectors are
  // determined only as a subspace): modified Gram-Schmidt in payload order, one warp
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(L.vec_ticket, 1u) == n_ctas - 1u ? 1u : 0u;
  __syncthreads();
  if (!s_last || w != 0 || k < 2) return;
  __threadfence();
  for (uint32_t a = 1; a < k; ++a) {
    const double la = gLam[gPerm[gIdx[a]]];
    bool changed = false;
    for (uint32_t b = 0; b < a; ++b) {
      const double lb = gLam[gPerm[gIdx[b]]];
      if (fabs(la - lb) > kSameEig || (given && fabs(la - lb) <= kCloseEig)) continue;   // (those are orthogonal already)
      volatile float* va = gShort + (int64_t)a * r;
      const volatile float* vb = gShort + (int64_t)b * r;
      double dot = 0.0;
      for (int i = lane; i < r; i += 32) dot = fma((double)va[i], (double)vb[i], dot);
      dot = warp_sum(dot);
      for (int i = lane; i < r; i += 32) va[i] = (float)((double)va[i] - dot * (double)vb[i]);
      __syncwarp();
      changed = true;
    }
    if (changed) {
      volatile float* va = gShort + (int64_t)a * r;
      double n2 = 0.0;
      for (int i = lane; i < r; i += 32) n2 = fma((double)va[i], (double)va[i], n2);
      n2 = warp_sum(n2);
      const double inv = n2 > 0.0 ? rsqrt(n2) : 0.0;
      for (int i = lane; i < r; i += 32) va[i] = (float)((double)va[i] * inv);
      __syncwarp();
    }
  }
}

// ---- host side ---------------------------------------------------------------------------------------------------
static size_t vec_smem_bytes(int rp_max) {
  return (size_t)(2 + kVecWork * kVecWarps) * rp_max * sizeof(double) + (size_t)(kVecStages * kVecGroup + 8) * rp_max * sizeof(float);
}

int sp_tridiag_max_rp() { return kTriMaxRp; }
int sp_tridiag_cluster_ctas() { return kTriCtas; }
int sp_tridiag_ctas_of(int rp) { return rp / kTriRows < 1 ? 1 : rp / kTriRows; }

// the eigenvalue kernel keeps d and e^2 of a layer in shared memory: more than the default 48 KB above a short side of
// about 3000.  Both tridiagonal routes need this (a batch may hold large layers only).  0 if it went through.
int sp_configure_bisect() {
  const int bytes = (int)(2 * (kMaxShort + 12) * sizeof(double));
  if (cudaFuncSetAttribute(sp_bisect_kernel<2, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess ||
      cudaFuncSetAttribute(sp_bisect_kernel<4, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess ||
      cudaFuncSetAttribute(sp_bisect_kernel<4, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return 0;
}

int sp_configure_tridiag() {
  // optional route: a GPU that refuses the cluster size or the shared memory simply reports it as unavailable
  if (cudaFuncSetAttribute(sp_tridiag_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaFuncSetAttribute(sp_eigvec_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vec_smem_bytes(kTriMaxRp)) != cudaSuccess ||
      sp_configure_bisect() != 0) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kTriCtas); cfg.blockDim = dim3(kTriThreads);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kTriCtas; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, sp_tridiag_cluster_kernel, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
  return n;
}

int launch_sp_tridiag(const SpLayer* d_layers, const ClusterCta* d_ctas, int n_clusters, uint32_t* d_timeout, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_clusters * kTriCtas); cfg.blockDim = dim3(kTriThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kTriCtas; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  return (int)cudaLaunchKernelEx(&cfg, sp_tridiag_cluster_kernel, d_layers, d_ctas, d_timeout);
}

void launch_sp_bisect(const SpLayer* d_layers, int n_layers, int r_max, int64_t n_eigenvalues, cudaStream_t st) {
  const int stride = (r_max + 9 + 1) & ~1;
  const size_t smem = 2 * (size_t)stride * sizeof(double);
  // two lanes per eigenvalue where there are many, else four (us, two | four: 18432 eigenvalues of 2048-row layers 601 | 764, 20000 of
  // 500-row layers 160 | 187, 4700 of the ResNet-18 set 112 | 74, 11000 of the VGG-11 set 1082 | 985)
  if (n_eigenvalues >= 16384) {
    sp_bisect_kernel<2, 64><<<dim3((r_max + 31) / 32, n_layers), 64, smem, st>>>(d_layers, stride);
  } else if (r_max > 2048) {
    // 64 KB of d and e^2 per CTA at 4096 rows: three CTAs per SM, so they are larger
    sp_bisect_kernel<4, 128><<<dim3((r_max + 31) / 32, n_layers), 128, smem, st>>>(d_layers, stride);
  } else {
    sp_bisect_kernel<4, 64><<<dim3((r_max + 15) / 16, n_layers), 64, smem, st>>>(d_layers, stride);
  }
}

void launch_sp_eigvec(const SpLayer* d_layers, int n_layers, int rp_max, cudaStream_t st) {
  // CTAs per layer (a CTA has an SM to itself): as many as keep the launch within one wave (100 layers of 64 rows with eight atoms each, four
  // CTAs | one: 56 | 44 us)
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int per = kVecCtasPerLayer;
  while (per > 1 && n_layers * per > sms) per /= 2;
  sp_eigvec_kernel<<<dim3(n_layers, per), kVecThreads, vec_smem_bytes(rp_max), st>>>(d_layers);
}

}  // namespace atomo
