// Spectral atoms, short sides above 512: short-side vectors of the kept atoms (the reduction that they belong to is in
// atomo_band.cu).  A vector of the tridiagonal T goes through the reflectors of the bulge chase and then through those of the
// panels: u = Q1 Q2 z.
#include <algorithm>
#include <cmath>

#include "atomo_kernels.cuh"
#include "atomo_twisted.cuh"

namespace atomo {

// ---- vectors of the kept atoms ------------------------------------------------------------------------------------
// Two phases per CTA.  (A) one warp per kept atom: the eigenvector of T by the twisted factorisation of the small
// route (work vectors in shared memory), normalised.  (B) the whole CTA takes its atoms through the
// reflectors, all in fp64 (the reflectors of the panels are fp32 numbers, and Q1 is exactly what the band reduction
// applied): first the chase's (vb_chase_back), one or two atoms at a time, then the panels' (vb_apply_reflectors), up to four at
// a time, so that their rows are read once.
// In fp32 (reflectors of the chase rounded, every application rounded) a kept atom's residual |A u - lambda u| / lambda_1 was
// 2.7e-8 instead of 1.0e-8 on 1024 x 4096 noise, its vectors orthogonal to 2.4e-7 instead of 4e-9: the eigenvector of the band
// fills eight times as many entries as one of a one-stage T, and each of its reflectors rounds them.
// Measured, before (a block barrier per sweep, four panel reflectors at a time, work vectors in global memory) | now: two layers of 4096 rows
// 8.0 | 3.7 ms, nine of 2048 rows 2.23 | 1.01, 96 of 1024 rows 1.66 | 1.02, one of 1023 rows 0.54 | 0.33.  What bounds it now:
// the panels (sums over all warps and conversions to fp64: 3500 cycles each at 1024 rows, 8500 at 4096), then the sweeps of the chase
// (290 and 640 cycles each).
// Tried and dropped: what the moves bring fetched once per turn instead of a load per sweep (spills: 3.8 -> 4.5 ms); eight warps per atom up
// to 1024 rows (1.02 -> 1.12 ms).
namespace {
constexpr int kVbThreads = 512;
constexpr int kVbWarps = kVbThreads / 32;
constexpr int kVbMaxCtas = 16;               // CTAs per layer (the kept atoms are dealt to them)
constexpr int kVbBatch = 4;                  // atoms per pass over the reflectors; two above a short side of 2048 (shared memory)
constexpr int kVbHalf = 2048;
constexpr double kVbSameEig = 1.0e-9;        // as on the small route
}  // namespace

namespace {
// The last CTA of a layer to finish orthogonalises kept atoms whose eigenvalues nearly coincide (their vectors are
// determined only as a subspace): modified Gram-Schmidt in payload order, one warp.  Called by every thread of the CTA.
__device__ __forceinline__ void vb_orthogonalise_equal(const SpLayer& L, uint32_t k, int n_ctas) {
  __shared__ uint32_t s_last;
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const int r = L.r;
  const uint32_t given = L.vec_ticket[1];
  const double* const gLam = L.lam64; const int* const gPerm = L.perm; const uint32_t* const gIdx = L.idx; float* const gShort = L.shortv;
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(L.vec_ticket, 1u) == (uint32_t)(n_ctas - 1) ? 1u : 0u;
  __syncthreads();
  if (!s_last || w != 0 || k < 2) return;
  __threadfence();
  for (uint32_t a = 1; a < k; ++a) {
    const double la = gLam[gPerm[gIdx[a]]];
    bool changed = false;
    for (uint32_t b = 0; b < a; ++b) {
      const double lb = gLam[gPerm[gIdx[b]]];
      if (fabs(la - lb) > kVbSameEig || (given && fabs(la - lb) <= kCloseEig)) continue;   // (those are orthogonal already)
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
}  // namespace


namespace {
// reduce-scatter of eight doubles over a warp: the lane ends with the sum of value lane / 4
__device__ __forceinline__ double vb_scatter8(const double (&v)[8], int lane) {
  double a[4], b[2], c;
  const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
#pragma unroll
  for (int i = 0; i < 4; ++i) a[i] = (h4 ? v[4 + i] : v[i]) + __shfl_xor_sync(0xffffffffu, h4 ? v[i] : v[4 + i], 16);
#pragma unroll
  for (int i = 0; i < 2; ++i) b[i] = (h3 ? a[2 + i] : a[i]) + __shfl_xor_sync(0xffffffffu, h3 ? a[i] : a[2 + i], 8);
  c = (h2 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, h2 ? b[0] : b[1], 4);
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  return c + __shfl_xor_sync(0xffffffffu, c, 1);
}

// z_b <- Q1 z_b for the nb vectors in s_z, the whole CTA, a panel at a time: z -= U (T (U^T z)).  A thread owns the columns tid,
// tid + THREADS, .. of the panel's eight rows, read once, in registers between the dots and the update; a column that has been
// updated makes room for the next panel's.  Panels shrink towards the last: a warp whose columns lie outside skips them.
// Reflectors kk >= nref of the last panel are rows of zeros.
template <int THREADS, int BATCH, int COLS>
__device__ __forceinline__ void vb_apply_reflectors(const float* __restrict__ gV, int64_t ldv, const double* __restrict__ gT, int r, int rp, int nref,
                                                    int nb, double* s_z, double (*s_part)[8 * BATCH], double* s_tot) {
  constexpr int kWarps = THREADS / 32;
  static_assert(BATCH <= kWarps, "a warp per vector adds the warps' parts");
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  if (nref <= 0) return;
  float q[8][COLS];
  auto load = [&](int base, int m) {
    const int h = tid + m * THREADS;
    const bool in = base >= 0 && h >= base + kBandWidth && h < r;   // reflector kk is zero below index kk + 8
    const float* v = gV + (int64_t)base * ldv + h;
#pragma unroll
    for (int x = 0; x < 8; ++x) q[x][m] = in ? __ldcg(v + x * ldv) : 0.0f;
  };
  const int top = (nref - 1) / 8 * 8;                          // the last panel's first reflector
#pragma unroll
  for (int m = 0; m < COLS; ++m) load(top, m);
  for (int base = top; base >= 0; base -= 8) {
    double2 t = make_double2(0.0, 0.0);                        // T[lane % 8][2 (lane / 8) ..]
    if (w < nb) t = __ldcg(reinterpret_cast<const double2*>(gT + (int64_t)(base / 8) * 64 + (lane & 7) * 8 + (lane >> 3) * 2));
    auto inside = [&](int m) { return 32 * w + 31 + m * THREADS >= base + kBandWidth && 32 * w + m * THREADS < r; };   // some of the warp's columns
#pragma unroll
    for (int b = 0; b < BATCH; ++b) {
      if (b < nb) {
        double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int m = 0; m < COLS; ++m) {
          if (inside(m)) {
            const int h = tid + m * THREADS;
            const double zh = h < r ? s_z[(size_t)b * rp + h] : 0.0;
#pragma unroll
            for (int x = 0; x < 8; ++x) acc[x] = fma((double)q[x][m], zh, acc[x]);
          }
        }
        const double sum = vb_scatter8(acc, lane);
        if ((lane & 3) == 0) s_part[w][8 * b + (lane >> 2)] = sum;
      }
    }
    __syncthreads();
    if (w < nb) {                                              // the vector of number w: lane's value lane % 8, of every fourth warp
      double p = 0.0;
#pragma unroll
      for (int ww = 0; ww < kWarps; ww += 4) p += s_part[ww + (lane >> 3)][8 * w + (lane & 7)];
      p += __shfl_xor_sync(0xffffffffu, p, 8);
      p += __shfl_xor_sync(0xffffffffu, p, 16);
      double c = t.x * __shfl_sync(0xffffffffu, p, (lane >> 3) * 2);
      c = fma(t.y, __shfl_sync(0xffffffffu, p, (lane >> 3) * 2 + 1), c);
      c += __shfl_xor_sync(0xffffffffu, c, 8);
      c += __shfl_xor_sync(0xffffffffu, c, 16);
      if (lane < 8) s_tot[8 * w + lane] = c;
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < BATCH; ++b) {
      if (b < nb) {
        double c[8];
#pragma unroll
        for (int x = 0; x < 8; ++x) c[x] = s_tot[8 * b + x];
#pragma unroll
        for (int m = 0; m < COLS; ++m) {
          if (inside(m)) {
            const int h = tid + m * THREADS;
            double z0 = 0.0, z1 = 0.0;
#pragma unroll
            for (int x = 0; x < 8; x += 2) { z0 = fma(c[x], (double)q[x][m], z0); z1 = fma(c[x + 1], (double)q[x + 1][m], z1); }
            if (h < r) s_z[(size_t)b * rp + h] -= z0 + z1;
          }
          if (b == nb - 1) load(base - 8, m);
        }
      }
    }
    // (two barriers separate a write to s_part or s_tot from the reads of the panel before)
  }
}
}  // namespace

// ---- back-transformation through the bulge chase -----------------------------------------------------------------------
// z <- H_first ... H_last z, the sweeps from the last to the first.  The reflectors of a sweep act on disjoint runs of eight
// entries, and from one sweep to the one before all runs move up by one entry.  A thread holds a run in registers; a
// move hands its last entry to the next thread (a shuffle, across warps through shared memory) and renames the others (the
// loop is unrolled over a whole turn of the names).  Entries only ever move towards the next warp, so warp w does the eight
// sweeps of a turn while warp w + 1 does those of the turn before: a block barrier per turn, not per sweep, and a warp takes up
// its work when its runs have come inside the matrix.  A lane's reflectors come straight into registers, DEPTH sweeps ahead.
// Bound: the reflectors, 4 r^2 bytes of fp64 per vector through one SM.
namespace {
template <int THREADS, int ATOMS, int DEPTH>
__device__ __forceinline__ void vb_chase_back(const double* __restrict__ gV2, const int r, double* s_z, const int z_stride, const int n_vecs,
                                              double (*s_edge)[THREADS / 32][8]) {
  constexpr int kPer = THREADS / ATOMS;                        // threads per vector
  static_assert(8 % DEPTH == 0, "a sweep's registers are the same in every turn");
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32, me = tid % kPer, wv = me / 32;
  double* const z = s_z + (size_t)(tid / kPer) * z_stride;
  const int turns = max(r - 2 + 7, 0) / 8;                     // the first sweeps of a partial turn act on nothing
  // the first turn in which one of the warp's entries is inside: before, they are all zeros
  const int first = tid / kPer < n_vecs ? max(0, (8 * turns + 256 * wv - r) / 8) : turns;
  const int j_first = 8 * (turns - first) - 1;
  const int64_t row = sp_chase_row(r);
  const double* from = gV2 + (j_first * row + wv * 256 + lane * 2);
  const int last = r - 3 - 8 * me;                             // the last sweep that has this thread's reflector
  double u[DEPTH][8];
  auto load = [&](double (&v)[8], int j) {
    const bool in = j >= 0 && j <= last;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double2 x = in ? __ldcg(reinterpret_cast<const double2*>(from + 64 * c)) : make_double2(0.0, 0.0);
      v[2 * c] = x.x; v[2 * c + 1] = x.y;
    }
    from -= row;
  };
  double x[8], carry = 0.0;                                    // carry: what the next turn's first move brings from the warp before
#pragma unroll
  for (int e = 0; e < 8; ++e) { const int at = j_first + 1 + me * 8 + e; x[e] = at < r ? z[at] : 0.0; }
#pragma unroll
  for (int s = 0; s < DEPTH; ++s) load(u[s], first < turns ? j_first - s : -1);
  for (int tick = 0; tick < turns + kPer / 32 - 1; ++tick) {
    const int b = tick - wv;
    if (b >= first && b < turns) {
#pragma unroll
      for (int s = 0; s < 8; ++s) {                            // entry e of the window sits in x[(e - s) mod 8]
        const int j = 8 * (turns - b) - 1 - s;
        if (s > 0 || b > first) {                              // the window moves up by one entry
          double in = __shfl_up_sync(0xffffffffu, x[(8 - s) % 8], 1);          // what was the last entry of the thread before
          if (lane == 0) in = wv == 0 ? (j + 1 < r ? z[j + 1] : 0.0) : s == 0 ? carry : s_edge[b & 1][w - 1][s - 1];
          x[(8 - s) % 8] = in;
        }
        double (&v)[8] = u[s % DEPTH];
        double d0 = 0.0, d1 = 0.0;
#pragma unroll
        for (int e = 0; e < 8; e += 2) { d0 = fma(v[e], x[(e - s + 8) % 8], d0); d1 = fma(v[e + 1], x[(e + 1 - s + 8) % 8], d1); }
        const double d = -2.0 * (d0 + d1);
#pragma unroll
        for (int e = 0; e < 8; ++e) x[(e - s + 8) % 8] = fma(d, v[e], x[(e - s + 8) % 8]);
        load(v, j - DEPTH);
        if (lane == 31) s_edge[b & 1][w][s] = x[(15 - s) % 8];
      }
      if (wv > 0) carry = s_edge[b & 1][w - 1][7];
    }
    __syncthreads();
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) { const int at = 1 + me * 8 + e; if (at < r) z[at] = x[(e + 1) % 8]; }   // after the seven moves of the last turn
  __syncthreads();
}
}  // namespace

// Short sides up to 1024, any number of layers: a small CTA (four warps) per kept atom at a time, sixteen CTAs per
// layer.  One warp forms the atom's eigenvector of T; the four warps then apply the reflectors together (a thread owns
// eight columns of every reflector row: the 16 loads of a group are in flight at once, the next group's are issued
// before this group's sums are exchanged).  With one warp per atom the same rows took four dependent batches of loads.
namespace {
constexpr int kVcThreads = 128;
constexpr int kVcWarps = kVcThreads / 32;
constexpr int kVcCtas = 16;                  // CTAs per layer
constexpr int kVcMaxRp = 1024;
}  // namespace

__global__ void __launch_bounds__(kVcThreads) sp_eigvec_big_cta_kernel(const SpLayer* __restrict__ layers,
                                                                       const int* __restrict__ big_layers) {
  const SpLayer& L = layers[big_layers[blockIdx.x]];
  if (L.rp > kVcMaxRp) return;                                 // larger layers: sp_eigvec_big_kernel
  extern __shared__ __align__(16) unsigned char vb_smem[];
  const int r = L.r, rp = L.rp;
  double* s_d = reinterpret_cast<double*>(vb_smem);            // [rp]
  double* s_e = s_d + rp;                                      // [rp]
  double* s_z = s_e + rp;                                      // [rp]
  double* const s_work = s_z + rp;                              // [2][rp], work vectors
  __shared__ double s_part[kVcWarps][8];
  __shared__ double s_tot[8];
  __shared__ double s_edge[2][kVcWarps][8];
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const uint32_t k = L.hdr->k, given = L.vec_ticket[1];
  const float* const gV = L.td_V; const int64_t ldv = L.td_ldv; const double* const gLam = L.lam64;
  const int* const gPerm = L.perm; const uint32_t* const gIdx = L.idx; float* const gShort = L.shortv;
  const int nref = max(r - kBandWidth - 1, 0);                 // a panel's reflector kk is zero up to index kk + 7
  const int slot = blockIdx.y;                                 // 0 .. 15
  if ((uint32_t)slot < k) {
    for (int i = tid; i < r; i += kVcThreads) { s_d[i] = L.td_d[i]; s_e[i] = i + 1 < r ? L.td_e[i] : 0.0; }
    __syncthreads();
    double* const wa = s_work;
    double* const wb = wa + rp;
    for (uint32_t a = slot; a < k; a += kVcCtas) {
      if (given && L.close_flag[a]) {                          // close to another kept atom's eigenvalue: sp_close_vectors has it
        for (int i = tid; i < r; i += kVcThreads) s_z[i] = L.tb_z[(int64_t)a * rp + i];
      } else if (w == 0) {
        const int ei = gPerm[gIdx[a]];                         // index of the atom's eigenvalue (ascending order)
        double lambda = gLam[ei];
        double n2 = 1.0;
        const double corr = twisted_vector(s_d, s_e, r, lambda, wa, wb, s_z, lane, &n2);
        double gap = 1.0e300;
        if (ei > 0) gap = fmin(gap, fabs(lambda - gLam[ei - 1]));
        if (ei + 1 < r) gap = fmin(gap, fabs(gLam[ei + 1] - lambda));
        if (finite64(corr) && !(fabs(corr) <= 1.0e-9 * gap)) {  // one Rayleigh-quotient step, then the vector again
          lambda += corr;
          __syncwarp();
          twisted_vector(s_d, s_e, r, lambda, wa, wb, s_z, lane, &n2);
        }
        __syncwarp();
        const double inv = n2 > 0.0 ? rsqrt(n2) : 0.0;
        for (int i = lane; i < r; i += 32) s_z[i] *= inv;
      }
      __syncthreads();
      vb_chase_back<kVcThreads, 1, 8>(L.bd_V2, r, s_z, rp, 1, s_edge);
      vb_apply_reflectors<kVcThreads, 1, kVcMaxRp / kVcThreads>(gV, ldv, L.bd_T, r, rp, nref, 1, s_z, s_part, s_tot);
      double n2 = 0.0;
      for (int i = tid; i < r; i += kVcThreads) n2 = fma(s_z[i], s_z[i], n2);
      n2 = warp_sum(n2);
      __syncthreads();
      if (lane == 0) s_part[w][0] = n2;
      __syncthreads();
      double tot = 0.0;
#pragma unroll
      for (int ww = 0; ww < kVcWarps; ++ww) tot += s_part[ww][0];
      const double inv = tot > 0.0 ? rsqrt(tot) : 0.0;
      for (int i = tid; i < r; i += kVcThreads) gShort[(int64_t)a * r + i] = (float)(s_z[i] * inv);
      __syncthreads();
    }
  }
  vb_orthogonalise_equal(L, k, kVcCtas);
}

// BATCH atoms at a time (through the chase as many as THREADS has warps for), COLS columns per thread: up to a short side of 2048, or above
template <int THREADS, int BATCH, int COLS, int DEPTH>
__global__ void __launch_bounds__(THREADS, 1) sp_eigvec_big_kernel(const SpLayer* __restrict__ layers,
                                                                      const int* __restrict__ big_layers) {
  constexpr int kRp = COLS * THREADS, kFew = THREADS * 8 / kRp, kWarps = THREADS / 32;
  const SpLayer& L = layers[big_layers[blockIdx.x]];
  if (L.rp <= kVcMaxRp || (L.rp <= kVbHalf) != (kRp <= kVbHalf)) return;   // another kernel's
  extern __shared__ __align__(16) unsigned char vb_smem[];
  const int r = L.r, rp = L.rp;
  double* s_z = reinterpret_cast<double*>(vb_smem);            // [BATCH][rp]
  double* s_d = s_z + (size_t)BATCH * rp;                      // [rp], phase A
  double* s_e = s_d + rp;                                      // [rp]
  __shared__ double s_ex[kWarps * (BATCH > 2 ? 8 * BATCH : 16)];   // what the warps exchange: in the chase's turns, in the panels' sums
  double (*const s_edge)[kWarps][8] = reinterpret_cast<double (*)[kWarps][8]>(s_ex);
  double (*const s_part)[8 * BATCH] = reinterpret_cast<double (*)[8 * BATCH]>(s_ex);
  __shared__ double s_tot[8 * BATCH];
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const int n_ctas = gridDim.y, cy = blockIdx.y;
  const uint32_t k = L.hdr->k, given = L.vec_ticket[1];
  const float* const gV = L.td_V; const int64_t ldv = L.td_ldv; const double* const gLam = L.lam64;
  const int* const gPerm = L.perm; const uint32_t* const gIdx = L.idx; float* const gShort = L.shortv;
  double* const gZ = L.tb_z;
  const int nref = max(r - kBandWidth - 1, 0);
  for (int i = tid; i < r; i += THREADS) { s_d[i] = L.td_d[i]; s_e[i] = i + 1 < r ? L.td_e[i] : 0.0; }
  __syncthreads();
  // ---- (A) this CTA's atoms are a = cy, cy + n_ctas, ...; as many warps as there is room for work vectors beside T share them ----
  constexpr int kWork = kRp <= kVbHalf ? 2 : 1;
  if (w < kWork) {
    double* const wa = s_e + rp + (size_t)w * 3 * rp;
    double* const wb = wa + rp; double* const zz = wb + rp;
    for (uint32_t a = cy + (uint32_t)n_ctas * w; a < k; a += (uint32_t)(n_ctas * kWork)) {
      if (given && L.close_flag[a]) continue;                  // in gZ already
      const int ei = gPerm[gIdx[a]];                           // index of the atom's eigenvalue (ascending order)
      double lambda = gLam[ei];
      double n2 = 1.0;
      const double corr = twisted_vector(s_d, s_e, r, lambda, wa, wb, zz, lane, &n2);
      double gap = 1.0e300;
      if (ei > 0) gap = fmin(gap, fabs(lambda - gLam[ei - 1]));
      if (ei + 1 < r) gap = fmin(gap, fabs(gLam[ei + 1] - lambda));
      if (finite64(corr) && !(fabs(corr) <= 1.0e-9 * gap)) {    // one Rayleigh-quotient step, then the vector again
        lambda += corr;
        __syncwarp();
        twisted_vector(s_d, s_e, r, lambda, wa, wb, zz, lane, &n2);
      }
      __syncwarp();
      const double inv = n2 > 0.0 ? rsqrt(n2) : 0.0;
      for (int i = lane; i < r; i += 32) gZ[(int64_t)a * rp + i] = zz[i] * inv;
      __syncwarp();
    }
  }
  __syncthreads();
  // ---- (B) back-transformation, BATCH of this CTA's atoms per pass over the reflectors ----
  const uint32_t n_mine = k > (uint32_t)cy ? (k - (uint32_t)cy + (uint32_t)n_ctas - 1u) / (uint32_t)n_ctas : 0u;
  for (uint32_t b0 = 0; b0 < n_mine; b0 += BATCH) {
    const int nb = (int)min((uint32_t)BATCH, n_mine - b0);
    for (int b = 0; b < BATCH; ++b) {
      const double* src = gZ + (int64_t)(cy + (b0 + b) * n_ctas) * rp;
      for (int i = tid; i < r; i += THREADS) s_z[(size_t)b * rp + i] = b < nb ? __ldcg(src + i) : 0.0;
    }
    __syncthreads();
    // a run per thread: one or two atoms at a time
    for (int b = 0; b < nb; b += kFew) vb_chase_back<THREADS, kFew, DEPTH>(L.bd_V2, r, s_z + (size_t)b * rp, rp, nb - b, s_edge);
    vb_apply_reflectors<THREADS, BATCH, COLS>(gV, ldv, L.bd_T, r, rp, nref, nb, s_z, s_part, s_tot);
    // normalise and file
    for (int b = 0; b < nb; ++b) {
      double n2 = 0.0;
      for (int i = tid; i < r; i += THREADS) n2 = fma(s_z[(size_t)b * rp + i], s_z[(size_t)b * rp + i], n2);
      n2 = warp_sum(n2);
      __syncthreads();
      if (lane == 0) s_part[w][0] = n2;
      __syncthreads();
      double tot = 0.0;
#pragma unroll
      for (int ww = 0; ww < kWarps; ++ww) tot += s_part[ww][0];
      const double inv = tot > 0.0 ? rsqrt(tot) : 0.0;
      float* dst = gShort + (int64_t)(cy + (b0 + b) * n_ctas) * r;
      for (int i = tid; i < r; i += THREADS) dst[i] = (float)(s_z[(size_t)b * rp + i] * inv);
    }
    __syncthreads();
  }
  vb_orthogonalise_equal(L, k, n_ctas);
}

// ---- host side ---------------------------------------------------------------------------------------------------
namespace {
// shared memory of the kernel with BATCH atoms and COLS columns per thread for a short side of rp: the vectors, T, the work
// vectors of one or two atoms
template <int BATCH> size_t vb_smem_bytes(int rp) { return (size_t)(BATCH + 2 + 3 * (rp <= kVbHalf ? 2 : 1)) * rp * sizeof(double); }
size_t vc_smem_bytes() { return (size_t)kVcMaxRp * 5 * sizeof(double); }
}  // namespace

// 0 if the kernels got their shared memory
int sp_configure_eigvec_big() {
  int bad = cudaFuncSetAttribute(sp_eigvec_big_kernel<kVbThreads / 2, kVbBatch, 8, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vb_smem_bytes<kVbBatch>(kVbHalf)) != cudaSuccess;
  bad |= cudaFuncSetAttribute(sp_eigvec_big_kernel<kVbThreads, kVbBatch, 4, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vb_smem_bytes<kVbBatch>(kVbHalf)) != cudaSuccess;
  bad |= cudaFuncSetAttribute(sp_eigvec_big_kernel<kVbThreads, 2, 8, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vb_smem_bytes<2>(kMaxShort)) != cudaSuccess;
  bad |= cudaFuncSetAttribute(sp_eigvec_big_cta_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vc_smem_bytes()) != cudaSuccess;
  if (bad) cudaGetLastError();
  return bad;
}

void launch_sp_eigvec_big(const SpLayer* d_layers, const int* d_big, int n_big, int rps, double budget, cudaStream_t st) {
  if (n_big <= 0) return;
  // layers up to a short side of 1024: a four-warp CTA per kept atom (each kernel's CTAs leave the others' layers at once)
  if (rps & 1) sp_eigvec_big_cta_kernel<<<dim3(n_big, kVcCtas), kVcThreads, vc_smem_bytes(), st>>>(d_layers, d_big);
  if (!(rps & 6)) return;
  // larger layers: CTAs per layer (1 to 16; the kept atoms are dealt to them), as many as keep the launch within one wave
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int per = 1;
  while (per < kVbMaxCtas && n_big * per * 2 <= sms) per *= 2;
  // up to a short side of 2048: one atom per CTA where the layer's CTAs are enough for the atoms to expect (the budget, and twice its root)
  // -- eight warps with twice the registers, eight sweeps of reflectors ahead --, else two at once on sixteen warps (us, one | two at
  // once: nine layers of 2048 rows at s = 2 1010 | 1183, one of 1100 at 6 448 | 500, ten of 1500 at 8 1325 | 991, 50 of 1200 at 7 2975 | 2580)
  const bool alone = budget + 2.0 * std::sqrt(budget) + 1.0 <= (double)per;
  if ((rps & 2) && alone) sp_eigvec_big_kernel<kVbThreads / 2, kVbBatch, 8, 8><<<dim3(n_big, per), kVbThreads / 2, vb_smem_bytes<kVbBatch>(kVbHalf), st>>>(d_layers, d_big);
  if ((rps & 2) && !alone) sp_eigvec_big_kernel<kVbThreads, kVbBatch, 4, 4><<<dim3(n_big, per), kVbThreads, vb_smem_bytes<kVbBatch>(kVbHalf), st>>>(d_layers, d_big);
  if (rps & 4) sp_eigvec_big_kernel<kVbThreads, 2, 8, 4><<<dim3(n_big, per), kVbThreads, vb_smem_bytes<2>(kMaxShort), st>>>(d_layers, d_big);
}

}  // namespace atomo
