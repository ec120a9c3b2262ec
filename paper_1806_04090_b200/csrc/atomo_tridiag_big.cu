// Spectral atoms, short sides above 512: short-side vectors of the kept atoms (the reduction that they belong to is in
// atomo_band.cu).  A vector of the tridiagonal T goes through the reflectors of the bulge chase and then through those of the
// panels: u = Q1 Q2 z.
#include <algorithm>

#include "atomo_kernels.cuh"
#include "atomo_twisted.cuh"

namespace atomo {

// ---- vectors of the kept atoms ------------------------------------------------------------------------------------
// Two phases per CTA.  (A) one warp per kept atom: the eigenvector of T by the twisted factorisation of the small
// route (work vectors in global memory), normalised.  (B) the whole CTA takes up to four of its atoms at once through the
// reflectors, all in fp64 (the reflectors of the panels are fp32 numbers, and Q1 is exactly what the band reduction
// applied): first the chase's (vb_chase_back), then the panels', four reflectors at a time.  There a thread owns the columns
// tid, tid + 512, ... of the four reflector rows (read once per group, kept in registers between the dot products and the
// update) and of every z (in shared memory; no other thread touches them), so the only exchange per group is the
// block-wide sum of the products p_i = u_i.z; with the group's 4 x 4 block T of the panel's triangular factor,
// z -= sum_i u_i (T p)_i.  The matrix of reflectors is read once per batch of atoms.
// In fp32 (reflectors of the chase rounded, every application rounded) a kept atom's residual |A u - lambda u| / lambda_1 was
// 2.7e-8 instead of 1.0e-8 on 1024 x 4096 noise, its vectors orthogonal to 2.4e-7 instead of 4e-9: the eigenvector of the band
// fills eight times as many entries as one of a one-stage T, and each of its reflectors rounds them.  Cost: two layers of 4096 rows 7.5 -> 8.3 ms for this and
// the back-projection, 96 of 1024 rows 1.7 -> 2.1.
namespace {
constexpr int kVbThreads = 512;
constexpr int kVbWarps = kVbThreads / 32;
constexpr int kVbSlots = 16;                 // work-vector sets per layer (phase A: 16 atoms at a time over the layer's CTAs)
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
      if (fabs(la - lb) > kVbSameEig) continue;
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
// the columns tid, tid + THREADS, ... of the four reflector rows base .. base + 3
template <int THREADS, int COLS>
__device__ __forceinline__ void vb_load_rows(const float* __restrict__ gV, int64_t ldv, int r, int base, float (&q)[4][COLS]) {
  const int tid = threadIdx.x;
  const float* v = gV + (int64_t)base * ldv;
#pragma unroll
  for (int m = 0; m < COLS; ++m) {
    const int h = tid + m * THREADS;
    const bool in = h >= base + kBandWidth && h < r;           // reflector kk is zero below index kk + 8
#pragma unroll
    for (int x = 0; x < 4; ++x) q[x][m] = in ? __ldcg(v + x * ldv + h) : 0.0f;
  }
}

// z_b <- Q1 z_b for the nb vectors in s_z, the whole CTA; the next group's rows are on their way while this group's sums are
// added up.  Reflectors kk >= nref of the last group are rows of zeros.
template <int THREADS, int BATCH, int COLS>
__device__ __forceinline__ void vb_apply_reflectors(const float* __restrict__ gV, int64_t ldv, const double* __restrict__ gT, int r, int rp, int nref,
                                                    int nb, double* s_z, double (*s_part)[4 * BATCH], double* s_tot) {
  constexpr int kSums = 4 * BATCH, kWarps = THREADS / 32;
  static_assert(kSums <= 32, "one warp adds the warps' parts");
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  float q[4][COLS], qn[4][COLS];
  const int top = (nref - 1) / 4 * 4;                          // the last group's first reflector
  if (nref > 0) vb_load_rows<THREADS, COLS>(gV, ldv, r, top, q);
  for (int base = nref > 0 ? top : -1; base >= 0; base -= 4) {
    double2 t01 = make_double2(0.0, 0.0), t23 = t01;           // row lane % 4 of the group's block of T
    if (w == 0) {
      const double* t = gT + (int64_t)(base / 8) * 64 + (base % 8 + lane % 4) * 8 + base % 8;
      t01 = __ldcg(reinterpret_cast<const double2*>(t)); t23 = __ldcg(reinterpret_cast<const double2*>(t) + 1);
    }
    double acc[kSums];
#pragma unroll
    for (int x = 0; x < kSums; ++x) acc[x] = 0.0;
#pragma unroll
    for (int m = 0; m < COLS; ++m) {
      const int h = tid + m * THREADS;
      if (h < r) {
#pragma unroll
        for (int b = 0; b < BATCH; ++b) {
          if (b < nb) {
            const double zh = s_z[(size_t)b * rp + h];
#pragma unroll
            for (int x = 0; x < 4; ++x) acc[4 * b + x] = fma((double)q[x][m], zh, acc[4 * b + x]);
          }
        }
      }
    }
    if (base >= 4) vb_load_rows<THREADS, COLS>(gV, ldv, r, base - 4, qn);
#pragma unroll
    for (int x = 0; x < kSums; ++x) {
      if (x < 4 * nb) {
        const double t = warp_sum(acc[x]);
        if (lane == 0) s_part[w][x] = t;
      }
    }
    __syncthreads();
    if (w == 0) {                                              // lane 4 b + i: (T p)_i of vector b
      double p = 0.0;
      if (lane < 4 * nb) {
#pragma unroll
        for (int ww = 0; ww < kWarps; ++ww) p += s_part[ww][lane];
      }
      const int l0 = lane & ~3;
      double s = t01.x * __shfl_sync(0xffffffffu, p, l0);      // (T is zero below its diagonal)
      s = fma(t01.y, __shfl_sync(0xffffffffu, p, l0 + 1), s);
      s = fma(t23.x, __shfl_sync(0xffffffffu, p, l0 + 2), s);
      s = fma(t23.y, __shfl_sync(0xffffffffu, p, l0 + 3), s);
      if (lane < 4 * nb) s_tot[lane] = s;
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < BATCH; ++b) {
      if (b < nb) {
        const double c0 = s_tot[4 * b], c1 = s_tot[4 * b + 1], c2 = s_tot[4 * b + 2], c3 = s_tot[4 * b + 3];
#pragma unroll
        for (int m = 0; m < COLS; ++m) {
          const int h = tid + m * THREADS;
          if (h < r) s_z[(size_t)b * rp + h] -= fma(c0, (double)q[0][m], fma(c1, (double)q[1][m], fma(c2, (double)q[2][m], c3 * (double)q[3][m])));
        }
      }
    }
    // (two barriers separate a write to s_part or s_tot from the reads of the group before)
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int m = 0; m < COLS; ++m) q[x][m] = qn[x][m];
  }
}
}  // namespace

// ---- back-transformation through the bulge chase -----------------------------------------------------------------------
// z <- H_first ... H_last z, the sweeps from the last to the first.  The reflectors of a sweep act on disjoint runs of eight
// entries, and from one sweep to the one before all runs move up by one entry.  A thread holds BPT runs in registers; a
// move hands its last entry to the next thread (a shuffle, across warps through shared memory) and renames the others (the
// loop is unrolled over a whole turn of the names).  The reflectors arrive through a ring in shared memory, kStages sweeps
// ahead, read once for all ATOMS vectors.  One block barrier per sweep.
namespace {
constexpr int kBackStages = 5;
template <int THREADS, int BPT, int ATOMS> constexpr size_t vb_ring_bytes() { return (size_t)kBackStages * (THREADS / ATOMS) * BPT * 8 * sizeof(double); }

template <int THREADS, int BPT, int ATOMS>
__device__ __forceinline__ void vb_chase_back(const double* __restrict__ gV2, const int ns, const int r, double* s_z, const int z_stride,
                                              double2* s_ring, double (*s_edge)[THREADS / 32]) {
  constexpr int kPer = THREADS / ATOMS;                        // threads per vector
  constexpr int kChunks = kPer * BPT * 4;                      // double2 per sweep
  constexpr int kW = 8 * BPT;                                  // entries per thread = sweeps per turn
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32, me = tid % kPer;
  double* const z = s_z + (size_t)(tid / kPer) * z_stride;
  const int sweeps = ((r - 2 + kW - 1) / kW) * kW;             // the first ones of a partial turn act on nothing
  auto place = [](int f) -> int {                              // chunk f of a sweep inside its stage (spread over the banks)
    const int th = f / (4 * BPT), c = f % (4 * BPT);
    return th * 4 * BPT + (c ^ (BPT == 1 ? (th >> 1) & 3 : th & 7));
  };
  // this thread's chunks of a sweep: where they go, the last sweep that has them, where they come from (sweep by sweep upwards)
  constexpr int kMine = (kChunks + THREADS - 1) / THREADS;
  uint32_t to[kMine];
  int last[kMine];
  const double* from[kMine];
#pragma unroll
  for (int c = 0; c < kMine; ++c) {
    const int f = tid + c * THREADS, t = f / 4;
    to[c] = (uint32_t)__cvta_generic_to_shared(s_ring + place(f));
    last[c] = f < kChunks ? min(r - 3, r - 3 - 8 * t) : -1;
    from[c] = gV2 + ((int64_t)(sweeps - 1) * ns + t) * 8 + (f & 3) * 2;
  }
  int fill = 0, use = 0;                                       // stages
  auto issue = [&](int j) {                                    // sweep j (none below 0: an empty group keeps the count)
    if (j >= 0) {
#pragma unroll
      for (int c = 0; c < kMine; ++c) {
        const bool ok = j <= last[c];
        if (kChunks % THREADS == 0 || tid + c * THREADS < kChunks)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to[c] + fill * (uint32_t)(kChunks * sizeof(double2))), "l"(ok ? from[c] : gV2), "r"(ok ? 16 : 0) : "memory");
        from[c] -= (int64_t)ns * 8;
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    fill = fill == kBackStages - 1 ? 0 : fill + 1;
  };
  double x[kW];
#pragma unroll
  for (int e = 0; e < kW; ++e) { const int at = sweeps + me * kW + e; x[e] = at < r ? z[at] : 0.0; }
  __syncthreads();
  for (int s = 0; s < kBackStages - 1; ++s) issue(sweeps - 1 - s);
  for (int j0 = sweeps - 1; j0 >= 0; j0 -= kW) {
#pragma unroll
    for (int s = 0; s < kW; ++s) {                             // entry e of the window sits in x[(e - s) mod kW]
      const int j = j0 - s;
      asm volatile("cp.async.wait_group %0;" ::"n"(kBackStages - 2) : "memory");
      __syncthreads();                                         // sweep j has landed for everybody; the stage of j + 1 is free
      issue(j - (kBackStages - 1));
      if (j < sweeps - 1) {                                    // the window moves up by one entry
        double in = __shfl_up_sync(0xffffffffu, x[(kW - s) % kW], 1);        // what was the last entry of the thread before
        if (lane == 0) in = me == 0 ? (j + 1 < r ? z[j + 1] : 0.0) : s_edge[(j + 1) & 1][w - 1];
        x[(kW - s) % kW] = in;
      }
      const double2* const st = s_ring + use * kChunks;
      use = use == kBackStages - 1 ? 0 : use + 1;
#pragma unroll
      for (int b = 0; b < BPT; ++b) {
        double u[8];
#pragma unroll
        for (int c = 0; c < 4; ++c) { const double2 v = st[place((me * BPT + b) * 4 + c)]; u[2 * c] = v.x; u[2 * c + 1] = v.y; }
        double d0 = 0.0, d1 = 0.0;
#pragma unroll
        for (int e = 0; e < 8; e += 2) { d0 = fma(u[e], x[(8 * b + e - s + 2 * kW) % kW], d0); d1 = fma(u[e + 1], x[(8 * b + e + 1 - s + 2 * kW) % kW], d1); }
        const double d = -2.0 * (d0 + d1);
#pragma unroll
        for (int e = 0; e < 8; ++e) x[(8 * b + e - s + 2 * kW) % kW] = fma(d, u[e], x[(8 * b + e - s + 2 * kW) % kW]);
      }
      if (lane == 31) s_edge[j & 1][w] = x[(2 * kW - 1 - s) % kW];
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
  for (int e = 0; e < kW; ++e) { const int at = 1 + me * kW + e; if (at < r) z[at] = x[(e + 1) % kW]; }   // after kW - 1 moves of the turn
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
constexpr int kVcCtas = 16;                  // CTAs per layer = work-vector sets per layer
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
  double2* s_ring = reinterpret_cast<double2*>(s_z + rp);
  __shared__ double s_part[kVcWarps][4];
  __shared__ double s_tot[4];
  __shared__ double s_edge[2][kVcWarps];
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const uint32_t k = L.hdr->k;
  const float* const gV = L.td_V; const int64_t ldv = L.td_ldv; const double* const gLam = L.lam64;
  const int* const gPerm = L.perm; const uint32_t* const gIdx = L.idx; float* const gShort = L.shortv;
  const int nref = max(r - kBandWidth - 1, 0);                 // a panel's reflector kk is zero up to index kk + 7
  const int slot = blockIdx.y;                                 // 0 .. 15
  if ((uint32_t)slot < k) {
    for (int i = tid; i < r; i += kVcThreads) { s_d[i] = L.td_d[i]; s_e[i] = i + 1 < r ? L.td_e[i] : 0.0; }
    __syncthreads();
    double* wa = L.tb_vecwork + (size_t)slot * 5 * rp;
    double* wb = wa + rp; double* wc = wb + rp; double* wd = wc + rp; double* zz = wd + rp;
    for (uint32_t a = slot; a < k; a += kVcCtas) {
      if (w == 0) {
        const int ei = gPerm[gIdx[a]];                         // index of the atom's eigenvalue (ascending order)
        double lambda = gLam[ei];
        int skip = 0;                                          // earlier kept atoms with the same eigenvalue: another twist index each
        for (uint32_t b2 = lane; b2 < a; b2 += 32) skip += fabs(gLam[gPerm[gIdx[b2]]] - lambda) <= kVbSameEig ? 1 : 0;
        skip = (int)warp_sum((uint32_t)skip);
        double n2 = 1.0;
        const double corr = twisted_vector(s_d, s_e, r, lambda, wa, wb, wc, wd, zz, lane, skip, &n2);
        double gap = 1.0e300;
        if (ei > 0) gap = fmin(gap, fabs(lambda - gLam[ei - 1]));
        if (ei + 1 < r) gap = fmin(gap, fabs(gLam[ei + 1] - lambda));
        if (finite64(corr) && skip == 0 && !(fabs(corr) <= 1.0e-9 * gap)) {  // one Rayleigh-quotient step, then the vector again
          lambda += corr;
          __syncwarp();
          twisted_vector(s_d, s_e, r, lambda, wa, wb, wc, wd, zz, lane, 0, &n2);
        }
        __syncwarp();
        const double inv = n2 > 0.0 ? rsqrt(n2) : 0.0;
        for (int i = lane; i < r; i += 32) s_z[i] = zz[i] * inv;
      }
      __syncthreads();
      vb_chase_back<kVcThreads, 1, 1>(L.bd_V2, (r + kBandWidth - 1) / kBandWidth, r, s_z, rp, s_ring, s_edge);
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

// BATCH atoms at a time, COLS columns per thread: up to a short side of 2048, or above
template <int BATCH, int COLS>
__global__ void __launch_bounds__(kVbThreads, 1) sp_eigvec_big_kernel(const SpLayer* __restrict__ layers,
                                                                      const int* __restrict__ big_layers) {
  constexpr int kRp = COLS * kVbThreads, kFew = kVbThreads * 8 / kRp;
  const SpLayer& L = layers[big_layers[blockIdx.x]];
  if (L.rp <= kVcMaxRp || (L.rp <= kVbHalf) != (kRp <= kVbHalf)) return;   // another kernel's
  extern __shared__ __align__(16) unsigned char vb_smem[];
  const int r = L.r, rp = L.rp;
  double* s_z = reinterpret_cast<double*>(vb_smem);            // [BATCH][rp]
  double* s_d = s_z + (size_t)BATCH * rp;                      // [rp], phase A
  double* s_e = s_d + rp;                                      // [rp]
  double2* s_ring = reinterpret_cast<double2*>(s_d);           // phase B
  __shared__ double s_edge[2][kVbWarps];
  __shared__ double s_part[kVbWarps][4 * BATCH];
  __shared__ double s_tot[4 * BATCH];
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const int n_ctas = gridDim.y, cy = blockIdx.y;
  const uint32_t k = L.hdr->k;
  const float* const gV = L.td_V; const int64_t ldv = L.td_ldv; const double* const gLam = L.lam64;
  const int* const gPerm = L.perm; const uint32_t* const gIdx = L.idx; float* const gShort = L.shortv;
  double* const gZ = L.tb_z;
  const int nref = max(r - kBandWidth - 1, 0);
  for (int i = tid; i < r; i += kVbThreads) { s_d[i] = L.td_d[i]; s_e[i] = i + 1 < r ? L.td_e[i] : 0.0; }
  __syncthreads();
  // ---- (A) this CTA's atoms are a = cy, cy + n_ctas, ...; warp w < slots-per-CTA takes every (slots-per-CTA)-th of them ----
  const int spc = kVbSlots / n_ctas;                           // work-vector sets of this CTA
  if (w < spc) {
    double* wa = L.tb_vecwork + (size_t)(cy * spc + w) * 5 * rp;
    double* wb = wa + rp; double* wc = wb + rp; double* wd = wc + rp; double* zz = wd + rp;
    for (uint32_t a = cy + (uint32_t)n_ctas * w; a < k; a += (uint32_t)(n_ctas * spc)) {
      const int ei = gPerm[gIdx[a]];                           // index of the atom's eigenvalue (ascending order)
      double lambda = gLam[ei];
      int skip = 0;                                            // earlier kept atoms with the same eigenvalue: another twist index each
      for (uint32_t b2 = lane; b2 < a; b2 += 32) skip += fabs(gLam[gPerm[gIdx[b2]]] - lambda) <= kVbSameEig ? 1 : 0;
      skip = (int)warp_sum((uint32_t)skip);
      double n2 = 1.0;
      const double corr = twisted_vector(s_d, s_e, r, lambda, wa, wb, wc, wd, zz, lane, skip, &n2);
      double gap = 1.0e300;
      if (ei > 0) gap = fmin(gap, fabs(lambda - gLam[ei - 1]));
      if (ei + 1 < r) gap = fmin(gap, fabs(gLam[ei + 1] - lambda));
      if (finite64(corr) && skip == 0 && !(fabs(corr) <= 1.0e-9 * gap)) {    // one Rayleigh-quotient step, then the vector again
        lambda += corr;
        __syncwarp();
        twisted_vector(s_d, s_e, r, lambda, wa, wb, wc, wd, zz, lane, 0, &n2);
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
      for (int i = tid; i < r; i += kVbThreads) s_z[(size_t)b * rp + i] = b < nb ? __ldcg(src + i) : 0.0;
    }
    __syncthreads();
    // few atoms: a run per thread and a turn of eight sweeps
    if (nb <= kFew) vb_chase_back<kVbThreads, 1, kFew>(L.bd_V2, (r + kBandWidth - 1) / kBandWidth, r, s_z, rp, s_ring, s_edge);
    else vb_chase_back<kVbThreads, COLS * BATCH / 8, BATCH>(L.bd_V2, (r + kBandWidth - 1) / kBandWidth, r, s_z, rp, s_ring, s_edge);
    vb_apply_reflectors<kVbThreads, BATCH, COLS>(gV, ldv, L.bd_T, r, rp, nref, nb, s_z, s_part, s_tot);
    // normalise and file
    for (int b = 0; b < nb; ++b) {
      double n2 = 0.0;
      for (int i = tid; i < r; i += kVbThreads) n2 = fma(s_z[(size_t)b * rp + i], s_z[(size_t)b * rp + i], n2);
      n2 = warp_sum(n2);
      __syncthreads();
      if (lane == 0) s_part[w][0] = n2;
      __syncthreads();
      double tot = 0.0;
#pragma unroll
      for (int ww = 0; ww < kVbWarps; ++ww) tot += s_part[ww][0];
      const double inv = tot > 0.0 ? rsqrt(tot) : 0.0;
      float* dst = gShort + (int64_t)(cy + (b0 + b) * n_ctas) * r;
      for (int i = tid; i < r; i += kVbThreads) dst[i] = (float)(s_z[(size_t)b * rp + i] * inv);
    }
    __syncthreads();
  }
  vb_orthogonalise_equal(L, k, n_ctas);
}

// ---- host side ---------------------------------------------------------------------------------------------------
namespace {
// shared memory of the kernel with BATCH atoms and COLS columns per thread for a short side of rp: the vectors, then the diagonals of
// T or the ring of reflectors (the larger of its two forms)
template <int BATCH, int COLS> size_t vb_smem_bytes(int rp) {
  const size_t ring = std::max(vb_ring_bytes<kVbThreads, 1, 8 / COLS>(), vb_ring_bytes<kVbThreads, COLS * BATCH / 8, BATCH>());
  return (size_t)rp * BATCH * sizeof(double) + std::max(ring, (size_t)rp * 2 * sizeof(double));
}
size_t vc_smem_bytes(int rp_max) { return (size_t)std::min(rp_max, kVcMaxRp) * 3 * sizeof(double) + vb_ring_bytes<kVcThreads, 1, 1>(); }
}  // namespace

int sp_eigvec_big_slots() { return kVbSlots; }

// 0 if the kernels got their shared memory
int sp_configure_eigvec_big() {
  int bad = cudaFuncSetAttribute(sp_eigvec_big_kernel<kVbBatch, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vb_smem_bytes<kVbBatch, 4>(kVbHalf)) != cudaSuccess;
  bad |= cudaFuncSetAttribute(sp_eigvec_big_kernel<2, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vb_smem_bytes<2, 8>(kMaxShort)) != cudaSuccess;
  bad |= cudaFuncSetAttribute(sp_eigvec_big_cta_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vc_smem_bytes(kVcMaxRp)) != cudaSuccess;
  if (bad) cudaGetLastError();
  return bad;
}

void launch_sp_eigvec_big(const SpLayer* d_layers, const int* d_big, int n_big, int rps, cudaStream_t st) {
  if (n_big <= 0) return;
  // layers up to a short side of 1024: a four-warp CTA per kept atom (each kernel's CTAs leave the others' layers at once)
  if (rps & 1) sp_eigvec_big_cta_kernel<<<dim3(n_big, kVcCtas), kVcThreads, vc_smem_bytes(kVcMaxRp), st>>>(d_layers, d_big);
  if (!(rps & 6)) return;
  // larger layers: CTAs per layer (1 to 16; the kept atoms are dealt to them), as many as keep the launch within one wave
  int dev = 0, sms = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int per = 1;
  while (per < kVbMaxCtas && n_big * per * 2 <= sms) per *= 2;
  if (rps & 2) sp_eigvec_big_kernel<kVbBatch, 4><<<dim3(n_big, per), kVbThreads, vb_smem_bytes<kVbBatch, 4>(kVbHalf), st>>>(d_layers, d_big);
  if (rps & 4) sp_eigvec_big_kernel<2, 8><<<dim3(n_big, per), kVbThreads, vb_smem_bytes<2, 8>(kMaxShort), st>>>(d_layers, d_big);
}

}  // namespace atomo
