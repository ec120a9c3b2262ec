// Spectral atoms, short sides above 512: short-side vectors of the kept atoms (the reduction that they belong to is in
// atomo_band.cu).  A vector of the tridiagonal T goes through the reflectors of the bulge chase and then through those of the
// panels: u = Q1 Q2 z.
#include <algorithm>

#include "atomo_kernels.cuh"
#include "atomo_twisted.cuh"

namespace atomo {

// ---- vectors of the kept atoms ------------------------------------------------------------------------------------
// Two phases per CTA.  (A) one warp per kept atom: the eigenvector of T by the twisted factorisation of the small
// route (work vectors in global memory), normalised, filed in the payload's slot of the atom.  (B) the whole CTA
// applies the reflectors to up to four of its atoms at once, u = H_0 H_1 ... H_{r-3} z with H = I - 2 v v^T, from the
// last reflector to the first, four at a time: a thread owns the columns tid, tid + 512, ... of the four reflector rows
// (read once per group, kept in registers between the dot products and the update) and of every z (in shared memory;
// no other thread touches them), so the only exchange per group is the block-wide sum of the products: v_i.z for
// every atom and the six v_i.v_j.  For a group applied in the order 0, 1, 2, 3:  c_0 = 2 v_0.z,
// c_i = 2 (v_i.z - sum_{j<i} c_j v_i.v_j),  z -= sum c_i v_i.  The matrix of reflectors is read once per four atoms
// instead of once per atom, by 512 threads instead of 32.
namespace {
constexpr int kVbThreads = 512;
constexpr int kVbWarps = kVbThreads / 32;
constexpr int kVbSlots = 16;                 // work-vector sets per layer (phase A: 16 atoms at a time over the layer's CTAs)
constexpr int kVbMaxCtas = 16;               // CTAs per layer (the kept atoms are dealt to them)
constexpr int kVbBatch = 4;                  // atoms per pass over the reflectors
constexpr int kVbSums = 4 * kVbBatch + 6;    // products summed per group
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
// the columns tid, tid + THREADS, ... of the four reflector rows top, top - 1, top - 2, top - 3 (rows below 0: zeros)
template <int THREADS, int COLS>
__device__ __forceinline__ void vb_load_rows(const float* __restrict__ gV, int64_t ldv, int r, int top, float (&q)[4][COLS]) {
  const int tid = threadIdx.x;
  const float* v0 = gV + (int64_t)top * ldv;
  const float* v1 = gV + (int64_t)max(top - 1, 0) * ldv;
  const float* v2 = gV + (int64_t)max(top - 2, 0) * ldv;
  const float* v3 = gV + (int64_t)max(top - 3, 0) * ldv;
  const bool e1 = top - 1 >= 0, e2 = top - 2 >= 0, e3 = top - 3 >= 0;
  const int h0 = max(top - 3, 0) + kBandWidth;                 // reflector kk is zero below index kk + 8
#pragma unroll
  for (int m = 0; m < COLS; ++m) {
    const int h = tid + m * THREADS;
    const bool in = h >= h0 && h < r;
    q[0][m] = in ? __ldcg(v0 + h) : 0.0f;
    q[1][m] = in && e1 ? __ldcg(v1 + h) : 0.0f;
    q[2][m] = in && e2 ? __ldcg(v2 + h) : 0.0f;
    q[3][m] = in && e3 ? __ldcg(v3 + h) : 0.0f;
  }
}

// z_b <- H_0 ... H_{nref-1} z_b for the nb vectors in s_z, the whole CTA.  PREFETCH: the next group's rows are on their
// way while this group's sums are added up (needs twice the registers for the rows: short sides up to 2048).
template <int THREADS, int BATCH, int COLS, bool PREFETCH>
__device__ __forceinline__ void vb_apply_reflectors(const float* __restrict__ gV, int64_t ldv, int r, int rp, int nref, int nb,
                                                    float* s_z, float (*s_part)[4 * BATCH + 6], float* s_tot) {
  constexpr int kSums = 4 * BATCH + 6, kWarps = THREADS / 32;
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  float q[4][COLS], qn[4][PREFETCH ? COLS : 1];
  if (PREFETCH && nref > 0) vb_load_rows<THREADS, COLS>(gV, ldv, r, nref - 1, q);
  for (int top = nref - 1; top >= 0; top -= 4) {
    if (!PREFETCH) vb_load_rows<THREADS, COLS>(gV, ldv, r, top, q);
    float acc[kSums];
#pragma unroll
    for (int x = 0; x < kSums; ++x) acc[x] = 0.0f;
#pragma unroll
    for (int m = 0; m < COLS; ++m) {
      const int h = tid + m * THREADS;
      if (h < r) {
        acc[0] = fmaf(q[1][m], q[0][m], acc[0]); acc[1] = fmaf(q[2][m], q[0][m], acc[1]); acc[2] = fmaf(q[2][m], q[1][m], acc[2]);
        acc[3] = fmaf(q[3][m], q[0][m], acc[3]); acc[4] = fmaf(q[3][m], q[1][m], acc[4]); acc[5] = fmaf(q[3][m], q[2][m], acc[5]);
#pragma unroll
        for (int b = 0; b < BATCH; ++b) {
          if (b < nb) {
            const float zh = s_z[(size_t)b * rp + h];
            acc[6 + 4 * b + 0] = fmaf(q[0][m], zh, acc[6 + 4 * b + 0]); acc[6 + 4 * b + 1] = fmaf(q[1][m], zh, acc[6 + 4 * b + 1]);
            acc[6 + 4 * b + 2] = fmaf(q[2][m], zh, acc[6 + 4 * b + 2]); acc[6 + 4 * b + 3] = fmaf(q[3][m], zh, acc[6 + 4 * b + 3]);
          }
        }
      }
    }
    if (PREFETCH && top - 4 >= 0) vb_load_rows<THREADS, COLS>(gV, ldv, r, top - 4, reinterpret_cast<float (&)[4][COLS]>(qn));
    const int n_sums = 6 + 4 * nb;
#pragma unroll
    for (int x = 0; x < kSums; ++x) {
      if (x < n_sums) {
        const float t = warp_sum(acc[x]);
        if (lane == 0) s_part[w][x] = t;
      }
    }
    __syncthreads();
    if (tid < n_sums) {
      float t = 0.0f;
#pragma unroll
      for (int ww = 0; ww < kWarps; ++ww) t += s_part[ww][tid];
      s_tot[tid] = t;
    }
    __syncthreads();
    const float g10 = s_tot[0], g20 = s_tot[1], g21 = s_tot[2], g30 = s_tot[3], g31 = s_tot[4], g32 = s_tot[5];
#pragma unroll
    for (int b = 0; b < BATCH; ++b) {
      if (b < nb) {
        const float c0 = 2.0f * s_tot[6 + 4 * b];
        const float c1 = 2.0f * (s_tot[6 + 4 * b + 1] - c0 * g10);
        const float c2 = 2.0f * (s_tot[6 + 4 * b + 2] - c0 * g20 - c1 * g21);
        const float c3 = 2.0f * (s_tot[6 + 4 * b + 3] - c0 * g30 - c1 * g31 - c2 * g32);
#pragma unroll
        for (int m = 0; m < COLS; ++m) {
          const int h = tid + m * THREADS;
          if (h < r) s_z[(size_t)b * rp + h] -= fmaf(c0, q[0][m], fmaf(c1, q[1][m], fmaf(c2, q[2][m], c3 * q[3][m])));
        }
      }
    }
    // (the next group's partial sums go to s_part only after the barrier that follows them in program order for the
    // slowest reader of s_tot: two barriers separate a write from the reads of the group before)
    if (PREFETCH) {
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int m = 0; m < COLS; ++m) q[x][m] = qn[x][PREFETCH ? m : 0];
    }
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
template <int THREADS, int BPT, int ATOMS> constexpr size_t vb_ring_bytes() { return (size_t)kBackStages * (THREADS / ATOMS) * BPT * 8 * sizeof(float); }

template <int THREADS, int BPT, int ATOMS>
__device__ __forceinline__ void vb_chase_back(const float* __restrict__ gV2, const int ns, const int r, float* s_z, const int z_stride,
                                              float4* s_ring, float (*s_edge)[THREADS / 32]) {
  constexpr int kPer = THREADS / ATOMS;                        // threads per vector
  constexpr int kChunks = kPer * BPT * 2;                      // float4 per sweep
  constexpr int kW = 8 * BPT;                                  // entries per thread = sweeps per turn
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32, me = tid % kPer;
  float* const z = s_z + (size_t)(tid / kPer) * z_stride;
  const int sweeps = ((r - 2 + kW - 1) / kW) * kW;             // the first ones of a partial turn act on nothing
  auto place = [](int f) -> int {                              // chunk f of a sweep inside its stage (spread over the banks)
    const int th = f / (2 * BPT), c = f % (2 * BPT);
    return th * 2 * BPT + (c ^ (BPT == 1 ? (th >> 2) & 1 : th & (2 * BPT - 1)));
  };
  // this thread's chunks of a sweep: where they go, the last sweep that has them, where they come from (sweep by sweep upwards)
  constexpr int kMine = (kChunks + THREADS - 1) / THREADS;
  uint32_t to[kMine];
  int last[kMine];
  const float* from[kMine];
#pragma unroll
  for (int c = 0; c < kMine; ++c) {
    const int f = tid + c * THREADS, t = f / 2;
    to[c] = (uint32_t)__cvta_generic_to_shared(s_ring + place(f));
    last[c] = f < kChunks ? min(r - 3, r - 3 - 8 * t) : -1;
    from[c] = gV2 + ((int64_t)(sweeps - 1) * ns + t) * 8 + (f & 1) * 4;
  }
  int fill = 0, use = 0;                                       // stages
  auto issue = [&](int j) {                                    // sweep j (none below 0: an empty group keeps the count)
    if (j >= 0) {
#pragma unroll
      for (int c = 0; c < kMine; ++c) {
        const bool ok = j <= last[c];
        if (kChunks % THREADS == 0 || tid + c * THREADS < kChunks)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to[c] + fill * (uint32_t)(kChunks * sizeof(float4))), "l"(ok ? from[c] : gV2), "r"(ok ? 16 : 0) : "memory");
        from[c] -= (int64_t)ns * 8;
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    fill = fill == kBackStages - 1 ? 0 : fill + 1;
  };
  float x[kW];
#pragma unroll
  for (int e = 0; e < kW; ++e) { const int at = sweeps + me * kW + e; x[e] = at < r ? z[at] : 0.0f; }
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
        float in = __shfl_up_sync(0xffffffffu, x[(kW - s) % kW], 1);        // what was the last entry of the thread before
        if (lane == 0) in = me == 0 ? (j + 1 < r ? z[j + 1] : 0.0f) : s_edge[(j + 1) & 1][w - 1];
        x[(kW - s) % kW] = in;
      }
      const float4* const st = s_ring + use * kChunks;
      use = use == kBackStages - 1 ? 0 : use + 1;
#pragma unroll
      for (int b = 0; b < BPT; ++b) {
        const float4 u0 = st[place((me * BPT + b) * 2)], u1 = st[place((me * BPT + b) * 2 + 1)];
        const float u[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
        float d0 = 0.0f, d1 = 0.0f;
#pragma unroll
        for (int e = 0; e < 8; e += 2) { d0 = fmaf(u[e], x[(8 * b + e - s + 2 * kW) % kW], d0); d1 = fmaf(u[e + 1], x[(8 * b + e + 1 - s + 2 * kW) % kW], d1); }
        const float d = -2.0f * (d0 + d1);
#pragma unroll
        for (int e = 0; e < 8; ++e) x[(8 * b + e - s + 2 * kW) % kW] = fmaf(d, u[e], x[(8 * b + e - s + 2 * kW) % kW]);
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
  float* s_z = reinterpret_cast<float*>(s_e + rp);             // [rp]
  float4* s_ring = reinterpret_cast<float4*>(s_z + rp);
  __shared__ float s_part[kVcWarps][10];
  __shared__ float s_tot[10];
  __shared__ float s_edge[2][kVcWarps];
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
        for (int i = lane; i < r; i += 32) s_z[i] = (float)(zz[i] * inv);
      }
      __syncthreads();
      vb_chase_back<kVcThreads, 1, 1>(L.bd_V2, (r + kBandWidth - 1) / kBandWidth, r, s_z, rp, s_ring, s_edge);
      vb_apply_reflectors<kVcThreads, 1, kVcMaxRp / kVcThreads, true>(gV, ldv, r, rp, nref, 1, s_z, s_part, s_tot);
      float n2f = 0.0f;
      for (int i = tid; i < r; i += kVcThreads) n2f = fmaf(s_z[i], s_z[i], n2f);
      n2f = warp_sum(n2f);
      __syncthreads();
      if (lane == 0) s_part[w][0] = n2f;
      __syncthreads();
      float tot = 0.0f;
#pragma unroll
      for (int ww = 0; ww < kVcWarps; ++ww) tot += s_part[ww][0];
      const float invf = tot > 0.0f ? rsqrtf(tot) : 0.0f;
      for (int i = tid; i < r; i += kVcThreads) gShort[(int64_t)a * r + i] = s_z[i] * invf;
      __syncthreads();
    }
  }
  vb_orthogonalise_equal(L, k, kVcCtas);
}

__global__ void __launch_bounds__(kVbThreads, 1) sp_eigvec_big_kernel(const SpLayer* __restrict__ layers,
                                                                      const int* __restrict__ big_layers) {
  const SpLayer& L = layers[big_layers[blockIdx.x]];
  if (L.rp <= 1024) return;                                    // smaller layers: sp_eigvec_big_cta_kernel
  extern __shared__ __align__(16) unsigned char vb_smem[];
  const int r = L.r, rp = L.rp;
  double* s_d = reinterpret_cast<double*>(vb_smem);            // [rp]
  double* s_e = s_d + rp;                                      // [rp]
  float* s_z = reinterpret_cast<float*>(s_e + rp);             // [kVbBatch][rp]
  float4* s_ring = reinterpret_cast<float4*>(s_z + (size_t)kVbBatch * rp);
  __shared__ float s_edge[2][kVbWarps];
  __shared__ float s_part[kVbWarps][kVbSums];
  __shared__ float s_tot[kVbSums];
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const int n_ctas = gridDim.y, cy = blockIdx.y;
  const uint32_t k = L.hdr->k;
  const float* const gV = L.td_V; const int64_t ldv = L.td_ldv; const double* const gLam = L.lam64;
  const int* const gPerm = L.perm; const uint32_t* const gIdx = L.idx; float* const gShort = L.shortv;
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
      for (int i = lane; i < r; i += 32) gShort[(int64_t)a * r + i] = (float)(zz[i] * inv);
      __syncwarp();
    }
  }
  __syncthreads();
  // ---- (B) back-transformation, kVbBatch of this CTA's atoms per pass over the reflectors ----
  const uint32_t n_mine = k > (uint32_t)cy ? (k - (uint32_t)cy + (uint32_t)n_ctas - 1u) / (uint32_t)n_ctas : 0u;
  for (uint32_t b0 = 0; b0 < n_mine; b0 += kVbBatch) {
    const int nb = (int)min((uint32_t)kVbBatch, n_mine - b0);
    for (int b = 0; b < nb; ++b) {
      const float* src = gShort + (int64_t)(cy + (b0 + b) * n_ctas) * r;
      for (int i = tid; i < r; i += kVbThreads) s_z[(size_t)b * rp + i] = src[i];
    }
    for (int b = nb; b < kVbBatch; ++b) for (int i = tid; i < r; i += kVbThreads) s_z[(size_t)b * rp + i] = 0.0f;
    __syncthreads();
    // one atom: a run per thread and a turn of eight sweeps; the turn of 32 that four atoms share the reflectors in is more
    // code than the instruction cache holds (one of 4096 entries: 9.0 -> 7.3 ms with the rest of the kernel)
    if (nb == 1) vb_chase_back<kVbThreads, 1, 1>(L.bd_V2, (r + kBandWidth - 1) / kBandWidth, r, s_z, rp, s_ring, s_edge);
    else vb_chase_back<kVbThreads, 4, kVbBatch>(L.bd_V2, (r + kBandWidth - 1) / kBandWidth, r, s_z, rp, s_ring, s_edge);
    if (rp <= 4 * kVbThreads) vb_apply_reflectors<kVbThreads, kVbBatch, 4, true>(gV, ldv, r, rp, nref, nb, s_z, s_part, s_tot);
    else vb_apply_reflectors<kVbThreads, kVbBatch, 8, true>(gV, ldv, r, rp, nref, nb, s_z, s_part, s_tot);
    // normalise and file
    for (int b = 0; b < nb; ++b) {
      float n2f = 0.0f;
      for (int i = tid; i < r; i += kVbThreads) n2f = fmaf(s_z[(size_t)b * rp + i], s_z[(size_t)b * rp + i], n2f);
      n2f = warp_sum(n2f);
      __syncthreads();
      if (lane == 0) s_part[w][0] = n2f;
      __syncthreads();
      float tot = 0.0f;
#pragma unroll
      for (int ww = 0; ww < kVbWarps; ++ww) tot += s_part[ww][0];
      const float invf = tot > 0.0f ? rsqrtf(tot) : 0.0f;
      float* dst = gShort + (int64_t)(cy + (b0 + b) * n_ctas) * r;
      for (int i = tid; i < r; i += kVbThreads) dst[i] = s_z[(size_t)b * rp + i] * invf;
    }
    __syncthreads();
  }
  vb_orthogonalise_equal(L, k, n_ctas);
}

// ---- host side ---------------------------------------------------------------------------------------------------
namespace {
size_t vb_smem_bytes(int rp_max) {
  return (size_t)rp_max * (2 * sizeof(double) + kVbBatch * sizeof(float)) + vb_ring_bytes<kVbThreads, 4, kVbBatch>();
}
size_t vc_smem_bytes(int rp_max) { return (size_t)std::min(rp_max, kVcMaxRp) * (2 * sizeof(double) + sizeof(float)) + vb_ring_bytes<kVcThreads, 1, 1>(); }
}  // namespace

int sp_eigvec_big_slots() { return kVbSlots; }

// 0 if the kernels got their shared memory
int sp_configure_eigvec_big() {
  int bad = cudaFuncSetAttribute(sp_eigvec_big_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vb_smem_bytes(kMaxShort)) != cudaSuccess;
  if (bad) cudaGetLastError();
  return bad;
}

void launch_sp_eigvec_big(const SpLayer* d_layers, const int* d_big, int n_big, int rp_max, cudaStream_t st) {
  if (n_big <= 0) return;
  // layers up to a short side of 1024: a four-warp CTA per kept atom (the other kernel's CTAs leave such layers at once,
  // and the other way round)
  sp_eigvec_big_cta_kernel<<<dim3(n_big, kVcCtas), kVcThreads, vc_smem_bytes(rp_max), st>>>(d_layers, d_big);
  if (rp_max <= kVcMaxRp) return;
  // larger layers: CTAs per layer (1 to 16; the kept atoms are dealt to them), as many as keep the launch within one wave
  static int sms = 0;
  if (sms == 0) { int dev = 0; if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) sms = 1; }
  int per = 1;
  while (per < kVbMaxCtas && n_big * per * 2 <= sms) per *= 2;
  sp_eigvec_big_kernel<<<dim3(n_big, per), kVbThreads, vb_smem_bytes(rp_max), st>>>(d_layers, d_big);
}

}  // namespace atomo
