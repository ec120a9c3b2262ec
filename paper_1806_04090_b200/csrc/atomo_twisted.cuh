// Eigenvector of a symmetric tridiagonal matrix for a given eigenvalue: twisted factorisation (device code shared by
// the two vector kernels of the tridiagonal routes; the work vectors may sit in shared or in global memory).
#pragma once
#include "atomo_common.cuh"

namespace atomo {

__device__ __forceinline__ bool finite64(double x) { return fabs(x) <= 1.7e308; }
constexpr double kPivMin = 1.0e-280;

// power of two that brings a pair of running minors to about one
__device__ __forceinline__ double minor_scale(double p, double pm) {
  const int ex = ((__double2hiint(fabs(p) + fabs(pm)) >> 20) & 0x7ff) - 1023;
  return __hiloint2double((1023 - max(min(ex, 1022), -1022)) << 20, 0);
}
// a zero or non-finite pivot is replaced, as a perturbed one would be
__device__ __forceinline__ double safe_pivot(double x) {
  if (!(fabs(x) >= kPivMin)) x = kPivMin;
  return finite64(x) ? x : 1.0e300;
}

// Twisted factorisation of T - lambda I by one warp: forward pivots D+_i = p_i / p_{i-1} from the leading principal minors
// p_i = (d_i - lambda) p_{i-1} - e_{i-1}^2 p_{i-2} (lane 0), backward pivots D- from the trailing ones (lane 1, the same
// instructions on mirrored addresses).  The recurrences carry no division: the minors are stored, the running pair is rescaled by a
// power of two every 8 steps (after it was stored; who divides finds the factor again from the two minors), and the
// quotients are taken by all lanes afterwards.  Twist index at the smallest |gamma_k| = |D+_k + D-_k - (d_k - lambda)|,
// z_k = 1, z_i = -(e_i / D+_i) z_{i+1} above and z_{i+1} = -(e_i / D-_{i+1}) z_i below.  Returns gamma_k / z^T z, the
// Rayleigh-quotient correction of lambda.  na, nb, z: r doubles each, in shared memory.
// Bound: the two serial loops.  Their operands are fetched eight steps at a time, so that a step is what the one warp issues (two
// products, two loads and a store), not a round trip to memory.
static __device__ __noinline__ double twisted_vector(const double* __restrict__ d, const double* __restrict__ e, int r, double lambda,
                                                     double* na, double* nb, double* z, int lane, double* znorm2) {
  constexpr int kStep = 8;
  bool dead = false;
  if (lane < 2) {
    const bool back = lane == 1;
    const int s = back ? -1 : 1;
    const double* pd = d + (back ? r - 1 : 0);
    const double* pe = e + (back ? r - 2 : 0);
    double* n = back ? nb + (r - 1) : na;
    double pm = 1.0, p = *pd - lambda;
    *n = p;
    int t = 1;
#pragma unroll 1
    for (; t + kStep <= r; t += kStep) {
      double dd[kStep], ee[kStep];
#pragma unroll
      for (int u = 0; u < kStep; ++u) { dd[u] = pd[s * (u + 1)]; ee[u] = pe[s * u]; }
      pd += s * kStep; pe += s * kStep;
#pragma unroll
      for (int u = 0; u < kStep; ++u) {
        const double pn = fma(dd[u] - lambda, p, -(ee[u] * ee[u]) * pm);
        n[s * (u + 1)] = pn;
        pm = p; p = pn;
      }
      n += s * kStep;
      const double sc = minor_scale(p, pm);
      p *= sc; pm *= sc;
    }
    for (; t < r; ++t) {
      pd += s; n += s;
      const double pn = fma(*pd - lambda, p, -(*pe * *pe) * pm);
      *n = pn;
      pm = p; p = pn; pe += s;
    }
    dead = p == 0.0;
  }
  // two zeros in a row (lambda a diagonal entry beside a zero off-diagonal one, to the last digit) end a sequence of minors: then
  // the pivots themselves, a division per step
  if (__any_sync(0xffffffffu, dead)) {
    if (lane < 2) {
      const bool back = lane == 1;
      double D = 1.0;
      for (int t = 0; t < r; ++t) {
        const int i = back ? r - 1 - t : t;
        const double ee = t == 0 ? 0.0 : e[back ? i : i - 1];
        D = safe_pivot(d[i] - lambda - ee * ee / D);
        (back ? nb : na)[i] = D;
      }
    }
    __syncwarp();
  } else {
    __syncwarp();
    // pivots in place: na <- D+ (from the last index down: a quotient needs the two minors before it), nb <- D- (upwards)
    const int top = (r - 1) / 32 * 32;
#pragma unroll 2
    for (int i0 = top; i0 >= 0; i0 -= 32) {
      const int i = i0 + lane;
      const double p = na[min(i, r - 1)], q1 = na[min(max(i - 1, 0), r - 1)], q2 = na[min(max(i - 2, 0), r - 1)];
      const double q = i == 0 ? 1.0 : (i - 1) % kStep == 0 && i > 1 ? q1 * minor_scale(q1, q2) : q1;
      __syncwarp();
      if (i < r) na[i] = safe_pivot(p / q);
      __syncwarp();
    }
#pragma unroll 2
    for (int i0 = 0; i0 <= top; i0 += 32) {
      const int i = i0 + lane, t = r - 1 - i;                    // (mirrored index)
      const double p = nb[min(i, r - 1)], q1 = nb[min(i + 1, r - 1)], q2 = nb[min(i + 2, r - 1)];
      const double q = t <= 0 ? 1.0 : (t - 1) % kStep == 0 && t > 1 ? q1 * minor_scale(q1, q2) : q1;
      __syncwarp();
      if (i < r) nb[i] = safe_pivot(p / q);
      __syncwarp();
    }
  }
  // twist index: the smallest |gamma| (lowest index on ties)
  double best = 1.0e300; int bk = 0x7fffffff;
#pragma unroll 4
  for (int i = lane; i < r; i += 32) {
    const double gam = fabs(na[i] + nb[i] - (d[i] - lambda));
    if (gam < best) { best = gam; bk = i; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
    if (ob < best || (ob == best && ok < bk)) { best = ob; bk = ok; }
  }
  if (bk == 0x7fffffff) bk = 0;                               // (non-finite input)
  const double gamma = na[bk] + nb[bk] - (d[bk] - lambda);
  __syncwarp();
  // multipliers: na[i] <- e_i / D+_i above the twist, e_i / D-_{i+1} from there
#pragma unroll 4
  for (int i = lane; i < r - 1; i += 32) na[i] = e[i] / (i < bk ? na[i] : nb[i + 1]);
  if (lane == 0) z[bk] = 1.0;
  __syncwarp();
  if (lane < 2) {                                             // lane 0 upwards from the twist, lane 1 downwards, in step
    const bool down = lane == 1;
    const int s = down ? 1 : -1, n = down ? r - 1 - bk : bk, longer = max(bk, r - 1 - bk);
    const double* pm = na + (down ? bk : bk - 1);
    double* pz = z + (down ? bk + 1 : bk - 1);
    double zz = 1.0;
#pragma unroll 1
    for (int t = 0; t < longer; t += kStep) {
      double m[kStep];
#pragma unroll
      for (int u = 0; u < kStep; ++u) m[u] = t + u < n ? pm[s * u] : 0.0;
#pragma unroll
      for (int u = 0; u < kStep; ++u) {
        zz = -m[u] * zz;
        if (t + u < n) pz[s * u] = zz;
      }
      pm += s * kStep; pz += s * kStep;
    }
  }
  __syncwarp();
  double n2 = 0.0;
#pragma unroll 4
  for (int i = lane; i < r; i += 32) n2 = fma(z[i], z[i], n2);
  n2 = warp_sum(n2);
  *znorm2 = n2;
  return gamma / n2;
}


}  // namespace atomo
