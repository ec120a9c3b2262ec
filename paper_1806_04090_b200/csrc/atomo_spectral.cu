// Spectral ATOMO (Section 5 of the paper): atoms are the rank-one terms sigma_i u_i v_i^T of the
// layer gradient seen as a matrix; only the singular values are sparsified.
//
//   sp_gram            A = G G^T (rows <= cols) or G^T G, r x r on the short side, fp32 products
//                      accumulated in short fp32 runs that are flushed into fp64
//   sp_scale           power-of-two normalisation of A by its trace (keeps squared row norms of
//                      small gradients away from the fp32 underflow range)
//   sp_jacobi_step     one step of a one-sided (Hestenes) Jacobi eigen-solver on the rows of
//                      X = [A | I]: row i is (x_i | v_i) with x_i = v_i^T A; orthogonal row
//                      rotations keep that relation and drive the x_i mutually orthogonal, i.e.
//                      x_i -> lambda_i v_i^T.  Blocks of B rows are paired round-robin; a CTA holds
//                      one block pair in shared memory, one warp per rotation.
//   sp_finalize_sample lambda_i = <x_i, v_i>, descending sort, sigma = sqrt(lambda), the
//                      probabilities of Algorithm 1, Philox Bernoulli draws (Eq. 2), ordered
//                      compaction of the kept ranks, short-side vectors of the kept atoms
//   sp_backproject     long-side vector of each kept atom, w_i = G^T u_i (or G v_i)
//   sp_finish_atoms    sigma_i = ||w_i||, coef_i = sigma_i / p_i, w_i normalised
//   sp_decode          G_hat = sum_k coef_k u_k v_k^T, one streaming write pass
#include <algorithm>

#include <type_traits>

#include "atomo_kernels.cuh"

namespace atomo {

// =================================================================================================
// init: V-part of X = identity (X was zero-filled by the caller)
// =================================================================================================
__global__ void sp_init_kernel(const SpLayer* __restrict__ layers) {
  const SpLayer& L = layers[blockIdx.x];
  if (!L.acc) return;
  const int64_t ldx = L.ldx;
  for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < L.rp; i += gridDim.y * blockDim.x)
    L.X[(int64_t)i * ldx + L.rp + i] = 1.0f;
}

void launch_sp_init(const SpLayer* d_layers, int n_layers, const TileRef*, int, cudaStream_t st) {
  sp_init_kernel<<<dim3(n_layers, 4), 256, 0, st>>>(d_layers);
}

// =================================================================================================
// Gram matrix of the short side.  64 x 64 output tile per CTA, 16 x 16 threads, 4 x 4 per thread.
// Short-side vector i is row i of G (rows <= cols) or column i of G (rows > cols).  A layer with a short side of up to 1024 has
// its K range cut into parts (ref.c: which part) of 512, or 2048 above 256, where they have more tiles (a 16384 x 18 layer was
// one CTA walking over 16384 rows: 1340 -> 235 us for a set with some); above there are tiles enough, and the parts' sums would
// cost more than they bring.  A layer gets at most kGramCtas CTAs, four per SM: more fill no idle SM, and the parts' sums, of which
// only the short side's own entries are kept, would outgrow the gradient (64 bytes per element of a 1 x n layer).  The parts
// depend on the layer alone, so that its sums do not change with the batch.
// =================================================================================================
constexpr int kGramTile = 64, kGramK = 16, kGramCtas = 4 * 148;
int sp_gram_part(int r, int len) {
  const int gt = (r + kGramTile - 1) / kGramTile, most = std::max(1, kGramCtas / (gt * (gt + 1) / 2)), part = r <= 256 ? 512 : 2048;
  if (r > 1024) return len;
  const int64_t even = ((int64_t)len + most - 1) / most;
  return (int)std::max<int64_t>(part, (even + 31) / 32 * 32);           // whole fp32 runs of 32 products
}
int sp_gram_split(int r, int len) { return (int)(((int64_t)len + sp_gram_part(r, len) - 1) / sp_gram_part(r, len)); }
int64_t sp_gram_sums(int r, int split) {
  const int64_t gt = (r + kGramTile - 1) / kGramTile, side = std::min((r + 3) / 4, 16);   // threads along a tile's side that hold entries
  return split > 1 ? gt * (gt + 1) / 2 * split * side * side * 16 : 0;
}

// kParts: short sides up to 1024, whose K range may be cut.  Larger layers have an instance of their own: with the code that adds
// parts up in the same kernel, the loop took 6.9 ms on two layers of 4096 x 4096, without it 6.5.
struct GramSmem {
  __align__(16) float As[kGramK][kGramTile + 4], Bs[kGramK][kGramTile + 4];
  bool last;
};
template <bool kParts>
__device__ __forceinline__ void gram_tile(const SpLayer& L, const TileRef& ref, GramSmem& sm) {
  float (&As)[kGramK][kGramTile + 4] = sm.As, (&Bs)[kGramK][kGramTile + 4] = sm.Bs;
  const int i0 = ref.a * kGramTile, j0 = ref.b * kGramTile;
  const bool diag = ref.a == ref.b;
  const float* __restrict__ G = L.G;
  const int64_t ld = L.ld;
  const int r = L.r, len = L.L;
  const bool tall = L.tall;
  const int t = threadIdx.x, ty = t / 16, tx = t % 16;
  float acc[4][4];
  double acc64[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) { acc[a][b] = 0.0f; acc64[a][b] = 0.0; }

  // the K range of a tile is cut into parts where a layer has few tiles
  const int c_lo = kParts ? ref.c * L.gram_part_len : 0, c_hi = kParts ? c_lo + min(len - c_lo, L.gram_part_len) : len;
  // this thread's entries of the next stage, fetched while the stage before is multiplied
  const int row = tall ? t / 16 : t / 4, col = (tall ? t % 16 : t % 4) * 4;
  float fa[4], fb[4];
  auto fetch = [&](int c0) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = tall ? c0 + row : c0 + col + j, ia = tall ? i0 + col + j : i0 + row, ib = tall ? j0 + col + j : j0 + row;
      fa[j] = ia < r && c < c_hi ? __ldg(G + (tall ? (int64_t)c * ld + ia : (int64_t)ia * ld + c)) : 0.0f;
      if (!diag) fb[j] = ib < r && c < c_hi ? __ldg(G + (tall ? (int64_t)c * ld + ib : (int64_t)ib * ld + c)) : 0.0f;
    }
  };
  fetch(c_lo);
  int flush = 0;
  for (int c0 = c_lo; c0 < c_hi; c0 += kGramK) {
    // As[kk][i] = x_{i0+i}[c0+kk], Bs likewise for j0
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (tall) { As[row][col + j] = fa[j]; if (!diag) Bs[row][col + j] = fb[j]; }
      else { As[col + j][row] = fa[j]; if (!diag) Bs[col + j][row] = fb[j]; }
    }
    if (c0 + kGramK < c_hi) fetch(c0 + kGramK);
    __syncthreads();
    const float(*Bp)[kGramTile + 4] = diag ? As : Bs;
#pragma unroll
    for (int kk = 0; kk < kGramK; ++kk) {
      const float4 a = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
      const float4 b = *reinterpret_cast<const float4*>(&Bp[kk][tx * 4]);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(av[p], bv[q], acc[p][q]);
    }
    __syncthreads();
    if (++flush == 2) {   // 32 products per fp32 run, then into fp64
      flush = 0;
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) { acc64[p][q] += (double)acc[p][q]; acc[p][q] = 0.0f; }
    }
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc64[p][q] += (double)acc[p][q];
  if (kParts && L.fma_split > 1) {                            // the last part to finish adds them up, in order
    const int n_split = L.fma_split;
    const int gt = (r + kGramTile - 1) / kGramTile, tile = ref.a * gt - ref.a * (ref.a - 1) / 2 + ref.b - ref.a;
    const int side = min((r + 3) / 4, 16), n_t = side * side; // threads whose 4 x 4 entries hold some of the matrix (short sides below 64: not all)
    const bool holds = ty < side && tx < side;
    double* const parts = L.gram_sums + (int64_t)tile * n_split * (16 * n_t) + ty * side + tx;
    double* const mine = parts + (int64_t)ref.c * (16 * n_t);
    if (holds) {
#pragma unroll
      for (int e = 0; e < 16; ++e) mine[e * n_t] = acc64[e / 4][e % 4];
    }
    __threadfence();
    __syncthreads();
    if (t == 0) sm.last = atomicAdd(L.fma_ticket + tile, 1u) == (uint32_t)(n_split - 1);
    __syncthreads();
    if (!sm.last) return;
    __threadfence();
#pragma unroll
    for (int e = 0; e < 16; ++e) acc64[e / 4][e % 4] = 0.0;
    for (int s = 0; s < n_split && holds; ++s) {
      const double* part = parts + (int64_t)s * (16 * n_t);
#pragma unroll
      for (int e = 0; e < 16; ++e) acc64[e / 4][e % 4] += __ldcg(part + e * n_t);
    }
  }
  const int64_t lda = L.lda;
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + ty * 4 + p, j = j0 + tx * 4 + q;
      if (i < r && j < r) {
        const float v = (float)acc64[p][q];
        L.A[(int64_t)i * lda + j] = v;
        if (!diag) L.A[(int64_t)j * lda + i] = v;
      }
    }
}

template <bool kParts>
__global__ void __launch_bounds__(256) sp_gram_kernel(const SpLayer* __restrict__ layers, const TileRef* __restrict__ tiles) {
  __shared__ GramSmem sm;
  const TileRef ref = tiles[blockIdx.x];
  gram_tile<kParts>(layers[ref.layer], ref, sm);
}

// The integer kernel's layers once more, where a vector's entries span more than its digits hold (i8_coarse): those tiles from fp32 products,
// over what the integer kernel left there.  Every call with such layers launches it, and nearly always its CTAs read one word and leave:
// four per SM deal the tiles of all layers among themselves, so that this costs a launch and no more.
__global__ void __launch_bounds__(256) sp_gram_coarse_kernel(const SpLayer* __restrict__ layers, int n_layers, const uint32_t* __restrict__ coarse) {
  __shared__ GramSmem sm;
  if (*coarse == 0u) return;
  const int t = threadIdx.x, grid = gridDim.x;
  int turn = 0;                                                // the CTA that the next layer's first tile goes to
  for (int l = 0; l < n_layers; ++l) {
    const SpLayer& L = layers[l];
    if (L.tc != 2) continue;
    const int gt = (L.r + kGramTile - 1) / kGramTile, n = gt * (gt + 1) / 2 * L.fma_split;
    for (int q = ((int)blockIdx.x + grid - turn) % grid; q < n; q += grid) {
      TileRef ref{l, 0, q / L.fma_split, q % L.fma_split};
      while (ref.b >= gt - ref.a) { ref.b -= gt - ref.a; ++ref.a; }
      ref.b += ref.a;
      const int i = (t < kGramTile ? ref.a : ref.b) * kGramTile + t % kGramTile;
      if (__syncthreads_or(t < 2 * kGramTile && i < L.r && i8_coarse(L.i8_stat[i]))) gram_tile<true>(L, ref, sm);
      __syncthreads();
    }
    turn = (turn + n) % grid;
  }
}

void launch_sp_gram_coarse(const SpLayer* d_layers, int n_layers, const uint32_t* d_coarse, cudaStream_t st) {
  sp_gram_coarse_kernel<<<kGramCtas, 256, 0, st>>>(d_layers, n_layers, d_coarse);
}

// d_tiles: n_tiles tiles, the last n_parts of them of short sides up to 1024 (or parts of such)
void launch_sp_gram(const SpLayer* d_layers, const TileRef* d_tiles, int n_tiles, int n_parts, cudaStream_t st) {
  if (n_tiles > n_parts) sp_gram_kernel<false><<<n_tiles - n_parts, 256, 0, st>>>(d_layers, d_tiles);
  if (n_parts > 0) sp_gram_kernel<true><<<n_parts, 256, 0, st>>>(d_layers, d_tiles + (n_tiles - n_parts));
}

// =================================================================================================
// scale A by a power of two so that trace(A) is about 1
// =================================================================================================
__global__ void __launch_bounds__(256) sp_trace_kernel(const SpLayer* __restrict__ layers) {
  const SpLayer& L = layers[blockIdx.x];
  const int64_t lda = L.lda;
  __shared__ float s_red[256];
  float tr = 0.0f;
  for (int i = threadIdx.x; i < L.r; i += 256) tr += L.A[(int64_t)i * lda + i];
  s_red[threadIdx.x] = tr;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) { if (threadIdx.x < o) s_red[threadIdx.x] += s_red[threadIdx.x + o]; __syncthreads(); }
  tr = s_red[0];
  float sc = 1.0f;
  if (tr > 0.0f && tr < 3.0e38f) sc = exp2f(-rintf(log2f(tr)));
  if (!(sc > 0.0f) || !(sc < 3.0e38f)) sc = 1.0f;
  if (threadIdx.x == 0) *L.scale = sc;
}

__global__ void __launch_bounds__(256) sp_scale_kernel(const SpLayer* __restrict__ layers) {
  const SpLayer& L = layers[blockIdx.x];
  const int64_t lda = L.lda;
  const float sc = *L.scale;
  if (sc == 1.0f) return;
  for (int i = blockIdx.y; i < L.r; i += gridDim.y)
    for (int j = threadIdx.x; j < L.r; j += 256) L.A[(int64_t)i * lda + j] *= sc;
}

// Start of a spectral encode call: the payload header (passed by value), the layer headers from their template in the
// table cache and the call's flag words -- a kernel instead of host-to-device copies and memsets, which would queue behind
// whatever the application has on the copy engine.
__global__ void __launch_bounds__(256) begin_kernel(uint8_t* __restrict__ pay, atomo_payload_header gh,
                                                    const atomo_layer_header* __restrict__ tmpl, int n_layers,
                                                    uint32_t* __restrict__ flags) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<atomo_payload_header*>(pay) = gh;
  if (blockIdx.x == 0 && threadIdx.x < 4) flags[threadIdx.x] = 0u;
  static_assert(sizeof(atomo_layer_header) % 16 == 0 && sizeof(atomo_payload_header) % 16 == 0, "headers are copied as 16-byte words");
  uint4* dst = reinterpret_cast<uint4*>(pay + sizeof(atomo_payload_header));
  const uint4* src = reinterpret_cast<const uint4*>(tmpl);
  const int n16 = n_layers * (int)(sizeof(atomo_layer_header) / 16);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += gridDim.x * blockDim.x) dst[i] = src[i];
}

void launch_sp_begin(uint8_t* pay, const atomo_payload_header& gh, const atomo_layer_header* d_tmpl, int n_layers,
                     uint32_t* d_flags, cudaStream_t st) {
  const int64_t n16 = n_layers * (int64_t)(sizeof(atomo_layer_header) / 16);
  begin_kernel<<<(int)std::max<int64_t>(1, std::min<int64_t>(32, (n16 + 255) / 256)), 256, 0, st>>>(pay, gh, d_tmpl, n_layers, d_flags);
}

// A decomposition supplied by the caller (test entry point): lambda_i = sigma_i^2 in the eigenvalue slots (scale 1),
// short-side vector i (rank-major input) in row i of X, which the caller zero-filled.
__global__ void __launch_bounds__(256) sp_load_svd_kernel(const SpLayer* __restrict__ layers, const float* const* __restrict__ sigma,
                                                          const float* const* __restrict__ vecs) {
  const SpLayer& L = layers[blockIdx.x];
  const float* sg = sigma[blockIdx.x];
  const float* vv = vecs[blockIdx.x];
  const int r = L.r;
  if (blockIdx.y == 0) {
    for (int i = threadIdx.x; i < r; i += 256) { const float x = sg[i]; L.lam[i] = x * x; }
    if (threadIdx.x == 0) *L.scale = 1.0f;
  }
  for (int i = blockIdx.y; i < r; i += gridDim.y)
    for (int j = threadIdx.x; j < r; j += 256) L.X[(int64_t)i * L.ldx + j] = vv[(int64_t)i * r + j];
}

void launch_sp_load_svd(const SpLayer* d_layers, int n_layers, const float* const* d_sigma, const float* const* d_vecs,
                        cudaStream_t st) {
  sp_load_svd_kernel<<<dim3(n_layers, 32), 256, 0, st>>>(d_layers, d_sigma, d_vecs);
}

void launch_sp_scale(const SpLayer* d_layers, int n_layers, int r_max, cudaStream_t st) {
  sp_trace_kernel<<<n_layers, 256, 0, st>>>(d_layers);
  // (a 4096-row layer on 32 CTAs took 300 us)
  sp_scale_kernel<<<dim3(n_layers, std::min(std::max(r_max / 8, 32), 512)), 256, 0, st>>>(d_layers);
}

// =================================================================================================
// Refinement of the singular values: sigma_i = || G^T u_i || (rows <= cols) or || G v_i || for every
// short-side vector, not only the kept ones.  The Gram route resolves eigenvalues only down to about
// eps * lambda_1, which for a long flat noise tail adds up in the nuclear norm; the norm of the projection
// is second-order accurate in the eigenvector error, so the tail comes out right as long as the
// vectors are orthonormal.  Tile = 64 vectors x 64 positions of the long side; each tile contributes
// one partial sum of squares per vector (summed in a fixed order by sp_finalize_sample).
// =================================================================================================
__global__ void __launch_bounds__(256) sp_rowinv_kernel(const SpLayer* __restrict__ layers) {
  const SpLayer& L = layers[blockIdx.x];
  if (!L.refine) return;
  const int lane = threadIdx.x % 32, w = threadIdx.x / 32;
  const int voff = L.acc ? L.rp : 0;
  for (int i = blockIdx.y * 8 + w; i < L.rp; i += gridDim.y * 8) {
    float n2 = 0.f;
    if (i < L.r) {
      const float* v = L.X + (int64_t)i * L.ldx + voff;
      for (int j = lane; j < L.r; j += 32) n2 = fmaf(v[j], v[j], n2);
    }
    n2 = warp_sum(n2);
    if (lane == 0) L.row_inv[i] = n2 > 0.f ? 1.0f / sqrtf(n2) : 0.f;
  }
}

__global__ void __launch_bounds__(256) sp_refine_kernel(const SpLayer* __restrict__ layers,
                                                        const TileRef* __restrict__ tiles) {
  __shared__ __align__(16) float As[kGramK][kGramTile + 4];   // As[k][a] = u_a[k0 + k]
  __shared__ __align__(16) float Bs[kGramK][kGramTile + 4];   // Bs[k][c] = G(k0 + k, c0 + c) seen from the short side
  __shared__ float s_sq[16][kGramTile];
  const TileRef ref = tiles[blockIdx.x];
  const SpLayer& L = layers[ref.layer];
  const int a0 = ref.a * kGramTile, c0 = ref.b * kGramTile;
  const float* __restrict__ G = L.G;
  const int64_t ld = L.ld, ldx = L.ldx;
  const int r = L.r, len = L.L;
  const int voff = L.acc ? L.rp : 0;
  const int t = threadIdx.x, ty = t / 16, tx = t % 16;
  float acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0f;
  for (int k0 = 0; k0 < r; k0 += kGramK) {
    {
      const int row = t / 4, k4 = (t % 4) * 4;               // vector a0 + row, components k0 + k4 ..
      const int a = a0 + row;
      const float inv = a < r ? L.row_inv[a] : 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = k0 + k4 + j;
        As[k4 + j][row] = (a < r && k < r) ? L.X[(int64_t)a * ldx + voff + k] * inv : 0.0f;
      }
    }
    if (!L.tall) {                                           // G[k][c]: contiguous in c
      const int kk = t / 16, c4 = (t % 16) * 4;
      const int k = k0 + kk;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = c0 + c4 + j;
        Bs[kk][c4 + j] = (k < r && c < len) ? __ldg(G + (int64_t)k * ld + c) : 0.0f;
      }
    } else {                                                 // G[c][k]: contiguous in k
      const int row = t / 4, k4 = (t % 4) * 4;
      const int c = c0 + row;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = k0 + k4 + j;
        Bs[k4 + j][row] = (k < r && c < len) ? __ldg(G + (int64_t)c * ld + k) : 0.0f;
      }
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kGramK; ++kk) {
      const float4 a = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
      const float4 b = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(av[p], bv[q], acc[p][q]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    float sq = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) sq = fmaf(acc[p][q], acc[p][q], sq);
    s_sq[tx][ty * 4 + p] = sq;
  }
  __syncthreads();
  if (t < kGramTile && a0 + t < r) {
    float tot = 0.f;
#pragma unroll
    for (int j = 0; j < 16; ++j) tot += s_sq[j][t];            // fixed order
    L.refine_partials[(int64_t)ref.b * L.rp + a0 + t] = tot;
  }
}

void launch_sp_refine(const SpLayer* d_layers, int n_layers, const TileRef* d_tiles, int n_tiles, cudaStream_t st) {
  if (n_tiles <= 0) return;
  sp_rowinv_kernel<<<dim3(n_layers, 16), 256, 0, st>>>(d_layers);
  sp_refine_kernel<<<n_tiles, 256, 0, st>>>(d_layers, d_tiles);
}

// =================================================================================================
// finalize + probabilities + sampling.  One CTA (512 threads) per layer.
// =================================================================================================
constexpr int kFinThreads = 512;

// x <- (T - mine)^{-1} x for a tridiagonal T, elimination with row interchanges, by one thread; u: [3][rp], the rows of the upper triangle.
// (Eight steps' operands are fetched ahead of the chain of each.)
__device__ __noinline__ void sp_solve_shifted(const double* __restrict__ d, const double* __restrict__ e, const int r, const int rp, const double mine,
                                              double* u, double* x) {
  constexpr double kLeast = 1.0e-14;                           // for pivots below: T is of trace 1, and its eigenvalues come to 4e-13
  constexpr int kStep = 8;
  double* const dd = u; double* const du = u + rp; double* const du2 = du + rp;
  double piv = d[0] - mine, up = r > 1 ? e[0] : 0.0, top = x[0];   // row i of the triangle and of the right side so far
  for (int i0 = 0; i0 + 1 < r; i0 += kStep) {
    double ee[kStep + 1], dn[kStep], xn[kStep];
#pragma unroll
    for (int q = 0; q <= kStep; ++q) ee[q] = i0 + q + 1 < r ? e[i0 + q] : 0.0;
#pragma unroll
    for (int q = 0; q < kStep; ++q) { const bool in = i0 + q + 1 < r; dn[q] = in ? d[i0 + q + 1] - mine : 0.0; xn[q] = in ? x[i0 + q + 1] : 0.0; }
#pragma unroll
    for (int q = 0; q < kStep; ++q) {
      if (i0 + q + 1 < r) {
        const double low = ee[q];
        const bool swap = fabs(low) > fabs(piv) && fabs(low) >= kLeast;   // the lower row has the larger pivot
        if (!swap && !(fabs(piv) >= kLeast)) piv = kLeast;
        const double inv = 1.0 / (swap ? low : piv), f = (swap ? piv : low) * inv;
        dd[i0 + q] = inv;
        du[i0 + q] = swap ? dn[q] : up;
        du2[i0 + q] = swap ? ee[q + 1] : 0.0;
        x[i0 + q] = swap ? xn[q] : top;
        piv = swap ? fma(-f, dn[q], up) : fma(-f, up, dn[q]);
        top = swap ? fma(-f, xn[q], top) : fma(-f, top, xn[q]);
        up = swap ? -f * ee[q + 1] : ee[q + 1];
      }
    }
  }
  if (!(fabs(piv) >= kLeast)) piv = kLeast;
  double x1 = top / piv, x2 = 0.0;
  x[r - 1] = x1;
  for (int i0 = r - 2; i0 >= 0; i0 -= kStep) {
    double a[kStep], b[kStep], c[kStep], y[kStep];
#pragma unroll
    for (int q = 0; q < kStep; ++q) {
      const int i = max(i0 - q, 0);
      a[q] = dd[i]; b[q] = du[i]; c[q] = du2[i]; y[q] = x[i];
    }
#pragma unroll
    for (int q = 0; q < kStep; ++q) {
      if (i0 - q >= 0) {
        const double v = fma(-c[q], x2, fma(-b[q], x1, y[q])) * a[q];
        x[i0 - q] = v; x2 = x1; x1 = v;
      }
    }
  }
}

// Vectors of T for kept atoms whose eigenvalues lie within kCloseEig of another kept atom's (equal to rounding, mostly: layers with equal or
// orthogonal rows, zero rows, ranks below the short side).  Worked out one by one, each from its own eigenvalue, they would be the same vector twice,
// or a vector and noise.  Inverse iteration with reorthogonalisation (the scheme of LAPACK's dstein): three steps from random starts, a warp per
// atom, each followed by Gram-Schmidt against the atoms before it.  The whole CTA.  Other layers pay for a comparison in shared memory.
// Against 64 bits, before | now: 8 x 1011 of +-1 (five equal eigenvalues), largest dot product of two kept vectors 0.58 | 1e-7.
// A whole encode, ms: 512 x 700 of +-1 with 56 atoms kept 7.35 | 4.21 (they need no Gram-Schmidt in the vector kernel), with six 1.12 | 1.37,
// identity of 4096 rows, 13 kept, 34.4 | 33.4.
__device__ __noinline__ void sp_close_vectors(const SpLayer& L, const uint32_t k, double* __restrict__ s_red) {
  constexpr int kWarps = kFinThreads / 32;
  static_assert(kCloseWork == 1 + 3 * kWarps, "room for a triangle per warp");
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32, r = L.r, rp = L.rp;
  double* const lam = L.close_work; double* const u = lam + rp + (int64_t)w * 3 * rp;
  uint32_t* const flag = L.close_flag;
  for (uint32_t a = tid; a < k; a += kFinThreads) lam[a] = L.lam64[L.perm[L.idx[a]]];
  __syncthreads();
  bool any = false;
  for (uint32_t a = tid; a < k; a += kFinThreads) {
    bool close = false;
    for (uint32_t b = 0; b < k; ++b) close |= b != a && fabs(lam[a] - lam[b]) <= kCloseEig;
    flag[a] = close ? 1u : 0u;
    any |= close;
  }
  if (!__syncthreads_or(any)) return;
  if (tid == 0) L.vec_ticket[1] = 1u;
  for (uint32_t a = 0; a < k; ++a) {                           // (uniform)
    if (!flag[a]) continue;
    for (int i = tid; i < r; i += kFinThreads) {
      uint32_t h = (uint32_t)i * 0x9e3779b1u ^ (a + 1u) * 0x85ebca77u;
      h ^= h >> 15; h *= 0x2c1b3c6du; h ^= h >> 12; h *= 0x297a2d39u; h ^= h >> 15;
      L.tb_z[(int64_t)a * rp + i] = (double)(int)h * 0x1p-31;
    }
  }
  __syncthreads();
  auto unit = [&](double* x) {                                 // to unit length (a zero or non-finite vector: to a unit vector)
    double n2 = 0.0;
    for (int i = tid; i < r; i += kFinThreads) n2 = fma(x[i], x[i], n2);
    n2 = warp_sum(n2);
    if (lane == 0) s_red[w] = n2;
    __syncthreads();
    n2 = 0.0;
    for (int q = 0; q < kWarps; ++q) n2 += s_red[q];
    const bool ok = n2 > 1.0e-280 && n2 < 1.0e300;
    const double inv = ok ? rsqrt(n2) : 0.0;
    for (int i = tid; i < r; i += kFinThreads) x[i] = ok ? x[i] * inv : i == 0 ? 1.0 : 0.0;
    __syncthreads();
  };
  for (int it = 0; it < 3; ++it) {
    for (uint32_t a = 0, turn = 0; a < k; ++a) {               // the flagged atoms, dealt to the warps
      if (!flag[a]) continue;
      if ((int)(turn++ % kWarps) == w && lane == 0) sp_solve_shifted(L.td_d, L.td_e, r, rp, lam[a], u, L.tb_z + (int64_t)a * rp);
    }
    __syncthreads();
    for (uint32_t a = 0; a < k; ++a) {
      if (!flag[a]) continue;
      const double mine = lam[a];
      double* const x = L.tb_z + (int64_t)a * rp;
      unit(x);
      for (int round = it < 2 ? 1 : 0; round < 2; ++round) {   // (the last step's vectors twice)
        for (uint32_t b0 = 0; b0 < a; b0 += kFinThreads) {     // dots, a warp each, then all of them out of x
          const uint32_t n = min((uint32_t)kFinThreads, a - b0);
          for (uint32_t q = w; q < n; q += kWarps) {
            double dot = 0.0;
            if (fabs(lam[b0 + q] - mine) <= kCloseEig) {
              const double* const z = L.tb_z + (int64_t)(b0 + q) * rp;
              for (int i = lane; i < r; i += 32) dot = fma(z[i], x[i], dot);
              dot = warp_sum(dot);
            }
            if (lane == 0) s_red[q] = dot;
          }
          __syncthreads();
          for (int i = tid; i < r; i += kFinThreads) {
            double v = x[i];
            for (uint32_t q = 0; q < n; ++q) if (s_red[q] != 0.0) v = fma(-s_red[q], L.tb_z[(int64_t)(b0 + q) * rp + i], v);
            x[i] = v;
          }
          __syncthreads();
        }
      }
      unit(x);
    }
  }
}

__global__ void __launch_bounds__(kFinThreads) sp_finalize_sample_kernel(const SpLayer* __restrict__ layers, double s,
                                                                         PhiloxKey key, uint32_t kind_step,
                                                                         int max_sweeps,
                                                                         const uint32_t* __restrict__ timeout_flag) {
  const SpLayer& L = layers[blockIdx.x];
  __shared__ float s_lam[kMaxShort];        // eigenvalues by row, later sigma by rank
  __shared__ float s_sig[kMaxShort];
  __shared__ double s_red[kFinThreads];
  __shared__ uint32_t s_scan[kFinThreads / 32];
  __shared__ double s_T, s_scur;
  __shared__ uint32_t s_nsat, s_bad, s_k;
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const int r = L.r, rp = L.rp;
  const int64_t ldx = L.ldx;
  const int voff = L.acc ? rp : 0;          // where the eigenvector sits in a row
  const float inv_scale = 1.0f / *L.scale;
  atomo_layer_header* h = L.hdr;
  if (tid == 0) { s_bad = 0; s_k = 0; }
  __syncthreads();

  // eigenvalue of A per row, one warp per row.  mode 0: lambda_i = <x_i, v_i> (Rayleigh quotient at v_i);
  // mode 1: lambda_i = ||x_i||^2 (row i = sigma_i w_i^T).  With refinement: the sum of the tiles' partial
  // squared norms of the projection (already in the units of G).
  if (L.lam_ready && !L.refine && !L.acc) {
    for (int i = tid; i < r; i += kFinThreads) {
      const float lam = L.lam[i] * inv_scale;
      if (!(fabsf(lam) <= 3.0e38f)) atomicOr(&s_bad, 1u);
      s_lam[i] = fmaxf(lam, 0.0f);
    }
  } else
  for (int i = w; i < r; i += kFinThreads / 32) {
    float lam;
    if (L.refine) {
      double d = 0.0;
      for (int tl = lane; tl < L.refine_tiles; tl += 32) d += (double)L.refine_partials[(int64_t)tl * rp + i];
      lam = (float)warp_sum(d);
    } else {
      // rows are zero-padded to rp floats (a multiple of 32): whole float4, several loads in flight
      const float4* x4 = reinterpret_cast<const float4*>(L.X + (int64_t)i * ldx);
      const float4* v4 = reinterpret_cast<const float4*>(L.X + (int64_t)i * ldx + voff);
      float d0 = 0.f, d1 = 0.f;
#pragma unroll 4
      for (int j = lane; j < rp / 4; j += 32) {
        const float4 a = x4[j], b = v4[j];
        d0 = fmaf(a.x, b.x, fmaf(a.y, b.y, d0));
        d1 = fmaf(a.z, b.z, fmaf(a.w, b.w, d1));
      }
      lam = warp_sum(d0 + d1) * inv_scale;
    }
    if (lane == 0) {
      if (!(fabsf(lam) <= 3.0e38f)) atomicOr(&s_bad, 1u);
      s_lam[i] = fmaxf(lam, 0.0f);
    }
  }
  __syncthreads();
  const bool bad = s_bad != 0;
  // rank (descending, ties: lower row first); sigma = sqrt(lambda).  The tridiagonal routes hand over ascending values, but for the
  // last digits: then two binary searches find the rank, else it is counted (r^2 comparisons by one CTA: 0.5 ms at 4096 rows)
  bool falls = false;
  for (int i = tid; i + 1 < r; i += kFinThreads) falls |= !(s_lam[i] <= s_lam[i + 1]);
  const bool ascending = !__syncthreads_or(falls);
  for (int i = tid; i < r; i += kFinThreads) {
    const float li = s_lam[i];
    int rank = 0;
    if (ascending) {
      int below = 0, upto = i;                                 // values below li, values up to li: [below, upto)
      for (int n = i; n > 0;) { const int half = n / 2; if (s_lam[below + half] < li) { below += half + 1; n -= half + 1; } else n = half; }
      for (int n = r - i; n > 0;) { const int half = n / 2; if (s_lam[upto + half] <= li) { upto += half + 1; n -= half + 1; } else n = half; }
      rank = r - upto + i - below;
    } else {
      for (int j = 0; j < r; ++j) { const float lj = s_lam[j]; rank += (lj > li) || (lj == li && j < i); }
    }
    s_sig[rank] = bad ? 0.0f : sqrtf(li);
    L.perm[rank] = i;
  }
  __syncthreads();
  // ||sigma||_1 in fp64, fixed tree
  double part = 0.0;
  for (int i = tid; i < r; i += kFinThreads) part += (double)s_sig[i];
  s_red[tid] = part;
  __syncthreads();
  for (int o = kFinThreads / 2; o > 0; o >>= 1) { if (tid < o) s_red[tid] += s_red[tid + o]; __syncthreads(); }
  if (tid == 0) {
    // Algorithm 1 on the sorted sigma: peel atoms while sigma_i * s > sum_{j >= i} sigma_j
    double T = s_red[0], sc = s;
    int i = 0;
    while (i < r && (double)s_sig[i] * sc > T) { T -= (double)s_sig[i]; sc -= 1.0; ++i; }
    if (i == r || !(T > 0.0)) T = 0.0;
    s_T = T; s_scur = sc; s_nsat = (uint32_t)i;
    h->n_sat = (uint32_t)i;
    h->c = (T > 0.0 && sc > 0.0) ? (float)(T / sc) : 0.0f;
    h->l1 = s_red[0];
  }
  __syncthreads();
  const double T = s_T, scur = s_scur;
  const int n_sat = (int)s_nsat;
  const double scale = (T > 0.0 && scur > 0.0) ? scur / T : 0.0;

  // probabilities, Bernoulli draws, ordered compaction of the kept ranks
  int* const s_kept = reinterpret_cast<int*>(s_lam);         // (the eigenvalues have been ranked; at most r atoms)
  uint32_t carry = 0;
  for (int base = 0; base < r; base += kFinThreads) {
    const int i = base + tid;
    float p = 0.0f;
    bool keep = false;
    if (i < r) {
      const float sg = s_sig[i];
      p = (i < n_sat) ? 1.0f : fminf((float)((double)sg * scale), 1.0f);
      if (!(sg > 0.0f)) p = 0.0f;
      const uint4 wd = atom_block_words((uint64_t)(i >> 2), L.layer, kind_step, key);
      const uint32_t word = (i & 3) == 0 ? wd.x : (i & 3) == 1 ? wd.y : (i & 3) == 2 ? wd.z : wd.w;
      keep = !bad && bernoulli_keep(p, word);
      if (L.sigma) L.sigma[i] = sg;
      if (L.prob) L.prob[i] = p;
    }
    const uint32_t ballot = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) {
      s_scan[w] = __popc(ballot);
      if (L.mask_words && base + w * 32 < r) L.mask_words[(base >> 5) + w] = ballot;
    }
    __syncthreads();
    uint32_t off = carry;
    for (int j = 0; j < w; ++j) off += s_scan[j];
    uint32_t total = 0;
    for (int j = 0; j < kFinThreads / 32; ++j) total += s_scan[j];
    if (keep) {
      const uint32_t pos = off + __popc(ballot & ((1u << lane) - 1u));
      if (pos < L.k_cap) { L.idx[pos] = (uint32_t)i; L.p_sel[pos] = p; s_kept[pos] = i; }
    }
    carry += total;
    __syncthreads();
  }
  if (tid == 0) {
    uint32_t status = ATOMO_OK;
    if (timeout_flag != nullptr && *timeout_flag != 0) status = ATOMO_ERR_TIMEOUT;
    else if (bad) status = ATOMO_ERR_NONFINITE;
    else if (carry > L.k_cap) status = ATOMO_ERR_CAPACITY;
    else if (h->sweeps >= (uint32_t)max_sweeps && L.rot_count[max_sweeps - 1] != 0) status = ATOMO_ERR_NOT_CONVERGED;
    h->status = status;
    // route 0 keeps an orthonormal basis whatever the sweep count, so its unconverged result is still an
    // unbiased estimator; route 1's rows are orthogonal only at convergence, so it keeps nothing
    const uint32_t k = (status == ATOMO_OK || (status == ATOMO_ERR_NOT_CONVERGED && L.acc)) ? carry : 0u;
    h->k = k;
    s_k = k;
  }
  __syncthreads();
  const uint32_t k = s_k;
  if (L.tri) {                             // tridiagonal route: the vectors of the kept atoms come from sp_eigvec_kernel, but for ..
    const float scale = *L.scale;          // .. neighbours within kCloseEig, or within the last digits of fp32
    bool close = false;
    for (uint32_t a = tid; a + 1 < k; a += kFinThreads) {
      const float hi = s_sig[s_kept[a]], lo = s_sig[s_kept[a + 1]];
      close |= (hi - lo) * (hi + lo) * scale <= (float)kCloseEig + 1.0e-6f * hi * hi * scale;
    }
    if (__syncthreads_or(close)) sp_close_vectors(L, k, s_red);
    return;
  }
  // short-side vectors of the kept atoms, normalised: payload shortv[a][0..r)
  for (uint32_t a = w; a < k; a += kFinThreads / 32) {
    const int row = L.perm[L.idx[a]];
    const float* v = L.X + (int64_t)row * ldx + voff;
    float n2 = 0.f;
    for (int j = lane; j < r; j += 32) n2 = fmaf(v[j], v[j], n2);
    n2 = warp_sum(n2);
    const float inv = n2 > 0.f ? 1.0f / sqrtf(n2) : 0.f;
    for (int j = lane; j < r; j += 32) L.shortv[(int64_t)a * r + j] = v[j] * inv;
  }
  // optional: every short-side vector (normalised), rank-major
  if (L.dbg_short) {
    for (int a = w; a < r; a += kFinThreads / 32) {
      const float* v = L.X + (int64_t)L.perm[a] * ldx + voff;
      float n2 = 0.f;
      for (int j = lane; j < r; j += 32) n2 = fmaf(v[j], v[j], n2);
      n2 = warp_sum(n2);
      const float inv = n2 > 0.f ? 1.0f / sqrtf(n2) : 0.f;
      for (int j = lane; j < r; j += 32) L.dbg_short[(int64_t)a * r + j] = v[j] * inv;
    }
  }
}

void launch_sp_finalize_sample(const SpLayer* d_layers, int n_layers, double s, PhiloxKey key, uint32_t kind_step,
                               int max_sweeps, const uint32_t* timeout_flag, cudaStream_t st) {
  sp_finalize_sample_kernel<<<n_layers, kFinThreads, 0, st>>>(d_layers, s, key, kind_step, max_sweeps, timeout_flag);
}

// =================================================================================================
// back-projection: long-side vector of each kept atom.
//   rows <= cols: w_a[c]   = sum_i G[i][c] u_a[i]   tile = 1024 columns x one chunk of rows (a multiple of 64, set
//                                                     per layer), 4 columns per thread, 16 row loads in flight (eight: 96 layers of
//                                                     1024 x 4096 369 us, sixteen 320 us = 5.0 TB/s);
//                                                     chunk partials go to bp_part and are summed in chunk
//                                                     order by sp_finish_atoms
//   rows >  cols: w_a[row] = sum_c G[row][c] v_a[c]   tile = 32 rows, warp per row (one chunk)
// =================================================================================================
constexpr int kBpThreads = 256, kBpAtoms = 8, kBpCols = 1024, kBpRows = 32, kBpChunk = 64;
int sp_bp_cols_per_tile() { return kBpCols; }
int sp_bp_rows_per_tile() { return kBpRows; }
int sp_bp_chunk_rows() { return kBpChunk; }

__global__ void __launch_bounds__(kBpThreads) sp_backproject_kernel(const SpLayer* __restrict__ layers,
                                                                    const TileRef* __restrict__ tiles) {
  __shared__ __align__(16) float s_u[kBpChunk][kBpAtoms];   // wide: the chunk's components of up to 8 short-side vectors
  extern __shared__ __align__(16) float s_v[];              // tall: kBpAtoms x r
  const TileRef ref = tiles[blockIdx.x];
  const SpLayer& L = layers[ref.layer];
  const uint32_t k = L.hdr->k;
  const int r = L.r, len = L.L;
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const float* __restrict__ G = L.G;
  const int64_t ld = L.ld;
  const bool vec = (ld % 4 == 0) && ((reinterpret_cast<uintptr_t>(G) & 15u) == 0);
  for (uint32_t a0 = 0; a0 < k; a0 += kBpAtoms) {
    const int na = min((uint32_t)kBpAtoms, k - a0);
    __syncthreads();
    if (!L.tall) {
      // a thread owns 4 consecutive columns: one 16-byte load per row, 16 rows in flight, 32 FMAs per row
      const int row_lo = ref.b * L.bp_chunk_rows, row_hi = min(r, row_lo + L.bp_chunk_rows);
      const int c = ref.a * kBpCols + 4 * tid;
      float acc[kBpAtoms][4];
#pragma unroll
      for (int a = 0; a < kBpAtoms; ++a) { acc[a][0] = 0.f; acc[a][1] = 0.f; acc[a][2] = 0.f; acc[a][3] = 0.f; }
      for (int i0 = row_lo; i0 < row_hi; i0 += kBpChunk) {
        const int ni = min(kBpChunk, row_hi - i0);
        if (i0 > row_lo) __syncthreads();
        for (int idx = tid; idx < kBpAtoms * kBpChunk; idx += kBpThreads) {
          const int i = idx / kBpAtoms, a = idx % kBpAtoms;
          s_u[i][a] = (a < na && i < ni) ? L.shortv[(int64_t)(a0 + a) * r + i0 + i] : 0.0f;
        }
        __syncthreads();
        if (c < len) {
          const float* gp = G + (int64_t)i0 * ld + c;
          const bool full4 = vec && c + 3 < len;
          for (int i = 0; i < ni; i += 16) {
            float4 g[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              g[u] = make_float4(0.f, 0.f, 0.f, 0.f);
              if (i + u < ni) {
                const float* src = gp + (int64_t)(i + u) * ld;
                if (full4) g[u] = __ldg(reinterpret_cast<const float4*>(src));
                else {
                  g[u].x = __ldg(src);
                  if (c + 1 < len) g[u].y = __ldg(src + 1);
                  if (c + 2 < len) g[u].z = __ldg(src + 2);
                  if (c + 3 < len) g[u].w = __ldg(src + 3);
                }
              }
            }
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              const float4 u0 = *reinterpret_cast<const float4*>(&s_u[i + u][0]);     // rows past ni hold zeros
              const float4 u1 = *reinterpret_cast<const float4*>(&s_u[i + u][4]);
              const float uu[kBpAtoms] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
              for (int a = 0; a < kBpAtoms; ++a) {
                acc[a][0] = fmaf(g[u].x, uu[a], acc[a][0]); acc[a][1] = fmaf(g[u].y, uu[a], acc[a][1]);
                acc[a][2] = fmaf(g[u].z, uu[a], acc[a][2]); acc[a][3] = fmaf(g[u].w, uu[a], acc[a][3]);
              }
            }
          }
        }
      }
      if (c < len) {
#pragma unroll
        for (int a = 0; a < kBpAtoms; ++a)
          if (a < na) {
            float* dst = L.bp_part + ((int64_t)ref.b * L.k_cap + a0 + a) * len + c;
            for (int j = 0; j < 4; ++j) if (c + j < len) dst[j] = acc[a][j];
          }
      }
    } else {
      for (int idx = tid; idx < na * r; idx += kBpThreads) s_v[idx] = L.shortv[(int64_t)a0 * r + idx];
      __syncthreads();
      for (int rr = w; rr < kBpRows; rr += kBpThreads / 32) {
        const int row = ref.a * kBpRows + rr;
        if (row >= len) break;
        float acc[kBpAtoms];
#pragma unroll
        for (int a = 0; a < kBpAtoms; ++a) acc[a] = 0.f;
        for (int c = lane; c < r; c += 32) {
          const float g = __ldg(G + (int64_t)row * ld + c);
#pragma unroll
          for (int a = 0; a < kBpAtoms; ++a) if (a < na) acc[a] = fmaf(g, s_v[a * r + c], acc[a]);
        }
#pragma unroll
        for (int a = 0; a < kBpAtoms; ++a) {
          acc[a] = warp_sum(acc[a]);
          if (a < na && lane == 0) L.bp_part[(int64_t)(a0 + a) * len + row] = acc[a];
        }
      }
    }
  }
}

int sp_configure() {
  const int e = sp_configure_eig();
  if (e != 0) return e;
  return (int)cudaFuncSetAttribute(sp_backproject_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   kBpAtoms * kMaxShort * (int)sizeof(float));
}

void launch_sp_backproject(const SpLayer* d_layers, const TileRef* d_tiles, int n_tiles, int r_max_tall, cudaStream_t st) {
  if (n_tiles > 0)
    sp_backproject_kernel<<<n_tiles, kBpThreads, kBpAtoms * r_max_tall * sizeof(float), st>>>(d_layers, d_tiles);
}

// w_a = sum over row chunks (in chunk order), sigma_a = ||w_a||, coef_a = sigma_a / p_a, long vector = w_a / sigma_a.
// One CTA per (layer, kept-atom slot); slots beyond the layer's k leave at once.
constexpr int kFinishThreads = 1024;
__global__ void __launch_bounds__(kFinishThreads) sp_finish_atoms_kernel(const SpLayer* __restrict__ layers, int k_cap_max) {
  const SpLayer& L = layers[blockIdx.x / k_cap_max];
  const uint32_t a = blockIdx.x % k_cap_max;
  if (a >= L.hdr->k) return;
  const int len = L.L, chunks = L.bp_chunks;
  __shared__ double s_red[kFinishThreads / 32];
  __shared__ float s_sg;
  double part = 0.0;
  float* out = L.longv + (int64_t)a * len;
  const float* in = L.bp_part + (int64_t)a * len;
  const int64_t chunk_stride = (int64_t)L.k_cap * len;
  for (int j = threadIdx.x; j < len; j += kFinishThreads) {
    float wv = 0.f;
#pragma unroll 8
    for (int ch = 0; ch < chunks; ++ch) wv += in[ch * chunk_stride + j];
    out[j] = wv;
    part += (double)wv * (double)wv;
  }
  part = warp_sum(part);
  if (threadIdx.x % 32 == 0) s_red[threadIdx.x / 32] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < kFinishThreads / 32; ++i) t += s_red[i];            // fixed order
    const float sg = (float)sqrt(t);
    L.coef[a] = sg / L.p_sel[a];
    s_sg = sg;
  }
  __syncthreads();
  const float sg = s_sg;
  const float inv = sg >= 1.17549435e-38f ? 1.0f / sg : 0.f;               // (a subnormal norm has no reciprocal: as zero)
  for (int j = threadIdx.x; j < len; j += kFinishThreads) out[j] *= inv;   // each thread rescales what it wrote itself
}

void launch_sp_finish_atoms(const SpLayer* d_layers, int n_layers, int k_cap_max, cudaStream_t st) {
  sp_finish_atoms_kernel<<<n_layers * k_cap_max, kFinishThreads, 0, st>>>(d_layers, k_cap_max);
}

// =================================================================================================
// decode: out[i][c] = sum_a coef_a rowvec_a[i] colvec_a[c] over the kept atoms of one payload, or of all payloads of an
// average: every output element is written once, whatever the number of atoms.
// A thread keeps 16 rows x 4 columns of sums in registers (4 x 4 where a layer has at most 128 columns) and walks over the
// atoms: one 16-byte load of the column vector and four broadcast loads of row entries (times coef, in shared memory) for 64
// multiply-adds.  Where rows are a multiple of 16 bytes a thread owns four neighbouring columns, else columns that lie a
// warp or more apart, so that single stores are still coalesced.  The layers come as a kernel argument, the payloads'
// headers are read by one lane each: three dependent reads of global memory before the first product.
// Bound: the writes of the output (96 layers of 1024 x 4096, one payload: 340 us, 4.7 TB/s), for an average of 24 atoms the multiply-adds as
// well: mean of eight ResNet-18 payloads 126 -> 42 us (before: eight atoms per pass over the output, 208 CTAs, headers
// read one after the other by every thread).
// =================================================================================================
constexpr int kDecThreads = 256, kDecAtoms = 32;               // atoms per round through shared memory
constexpr int kDecCols = 1024, kDecMaxRows = 128;              // columns and at most rows of a CTA

// `single` (one payload) or `list[0 .. n_payloads)`: the kept atoms of all payloads are walked as one sequence, payload after
// payload; `scale` multiplies every term (1, or 1 / n_payloads for the average).
template <int N>
__global__ void __launch_bounds__(kDecThreads, 2) sp_decode_kernel(const __grid_constant__ SpDecodeBatch<N> B, const uint8_t* __restrict__ single,
                                                                   const uint8_t* const* __restrict__ list, const int n_payloads, const float scale) {
  __shared__ __align__(16) float s_rc[kDecAtoms][kDecMaxRows]; // scale * coef_a * rowvec_a[i] of the CTA's rows
  __shared__ const float *s_row[kDecAtoms], *s_col[kDecAtoms];
  __shared__ float s_cf[kDecAtoms];
  __shared__ const float *s_rows[32], *s_cols[32], *s_vals[32];  // the arrays of a round's payloads
  __shared__ int s_first[32], s_k[32];                           // ... and their atoms in the sequence
  __shared__ int s_total;
  int v = 0;
  if (N > 1) {                                                 // the last layer whose first CTA is not above this one
    int hi = B.n;
    while (hi - v > 1) { const int m = (v + hi) / 2; if (B.v[m].cta0 <= blockIdx.x) v = m; else hi = m; }
  }
  const SpDecodeLayer& D = B.v[v];
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const int64_t rows = D.rows, cols = D.cols;
  const bool tall = rows > cols;
  const int64_t r = tall ? cols : rows, len = tall ? rows : cols;
  const int64_t rlen = tall ? len : r, clen = tall ? r : len;  // lengths of the row- and column-indexed vectors
  const uint32_t local = blockIdx.x - D.cta0, n_cb = (uint32_t)((cols + kDecCols - 1) / kDecCols);
  const int width = D.width, my_col = tid & (width - 1), grp = tid / width;   // threads per row, position, row group
  const int64_t i0 = (int64_t)(local / n_cb) * D.cta_rows, c0 = (int64_t)(local % n_cb) * kDecCols;
  const int n_rows = (int)min((int64_t)D.cta_rows, rows - i0);
  const bool quad = (cols % 4 == 0) && ((reinterpret_cast<uintptr_t>(D.out) & 15u) == 0);
  const int64_t c = quad ? c0 + 4 * my_col : c0 + my_col;      // first column of the thread, then every dc-th
  const int dc = quad ? 1 : width;
  const int64_t c_end = min(cols, c0 + 4 * width);
  float* const out = D.out + i0 * cols;
  const int row_bits = __ffs(D.cta_rows) - 1;                  // (a power of two)
  bool staged = false;                                         // all atoms fit shared memory and are there
  // a block of rows: rounds of 32 payloads, their atoms 32 at a time
  auto block = [&](auto rows_tag, const int row_lo) {
    constexpr int kRows = decltype(rows_tag)::value;
    float acc[kRows][4];
#pragma unroll
    for (int i = 0; i < kRows; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
    for (int p0 = 0; p0 < n_payloads; p0 += 32) {
      if (w == 0 && !staged) {
        // a payload normally comes from another rank: its header is checked before anything it points to is read.  The
        // layer headers must exist (layer index below n_layers) and every array must lie inside total_bytes; a header
        // that fails contributes zeros, and the status word is written only where it is known to be a status word
        uint32_t k = 0;
        if (p0 + lane < n_payloads) {
          const uint8_t* payload = list ? list[p0 + lane] : single;
          const atomo_payload_header* gh = reinterpret_cast<const atomo_payload_header*>(payload);
          const bool has_hdr = gh->magic == ATOMO_MAGIC && (uint32_t)D.layer < gh->n_layers &&
                               sizeof(atomo_payload_header) + (uint64_t)gh->n_layers * sizeof(atomo_layer_header) <= gh->total_bytes;
          const atomo_layer_header* h = reinterpret_cast<const atomo_layer_header*>(payload + sizeof(atomo_payload_header)) +
                                        (has_hdr ? D.layer : 0);
          bool ok = has_hdr && gh->kind == ATOMO_KIND_SPECTRAL && h->rows == rows && h->cols == cols && h->k <= h->k_cap;
          if (ok) {
            const uint64_t kc = h->k_cap, tb = gh->total_bytes;
            ok = h->off_idx <= tb && kc * 4 <= tb - h->off_idx && h->off_val <= tb && kc * 4 <= tb - h->off_val &&
                 h->off_short <= tb && kc * (uint64_t)r * 4 <= tb - h->off_short &&
                 h->off_long <= tb && kc * (uint64_t)len * 4 <= tb - h->off_long;
          }
          if (ok) {
            k = h->k;
            s_rows[lane] = reinterpret_cast<const float*>(payload + (tall ? h->off_long : h->off_short));
            s_cols[lane] = reinterpret_cast<const float*>(payload + (tall ? h->off_short : h->off_long));
            s_vals[lane] = reinterpret_cast<const float*>(payload + h->off_val);
          } else if (has_hdr && local == 0 && row_lo == 0) raise_status(const_cast<atomo_layer_header*>(h), ATOMO_ERR_PAYLOAD);
        }
        uint32_t upto = k;                                     // atoms of the payloads up to this lane's
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const uint32_t x = __shfl_up_sync(0xffffffffu, upto, o); if (lane >= o) upto += x; }
        s_first[lane] = (int)(upto - k); s_k[lane] = (int)k;
        if (lane == 31) s_total = (int)upto;
      }
      __syncthreads();
      const int total = s_total;
      for (int a0 = 0; a0 < total; a0 += kDecAtoms) {
        const int na = min(kDecAtoms, total - a0);
        if (!staged) {
          if (w == 0) {
            const int first = s_first[lane], lo = max(first, a0), hi = min(first + s_k[lane], a0 + na);
            for (int t = lo; t < hi; ++t) {
              const int64_t a = t - first;
              s_row[t - a0] = s_rows[lane] + a * rlen + i0;
              s_col[t - a0] = s_cols[lane] + a * clen;
              s_cf[t - a0] = __ldg(s_vals[lane] + a) * scale;
            }
          }
          __syncthreads();
          for (int q = tid; q < na << row_bits; q += kDecThreads) {
            const int a = q >> row_bits, i = q & (D.cta_rows - 1);
            s_rc[a][i] = i < n_rows ? __ldg(s_row[a] + i) * s_cf[a] : 0.0f;
          }
          __syncthreads();
          staged = n_payloads <= 32 && total <= kDecAtoms;
        }
        if (c < cols) {
          auto entries = [&](int a) {
            const float* src = s_col[a] + c;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (quad && (reinterpret_cast<uintptr_t>(src) & 15u) == 0) x = __ldg(reinterpret_cast<const float4*>(src));
            else {
              x.x = __ldg(src);
              if (c + dc < c_end) x.y = __ldg(src + dc);
              if (c + 2 * dc < c_end) x.z = __ldg(src + 2 * dc);
              if (c + 3 * dc < c_end) x.w = __ldg(src + 3 * dc);
            }
            return x;
          };
          const float* rc = &s_rc[0][row_lo + grp * kRows];
          auto add = [&](const float4 x, int a) {
#pragma unroll
            for (int i = 0; i < kRows; i += 4) {
              const float4 q = *reinterpret_cast<const float4*>(rc + (size_t)a * kDecMaxRows + i);
              const float y[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                acc[i + u][0] = fmaf(y[u], x.x, acc[i + u][0]); acc[i + u][1] = fmaf(y[u], x.y, acc[i + u][1]);
                acc[i + u][2] = fmaf(y[u], x.z, acc[i + u][2]); acc[i + u][3] = fmaf(y[u], x.w, acc[i + u][3]);
              }
            }
          };
          int a = 0;
          for (; a + 4 <= na; a += 4) {                        // four loads in flight
            const float4 x0 = entries(a), x1 = entries(a + 1), x2 = entries(a + 2), x3 = entries(a + 3);
            add(x0, a); add(x1, a + 1); add(x2, a + 2); add(x3, a + 3);
          }
          for (; a < na; ++a) add(entries(a), a);
        }
        if (!staged) __syncthreads();
      }
      if (!staged) __syncthreads();
    }
    if (c < cols) {
      float* o = out + (int64_t)(row_lo + grp * kRows) * cols + c;
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        if (row_lo + grp * kRows + i < n_rows) {
          if (quad) *reinterpret_cast<float4*>(o) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
          else {
#pragma unroll
            for (int j = 0; j < 4; ++j) if (c + j * dc < c_end) o[j * dc] = acc[i][j];
          }
        }
        o += cols;
      }
    }
  };
  if (width >= 64) { for (int lo = 0; lo < n_rows; lo += 16 * (kDecThreads / width)) block(std::integral_constant<int, 16>{}, lo); }
  else { for (int lo = 0; lo < n_rows; lo += 4 * (kDecThreads / width)) block(std::integral_constant<int, 4>{}, lo); }
}

// The layers of a decode in launches of up to kSpDecodeBatch of them; returns their number.  The thread layout of a layer
// follows from its columns.  A CTA takes one block of rows; four where the call has CTAs enough to fill the GPU many times
// over (what a CTA reads before its first product then counts less).
int launch_sp_decode(const uint8_t* payload, const uint8_t* const* d_payloads, int n_payloads, const int64_t* rows, const int64_t* cols,
                     float* const* out, int n_layers, cudaStream_t st) {
  auto describe = [&](int l, int blocks, uint32_t cta0) {
    SpDecodeLayer D{out[l], rows[l], cols[l], l, 8, 0, cta0};
    while (4 * D.width < std::min<int64_t>(cols[l], kDecCols)) D.width *= 2;
    D.cta_rows = std::min((D.width >= 64 ? 16 : 4) * (kDecThreads / D.width) * blocks, kDecMaxRows);
    return D;
  };
  auto ctas_of = [](const SpDecodeLayer& D) {
    return (uint64_t)((D.rows + D.cta_rows - 1) / D.cta_rows) * (uint64_t)((D.cols + kDecCols - 1) / kDecCols);
  };
  uint64_t total = 0;
  for (int l = 0; l < n_layers; ++l) total += ctas_of(describe(l, 1, 0));
  const int blocks = total >= 8192 ? 4 : 1;
  const float scale = payload ? 1.0f : 1.0f / (float)n_payloads;
  int n_launch = 0;
  for (int l = 0; l < n_layers; ++n_launch) {
    uint64_t ctas = 0;
    auto run = [&](auto& B, int most) {
      for (B.n = 0; B.n < most && l < n_layers; ++B.n, ++l) {
        const SpDecodeLayer D = describe(l, blocks, (uint32_t)ctas);
        if (B.n > 0 && ctas + ctas_of(D) > 0x7fffffffull) break;
        B.v[B.n] = D;
        ctas += ctas_of(D);
      }
      sp_decode_kernel<<<(unsigned)ctas, kDecThreads, 0, st>>>(B, payload, d_payloads, n_payloads, scale);
    };
    if (n_layers - l == 1) { SpDecodeBatch<1> B{}; run(B, 1); }
    else if (n_layers - l <= 24) { SpDecodeBatch<24> B{}; run(B, 24); }   // (a kilobyte of arguments)
    else { SpDecodeBatch<kSpDecodeBatch> B{}; run(B, kSpDecodeBatch); }
  }
  return n_launch;
}

}  // namespace atomo
