// Device-side descriptors and kernel launchers shared by the API translation unit.
#pragma once
#include "atomo_common.cuh"

namespace atomo {

// ================================= entry-wise path ===============================================
constexpr int kEwMaxRounds = 64;      // water-filling rounds; Algorithm 1 saturates < ceil(s) atoms,
                                      // a round usually takes many at once

constexpr int kEwBatch = 24;          // vectors per launch (their descriptors travel as a kernel argument)
constexpr int kEwBarrierStride = 32;  // words between the barrier counters of two vectors (a line each: arrivals; two-kernel form: CTAs that are done with them)

struct EwPartial { double sum; float amax; uint32_t cnt; };

struct EwState {
  double T0;        // ||g||_1
  float scale;      // p_i = |g_i| * scale for atoms with |g| <= theta
  float c;          // weight of the kept atoms with p < 1
  float theta, amax;// atoms with |g| > theta have p = 1; max |g|
  uint32_t n_sat, rounds, nonfinite;
  uint32_t list_chunks; // one-kernel form: chunks whose keep decisions were taken on the candidate list (test introspection)
};

struct EwVec {
  const float* g; int64_t n, n_tiles;
  uint8_t* pay; atomo_layer_header* hdr;                       // payload
  uint64_t off_idx, off_val, off_tiles, off_sat;
  uint32_t layer, k_cap, sat_cap;
  int compact, candidates;                                     // payload format; keep a candidate list during the first pass (else read the chunk twice)
  int n_ctas, cta0;                                            // chunks (CTAs) of this vector, its first CTA in the launch
  EwPartial* partials; EwState* state;                         // workspace: [3][n_ctas], one record
  uint64_t* chunk_status;                                      // [chunks] ready flag (bit 63) | saturated << 32 | kept atoms of the chunk
  uint32_t* barrier; uint32_t* ticket;                         // arrivals at the vector's barriers; next chunk (two-kernel form)
  uint32_t* mask_words; float* prob_out; int64_t n_words;      // debug outputs or nullptr / 0
};
struct EwBegin { atomo_payload_header gh; int on; };           // the payload header, written by the call's first launch
template <int N> struct EwBatch {
  EwVec v[N];
  int n, scratch_words;
  double s; PhiloxRoundKeys key; uint32_t kind_step;
  EwBegin begin;
};

struct EwDecode { float* out; int64_t n; int layer; uint32_t tile0; };
template <int N> struct EwDecodeBatch { EwDecode v[N]; int n; const uint8_t* payload; };
struct EwLqPart { double sum, sq, amax; };

int ew_configure();                                            // shared memory opt-in; cudaError_t
int ew_plan(EwVec* v, int n_vecs, bool list);                  // CTAs of the one-kernel form (sets n_ctas, cta0), 0: does not fit one wave
bool ew_list_pays(int64_t n, int64_t n_tiles, int n_ctas, double s);   // whether the candidate list is worth keeping at this budget
template <int N> int launch_ew_encode(EwBatch<N>& B, bool list, cudaStream_t st);       // cudaError_t
int ew_solve_ctas(int64_t n_tiles);                            // two-kernel form: CTAs of the solve, chunks of the sampling
int ew_pack_ctas(int64_t n_tiles);
int launch_ew_solve(EwBatch<1>& B, int solve_ctas, int pack_ctas, cudaStream_t st);     // cudaError_t, both
int launch_ew_sample_pack(EwBatch<1>& B, int pack_ctas, cudaStream_t st);
template <int N> void launch_ew_decode(const EwDecodeBatch<N>& B, uint32_t n_tiles, cudaStream_t st);
template <int N> void launch_ew_decode_average(const EwDecodeBatch<N>& B, uint32_t n_tiles, const uint8_t* const* d_payloads,
                                               int n_payloads, cudaStream_t st);
int ew_tile_elems();
void launch_ew_lq(const float* g, int64_t n, int pass, double q, double inv_amax, EwLqPart* part, uint32_t* ticket,
                  EwLqPart* result, int max_ctas, cudaStream_t st);

// ================================= spectral path =================================================
constexpr int kMaxShort = 4096;       // largest short side (atoms per layer)
constexpr int kBandWidth = 8;         // sub-diagonals between the two stages of the large layers' reduction
// doubles that a sweep of the chase takes in bd_V2: its steps in groups of 32, in a group the steps' entries 0 and 1, then 2 and
// 3, .. (a warp of the back-transformation, a reflector per lane, reads whole lines)
__host__ __device__ inline int64_t sp_chase_row(int r) { return (int64_t)((r + 255) / 256) * 256; }
// kept atoms whose eigenvalues are this close (scaled units: trace 1) get their vectors of T together (sp_close_vectors): eigenvalues come to 4e-13 at
// worst, and a vector of its own to that over the distance
constexpr double kCloseEig = 2.0e-11;
constexpr int kCloseWork = 1 + 3 * 16;   // rows of that kernel's workspace
constexpr int kSmemRowsMaxRp = 4096;  // largest padded short side the shared-memory Jacobi kernel holds

// what the digits of a short-side vector say of its range (integer Gram kernel; q = the entry in units of 2^(E - 30))
struct I8Stat {
  unsigned long long rest;     // what the digit pairs p + q <= 3 lack of the vector's square (signed, in units of 2^16)
  unsigned long long square;   // sum of the squares of the leading digits (units of 2^(E - 6))
  unsigned long long counts;   // entries other than zero << 32 | those of them below 2^(E - 9)
};
// more than a quarter of the entries that are not zero have fewer than 22 bits: the FMA kernel forms this vector's row of A
__device__ __forceinline__ bool i8_coarse(const I8Stat& s) { return 4 * (s.counts & 0xffffffffull) > (s.counts >> 32); }

struct SpLayer {
  const float* G; int rows, cols; int64_t ld;
  int r, L, tall;              // short side, long side, rows > cols
  int rp, B, nb;               // padded short side, Jacobi block rows, number of blocks (even)
  uint32_t layer, k_cap;
  int acc;                     // eigen-solver route: 1 = rows [x | v] of [A | I] (mode 0), 0 = rows of L^T (mode 1)
  int ldx;                     // floats per row of X: 2 rp (acc) or rp
  float* A; int64_t lda;       // scaled Gram matrix, r x r valid (mode 0: the left half of X)
  float* X;                    // rp x ldx working rows of the Jacobi solver
  atomo_layer_header* hdr;     // payload
  uint32_t* idx; float* coef; float* shortv; float* longv;
  float* lam;                  // rp   squared norm per row of X as the cluster eigen-solve left it (scaled units)
  int lam_ready;               // lam was written by the eigen-solve (cluster form): finalize need not re-read X for it
  int* perm;                   // r    rank -> row
  float* sigma; float* prob;   // r    descending (debug buffers or workspace)
  uint32_t* mask_words;        // ceil(r/32)
  float* p_sel;                // k_cap: p of the kept atoms
  float* bp_part;              // [bp_chunks][k_cap][L] row-chunk partial sums of the long vectors
  int bp_tiles, bp_chunks, bp_chunk_rows;
  uint32_t* rot_count;         // [max_sweeps] rotations applied in each sweep
  uint32_t* step_bar;          // arrivals of the layer's CTAs at the step barrier of the persistent eigen-solve
  float* scale;                // 1 float: power-of-two scaling applied to A
  float* chol_dd;              // 32 x 32 + 32 floats: diagonal block of the current Cholesky panel, published by its owner
  float* dbg_short;            // r x r or nullptr
  int tc;                      // kernel of the Gram matrix: 0 FMA, 1 TF32 on tensor cores, 2 8-bit integers on tensor cores
  int gram_split;              // Gram matrix on tensor cores: CTAs per output tile (parts of the K range), 1 = no split
  float* gram_part;            // [tiles][gram_split][128 x 128] partial tiles (column-major) when gram_split > 1
  int fma_split, gram_part_len;   // FMA kernel: parts of the K range, length of a part
  double* gram_sums;           // FMA kernel: [tiles][gram_split][16][threads that hold entries] partial tiles; integer kernel: [tiles][gram_split][128 x 128]
  uint32_t *gram_ticket, *fma_ticket;   // [tiles] parts finished; zeroed per call
  int8_t* i8_dig; int64_t i8_ld;   // integer kernel: [4][r][i8_ld] digits of the short-side vectors
  uint32_t* i8_max;            // r: bits of the vectors' largest magnitudes; zeroed per call
  I8Stat* i8_stat;             // r; zeroed per call
  int refine, refine_tiles;    // singular values from the projection norms; tiles along the long side
  float* row_inv;              // rp: 1 / norm of each short-side vector as stored in X
  float* refine_partials;      // [refine_tiles][rp] partial squared norms
  // tridiagonal route (short side <= 512): T = Q^T A Q, its eigenvalues, vectors of the kept atoms only
  int tri;                     // this layer takes the tridiagonal route: 1 = registers of a cluster (rp <= 512), 2 = two stages, A in global memory
  double* td_d; double* td_e;  // rp each: diagonal and off-diagonal of T
  int td_ldv;                  // floats per row of td_V: r rounded up to a multiple of 4 (16-byte rows)
  float* td_V;                 // r x td_ldv: row k = v_k / ||v_k|| (zero up to index k), fp32 for the back-transformation: H_k = I - 2 u u^T
  double* lam64;               // rp: eigenvalues of T, ascending (scaled units); lam holds the same in fp32
  uint32_t* vec_ticket;        // [2] CTAs of the vector kernel that finished this layer, whether some atoms come from tb_z; zeroed per call
  // tridiagonal route for short sides above 512 (tri = 2): dense -> band -> tridiagonal
  float* bd_UW;                // [rows padded to strips][16] U and W of the panel before
  float* bd_X;                 // [rows padded to strips][8] entries of the next panel
  double* bd_part;             // [parts][rows padded to strips][8] partial products
  double* bd_S;                // [3][128] U^T A U and U^T U of three panels in turn
  double* bd_G;                // [half strips][36] dots of the next panel's columns
  double* bd_band;             // [r][9] the band, by column
  double* bd_T;                // [panels][64] T of the panels: Q1 is the product of I - U T U^T
  double* bd_V2;               // [r][sp_chase_row] reflectors of the chase, by sweep
  uint32_t* bd_bar;            // arrivals at the layer's barriers; zeroed per call
  double* tb_z;                // [k_cap][rp] the kept atoms' eigenvectors of T: those of close eigenvalues, above 1024 rows all
  double* close_work;          // [kCloseWork][rp] for the former: their eigenvalues, an upper triangle per warp
  uint32_t* close_flag;        // [k_cap] which those are (valid where vec_ticket[1] is set)
};

// a layer of a spectral decode: threads per output row, rows per CTA, the layer's first CTA
struct SpDecodeLayer { float* out; int64_t rows, cols; int32_t layer, width, cta_rows; uint32_t cta0; };
constexpr int kSpDecodeBatch = 128;
template <int N> struct SpDecodeBatch { SpDecodeLayer v[N]; int n; };

struct TileRef { int32_t layer, a, b, c; };

// payload header (by value), layer headers from a device template, the call's four flag words
void launch_sp_begin(uint8_t* pay, const atomo_payload_header& gh, const atomo_layer_header* d_tmpl, int n_layers,
                     uint32_t* d_flags, cudaStream_t st);
void launch_sp_init(const SpLayer* d_layers, int n_layers, const TileRef* d_diag_tiles, int n_diag_tiles, cudaStream_t st);
int sp_gram_part(int r, int len);                                // FMA kernel: length of a part of the K range, parts, doubles for their sums
int sp_gram_split(int r, int len);
int64_t sp_gram_sums(int r, int split);
void launch_sp_gram(const SpLayer* d_layers, const TileRef* d_tiles, int n_tiles, int n_parts, cudaStream_t st);
// behind the integer kernel: the tiles of its layers that hold a vector too wide for its digits (d_coarse: whether there are any)
void launch_sp_gram_coarse(const SpLayer* d_layers, int n_layers, const uint32_t* d_coarse, cudaStream_t st);
void launch_sp_scale(const SpLayer* d_layers, int n_layers, int r_max, cudaStream_t st);   // trace, then scaling
void launch_sp_load_svd(const SpLayer* d_layers, int n_layers, const float* const* d_sigma, const float* const* d_vecs,
                        cudaStream_t st);                                       // a decomposition given by the caller
// one Jacobi step (global step index t) for every layer of the batch
void launch_sp_jacobi_step(const SpLayer* d_layers, const TileRef* d_pairs, int n_pairs, int row_floats_max,
                           int t, int max_sweeps, float tol, cudaStream_t st);
// whole eigen-solve of a group of layers in one cooperative launch (block pairs co-resident); returns a cudaError_t
int sp_jacobi_persistent_capacity(int row_floats_max);
int launch_sp_jacobi_persistent(const SpLayer* d_layers, const TileRef* d_pairs, int n_pairs, int row_floats_max,
                                int max_sweeps, float tol, uint32_t* d_state, cudaStream_t st);
// layers of up to 1024 rows: clusters of 8 CTAs; more rows: cooperative launch.  Both return a cudaError_t
// cluster form of the persistent eigen-solve (layers of up to 16 block pairs); one entry per CTA of a cluster
struct ClusterCta { int32_t layer, slot, base_rank, pad; };       // layer < 0: this CTA only keeps the barriers
int sp_jacobi_cluster_ctas();                                     // CTAs per cluster
int sp_jacobi_cluster_max_rp();                                   // largest padded short side it takes
int sp_jacobi_cluster_capacity(int rp_max);                       // co-resident clusters (0: not available here)
int launch_sp_jacobi_cluster(const SpLayer* d_layers, const ClusterCta* d_ctas, int n_clusters, int rp_max, int max_sweeps,
                             float tol, cudaStream_t st);         // returns a cudaError_t
// tridiagonal route (atomo_tridiag.cu)
int sp_tridiag_max_rp();
int sp_tridiag_cluster_ctas();
int sp_tridiag_ctas_of(int rp);                                   // CTAs a layer of padded short side rp takes
int sp_configure_tridiag();                                       // co-resident clusters (0: route not available)
int launch_sp_tridiag(const SpLayer* d_layers, const ClusterCta* d_ctas, int n_clusters, uint32_t* d_timeout, cudaStream_t st);  // cudaError_t
void launch_sp_bisect(const SpLayer* d_layers, int n_layers, int r_max, int64_t n_eigenvalues, cudaStream_t st);
void launch_sp_eigvec(const SpLayer* d_layers, int n_layers, int rp_max, cudaStream_t st);
// tridiagonal route for short sides above 512 (atomo_band.cu, vectors in atomo_tridiag_big.cu)
int sp_band_max_r();
int sp_band_strips(int r);
int sp_band_steps(int r);
int sp_band_form(int r_max, int64_t strips);                      // instance of the band kernel for a batch
int sp_band_parts(int form);                                      // tasks that a strip's columns are split into
int sp_band_capacity(int form, int r_max);                        // co-resident CTAs of the band reduction (0: not available)
int sp_configure_band();                                          // 0 if available
int launch_sp_band(const SpLayer* d_layers, const ClusterCta* d_ctas, int n_ctas, int form, int r_max, uint32_t* d_timeout, cudaStream_t st);  // cudaError_t
int sp_chase_capacity(int ctas);                                  // clusters of that many CTAs side by side (0: not available)
int sp_chase_ctas(int r, int n, int wide_capacity);               // CTAs per layer of the chase, for n layers of its size
int launch_sp_chase(const SpLayer* d_layers, const int* d_list, int n, int ctas, cudaStream_t st);   // cudaError_t
int sp_configure_eigvec_big();                                    // 0 if available
int sp_configure_bisect();                                        // 0 if the eigenvalue kernel got its shared memory
// rps: which padded short sides are among them (bit 0: up to 1024, bit 1: up to 2048, bit 2: above)
void launch_sp_eigvec_big(const SpLayer* d_layers, const int* d_big, int n_big, int rps, double budget, cudaStream_t st);
int launch_sp_cholesky(const SpLayer* d_layers, int n_layers, int rp_max, cudaStream_t st);
int launch_sp_cholesky_big(const SpLayer* d_layers, const TileRef* d_ctas, int n_ctas, int max_panels, cudaStream_t st);
int sp_cholesky_big_rows_per_cta();
int sp_configure_eig();
// convergence bookkeeping after t_done steps were enqueued
void launch_sp_check(const SpLayer* d_layers, int n_layers, int t_done, int max_sweeps, uint32_t* d_all_done,
                     cudaStream_t st);
void launch_sp_refine(const SpLayer* d_layers, int n_layers, const TileRef* d_tiles, int n_tiles, cudaStream_t st);
// timeout_flag (device, may be null): non-zero means a bounded wait of an earlier kernel of the call ran out;
// every layer then reports ATOMO_ERR_TIMEOUT and keeps nothing
void launch_sp_finalize_sample(const SpLayer* d_layers, int n_layers, double s, PhiloxKey key,
                               uint32_t kind_step, int max_sweeps, const uint32_t* timeout_flag, cudaStream_t st);
void launch_sp_backproject(const SpLayer* d_layers, const TileRef* d_tiles, int n_tiles, int r_max, cudaStream_t st);
void launch_sp_finish_atoms(const SpLayer* d_layers, int n_layers, int k_cap_max, cudaStream_t st);
// decode of one payload, or (payload null) the mean of n_payloads of them whose addresses are in device memory
int launch_sp_decode(const uint8_t* payload, const uint8_t* const* d_payloads, int n_payloads, const int64_t* rows, const int64_t* cols,
                     float* const* out, int n_layers, cudaStream_t st);      // launches
int sp_configure();          // opt in to large dynamic shared memory; returns cudaError_t
// tensor-core Gram kernel (atomo_tc.cu)
int sp_tc_configure();       // driver entry point for tensor maps + shared memory opt-in; returns cudaError_t
bool sp_tc_eligible(const float* g, int rows, int cols, int64_t ld);
int sp_tc_make_map(void* out_map, const float* g, int rows, int cols, int64_t ld);   // 0 on success
int sp_tc_map_bytes();
int sp_tc_tile();
void launch_sp_gram_tc(const SpLayer* d_layers, const void* d_maps, const TileRef* d_tiles, int n_tiles, uint32_t* d_err,
                       cudaStream_t st);
// integer Gram kernel (atomo_i8.cu)
int sp_i8_configure();                                           // 0 if the kernel got its shared memory
int64_t sp_i8_pitch(int len);                                    // bytes per vector and digit
int sp_i8_stages(int len);
int sp_i8_min_split(int len);                                    // fewest parts of the K range
int64_t sp_i8_sums(int r, int split);                            // doubles for partial tiles
bool sp_i8_by_rows(int len, bool tall);                           // digits in one pass over G
void sp_i8_prep_tiles(int r, int len, bool tall, int* short_tiles, int* long_tiles);
int sp_i8_make_map(void* out_map, const int8_t* digits, int r, int len, int64_t pitch);   // 0 on success
// d_prep: n_prep tiles, the first n_rows of them of layers by rows
void launch_sp_gram_i8(const SpLayer* d_layers, const void* d_maps, const TileRef* d_prep, int n_rows, int n_prep, const TileRef* d_tiles, int n_tiles,
                       uint32_t* d_err, uint32_t* d_coarse, cudaStream_t st);
int sp_bp_rows_per_tile();
int sp_bp_cols_per_tile();
int sp_bp_chunk_rows();

}  // namespace atomo
