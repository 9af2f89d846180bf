// Internal interface between the host layer (lordo_api.cu) and the kernel files.
#pragma once
#include "lordo_common.cuh"
#include "lordo_plan.h"

namespace lordo {

// Elements per partial sum of squares: 32768, or less where that leaves less than a wave of blocks (eight fit an SM),
// then about one wave, down to 2048 (256 threads of 8). Smaller blocks cost more in counters and exits than they
// balance (five ragged matrices, 15 million elements: blocks of 2048 29 us, 1038 blocks 13 us), larger ones end apart
// (4096 x 11008, K = 4: blocks of 131072 70 us, of 32768 58 us).
inline long long sq_chunk(long long elements) {
  const long long c = (elements / (8 * kPlannedSms) + 2047) / 2048 * 2048;
  return c < 2048 ? 2048 : c > 32768 ? 32768 : c;
}

// Launch of a kernel that calls dep_begin() in every thread before it touches anything that another kernel writes. Its
// blocks take their places and set themselves up under the end of the kernel before it: 2 to 3 us less per
// launch in a chain of small kernels (256 x 256 step in check mode 34.6 -> 28.2 us, refresh of 7 layers of 768 700 -> 672 us).
template <class... Params, class... Args>
inline cudaError_t launch_dep(void (*kernel)(Params...), dim3 grid, unsigned threads_x, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  lc.gridDim = grid; lc.blockDim = dim3(threads_x, 1, 1); lc.dynamicSmemBytes = smem; lc.stream = st;
  lc.attrs = &at; lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, kernel, Params(args)...);
}

struct RandomKeys {
  unsigned long long key[64];
};

// ---------------------------------------------------------------------------------------------
// Grouped fp32 GEMM with fused operand formation and epilogues (FFMA path).
//   C[M x N] = A[M x Kd] * B[Kd x N]        (+ second accumulator: A' * B2, A' = A or A o A)
// B, B2 are stored row-major [Kd][N]. A is stored [M][Kd] (ATRANS = 0) or [Kd][M] (ATRANS = 1).
// ---------------------------------------------------------------------------------------------
enum OperandKind {
  OP_PLAIN = 0,  // (*s0_ptr) * p0[idx] + p1[idx]        (s0_ptr, p1 optional)
  OP_UHAT = 1,   // inv_bc1 * p0[idx]                      bias-corrected first moment
  OP_VRES = 2    // inv_bc2 * p1[idx] - (inv_bc1 * p0[idx])^2
};

struct Operand {
  const void* p0;
  const void* const* p0_ind;  // if set: p0 = *p0_ind (a per-call pointer table entry)
  long long p0_off;           // element offset added to p0
  const void* p1;
  const float* s0_ptr;
  long long ld;
  int dt0, dt1, kind, pad;
};

enum EpilogueKind { EPI_STORE = 0, EPI_APPLY = 1, EPI_ROTATE = 2 };

struct Epilogue {
  int kind, pad;
  float* C;         // STORE: C[row*ldc + col] = acc (pad != 0: += acc)
  long long ldc;
  // APPLY (Algorithm 1: error-feedback line and the model update), row = weight row, col = column
  void* W;
  void* E;
  const void* const* G_ind;
  long long G_off;
  const float* dcol;
  const float* cptr;
  // ROTATE (Algorithm 1: moment-rotation lines)
  float* u_out;
  float* v_out;
  // STORE and APPLY, a matrix projected from the right: output element (row, col) belongs to memory
  // element col * ldt + row (the product is formed for the transposed problem). STORE: ldt = ldc.
  int trans, pad2;
  long long ldt;
};

// Columns of an output tile of the fp32 products (rows: 64), with one product or two.
__host__ __device__ constexpr int gemm_columns(int dual) { return dual ? 32 : 64; }
struct GemmProblem {
  int M, N, Kd, tiles_n;
  long long tile_start;  // first tile of this problem within its launch
  Operand A, B, B2;
  Epilogue epi;
};

struct GemmScalars {
  float lr, omega, inv_bc1, inv_bc2, bc1, bc2;
  int form, ef, w_dt, e_dt, g_dt, a_square;
};

void launch_gemm(const GemmProblem* probs, int nprobs, long long total_tiles, ProductSplit split, int atrans, int dual, int carry,
                 const GemmScalars& sc, cudaStream_t st);
cudaError_t gemm_configure();

// ---------------------------------------------------------------------------------------------
// Tensor-core path of the inner step (bf16 operands, fp32 accumulation), see lordo_tc.cu.
// One TcProblem per (matrix, worker); a launch covers `strips` 128-column strips in total.
// ---------------------------------------------------------------------------------------------
struct TcProblem {
  long long strip_start;       // first strip of this problem within the launch
  int m, n, r;
  int r_k;                     // r rounded up to 64: k extent of P16, gT16, uT16
  int r_n;                     // r rounded up to 16: rows of PT16
  int m_k;                     // m rounded up to 64: k extent of PT16, rows of P16
  const __nv_bfloat16* PT16;   // [r_n][m_k]  P^T, zero padded
  const __nv_bfloat16* P16;    // [m_k][r_k]  P, zero padded
  // Low-rank gradient and normalised low-rank update U~, transposed, private to the projection and
  // update kernels:
  // [strip][r_k/8][128 columns][8], i.e. the 16-byte pieces of one k-chunk of a strip's columns lie
  // side by side and a warp moves 512 contiguous bytes.
  __nv_bfloat16* gT16;
  __nv_bfloat16* uT16;
  float* u;                    // [r][n] of this worker
  float* v;
  float* dcol;                 // [n]
  void* W;                     // [m][n] of this worker
  void* E;
  const void* const* G_ind;    // entry of the per-call gradient pointer table
  long long G_off;             // element offset of this worker inside it
  const float* cptr;           // clip coefficient
  int mat, replica, pcopy;     // matrix index, worker index, which copy of P (0 for Global)
  int tr;                      // 1: W, G, E are stored transposed with respect to this problem (a matrix projected from the
                               // right): m counts their columns, n their rows
  float* tb;                   // [r][n] time buffer of this worker (+= lr * U~ every step), or null
  // TMA-fed projection: nsplit CTA pairs per 256 columns (2 when 256 < r <= 512: one per half of the rank), and
  // the second half's share of the column scale of the full-rank QHM term
  float* dcol2;                // [n], or null when nsplit == 1
  int nsplit, pad2;
};

// Tensor maps (opaque 128-byte objects encoded on the host) of one matrix for the TMA-fed kernels.
// "sw": 64 x 64 boxes with the 128-byte swizzle (operands of the projection, and the tiles the update
// epilogue reads and writes in place); "st": 64 x 16 boxes with the same swizzle.
struct alignas(128) TmaMatMaps {
  unsigned char e_sw[128], pt[128], p16[128], w_sw[128];
  // a matrix projected from the right: W as 64 x 128 boxes, and stores of 32 rows of a 64-column tile
  unsigned char w_kb[128], e_st32[128], w_st32[128];
  // refresh: E and Delta16 as 64 x 128 swizzled boxes ("kb", rows of S as MMA rows), Delta16 as
  // 64 x 64 swizzled boxes, and the three bf16 right-hand sides [batch][Kd][r]
  unsigned char e_kb[128], d_kb[128], d_sw[128], om16[128], pn16[128], zq16[128];
  unsigned char e_st[128], w_st[128];  // stores of one row group of the update epilogue
  // refresh on tensor cores, all over hi|lo bf16 planes [2 x batch][rows][cols], 64 x 64 swizzled boxes
  // unless noted: the matrix being orthonormalised with m rows and with n rows (also as 64 x 128 boxes,
  // rows as MMA rows), R^-1, P; 64 x 32 boxes of Rot^T and of Rot^T o Rot^T
  unsigned char xm_sw[128], xm_kb[128], xn_sw[128], xn_kb[128], rinv_sw[128], phl_sw[128], rt_32[128], sq_32[128];
  unsigned char s_sw[128], s_kb[128];  // the Local signal c G + E in bf16, [K][m][n], as 64 x 64 and as 64 x 128 boxes
};
struct alignas(128) TmaGradMaps {  // re-encoded whenever the caller's gradient pointer changes
  unsigned char g_sw[128], g_kb[128];
};
// ... with fp32 storage one map per matrix, of boxes of 32 rows x 128 columns as they are stored
__device__ __forceinline__ const unsigned char* grad_map_f32(const TmaGradMaps* maps, int mat) { return maps->g_sw + 128ll * mat; }

struct TcPrep {
  const float* P;              // [m][r]
  __nv_bfloat16* P16;
  __nv_bfloat16* PT16;
  long long m;
  int r, r_k, m_k, pad;
};

cudaError_t tc_configure(int r_n_max);
void launch_prep_projection(const TcPrep* items, const long long* blk_start, int nitems, long long total_blocks, cudaStream_t st);
// G and E in fp32, ranks up to 256 (mixed storage and larger ranks run on the fp32 path).
void launch_project_tc(const TcProblem* probs, int nprobs, long long total_strips, int r_n_max, int steps, int sm_count, const StepScalars& sc,
                       unsigned* status, cudaStream_t st);
// TMA-fed persistent kernels (lordo_tma.cu): all of bf16 storage, the update of fp32 storage.
cudaError_t tma_configure();      // bf16 storage
cudaError_t tma_configure_f32();  // fp32 storage
int project_pairs(int sm_count);  // CTA pairs of the projection that the device holds at once
void launch_project_tma(const TcProblem* probs, const TcSeg* segs, const int* start, int pairs, const TmaMatMaps* maps,
                        const TmaGradMaps* gmaps, const StepScalars& sc, unsigned* status, cudaStream_t st);
// f32: fp32 storage. mode 0: r <= 256, one sweep; modes 1 and 2: the two sweeps for 256 < r <= 512. side 0: every problem is
// stored as it is (tr = 0), 1: every one transposed, 2: some of either. With fp32 storage mode and side are 0.
void launch_apply_tma(const TcProblem* probs, const TcSeg* segs, const int* start, int ctas, const TmaMatMaps* maps, const TmaGradMaps* gmaps,
                      const StepScalars& sc, int f32, int mode, int side, unsigned* status, cudaStream_t st);

void launch_selftest_wait(unsigned* status, cudaStream_t st);

// Diagnostics: MSSV = ||Rot||_F^2 / r of every rotation matrix of the last refresh, and ||E||_F per
// (matrix, worker).
struct DiagProblem {
  const float* rot;  // r x r
  int r, pad;
};
void launch_mssv(const DiagProblem* probs, int nprobs, float* out, cudaStream_t st);
void launch_error_norms(const MatDev* mats, int n_mats, int K, int e_dt, float* out, cudaStream_t st);

// Cholesky factor of a batch of r x r Gram matrices and the inverse of its transpose:
// gram = R^T R (R upper triangular, positive diagonal); rinv = R^-1, row-major, zeros below the
// diagonal. lwork: r*r floats per problem.
struct CholProblem {
  const float* gram;
  float* lwork;
  float* rinv;
  __nv_bfloat16* rinv16;  // R^-1 as three bf16 planes, `plane` elements apart, zeros below the diagonal; or null: then the zeros
  long long plane;        // are written to rinv instead
  int r, pad;
};
void launch_chol_inverse(const CholProblem* probs, int nprobs, int r_max, unsigned* status, cudaStream_t st);
cudaError_t chol_configure();

// Rayleigh-Ritz truncation of an oversampled basis: C = (Q^T S)(Q^T S)^T is w x w symmetric (w = r + p
// <= 600). The kernel diagonalises C with a parallel cyclic Jacobi method (one CTA per problem) and
// writes Mr [w][r] = the first r columns of the projector V_r V_r^T onto the eigenvectors of the r
// largest eigenvalues. C is destroyed; work holds 3 w*w floats.
struct EigProblem {
  float* C;
  float* work;
  float* Mr;
  int w, r;
};
void launch_jacobi_projector(const EigProblem* probs, int nprobs, int w_max, cudaStream_t st);

// Grouped helpers of the refresh: random sketches and device-to-device copies for many matrices
// in one launch each. blk_start is the first 256-thread block of the entry within the launch.
struct RandProblem {
  float* out;            // fp32 output, may be null
  __nv_bfloat16* out16;  // bf16 output, may be null
  long long count, blk_start;
  int purpose, mat, replica, pad;
};
struct CopyProblem {
  void* dst;
  const void* src;
  long long chunks, blk_start;  // 16-byte chunks
};
void launch_fill_random_grouped(const RandProblem* probs, int nprobs, long long total_blocks, unsigned long long seed, long long index,
                                cudaStream_t st);
void launch_copy_grouped(const CopyProblem* probs, int nprobs, long long total_blocks, cudaStream_t st);
// fp32 -> bf16 copies (rounded to nearest) of many buffers, 4096 elements per block.
struct ConvProblem {
  const float* src;
  __nv_bfloat16* dst;
  long long count, blk_start;  // count is a multiple of 8
};
void launch_convert_grouped(const ConvProblem* probs, int nprobs, long long total_blocks, cudaStream_t st);

// "Planes": a value x as bf16 numbers p0, p1 (, p2), each the rounding residual of the ones before it, stored as
// arrays of their own a fixed distance apart. Products of such operands sum pairs of planes: (0,0), (0,1), (1,0) with
// two planes (16 bits of each operand), (1,1), (0,2), (2,0) as well with three (24 bits, the accuracy of an fp32
// product).

// Moments of one worker in a new basis (lordo_rotate.cu), in place. map_rt, map_sq: 64 x 32 swizzled boxes over the two planes of
// Rot^T and of its square, entry b of nb. Items are what a CTA pair works on at a time: two strips of 128
// columns, or one when nsplit = 2 (r > 256).
struct RotateProblem {
  float *u, *v;               // [r][n]
  const void *map_rt, *map_sq;
  long long item_start;       // first item of this problem within the launch
  int n, r, r_n, b, nb, nsplit;
};
cudaError_t rotate_configure();
void launch_rotate(const RotateProblem* probs, int nprobs, long long items, int r_max, int sm_count, const GemmScalars& sc, unsigned* status, cudaStream_t st);

// Gram matrix of a tensor-core QR from its partial products: gram = sum_s S_s + sum_s (T_s + T_s^T), the S
// and T of `ns` ranges of k each, all r x r, S first. With X ~ p0 + p1 + p2, S = p1^T p1 + p0^T p0 and
// T = p0^T p2 + p0^T p1, so that four of the six pairs of planes are multiplied.
struct GramProblem {
  const float* part;
  float* gram;
  long long blk_start;
  int r, ns;
};
void launch_gram_sum(const GramProblem* probs, int nprobs, long long total_blocks, cudaStream_t st);

// Rot = P'^T P from its products over `ns` ranges of k, with the two right-hand sides of the moments' rotation:
// Rot^T and Rot^T o Rot^T as two bf16 planes each, `plane` elements apart.
struct RotProblem {
  const float* part;  // [ns][r][r]
  float* rot;         // [r][r]
  __nv_bfloat16 *rt16, *sq16;
  long long plane, blk_start;
  int r, ns;
};
void launch_rot_sum(const RotProblem* probs, int nprobs, long long total_blocks, cudaStream_t st);

// A new basis in place of the old one, one block per 64 x 64 tile: the columns of Q scaled to unit length (the
// tensor cores' fp32 accumulation truncates and leaves them a few 1e-6 off; the off-diagonal part is at
// fp32 level) become P, its operand copies P16 and PT16 and two planes for Rot; the old P becomes two planes too.
// sq: sums of squares of Q's columns over chunks of kNormRows rows, [chunks][r], from launch_colsq.
constexpr int kNormRows = 256;
struct BasisProblem {
  const float* Q;                    // [m][r]
  double* sq;
  float* P;                          // [m][r]
  __nv_bfloat16 *q16, *p16;          // planes of the new and of the old basis, q_plane and p_plane elements apart
  __nv_bfloat16 *P16, *PT16;         // [m_k][r_k], [r_n][m_k]
  long long q_plane, p_plane;
  long long sq_start, tile_start;    // first block of this problem in the two launches
  long long m;
  int r, r_k, m_k, pad;
};
void launch_colsq(const BasisProblem* probs, int nprobs, long long total_blocks, cudaStream_t st);
void launch_commit_basis(const BasisProblem* probs, int nprobs, long long total_blocks, cudaStream_t st);

// Tensor-core sketch products of the refresh (lordo_tma.cu): C[M x r] (fp32) = S * B with the big
// signal matrix S streamed by TMA as bf16 (optionally formed as c*G + E in shared memory) and
// B [Kd][r] in bf16. a_mn = 1: S is stored [Kd][M] (the product S^T P'); 0: stored [M][Kd].
// Where the result is only an operand of a later product it leaves the kernel as its bf16 planes: an fp32 store, a
// pass to split it and a launch less per product (4096 x 11008, r = 512, K = 16: refresh 14.8 -> 13.6 ms).
struct SkProblem {
  long long tile_start;      // first 256-row tile (128 rows per CTA of a pair) of this problem within the launch
  int M, Kd, r, r_n;
  int a_mn, a_c2, b_c2;      // third TMA coordinate (worker / batch index) of A and of B
  // operands split in bf16 planes: the k loop runs over pairs of planes, pair s being nibble s of pa (plane of A)
  // and of pb (plane of B); a problem covers the steps [j0, j1) of 64 k of the pairs laid end to end
  unsigned pa, pb;
  int j0, j1;
  int a_pl, b_pl;            // third-coordinate distance between the planes of A and of B
  const void* map_a;         // 64 x 64 swizzled boxes (a_mn) or 64 x 128 swizzled boxes
  const void* map_e;         // same shape over E, or null
  const void* map_b;         // 64 x 64 swizzled boxes over B [batch][Kd][r]
  const float* cptr;         // scale of A when map_e is set (clip coefficient), else null
  float* C;                  // fp32 output, or null: then `planes` bf16 planes (1 or 3), C16 [M][r] and `plane` elements on.
  long long ldc;             // C16 may be A's own storage: a tile reads no rows of A but those it writes, and has read them all
  __nv_bfloat16* C16;
  long long plane;
  int planes;
  // with map_e: where c G + E is kept in bf16, as stored [S_rows][S_cols], for the products that follow; or null
  int S_rows, S_cols;
  int tri;                   // B is upper triangular (used above r = 256)
  __nv_bfloat16* S16;
};
// with_e: map_e and cptr are set in every problem of the launch, else in none
void launch_sketch_tma(const SkProblem* probs, int nprobs, long long total_tiles, int grid, int big, int with_e, unsigned* status, cudaStream_t st);

// streaming kernels
// tickets: n_mats * K + K counters, zero before the first launch (every launch leaves them at zero)
void launch_clip(const MatDev* mats, const void* const* G, const long long* chunk_start, int n_mats, int K, int g_dt, long long chunk,
                 double* partial, long long total_chunks, float rho, int scope, float* coef, double* sumsq, unsigned* tickets, unsigned* status,
                 cudaStream_t st);
void launch_fill_float(float* p, long long count, float value, cudaStream_t st);
constexpr int kMomCols = 32;  // columns of the low-rank arrays per block of the moment update
void launch_moments(const MatDev* mats, const long long* tile_start, int n_mats, long long total_tiles, const StepScalars& sc,
                    cudaStream_t st);
void launch_outer_weights(const MatDev* mats, const long long* blk_start, int n_mats, long long total_blocks, int K, int w_dt,
                          int outer, float eta_s, float mu_s, float delta_scale, cudaStream_t st);
void launch_outer_states(const MatDev* mats, const long long* blk_start, int n_mats, long long total_blocks, int K, int which,
                         cudaStream_t st);
void launch_init_weights(const MatDev* mats, const long long* blk_start, int n_mats, long long total_blocks, int K, int w_dt,
                         cudaStream_t st);
void launch_identity_projection(float* P, long long m, int r, int copies, cudaStream_t st);
void launch_fill_random(float* out, long long count, long long batch_stride, const RandomKeys& keys, int batch, cudaStream_t st);

}  // namespace lordo
