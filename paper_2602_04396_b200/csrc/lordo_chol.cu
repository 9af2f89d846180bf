// Cholesky factor of a Gram matrix and the inverse of its triangular factor, one cluster of CTAs per problem.
//
//   gram = L L^T,  rinv = (L^-1)^T = R^-1 (row-major, zeros below the diagonal)
//
// Both triangles come out of one sweep over 32-column panels k. With Z the stack of the rows of L below the
// panel and of the rows of rinv above it, every 32 x 32 block of the panel's column is
//   M = init - sum_{j<k} Z_j L_kj^T          init = the Gram block (rows of L), 0 (rows of rinv), I (the
//   Z_k = M Lkk^-T                           panel's own rows of rinv)
// so the whole kernel is one kind of product, both factors stored with the summation index contiguous. The
// sums run in fp64 on the tensor cores (mma.sync m8n8k4, measured at 64 FMA a clock and SM, the rate of the
// fp64 pipe), L and rinv are kept in fp32. A row block belongs to CTA (block mod cluster size); the block of
// the diagonal is summed, factored and inverted by every CTA for itself, which leaves one barrier a panel.
// While one warp factors the diagonal block of panel k, the others already sum panel k + 1 over the panels
// before k, so that a panel waits for the newest 32 columns only.
//
// What bounds it: the r columns of the diagonal blocks, 165 to 200 clocks each (some 45 instructions of one warp), and per panel one trip
// to L2 for the newest columns, the small products and the barrier (14 thousand clocks a panel at r = 256, 17 with 270 clocks a
// column); for few CTAs per matrix the fp64 products. r = 512 and 16 matrices, r = 256 and 7, r = 128 and 56, us: one CTA per matrix
// with a thread per row 2200, 580, 197; clusters that summed a whole panel at its turn 654, 131, 62; that sum a panel ahead 312, 77, 46;
// with the factor free of roots, the diagonal block handed to it summed, units by the panels they have, and a unit instead of
// the inverse on the factor's scheduler (products of all four units on three schedulers: 296) 265, 66, 43. Every block's sum as
// quarters of 16 x 16 on four warps was slower (four sums in flight a warp instead of sixteen; 354, 86, 48), and so were units that hand steps
// to one another (registers; 346, 80, 55).
#include "lordo_kernels.h"
#include "lordo_recip.cuh"

namespace lordo {
namespace {

constexpr int kB = 32;                       // panel width
constexpr int kCholWarps = 8;                // 255 registers a thread: with 168 the column chain takes twice as long
constexpr int kUnits = 4;                    // partial sums of 32 x 32 blocks in flight, one per warp
constexpr int kLd = 36;                      // row stride of the partial sums and of the inverse: 8 rows x 4 columns meet no bank twice
constexpr int kPartDoubles = kB * kLd;
constexpr size_t kCholSmem = sizeof(double) * (size_t)((5 + kUnits) * kPartDoubles + 2 * kB * kB + 3 * kB);

__device__ __forceinline__ void dmma(double& c0, double& c1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1},{%2},{%3},{%0,%1};" : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}

// Sums of products of rows: lane l of a warp holds rows l/4 + 8i of both 32-row blocks (rows from r on read as
// zeros). The columns may be dealt to the lanes in any order as long as it is the same on both sides.
// DIAG: both blocks are the same one, so its rows are fetched once and only the 8 x 8 tiles on and above the diagonal are
// multiplied (every CTA of a cluster sums the diagonal block for itself: in the kernel whose factor took roots, r = 512, 16 matrices
// 359 -> 345 us, r = 256, 7 matrices 90 -> 88 us).
// c += X_cols L_cols^T over 8 columns from `col` on.
template <bool DIAG>
__device__ __forceinline__ void block_cols(double (&c)[4][4][2], const float* X, int xr, const float* L, int lr, int r, int col) {
  const int lane = threadIdx.x & 31, row = lane >> 2, kc = col + (lane & 3) * 2;
  float2 a[4], b[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int ra = xr + row + 8 * i, rb = lr + row + 8 * i;
    a[i] = b[i] = make_float2(0.f, 0.f);
    if (ra < r) a[i] = *reinterpret_cast<const float2*>(X + (size_t)ra * r + kc);
    if (DIAG) b[i] = a[i];
    else if (rb < r) b[i] = *reinterpret_cast<const float2*>(L + (size_t)rb * r + kc);
  }
#pragma unroll
  for (int t = 0; t < 2; ++t)
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int n = DIAG ? i : 0; n < 4; ++n) dmma(c[i][n][0], c[i][n][1], (double)(t ? a[i].y : a[i].x), (double)(t ? b[n].y : b[n].x));
}

template <bool DIAG>
__device__ __forceinline__ void fetch16(float4 (&a)[4], float4 (&b)[4], const float* X, int xr, const float* L, int lr, int r, int col) {
  const int lane = threadIdx.x & 31, row = lane >> 2, kc = col + (lane & 3) * 4;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int ra = xr + row + 8 * i, rb = lr + row + 8 * i;
    a[i] = b[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (ra < r) a[i] = *reinterpret_cast<const float4*>(X + (size_t)ra * r + kc);
    if (!DIAG && rb < r) b[i] = *reinterpret_cast<const float4*>(L + (size_t)rb * r + kc);
  }
}
template <bool DIAG>
__device__ __forceinline__ void mma16(double (&c)[4][4][2], const float4 (&a)[4], const float4 (&b)[4]) {
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    double bv[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const float4& v = DIAG ? a[n] : b[n];
      bv[n] = (double)(t == 0 ? v.x : t == 1 ? v.y : t == 2 ? v.z : v.w);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double av = DIAG ? bv[i] : (double)(t == 0 ? a[i].x : t == 1 ? a[i].y : t == 2 ? a[i].z : a[i].w);
#pragma unroll
      for (int n = DIAG ? i : 0; n < 4; ++n) dmma(c[i][n][0], c[i][n][1], av, bv[n]);
    }
  }
}
// c += X_j L_j^T over the 32-column blocks j = j0, j0 + dj, ... < j1, 16 columns on their way while 16 are multiplied.
template <bool DIAG>
__device__ __forceinline__ void block_sum(double (&c)[4][4][2], const float* X, int xr, const float* L, int lr, int r, int j0, int j1, int dj) {
  if (j0 >= j1) return;
  float4 a0[4], b0[4], a1[4], b1[4];
  fetch16<DIAG>(a0, b0, X, xr, L, lr, r, j0 * kB);
#pragma unroll 1
  for (int j = j0; j < j1; j += dj) {
    fetch16<DIAG>(a1, b1, X, xr, L, lr, r, j * kB + 16);
    mma16<DIAG>(c, a0, b0);
    if (j + dj < j1) fetch16<DIAG>(a0, b0, X, xr, L, lr, r, (j + dj) * kB);
    mma16<DIAG>(c, a1, b1);
  }
}

// c += X_cols L_cols^T over the quarters slice, slice + of, ... of the 32 columns from `col` on, all loads before the first product.
__device__ __forceinline__ void newest(double (&c)[4][4][2], const float* X, int xr, const float* L, int lr, int r, int col, int slice, int of) {
  if (of == 1) {
    float4 a0[4], b0[4], a1[4], b1[4];
    fetch16<false>(a0, b0, X, xr, L, lr, r, col);
    fetch16<false>(a1, b1, X, xr, L, lr, r, col + 16);
    mma16<false>(c, a0, b0);
    mma16<false>(c, a1, b1);
  } else if (of == 2) {
    float4 a0[4], b0[4];
    fetch16<false>(a0, b0, X, xr, L, lr, r, col + 16 * slice);
    mma16<false>(c, a0, b0);
  } else {
    for (int h = slice; h < 4; h += of) block_cols<false>(c, X, xr, L, lr, r, col + h * 8);
  }
}

__device__ __forceinline__ void clear(double (&c)[4][4][2]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int n = 0; n < 4; ++n) c[i][n][0] = c[i][n][1] = 0.0;
}

__device__ __forceinline__ void store_part(double* p, const double (&c)[4][4][2]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int n = 0; n < 4; ++n)
      *reinterpret_cast<double2*>(p + (8 * i + (lane >> 2)) * kLd + 8 * n + 2 * (lane & 3)) = make_double2(c[i][n][0], c[i][n][1]);
}

// Which unit sums what. Of the t-th block: its place in the matrix, its first unit and the number of its units. Of unit x: its block (the
// number among the CTA's, -1: none) and its place among the block's units.
struct Plan {
  int block[kUnits], first[kUnits], of[kUnits];
  int tile[kUnits], slice[kUnits];
};

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t x;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(x));
  return x;
}
__device__ __forceinline__ uint32_t cluster_nctarank() {
  uint32_t x;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(x));
  return x;
}

}  // namespace

__global__ void __launch_bounds__(kCholWarps * 32, 1) chol_inverse_kernel(const CholProblem* __restrict__ probs, unsigned* __restrict__ status) {
  dep_begin();
  extern __shared__ __align__(16) double csm[];
  double* dpart = csm;                               // [4] parts of the diagonal block's sum
  double* part = dpart + 4 * kPartDoubles;           // [kUnits] partial sums of the other blocks
  double* Xs = part + kUnits * kPartDoubles;         // [kB][kB] columns of the diagonal block's factor, not divided by their pivots
  double* Ts = Xs + kB * kB;                         // ... and divided
  double* piv = Ts + kB * kB;                        // [kB] pivots
  double* floors = piv + kB;                         // [2][kB] least pivots of this panel and the next
  double* Li = floors + 2 * kB;                      // [kB][kLd] inverse of the diagonal block of L
  __shared__ float wmax[kCholWarps];
  __shared__ Plan plans[3], late[2];                 // of this panel, the next and the one after it; of blocks that find no unit at first, in turn
  __shared__ float ga[2 * kB * kB];                  // the Gram matrix' diagonal blocks of this panel and the next, for warp 0

  // handed round, so that the compiler sees that the lanes of a warp agree on what depends on them
  const uint32_t rank = __shfl_sync(0xffffffffu, cluster_ctarank(), 0), csize = __shfl_sync(0xffffffffu, cluster_nctarank(), 0);
  const CholProblem pb = probs[blockIdx.x / csize];
  const int r = pb.r, nb = (r + kB - 1) / kB;
  const float* A = pb.gram;
  float* L = pb.lwork;   // [r][r], blocks below the diagonal
  float* Z = pb.rinv;    // [r][r], upper triangle
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  constexpr int nt = kCholWarps * 32;

  // zeros below the diagonal of rinv (this CTA's row blocks), largest diagonal element
  for (int b = (int)rank; b < nb; b += (int)csize) {
    const int rows = r - b * kB < kB ? r - b * kB : kB;
    for (int e = tid; e < rows * b * (kB / 4); e += nt) {
      const int rr = e / (b * (kB / 4)), cc = e - rr * (b * (kB / 4));
      const size_t at = (size_t)(b * kB + rr) * r + cc * 4;
      if (!pb.rinv16) *reinterpret_cast<float4*>(Z + at) = make_float4(0.f, 0.f, 0.f, 0.f);
      else
        for (int p = 0; p < 3; ++p) *reinterpret_cast<uint2*>(pb.rinv16 + p * pb.plane + at) = make_uint2(0u, 0u);
    }
  }
  float md = 0.f;
  for (int i = tid; i < r; i += nt) md = fmaxf(md, fabsf(A[(size_t)i * r + i]));
  for (int o = 16; o > 0; o >>= 1) md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, o));
  if (lane == 0) wmax[warp] = md;
  __syncthreads();
  md = wmax[0];
  for (int w = 1; w < kCholWarps; ++w) md = fmaxf(md, wmax[w]);
  // A pivot is the squared distance of column j of the factored matrix from the span of the columns
  // before it. Below kBreakdown times the column's own squared norm that distance is inside the
  // rounding noise of an fp32 Gram matrix: the column is treated as dependent, the flag is raised and
  // the pivot is clamped so that everything stays finite.
  constexpr float kBreakdown = 3e-5f;
  const float abs_floor = md > 0.f ? md * 1e-12f : 1.f;

  // Warp 0 factors the diagonal block, warp 7 inverts it, warps 1 and 2 sum it, the other four are the units that sum the row blocks. The
  // factor shares its scheduler with the last unit, which is idle first.
  const int u = warp == 3 ? 0 : warp == 5 ? 1 : warp == 6 ? 2 : warp == 4 ? 3 : kUnits;
  const int own = (int)rank < nb ? (nb - 1 - (int)rank) / (int)csize + 1 : 0;  // this CTA's row blocks: rank, rank + csize, ...
  const bool ahead = own <= kUnits;  // every block of a panel has a unit of its own, so its sum may begin early
  auto has = [&](int k) { return k % (int)csize == (int)rank; };
  auto tiles = [&](int k) { return own - (has(k) ? 1 : 0); };                  // ... without the block of the diagonal
  auto tile_block = [&](int k, int t) { return (int)rank + (int)csize * ((has(k) && t >= k / (int)csize) ? t + 1 : t); };
  // The panels behind the blocks' sums, dealt out to the units (a block above the diagonal has panels from itself on): every block has
  // a unit, those left over go, one after the other, to the block with the most panels a unit. With as many units for each
  // block one was idle with three blocks, and a block of two panels had as many as one of fourteen. Laid down by a warp, two panels ahead or
  // while it has nothing else to do: by one thread, between two barriers that all wait at, it took a tenth where a matrix has one CTA
  // (r = 192 and 148 matrices 140 us, now 128; r = 256 and 300 543, now 494).
  auto lay_out = [&](Plan& pl, int k, int t0, int cnt) {
    int block[kUnits], n[kUnits], of[kUnits];
#pragma unroll
    for (int t = 0; t < kUnits; ++t) {
      block[t] = t < cnt ? tile_block(k, t0 + t) : 0;
      n[t] = block[t] > k ? k : k - block[t];
      of[t] = t < cnt ? 1 : 0;
    }
#pragma unroll
    for (int left = 1; left < kUnits; ++left) {
      if (cnt == 0 || left > kUnits - cnt) continue;
      int best = 0, bn = n[0], bof = of[0];
#pragma unroll
      for (int t = 1; t < kUnits; ++t)
        if (t < cnt && n[t] * bof > bn * of[t]) { best = t; bn = n[t]; bof = of[t]; }
#pragma unroll
      for (int t = 0; t < kUnits; ++t) of[t] += t == best ? 1 : 0;
    }
    int first = 0, mine = 0, count = 0, tile = -1, slice = 0;
#pragma unroll
    for (int t = 0, at = 0; t < kUnits; at += of[t], ++t) {
      if (lane == t) { first = at; mine = block[t]; count = of[t]; }
      if (lane >= at && lane < at + of[t]) { tile = t; slice = lane - at; }
    }
    if (lane < kUnits) { pl.block[lane] = mine; pl.first[lane] = first; pl.of[lane] = count; pl.tile[lane] = tile; pl.slice[lane] = slice; }
  };
  auto a_diag = [&](int k, int j) {  // element (lane, j) of the Gram matrix' diagonal block; A is symmetric
    const int k0 = k * kB, kw = r - k0 < kB ? r - k0 : kB;
    return lane < kw && j < kw ? A[(size_t)(k0 + j) * r + k0 + lane] : (lane == j ? 1.f : 0.f);
  };

  double c[4][4][2];  // a product warp's sum, begun one panel ahead
  clear(c);
  auto stage_diag = [&](int k) {
    float t[kB];  // all loads before the first store (one after the other they took half a panel's time)
#pragma unroll
    for (int j = 0; j < kB; ++j) t[j] = a_diag(k, j);
#pragma unroll
    for (int j = 0; j < kB; ++j) {
      ga[((k & 1) * kB + j) * kB + lane] = t[j];
      if (lane == j) floors[(k & 1) * kB + j] = k * kB + j < r ? (double)fmaxf(kBreakdown * t[j], abs_floor) : 0.0;
    }
  };
  if (warp == 0) stage_diag(0);
  if (warp > 1 && warp < 4 && warp - 2 < nb) lay_out(plans[warp - 2], warp - 2, 0, min(tiles(warp - 2), kUnits));
  __syncthreads();

#pragma unroll 1
  for (int k = 0; k < nb; ++k) {
    const int k0 = k * kB, kw = r - k0 < kB ? r - k0 : kB;  // this panel's columns
    const bool has_k = has(k);
    const int ntiles = tiles(k), first = ntiles < kUnits ? ntiles : kUnits;

    // ---- the newest 32 columns (or, without a head start, all of them) and the sums to shared memory
    if (u == kUnits) {
      const int w = warp == 7 ? 3 : warp;
      if (k > 0) block_cols<true>(c, L, k0, L, k0, r, k0 - kB + w * 8);
      store_part(dpart + w * kPartDoubles, c);
      clear(c);
      asm volatile("bar.sync 1, 128;" ::: "memory");
#pragma unroll
      for (int j = 0; j < 8; ++j) {  // what is left of the diagonal block, for warp 0: eight columns each
        const double* q = dpart + (w * 8 + j) * kLd + lane;  // symmetric too
        Ts[(w * 8 + j) * kB + lane] =
            (double)ga[((k & 1) * kB + w * 8 + j) * kB + lane] - ((q[0] + q[kPartDoubles]) + (q[2 * kPartDoubles] + q[3 * kPartDoubles]));
      }
      if (warp == 0) asm volatile("bar.sync 10, 128;" ::: "memory");
      else asm volatile("bar.arrive 10, 128;" ::: "memory");
    } else {
      const Plan& pl = plans[k % 3];
      const int t = pl.tile[u];
      if (t >= 0) {
        const int b = pl.block[t], sl = pl.slice[u], of = pl.of[t];
        const float* X = b > k ? L : Z;
        if (!ahead) block_sum<false>(c, X, b * kB, L, k0, r, (b > k ? 0 : b) + sl, k, of);
        else if (k > 0) newest(c, X, b * kB, L, k0, r, k0 - kB, sl, of);
        store_part(part + u * kPartDoubles, c);
        clear(c);
      }
    }

    if (warp == 0) {
      // Factor X D^-1 X^T of the diagonal block: lane i holds row i of what is left of the block, X_j its column j, d_j the pivot. Every lane
      // works out every pivot for itself, from the element b beside the pivot before it and the diagonal element D that were
      // handed round a column earlier: D - b b / d = D - b b r0 (1 + e), see lordo_recip.cuh. Nothing here is scaled by a root: the
      // columns behind X_j need X_j, which is in shared memory before its pivot is known, and X_j / d_j. With the roots on the way a column
      // took 270 clocks, now 165: some 45 instructions of one warp.
      const double* fl = floors + (k & 1) * kB;
      double a[kB], dg = 1.0;
#pragma unroll
      for (int j = 0; j < kB; ++j) {
        a[j] = Ts[j * kB + lane];
        if (lane == j) dg = a[j];
      }
      Xs[lane] = a[0];
      __syncwarp();
      bool broke = false;
      auto pivot = [&](double x, double least) {  // x, or the floor where it is not above it (NaN neither)
        const int h = __double2hiint(x);
        const bool low = !(h > __double2hiint(least) && h < 0x7FF00000);
        broke |= low;
        return low ? least : x;
      };
      double d = pivot(__shfl_sync(0xffffffffu, dg, 0), fl[0]);
      double b = __shfl_sync(0xffffffffu, a[0], 1), D = __shfl_sync(0xffffffffu, dg, 1);
#pragma unroll
      for (int j = 0; j < kB; ++j) {
        double r0, e, dn = 1.0;
        recip_parts(d, r0, e);
        const double t0 = a[j] * r0, t = fma(t0, e, t0);  // X_j / d_j
        if (j + 1 < kB) {
          const double p = (b * b) * r0;
          dn = fma(-p, e, D - p);
          a[j + 1] = fma(-t, b, a[j + 1]);
          dg = fma(-t, a[j], dg);
          Xs[(j + 1) * kB + lane] = a[j + 1];
        }
        if (j + 2 < kB) {
          b = __shfl_sync(0xffffffffu, a[j + 1], j + 2);
          D = __shfl_sync(0xffffffffu, dg, j + 2);
        }
        Ts[j * kB + lane] = t;
        if (lane == 0) piv[j] = d;
        if (j + 1 < kB) d = pivot(dn, fl[j + 1]);
        __syncwarp();
        if (j % 4 == 3) asm volatile("bar.arrive %0, 64;" ::"r"(2 + j / 4) : "memory");  // four more columns for the inverse
#pragma unroll
        for (int j2 = (j + 2) & ~1; j2 < kB; j2 += 2) {
          const double2 v = *reinterpret_cast<const double2*>(Xs + j * kB + j2);
          if (j2 > j + 1) a[j2] = fma(-t, v.x, a[j2]);
          a[j2 + 1] = fma(-t, v.y, a[j2 + 1]);
        }
      }
      if (broke && rank == 0 && lane == 0) atomicOr(status, LORDO_FLAG_QR_BREAKDOWN);
      clear(c);  // not held in registers meanwhile
    } else if (warp < 3) {
      if (warp == 2 && k + 1 < nb) stage_diag(k + 1);
      if (warp == 1 && k + 2 < nb) lay_out(plans[(k + 2) % 3], k + 2, 0, min(tiles(k + 2), kUnits));
      __syncwarp();
      if (k + 1 < nb) block_sum<true>(c, L, k0 + kB, L, k0 + kB, r, warp - 1, k, 2);
    } else if (warp == 7) {
      // inverse of the diagonal block, column `lane`, four columns of the factor behind warp 0; its rows are divided by the pivots' roots
      double x[kB], y = 0.0;
#pragma unroll
      for (int i = 0; i < kB; ++i) x[i] = lane == i ? 1.0 : 0.0;
#pragma unroll
      for (int p = 0; p < kB; ++p) {
        if (p % 4 == 0) {
          asm volatile("bar.sync %0, 64;" ::"r"(2 + p / 4) : "memory");
          y = recip_sqrt(piv[p + (lane & 3)]);
        }
        Li[p * kLd + lane] = x[p] * __shfl_sync(0xffffffffu, y, p & 3);
#pragma unroll
        for (int i = (p + 1) & ~1; i < kB; i += 2) {
          const double2 v = *reinterpret_cast<const double2*>(Ts + p * kB + i);
          if (i > p) x[i] = fma(-v.x, x[p], x[i]);
          x[i + 1] = fma(-v.y, x[p], x[i + 1]);
        }
      }
      clear(c);
    } else if (ahead && k + 1 < nb) {
      const Plan& pl = plans[(k + 1) % 3];
      const int t = pl.tile[u];
      if (t >= 0) {
        const int b = pl.block[t];
        block_sum<false>(c, b > k + 1 ? L : Z, b * kB, L, k0 + kB, r, (b > k + 1 ? 0 : b) + pl.slice[u], k, pl.of[t]);
      }
    } else if (!ahead && u == 0 && ntiles > kUnits) {
      lay_out(late[0], k, kUnits, min(ntiles - kUnits, kUnits));
    }

    // ---- Z_k = M Lkk^-T, eight rows of a block per warp and turn; the panel's own rows of rinv are Lkk^-T itself
    const int lr = lane >> 2, lc = lane & 3;
    auto gram_init = [&](int b, int row, float (&g)[8]) {  // below the diagonal k0 + 32 <= row, so the columns exist
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) g[kk] = b > k && row < r ? A[(size_t)row * r + k0 + kk * 4 + lc] : 0.f;
    };
    auto put = [&](int b, int row, int col, float x, float y) {
      *reinterpret_cast<float2*>((b > k ? L : Z) + (size_t)row * r + k0 + col) = make_float2(x, y);
      if (b <= k && pb.rinv16) {
        __nv_bfloat16* o16 = pb.rinv16 + (size_t)row * r + k0 + col;
#pragma unroll
        for (int p = 0; p < 3; ++p, o16 += pb.plane) {
          const uint32_t w = pack_bf16x2(x, y);
          *reinterpret_cast<uint32_t*>(o16) = w;
          x -= __uint_as_float(w << 16);
          y -= __uint_as_float(w & 0xFFFF0000u);
        }
      }
    };
    // The 32 columns are summed in two halves side by side: a product waits 26 clocks for the one before it in its sum.
    auto finish = [&](const Plan& pl, int t, int r8, const float (&g)[8]) {
      const int b = pl.block[t], of = pl.of[t];
      double z[2][4][2], m[8];
#pragma unroll
      for (int n = 0; n < 8; ++n) z[n >> 2][n & 3][0] = z[n >> 2][n & 3][1] = 0.0;
      const double* q0 = part + pl.first[t] * kPartDoubles + (r8 + lr) * kLd + lc;
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) m[kk] = (double)g[kk];
#pragma unroll
      for (int sl = 0; sl < kUnits; ++sl)
        if (sl < of) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) m[kk] -= q0[(size_t)sl * kPartDoubles + kk * 4];
        }
#pragma unroll
      for (int kk = 0; kk < 8; ++kk)
#pragma unroll
        for (int n = kk / 2; n < 4; ++n) dmma(z[kk & 1][n][0], z[kk & 1][n][1], m[kk], Li[(8 * n + lr) * kLd + kk * 4 + lc]);  // zeros right of its diagonal
      const int row = b * kB + r8 + lr;
      if (row < r) {
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const int col = 8 * n + 2 * lc;
          if (col < kw) put(b, row, col, (float)(z[0][n][0] + z[1][n][0]), (float)(z[0][n][1] + z[1][n][1]));
        }
      }
    };
    float g[2][8];
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (warp + 8 * h < first * 4) {
        const int b = plans[k % 3].block[(warp + 8 * h) >> 2];
        gram_init(b, b * kB + (warp & 3) * 8 + lr, g[h]);
      }
    __syncthreads();  // the inverse of the diagonal block and the sums of the first blocks are there
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (warp + 8 * h < first * 4) finish(plans[k % 3], (warp + 8 * h) >> 2, (warp & 3) * 8, g[h]);
    if (has_k) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = warp * 4 + 2 * h + (lane >> 4), col = 2 * (lane & 15);
        if (row < kw && col < kw) put(k, k0 + row, col, (float)Li[col * kLd + row], (float)Li[(col + 1) * kLd + row]);
      }
    }
    for (int base = kUnits, i = 0; base < ntiles; base += kUnits, i ^= 1) {
      const Plan& pl = late[i];
      const int cnt = min(ntiles - base, kUnits), more = min(ntiles - base - kUnits, kUnits);
      __syncthreads();  // the blocks before are done with their sums
      if (u < kUnits) {
        const int t = pl.tile[u], b = pl.block[t];
        block_sum<false>(c, b > k ? L : Z, b * kB, L, k0, r, (b > k ? 0 : b) + pl.slice[u], k, pl.of[t]);
        store_part(part + u * kPartDoubles, c);
        clear(c);
      } else if (warp == 7 && more > 0) {
        lay_out(late[i ^ 1], k, base + kUnits, more);
      }
      __syncthreads();
      for (int q = warp; q < cnt * 4; q += kCholWarps) {
        const int b = pl.block[q >> 2];
        gram_init(b, b * kB + (q & 3) * 8 + lr, g[0]);
        finish(pl, q >> 2, (q & 3) * 8, g[0]);
      }
    }
    // the panel is in memory for every CTA of the cluster
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

static int g_clusters[9] = {};  // clusters of c CTAs that the device holds at once, set by chol_configure (one device model per process)

static cudaLaunchConfig_t chol_launch(cudaLaunchAttribute* at, int nprobs, int c, cudaStream_t st) {
  cudaLaunchConfig_t lc = {};
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = (unsigned)c; at->val.clusterDim.y = 1; at->val.clusterDim.z = 1;
  lc.gridDim = dim3((unsigned)(nprobs * c), 1, 1); lc.blockDim = dim3(kCholWarps * 32, 1, 1); lc.dynamicSmemBytes = kCholSmem; lc.stream = st;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_dep
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at; lc.numAttrs = 2;
  return lc;
}

void launch_chol_inverse(const CholProblem* probs, int nprobs, int r_max, unsigned* status, cudaStream_t st) {
  const int c = factor_ctas((r_max + kB - 1) / kB, nprobs, g_clusters);
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t lc = chol_launch(at, nprobs, c, st);
  cudaLaunchKernelEx(&lc, chol_inverse_kernel, probs, status);
}

cudaError_t chol_configure() {
  cudaError_t e = cudaFuncSetAttribute(chol_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCholSmem);
  for (int c = 2; c <= 8 && e == cudaSuccess; ++c) {
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t lc = chol_launch(at, 256, c, nullptr);
    lc.numAttrs = 1;  // the cluster size alone
    e = cudaOccupancyMaxActiveClusters(&g_clusters[c], chol_inverse_kernel, &lc);
  }
  return e;
}

}  // namespace lordo
