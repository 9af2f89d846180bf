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
// What bounds it: the r columns of the diagonal blocks, 300 clocks each (some 70 instructions of one warp),
// and per panel one trip to L2 for the newest columns, the small products and the barrier; for few CTAs per matrix
// the fp64 products. One CTA per matrix with a thread per row took 2200 us for r = 512 and 16 matrices, 580 us
// for r = 256 and 7, 197 us for r = 128 and 56; clusters that summed a whole panel at its turn 654, 131 and 62 us;
// clusters that sum a panel ahead
// 360, 99 and 56 us (first launch of a stream), with the next diagonal block staged by the inverting warp and the pivots worked
// out by every lane 345, 88 and 53 us. (Scaling the block so that rsqrt.approx needs no care, and handing the factoring
// warp its block summed, both made the column chain slower.)
#include "lordo_kernels.h"
#include "lordo_recip.cuh"

namespace lordo {
namespace {

constexpr int kB = 32;                       // panel width
constexpr int kCholWarps = 8;                // 255 registers a thread: with 168 the column chain takes twice as long
constexpr int kUnits = 4;                    // partial sums of 32 x 32 blocks in flight, one per warp
constexpr int kLd = 36;                      // row stride of the partial sums and of the inverse: 8 rows x 4 columns meet no bank twice
constexpr int kPartDoubles = kB * kLd;
constexpr size_t kCholSmem = sizeof(double) * (size_t)((4 + kUnits) * kPartDoubles + kB * kB + kB + kB * kLd);

__device__ __forceinline__ void dmma(double& c0, double& c1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1},{%2},{%3},{%0,%1};" : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}

// Sums of products of rows: lane l of a warp holds rows l/4 + 8i of both 32-row blocks (rows from r on read as
// zeros). The columns may be dealt to the lanes in any order as long as it is the same on both sides.
// DIAG: both blocks are the same one, so its rows are fetched once and only the 8 x 8 tiles on and above the diagonal are
// multiplied (every CTA of a cluster sums the diagonal block for itself: r = 512, 16 matrices
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
  double* Lc = part + kUnits * kPartDoubles;         // [kB][kB] columns of the diagonal block of L
  double* dinv = Lc + kB * kB;                       // [kB] 1 / its diagonal
  double* Li = dinv + kB;                            // [kB][kLd] inverse of the diagonal block
  __shared__ float wmax[kCholWarps];
  __shared__ float ga[2 * kB * kB];                  // the Gram matrix' diagonal blocks of this panel and the next, for warp 0

  const uint32_t rank = cluster_ctarank(), csize = cluster_nctarank();
  const CholProblem pb = probs[blockIdx.x / csize];
  const int r = pb.r, nb = (r + kB - 1) / kB;
  const float* A = pb.gram;
  float* L = pb.lwork;   // [r][r], blocks below the diagonal
  float* Z = pb.rinv;    // [r][r], upper triangle
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
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

  // Warps 0 and 4 (one scheduler's fp64 pipe, kept free of the products) factor and invert the diagonal block,
  // warps 1 and 2 sum the diagonal block, the other four the row blocks.
  const int u = warp == 3 ? 0 : warp > 4 ? warp - 4 : kUnits;
  const int own = (int)rank < nb ? (nb - 1 - (int)rank) / (int)csize + 1 : 0;  // this CTA's row blocks: rank, rank + csize, ...
  const bool ahead = own <= kUnits;  // every block of a panel has a warp of its own, so its sum may begin early
  auto has = [&](int k) { return k % (int)csize == (int)rank; };
  auto tiles = [&](int k) { return own - (has(k) ? 1 : 0); };                  // ... without the block of the diagonal
  auto tile_block = [&](int k, int t) { return (int)rank + (int)csize * ((has(k) && t >= k / (int)csize) ? t + 1 : t); };
  // slices of the summation index per block, so that a batch of `cnt` blocks has work for every warp
  auto slices = [&](int cnt) { return cnt > 0 && cnt <= kUnits ? kUnits / cnt : 1; };
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
    for (int j = 0; j < kB; ++j) ga[((k & 1) * kB + j) * kB + lane] = t[j];
  };
  if (warp == 0) stage_diag(0);

#pragma unroll 1
  for (int k = 0; k < nb; ++k) {
    const int k0 = k * kB, kw = r - k0 < kB ? r - k0 : kB;  // this panel's columns
    const bool has_k = has(k);
    const int ntiles = tiles(k), first = ntiles < kUnits ? ntiles : kUnits;

    // ---- the newest 32 columns (or, without a head start, all of them) and the sums to shared memory
    if (u == kUnits) {
      const int w = warp == 4 ? 3 : warp;
      if (k > 0) block_cols<true>(c, L, k0, L, k0, r, k0 - kB + w * 8);
      store_part(dpart + w * kPartDoubles, c);
      clear(c);
    } else if (u < first * slices(first)) {
      const int s = slices(first), b = tile_block(k, u / s), sl = u % s;
      const float* X = b > k ? L : Z;
      if (!ahead) block_sum<false>(c, X, b * kB, L, k0, r, (b > k ? 0 : b) + sl, k, s);
      else if (k > 0)
        for (int h = sl; h < 4; h += s) block_cols<false>(c, X, b * kB, L, k0, r, k0 - kB + h * 8);
      store_part(part + u * kPartDoubles, c);
      clear(c);
    }

    if (warp == 0) {
      // Factor of the diagonal block: lane i holds row i of what is left of the block. Every lane works out every pivot d
      // for itself, from the element b beside the pivot before it and the diagonal element D that were handed round a column
      // earlier: D - b b / d = D - b b r0 (1 + e), see lordo_recip.cuh, and the next column's elements likewise; the square
      // root, the column of L and the update of the columns behind the next one fill the gaps. (No chain is what is left: a column is some 70 instructions of one warp, which issues one
      // every four clocks. Handing two elements round and updating the columns behind one column late: slower, registers.)
      asm volatile("bar.sync 1, 128;" ::: "memory");
      const float* gk = ga + (k & 1) * kB * kB;
      double a[kB], dg = 1.0;
#pragma unroll
      for (int j = 0; j < kB; ++j) {
        const double* q = dpart + j * kLd + lane;  // symmetric too
        a[j] = (double)gk[j * kB + lane] - ((q[0] + q[kPartDoubles]) + (q[2 * kPartDoubles] + q[3 * kPartDoubles]));
        if (lane == j) dg = a[j];
      }
      bool broke = false;
      auto pivot = [&](double x, int j) {  // x, or the floor where it is not above it (NaN neither)
        const double fl = j < kw ? (double)fmaxf(kBreakdown * gk[j * kB + j], abs_floor) : 0.0;
        const int h = __double2hiint(x);
        const bool low = !(h > __double2hiint(fl) && h < 0x7FF00000);
        broke |= low;
        return low ? fl : x;
      };
      double d = pivot(__shfl_sync(0xffffffffu, dg, 0), 0);
      double b = __shfl_sync(0xffffffffu, a[0], 1), D = __shfl_sync(0xffffffffu, dg, 1);
#pragma unroll
      for (int j = 0; j < kB; ++j) {
        double r0, e, dn = 1.0;
        recip_parts(d, r0, e);
        const double aj = a[j];
        auto minus = [&](double x, double pq) { const double p = pq * r0; return fma(-p, e, x - p); };  // x - pq / d
        if (j + 1 < kB) {
          dn = minus(D, b * b);
          a[j + 1] = minus(a[j + 1], aj * b);  // rows from j on; those above are done with
          dg = minus(dg, aj * aj);
        }
        if (j + 2 < kB) {
          b = __shfl_sync(0xffffffffu, a[j + 1], j + 2);
          D = __shfl_sync(0xffffffffu, dg, j + 2);
        }
        const double y = recip_sqrt(d);  // 1 / L_jj
        const double l = lane == j ? d * y : (lane > j ? aj * y : 0.0);
        Lc[j * kB + lane] = l;
        if (lane == 0) dinv[j] = y;
        if (j + 1 < kB) d = pivot(dn, j + 1);
        __syncwarp();
        if (j % 8 == 7) asm volatile("bar.arrive %0, 64;" ::"r"(2 + j / 8) : "memory");  // eight more columns for the inverse
#pragma unroll
        for (int j2 = (j + 2) & ~1; j2 < kB; j2 += 2) {
          const double2 v = *reinterpret_cast<const double2*>(Lc + j * kB + j2);
          if (j2 > j + 1) a[j2] -= l * v.x;
          a[j2 + 1] -= l * v.y;
        }
      }
      if (broke && rank == 0 && lane == 0) atomicOr(status, LORDO_FLAG_QR_BREAKDOWN);
      clear(c);  // not held in registers meanwhile
    } else if (warp < 3) {
      asm volatile("bar.arrive 1, 128;" ::: "memory");
      if (k + 1 < nb) block_sum<true>(c, L, k0 + kB, L, k0 + kB, r, warp - 1, k, 2);
    } else if (warp == 4) {
      asm volatile("bar.arrive 1, 128;" ::: "memory");
      if (k + 1 < nb) stage_diag(k + 1);  // before the first columns are there
      // inverse of the diagonal block, column `lane`, eight columns of the factor behind warp 0
      double x[kB];
#pragma unroll
      for (int i = 0; i < kB; ++i) x[i] = lane == i ? 1.0 : 0.0;
#pragma unroll
      for (int p = 0; p < kB; ++p) {
        if (p % 8 == 0) asm volatile("bar.sync %0, 64;" ::"r"(2 + p / 8) : "memory");
        x[p] *= dinv[p];
        Li[p * kLd + lane] = x[p];
#pragma unroll
        for (int i = (p + 1) & ~1; i < kB; i += 2) {
          const double2 v = *reinterpret_cast<const double2*>(Lc + p * kB + i);
          if (i > p) x[i] -= v.x * x[p];
          x[i + 1] -= v.y * x[p];
        }
      }
      clear(c);
    } else if (ahead && k + 1 < nb) {
      const int n1 = tiles(k + 1), s = slices(n1);
      if (u < n1 * s) {
        const int b = tile_block(k + 1, u / s), sl = u % s;
        block_sum<false>(c, b > k + 1 ? L : Z, b * kB, L, k0 + kB, r, (b > k + 1 ? 0 : b) + sl, k, s);
      }
    }

    // ---- Z_k = M Lkk^-T, eight rows of a block per warp and turn; the panel's own rows of rinv with the first batch
    const int lr = lane >> 2, lc = lane & 3;
    auto gram_init = [&](int b, int row, float (&g)[8]) {  // below the diagonal k0 + 32 <= row, so the columns exist
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) g[kk] = b > k && row < r ? A[(size_t)row * r + k0 + kk * 4 + lc] : 0.f;
    };
    float g[8];
    if (warp < first * 4) gram_init(tile_block(k, warp >> 2), tile_block(k, warp >> 2) * kB + (warp & 3) * 8 + lr, g);
    __syncthreads();  // the inverse of the diagonal block and the sums of the first batch are there
    for (int base = 0; base < ntiles || base == 0; base += kUnits) {
      const int cnt = ntiles - base < kUnits ? ntiles - base : kUnits;
      const int s = slices(cnt);
      if (base > 0) {
        __syncthreads();  // the batch before is done with its sums
        if (u < cnt * s) {
          const int b = tile_block(k, base + u / s);
          block_sum<false>(c, b > k ? L : Z, b * kB, L, k0, r, (b > k ? 0 : b) + u % s, k, s);
          store_part(part + u * kPartDoubles, c);
          clear(c);
        }
        __syncthreads();
      }
      const int strips = cnt * 4 + (base == 0 && has_k ? 4 : 0);
      for (int q = warp; q < strips; q += kCholWarps) {
        const int t = q >> 2, r8 = (q & 3) * 8;
        const bool diag = t == cnt;
        const int b = diag ? k : tile_block(k, base + t);
        const int row = b * kB + r8 + lr;
        if (!diag && (q != warp || base > 0)) gram_init(b, row, g);
        double z[4][2];
#pragma unroll
        for (int n = 0; n < 4; ++n) z[n][0] = z[n][1] = 0.0;
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const int col = kk * 4 + lc;
          double m;
          if (diag) {
            m = r8 + lr == col ? 1.0 : 0.0;
          } else {
            const double* q0 = part + (size_t)t * s * kPartDoubles + (r8 + lr) * kLd + col;
            double sum = 0.0;
#pragma unroll
            for (int sl = 0; sl < kUnits; ++sl)
              if (sl < s) sum += q0[(size_t)sl * kPartDoubles];
            m = (double)g[kk] - sum;
          }
#pragma unroll
          for (int n = 0; n < 4; ++n) dmma(z[n][0], z[n][1], m, Li[(8 * n + lr) * kLd + col]);
        }
        if (row < r) {
          float* out = (b > k ? L : Z) + (size_t)row * r + k0;
#pragma unroll
          for (int n = 0; n < 4; ++n) {
            const int col = 8 * n + 2 * lc;
            if (col >= kw) continue;
            float x = (float)z[n][0], y = (float)z[n][1];
            *reinterpret_cast<float2*>(out + col) = make_float2(x, y);
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
          }
        }
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

// CTAs per problem: as many, up to the portable cluster size, as leave every problem a place on the device at
// once (fifteen clusters of seven or eight fit, 22 of six: r = 512, 16 problems 375 us with four CTAs each, 325 with
// six) and every CTA about two row blocks.
void launch_chol_inverse(const CholProblem* probs, int nprobs, int r_max, unsigned* status, cudaStream_t st) {
  const int panels = (r_max + kB - 1) / kB;
  int c = 8;
  while (c > 1 && (2 * c > panels + 1 || nprobs > g_clusters[c])) --c;
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
