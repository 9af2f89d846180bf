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
//
// What bounds it: the chain of r columns (a reciprocal square root and two multiply-adds each) and one pass
// over the stored factors out of L2 per panel. Against one CTA per matrix with a thread per row: r = 512, 16
// matrices 2200 -> 669 us; r = 256, 7 matrices 580 -> 136 us; r = 128, 56 matrices 197 -> 67 us.
#include "lordo_kernels.h"

namespace lordo {
namespace {

constexpr int kB = 32;                       // panel width
constexpr int kCholWarps = 12;               // 4 on the diagonal block, 8 on the other blocks of the panel
constexpr int kUnits = 8;                    // partial sums of 32 x 32 blocks in flight, one per warp
constexpr int kLd = 40;                      // row stride of a partial sum: 16-byte stores of two rows meet no bank twice
constexpr int kPartDoubles = kB * kLd;
constexpr size_t kCholSmem = sizeof(double) * (size_t)((4 + kUnits) * kPartDoubles + kB * (2 * kB + 1) + kB);

__device__ __forceinline__ void dmma(double& c0, double& c1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1},{%2},{%3},{%0,%1};" : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}

// c (+)= X_j L_j^T over the 32-column blocks j = j0, j0 + dj, ... < j1 of two row blocks (32 rows from xr, lr on).
// Lane l holds rows l/4 + 8a and, of every 8 columns, columns 2(l%4) and +1: the same permutation of the
// summation index on both sides. Rows from r on read as zeros.
__device__ __forceinline__ void block_sum(double (&c)[4][4][2], const float* X, int xr, const float* L, int lr, int r, int j0, int j1, int dj) {
  const int lane = threadIdx.x & 31, row = lane >> 2, kc = (lane & 3) * 2;
  float2 a[4], b[4];
  auto fetch = [&](int col) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int ra = xr + row + 8 * i, rb = lr + row + 8 * i;
      a[i] = b[i] = make_float2(0.f, 0.f);
      if (ra < r) a[i] = *reinterpret_cast<const float2*>(X + (size_t)ra * r + col);
      if (rb < r) b[i] = *reinterpret_cast<const float2*>(L + (size_t)rb * r + col);
    }
  };
  if (j0 < j1) fetch(j0 * kB + kc);
  for (int j = j0; j < j1; j += dj) {
#pragma unroll 1
    for (int h = 0; h < 4; ++h) {
      double av[4][2], bv[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) { av[i][0] = a[i].x; av[i][1] = a[i].y; bv[i][0] = b[i].x; bv[i][1] = b[i].y; }
      if (h < 3) fetch(j * kB + (h + 1) * 8 + kc);  // the next 8 columns are on their way while these are multiplied
      else if (j + dj < j1) fetch((j + dj) * kB + kc);
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int n = 0; n < 4; ++n) dmma(c[i][n][0], c[i][n][1], av[i][t], bv[n][t]);
    }
  }
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
  extern __shared__ __align__(16) double csm[];
  double* dpart = csm;                               // [4] quarters of the diagonal block's sum
  double* part = dpart + 4 * kPartDoubles;           // [kUnits] partial sums of the other blocks
  double* Li = part + kUnits * kPartDoubles;         // [kB][kB + 1] inverse of the diagonal block of L
  double* Lc = Li + kB * (kB + 1);                   // [kB][kB] columns of the diagonal block of L
  double* dinv = Lc + kB * kB;                       // [kB] 1 / its diagonal
  __shared__ float wmax[kCholWarps];

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

  for (int k = 0; k < nb; ++k) {
    const int k0 = k * kB, kw = r - k0 < kB ? r - k0 : kB;  // this panel's columns
    // this CTA's other row blocks: b = rank, rank + csize, ... without k
    const int own = ((int)rank < nb ? (nb - 1 - (int)rank) / (int)csize + 1 : 0);
    const bool has_k = k % (int)csize == (int)rank;
    const int ntiles = own - (has_k ? 1 : 0);
    const int kpos = k / (int)csize;  // position of k in this CTA's list when has_k
    auto tile_block = [&](int t) { return (int)rank + (int)csize * ((has_k && t >= kpos) ? t + 1 : t); };
    // slices of the summation index per block, so that a batch of `cnt` blocks has work for every warp
    auto slices = [&](int cnt) {
      const int s = cnt > 0 ? kUnits / cnt : 1;
      return s < 1 ? 1 : s > k && k > 0 ? k : k > 0 ? s : 1;
    };
    auto unit = [&](int base, int cnt, int s) {  // a warp's share of a batch of `cnt` blocks in `s` slices each
      const int u = warp - 4;
      if (u >= cnt * s) return;
      const int b = tile_block(base + u / s), sl = u % s;
      double c[4][4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int n = 0; n < 4; ++n) c[i][n][0] = c[i][n][1] = 0.0;
      block_sum(c, b > k ? L : Z, b * kB, L, k0, r, (b > k ? 0 : b) + sl, k, s);
      store_part(part + u * kPartDoubles, c);
    };
    const int first = ntiles < kUnits ? ntiles : kUnits;  // blocks of the first batch

    if (warp < 4) {
      double c[4][4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int n = 0; n < 4; ++n) c[i][n][0] = c[i][n][1] = 0.0;
      block_sum(c, L, k0, L, k0, r, warp, k, 4);
      store_part(dpart + warp * kPartDoubles, c);
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (warp == 0) {
        // Factor of the diagonal block: lane i holds row i of what is left of the block. The next pivot is kept
        // up to date by its own lane (dg), so that the chain from column to column is a reciprocal square root
        // (one Newton step in fp64 on rsqrtf's 22 bits: 44 bits) and two multiply-adds; the update of the
        // columns behind the next one runs beside it.
        double a[kB], dg = 1.0;
        float own_floor = 0.f;
#pragma unroll
        for (int j = 0; j < kB; ++j) {
          const bool in = lane < kw && j < kw;
          double s = in ? (double)A[(size_t)(k0 + j) * r + k0 + lane] : (lane == j ? 1.0 : 0.0);  // A is symmetric
          if (in && lane == j) own_floor = fmaxf(kBreakdown * (float)s, abs_floor);
          const double* q = dpart + lane * kLd + j;
          s -= ((q[0] + q[kPartDoubles]) + (q[2 * kPartDoubles] + q[3 * kPartDoubles]));
          a[j] = s;
          if (lane == j) dg = s;
        }
        bool broke = false;
#pragma unroll
        for (int j = 0; j < kB; ++j) {
          double d = __shfl_sync(0xffffffffu, dg, j);
          float df = (float)d;
          const float fl = __shfl_sync(0xffffffffu, own_floor, j);
          if (!(df > fl)) {  // also catches NaN
            broke = true;
            df = fl;
            d = (double)fl;
          }
          const double y0 = (double)rsqrtf(df);
          const double y = fma(y0 * fma(-d * y0, y0, 1.0), 0.5, y0);  // 1 / L_jj
          const double l = lane == j ? d * y : (lane > j ? a[j] * y : 0.0);
          dg -= l * l;
          Lc[j * kB + lane] = l;
          if (lane == 0) dinv[j] = y;
          __syncwarp();
          if (j % 8 == 7) asm volatile("bar.arrive %0, 64;" ::"r"(2 + j / 8) : "memory");  // eight more columns for the inverse
#pragma unroll
          for (int j2 = j + 1; j2 < kB; ++j2) a[j2] -= l * Lc[j * kB + j2];
        }
        if (broke && lane == 0 && rank == 0) atomicOr(status, LORDO_FLAG_QR_BREAKDOWN);
      } else if (warp == 1) {
        // inverse of the diagonal block, column `lane`, eight columns of the factor behind warp 0
        double x[kB];
#pragma unroll
        for (int i = 0; i < kB; ++i) x[i] = lane == i ? 1.0 : 0.0;
#pragma unroll
        for (int p = 0; p < kB; ++p) {
          if (p % 8 == 0) asm volatile("bar.sync %0, 64;" ::"r"(2 + p / 8) : "memory");
          x[p] *= dinv[p];
          Li[p * (kB + 1) + lane] = x[p];
#pragma unroll
          for (int i = p + 1; i < kB; ++i) x[i] -= Lc[p * kB + i] * x[p];
        }
      }
    } else {
      unit(0, first, slices(first));
    }
    __syncthreads();  // the inverse of the diagonal block and the partial sums of the first batch are there

    for (int base = 0; base < ntiles || base == 0; base += kUnits) {
      const int cnt = ntiles - base < kUnits ? ntiles - base : kUnits;
      const int s = slices(cnt);
      if (base > 0) {
        __syncthreads();  // the batch before is done with its partial sums
        if (warp >= 4) unit(base, cnt, s);
        __syncthreads();
      }
      // Z_k = M Lkk^-T, eight rows of a block per warp and turn; the panel's own rows of rinv with the first batch
      const int strips = cnt * 4 + (base == 0 && has_k ? 4 : 0);
      for (int q = warp; q < strips; q += kCholWarps) {
        const int t = q >> 2, r8 = (q & 3) * 8;
        const bool diag = t == cnt;
        const int b = diag ? k : tile_block(base + t);
        const int row = b * kB + r8 + (lane >> 2);
        double c[4][2];
#pragma unroll
        for (int n = 0; n < 4; ++n) c[n][0] = c[n][1] = 0.0;
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const int col = kk * 4 + (lane & 3);
          double m;
          if (diag) {
            m = (r8 + (lane >> 2)) == col ? 1.0 : 0.0;
          } else {
            m = (b > k && row < r) ? (double)A[(size_t)row * r + k0 + col] : 0.0;  // below the diagonal k0 + 32 <= row, so the columns exist
            const double* q0 = part + (size_t)t * s * kPartDoubles + (r8 + (lane >> 2)) * kLd + col;
            double sum = 0.0;
            for (int sl = 0; sl < s; ++sl) sum += q0[(size_t)sl * kPartDoubles];
            m -= sum;
          }
#pragma unroll
          for (int n = 0; n < 4; ++n) dmma(c[n][0], c[n][1], m, Li[(8 * n + (lane >> 2)) * (kB + 1) + col]);
        }
        if (row < r) {
          float* out = (b > k ? L : Z) + (size_t)row * r + k0;
#pragma unroll
          for (int n = 0; n < 4; ++n) {
            const int col = 8 * n + 2 * (lane & 3);
            if (col >= kw) continue;
            float x = (float)c[n][0], y = (float)c[n][1];
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
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

// CTAs per problem: as many as the device has room for, up to the portable cluster size. More than half the
// problem's panels would idle.
void launch_chol_inverse(const CholProblem* probs, int nprobs, int r_max, int sm_count, unsigned* status, cudaStream_t st) {
  const int panels = (r_max + kB - 1) / kB;
  int c = 1;
  while (c < 8 && 2 * c <= panels && 2 * c * nprobs <= sm_count) c *= 2;
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)c; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
  lc.gridDim = dim3((unsigned)(nprobs * c), 1, 1); lc.blockDim = dim3(kCholWarps * 32, 1, 1); lc.dynamicSmemBytes = kCholSmem; lc.stream = st;
  lc.attrs = &at; lc.numAttrs = 1;
  cudaLaunchKernelEx(&lc, chol_inverse_kernel, probs, status);
}

cudaError_t chol_configure() { return cudaFuncSetAttribute(chol_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCholSmem); }

}  // namespace lordo
