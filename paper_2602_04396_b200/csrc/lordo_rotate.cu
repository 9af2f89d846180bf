// Rotation of the moments into a new basis (Algorithm 1, moment-rotation lines), in place, one pass over u and v:
//
//   u <- bc1 (Rot u^),  v <- bc2 |(Rot o Rot)(v^ - u^ u^) + (Rot u^)^2|,   u^ = u / bc1, v^ = v / bc2
//
// For a strip of 128 columns both products are tcgen05.mma with the strip's columns as M, the new ranks as N and
// the old ranks as the contraction, fp32 accumulators side by side in tensor memory. Every operand is two bf16
// planes (16 bits); the products are hi lo + lo hi + hi hi. The planes of Rot^T and of its square come by TMA; the
// planes of u^ and of v^ - u^ u^ are formed from u and v in registers on their way into shared memory.
//
// CTA pairs (clusters of two). PAIR (every r <= 256): two strips, one per CTA, every MMA spanning both (M = 256,
// cta_group::2), so that each CTA loads and keeps only half of the columns of Rot^T. Otherwise the CTAs multiply on their
// own: a strip each, or, for r > 256, the same strip and half of the new ranks each; the second reading of u
// and v then comes out of L2, and neither writes before both have read.
//
// What bounds it: the planes of Rot^T and its square, which every strip pulls out of L2 again (256 KB at r = 256, beside
// 512 KB of u and v). Accumulators fill tensor memory, so a strip's products wait for the epilogue of the one before it;
// its first stages are filled meanwhile. 8 workers of 7 matrices of 2048 (r = 256): 447 us as separate passes (planes, two
// products, combination), 242 us with whole planes in each CTA and one set of warps for both ends, 183 us now; of 768
// (r = 128): 117, 59, 46 us; 16 workers of 4096 x 11008 (r = 512): 1050, 747, 696 us.
#include <algorithm>

#include "lordo_kernels.h"
#include "lordo_umma.cuh"

namespace lordo {

using namespace umma;

namespace {

constexpr int kStrip = 128, kRows = 32;  // columns of a strip, old ranks per stage
constexpr uint32_t kPlaneA = 8192;       // one plane of a stage: [2 groups of 64][32 rows][64] bf16
constexpr int kMaxStages = 3, kFormWarps = 8, kEpiWarps = 8;
constexpr int kThreads = (2 + kFormWarps + kEpiWarps) * 32;
constexpr size_t kSmem = 196608 + 1024;  // two stages with whole planes of Rot^T (4 groups of 64 columns), three with half

// as smem_desc_mn128, with 32 rows per 64-element group: the next group is 4096 bytes on
__device__ __forceinline__ uint64_t desc_mn_rows32(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(4096u >> 4) << 16;
  d |= (uint64_t)(1024u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

__device__ __forceinline__ int find_rotate(const RotateProblem* __restrict__ probs, int nprobs, long long item) {
  int lo = 0, hi = nprobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].item_start <= item) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Eight neighbouring values as two planes of 16 bytes.
__device__ __forceinline__ void store_planes(unsigned char* hi, unsigned char* lo, const float (&x)[8]) {
  uint32_t h[4], l[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    h[j] = pack2_bf16(x[2 * j], x[2 * j + 1]);
    l[j] = pack2_bf16(x[2 * j] - __uint_as_float(h[j] << 16), x[2 * j + 1] - __uint_as_float(h[j] & 0xFFFF0000u));
  }
  *reinterpret_cast<uint4*>(hi) = make_uint4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<uint4*>(lo) = make_uint4(l[0], l[1], l[2], l[3]);
}

}  // namespace

template <bool PAIR>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    rotate_kernel(const RotateProblem* __restrict__ probs, int nprobs, long long items, float inv_bc1, float inv_bc2, float bc1, float bc2,
                  unsigned* __restrict__ status) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr uint32_t kPlaneB = PAIR ? 8192 : 16384, kStage = 4 * kPlaneA + 4 * kPlaneB;
  constexpr int kStages = 196608 / kStage, kCtas = PAIR ? 2 : 1;  // CTAs behind one MMA
  // PAIR: full_a (here: A and B of both CTAs) and acc_empty are waited on by the MMA thread of the pair's first CTA only and
  // fed by the warps of both; empty_bar and acc_full are signalled in both CTAs by that thread's commits
  // peer_read: two barriers in turn, one per split strip. The other CTA arrives for a strip as soon as all warps here have arrived
  // for the one before it, whether or not each of them has seen that phase complete; on a single barrier a warp that
  // polls late would find the parity of the phase after it. Nobody arrives for the strip after the next before
  // every warp here has arrived for the next, hence has seen this one.
  __shared__ uint64_t full_a[kMaxStages], full_b[kMaxStages], empty_bar[kMaxStages], acc_full, acc_empty, peer_read[2];
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const uint32_t rank = cluster_rank();
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(&full_a[s], kCtas * kFormWarps); mbar_init(&full_b[s], 1); mbar_init(&empty_bar[s], 1); }
    mbar_init(&acc_full, 1); mbar_init(&acc_empty, kCtas * kEpiWarps); for (int b = 0; b < 2; ++b) mbar_init(&peer_read[b], kEpiWarps);
    mbar_init_fence();
  }
  if (warp == 1) {
    if (PAIR) tmem_alloc_pair(&tmem_slot, 512);
    else tmem_alloc(&tmem_slot, 512);
  }
  tc_fence_before_sync();
  cluster_sync();  // both CTAs' barriers exist before either reaches into the other
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  dep_begin();

  const long long first = blockIdx.x >> 1, step = gridDim.x >> 1;
  if (warp == 0) {
    // ---------------- TMA producer: planes of Rot^T and of its square -----------------------------
    {
      const uint32_t one = elect_one();
      uint32_t it = 0;
      bool ok = true;
      for (long long item = first; item < items && ok; item += step) {
        const RotateProblem* __restrict__ pr = probs + find_rotate(probs, nprobs, item);
        // the columns of Rot^T that this CTA keeps
        const int c0 = PAIR ? (int)rank * (pr->r_n / 2) : pr->nsplit == 2 ? (int)rank * 256 : 0;
        const int cols = PAIR ? pr->r_n / 2 : min(pr->r_n - c0, 256);
        const int nbox = (cols + 63) / 64, nkb = (pr->r + kRows - 1) / kRows;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = it % kStages;
          ok = mbar_wait_warp(&empty_bar[s], ((it / kStages) & 1u) ^ 1u, status);
          if (!ok) break;
          unsigned char* base = smem + s * kStage + 4 * kPlaneA;
          mbar_expect_tx(&full_b[s], 4u * (uint32_t)nbox * 4096u, one);
          for (int p = 0; p < 4; ++p)  // Rot^T hi, lo, square hi, lo
            for (int x = 0; x < nbox; ++x)
              tma_load_3d(base + p * kPlaneB + x * 4096, p < 2 ? pr->map_rt : pr->map_sq, c0 + x * 64, kb * kRows, (p & 1) * pr->nb + pr->b,
                          &full_b[s], one);
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issue --------------------------------------------------------------------
    if (!PAIR || rank == 0) {
      const uint32_t one = elect_one();
      uint32_t it = 0, si = 0;
      bool ok = true;
      const uint32_t eb0 = cluster_addr(&empty_bar[0], 0), eb1 = cluster_addr(&empty_bar[0], 1);
      const uint32_t af0 = cluster_addr(&acc_full, 0), af1 = cluster_addr(&acc_full, 1);
      for (long long item = first; item < items && ok; item += step, ++si) {
        const RotateProblem* __restrict__ pr = probs + find_rotate(probs, nprobs, item);
        const int r_lo = pr->nsplit == 2 ? (int)rank * 256 : 0, n_h = min(pr->r_n - r_lo, 256);
        const int nkb = (pr->r + kRows - 1) / kRows;
        const uint32_t idesc = idesc_bf16_f32(128 * kCtas, (uint32_t)n_h) | kIdescAMajorMN | (1u << 16);  // both operands MN-major
        ok = mbar_wait_warp(&acc_empty, (si & 1u) ^ 1u, status);
        for (int kb = 0; kb < nkb && ok; ++kb, ++it) {
          const int s = it % kStages;
          if (!PAIR) ok = mbar_wait_warp(&full_b[s], (it / kStages) & 1u, status);
          if (ok) ok = mbar_wait_warp(&full_a[s], (it / kStages) & 1u, status);
          if (!ok) break;
          tc_fence_after_sync();
          const uint32_t a = smem_u32(smem + s * kStage), b = a + 4 * kPlaneA;
#pragma unroll
          for (int k16 = 0; k16 < 2; ++k16)
#pragma unroll
            for (int d = 0; d < 2; ++d) {
              const uint32_t ah = a + 2 * d * kPlaneA + k16 * 2048, bh = b + 2 * d * kPlaneB + k16 * 2048, acc = tmem + 256 * d;
              const uint32_t more = (kb > 0 || k16 > 0) ? 1u : 0u;
              if (PAIR) {
                mma_bf16_pair(acc, desc_mn_rows32(ah), desc_mn_rows32(bh + kPlaneB), idesc, more, one);
                mma_bf16_pair(acc, desc_mn_rows32(ah + kPlaneA), desc_mn_rows32(bh), idesc, 1u, one);
                mma_bf16_pair(acc, desc_mn_rows32(ah), desc_mn_rows32(bh), idesc, 1u, one);
              } else {
                mma_bf16(acc, desc_mn_rows32(ah), desc_mn_rows32(bh + kPlaneB), idesc, more, one);
                mma_bf16(acc, desc_mn_rows32(ah + kPlaneA), desc_mn_rows32(bh), idesc, 1u, one);
                mma_bf16(acc, desc_mn_rows32(ah), desc_mn_rows32(bh), idesc, 1u, one);
              }
            }
          if (one) {
            if (PAIR) { mma_commit_pair(eb0 + 8u * s); mma_commit_pair(eb1 + 8u * s); }
            else mma_commit(&empty_bar[s]);
          }
        }
        if (ok && one) {
          if (PAIR) { mma_commit_pair(af0); mma_commit_pair(af1); }
          else mma_commit(&acc_full);
        }
      }
    }
  } else if (warp < 2 + kFormWarps) {
    // ---------------- planes of u^ and v^ - u^ u^ ---------------------------------------------------
    const int wt = tid - 64, ck = wt & 15, wr = wt >> 4;  // 8 columns from 8 ck on, rows wr and wr + 16 of a stage
    const uint32_t ready = cluster_addr(&full_a[0], 0);
    uint32_t it = 0;
    bool ok = true;
    for (long long item = first; item < items && ok; item += step) {
      const RotateProblem* __restrict__ pr = probs + find_rotate(probs, nprobs, item);
      const int lp = (int)(item - pr->item_start), n = pr->n, r = pr->r;
      const int n0 = (pr->nsplit == 2 ? lp : 2 * lp + (int)rank) * kStrip, nkb = (r + kRows - 1) / kRows;
      const float* __restrict__ up = pr->u;
      const float* __restrict__ vp = pr->v;
      const bool in = n0 + ck * 8 < n;  // n is a multiple of 8
      float4 un[2][2], vn[2][2];        // the coming stage's rows
      auto fetch = [&](int kb) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int row = kb * kRows + wr + 16 * i;
          const size_t at = (size_t)row * n + n0 + ck * 8;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            un[i][h] = vn[i][h] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (in && row < r) {
              un[i][h] = __ldcs(reinterpret_cast<const float4*>(up + at) + h);
              vn[i][h] = __ldcs(reinterpret_cast<const float4*>(vp + at) + h);
            }
          }
        }
      };
      fetch(0);
      for (int kb = 0; kb < nkb; ++kb, ++it) {
        const int s = it % kStages;
        float x[2][8], w[2][8];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float u8[8] = {un[i][0].x, un[i][0].y, un[i][0].z, un[i][0].w, un[i][1].x, un[i][1].y, un[i][1].z, un[i][1].w};
          const float v8[8] = {vn[i][0].x, vn[i][0].y, vn[i][0].z, vn[i][0].w, vn[i][1].x, vn[i][1].y, vn[i][1].z, vn[i][1].w};
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            x[i][j] = inv_bc1 * u8[j];
            w[i][j] = inv_bc2 * v8[j] - x[i][j] * x[i][j];
          }
        }
        if (kb + 1 < nkb) fetch(kb + 1);
        ok = mbar_wait(&empty_bar[s], ((it / kStages) & 1u) ^ 1u, status);
        if (!ok) break;
        unsigned char* base = smem + s * kStage;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int row = wr + 16 * i;
          const uint32_t off = (uint32_t)((ck >> 3) * 4096 + (row >> 3) * 1024 + (row & 7) * 128 + (((ck & 7) ^ (row & 7)) << 4));
          store_planes(base + off, base + kPlaneA + off, x[i]);
          store_planes(base + 2 * kPlaneA + off, base + 3 * kPlaneA + off, w[i]);
        }
        fence_async_smem();
        if (PAIR) ok = mbar_wait(&full_b[s], (it / kStages) & 1u, status);  // passed on together with this CTA's half of Rot^T
        if (!ok) break;
        __syncwarp();
        if (lane == 0) {
          if (PAIR) mbar_arrive_cluster(ready + 8u * s);
          else mbar_arrive(&full_a[s]);
        }
      }
    }
  } else {
    // ---------------- the rotated moments out of tensor memory ---------------------------------------
    const int q = warp & 3, half = (warp - (2 + kFormWarps)) >> 2;
    const uint32_t peer = cluster_addr(&peer_read[0], rank ^ 1u), drained = cluster_addr(&acc_empty, 0);
    uint32_t si = 0, split_items = 0;
    bool ok = true;
    for (long long item = first; item < items && ok; item += step, ++si) {
      const RotateProblem* __restrict__ pr = probs + find_rotate(probs, nprobs, item);
      const bool split = !PAIR && pr->nsplit == 2;
      const int lp = (int)(item - pr->item_start), n = pr->n, r = pr->r;
      const int r_lo = split ? (int)rank * 256 : 0, n_h = min(pr->r_n - r_lo, 256);
      const int col = (split ? lp : 2 * lp + (int)rank) * kStrip + q * 32 + lane;
      float* __restrict__ up = pr->u;
      float* __restrict__ vp = pr->v;
      ok = mbar_wait<32>(&acc_full, si & 1u, status);
      if (!ok) break;
      tc_fence_after_sync();
      if (split) {  // the other CTA has read this strip too
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(peer + 8u * (split_items & 1u));
        ok = mbar_wait<32>(&peer_read[split_items & 1u], (split_items >> 1) & 1u, status);
        ++split_items;
        if (!ok) break;
      }
      for (int ch = half; ch < n_h / 16; ch += 2) {
        float g[16], d[16];
        const uint32_t at = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ch * 16);
        tmem_ld16x2(at, at + 256, g, d);
        if (col < n) {
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int row = r_lo + ch * 16 + i;
            if (row < r) {
              const size_t to = (size_t)row * n + col;
              up[to] = bc1 * g[i];
              vp[to] = bc2 * fabsf(d[i] + g[i] * g[i]);
            }
          }
        }
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) {
        if (PAIR) mbar_arrive_cluster(drained);
        else mbar_arrive(&acc_empty);
      }
    }
  }
  tc_fence_before_sync();
  __syncwarp();
  cluster_sync();  // neither CTA leaves while the other may still signal its barriers
  if (warp == 1) {
    if (PAIR) tmem_free_pair(tmem, 512);
    else tmem_free(tmem, 512);
  }
}

static int g_rotate_pairs = 0;  // CTA pairs that the device holds at once, set by rotate_configure (one device model per process)

cudaError_t rotate_configure() {
  cudaError_t e = cudaFuncSetAttribute(rotate_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(rotate_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 2; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
  lc.gridDim = dim3(2048, 1, 1); lc.blockDim = dim3(kThreads, 1, 1); lc.dynamicSmemBytes = kSmem;
  lc.attrs = &at; lc.numAttrs = 1;
  return cudaOccupancyMaxActiveClusters(&g_rotate_pairs, rotate_kernel<true>, &lc);
}

void launch_rotate(const RotateProblem* probs, int nprobs, long long items, int r_max, int sm_count, const GemmScalars& sc, unsigned* status,
                   cudaStream_t st) {
  if (items <= 0) return;
  long long pairs = sm_count / 2;
  if (g_rotate_pairs > 0) pairs = std::min<long long>(pairs, g_rotate_pairs);
  const dim3 grid(2u * (unsigned)std::min(items, pairs));
  if (r_max <= 256) launch_dep(rotate_kernel<true>, grid, kThreads, kSmem, st, probs, nprobs, items, sc.inv_bc1, sc.inv_bc2, sc.bc1, sc.bc2, status);
  else launch_dep(rotate_kernel<false>, grid, kThreads, kSmem, st, probs, nprobs, items, sc.inv_bc1, sc.inv_bc2, sc.bc1, sc.bc2, status);
}

}  // namespace lordo
