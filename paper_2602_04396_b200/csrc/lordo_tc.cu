// Tensor-core (tcgen05 + tensor memory) projection of the inner step with fp32 storage, "fast mode":
//
//   project_tc_kernel  g^T = (cG+E)^T P  for one 128-column strip of one (matrix, worker), swept
//                      down the m rows; the low-rank moment update (Algorithm 1: u, v lines and the
//                      bracket of the update cases) runs in its epilogue straight out of tensor
//                      memory, so the low-rank gradient never goes to global memory in fp32.
//
// Where there are fewer strips than SMs, the rows of a strip are dealt out over a cluster of CTAs that exchange their partial
// accumulators through distributed shared memory, each finishing every S-th 16 ranks: 2048 x 2048, r = 128, K = 4 (64 strips) 98 -> 42 us.
//
// Orientation: the strip's columns (n) are the 128 lanes of tensor memory, so every epilogue
// thread owns one column and a warp touches 32 consecutive columns of a row of G, E, W, u or v.
// bf16 operands, fp32 accumulation. Operand tiles are written to shared memory by the kernels
// themselves (the streamed operand has to be formed as c*G + E and transposed anyway).
#include <algorithm>

#include "lordo_kernels.h"
#include "lordo_umma.cuh"

namespace lordo {

using namespace umma;

namespace {

constexpr int kStrip = 128;        // columns per strip = MMA M
constexpr int kProjThreads = 288;  // 8 producer/epilogue warps + 1 MMA warp

__device__ __forceinline__ int find_problem(const TcProblem* __restrict__ probs, int nprobs, long long strip) {
  int lo = 0, hi = nprobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].strip_start <= strip) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Storage type of G and E: fp32 alone (bf16 storage takes the TMA-fed projection), although the kernel is written for either and for ranks up
// to 512: as a plain function its loop compiles into one that is up to 2 % slower, and without the branches for ranks above 256, which
// nothing reaches, up to 5 % (2832 x 752, r = 256, K = 1 104.9 and 109.5 us).
template <bool BF16>
struct Elem;
template <>
struct Elem<false> {
  using one = float;
  using pair = float2;
  static __device__ __forceinline__ float2 cvt2(pair x) { return x; }
};

}  // namespace

// ---------------------------------------------------------------------------------------------
// P (fp32 [m][r]) -> P16 [m_r][r_k] and PT16 [r_n][m_k] in bf16; the pads stay zero.
// ---------------------------------------------------------------------------------------------
// One block per 64 x 64 tile of P: rows of P16 and, through a transposed tile in shared memory, rows of
// PT16 are both written as runs of consecutive addresses.
__global__ void __launch_bounds__(256) prep_projection_kernel(const TcPrep* __restrict__ items, const long long* __restrict__ blk_start,
                                                              int nitems) {
  dep_begin();
  __shared__ __nv_bfloat16 tile[64][66];
  const long long blk = blockIdx.x;
  const int i = find_segment(blk_start, nitems, blk);
  const TcPrep it = items[i];
  const long long local = blk - blk_start[i];
  const int tiles_c = (it.r + 63) / 64;
  const long long row0 = (local / tiles_c) * 64;
  const int col0 = (int)(local % tiles_c) * 64;
  for (int e = threadIdx.x; e < 64 * 64; e += 256) {
    const int rr = e >> 6, cc = e & 63;
    const long long row = row0 + rr;
    const int col = col0 + cc;
    if (row < it.m && col < it.r) {
      const __nv_bfloat16 h = __float2bfloat16_rn(it.P[row * it.r + col]);
      it.P16[row * it.r_k + col] = h;
      tile[rr][cc] = h;
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 64 * 64; e += 256) {
    const int cc = e >> 6, rr = e & 63;
    const long long row = row0 + rr;
    const int col = col0 + cc;
    if (row < it.m && col < it.r) it.PT16[(long long)col * it.m_k + row] = tile[rr][cc];
  }
}

// ---------------------------------------------------------------------------------------------
// project + moments
// ---------------------------------------------------------------------------------------------
template <bool BF16>
__global__ void __launch_bounds__(kProjThreads, 2) project_tc_kernel(const TcProblem* __restrict__ probs, int nprobs, StepScalars sc,
                                                                     unsigned* __restrict__ status) {
  using EL = Elem<BF16>;
  using one_t = typename EL::one;
  using pair_t = typename EL::pair;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t full_bar[2], empty_bar[2], done_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ float dsum_s[kStrip];
  const uint32_t rank = cluster_rank(), S = cluster_size();

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const long long strip = blockIdx.x / S;
  const TcProblem* __restrict__ prp = probs + find_problem(probs, nprobs, strip);
  const int m = prp->m, n = prp->n, r = prp->r, r_n = prp->r_n, m_k = prp->m_k, r_k = prp->r_k;
  const long long n0 = (strip - prp->strip_start) * kStrip;
  // this CTA's steps of 64 rows
  const int kb0 = (int)((long long)(m_k / 64) * rank / S), kb1 = (int)((long long)(m_k / 64) * (rank + 1) / S);
  const uint32_t a_bytes = kStrip * 128, b_bytes = (uint32_t)r_n * 128, stage_bytes = a_bytes + ((b_bytes + 1023) & ~1023u);
  const uint32_t ncols = tmem_cols_pow2((uint32_t)r_n);

  if (tid == 0) {
    for (int s = 0; s < 2; ++s) { mbar_init(&full_bar[s], 256); mbar_init(&empty_bar[s], 1); }
    mbar_init(&done_bar, 1);
    mbar_init_fence();
  }
  if (warp == 8) tmem_alloc(&tmem_slot, ncols);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  dep_begin();

  if (warp < 8) {
    // ---------------- producers: form (cG+E)^T tiles and copy P^T tiles -----------------------
    const int cp = tid & 63, kg = tid >> 6;  // column pair 0..63, k-group of 16 rows 0..3
    const long long col = n0 + 2 * cp;
    const bool col_ok = col < n;
    const long long colc = col_ok ? col : (long long)n - 2;  // loads stay in bounds, results are masked
    const one_t* __restrict__ Gp = reinterpret_cast<const one_t*>(*prp->G_ind) + prp->G_off;
    const bool have_e = sc.ef != 0;
    const one_t* __restrict__ Ep = have_e ? reinterpret_cast<const one_t*>(prp->E) : Gp;
    const one_t* __restrict__ Gc = Gp + colc;
    const one_t* __restrict__ Ec = Ep + colc;
    const float c = *prp->cptr;
    const float es = have_e ? 1.f : 0.f;
    const __nv_bfloat16* __restrict__ PT = prp->PT16;
    const int pt_chunks = r_n * 8;
    bool ok = true;
    for (int kb = kb0; kb < kb1 && ok; ++kb) {
      const int s = (kb - kb0) & 1, use = (kb - kb0) >> 1;
      pair_t rg[16], re[16];
      const int rbase = kb * 64 + kg * 16;
      if (rbase + 16 <= m) {
        const size_t base = (size_t)rbase * (size_t)n;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          rg[j] = *reinterpret_cast<const pair_t*>(Gc + base + (size_t)(unsigned)(j * n));
          re[j] = *reinterpret_cast<const pair_t*>(Ec + base + (size_t)(unsigned)(j * n));
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const size_t off = (size_t)(unsigned)min(rbase + j, m - 1) * (size_t)n;
          rg[j] = *reinterpret_cast<const pair_t*>(Gc + off);
          re[j] = *reinterpret_cast<const pair_t*>(Ec + off);
        }
      }
      uint4 pt[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        int idx = tid + t * 256;
        idx = idx < pt_chunks ? idx : pt_chunks - 1;
        pt[t] = *reinterpret_cast<const uint4*>(PT + (long long)(idx >> 3) * m_k + kb * 64 + (idx & 7) * 8);
      }
      float2 a[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float2 g = EL::cvt2(rg[j]), e = EL::cvt2(re[j]);
        const float live = (col_ok && rbase + j < m) ? 1.f : 0.f;
        a[j] = make_float2(live * (c * g.x + es * e.x), live * (c * g.y + es * e.y));
      }
      ok = mbar_wait(&empty_bar[s], (uint32_t)((use & 1) ^ 1), status);
      if (!ok) break;
      unsigned char* sA = smem + s * stage_bytes;
      unsigned char* sB = sA + a_bytes;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint4 lo, hi;
        lo.x = pack2_bf16(a[8 * q + 0].x, a[8 * q + 1].x); lo.y = pack2_bf16(a[8 * q + 2].x, a[8 * q + 3].x);
        lo.z = pack2_bf16(a[8 * q + 4].x, a[8 * q + 5].x); lo.w = pack2_bf16(a[8 * q + 6].x, a[8 * q + 7].x);
        hi.x = pack2_bf16(a[8 * q + 0].y, a[8 * q + 1].y); hi.y = pack2_bf16(a[8 * q + 2].y, a[8 * q + 3].y);
        hi.z = pack2_bf16(a[8 * q + 4].y, a[8 * q + 5].y); hi.w = pack2_bf16(a[8 * q + 6].y, a[8 * q + 7].y);
        *reinterpret_cast<uint4*>(sA + swz_chunk(2 * cp, kg * 2 + q)) = lo;
        *reinterpret_cast<uint4*>(sA + swz_chunk(2 * cp + 1, kg * 2 + q)) = hi;
      }
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const int idx = tid + t * 256;
        if (idx < pt_chunks) *reinterpret_cast<uint4*>(sB + swz_chunk(idx >> 3, idx & 7)) = pt[t];
      }
      if (r_n > 256) {  // rows 256.. of the P^T tile: not reached, see Elem
        for (int idx = 2048 + tid; idx < pt_chunks; idx += 256) {
          const uint4 v = *reinterpret_cast<const uint4*>(PT + (long long)(idx >> 3) * m_k + kb * 64 + (idx & 7) * 8);
          *reinterpret_cast<uint4*>(sB + swz_chunk(idx >> 3, idx & 7)) = v;
        }
      }
      fence_async_smem();
      mbar_arrive(&full_bar[s]);
    }

  } else {
    // ---------------- MMA issue ---------------------------------------------------------------
    const uint32_t one = elect_one();
    const uint32_t n_lo = r_n > 256 ? 256u : (uint32_t)r_n, n_hi = r_n > 256 ? (uint32_t)(r_n - 256) : 0u;
    const uint32_t idesc_lo = idesc_bf16_f32(128, n_lo), idesc_hi = idesc_bf16_f32(128, n_hi);
    bool ok = true;
    for (int kb = kb0; kb < kb1 && ok; ++kb) {
      const int s = (kb - kb0) & 1, use = (kb - kb0) >> 1;
      ok = mbar_wait_warp(&full_bar[s], (uint32_t)(use & 1), status);
      if (!ok) break;
      tc_fence_after_sync();
      const uint32_t sA = smem_u32(smem + s * stage_bytes), sB = sA + a_bytes;
#pragma unroll
      for (int k16 = 0; k16 < 4; ++k16) {
        const uint32_t acc = (kb > kb0 || k16 > 0) ? 1u : 0u;
        mma_bf16(tmem, smem_desc_k128(sA + k16 * 32), smem_desc_k128(sB + k16 * 32), idesc_lo, acc, one);
        if (n_hi) mma_bf16(tmem + 256, smem_desc_k128(sA + k16 * 32), smem_desc_k128(sB + 256 * 128 + k16 * 32), idesc_hi, acc, one);
      }
      if (one) mma_commit(&empty_bar[s]);
    }
    if (one) mma_commit(&done_bar);
  }

  // ---------------- partial accumulators of the ranks that other CTAs finish ---------------------
  // exch [chunk of 16 ranks not finished here][16][128 columns], over the stages that nothing reads any more
  float* exch = reinterpret_cast<float*>(smem);
  const int nch = r_n / 16, q = warp & 3;
  auto foreign = [&](int ch, int of) { return ch - (ch > of ? (ch - of + (int)S - 1) / (int)S : 0); };  // place of chunk ch in CTA `of`
  bool done = true;
  if (warp < 8) {
    done = mbar_wait<64>(&done_bar, 0u, status);
    tc_fence_after_sync();
    if (S > 1)
      for (int ch = warp >> 2; ch < nch; ch += 2) {
        if (ch % (int)S == (int)rank) continue;
        float g[16];
        tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ch * 16), g);
        float* to = exch + (size_t)foreign(ch, (int)rank) * 16 * kStrip + q * 32 + lane;
#pragma unroll
        for (int i = 0; i < 16; ++i) to[i * kStrip] = g[i];
      }
  }
  __syncwarp();
  if (S > 1) cluster_sync();
  if (warp < 8) {
    // ---------------- epilogue: moments on this thread's column ------------------------------
    const int half = warp >> 2;
    const long long ecol = n0 + q * 32 + lane;
    const bool e_ok = done && ecol < n;
    const long long ecolc = ecol < n ? ecol : (long long)n - 1;
    float* __restrict__ up_ = prp->u;
    float* __restrict__ vp_ = prp->v;
    const size_t lr_off = (size_t)(n0 / kStrip) * (size_t)r_k * kStrip + (size_t)(q * 32 + lane) * 8;  // this column's 16-byte pieces
    __nv_bfloat16* __restrict__ gT = prp->gT16 + lr_off;
    __nv_bfloat16* __restrict__ uT = prp->uT16 + lr_off;
    const float b1 = sc.beta1, b2 = sc.beta2, w = sc.omega;
    const bool low = sc.form == LORDO_QHM_LOW;
    float dsum = 0.f;
    for (int ch = (int)rank + (int)S * half; ch < nch; ch += 2 * (int)S) {
      float u[16], v[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const size_t idx = (size_t)(unsigned)min(ch * 16 + i, r - 1) * (size_t)n + (size_t)ecolc;
        u[i] = up_[idx];
        v[i] = vp_[idx];
      }
      float g[16];
      tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ch * 16), g);
      for (uint32_t o = 0; o < S; ++o) {  // the other CTAs' partial sums
        if (o == rank) continue;
        const uint32_t from = cluster_addr(exch + (size_t)foreign(ch, (int)o) * 16 * kStrip + q * 32 + lane, o);
#pragma unroll
        for (int i = 0; i < 16; ++i) g[i] += ld_cluster_f32(from + (uint32_t)(i * kStrip * 4));
      }
      uint32_t gp[8], upk[8];
#pragma unroll
      for (int i = 0; i < 16; i += 2) {
        float o[2];
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const int row = ch * 16 + i + t;
          const float gg = g[i + t];
          const float un = b1 * u[i + t] + (1.f - b1) * gg;
          const float vn = b2 * v[i + t] + (1.f - b2) * gg * gg;
          const float uh = un * sc.inv_bc1;
          const float D = sqrtf(vn * sc.inv_bc2) + sc.eps;
          o[t] = low ? (w * uh + (1.f - w) * gg) / D : uh / D;
          if (e_ok && row < r) {
            const size_t idx = (size_t)(unsigned)row * (size_t)n + (size_t)ecol;
            up_[idx] = un;
            vp_[idx] = vn;
            if (prp->tb) prp->tb[idx] += sc.lr * o[t];
            dsum += D;
          } else {
            o[t] = 0.f;
          }
        }
        gp[i >> 1] = pack2_bf16(g[i], g[i + 1]);
        upk[i >> 1] = pack2_bf16(o[0], o[1]);
      }
      if (e_ok) {
        uint4* gd = reinterpret_cast<uint4*>(gT + (size_t)ch * 2048);  // k-chunks 2 ch and 2 ch + 1, 128 pieces apart
        uint4* ud = reinterpret_cast<uint4*>(uT + (size_t)ch * 2048);
        gd[0] = make_uint4(gp[0], gp[1], gp[2], gp[3]); gd[128] = make_uint4(gp[4], gp[5], gp[6], gp[7]);
        ud[0] = make_uint4(upk[0], upk[1], upk[2], upk[3]); ud[128] = make_uint4(upk[4], upk[5], upk[6], upk[7]);
      }
    }
    if (sc.form == LORDO_QHM_FULL) {  // mu(D): mean over the rank axis, one value per column
      if (half == 1) dsum_s[q * 32 + lane] = dsum;
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (half == 0) {
        dsum += dsum_s[q * 32 + lane];
        if (S == 1 && e_ok) prp->dcol[ecol] = dsum / (float)r;
        dsum_s[q * 32 + lane] = dsum;  // the cluster's first CTA adds them up below
      }
    }
  }
  if (S > 1) {
    cluster_sync();
    if (rank == 0 && sc.form == LORDO_QHM_FULL && tid < kStrip && n0 + tid < n) {
      float dsum = dsum_s[tid];
      for (uint32_t o = 1; o < S; ++o) dsum += ld_cluster_f32(cluster_addr(dsum_s + tid, o));
      prp->dcol[n0 + tid] = dsum / (float)r;
    }
    cluster_sync();  // nobody leaves while its partial sums may still be read
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 8) tmem_free(tmem, ncols);
}

// ---------------------------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------------------------
// two stages, or the partial accumulators that a CTA of a cluster of four hands to the others
size_t project_tc_smem(int r_n_max) {
  const size_t stage = (size_t)kStrip * 128 + (((size_t)r_n_max * 128 + 1023) & ~size_t(1023));
  const size_t nch = (size_t)r_n_max / 16;
  return std::max(2 * stage, (nch - nch / 4) * 16 * kStrip * sizeof(float)) + 1024;
}
cudaError_t tc_configure(int r_n_max) {
  return cudaFuncSetAttribute(project_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)project_tc_smem(r_n_max));
}

void launch_prep_projection(const TcPrep* items, const long long* blk_start, int nitems, long long total_blocks, cudaStream_t st) {
  launch_dep(prep_projection_kernel, dim3((unsigned)total_blocks), 256, 0, st, items, blk_start, nitems);
}
// `steps`: 64-row steps of the problem with the fewest
void launch_project_tc(const TcProblem* probs, int nprobs, long long total_strips, int r_n_max, int steps, int sm_count, const StepScalars& sc,
                       unsigned* status, cudaStream_t st) {
  // two CTAs fit an SM; each is left four steps at least
  int c = 1;
  while (c < 4 && total_strips * 2 * c <= 2 * (long long)sm_count && steps >= 8 * c) c *= 2;
  // Begun under the end of the kernel before it (as launch_dep does), or as clusters of one, its CTAs are not spread over the SMs
  // but land two to an SM while others idle: four ragged matrices, r up to 256, 54 strips, step 355 us, plainly launched 285 us.
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)c; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
  lc.gridDim = dim3((unsigned)(total_strips * c), 1, 1); lc.blockDim = dim3(kProjThreads, 1, 1); lc.dynamicSmemBytes = project_tc_smem(r_n_max);
  lc.stream = st; lc.attrs = &at; lc.numAttrs = c > 1 ? 1 : 0;
  cudaLaunchKernelEx(&lc, project_tc_kernel<false>, probs, nprobs, sc, status);
}
}  // namespace lordo
