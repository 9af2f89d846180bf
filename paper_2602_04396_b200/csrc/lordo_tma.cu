// TMA-fed, persistent tensor-core kernels of the inner step: the projection for bf16 storage of G, E and W, the update for either.
//
//   project_tma_kernel  The streamed operand never passes through registers as single elements:
//                       TMA brings 64-row tiles of G, E (and of P^T) into 128B-swizzled shared
//                       memory, four warps turn the G tile into c*G + E in place (16-byte vector
//                       operations, layout-agnostic), and the tile is consumed as an MN-major
//                       operand by tcgen05.mma. Two accumulator buffers in tensor memory let the
//                       moment-update epilogue of one strip run under the main loop of the next
//                       (ranks above 256 as two half-rank strips, see the kernel). Runs as CTA
//                       pairs (clusters of two, tcgen05 cta_group::2): one strip per CTA, each CTA
//                       holding half of the rows of the P^T tile.
//   apply_tma_kernel    The strip's two low-rank operands (g^T, U~^T) live in tensor memory as the
//                       A operands; rows of P and the tiles of G, E, W arrive by TMA; the epilogue
//                       works on the swizzled tiles in shared memory (four neighbouring columns per
//                       thread, 8-byte accesses) and the updated E and W tiles leave by TMA stores.
//
// One CTA per SM; a CTA (the update kernel) or a CTA pair (the projection) walks its own list of
// 128-column strips or parts of strips, or of pairs of strips. Every role walks the same list, so stage
// and phase counters stay in step without further communication.
#include <algorithm>

#include "lordo_kernels.h"
#include "lordo_umma.cuh"

namespace lordo {

using namespace umma;

namespace {

constexpr int kStrip = 128;

__device__ __forceinline__ float bf_lo(uint32_t x) { return __uint_as_float(x << 16); }
__device__ __forceinline__ float bf_hi(uint32_t x) { return __uint_as_float(x & 0xFFFF0000u); }

// ---- projection ---------------------------------------------------------------------------------
constexpr int kPStages = 4;
constexpr uint32_t kPStageBytes = 49152;  // G 16 KB | E 16 KB | this CTA's rows of the P^T tile, up to 16 KB
constexpr int kPXformWarps = 4, kPEpiWarps = 16;
constexpr int kPThreads = (2 + kPXformWarps + kPEpiWarps) * 32;  // 704

// ---- update -------------------------------------------------------------------------------------
constexpr int kARows = 64, kARows32 = 32; // rows of W per step = MMA N, with bf16 and with fp32 storage
constexpr int kAInStages = 3, kAInStages32 = 4;  // G | E | W tiles, 16 KB each
constexpr uint32_t kAInStageBytes = 49152;
constexpr int kAPStages = 2;              // rows of P, up to 32 KB
constexpr uint32_t kAPStageBytes = 32768;
constexpr int kAEpiWarps = 16;
constexpr int kAThreads = (3 + kAEpiWarps) * 32;  // 608: TMA inputs, MMA, 16 epilogue warps, TMA rows of P

}  // namespace

// =================================================================================================
// 256 < r <= 512: the accumulator of a whole strip would fill all 512 columns of tensor memory and leave
// no second buffer, so such a problem is dealt out as two strips per 128 columns, one per half of the
// rank (rows [0, 256) and [256, r) of P^T, of the moments and of the low-rank operands). The two halves
// are neighbours in the strip list, hence run on neighbouring CTAs at the same time, and the second
// read of the G and E tiles is served by L2. Each half is then the r <= 256 pipeline: four stages, two
// accumulator buffers, the moment epilogue of one strip under the main loop of the next.
//
// The kernel runs as CTA pairs (clusters of two, tcgen05 cta_group::2): a pair works on two neighbouring
// strips of a problem (and the same half of the rank), one per CTA, and every MMA spans both (M = 256),
// so each CTA fetches and keeps only half of the rows of the P^T tile. Each CTA's loads complete on
// its own barrier; its transform warps pass the stage on to the MMA thread of the pair's first CTA.
// A problem with an odd number of strips ends in a pair whose second CTA reads zeros and stores nothing.
//
// Sixteen epilogue warps: the moment update (two loads, two stores, a square root and a division per low-rank
// element) is as long as the k loop at r = m / 8 with eight. 14 layers of 2048 (r = 256, K = 8) 882 -> 790 us, 7 layers of
// 768 (r = 128) 118 -> 91 us, the second with the strips dealt out by length as well.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPThreads, 1)
    project_tma_kernel(const TcProblem* __restrict__ probs, const TcSeg* __restrict__ segs, const int* __restrict__ start,
                       const TmaMatMaps* __restrict__ maps, const TmaGradMaps* __restrict__ gmaps, StepScalars sc, unsigned* __restrict__ status) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int ST = kPStages;
  constexpr uint32_t SB = kPStageBytes;
  // xform_bar and acc_empty are waited on by the MMA thread of the pair's first CTA only and fed by the
  // warps of both CTAs; empty_bar and acc_full are signalled in both CTAs by that thread's commits
  __shared__ uint64_t full_bar[kPStages], xform_bar[kPStages], empty_bar[kPStages], acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ float dsum_s[3][kStrip];

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const bool ef = sc.ef != 0;
  const uint32_t rank = cluster_rank();
  const int seg_begin = start[blockIdx.x >> 1], seg_end = start[(blockIdx.x >> 1) + 1];

  if (tid == 0) {
    for (int s = 0; s < ST; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&xform_bar[s], 2 * kPXformWarps); mbar_init(&empty_bar[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 2 * kPEpiWarps); }
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc_pair(&tmem_slot, 512);
  tc_fence_before_sync();
  cluster_sync();  // both CTAs' barriers exist before either reaches into the other
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  dep_begin();
  // pair lp of a problem -> this CTA's 128 columns and its half of the rank (split problems: the two
  // halves of a column pair are neighbouring pairs)
#define LORDO_PAIR_COORDS(pr, lp)                                                              \
  const int cs = 2 * ((pr)->nsplit == 2 ? lp >> 1 : lp) + (int)rank;                          \
  const int r_lo = (pr)->nsplit == 2 ? (lp & 1) * 256 : 0;

  if (warp == 0) {
    // ---------------- TMA producer ------------------------------------------------------------
    {
      const uint32_t one = elect_one();
      uint32_t it = 0;
      bool ok = true;
      for (int e = seg_begin; e < seg_end && ok; ++e) {
        const TcProblem* __restrict__ pr = probs + segs[e].prob;
        LORDO_PAIR_COORDS(pr, segs[e].strip)
        const int n0 = cs * kStrip;
        const TmaMatMaps* mm = maps + pr->mat;
        const TmaGradMaps* gm = gmaps + pr->mat;
        const int nkb = pr->m_k / 64, rep = pr->replica, pc = pr->pcopy;
        const int pt_rows = pr->r_n <= 256 ? pr->r_n / 2 : 128;  // rows of one P^T box: a CTA's half of an MMA's N
        const int n_h = pr->r_n - r_lo < 256 ? pr->r_n - r_lo : 256;
        const int pt_row0 = r_lo + (int)rank * (n_h / 2);
        const uint32_t tx = 16384u + (ef ? 16384u : 0u) + (uint32_t)pt_rows * 128u;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = it % ST;
          ok = mbar_wait_warp(&empty_bar[s], ((it / ST) & 1u) ^ 1u, status);
          if (!ok) break;
          unsigned char* base = smem + s * SB;
          mbar_expect_tx(&full_bar[s], tx, one);
          if (pr->tr) {  // stored transposed: the strip's 128 elements are stored rows, the k-block 64 stored columns
            tma_load_3d(base, gm->g_kb, kb * 64, n0, rep, &full_bar[s], one);
            if (ef) tma_load_3d(base + 16384, mm->e_kb, kb * 64, n0, rep, &full_bar[s], one);
          } else {
            tma_load_3d(base, gm->g_sw, n0, kb * 64, rep, &full_bar[s], one);
            tma_load_3d(base + 8192, gm->g_sw, n0 + 64, kb * 64, rep, &full_bar[s], one);
            if (ef) {
              tma_load_3d(base + 16384, mm->e_sw, n0, kb * 64, rep, &full_bar[s], one);
              tma_load_3d(base + 24576, mm->e_sw, n0 + 64, kb * 64, rep, &full_bar[s], one);
            }
          }
          tma_load_3d(base + 32768, mm->pt, kb * 64, pt_row0, pc, &full_bar[s], one);  // rows past r_n arrive as zeros
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issue ---------------------------------------------------------------
    if (rank == 0) {
      const uint32_t one = elect_one();
      uint32_t it = 0, si = 0;
      bool ok = true;
      // the barriers the commits arrive on, in this CTA and in the other (8 bytes apart within an array)
      const uint32_t eb0 = cluster_addr(&empty_bar[0], 0), eb1 = cluster_addr(&empty_bar[0], 1);
      const uint32_t af0 = cluster_addr(&acc_full[0], 0), af1 = cluster_addr(&acc_full[0], 1);
      for (int e = seg_begin; e < seg_end && ok; ++e, ++si) {
        const TcProblem* __restrict__ pr = probs + segs[e].prob;
        const int r_lo = pr->nsplit == 2 ? (segs[e].strip & 1) * 256 : 0;
        const int nkb = pr->m_k / 64;
        const uint32_t n_h = (uint32_t)(pr->r_n - r_lo < 256 ? pr->r_n - r_lo : 256);
        const bool tr = pr->tr != 0;  // the tile then lies as [128 strip elements][64 k]: a K-major operand
        const uint32_t idesc = idesc_bf16_f32(256, n_h) | (tr ? 0u : kIdescAMajorMN);
        const uint32_t buf = si & 1u;
        ok = mbar_wait_warp(&acc_empty[buf], ((si >> 1) & 1u) ^ 1u, status);
        if (!ok) break;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = it % ST;
          ok = mbar_wait_warp(&xform_bar[s], (it / ST) & 1u, status);
          if (!ok) break;
          tc_fence_after_sync();
          const uint32_t sA = smem_u32(smem + s * SB), sB = sA + 32768;
#pragma unroll
          for (int k16 = 0; k16 < 4; ++k16)
            mma_bf16_pair(tmem + buf * 256, tr ? smem_desc_k128(sA + k16 * 32) : smem_desc_mn128(sA + k16 * 2048), smem_desc_k128(sB + k16 * 32),
                          idesc, (kb > 0 || k16 > 0) ? 1u : 0u, one);
          if (one) { mma_commit_pair(eb0 + 8u * s); mma_commit_pair(eb1 + 8u * s); }
        }
        if (ok && one) { mma_commit_pair(af0 + 8u * buf); mma_commit_pair(af1 + 8u * buf); }
      }
    }
  } else if (warp < 2 + kPXformWarps) {
    // ---------------- transform: G tile <- c*G + E, in place ------------------------------------
    const int xt = tid - 64;
    uint32_t it = 0;
    bool ok = true;
    const uint32_t xf = cluster_addr(&xform_bar[0], 0);
    for (int e = seg_begin; e < seg_end && ok; ++e) {
      const TcProblem* __restrict__ pr = probs + segs[e].prob;
      const int nkb = pr->m_k / 64;
      const float c = *pr->cptr;
      for (int kb = 0; kb < nkb; ++kb, ++it) {
        const int s = it % ST;
        ok = mbar_wait(&full_bar[s], (it / ST) & 1u, status);
        if (!ok) break;
        uint4* G = reinterpret_cast<uint4*>(smem + s * SB);
        const uint4* E = G + 1024;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int idx = xt + i * 128;
          const uint4 g = G[idx];
          uint4 e = make_uint4(0u, 0u, 0u, 0u);
          if (ef) e = E[idx];
          uint4 a;
          a.x = pack2_bf16(fmaf(c, bf_lo(g.x), bf_lo(e.x)), fmaf(c, bf_hi(g.x), bf_hi(e.x)));
          a.y = pack2_bf16(fmaf(c, bf_lo(g.y), bf_lo(e.y)), fmaf(c, bf_hi(g.y), bf_hi(e.y)));
          a.z = pack2_bf16(fmaf(c, bf_lo(g.z), bf_lo(e.z)), fmaf(c, bf_hi(g.z), bf_hi(e.z)));
          a.w = pack2_bf16(fmaf(c, bf_lo(g.w), bf_lo(e.w)), fmaf(c, bf_hi(g.w), bf_hi(e.w)));
          G[idx] = a;
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(xf + 8u * s);  // this CTA's half of the stage is ready for the pair's MMAs
      }
    }
  } else {
    // ---------------- epilogue: moments on this thread's column, out of tensor memory -----------
    const int q = warp & 3, part = (warp - (2 + kPXformWarps)) >> 2;
    const float b1 = sc.beta1, b2 = sc.beta2, w = sc.omega;
    const bool low = sc.form == LORDO_QHM_LOW;
    uint32_t si = 0;
    bool ok = true;
    const uint32_t ae = cluster_addr(&acc_empty[0], 0);
    for (int e = seg_begin; e < seg_end && ok; ++e, ++si) {
      const TcProblem* __restrict__ pr = probs + segs[e].prob;
      LORDO_PAIR_COORDS(pr, segs[e].strip)
      const int n = pr->n, r = pr->r, r_k = pr->r_k;
      const int rn_h = pr->r_n - r_lo < 256 ? pr->r_n - r_lo : 256;  // rank rows of this strip, padded to 16
      const long long n0 = (long long)cs * kStrip;
      const long long ecol = n0 + q * 32 + lane;
      const bool e_ok = ecol < n;
      const long long ecolc = e_ok ? ecol : (long long)n - 1;
      float* __restrict__ up_ = pr->u;
      float* __restrict__ vp_ = pr->v;
      float* __restrict__ tb_ = pr->tb;
      // this column's 16-byte pieces inside the strip's block [r_k/8][128][8], from k-chunk r_lo/8 on
      const size_t lr_off = (size_t)cs * (size_t)r_k * 128 + (size_t)r_lo * 128 + (size_t)(q * 32 + lane) * 8;
      __nv_bfloat16* __restrict__ gT = pr->gT16 + lr_off;
      __nv_bfloat16* __restrict__ uT = pr->uT16 + lr_off;
      const uint32_t buf = si & 1u;
      ok = mbar_wait<64>(&acc_full[buf], (si >> 1) & 1u, status);
      if (!ok) break;
      tc_fence_after_sync();
      float dsum = 0.f;
      for (int ch = part; ch < rn_h / 16; ch += kPEpiWarps / 4) {
        float u[16], v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const size_t idx = (size_t)(unsigned)min(r_lo + ch * 16 + i, r - 1) * (size_t)n + (size_t)ecolc;
          u[i] = up_[idx];
          v[i] = vp_[idx];
        }
        float g[16];
        tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + buf * 256 + (uint32_t)(ch * 16), g);
        uint32_t gp[8], upk[8];
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
          float o[2];
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            const int row = r_lo + ch * 16 + i + t;
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
              if (tb_) tb_[idx] += sc.lr * o[t];
              dsum += D;
            } else {
              o[t] = 0.f;
            }
          }
          gp[i >> 1] = pack2_bf16(g[i], g[i + 1]);
          upk[i >> 1] = pack2_bf16(o[0], o[1]);
        }
        if (e_ok) {
          uint4* gd = reinterpret_cast<uint4*>(gT + (size_t)ch * 2048);  // k-chunks 2ch and 2ch+1, 128 pieces apart
          uint4* ud = reinterpret_cast<uint4*>(uT + (size_t)ch * 2048);
          gd[0] = make_uint4(gp[0], gp[1], gp[2], gp[3]); gd[128] = make_uint4(gp[4], gp[5], gp[6], gp[7]);
          ud[0] = make_uint4(upk[0], upk[1], upk[2], upk[3]); ud[128] = make_uint4(upk[4], upk[5], upk[6], upk[7]);
        }
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(ae + 8u * buf);
      if (sc.form == LORDO_QHM_FULL) {  // mu(D): mean over the rank axis, one value per column (a split problem: this half's share)
        if (part > 0) dsum_s[part - 1][q * 32 + lane] = dsum;
        asm volatile("bar.sync 1, %0;" ::"n"(kPEpiWarps * 32) : "memory");
        if (part == 0 && e_ok)
          (r_lo ? pr->dcol2 : pr->dcol)[ecol] = ((dsum + dsum_s[0][q * 32 + lane]) + (dsum_s[1][q * 32 + lane] + dsum_s[2][q * 32 + lane])) / (float)r;
        asm volatile("bar.sync 1, %0;" ::"n"(kPEpiWarps * 32) : "memory");
      }
    }
  }
#undef LORDO_PAIR_COORDS
  tc_fence_before_sync();
  __syncwarp();
  cluster_sync();  // neither CTA leaves while the other may still signal one of its barriers
  if (warp == 1) tmem_free_pair(tmem, 512);
}

// =================================================================================================
// MODE 0: r <= 256, both products in one sweep. For 256 < r <= 512 one low-rank operand alone fills
// 256 columns of tensor memory, so the update is two sweeps of the same kernel: MODE 1 does the
// error-feedback line (operand g^T, tiles G and E), MODE 2 the model update (operand U~^T, tiles G, W).
// SIDE 1: the problems of this launch are matrices projected from the right, whose W, G, E are stored
// transposed with respect to the problem: a strip is 128 stored rows, a step 64 stored columns, and the
// accumulator tile (lane = strip element, column = step element) already lies the way the tiles are
// stored, so a thread works on 16 neighbouring stored columns of its own row. SIDE 2: both kinds, told apart piece by
// piece; as two launches, each with its own start and end, five ragged matrices took 28 + 31 us, as one 46 us.
// F32: fp32 storage. A step is half as many rows, so a tile is as large and the accumulator half; tiles lie unswizzled, a row of 512 bytes
// after the other, and a thread works on one column. The rows of P take half the room, which gives a fourth stage of tiles. Bound by HBM and,
// where strips are few, by what an SM can have on its way. The kernel before it loaded G, E and W into registers itself, half of a step ahead:
// whole steps of 2048 x 2048, r = 128, K = 4 131 -> 120 us, 2048 x 5632, r = 256, K = 4 488 -> 412, seven matrices of 768 with two workers
// (strips of 12 and of 48 steps, all cut in the same number of parts) 354 -> 208, one 64 x 64 21.0 -> 21.1.
template <int MODE, int SIDE, bool F32>
__global__ void __launch_bounds__(kAThreads, 1) apply_tma_kernel(const TcProblem* __restrict__ probs, const TcSeg* __restrict__ segs,
                                                                 const int* __restrict__ start, const TmaMatMaps* __restrict__ maps,
                                                                 const TmaGradMaps* __restrict__ gmaps, StepScalars sc,
                                                                 unsigned* __restrict__ status) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  static_assert(!F32 || (MODE == 0 && SIDE == 0), "fp32 storage: ranks up to 256, matrices projected from the left");
  constexpr int ROWS = F32 ? kARows32 : kARows;
  constexpr uint32_t PSB = MODE ? 65536u : F32 ? kAPStageBytes / 2 : kAPStageBytes;  // one stage of rows of P
  constexpr int INST = F32 ? kAInStages32 : kAInStages;
  constexpr bool DO_E = MODE != 2, DO_W = MODE != 1;
  constexpr uint32_t A2COL = MODE ? 0u : 128u;             // first column of the U~^T operand
  // a stage holds the tiles the mode works on: G | E | W (MODE 0), G | E (MODE 1), G | W (MODE 2)
  constexpr uint32_t ISB = MODE ? 32768u : kAInStageBytes;
  constexpr uint32_t EOFF = 16384u, WOFF = MODE == 2 ? 16384u : 32768u;
  unsigned char* sP = smem;                      // kAPStages stages of rows of P
  unsigned char* sIn = smem + kAPStages * PSB;   // INST stages of tiles
  __shared__ uint64_t p_full[kAPStages], p_empty[kAPStages], in_full[INST], in_free[INST], acc_full[2], acc_empty[2], x_ready;
  __shared__ uint32_t tmem_slot;

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const bool ef = sc.ef != 0;
  const int seg_begin = start[blockIdx.x], seg_end = start[blockIdx.x + 1];

  if (tid == 0) {
    for (int s = 0; s < kAPStages; ++s) { mbar_init(&p_full[s], 1); mbar_init(&p_empty[s], 1); }
    for (int s = 0; s < INST; ++s) { mbar_init(&in_full[s], 1); mbar_init(&in_free[s], 4); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], kAEpiWarps * 32); }
    mbar_init(&x_ready, kAEpiWarps * 32);
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc(&tmem_slot, 512);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  dep_begin();
  // tensor memory: columns [0,256) the low-rank operands, two bf16 per column (MODE 0: g^T then U~^T,
  // 128 columns each); [256,512) two buffers of two accumulators

  if (warp == 0) {
    // ---------------- TMA producer: tiles of G, E, W ---------------------------------------------
    {
      const uint32_t one = elect_one();
      uint32_t jt = 0;
      bool ok = true;
      for (int e = seg_begin; e < seg_end && ok; ++e) {
        const TcSeg sg = segs[e];
        const TcProblem* __restrict__ pr = probs + sg.prob;
        const int n0 = sg.strip * kStrip;
        const TmaMatMaps* mm = maps + pr->mat;
        const TmaGradMaps* gm = gmaps + pr->mat;
        const int rep = pr->replica;
        for (int t = sg.t0; t < sg.t1; ++t, ++jt) {
          const int is = jt % INST;
          ok = mbar_wait_warp(&in_free[is], ((jt / INST) & 1u) ^ 1u, status);
          if (!ok) break;
          unsigned char* base = sIn + is * ISB;
          const bool ld_e = DO_E && ef;
          mbar_expect_tx(&in_full[is], 16384u + (ld_e ? 16384u : 0u) + (DO_W ? 16384u : 0u), one);
          if (F32) {  // one box of 32 rows x 128 columns per tile
            tma_load_3d(base, grad_map_f32(gmaps, pr->mat), n0, t * ROWS, rep, &in_full[is], one);
            if (ld_e) tma_load_3d(base + EOFF, mm->e_kb, n0, t * ROWS, rep, &in_full[is], one);
            tma_load_3d(base + WOFF, mm->w_kb, n0, t * ROWS, rep, &in_full[is], one);
          } else if (SIDE == 1 || (SIDE == 2 && pr->tr)) {  // one box of 128 stored rows x 64 stored columns per tile
            tma_load_3d(base, gm->g_kb, t * ROWS, n0, rep, &in_full[is], one);
            if (ld_e) tma_load_3d(base + EOFF, mm->e_kb, t * ROWS, n0, rep, &in_full[is], one);
            if (DO_W) tma_load_3d(base + WOFF, mm->w_kb, t * ROWS, n0, rep, &in_full[is], one);
          } else {
            for (int hh = 0; hh < 2; ++hh) {  // two 64-column halves per tile, 8 KB each
              tma_load_3d(base + hh * 8192, gm->g_sw, n0 + hh * 64, t * ROWS, rep, &in_full[is], one);
              if (ld_e) tma_load_3d(base + EOFF + hh * 8192, mm->e_sw, n0 + hh * 64, t * ROWS, rep, &in_full[is], one);
              if (DO_W) tma_load_3d(base + WOFF + hh * 8192, mm->w_sw, n0 + hh * 64, t * ROWS, rep, &in_full[is], one);
            }
          }
        }
      }
    }
  } else if (warp == 2 + kAEpiWarps) {
    // ---------------- TMA producer: rows of P ---------------------------------------------------
    {
      const uint32_t one = elect_one();
      uint32_t jt = 0;
      bool ok = true;
      for (int e = seg_begin; e < seg_end && ok; ++e) {
        const TcSeg sg = segs[e];
        const TcProblem* __restrict__ pr = probs + sg.prob;
        const TmaMatMaps* mm = maps + pr->mat;
        const int nkb = pr->r_k / 64, pc = pr->pcopy;
        for (int t = sg.t0; t < sg.t1; ++t, ++jt) {
          const int ps = jt % kAPStages;
          ok = mbar_wait_warp(&p_empty[ps], ((jt / kAPStages) & 1u) ^ 1u, status);
          if (!ok) break;
          mbar_expect_tx(&p_full[ps], (uint32_t)nkb * (ROWS * 128u), one);
          for (int kb = 0; kb < nkb; ++kb) tma_load_3d(sP + ps * PSB + kb * (ROWS * 128), mm->p16, kb * 64, t * ROWS, pc, &p_full[ps], one);
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issue: A operands from tensor memory ----------------------------------
    {
      const uint32_t idesc = idesc_bf16_f32(128, ROWS), one = elect_one();
      uint32_t jt = 0, si = 0;
      bool ok = true;
      for (int e = seg_begin; e < seg_end && ok; ++e, ++si) {
        const TcSeg sg = segs[e];
        const TcProblem* __restrict__ pr = probs + sg.prob;
        const int nkb = pr->r_k / 64;
        ok = mbar_wait_warp(&x_ready, si & 1u, status);
        if (!ok) break;
        for (int t = sg.t0; t < sg.t1; ++t, ++jt) {
          const int ps = jt % kAPStages;
          const uint32_t b = jt & 1u;
          ok = mbar_wait_warp(&p_full[ps], (jt / kAPStages) & 1u, status);
          if (ok) ok = mbar_wait_warp(&acc_empty[b], ((jt >> 1) & 1u) ^ 1u, status);
          if (!ok) break;
          tc_fence_after_sync();
          const uint32_t pbase = smem_u32(sP + ps * PSB);
          const uint32_t d1 = tmem + 256 + b * 128, d2 = d1 + 64;
          for (int kb = 0; kb < nkb; ++kb) {
#pragma unroll
            for (int k16 = 0; k16 < 4; ++k16) {
              const uint32_t acc = (kb > 0 || k16 > 0) ? 1u : 0u;
              const uint64_t bd = smem_desc_k128(pbase + kb * (ROWS * 128) + k16 * 32);
              const uint32_t acol = (uint32_t)(kb * 4 + k16) * 8;
              if (DO_E) mma_bf16_ts(d1, tmem + acol, bd, idesc, acc, one);
              if (DO_W) mma_bf16_ts(d2, tmem + A2COL + acol, bd, idesc, acc, one);
            }
          }
          if (one) {
            mma_commit(&p_empty[ps]);
            mma_commit(&acc_full[b]);
          }
        }
      }
    }
  } else {
    // ---------------- epilogue: 4 columns x 4 rows per thread and step ---------------------------
    // Lane l = 8a + b of a warp's lane quarter holds strip column 32q + 4b + a, so that the two
    // 16-lane accumulator loads hand thread t the four neighbouring columns 4(t/4)..+3 of rows
    // 2(t%4), +1, +8, +9 of its row group: 8-byte accesses to the swizzled tiles, free of conflicts.
    const int ew = warp - 2;
    const int q = warp & 3, grp = ew >> 2;  // lane quarter (fixed by the hardware), row group 0..3
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    const int tb = lane >> 2, tr = lane & 3;
    const int ecol0 = q * 32 + 4 * tb;  // first of this thread's four epilogue columns
    // byte offsets inside a 16 KB tile (two halves of 64 rows x 128 bytes, 128-byte swizzle)
    uint32_t toff[4];
#pragma unroll
    for (int ri = 0; ri < 4; ++ri) {
      const int rho = grp * 16 + (ri >> 1) * 8 + 2 * tr + (ri & 1);
      const int chunk = 4 * (q & 1) + (tb >> 1);
      toff[ri] = (uint32_t)((q >> 1) * 8192 + rho * 128 + ((chunk ^ (rho & 7)) << 4) + 8 * (tb & 1));
    }
    const float lr = sc.lr, om = sc.omega;
    const bool full = sc.form == LORDO_QHM_FULL;
    const float a2w = full ? om : 1.f;
    uint32_t jt = 0, si = 0;
    bool ok = true;
    for (int e = seg_begin; e < seg_end && ok; ++e, ++si) {
      const TcSeg sg = segs[e];
      const TcProblem* __restrict__ pr = probs + sg.prob;
      const int n = pr->n, r_k = pr->r_k;
      const int n0 = sg.strip * kStrip;
      const TmaMatMaps* mm = maps + pr->mat;
      const int rep = pr->replica;
      const bool tr_p = SIDE == 1 || (SIDE == 2 && pr->tr);
      const int colq = tr_p || F32 ? q * 32 + lane : q * 32 + 4 * (lane & 7) + (lane >> 3);  // strip element this lane's operands belong to
      const long long col = (long long)n0 + colq;
      const float c = *pr->cptr;
      float cd[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        // right side, fp32: one strip element per thread (its own row or column); else the four columns of the thread's epilogue block
        const long long ec = tr_p || F32 ? col : (long long)n0 + ecol0 + j;
        const long long ecc = ec < n ? ec : (long long)n - 1;
        cd[j] = full ? (1.f - om) * c / (pr->dcol[ecc] + (pr->dcol2 ? pr->dcol2[ecc] : 0.f)) : 0.f;
      }
      // this thread's quarter of its column's low-rank operands -> tensor memory (r_k/8 columns each)
      {
        const int per = r_k / 8;  // 32-bit columns of one operand handled by this row group
        // strip block [r_k/8][128][8]: this row group's k-chunks, this lane's column; a warp reads 512
        // contiguous bytes per instruction
        const size_t lr_off = (size_t)sg.strip * (size_t)r_k * 128 + (size_t)grp * (r_k / 32) * 1024 + (size_t)colq * 8;
        const uint4* __restrict__ g16 = reinterpret_cast<const uint4*>(pr->gT16 + lr_off);
        const uint4* __restrict__ u16 = reinterpret_cast<const uint4*>(pr->uT16 + lr_off);
        const bool live = col < n;
        for (int c0 = 0; c0 < per; c0 += 8) {
          if (DO_E) {
            uint4 glo = g16[(c0 >> 2) * 128], ghi = g16[(c0 >> 2) * 128 + 128];
            if (!live) glo = ghi = make_uint4(0u, 0u, 0u, 0u);
            tmem_st8(tmem + lane_base + (uint32_t)(grp * per + c0), glo, ghi);
          }
          if (DO_W) {
            uint4 ulo = u16[(c0 >> 2) * 128], uhi = u16[(c0 >> 2) * 128 + 128];
            if (!live) ulo = uhi = make_uint4(0u, 0u, 0u, 0u);
            tmem_st8(tmem + lane_base + A2COL + (uint32_t)(grp * per + c0), ulo, uhi);
          }
        }
        tmem_st_wait();
        tc_fence_before_sync();
        mbar_arrive(&x_ready);
      }
      for (int t = sg.t0; t < sg.t1; ++t, ++jt) {
        const int is = jt % INST;
        const uint32_t b = jt & 1u;
        unsigned char* base = sIn + is * ISB;
        ok = mbar_wait<32>(&in_full[is], (jt / INST) & 1u, status);
        if (ok) ok = mbar_wait<32>(&acc_full[b], (jt >> 1) & 1u, status);
        if (!ok) break;
        tc_fence_after_sync();
        if constexpr (F32) {
          // this thread: column 32 q + lane of the strip, rows 8 grp .. +7 of the step; a warp reads 128 bytes of a row
          float a1[8], a2[8];
          const uint32_t taddr = tmem + lane_base + 256 + b * 128 + (uint32_t)(grp * 8);
          tmem_ld8x2(taddr, taddr + 64, a1, a2);
          tc_fence_before_sync();
          mbar_arrive(&acc_empty[b]);
          float* at = reinterpret_cast<float*>(base) + grp * 8 * kStrip + q * 32 + lane;
          float *ae = at + EOFF / 4, *aw = at + WOFF / 4;
          float g[8], w[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) { g[i] = at[i * kStrip]; w[i] = aw[i * kStrip]; }
          if (ef) {
            float e[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) e[i] = ae[i * kStrip];
#pragma unroll
            for (int i = 0; i < 8; ++i) ae[i * kStrip] = (c * g[i] + e[i]) - a1[i];
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) aw[i * kStrip] = w[i] - lr * (cd[0] * g[i] + a2w * a2[i]);
          fence_async_smem();
          asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
          if ((ew & 3) == 0 && lane == 0) {  // a row group's 8 rows
            const int row = t * ROWS + grp * 8;
            if (row < pr->m) {
              if (ef) tma_store_3d(mm->e_st, n0, row, rep, base + EOFF + grp * 4096);
              tma_store_3d(mm->w_st, n0, row, rep, base + WOFF + grp * 4096);
            }
            tma_store_commit();
            tma_store_wait_read();
            mbar_arrive(&in_free[is]);
          }
        } else if (tr_p) {
          // this thread: stored row 32q + lane of the strip, stored columns 16 grp .. +15 of the step
          const int row = q * 32 + lane;
          const uint32_t o0 = swz_chunk(row, 2 * grp), o1 = swz_chunk(row, 2 * grp + 1);
          float a1[16], a2[16];
          const uint32_t taddr = tmem + lane_base + 256 + b * 128 + (uint32_t)(grp * 16);
          if (DO_E && DO_W) tmem_ld16x2(taddr, taddr + 64, a1, a2);
          else if (DO_E) tmem_ld16(taddr, a1);
          else tmem_ld16(taddr + 64, a2);
          tc_fence_before_sync();
          mbar_arrive(&acc_empty[b]);
          const uint4 gq[2] = {*reinterpret_cast<const uint4*>(base + o0), *reinterpret_cast<const uint4*>(base + o1)};
          const float cdv = cd[0];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const uint32_t off = h ? o1 : o0;
            const uint32_t gw[4] = {gq[h].x, gq[h].y, gq[h].z, gq[h].w};
            if (DO_E && ef) {
              const uint4 eq = *reinterpret_cast<const uint4*>(base + EOFF + off);
              const uint32_t ew4[4] = {eq.x, eq.y, eq.z, eq.w};
              uint32_t o[4];
#pragma unroll
              for (int j = 0; j < 4; ++j)
                o[j] = pack2_bf16((c * bf_lo(gw[j]) + bf_lo(ew4[j])) - a1[8 * h + 2 * j], (c * bf_hi(gw[j]) + bf_hi(ew4[j])) - a1[8 * h + 2 * j + 1]);
              *reinterpret_cast<uint4*>(base + EOFF + off) = make_uint4(o[0], o[1], o[2], o[3]);
            }
            if (DO_W) {
              const uint4 wq = *reinterpret_cast<const uint4*>(base + WOFF + off);
              const uint32_t ww[4] = {wq.x, wq.y, wq.z, wq.w};
              uint32_t o[4];
#pragma unroll
              for (int j = 0; j < 4; ++j)
                o[j] = pack2_bf16(bf_lo(ww[j]) - lr * (cdv * bf_lo(gw[j]) + a2w * a2[8 * h + 2 * j]),
                                  bf_hi(ww[j]) - lr * (cdv * bf_hi(gw[j]) + a2w * a2[8 * h + 2 * j + 1]));
              *reinterpret_cast<uint4*>(base + WOFF + off) = make_uint4(o[0], o[1], o[2], o[3]);
            }
          }
          // the four warps that share 32 stored rows hand them to the TMA engine on their own
          fence_async_smem();
          asm volatile("bar.sync %0, 128;" ::"r"(6 + q) : "memory");
          if (grp == 0 && lane == 0) {
            if (n0 + q * 32 < n) {
              if (DO_E && ef) tma_store_3d(mm->e_st32, t * ROWS, n0 + q * 32, rep, base + EOFF + q * 4096);
              if (DO_W) tma_store_3d(mm->w_st32, t * ROWS, n0 + q * 32, rep, base + WOFF + q * 4096);
            }
            tma_store_commit();
            tma_store_wait_read();
            mbar_arrive(&in_free[is]);
          }
        } else {
          const uint32_t taddr = tmem + lane_base + 256 + b * 128 + (uint32_t)(grp * 16);
          // both accumulators come out of tensor memory together and the buffer goes back to the MMA
          // warp before any arithmetic. a?[h][4k + 2jj + p]: column 2h + jj, row 8k + 2(t%4) + p.
          float a1[2][8], a2[2][8];
  #pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (DO_E) tmem_ld_16x256b_x2(taddr + ((uint32_t)(h * 16) << 16), a1[h]);       // (P g)^T
            if (DO_W) tmem_ld_16x256b_x2(taddr + 64 + ((uint32_t)(h * 16) << 16), a2[h]);  // (P U~)^T
          }
          tmem_ld_wait();
  #pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (DO_E) tmem_ld_pin8(a1[h]);
            if (DO_W) tmem_ld_pin8(a2[h]);
          }
          tc_fence_before_sync();
          mbar_arrive(&acc_empty[b]);
          uint2 gv[4], ev[4], wv[4];
  #pragma unroll
          for (int ri = 0; ri < 4; ++ri) {
            gv[ri] = *reinterpret_cast<const uint2*>(base + toff[ri]);
            if (DO_E && ef) ev[ri] = *reinterpret_cast<const uint2*>(base + EOFF + toff[ri]);
            if (DO_W) wv[ri] = *reinterpret_cast<const uint2*>(base + WOFF + toff[ri]);
          }
  #pragma unroll
          for (int ri = 0; ri < 4; ++ri) {
            const int k = ri >> 1, p = ri & 1;
            const float g0 = bf_lo(gv[ri].x), g1 = bf_hi(gv[ri].x), g2 = bf_lo(gv[ri].y), g3 = bf_hi(gv[ri].y);
            if (DO_E && ef) {
              const float e0 = (c * g0 + bf_lo(ev[ri].x)) - a1[0][4 * k + p];
              const float e1 = (c * g1 + bf_hi(ev[ri].x)) - a1[0][4 * k + 2 + p];
              const float e2 = (c * g2 + bf_lo(ev[ri].y)) - a1[1][4 * k + p];
              const float e3 = (c * g3 + bf_hi(ev[ri].y)) - a1[1][4 * k + 2 + p];
              *reinterpret_cast<uint2*>(base + EOFF + toff[ri]) = make_uint2(pack2_bf16(e0, e1), pack2_bf16(e2, e3));
            }
            if (DO_W) {
              const float w0 = bf_lo(wv[ri].x) - lr * (cd[0] * g0 + a2w * a2[0][4 * k + p]);
              const float w1 = bf_hi(wv[ri].x) - lr * (cd[1] * g1 + a2w * a2[0][4 * k + 2 + p]);
              const float w2 = bf_lo(wv[ri].y) - lr * (cd[2] * g2 + a2w * a2[1][4 * k + p]);
              const float w3 = bf_hi(wv[ri].y) - lr * (cd[3] * g3 + a2w * a2[1][4 * k + 2 + p]);
              *reinterpret_cast<uint2*>(base + WOFF + toff[ri]) = make_uint2(pack2_bf16(w0, w1), pack2_bf16(w2, w3));
            }
          }
          // the four warps of a row group hand their 16 rows to the TMA engine on their own
          fence_async_smem();
          asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
          if ((ew & 3) == 0 && lane == 0) {
            unsigned char* sb = base + grp * 2048;
            const int row = t * ROWS + grp * 16;
            for (int hh = 0; hh < 2; ++hh) {
              if (n0 + hh * 64 >= n) break;
              if (DO_E && ef) tma_store_3d(mm->e_st, n0 + hh * 64, row, rep, sb + EOFF + hh * 8192);
              if (DO_W) tma_store_3d(mm->w_st, n0 + hh * 64, row, rep, sb + WOFF + hh * 8192);
            }
            tma_store_commit();
            tma_store_wait_read();
            mbar_arrive(&in_free[is]);
          }
        }
      }
    }
    if ((grp == 0 || (ew & 3) == 0) && lane == 0) tma_store_wait_all();
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_free(tmem, 512);
}

// =================================================================================================
cudaError_t sketch_configure();

// How many CTA pairs of `kernel` the device holds at once. A persistent kernel that launched more would
// still be correct (no pair waits for another pair), but the pairs that start late would double its time.
template <typename Kernel>
static cudaError_t max_resident_pairs(Kernel kernel, int threads, size_t smem, int* pairs) {
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 2; at.val.clusterDim.y = 1; at.val.clusterDim.z = 1;
  lc.gridDim = dim3(2048, 1, 1); lc.blockDim = dim3((unsigned)threads, 1, 1); lc.dynamicSmemBytes = smem;
  lc.attrs = &at; lc.numAttrs = 1;
  return cudaOccupancyMaxActiveClusters(pairs, kernel, &lc);
}
static int g_project_pairs = 0, g_sketch_pairs = 0;  // set by tma_configure, per process (one device model per process)

cudaError_t tma_configure() {
  cudaError_t e = sketch_configure();
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(project_tma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kPStages * kPStageBytes + 1024));
  if (e != cudaSuccess) return e;
  e = max_resident_pairs(project_tma_kernel, kPThreads, kPStages * kPStageBytes + 1024, &g_project_pairs);
  if (e != cudaSuccess) return e;
  const int smem = (int)(kAPStages * 65536 + kAInStages * 32768 + 1024);  // the largest of the three modes
  const void* kernels[9] = {(const void*)apply_tma_kernel<0, 0, false>, (const void*)apply_tma_kernel<1, 0, false>, (const void*)apply_tma_kernel<2, 0, false>,
                            (const void*)apply_tma_kernel<0, 1, false>, (const void*)apply_tma_kernel<1, 1, false>, (const void*)apply_tma_kernel<2, 1, false>,
                            (const void*)apply_tma_kernel<0, 2, false>, (const void*)apply_tma_kernel<1, 2, false>, (const void*)apply_tma_kernel<2, 2, false>};
  for (const void* k : kernels)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return e;
}

cudaError_t tma_configure_f32() {
  return cudaFuncSetAttribute(apply_tma_kernel<0, 0, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kAPStages * kAPStageBytes / 2 + kAInStages32 * kAInStageBytes + 1024));
}

int project_pairs(int sm_count) { return g_project_pairs > 0 ? std::min(sm_count / 2, g_project_pairs) : sm_count / 2; }

void launch_project_tma(const TcProblem* probs, const TcSeg* segs, const int* start, int pairs, const TmaMatMaps* maps,
                        const TmaGradMaps* gmaps, const StepScalars& sc, unsigned* status, cudaStream_t st) {
  if (pairs <= 0) return;
  launch_dep(project_tma_kernel, dim3(2u * (unsigned)pairs), kPThreads, kPStages * kPStageBytes + 1024, st, probs, segs, start, maps, gmaps, sc, status);
}
void launch_apply_tma(const TcProblem* probs, const TcSeg* segs, const int* start, int ctas, const TmaMatMaps* maps, const TmaGradMaps* gmaps,
                      const StepScalars& sc, int f32, int mode, int side, unsigned* status, cudaStream_t st) {
  if (ctas <= 0) return;
  const size_t small = kAPStages * kAPStageBytes + kAInStages * kAInStageBytes + 1024, large = kAPStages * 65536 + kAInStages * 32768 + 1024;
#define LORDO_APPLY(M, T, SM) launch_dep(apply_tma_kernel<M, T, false>, dim3((unsigned)ctas), kAThreads, SM, st, probs, segs, start, maps, gmaps, sc, status)
#define LORDO_APPLY_SIDE(T)                    \
  if (mode == 0) LORDO_APPLY(0, T, small);      \
  else if (mode == 1) LORDO_APPLY(1, T, large); \
  else LORDO_APPLY(2, T, large)
  // Begun early at every rank. With the kernel before it that cost 12 to 25 % at r_k = 256; with this one, launched plainly,
  // 61 steps of random shapes with r_k = 256 are 1 % slower (median; the ten shortest 1 to 5 %), one is 6 % faster (six matrices, one of r = 256).
  if (f32)
    launch_dep(apply_tma_kernel<0, 0, true>, dim3((unsigned)ctas), kAThreads, kAPStages * kAPStageBytes / 2 + kAInStages32 * kAInStageBytes + 1024, st, probs, segs,
               start, maps, gmaps, sc, status);
  else if (side == 0) { LORDO_APPLY_SIDE(0); }
  else if (side == 1) { LORDO_APPLY_SIDE(1); }
  else { LORDO_APPLY_SIDE(2); }
#undef LORDO_APPLY_SIDE
#undef LORDO_APPLY
}

}  // namespace lordo

// =================================================================================================
// Sketch products of the refresh: C = S * B (fp32 out), S streamed by TMA. Same pipeline as the
// projection: TMA -> (optional c*G + E in place) -> tcgen05.mma -> epilogue out of tensor memory,
// two accumulator buffers.
//
// The kernel runs as CTA pairs (clusters of two, tcgen05 cta_group::2): a pair works on 256 rows of
// S, 128 per CTA, and every MMA spans both CTAs (M = 256), so each CTA fetches and keeps only half of
// the columns of B. With both operands in shared memory an MMA of one CTA reads 4 KB of A and 8 KB of B
// per 16-deep step at r = 256, more than the shared memory can feed at the tensor cores' rate; the
// pair halves B's share and its L2 traffic, and the freed shared memory holds one more stage. Each
// CTA's loads complete on its own barrier; its transform warps (which form c*G + E where asked) pass
// the stage on to the MMA thread of the pair's first CTA. The table counts tiles in pairs; a problem
// with an odd number of 128-row tiles ends in a pair whose second CTA reads zeros and stores nothing.
// =================================================================================================
namespace lordo {
using namespace umma;
namespace {
constexpr int kSMaxStages = 6;
constexpr uint32_t kSSmemBytes = 196608 + 1024;  // stages of A 16 KB [| E 16 KB] | B 16 KB, or 32 KB for r > 256
constexpr int kSThreads = (2 + 4 + 8) * 32;  // TMA, MMA, 4 transform warps, 8 epilogue warps
constexpr uint32_t kIdescBMajorMN = 1u << 16;

__device__ __forceinline__ int find_sk(const SkProblem* __restrict__ probs, int nprobs, long long tile) {
  int lo = 0, hi = nprobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].tile_start <= tile) lo = mid; else hi = mid - 1;
  }
  return lo;
}
}  // namespace

namespace {
// Columns of B that take part in the 64-deep step kb: of the first n_lo all but skip_lo, of the other n_hi all but skip_hi. With
// an upper triangular B (R^-1) the columns below 64 kb are zero there and cost neither loads nor MMAs; the first step of a
// pair of planes has them all, so it may overwrite the accumulator. r = 512, 16 workers: 11008 rows 385 -> 301 us, 4096 rows
// 160 -> 125 us. For r <= 256 the table's word is not looked at: the products with R^-1 of r = 256 gain 2 us each, but widths that may change
// from step to step cost each of a refresh's other launches up to a microsecond. Whole refreshes with the word looked at everywhere: 7
// matrices of 768, r = 128 507 -> 511 us; of 2048, r = 192 493 -> 495 us, r = 256 600 -> 597 us; two iterations of r = 256 1042 -> 1032 us.
struct SkCols {
  int lo, hi, skip_lo, skip_hi;
  __device__ __forceinline__ SkCols(int n_lo, int n_hi, int tri, int kb) {
    const int skip = tri ? kb * 64 : 0;
    skip_lo = skip < n_lo ? skip : n_lo;
    skip_hi = skip > 256 ? skip - 256 : 0;
    lo = n_lo - skip_lo;
    hi = n_hi - skip_hi;
  }
};
}  // namespace

// BIG: ranks above 256. WITH_E: the problems' A is c G + E, formed from two tiles; without, the stage is a third or a
// quarter smaller and the pipeline one or two stages deeper.
template <bool BIG, bool WITH_E>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSThreads, 1)
    sketch_tma_kernel(const SkProblem* __restrict__ probs, int nprobs, long long total_tiles, unsigned* __restrict__ status) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr uint32_t BOFF = WITH_E ? 32768u : 16384u;
  constexpr uint32_t SB = BOFF + (BIG ? 32768u : 16384u);  // A 16 KB | E 16 KB | this CTA's columns of B: up to 2 (+ 2) boxes of 8 KB
  constexpr int ST = 196608 / SB;
  static_assert(ST * SB + 1024 <= kSSmemBytes, "stages do not fit the shared memory asked for");
  // xform_bar and acc_empty are waited on by the MMA thread of the pair's first CTA only and fed by the
  // warps of both CTAs; empty_bar and acc_full are signalled in both CTAs by that thread's commits
  __shared__ uint64_t full_bar[kSMaxStages], xform_bar[kSMaxStages], empty_bar[kSMaxStages], acc_full[2], acc_empty[2];
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const uint32_t rank = cluster_rank();
  const long long tile_first = blockIdx.x >> 1, tile_step = gridDim.x >> 1;  // tiles of 256 rows, one per pair

  if (tid == 0) {
    for (int s = 0; s < ST; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&xform_bar[s], 8); mbar_init(&empty_bar[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 16); }
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc_pair(&tmem_slot, 512);
  tc_fence_before_sync();
  cluster_sync();  // both CTAs' barriers exist before either reaches into the other
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  dep_begin();

  if (warp == 0) {
    {
      const uint32_t one = elect_one();
      uint32_t it = 0;
      bool ok = true;
      for (long long tile = tile_first; tile < total_tiles && ok; tile += tile_step) {
        const SkProblem* __restrict__ pr = probs + find_sk(probs, nprobs, tile);
        const int m0 = (2 * (int)(tile - pr->tile_start) + (int)rank) * 128;
        const int nkb1 = (pr->Kd + 63) / 64;
        // this CTA's columns of B: half of the first 256 (one MMA) and half of the rest (a second MMA)
        const int n_lo = pr->r_n < 256 ? pr->r_n : 256, n_hi = pr->r_n - n_lo;
        const int j1 = pr->j1, tri = BIG ? pr->tri : 0;
        int seg = pr->j0 / nkb1, kb = pr->j0 - seg * nkb1;
        for (int j = pr->j0; j < j1; ++j, ++it, ++kb) {
          if (kb == nkb1) { kb = 0; ++seg; }
          const int a_c2 = pr->a_c2 + (int)((pr->pa >> (4 * seg)) & 15u) * pr->a_pl, b_c2 = pr->b_c2 + (int)((pr->pb >> (4 * seg)) & 15u) * pr->b_pl;
          const int s = it % ST;
          const SkCols cols(n_lo, n_hi, tri, kb);
          const int c_lo = cols.skip_lo + (int)rank * (cols.lo / 2), c_hi = 256 + cols.skip_hi + (int)rank * (cols.hi / 2);
          const int nbox_lo = (cols.lo / 2 + 63) / 64, nbox_hi = (cols.hi / 2 + 63) / 64;
          ok = mbar_wait_warp(&empty_bar[s], ((it / ST) & 1u) ^ 1u, status);
          if (!ok) break;
          unsigned char* base = smem + s * SB;
          mbar_expect_tx(&full_bar[s], 16384u + (WITH_E ? 16384u : 0u) + (uint32_t)(nbox_lo + nbox_hi) * 8192u, one);
          if (pr->a_mn) {  // S stored [Kd][M]: two boxes of 64 k-rows x 64 columns
            tma_load_3d(base, pr->map_a, m0, kb * 64, a_c2, &full_bar[s], one);
            tma_load_3d(base + 8192, pr->map_a, m0 + 64, kb * 64, a_c2, &full_bar[s], one);
            if (WITH_E) {
              tma_load_3d(base + 16384, pr->map_e, m0, kb * 64, a_c2, &full_bar[s], one);
              tma_load_3d(base + 24576, pr->map_e, m0 + 64, kb * 64, a_c2, &full_bar[s], one);
            }
          } else {         // S stored [M][Kd]: one box of 128 rows x 64 k
            tma_load_3d(base, pr->map_a, kb * 64, m0, a_c2, &full_bar[s], one);
            if (WITH_E) tma_load_3d(base + 16384, pr->map_e, kb * 64, m0, a_c2, &full_bar[s], one);
          }
          for (int x = 0; x < nbox_lo; ++x) tma_load_3d(base + BOFF + x * 8192, pr->map_b, c_lo + x * 64, kb * 64, b_c2, &full_bar[s], one);
          for (int x = 0; x < nbox_hi; ++x) tma_load_3d(base + BOFF + 16384 + x * 8192, pr->map_b, c_hi + x * 64, kb * 64, b_c2, &full_bar[s], one);
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      const uint32_t one = elect_one();
      uint32_t it = 0, si = 0;
      bool ok = true;
      // the barriers the commits arrive on, in this CTA and in the other (8 bytes apart within an array)
      const uint32_t eb0 = cluster_addr(&empty_bar[0], 0), eb1 = cluster_addr(&empty_bar[0], 1);
      const uint32_t af0 = cluster_addr(&acc_full[0], 0), af1 = cluster_addr(&acc_full[0], 1);
      for (long long tile = tile_first; tile < total_tiles && ok; tile += tile_step, ++si) {
        const SkProblem* __restrict__ pr = probs + find_sk(probs, nprobs, tile);
        const int nkb = pr->j1 - pr->j0;
        const bool a_mn = pr->a_mn != 0;
        const int n_lo = pr->r_n < 256 ? pr->r_n : 256, n_hi = pr->r_n - n_lo, tri = BIG ? pr->tri : 0, nkb1 = (pr->Kd + 63) / 64;
        const uint32_t majors = kIdescBMajorMN | (a_mn ? kIdescAMajorMN : 0u);
        int kk = pr->j0 % nkb1;  // 64-deep step within a pair of planes
        const uint32_t buf = BIG ? 0u : (si & 1u);
        ok = mbar_wait_warp(&acc_empty[buf], ((BIG ? si : (si >> 1)) & 1u) ^ 1u, status);
        if (!ok) break;
        for (int kb = 0; kb < nkb; ++kb, ++it, ++kk) {
          if (kk == nkb1) kk = 0;
          const int s = it % ST;
          const SkCols cols(n_lo, n_hi, tri, kk);
          const uint32_t idesc = idesc_bf16_f32(256, cols.lo ? (uint32_t)cols.lo : 16u) | majors, idesc_hi = idesc_bf16_f32(256, cols.hi ? (uint32_t)cols.hi : 16u) | majors;
          ok = mbar_wait_warp(&xform_bar[s], (it / ST) & 1u, status);
          if (!ok) break;
          tc_fence_after_sync();
          const uint32_t sA = smem_u32(smem + s * SB), sB = sA + BOFF;
#pragma unroll
          for (int k16 = 0; k16 < 4; ++k16) {
            const uint64_t ad = a_mn ? smem_desc_mn128(sA + k16 * 2048) : smem_desc_k128(sA + k16 * 32);
            if (!BIG || cols.lo) mma_bf16_pair(tmem + buf * 256 + cols.skip_lo, ad, smem_desc_mn128(sB + k16 * 2048), idesc, (kb > 0 || k16 > 0) ? 1u : 0u, one);
            if (BIG && cols.hi) mma_bf16_pair(tmem + 256 + cols.skip_hi, ad, smem_desc_mn128(sB + 2 * 8192 + k16 * 2048), idesc_hi, (kb > 0 || k16 > 0) ? 1u : 0u, one);
          }
          if (one) { mma_commit_pair(eb0 + 8u * s); mma_commit_pair(eb1 + 8u * s); }
        }
        if (ok && one) { mma_commit_pair(af0 + 8u * buf); mma_commit_pair(af1 + 8u * buf); }
      }
    }
  } else if (warp < 6) {
    const int xt = tid - 64;
    uint32_t it = 0;
    bool ok = true;
    const uint32_t xf = cluster_addr(&xform_bar[0], 0);
    for (long long tile = tile_first; tile < total_tiles && ok; tile += tile_step) {
      const SkProblem* __restrict__ pr = probs + find_sk(probs, nprobs, tile);
      const int nkb = pr->j1 - pr->j0;
      const float c = WITH_E ? *pr->cptr : 1.f;
      __nv_bfloat16* S16 = WITH_E ? pr->S16 : nullptr;
      const bool a_mn = pr->a_mn != 0;
      const int m0 = (2 * (int)(tile - pr->tile_start) + (int)rank) * 128;
      for (int kb = 0; kb < nkb; ++kb, ++it) {
        const int s = it % ST;
        ok = mbar_wait(&full_bar[s], (it / ST) & 1u, status);
        if (!ok) break;
        if (WITH_E) {
          uint4* G = reinterpret_cast<uint4*>(smem + s * SB);
          const uint4* E = G + 1024;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int idx = xt + i * 128;
            const uint4 g = G[idx], e = E[idx];
            uint4 a;
            a.x = pack2_bf16(fmaf(c, bf_lo(g.x), bf_lo(e.x)), fmaf(c, bf_hi(g.x), bf_hi(e.x)));
            a.y = pack2_bf16(fmaf(c, bf_lo(g.y), bf_lo(e.y)), fmaf(c, bf_hi(g.y), bf_hi(e.y)));
            a.z = pack2_bf16(fmaf(c, bf_lo(g.z), bf_lo(e.z)), fmaf(c, bf_hi(g.z), bf_hi(e.z)));
            a.w = pack2_bf16(fmaf(c, bf_lo(g.w), bf_lo(e.w)), fmaf(c, bf_hi(g.w), bf_hi(e.w)));
            G[idx] = a;
            if (S16) {  // every tile passes here once: eight lanes hold 128 neighbouring bytes of a stored row
              const int in_box = a_mn ? (idx >> 3) & 63 : idx >> 3, c8 = ((idx & 7) ^ (in_box & 7)) * 8;
              const int row = (a_mn ? kb * 64 : m0) + in_box, col = (a_mn ? m0 + (idx >> 9) * 64 : kb * 64) + c8;
              if (row < pr->S_rows && col < pr->S_cols) *reinterpret_cast<uint4*>(S16 + (size_t)row * pr->S_cols + col) = a;
            }
          }
          fence_async_smem();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(xf + 8u * s);  // this CTA's half of the stage is ready for the pair's MMAs
      }
    }
  } else {
    // epilogue: lane = row of the tile, r_n fp32 columns out of tensor memory, every other 16 of them per warp
    const int q = warp & 3, half = (warp - 6) >> 2;
    uint32_t si = 0;
    bool ok = true;
    const uint32_t ae = cluster_addr(&acc_empty[0], 0);
    for (long long tile = tile_first; tile < total_tiles && ok; tile += tile_step, ++si) {
      const SkProblem* __restrict__ pr = probs + find_sk(probs, nprobs, tile);
      const long long row = (2 * (tile - pr->tile_start) + rank) * 128 + q * 32 + lane;
      const bool row_ok = row < pr->M;
      float* __restrict__ crow = pr->C + (row_ok ? row : 0) * pr->ldc;
      const int r = pr->r, r_n = pr->r_n, planes = pr->planes;
      const uint32_t buf = BIG ? 0u : (si & 1u);
      ok = mbar_wait<64>(&acc_full[buf], (BIG ? si : (si >> 1)) & 1u, status);
      if (!ok) break;
      tc_fence_after_sync();
      for (int ch = half; ch < r_n / 16; ch += 2) {
        float v[16];
        tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + buf * 256 + (uint32_t)(ch * 16), v);
        if (planes) {
          // rounded to bf16, the residual being the next plane's value
          __nv_bfloat16* d = pr->C16 + (row_ok ? row : 0) * r + ch * 16;
          for (int p = 0; p < planes; ++p, d += pr->plane) {
            uint32_t w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              w[j] = pack2_bf16(v[2 * j], v[2 * j + 1]);
              v[2 * j] -= bf_lo(w[j]);
              v[2 * j + 1] -= bf_hi(w[j]);
            }
            if (row_ok) {
              *reinterpret_cast<uint4*>(d) = make_uint4(w[0], w[1], w[2], w[3]);
              if (ch * 16 + 8 < r) *reinterpret_cast<uint4*>(d + 8) = make_uint4(w[4], w[5], w[6], w[7]);
            }
          }
        } else if (row_ok) {
#pragma unroll
          for (int j = 0; j < 16; j += 4)
            if (ch * 16 + j < r) *reinterpret_cast<float4*>(crow + ch * 16 + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        }
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(ae + 8u * buf);
    }
  }
  tc_fence_before_sync();
  __syncwarp();
  cluster_sync();  // neither CTA leaves while the other may still signal one of its barriers
  if (warp == 1) tmem_free_pair(tmem, 512);
}

cudaError_t sketch_configure() {
  cudaError_t e = cudaFuncSetAttribute(sketch_tma_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSSmemBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(sketch_tma_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSSmemBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(sketch_tma_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSSmemBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(sketch_tma_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSSmemBytes);
  if (e != cudaSuccess) return e;
  return max_resident_pairs(sketch_tma_kernel<true, true>, kSThreads, kSSmemBytes, &g_sketch_pairs);
}
// total_tiles counts tiles of 256 rows (tile_start in `probs` does too); a CTA pair per SM pair.
void launch_sketch_tma(const SkProblem* probs, int nprobs, long long total_tiles, int grid, int big, int with_e, unsigned* status, cudaStream_t st) {
  if (total_tiles <= 0 || grid < 2) return;
  long long pairs = grid / 2;
  if (g_sketch_pairs > 0 && pairs > g_sketch_pairs) pairs = g_sketch_pairs;
  const unsigned g = 2u * (unsigned)(total_tiles < pairs ? total_tiles : pairs);
#define LORDO_SKETCH(B, E) launch_dep(sketch_tma_kernel<B, E>, dim3(g), kSThreads, kSSmemBytes, st, probs, nprobs, total_tiles, status)
  if (big && with_e) LORDO_SKETCH(true, true);
  else if (big) LORDO_SKETCH(true, false);
  else if (with_e) LORDO_SKETCH(false, true);
  else LORDO_SKETCH(false, false);
#undef LORDO_SKETCH
}

}  // namespace lordo

// =================================================================================================
// Self-test of the bounded wait: one thread waits on an mbarrier phase that nothing completes. The
// wait must give up after its limit, set LORDO_FLAG_DEVICE_TIMEOUT in *status and let the kernel end.
// =================================================================================================
namespace lordo {
__global__ void selftest_wait_kernel(unsigned* __restrict__ status) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    umma::mbar_init(&bar, 1);
    umma::mbar_init_fence();
    (void)umma::mbar_wait(&bar, 0u, status);
  }
}
void launch_selftest_wait(unsigned* status, cudaStream_t st) { selftest_wait_kernel<<<1, 32, 0, st>>>(status); }
}  // namespace lordo
