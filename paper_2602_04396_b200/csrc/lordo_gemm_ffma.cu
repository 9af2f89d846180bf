// Grouped fp32 FFMA GEMM with fused operand formation and epilogues: the fp32-accurate ("check
// mode") realisation of every contraction of the path -- P^T(cG+E), P g, P U~, the sketch and
// subspace-iteration products, Gram matrices, R^-1 application, Rot = P'^T P and the rotation of
// the moments. 64 x 64 output tile (64 x 32 with two products), 16-deep k-slices, 256 threads of 4 rows or 128 of 8.
// Products are formed and summed in fp32 inside a k-slice; the slice sums are carried across slices
// in fp64, so a result is accurate to fp32 rounding whatever the contraction length.
#include "lordo_kernels.h"

namespace lordo {

constexpr int BM = 64, BK = 16, PADS = 4;

// An operand as the main loop reads it, resolved once per tile.
struct Source {
  const void *p0, *p1;
  long long ld;
  float s0;
  int dt0, dt1, kind;
};
__device__ __forceinline__ Source resolve(const Operand& op) {
  Source s;
  const void* base = op.p0_ind ? *op.p0_ind : op.p0;
  s.p0 = reinterpret_cast<const char*>(base) + op.p0_off * (op.dt0 == LORDO_F32 ? 4 : 2);
  s.p1 = op.p1; s.ld = op.ld; s.s0 = 1.f; s.dt0 = op.dt0; s.dt1 = op.dt1; s.kind = op.kind;
  return s;
}

// Four consecutive stored elements of an operand as loaded; their value is formed when they are put into shared memory, so that
// nothing waits for a load before that.
struct Raw {
  float4 a, b;
};
// What one thread fetches of an operand, slice after slice: once or twice four elements, where they are next, how far the ones after them, and
// their k (of the row, or of the first of the four where k runs along the contiguous side). The contiguous side of every operand is
// a multiple of four, so four elements are inside or outside together; with two products and eight rows a thread the second
// four come from B2 at B's index, so both have one ld (the plans are checked for either).
struct Feed {
  long long at, step, second;
  int k, second_k, end, second_end;  // end: the contraction's length, or 0 where the other side's index is outside
};
__device__ __forceinline__ void feed_one(const Source& op, long long at, bool in, Raw& o) {
  o.a = o.b = make_float4(0.f, 0.f, 0.f, 0.f);
  if (in) {
    o.a = load4(op.p0, op.dt0, at);
    if (op.p1) o.b = load4(op.p1, op.dt1, at);
  }
}
template <int NL>
__device__ __forceinline__ void feed_next(const Source& op, const Source& op2, Feed& f, Raw (&o)[NL]) {
  feed_one(op, f.at, f.k < f.end, o[0]);
  if constexpr (NL > 1) feed_one(op2, f.at + f.second, f.k + f.second_k < f.second_end, o[1]);
  f.at += f.step;
  f.k += BK;
}
__device__ __forceinline__ float4 source_value(const Source& op, const Raw& x, const GemmScalars& sc) {
  if (op.kind == OP_PLAIN) return make_float4(op.s0 * x.a.x + x.b.x, op.s0 * x.a.y + x.b.y, op.s0 * x.a.z + x.b.z, op.s0 * x.a.w + x.b.w);
  const float4 u = make_float4(sc.inv_bc1 * x.a.x, sc.inv_bc1 * x.a.y, sc.inv_bc1 * x.a.z, sc.inv_bc1 * x.a.w);
  if (op.kind == OP_UHAT) return u;
  return make_float4(sc.inv_bc2 * x.b.x - u.x * u.x, sc.inv_bc2 * x.b.y - u.y * u.y, sc.inv_bc2 * x.b.z - u.z * u.z, sc.inv_bc2 * x.b.w - u.w * u.w);
}

// One output row, columns col .. col+3 (N is a multiple of 4).
template <int DUAL>
__device__ __forceinline__ void gemm_epilogue(const Epilogue& ep, const GemmScalars& sc, int N, long long row, long long col, const float (&a)[4],
                                              const float (&a2)[4]) {
  if (ep.kind == EPI_STORE && ep.trans) {  // C[col][row]
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float* cp = ep.C + (col + j) * ep.ldc + row;
      *cp = ep.pad ? *cp + a[j] : a[j];
    }
  } else if (ep.kind == EPI_STORE) {
    float4* cp = reinterpret_cast<float4*>(ep.C + row * ep.ldc + col);
    float4 o = make_float4(a[0], a[1], a[2], a[3]);
    if (ep.pad) {  // accumulate into C
      const float4 old = *cp;
      o.x += old.x; o.y += old.y; o.z += old.z; o.w += old.w;
    }
    *cp = o;
  } else if (ep.kind == EPI_APPLY && ep.trans) {
    // the product was formed for the transposed problem: output (row, col) is weight element (col, row),
    // and the full-rank QHM scale belongs to the output column = the weight's row
    if constexpr (DUAL) {
      const float c = *ep.cptr;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long long idx = (col + j) * ep.ldt + row;
        const float g = load1(*ep.G_ind, sc.g_dt, ep.G_off + idx);
        const float w = load1(ep.W, sc.w_dt, idx);
        float upd = a2[j];
        if (sc.form == LORDO_QHM_FULL) upd = (1.f - sc.omega) * (c * g) / ep.dcol[col + j] + sc.omega * upd;
        if (sc.ef) store1(ep.E, sc.e_dt, idx, (c * g + load1(ep.E, sc.e_dt, idx)) - a[j]);
        store1(ep.W, sc.w_dt, idx, w - sc.lr * upd);
      }
    }
  } else if (ep.kind == EPI_APPLY) {
    if constexpr (DUAL) {
      const long long idx = row * (long long)N + col;
      const float c = *ep.cptr;
      const float4 g = load4(*ep.G_ind, sc.g_dt, ep.G_off + idx);
      const float4 w = load4(ep.W, sc.w_dt, idx);
      float4 upd = make_float4(a2[0], a2[1], a2[2], a2[3]);
      if (sc.form == LORDO_QHM_FULL) {
        const float4 d = *reinterpret_cast<const float4*>(ep.dcol + col);
        const float w1 = 1.f - sc.omega;
        upd.x = w1 * (c * g.x) / d.x + sc.omega * upd.x;
        upd.y = w1 * (c * g.y) / d.y + sc.omega * upd.y;
        upd.z = w1 * (c * g.z) / d.z + sc.omega * upd.z;
        upd.w = w1 * (c * g.w) / d.w + sc.omega * upd.w;
      }
      if (sc.ef) {
        const float4 e = load4(ep.E, sc.e_dt, idx);
        float4 en;
        en.x = (c * g.x + e.x) - a[0];
        en.y = (c * g.y + e.y) - a[1];
        en.z = (c * g.z + e.z) - a[2];
        en.w = (c * g.w + e.w) - a[3];
        store4(ep.E, sc.e_dt, idx, en);
      }
      store4(ep.W, sc.w_dt, idx, make_float4(w.x - sc.lr * upd.x, w.y - sc.lr * upd.y, w.z - sc.lr * upd.z, w.w - sc.lr * upd.w));
    }
  } else {  // EPI_ROTATE: a = Rot u^, a2 = (Rot o Rot)(v^ - u^ o u^)
    if constexpr (DUAL) {
      const long long idx = row * (long long)N + col;
      float4 un, vn;
      un.x = sc.bc1 * a[0]; un.y = sc.bc1 * a[1]; un.z = sc.bc1 * a[2]; un.w = sc.bc1 * a[3];
      vn.x = sc.bc2 * fabsf(a2[0] + a[0] * a[0]);
      vn.y = sc.bc2 * fabsf(a2[1] + a[1] * a[1]);
      vn.z = sc.bc2 * fabsf(a2[2] + a[2] * a[2]);
      vn.w = sc.bc2 * fabsf(a2[3] + a[3] * a[3]);
      *reinterpret_cast<float4*>(ep.u_out + idx) = un;
      *reinterpret_cast<float4*>(ep.v_out + idx) = vn;
    }
  }
}

// Four partial sums of the CTA of rank `rank` of the cluster.
__device__ __forceinline__ void partials_of(const double* p, unsigned rank, double (&v)[4]) {
  const unsigned here = (unsigned)__cvta_generic_to_shared(p);
  unsigned there;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(here), "r"(rank));
  asm volatile("ld.shared::cluster.v2.f64 {%0,%1}, [%2];" : "=d"(v[0]), "=d"(v[1]) : "r"(there) : "memory");
  asm volatile("ld.shared::cluster.v2.f64 {%0,%1}, [%2];" : "=d"(v[2]), "=d"(v[3]) : "r"(there + 16u) : "memory");
}

// A cluster of CTAs works on one output tile, each on a range of k; the partial sums meet in fp64 through
// distributed shared memory, every CTA finishing its share of the tile's rows (see lordo_plan.h for the size).
// CARRY = 1: slice sums carried across k-slices in fp64 (parity mode). CARRY = 0: plain fp32
// accumulation, half the registers (the fp32 work of the fast mode: QR and moment rotation).
// With two products a tile is half as wide (gemm_columns): a thread then holds two columns of each, two CTAs fit an SM and the
// loads of one's epilogue (G, E, W) run under the other's products. Three ragged matrices with three workers, r up to 136: update
// 175 us with 256 threads of 4 x 4 outputs, 146 with 512 threads of 4 x 2, 120 with 256 of 4 x 2 of each.
// RN: rows per thread. A slice is latency as long as few warps run (fragments out of shared memory, conversions for the carry, a barrier):
// 3400 clocks of two CTAs an SM where the multiply-adds take 1000. Eight rows make twice as many independent ones per fragment, three
// CTAs fit an SM, and the sums' registers leave room for one slice on its way instead of two. Where CTAs are few, four rows in
// twice as many warps end sooner (256 x 256, r = 16 step 21.6 and 23.5 us; see split_by_time). With the sums of fast mode in 32 bits there are
// registers for four rows to do as well (refresh of 768 x 1536, r = 128, K = 4 with eight 944 us, with four 752). Steps of three ragged
// matrices with three workers, r up to 136: 186 -> 170 us; of 600 x 3000, r = 200, K = 2 252 -> 216; of 2048 x 2048, r = 128, K = 4 659 -> 584.
// Loads by a pointer that moves on from slice to slice instead of an index formed anew gave 3 % of a step (192 -> 186, 262 -> 252).

__device__ __forceinline__ void load_columns(float (&x)[4], const float* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}
__device__ __forceinline__ void load_columns(float (&x)[2], const float* p) {
  const float2 v = *reinterpret_cast<const float2*>(p);
  x[0] = v.x; x[1] = v.y;
}

// Two fp32 multiply-adds in one instruction, each rounded like fmaf. The main loop is bound by the issue of instructions
// (16 multiply-adds, two loads from shared memory): rows in pairs and columns doubled up make 14 of 18
// (three ragged matrices with three workers, projection 84 -> 78 us).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pair_of(float lo, float hi) {
  f32x2 p;
  asm("mov.b64 %0, {%1, %2};" : "=l"(p) : "f"(lo), "f"(hi));
  return p;
}
__device__ __forceinline__ void unpair(f32x2 p, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 square2(f32x2 a) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %1;" : "=l"(d) : "l"(a));
  return d;
}

template <int ATRANS, int DUAL, int CARRY, int RN>
__global__ void __launch_bounds__(1024 / RN, RN == 8 ? 3 : 2) gemm_ffma_kernel(const GemmProblem* __restrict__ probs, int nprobs, GemmScalars sc) {
  constexpr int NT = 1024 / RN, NL = 256 / NT, BN = gemm_columns(DUAL), CN = BN * BM / RN / NT;  // output columns per thread
  __shared__ __align__(16) float sA[2][BK][BM + PADS];
  __shared__ __align__(16) float sB[2][BK][BN + PADS];
  __shared__ __align__(16) float sB2[2][DUAL ? BK : 1][BN + PADS];
  extern __shared__ __align__(16) double part[];  // [1 or 2 products][BM][BN] partial sums of this CTA, clusters only
  unsigned rank, csize;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(csize));

  // locate the problem of this block
  const long long blk = blockIdx.x / csize;
  int lo = 0, hi = nprobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].tile_start <= blk) lo = mid; else hi = mid - 1;
  }
  const GemmProblem& pr = probs[lo];
  const long long local = blk - pr.tile_start;
  const int tile_m = (int)(local / pr.tiles_n), tile_n = (int)(local - (long long)tile_m * pr.tiles_n);
  const int M = pr.M, N = pr.N, Kd = pr.Kd;
  const long long m0 = (long long)tile_m * BM, n0 = (long long)tile_n * BN;

  Source A = resolve(pr.A), B = resolve(pr.B);
  const Source B2 = resolve(DUAL ? pr.B2 : pr.B);
  dep_begin();  // the tables are constant, and gradient pointers are copied in front of the kernel before this one
  if (pr.A.s0_ptr) A.s0 = *pr.A.s0_ptr;
  if (pr.B.s0_ptr) B.s0 = *pr.B.s0_ptr;

  const int t = threadIdx.x;
  const int tx = t % (BN / CN), ty = t / (BN / CN);
  // loaders, NL float4 of each operand a slice; with two products B and B2 share them, one each or one by each half of the threads
  const bool second = DUAL && NL == 1 && t >= NT / 2;
  const int lt = DUAL && NL == 1 ? t & (NT / 2 - 1) : t;
  const int bk = lt / (BN / 4), bc = lt % (BN / 4) * 4;  // row, columns four at a time; the second float4 NT / (BN / 4) rows on, or in B2
  const Source Bm = second ? B2 : B;
  // A. ATRANS: as B (stored [Kd][M]), the second 8 rows of k on. Otherwise stored [M][Kd]: row t/4, k (t%4)*4, the second 32 rows on.
  const int ar = ATRANS ? (t >> 4) : (t >> 2), ac = ATRANS ? (t & 15) * 4 : (t & 3) * 4;

  f32x2 acc[RN / 2][CN], acc2[DUAL ? RN / 2 : 1][CN];  // rows in pairs
  double tot[CARRY ? RN : 1][CN], tot2[(CARRY && DUAL) ? RN : 1][CN];
#pragma unroll
  for (int i = 0; i < RN; ++i)
#pragma unroll
    for (int j = 0; j < CN; ++j) {
      acc[i / 2][j] = 0ull;
      if constexpr (CARRY) tot[i][j] = 0.0;
      if constexpr (DUAL) {
        acc2[i / 2][j] = 0ull;
        if constexpr (CARRY) tot2[i][j] = 0.0;
      }
    }

  // One or two slices of k are on their way in registers while another, in one of two buffers, is multiplied.
  constexpr int kSecond = DUAL ? 0 : NT / (BN / 4);
  struct Slice {
    Raw a[NL], b[NL];
  };
  // this CTA's range of k
  const int per = ((Kd + BK - 1) / BK + (int)csize - 1) / (int)csize * BK;
  const int kbeg = min((int)rank * per, Kd), kend = min(kbeg + per, Kd);
  Feed fa, fb;
  if (ATRANS) fa = {(long long)(kbeg + ar) * A.ld + m0 + ac, (long long)BK * A.ld, 8 * A.ld, kbeg + ar, 8, m0 + ac < M ? Kd : 0, m0 + ac < M ? Kd : 0};
  else fa = {(m0 + ar) * A.ld + kbeg + ac, BK, 32 * A.ld, kbeg + ac, 0, m0 + ar < M ? Kd : 0, m0 + ar + 32 < M ? Kd : 0};
  fb = {(long long)(kbeg + bk) * Bm.ld + n0 + bc, (long long)BK * Bm.ld, kSecond * Bm.ld, kbeg + bk, kSecond, n0 + bc < N ? Kd : 0, n0 + bc < N ? Kd : 0};
  auto fetch = [&](Slice& s) {
    feed_next<NL>(A, A, fa, s.a);
    feed_next<NL>(Bm, DUAL ? B2 : B, fb, s.b);
  };
  auto stash = [&](const Slice& s, int buf) {
#pragma unroll
    for (int h = 0; h < NL; ++h) {
      const float4 v = source_value(A, s.a[h], sc);
      if (ATRANS) {
        *reinterpret_cast<float4*>(&sA[buf][ar + 8 * h][ac]) = v;
      } else {
        sA[buf][ac + 0][ar + 32 * h] = v.x; sA[buf][ac + 1][ar + 32 * h] = v.y; sA[buf][ac + 2][ar + 32 * h] = v.z; sA[buf][ac + 3][ar + 32 * h] = v.w;
      }
      const bool to2 = DUAL && (NL == 1 ? second : h == 1);
      *reinterpret_cast<float4*>(to2 ? &sB2[buf][DUAL ? bk : 0][bc] : &sB[buf][bk + kSecond * h][bc]) = source_value(DUAL && h ? B2 : Bm, s.b[h], sc);
    }
  };
  Slice x0, x1;
  if (kbeg < kend) fetch(x0);
  if (RN == 4 && kbeg + BK < kend) fetch(x1);
  if (kbeg < kend) stash(x0, 0);
  __syncthreads();
  int buf = 0;
  auto multiply = [&]() {
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      f32x2 a[RN / 2];
#pragma unroll
      for (int h = 0; h < RN / 4; ++h) {
        const float4 a4 = *reinterpret_cast<const float4*>(&sA[buf][kk][ty * RN + 4 * h]);
        a[2 * h] = pair_of(a4.x, a4.y); a[2 * h + 1] = pair_of(a4.z, a4.w);
      }
      float b[CN], c[CN];
      load_columns(b, &sB[buf][kk][tx * CN]);
#pragma unroll
      for (int j = 0; j < CN; ++j) {
        const f32x2 bb = pair_of(b[j], b[j]);
#pragma unroll
        for (int p = 0; p < RN / 2; ++p) acc[p][j] = fma2(a[p], bb, acc[p][j]);
      }
      if constexpr (DUAL) {
        load_columns(c, &sB2[buf][kk][tx * CN]);
        f32x2 a2[RN / 2];
#pragma unroll
        for (int p = 0; p < RN / 2; ++p) a2[p] = sc.a_square ? square2(a[p]) : a[p];
#pragma unroll
        for (int j = 0; j < CN; ++j) {
          const f32x2 cc = pair_of(c[j], c[j]);
#pragma unroll
          for (int p = 0; p < RN / 2; ++p) acc2[p][j] = fma2(a2[p], cc, acc2[p][j]);
        }
      }
    }
    if constexpr (CARRY) {
#pragma unroll
      for (int p = 0; p < RN / 2; ++p)
#pragma unroll
        for (int j = 0; j < CN; ++j) {
          float lo, hi;
          unpair(acc[p][j], lo, hi);
          tot[2 * p][j] += (double)lo; tot[2 * p + 1][j] += (double)hi;
          acc[p][j] = 0ull;
          if constexpr (DUAL) {
            unpair(acc2[p][j], lo, hi);
            tot2[2 * p][j] += (double)lo; tot2[2 * p + 1][j] += (double)hi;
            acc2[p][j] = 0ull;
          }
        }
    }
  };
  // on entry to a turn `far` is free, `near` holds the slice after the one in `buf` (RN = 8: they are one)
  auto turn = [&](int k0, Slice& far, const Slice& near) {
    if (k0 + (RN == 4 ? 2 : 1) * BK < kend) fetch(far);
    multiply();
    if (k0 + BK < kend) {
      stash(near, buf ^ 1);
      __syncthreads();
    }
    buf ^= 1;
  };
  if constexpr (RN == 4) {
    for (int k0 = kbeg; k0 < kend; k0 += 2 * BK) {
      turn(k0, x0, x1);
      if (k0 + BK < kend) turn(k0 + BK, x1, x0);
    }
  } else {
    for (int k0 = kbeg; k0 < kend; k0 += BK) turn(k0, x0, x0);
  }
  float out[RN][CN], out2[DUAL ? RN : 1][CN];  // without the carry: the sums
  if constexpr (!CARRY) {
#pragma unroll
    for (int p = 0; p < RN / 2; ++p)
#pragma unroll
      for (int j = 0; j < CN; ++j) {
        unpair(acc[p][j], out[2 * p][j], out[2 * p + 1][j]);
        if constexpr (DUAL) unpair(acc2[p][j], out2[2 * p][j], out2[2 * p + 1][j]);
      }
  }
  const Epilogue& ep = pr.epi;
  if (DUAL || csize > 1) {
#pragma unroll
    for (int i = 0; i < RN; ++i)
#pragma unroll
      for (int j = 0; j < CN; j += 2) {
        double* o = part + (ty * RN + i) * BN + tx * CN + j;
        if constexpr (CARRY) *reinterpret_cast<double2*>(o) = make_double2(tot[i][j], tot[i][j + 1]);
        else *reinterpret_cast<double2*>(o) = make_double2((double)out[i][j], (double)out[i][j + 1]);
        if constexpr (CARRY && DUAL) *reinterpret_cast<double2*>(o + BM * BN) = make_double2(tot2[i][j], tot2[i][j + 1]);
        else if constexpr (DUAL) *reinterpret_cast<double2*>(o + BM * BN) = make_double2((double)out2[i][j], (double)out2[i][j + 1]);
      }
    if (csize > 1) asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    else __syncthreads();
    const int rows = BM / (int)csize;
    for (int e = t; e < rows * (BN / 4); e += NT) {
      const int lr = (int)rank * rows + e / (BN / 4), lc = (e % (BN / 4)) * 4;
      const long long row = m0 + lr, col = n0 + lc;
      if (row >= M || col >= N) continue;
      double s1[4] = {0.0, 0.0, 0.0, 0.0}, s2[4] = {0.0, 0.0, 0.0, 0.0};
      for (unsigned q = 0; q < csize; ++q) {
        double v[4];
        partials_of(part + lr * BN + lc, q, v);
#pragma unroll
        for (int j = 0; j < 4; ++j) s1[j] += v[j];
        if constexpr (DUAL) {
          partials_of(part + BM * BN + lr * BN + lc, q, v);
#pragma unroll
          for (int j = 0; j < 4; ++j) s2[j] += v[j];
        }
      }
      const float a1[4] = {(float)s1[0], (float)s1[1], (float)s1[2], (float)s1[3]}, a2[4] = {(float)s2[0], (float)s2[1], (float)s2[2], (float)s2[3]};
      gemm_epilogue<DUAL>(ep, sc, N, row, col, a1, a2);
    }
    // nobody leaves while its partial sums may still be read
    if (csize > 1) asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    return;
  }
  if constexpr (!DUAL) {
    // each thread owns rows m0+ty*RN.., columns n0+tx*4..+3
    const long long col = n0 + tx * 4;
    if (col >= N) return;
#pragma unroll
    for (int i = 0; i < RN; ++i) {
      const long long row = m0 + ty * RN + i;
      if (row >= M) break;
      if constexpr (CARRY) {
#pragma unroll
        for (int j = 0; j < 4; ++j) out[i][j] = (float)tot[i][j];
      }
      gemm_epilogue<0>(ep, sc, N, row, col, out[i], out[i]);
    }
  }
}

// Rows per thread and CTAs per output tile: see lordo_plan.h.
void launch_gemm(const GemmProblem* probs, int nprobs, long long total_tiles, ProductSplit split, int atrans, int dual, int carry,
                 const GemmScalars& sc, cudaStream_t st) {
  const int c = split.ctas;
  const bool eight = split.rows == 8;
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)c; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // as launch_dep
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.gridDim = dim3((unsigned)(total_tiles * c), 1, 1); lc.blockDim = dim3(eight ? 128 : 256, 1, 1); lc.stream = st;
  lc.dynamicSmemBytes = c > 1 || dual ? sizeof(double) * BM * gemm_columns(dual) * (dual ? 2 : 1) : 0;
  lc.attrs = at; lc.numAttrs = 2;
#define LORDO_GEMM(A, B)                                                                     \
  if (eight) cudaLaunchKernelEx(&lc, gemm_ffma_kernel<A, B, 1, 8>, probs, nprobs, sc);        \
  else if (carry) cudaLaunchKernelEx(&lc, gemm_ffma_kernel<A, B, 1, 4>, probs, nprobs, sc);   \
  else cudaLaunchKernelEx(&lc, gemm_ffma_kernel<A, B, 0, 4>, probs, nprobs, sc)
  if (atrans && !dual) LORDO_GEMM(1, 0);
  else if (!atrans && !dual) LORDO_GEMM(0, 0);
  else if (!atrans && dual) LORDO_GEMM(0, 1);
  else LORDO_GEMM(1, 1);
#undef LORDO_GEMM
}

// With its partial sums a CTA exceeds the 48 KB of shared memory that a launch may ask for unannounced.
cudaError_t gemm_configure() {
  const int one = (int)(sizeof(double) * BM * gemm_columns(0)), two = (int)(2 * sizeof(double) * BM * gemm_columns(1));
  cudaError_t e = cudaSuccess;
  auto set = [&](const void* kernel, int smem) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  };
  set((const void*)gemm_ffma_kernel<0, 0, 0, 4>, one); set((const void*)gemm_ffma_kernel<0, 0, 1, 4>, one); set((const void*)gemm_ffma_kernel<0, 0, 1, 8>, one);
  set((const void*)gemm_ffma_kernel<1, 0, 0, 4>, one); set((const void*)gemm_ffma_kernel<1, 0, 1, 4>, one); set((const void*)gemm_ffma_kernel<1, 0, 1, 8>, one);
  set((const void*)gemm_ffma_kernel<0, 1, 0, 4>, two); set((const void*)gemm_ffma_kernel<0, 1, 1, 4>, two); set((const void*)gemm_ffma_kernel<0, 1, 1, 8>, two);
  set((const void*)gemm_ffma_kernel<1, 1, 0, 4>, two); set((const void*)gemm_ffma_kernel<1, 1, 1, 4>, two); set((const void*)gemm_ffma_kernel<1, 1, 1, 8>, two);
  return e;
}

// ---------------------------------------------------------------------------------------------
// Parallel cyclic Jacobi eigen-solver of a small symmetric matrix + the projector it is wanted for.
// A sweep is w - 1 steps (w made even with a dummy index); a step rotates w/2 disjoint index pairs
// (round-robin tournament order). Rotations of disjoint pairs commute, so a step is
//   C <- J^T C J,  V^T <- J^T V^T,  J = product of the step's plane rotations,
// done pair by pair: a warp forms rows p and q of J^T C from the old rows p and q (coalesced reads),
// keeps them in shared memory, applies the column rotations there and writes the two new rows.
// Old and new matrices are separate buffers, swapped after every step.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(512) jacobi_projector_kernel(const EigProblem* __restrict__ probs) {
  extern __shared__ float jsm[];
  const EigProblem pb = probs[blockIdx.x];
  const int w = pb.w, r = pb.r;
  const int we = (w + 1) & ~1;           // even number of players
  float* cc = jsm;                       // [we] own-row coefficient
  float* ss = cc + we;                   // [we] partner-row coefficient
  int* partner = reinterpret_cast<int*>(ss + we);  // [we]
  float* rowbuf = reinterpret_cast<float*>(partner + we);  // [16][2][w]
  __shared__ double red[16];
  __shared__ int done_s;
  const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
  float* Ca = pb.C;
  float* Cb = pb.work;
  float* Va = pb.work + (long long)w * w;
  float* Vb = pb.work + 2LL * w * w;
  for (long long e = t; e < (long long)w * w; e += 512) Va[e] = (e / w == e % w) ? 1.f : 0.f;  // V^T = I
  __syncthreads();

  for (int sweep = 0; sweep < 14; ++sweep) {
    // off-diagonal and diagonal weight: stop when the matrix is diagonal to fp32 accuracy
    double off = 0.0, dg = 0.0;
    for (long long e = t; e < (long long)w * w; e += 512) {
      const double x = (double)Ca[e];
      if (e / w == e % w) dg += x * x; else off += x * x;
    }
    for (int o = 16; o > 0; o >>= 1) { off += __shfl_xor_sync(0xffffffffu, off, o); dg += __shfl_xor_sync(0xffffffffu, dg, o); }
    if (lane == 0) red[wp] = off;
    __syncthreads();
    if (t == 0) { double s0 = 0.0; for (int k = 0; k < 16; ++k) s0 += red[k]; red[0] = s0; }
    __syncthreads();
    const double off_all = red[0];
    __syncthreads();
    if (lane == 0) red[wp] = dg;
    __syncthreads();
    if (t == 0) { double s0 = 0.0; for (int k = 0; k < 16; ++k) s0 += red[k]; done_s = off_all <= 1e-14 * (double)w * (double)w * s0; }
    __syncthreads();
    if (done_s) break;

    for (int step = 0; step < we - 1; ++step) {
      // ---- rotations of this step's pairs
      for (int k = t; k < we / 2; k += 512) {
        const int p = (step + k) % (we - 1);
        const int q = (k == 0) ? we - 1 : (step + we - 1 - k) % (we - 1);
        float c = 1.f, s = 0.f;
        if (p < w && q < w) {
          const double apq = (double)Ca[(long long)p * w + q];
          if (apq != 0.0) {
            const double app = (double)Ca[(long long)p * w + p], aqq = (double)Ca[(long long)q * w + q];
            const double theta = (aqq - app) / (2.0 * apq);
            const double tt = (theta >= 0.0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
            const double cd = 1.0 / sqrt(tt * tt + 1.0);
            c = (float)cd; s = (float)(tt * cd);
          }
        }
        // new row p = c row p - s row q ; new row q = s row p + c row q
        if (p < we) { partner[p] = q; cc[p] = c; ss[p] = -s; }
        if (q < we) { partner[q] = p; cc[q] = c; ss[q] = s; }
      }
      __syncthreads();
      // ---- rows of J^T C J and of J^T V^T, a pair of rows per warp: both new rows come from the same two
      // old rows, which are read once
      float* rbp = rowbuf + wp * 2 * w;
      float* rbq = rbp + w;
      for (int k = wp; k < we / 2; k += 16) {
        int p = (step + k) % (we - 1);
        int q = (k == 0) ? we - 1 : (step + we - 1 - k) % (we - 1);
        float c = cc[p], sn = -ss[p];  // new row p = c row p - sn row q ; new row q = sn row p + c row q
        const bool single = q >= w || p >= w;  // paired with the dummy index: the row is copied
        if (p >= w) p = q;
        if (single) { q = p; c = 1.f; sn = 0.f; }
#pragma unroll 4
        for (int j = lane; j < w; j += 32) {
          const float cp = Ca[(long long)p * w + j], cq = Ca[(long long)q * w + j];
          const float vp = Va[(long long)p * w + j], vq = Va[(long long)q * w + j];
          rbp[j] = c * cp - sn * cq;
          rbq[j] = sn * cp + c * cq;
          Vb[(long long)p * w + j] = c * vp - sn * vq;
          if (!single) Vb[(long long)q * w + j] = sn * vp + c * vq;
        }
        __syncwarp();
#pragma unroll 4
        for (int j = lane; j < w; j += 32) {
          int pj = partner[j];
          float cj = cc[j], sj = ss[j];
          if (pj >= w) { pj = j; cj = 1.f; sj = 0.f; }
          Cb[(long long)p * w + j] = cj * rbp[j] + sj * rbp[pj];
          if (!single) Cb[(long long)q * w + j] = cj * rbq[j] + sj * rbq[pj];
        }
        __syncwarp();
      }
      __syncthreads();
      float* x = Ca; Ca = Cb; Cb = x;
      x = Va; Va = Vb; Vb = x;
    }
  }
  __syncthreads();
  // ---- eigenvalues = diagonal of Ca; rank of each (0 = largest), kept in `partner`
  for (int i = t; i < w; i += 512) {
    const float li = Ca[(long long)i * w + i];
    int rk = 0;
    for (int j = 0; j < w; ++j) {
      const float lj = Ca[(long long)j * w + j];
      rk += (lj > li || (lj == li && j < i)) ? 1 : 0;
    }
    partner[i] = rk;
  }
  __syncthreads();
  // ---- Mr[a][b] = sum over the r leading eigenvectors v of v[a] v[b], b < r  (rows of V^T are eigenvectors)
  for (long long e = t; e < (long long)w * r; e += 512) {
    const int a = (int)(e / r), b = (int)(e - (long long)a * r);
    double acc = 0.0;
    for (int i = 0; i < w; ++i)
      if (partner[i] < r) acc += (double)Va[(long long)i * w + a] * (double)Va[(long long)i * w + b];
    pb.Mr[e] = (float)acc;
  }
}

void launch_jacobi_projector(const EigProblem* probs, int nprobs, int w_max, cudaStream_t st) {
  const int we = (w_max + 1) & ~1;
  const size_t smem = sizeof(float) * (size_t)(3 * we + 32 * w_max);
  static bool configured = false;  // w <= 600 (checked at init): at most 84 KB
  if (!configured) {
    cudaFuncSetAttribute(jacobi_projector_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(float) * (3 * 600 + 32 * 600)));
    configured = true;
  }
  jacobi_projector_kernel<<<nprobs, 512, smem, st>>>(probs);
}

}  // namespace lordo
