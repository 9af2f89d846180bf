// Streaming (HBM-bound) kernels of the LoRDO hot path: clip norm, low-rank moment update,
// outer synchronisation, sketch generator. All grouped over the whole list of matrices.
#include "lordo_kernels.h"

namespace lordo {

// ---------------------------------------------------------------------------------------------
// Clip coefficient (Algorithm 1, line "clip"): c = min(1, rho / (||G_k||_2 + 1e-6))
// One block per `chunk` elements writes a partial sum of squares; the last block of a (matrix, worker) to
// finish adds that pair's partial sums, the last pair of a worker the matrices' sums, both in a fixed order
// whichever block it is. Bound by HBM (7 TB/s on 14 layers of 2048); with the two sums as kernels of their own a small
// step spent 8 us more on launches, and 256 x 256 with chunks of 32768 had four blocks (step 40.0 -> 34.6 us).
// The sums of a block meet by shuffles and one barrier (as a tree of nine barriers: 256 x 256 step 20.8 us, now 20.5).
// ---------------------------------------------------------------------------------------------
// All threads return the sum of x, always in the same order; `red` is not used again before a barrier.
__device__ __forceinline__ double block_sum_256(double x, double* red) {
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  double s = 0.0;
#pragma unroll
  for (int w = 0; w < 8; ++w) s += red[w];
  return s;
}

template <bool BF16>
__global__ void __launch_bounds__(256) clip_kernel(const MatDev* __restrict__ mats, const void* const* __restrict__ G,
                                                   const long long* __restrict__ chunk_start, int n_mats, int K, long long chunk, double* partial,
                                                   float rho, int scope, float* __restrict__ coef, double* sumsq, unsigned* __restrict__ tickets,
                                                   unsigned* __restrict__ status) {
  __shared__ double red[3][8];
  __shared__ bool last_s;
  const int t = threadIdx.x;
  const long long blk = blockIdx.x;
  const int i = find_segment(chunk_start, n_mats, blk);  // the tables are constant
  const long long elems = mats[i].m * mats[i].n;
  dep_begin();
  const unsigned chunks = (unsigned)((elems + chunk - 1) / chunk);
  const unsigned local = (unsigned)(blk - chunk_start[i]);
  const int k = (int)(local / chunks);
  const long long begin = (long long)(local - (unsigned)k * chunks) * chunk;
  const long long end = begin + chunk < elems ? begin + chunk : elems;
  constexpr int kBytes = BF16 ? 2 : 4;
  const char* g = reinterpret_cast<const char*>(G[i]) + (long long)k * elems * kBytes;
  float sum[4] = {0.f, 0.f, 0.f, 0.f};  // of at most 128 squares each
  for (long long e = begin + 8ll * t; e < end; e += 4 * 8 * 256) {  // elems is a multiple of 8
    uint4 x[4][BF16 ? 1 : 2];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long at = e + u * 8 * 256;
#pragma unroll
      for (int h = 0; h < (BF16 ? 1 : 2); ++h)
        x[u][h] = at < end ? reinterpret_cast<const uint4*>(g + at * kBytes)[h] : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int h = 0; h < (BF16 ? 1 : 2); ++h) {
        const uint32_t w[4] = {x[u][h].x, x[u][h].y, x[u][h].z, x[u][h].w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (BF16) {
            const float lo = __uint_as_float(w[j] << 16), hi = __uint_as_float(w[j] & 0xFFFF0000u);
            sum[u] += lo * lo + hi * hi;
          } else {
            const float v = __uint_as_float(w[j]);
            sum[u] += v * v;
          }
        }
      }
  }
  const double s = block_sum_256(((double)sum[0] + (double)sum[1]) + ((double)sum[2] + (double)sum[3]), red[0]);
  if (t == 0) {
    partial[blk] = s;
    __threadfence();
    last_s = atomicInc(tickets + (long long)i * K + k, chunks - 1) == chunks - 1;  // back to zero with the last block
  }
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  const double* p = partial + chunk_start[i] + (long long)k * chunks;
  double a = 0.0;
  for (unsigned c = t; c < chunks; c += 256) a += __ldcg(p + c);  // written by other SMs meanwhile: not from this one's L1
  const double s_i = block_sum_256(a, red[1]);
  if (t == 0) {
    sumsq[(long long)i * K + k] = s_i;
    if (scope == 1) coef[(long long)i * K + k] = fminf(1.f, rho / ((float)sqrt(s_i) + 1e-6f));
    __threadfence();
    last_s = atomicInc(tickets + (long long)n_mats * K + k, (unsigned)n_mats - 1) == (unsigned)n_mats - 1;
  }
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  a = 0.0;
  for (int m = t; m < n_mats; m += 256) a += __ldcg(sumsq + (long long)m * K + k);
  const double total = block_sum_256(a, red[2]);
  if (t == 0 && !isfinite(total)) atomicOr(status, LORDO_FLAG_NONFINITE_GRAD);
  const float c = fminf(1.f, rho / ((float)sqrt(total) + 1e-6f));
  if (scope == 0)
    for (int m = t; m < n_mats; m += 256) coef[(long long)m * K + k] = c;
}

__global__ void fill_float_kernel(float* __restrict__ p, long long count, float value) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) p[i] = value;
}

// ---------------------------------------------------------------------------------------------
// Low-rank moment update (Algorithm 1: u, v lines and the bracket of the update cases).
//   u <- b1 u + (1-b1) g ; v <- b2 v + (1-b2) g*g ; u^ = u/(1-b1^s) ; v^ = v/(1-b2^s)
//   D = sqrt(v^) + eps ; U~ = u^/D (no / full-rank QHM) or (w u^ + (1-w) g)/D (low-rank QHM)
//   full-rank QHM also needs mu(D) = mean over the rank axis, one value per column.
// One block = kMomCols columns of one (matrix, replica), eight lanes across and 32 rows of ranks down: bound by latency
// at the sizes of check mode (a rank's loads, square root and division take about a microsecond), so a thread has few ranks
// and a full line per row of a block is all the width that the loads need. With 128 columns a block three ragged
// matrices with three workers (r up to 136) took 20 us, now 9; 256 columns, r = 16, two workers 5.3, now 4.5 us.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) moments_kernel(const MatDev* __restrict__ mats, const long long* __restrict__ tile_start,
                                                      int n_mats, StepScalars sc) {
  constexpr int LANES = kMomCols / 4, ROWS = 256 / LANES;
  const int lane = threadIdx.x % LANES, row = threadIdx.x / LANES;
  const long long blk = blockIdx.x;
  const int i = find_segment(tile_start, n_mats, blk);  // the tables are constant
  const MatDev md = mats[i];
  dep_begin();
  const long long n = md.ln;  // columns of the low-rank arrays
  const int r = md.r;
  const long long ctiles = (n + kMomCols - 1) / kMomCols;
  const long long local = blk - tile_start[i];
  const int k = (int)(local / ctiles);
  const long long col = (local - (long long)k * ctiles) * kMomCols + 4ll * lane;
  const bool active = col < n;
  const long long base = (long long)k * r * n + col;
  const float b1 = sc.beta1, b2 = sc.beta2, w = sc.omega;
  float dsum0 = 0.f, dsum1 = 0.f, dsum2 = 0.f, dsum3 = 0.f;
  if (active) {
#pragma unroll 2
    for (int a = row; a < r; a += ROWS) {
      const long long idx = base + (long long)a * n;
      const float4 g = *reinterpret_cast<const float4*>(md.ghat + idx);
      float4 u = *reinterpret_cast<const float4*>(md.u + idx);
      float4 v = *reinterpret_cast<const float4*>(md.v + idx);
      float4 o;
#define LORDO_MOM(c)                                                              \
  {                                                                               \
    u.c = b1 * u.c + (1.f - b1) * g.c;                                            \
    v.c = b2 * v.c + (1.f - b2) * g.c * g.c;                                      \
    const float uh = u.c * sc.inv_bc1;                                            \
    const float D = sqrtf(v.c * sc.inv_bc2) + sc.eps;                             \
    o.c = (sc.form == LORDO_QHM_LOW) ? (w * uh + (1.f - w) * g.c) / D : uh / D;   \
    dsum_##c += D;                                                                \
  }
      float dsum_x = 0.f, dsum_y = 0.f, dsum_z = 0.f, dsum_w = 0.f;
      LORDO_MOM(x) LORDO_MOM(y) LORDO_MOM(z) LORDO_MOM(w)
#undef LORDO_MOM
      dsum0 += dsum_x; dsum1 += dsum_y; dsum2 += dsum_z; dsum3 += dsum_w;
      *reinterpret_cast<float4*>(md.u + idx) = u;
      *reinterpret_cast<float4*>(md.v + idx) = v;
      *reinterpret_cast<float4*>(md.util + idx) = o;
      if (md.T) {  // up-link time buffer
        float4 tb = *reinterpret_cast<const float4*>(md.T + idx);
        tb.x += sc.lr * o.x; tb.y += sc.lr * o.y; tb.z += sc.lr * o.z; tb.w += sc.lr * o.w;
        *reinterpret_cast<float4*>(md.T + idx) = tb;
      }
    }
  }
  if (sc.form == LORDO_QHM_FULL) {  // uniform over the grid
    // the four rows of a warp, then the warps, in a fixed order
    __shared__ float4 red[8][LANES];
    float4 s = make_float4(dsum0, dsum1, dsum2, dsum3);
#pragma unroll
    for (int o = LANES; o < 32; o <<= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, o); s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
      s.z += __shfl_xor_sync(0xffffffffu, s.z, o); s.w += __shfl_xor_sync(0xffffffffu, s.w, o);
    }
    if ((threadIdx.x & 31) < LANES) red[threadIdx.x >> 5][lane] = s;
    __syncthreads();
    if (row == 0 && active) {
      s = red[0][lane];
#pragma unroll
      for (int y = 1; y < 8; ++y) {
        const float4 t = red[y][lane];
        s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
      }
      const float inv_r = 1.f / (float)r;
      s.x *= inv_r; s.y *= inv_r; s.z *= inv_r; s.w *= inv_r;
      *reinterpret_cast<float4*>(md.dcol + (long long)k * n + col) = s;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Outer synchronisation (Algorithm 1, synchronisation lines; appendix "Unrolled low-rank
// updates": Delta = old - new, theta <- theta - eta_s Delta).
// One thread = 4 consecutive weights of one matrix, all K replicas.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) outer_weights_kernel(const MatDev* __restrict__ mats, const long long* __restrict__ blk_start,
                                                            int n_mats, int K, int w_dt, int outer, float eta_s, float mu_s,
                                                            float delta_scale) {
  dep_begin();
  const long long blk = blockIdx.x;
  const int i = find_segment(blk_start, n_mats, blk);
  const MatDev md = mats[i];
  const long long elems = md.m * md.n;
  const long long e = ((blk - blk_start[i]) * 256 + threadIdx.x) * 4;
  if (e >= elems) return;
  const float4 x0 = *reinterpret_cast<const float4*>(md.X0 + e);
  float4 d, xn;
  if (delta_scale != 0.f) {  // the pseudo-gradient was rebuilt from the time buffers into Delta
    d = *reinterpret_cast<const float4*>(md.Delta + e);
    d.x *= delta_scale; d.y *= delta_scale; d.z *= delta_scale; d.w *= delta_scale;
  } else {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
      const float4 w = load4(md.W, w_dt, (long long)k * elems + e);
      s.x += w.x; s.y += w.y; s.z += w.z; s.w += w.w;
    }
    const float inv_k = 1.f / (float)K;
    d.x = x0.x - s.x * inv_k; d.y = x0.y - s.y * inv_k; d.z = x0.z - s.z * inv_k; d.w = x0.w - s.w * inv_k;
  }
  if (outer == LORDO_OUTER_NESTEROV) {
    float4 b = *reinterpret_cast<const float4*>(md.B + e);
    b.x = mu_s * b.x + d.x; b.y = mu_s * b.y + d.y; b.z = mu_s * b.z + d.z; b.w = mu_s * b.w + d.w;
    *reinterpret_cast<float4*>(md.B + e) = b;
    xn.x = x0.x - eta_s * (d.x + mu_s * b.x); xn.y = x0.y - eta_s * (d.y + mu_s * b.y);
    xn.z = x0.z - eta_s * (d.z + mu_s * b.z); xn.w = x0.w - eta_s * (d.w + mu_s * b.w);
  } else {
    xn.x = x0.x - d.x; xn.y = x0.y - d.y; xn.z = x0.z - d.z; xn.w = x0.w - d.w;
  }
  *reinterpret_cast<float4*>(md.Delta + e) = d;
  *reinterpret_cast<float4*>(md.X0 + e) = xn;
#pragma unroll 4
  for (int k = 0; k < K; ++k) store4(md.W, w_dt, (long long)k * elems + e, xn);
}

// u, v <- mean over replicas (Algorithm 1, "Sync u / v" lines). which: bit 0 = u, bit 1 = v,
// bit 2 = the time buffers (Global rule: one basis, so their mean is all the rebuilt pseudo-gradient needs).
__global__ void __launch_bounds__(256) outer_states_kernel(const MatDev* __restrict__ mats, const long long* __restrict__ blk_start,
                                                           int n_mats, int K, int which) {
  dep_begin();
  const long long blk = blockIdx.x;
  const int i = find_segment(blk_start, n_mats, blk);
  const MatDev md = mats[i];
  const long long elems = (long long)md.r * md.ln;
  const long long e = ((blk - blk_start[i]) * 256 + threadIdx.x) * 4;
  if (e >= elems) return;
  const float inv_k = 1.f / (float)K;
  for (int t = 0; t < 3; ++t) {
    if (!((which >> t) & 1)) continue;
    float* p = t == 0 ? md.u : (t == 1 ? md.v : md.T);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
      const float4 x = *reinterpret_cast<const float4*>(p + (long long)k * elems + e);
      s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
    }
    s.x *= inv_k; s.y *= inv_k; s.z *= inv_k; s.w *= inv_k;
#pragma unroll 4
    for (int k = 0; k < K; ++k) *reinterpret_cast<float4*>(p + (long long)k * elems + e) = s;
  }
}

// ---------------------------------------------------------------------------------------------
// init helpers
// ---------------------------------------------------------------------------------------------
// Copies W[0] to replicas 1..K-1 and to X0 (fp32).
__global__ void __launch_bounds__(256) init_weights_kernel(const MatDev* __restrict__ mats, const long long* __restrict__ blk_start,
                                                           int n_mats, int K, int w_dt) {
  const long long blk = blockIdx.x;
  const int i = find_segment(blk_start, n_mats, blk);
  const MatDev md = mats[i];
  const long long elems = md.m * md.n;
  const long long e = ((blk - blk_start[i]) * 256 + threadIdx.x) * 4;
  if (e >= elems) return;
  const float4 w = load4(md.W, w_dt, e);
  *reinterpret_cast<float4*>(md.X0 + e) = w;
  for (int k = 1; k < K; ++k) store4(md.W, w_dt, (long long)k * elems + e, w);
}

__global__ void identity_projection_kernel(float* __restrict__ P, long long m, int r, int copies) {
  const long long total = m * r * copies;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= total) return;
  const long long within = idx % (m * r);
  const long long row = within / r;
  const int col = (int)(within - row * r);
  P[idx] = (row == col) ? 1.f : 0.f;
}

// out[c] = popcount(mix64(key + golden*(c+1))) - 32 ; batch entry b uses keys[b].
__global__ void __launch_bounds__(256) fill_random_kernel(float* __restrict__ out, long long count, long long batch_stride,
                                                          RandomKeys keys) {
  const long long c = (long long)blockIdx.x * 256 + threadIdx.x;
  if (c >= count) return;
  const unsigned long long w = mix64(keys.key[blockIdx.y] + kGolden * (unsigned long long)(c + 1));
  out[(long long)blockIdx.y * batch_stride + c] = (float)(__popcll(w) - 32);
}

// The same generator for many matrices in one launch; the key of each is derived on the device.
// Bound by integer instructions: about 27 an entry, nearly all of them the two 64-bit products and three shifts of the mixer.
// So the key (five more of them) is derived once per block and not once per thread, and neither the float nor its
// bf16 bits come from a conversion, which like popc issue at an eighth of the rate: an integer below 2^22 added to the bits of
// 2^23 is a float, and the high half of a float that is an integer in [-32, 32] is its bf16.
// 90 million entries (16 workers, 11008 x 512) 197 -> 131 us, 7 matrices of 768 with 8 workers 26.7 -> 20.3 us.
__global__ void __launch_bounds__(256) fill_random_grouped_kernel(const RandProblem* __restrict__ probs, int nprobs,
                                                                  unsigned long long seed, long long index) {
  __shared__ unsigned long long s_key;
  __shared__ int s_prob;
  const long long blk = blockIdx.x;
  if (threadIdx.x == 0) {  // the table is constant
    int lo = 0, hi = nprobs - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (probs[mid].blk_start <= blk) lo = mid; else hi = mid - 1;
    }
    s_prob = lo;
    s_key = stream_key(seed, probs[lo].purpose, probs[lo].mat, index, probs[lo].replica);
  }
  __syncthreads();
  const RandProblem pb = probs[s_prob];
  const long long c0 = ((blk - pb.blk_start) * 256 + threadIdx.x) * 8;  // eight consecutive entries per thread (count is a multiple of 8)
  const unsigned long long x0 = s_key + kGolden * (unsigned long long)(c0 + 1);
  float val[8];
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const unsigned long long w = mix64(x0 + kGolden * (unsigned long long)x);
    val[x] = __int_as_float(0x4B000000 + __popc((unsigned)w) + __popc((unsigned)(w >> 32))) - 8388640.f;
  }
  dep_begin();
  if (c0 >= pb.count) return;
  if (pb.out) {
    *reinterpret_cast<float4*>(pb.out + c0) = make_float4(val[0], val[1], val[2], val[3]);
    *reinterpret_cast<float4*>(pb.out + c0 + 4) = make_float4(val[4], val[5], val[6], val[7]);
  }
  if (pb.out16) {
    unsigned h[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) h[x] = __byte_perm(__float_as_uint(val[2 * x]), __float_as_uint(val[2 * x + 1]), 0x7632);
    *reinterpret_cast<uint4*>(pb.out16 + c0) = make_uint4(h[0], h[1], h[2], h[3]);
  }
}

__device__ __forceinline__ void split_store4(__nv_bfloat16* dst, long long plane, int planes, long long e, float4 v) {
  for (int p = 0; p < planes; ++p) {
    const float4 h = make_float4(__bfloat162float(__float2bfloat16_rn(v.x)), __bfloat162float(__float2bfloat16_rn(v.y)),
                                 __bfloat162float(__float2bfloat16_rn(v.z)), __bfloat162float(__float2bfloat16_rn(v.w)));
    store4(dst + p * plane, LORDO_BF16, e, h);
    v = make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w);  // exact: the residual of a rounding to 8 bits
  }
}

// Four vectors per thread in flight: 7 matrices of 2048 (51 million elements) 84 -> 40 us.
__global__ void __launch_bounds__(256) convert_grouped_kernel(const ConvProblem* __restrict__ probs, int nprobs) {
  const long long blk = blockIdx.x;
  int lo = 0, hi = nprobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].blk_start <= blk) lo = mid; else hi = mid - 1;
  }
  const ConvProblem pb = probs[lo];
  dep_begin();  // the tables are constant
  const long long e = (blk - pb.blk_start) * 4096 + threadIdx.x * 4;
  float4 v[4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (e + i * 1024 < pb.count) v[i] = *reinterpret_cast<const float4*>(pb.src + e + i * 1024);
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (e + i * 1024 < pb.count) store4(pb.dst, LORDO_BF16, e + i * 1024, v[i]);
}

// One block per 32 x 32 block on or below the diagonal, which it also mirrors; the partial products meet in
// fp64, so that what is left of the tensor cores' truncating accumulation is that of one range of k. The mirrored
// block of T is summed as it lies and turned over once, in fp64, so the ranges' loads wait for nothing.
// Bound by the reads of the partial products: 56 matrices of r = 128 14.5 -> 10.5 us, 7 of r = 256 20 -> 12.6 us, six launches
// over 16 matrices of r = 512 283 -> 246 us, against two barriers a range
__global__ void __launch_bounds__(256) gram_sum_kernel(const GramProblem* __restrict__ probs, int nprobs) {
  __shared__ double tt[32][33];
  const long long blk = blockIdx.x;
  int lo = 0, hi = nprobs - 1;
  while (lo < hi) {  // the tables are constant
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].blk_start <= blk) lo = mid; else hi = mid - 1;
  }
  const GramProblem pb = probs[lo];
  const int r = pb.r;
  const size_t rr = (size_t)r * r;
  int bi = 0, rest = (int)(blk - pb.blk_start);
  while (rest > bi) rest -= ++bi;  // block row bi has bi + 1 blocks
  const int bj = rest;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  double acc[4] = {0.0, 0.0, 0.0, 0.0}, mir[4] = {0.0, 0.0, 0.0, 0.0};
  size_t at[4], am[4];  // elements outside the matrix: its first one, summed and not used
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = bi * 32 + y + 8 * q, j = bj * 32 + x, i2 = bj * 32 + y + 8 * q, j2 = bi * 32 + x;
    at[q] = i < r && j < r ? (size_t)i * r + j : 0;
    am[q] = i2 < r && j2 < r ? (size_t)i2 * r + j2 : 0;
  }
  dep_begin();
#pragma unroll 2
  for (int s = 0; s < pb.ns; ++s) {
    const float* S = pb.part + s * rr;
    const float* T = pb.part + (pb.ns + s) * rr;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      acc[q] += (double)S[at[q]] + (double)T[at[q]];
      mir[q] += (double)T[am[q]];
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) tt[y + 8 * q][x] = mir[q];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) acc[q] += tt[x][y + 8 * q];
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = bi * 32 + y + 8 * q, j = bj * 32 + x;
    tt[y + 8 * q][x] = acc[q];
    if (i < r && j < r && (bi != bj || j <= i)) pb.gram[(size_t)i * r + j] = (float)acc[q];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = bj * 32 + y + 8 * q, j = bi * 32 + x;
    if (i < r && j < r && (bi != bj || j > i)) pb.gram[(size_t)i * r + j] = (float)tt[x][y + 8 * q];
  }
}

// One block per 32 x 32 block of Rot, whose transpose it writes. Sixteen loads of a thread are in
// flight: 7 matrices of r = 256 22.7 us with one row after the other, now 12.7.
__global__ void __launch_bounds__(256) rot_sum_kernel(const RotProblem* __restrict__ probs, int nprobs) {
  __shared__ float tt[32][33];
  const long long blk = blockIdx.x;
  int lo = 0, hi = nprobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].blk_start <= blk) lo = mid; else hi = mid - 1;
  }
  const RotProblem pb = probs[lo];
  const int r = pb.r, nb = (r + 31) / 32;
  const int bi = (int)(blk - pb.blk_start) / nb, bj = (int)(blk - pb.blk_start) - bi * nb;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  double a[4] = {0.0, 0.0, 0.0, 0.0};
  size_t at[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = bi * 32 + y + 8 * q, j = bj * 32 + x;
    at[q] = i < r && j < r ? (size_t)i * r + j : 0;
  }
  dep_begin();
#pragma unroll 4
  for (int s = 0; s < pb.ns; ++s) {
#pragma unroll
    for (int q = 0; q < 4; ++q) a[q] += (double)pb.part[(size_t)s * r * r + at[q]];
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (bi * 32 + y + 8 * q < r && bj * 32 + x < r) pb.rot[at[q]] = (float)a[q];
    tt[y + 8 * q][x] = (float)a[q];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 256; e += 256) {  // four neighbouring elements of a row of Rot^T per thread
    const int i = bj * 32 + (e >> 3), j = bi * 32 + (e & 7) * 4;
    if (i < r && j < r) {  // r is a multiple of 8
      const int c = e >> 3, k = (e & 7) * 4;
      const float4 t = make_float4(tt[k][c], tt[k + 1][c], tt[k + 2][c], tt[k + 3][c]);
      const long long at = (long long)i * r + j;
      split_store4(pb.rt16, pb.plane, 2, at, t);
      split_store4(pb.sq16, pb.plane, 2, at, make_float4(t.x * t.x, t.y * t.y, t.z * t.z, t.w * t.w));
    }
  }
}

// Sums of squares of 128 columns over kNormRows rows, in fp64. One block per 32 columns over all rows took 346 us
// for 7 matrices of up to 5632 x 256 (and 400 us for 16 of 4096 x 512).
__global__ void __launch_bounds__(256) colsq_kernel(const BasisProblem* __restrict__ probs, int nprobs) {
  __shared__ double red[8][128];
  const long long blk = blockIdx.x;
  int lo = 0, hi = nprobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].sq_start <= blk) lo = mid; else hi = mid - 1;
  }
  const BasisProblem pb = probs[lo];
  const int nc = (pb.r + 127) / 128;
  dep_begin();  // the tables are constant
  const long long chunk = (blk - pb.sq_start) / nc;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c0 = (int)(blk - pb.sq_start - chunk * nc) * 128;
  const int col = c0 + 4 * lane;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  if (col < pb.r) {
    const long long end = min((long long)pb.m, (chunk + 1) * kNormRows);
#pragma unroll 4
    for (long long row = chunk * kNormRows + w; row < end; row += 8) {
      const float4 v = *reinterpret_cast<const float4*>(pb.Q + row * pb.r + col);
      s[0] += (double)v.x * (double)v.x; s[1] += (double)v.y * (double)v.y;
      s[2] += (double)v.z * (double)v.z; s[3] += (double)v.w * (double)v.w;
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) red[w][4 * lane + i] = s[i];
  __syncthreads();
  if (threadIdx.x < 128 && c0 + threadIdx.x < pb.r) {
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += red[k][threadIdx.x];
    pb.sq[chunk * pb.r + c0 + threadIdx.x] = t;
  }
}

__global__ void __launch_bounds__(256) commit_basis_kernel(const BasisProblem* __restrict__ probs, int nprobs) {
  dep_begin();
  __shared__ __nv_bfloat16 tile[64][66];
  __shared__ float scale[64];
  __shared__ double part[4][64];
  const long long blk = blockIdx.x;
  int lo = 0, hi = nprobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].tile_start <= blk) lo = mid; else hi = mid - 1;
  }
  const BasisProblem pb = probs[lo];
  const int r = pb.r, nc = (r + 63) / 64;
  const long long row0 = (blk - pb.tile_start) / nc * 64;
  const int col0 = (int)((blk - pb.tile_start) % nc) * 64;
  const int t = threadIdx.x;
  float4 q[4], p[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int rr = (t >> 4) + 16 * i, cc = (t & 15) * 4;
    q[i] = p[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row0 + rr < pb.m && col0 + cc < r) {
      const long long at = (row0 + rr) * r + col0 + cc;
      q[i] = *reinterpret_cast<const float4*>(pb.Q + at);
      p[i] = *reinterpret_cast<const float4*>(pb.P + at);
    }
  }
  {
    const int c = t & 63, w = t >> 6;
    double s = 0.0;
    if (col0 + c < r) {
      const int chunks = (int)((pb.m + kNormRows - 1) / kNormRows);
      for (int k = w; k < chunks; k += 4) s += pb.sq[(long long)k * r + col0 + c];
    }
    part[w][c] = s;
  }
  __syncthreads();
  if (t < 64) {
    const double s = (part[0][t] + part[1][t]) + (part[2][t] + part[3][t]);
    scale[t] = (float)(s > 0.0 ? 1.0 / sqrt(s) : 1.0);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int rr = (t >> 4) + 16 * i, cc = (t & 15) * 4;
    if (row0 + rr < pb.m && col0 + cc < r) {
      const long long at = (row0 + rr) * r + col0 + cc;
      const float4 n = make_float4(q[i].x * scale[cc], q[i].y * scale[cc + 1], q[i].z * scale[cc + 2], q[i].w * scale[cc + 3]);
      *reinterpret_cast<float4*>(pb.P + at) = n;
      split_store4(pb.q16, pb.q_plane, 2, at, n);
      split_store4(pb.p16, pb.p_plane, 2, at, p[i]);
      store4(pb.P16, LORDO_BF16, (row0 + rr) * pb.r_k + col0 + cc, n);
      tile[rr][cc] = __float2bfloat16_rn(n.x); tile[rr][cc + 1] = __float2bfloat16_rn(n.y);
      tile[rr][cc + 2] = __float2bfloat16_rn(n.z); tile[rr][cc + 3] = __float2bfloat16_rn(n.w);
    }
  }
  __syncthreads();
  for (int e = t; e < 64 * 64; e += 256) {
    const int cc = e >> 6, rr = e & 63;
    if (row0 + rr < pb.m && col0 + cc < r) pb.PT16[(long long)(col0 + cc) * pb.m_k + row0 + rr] = tile[rr][cc];
  }
}

// Device-to-device copies of many buffers in one launch (16-byte chunks).
__global__ void __launch_bounds__(256) copy_grouped_kernel(const CopyProblem* __restrict__ probs, int nprobs) {
  const long long blk = blockIdx.x;
  int lo = 0, hi = nprobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (probs[mid].blk_start <= blk) lo = mid; else hi = mid - 1;
  }
  const CopyProblem pb = probs[lo];
  dep_begin();  // the tables are constant
  const long long c = ((blk - pb.blk_start) * 256 + threadIdx.x) * 4;
  const uint4* __restrict__ src = reinterpret_cast<const uint4*>(pb.src);
  uint4* __restrict__ dst = reinterpret_cast<uint4*>(pb.dst);
  uint4 v[4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (c + i < pb.chunks) v[i] = src[c + i];
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (c + i < pb.chunks) dst[c + i] = v[i];
}

// Mean squared singular value of Rot = P'^T P (the paper's MSSV metric): the sum of the squared
// singular values of a matrix is its squared Frobenius norm. One block per rotation matrix.
__global__ void __launch_bounds__(256) mssv_kernel(const DiagProblem* __restrict__ probs, float* __restrict__ out) {
  const DiagProblem pb = probs[blockIdx.x];
  const long long count = (long long)pb.r * pb.r;
  double a = 0.0;
  for (long long e = threadIdx.x; e < count; e += 256) { const double x = (double)pb.rot[e]; a += x * x; }
  __shared__ double red[256];
  red[threadIdx.x] = a;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = (float)(red[0] / (double)pb.r);
}

// ||E||_F of one (matrix, worker) per block.
__global__ void __launch_bounds__(256) error_norms_kernel(const MatDev* __restrict__ mats, int K, int e_dt, float* __restrict__ out) {
  const int i = blockIdx.x, k = blockIdx.y;
  const long long elems = mats[i].m * mats[i].n;
  const void* E = mats[i].E;
  double a = 0.0;
  for (long long e = 4ll * threadIdx.x; e < elems; e += 4ll * 256) {  // elems is a multiple of 8
    const float4 x = load4(E, e_dt, (long long)k * elems + e);
    a += (double)(x.x * x.x + x.y * x.y) + (double)(x.z * x.z + x.w * x.w);
  }
  __shared__ double red[256];
  red[threadIdx.x] = a;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[(long long)i * K + k] = (float)sqrt(red[0]);
}

// ---------------------------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------------------------
void launch_mssv(const DiagProblem* probs, int nprobs, float* out, cudaStream_t st) { mssv_kernel<<<nprobs, 256, 0, st>>>(probs, out); }
void launch_error_norms(const MatDev* mats, int n_mats, int K, int e_dt, float* out, cudaStream_t st) {
  error_norms_kernel<<<dim3(n_mats, K), 256, 0, st>>>(mats, K, e_dt, out);
}
void launch_fill_random_grouped(const RandProblem* probs, int nprobs, long long total_blocks, unsigned long long seed, long long index,
                                cudaStream_t st) {
  launch_dep(fill_random_grouped_kernel, dim3((unsigned)total_blocks), 256, 0, st, probs, nprobs, seed, index);
}
void launch_convert_grouped(const ConvProblem* probs, int nprobs, long long total_blocks, cudaStream_t st) {
  launch_dep(convert_grouped_kernel, dim3((unsigned)total_blocks), 256, 0, st, probs, nprobs);
}
void launch_gram_sum(const GramProblem* probs, int nprobs, long long total_blocks, cudaStream_t st) {
  launch_dep(gram_sum_kernel, dim3((unsigned)total_blocks), 256, 0, st, probs, nprobs);
}
void launch_rot_sum(const RotProblem* probs, int nprobs, long long total_blocks, cudaStream_t st) {
  launch_dep(rot_sum_kernel, dim3((unsigned)total_blocks), 256, 0, st, probs, nprobs);
}
void launch_colsq(const BasisProblem* probs, int nprobs, long long total_blocks, cudaStream_t st) {
  launch_dep(colsq_kernel, dim3((unsigned)total_blocks), 256, 0, st, probs, nprobs);
}
void launch_commit_basis(const BasisProblem* probs, int nprobs, long long total_blocks, cudaStream_t st) {
  launch_dep(commit_basis_kernel, dim3((unsigned)total_blocks), 256, 0, st, probs, nprobs);
}
void launch_copy_grouped(const CopyProblem* probs, int nprobs, long long total_blocks, cudaStream_t st) {
  launch_dep(copy_grouped_kernel, dim3((unsigned)total_blocks), 256, 0, st, probs, nprobs);
}
void launch_clip(const MatDev* mats, const void* const* G, const long long* chunk_start, int n_mats, int K, int g_dt, long long chunk,
                 double* partial, long long total_chunks, float rho, int scope, float* coef, double* sumsq, unsigned* tickets, unsigned* status,
                 cudaStream_t st) {
  if (g_dt == LORDO_BF16)
    launch_dep(clip_kernel<true>, dim3((unsigned)total_chunks), 256, 0, st, mats, G, chunk_start, n_mats, K, chunk, partial, rho, scope, coef, sumsq, tickets, status);
  else
    launch_dep(clip_kernel<false>, dim3((unsigned)total_chunks), 256, 0, st, mats, G, chunk_start, n_mats, K, chunk, partial, rho, scope, coef, sumsq, tickets, status);
}
void launch_fill_float(float* p, long long count, float value, cudaStream_t st) {
  fill_float_kernel<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(p, count, value);
}
void launch_moments(const MatDev* mats, const long long* tile_start, int n_mats, long long total_tiles, const StepScalars& sc,
                    cudaStream_t st) {
  launch_dep(moments_kernel, dim3((unsigned)total_tiles), 256, 0, st, mats, tile_start, n_mats, sc);
}
void launch_outer_weights(const MatDev* mats, const long long* blk_start, int n_mats, long long total_blocks, int K, int w_dt,
                          int outer, float eta_s, float mu_s, float delta_scale, cudaStream_t st) {
  launch_dep(outer_weights_kernel, dim3((unsigned)total_blocks), 256, 0, st, mats, blk_start, n_mats, K, w_dt, outer, eta_s, mu_s, delta_scale);
}
void launch_outer_states(const MatDev* mats, const long long* blk_start, int n_mats, long long total_blocks, int K, int which,
                         cudaStream_t st) {
  launch_dep(outer_states_kernel, dim3((unsigned)total_blocks), 256, 0, st, mats, blk_start, n_mats, K, which);
}
void launch_init_weights(const MatDev* mats, const long long* blk_start, int n_mats, long long total_blocks, int K, int w_dt,
                         cudaStream_t st) {
  init_weights_kernel<<<(unsigned)total_blocks, 256, 0, st>>>(mats, blk_start, n_mats, K, w_dt);
}
void launch_identity_projection(float* P, long long m, int r, int copies, cudaStream_t st) {
  const long long total = m * r * copies;
  identity_projection_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(P, m, r, copies);
}
void launch_fill_random(float* out, long long count, long long batch_stride, const RandomKeys& keys, int batch, cudaStream_t st) {
  fill_random_kernel<<<dim3((unsigned)((count + 255) / 256), batch), 256, 0, st>>>(out, count, batch_stride, keys);
}

}  // namespace lordo
