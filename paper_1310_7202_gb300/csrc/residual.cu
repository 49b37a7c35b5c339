// Error of Eq. (1) / Eq. (relErr): R = P A Q - L U.
//   ||R||_F: a tiled L*U product accumulated in FP64 with the residual and its square formed
//            in the epilogue (A read through the P/Q gathers); per-CTA partial sums are added
//            in a fixed order.
//   ||R||_2: power iteration x <- R^T R x / ||R^T R x|| from a fixed start vector, with R
//            applied as two skinny products per half-step (P A Q x - L (U x), and its
//            transpose), every reduction in FP64 and in a fixed order.
//
// FP64 multiply-adds and conversions run at 1/64 of the FP32 rate and bound all three passes
// over the m x n elements (||R||_F at 8192^2, k = 200: 23.7 ms, the two halves of an iteration
// 0.27 + 0.26 ms). With FP32 or BF16 A and FP32 factors these passes therefore use exact FP32
// arithmetic: an FP32 product is the sum of two floats (a multiply and a fused multiply-add),
// an FP64 vector entry the sum of three, and sums are kept as three floats, the first two with
// the exact rounding error of every addition carried down (Knuth's two-sum), so that nothing
// above 2^-70 or so of the terms is dropped, where FP64 rounds every addition at 2^-53. It
// holds while no term leaves the FP32 range; k_range looks for the largest magnitudes of A, L
// and U first. Where one is outside [2^-20, 2^40] (also for Inf, NaN and all-zero operands), or
// where by them A times y = (PAQ - LU) x, ||x|| = 1, could pass 2^126 in a sum over a chunk of
// rows (y is not known beforehand), the passes take their FP64 form.
#include "common.cuh"
#include "residual.cuh"

namespace rlu {

static constexpr int RS_RB = 64;  // row blocks of the transposed product

template <typename T> __device__ __forceinline__ double to_d(T v) { return (double)v; }
template <> __device__ __forceinline__ double to_d<__nv_bfloat16>(__nv_bfloat16 v) {
  return (double)__bfloat162float(v);
}

// a + b = s + e exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
struct Acc3 {  // s1 + s2 + s3
  float s1, s2, s3;
  // + a b
  __device__ __forceinline__ void mac(float a, float b) {
    const float p = __fmul_rn(a, b), e = __fmaf_rn(a, b, -p);
    float r, t, r1, r2;
    two_sum(s1, p, s1, r);
    two_sum(e, r, t, r1);
    two_sum(s2, t, s2, r2);
    s3 = __fadd_rn(s3, __fadd_rn(r1, r2));
  }
  // + a (b1 + b2 + b3), the b's parts of one FP64 value
  __device__ __forceinline__ void mac(float a, float b1, float b2, float b3) {
    const float p = __fmul_rn(a, b1), e = __fmaf_rn(a, b1, -p);
    const float q = __fmul_rn(a, b2), f = __fmaf_rn(a, b2, -q);
    float r, t, r1, r2, r3;
    two_sum(s1, p, s1, r);
    two_sum(e, q, t, r1);
    two_sum(t, r, t, r2);
    two_sum(s2, t, s2, r3);
    s3 = __fadd_rn(s3, __fadd_rn(__fmaf_rn(a, b3, f), __fadd_rn(__fadd_rn(r1, r2), r3)));
  }
  __device__ __forceinline__ double value() const {
    return (double)s1 + ((double)s2 + (double)s3);
  }
};
__device__ __forceinline__ void split3(double x, float& x1, float& x2, float& x3) {
  x1 = (float)x;
  const double r = x - (double)x1;
  x2 = (float)r;
  x3 = (float)(r - (double)x2);
}
template <typename T> __device__ __forceinline__ float to_f(T v) { return (float)v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}
// Whether the types have the FP32 form, and whether the operands' magnitudes (k_range) do.
template <typename TA, typename TLU> __host__ __device__ constexpr bool has_f32() {
  return sizeof(TA) <= 4 && sizeof(TLU) == 4;
}
__device__ __forceinline__ bool in_range(const uint32_t* mx) {
  bool ok = true;
#pragma unroll
  for (int i = 0; i < 3; ++i) ok &= mx[i] >= 0x35800000u && mx[i] <= 0x53800000u;  // 2^-20, 2^40
  return ok;
}

// Largest |entry| of A, L (m x k column-major) and U (k x n row-major) as float bits (a NaN
// counts as larger than Inf) in mx[0..2]; mx[0] = 0, out of range, where the three together allow
// too large a product (lu_exp and top_exp: range_limits). mx[3] counts blocks; all four are zero
// on entry.
template <typename TA, typename TLU>
__global__ void __launch_bounds__(256) k_range(ResidualArgs a, int lu_exp, int top_exp,
                                               uint32_t* __restrict__ mx) {
  uint32_t big[3] = {0, 0, 0};
  auto scan = [&](auto* p, int64_t rows, int64_t cols, int64_t ld, uint32_t& b) {
    for (int64_t r = blockIdx.x; r < rows; r += gridDim.x)
#pragma unroll 4
      for (int64_t c = threadIdx.x; c < cols; c += 256)
        b = max(b, __float_as_uint(fabsf(to_f(p[r * ld + c]))));
  };
  scan(static_cast<const TA*>(a.A), a.m, a.n, a.lda, big[0]);
  scan(static_cast<const TLU*>(a.L), a.k, a.m, a.ldl, big[1]);
  scan(static_cast<const TLU*>(a.U), a.k, a.n, a.ldu, big[2]);
  __shared__ uint32_t red[3][8];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const uint32_t w = __reduce_max_sync(0xffffffffu, big[i]);
    if ((threadIdx.x & 31) == 0) red[i][threadIdx.x >> 5] = w;
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  if (threadIdx.x < 3) {  // one atomic a block; one a warp cost more than the count below
    uint32_t w = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) w = max(w, red[threadIdx.x][q]);
    atomicMax(mx + threadIdx.x, w);
    __threadfence();
  }
  __syncwarp();
  if (threadIdx.x == 0 && atomicAdd(mx + 3, 1u) == gridDim.x - 1) {  // the last block
    __threadfence();
    int e[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) e[i] = (int)(__ldcg(mx + i) >> 23);
    if (e[0] + max(e[0], e[1] + e[2] + lu_exp) > top_exp) mx[0] = 0;
  }
}
struct RangeLimits { int lu_exp, top_exp; };
// |(PAQ - LU) x| <= sqrt(n) (max|A| + k max|L| max|U|), and its products with A over a chunk of
// rows stay below 2^126; a maximum is below 2^(e - 126), e its exponent field.
static RangeLimits range_limits(const ResidualArgs& a) {
  auto log2_up = [](int64_t v) {  // smallest e with v <= 2^e
    int e = 0;
    while (((int64_t)1 << e) < v) ++e;
    return e;
  };
  return {log2_up(a.k) - 126,
          126 + 2 * 126 - 1 - (log2_up(a.n) + 1) / 2 - log2_up(ceil_div(a.m, RS_RB))};
}

static constexpr int RS_BM = 64, RS_BN = 64, RS_BK = 16;

// ||R||_F, FP32 form: tiles as below, the residual a - sum l u accumulated exactly from a.
template <typename TA>
__device__ __forceinline__ double residual_tile_f32(const ResidualArgs& a, float (*Ls)[RS_BM + 1],
                                                    float (*Us)[RS_BN + 1]) {
  const TA* __restrict__ A = static_cast<const TA*>(a.A);
  const float* __restrict__ L = static_cast<const float*>(a.L);
  const float* __restrict__ U = static_cast<const float*>(a.U);
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int64_t m0 = (int64_t)blockIdx.y * RS_BM, n0 = (int64_t)blockIdx.x * RS_BN;
  Acc3 acc[4][4];
  bool in[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t gi = m0 + ty + 16 * i;
    const int64_t prow = gi < a.m ? (int64_t)a.P[gi] * a.lda : 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t gj = n0 + tx + 16 * j;
      in[i][j] = gi < a.m && gj < a.n;
      acc[i][j] = Acc3{in[i][j] ? to_f(A[prow + a.Q[gj]]) : 0.f, 0.f, 0.f};
    }
  }
  for (int t0 = 0; t0 < a.k; t0 += RS_BK) {
    for (int e = tid; e < RS_BK * RS_BM; e += 256) {
      const int kk = e / RS_BM, r = e % RS_BM, t = t0 + kk;
      Ls[kk][r] = (m0 + r < a.m && t < a.k) ? -L[(int64_t)t * a.ldl + m0 + r] : 0.f;
    }
    for (int e = tid; e < RS_BK * RS_BN; e += 256) {
      const int kk = e / RS_BN, c = e % RS_BN, t = t0 + kk;
      Us[kk][c] = (n0 + c < a.n && t < a.k) ? U[(int64_t)t * a.ldu + n0 + c] : 0.f;
    }
    __syncthreads();
#pragma unroll 2
    for (int kk = 0; kk < RS_BK; ++kk) {
      float lv[4], uv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) lv[i] = Ls[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) uv[j] = Us[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j].mac(lv[i], uv[j]);
    }
    __syncthreads();
  }
  double sq = 0.0;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double r = acc[i][j].value();
      if (in[i][j]) sq = fma(r, r, sq);
    }
  return sq;
}

template <typename TA, typename TLU>
__device__ __forceinline__ double residual_tile_f64(const ResidualArgs& a,
                                                    double (*Ls)[RS_BM + 1],
                                                    double (*Us)[RS_BN + 1]) {
  const TA* __restrict__ A = static_cast<const TA*>(a.A);
  const TLU* __restrict__ L = static_cast<const TLU*>(a.L);
  const TLU* __restrict__ U = static_cast<const TLU*>(a.U);
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int64_t m0 = (int64_t)blockIdx.y * RS_BM, n0 = (int64_t)blockIdx.x * RS_BN;
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  for (int t0 = 0; t0 < a.k; t0 += RS_BK) {
    for (int e = tid; e < RS_BK * RS_BM; e += 256) {
      const int kk = e / RS_BM, r = e % RS_BM;
      const int64_t gi = m0 + r;
      const int t = t0 + kk;
      Ls[kk][r] = (gi < a.m && t < a.k) ? to_d(L[(int64_t)t * a.ldl + gi]) : 0.0;
    }
    for (int e = tid; e < RS_BK * RS_BN; e += 256) {
      const int kk = e / RS_BN, c = e % RS_BN;
      const int64_t gj = n0 + c;
      const int t = t0 + kk;
      Us[kk][c] = (gj < a.n && t < a.k) ? to_d(U[(int64_t)t * a.ldu + gj]) : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < RS_BK; ++kk) {
      double lv[4], uv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) lv[i] = Ls[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) uv[j] = Us[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(lv[i], uv[j], acc[i][j]);
    }
    __syncthreads();
  }
  double sq = 0.0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t gi = m0 + ty + 16 * i;
    if (gi >= a.m) continue;
    const int64_t prow = (int64_t)a.P[gi] * a.lda;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t gj = n0 + tx + 16 * j;
      if (gj >= a.n) continue;
      const double r = to_d(A[prow + a.Q[gj]]) - acc[i][j];
      sq = fma(r, r, sq);
    }
  }
  return sq;
}

template <typename TA, typename TLU, bool F32>
__global__ void __launch_bounds__(256) k_residual_fro(ResidualArgs a, double* __restrict__ partial,
                                                      const uint32_t* __restrict__ mx) {
  __shared__ double tiles[2][RS_BK][RS_BM + 1];
  __shared__ double red[256];
  const int tid = threadIdx.x;
  double sq;
  bool done = false;
  if constexpr (F32) {
    if (in_range(mx)) {
      sq = residual_tile_f32<TA>(a, reinterpret_cast<float(*)[RS_BM + 1]>(&tiles[0][0][0]),
                                 reinterpret_cast<float(*)[RS_BN + 1]>(&tiles[1][0][0]));
      done = true;
    }
  }
  if (!done) sq = residual_tile_f64<TA, TLU>(a, tiles[0], tiles[1]);
  red[tid] = sq;
  __syncthreads();
  for (int off = 128; off > 0; off >>= 1) {
    if (tid < off) red[tid] += red[tid + off];
    __syncthreads();
  }
  if (tid == 0) partial[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = red[0];
}

// out[0] = sqrt(sum of in[0..count)) if take_sqrt else the sum; one block, fixed order.
__global__ void k_sum_sqrt(const double* __restrict__ in, int64_t count, double* __restrict__ out,
                           bool take_sqrt) {
  __shared__ double red[256];
  double s = 0.0;
  for (int64_t e = threadIdx.x; e < count; e += 256) s += in[e];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int off = 128; off > 0; off >>= 1) {
    if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = take_sqrt ? sqrt(red[0]) : red[0];
}

// ---- power iteration pieces -----------------------------------------------------------
// Sum of squares of 64 values, one per thread of the block's first two warps, to out.
__device__ __forceinline__ void sum_sq64(double v, double* __restrict__ out) {
  __shared__ double half[2];
  double s = v * v;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (threadIdx.x == 0 || threadIdx.x == 32) half[threadIdx.x >> 5] = s;
  asm volatile("bar.sync 1, 64;\n" ::: "memory");
  if (threadIdx.x == 0) *out = half[0] + half[1];
}

// fixed start vector z_j = 1 + (j mod 7)/7, normalised later; sq: each block's sum of squares
// (64 entries a block, as k_finish_z's)
__global__ void __launch_bounds__(64) k_init_x(double* z, int64_t n, double* __restrict__ sq) {
  const int64_t j = blockIdx.x * 64ll + threadIdx.x;
  const double v = j < n ? 1.0 + (double)(j % 7) / 7.0 : 0.0;
  if (j < n) z[j] = v;
  sum_sq64(v, sq + blockIdx.x);
}

// Sum of count values of sq in every thread of a 256-thread block (the same order in each).
__device__ __forceinline__ double block_total(const double* __restrict__ sq, int64_t count) {
  __shared__ double red[8];
  double s = 0.0;
  for (int64_t e = threadIdx.x; e < count; e += 256) s += sq[e];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  s = 0.0;
#pragma unroll
  for (int w = 0; w < 8; ++w) s += red[w];
  return s;
}

// x = z / ||z||, ||z||^2 from its blocks' partial sums sq; xq[Q[j]] = x[j], and its three float
// parts in planes of xs (xs + n, xs + 2 n).
__global__ void __launch_bounds__(256) k_scatter_q(const double* __restrict__ z,
                                                   const double* __restrict__ sq, int64_t count,
                                                   const int32_t* __restrict__ Q, int64_t n,
                                                   double* __restrict__ x, double* __restrict__ xq,
                                                   float* __restrict__ xs) {
  const double nrm = sqrt(block_total(sq, count));
  const double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
  for (int64_t j = blockIdx.x * 256ll + threadIdx.x; j < n; j += gridDim.x * 256ll) {
    const int64_t c = Q[j];
    const double v = z[j] * inv;
    x[j] = v;
    xq[c] = v;
    split3(v, xs[c], xs[n + c], xs[2 * n + c]);
  }
}

// sqrt of the sum of count partial sums (one block)
__global__ void __launch_bounds__(256) k_norm(const double* __restrict__ sq, int64_t count,
                                              double* __restrict__ out) {
  const double nrm = sqrt(block_total(sq, count));
  if (threadIdx.x == 0) out[0] = nrm;
}

// u[t] = sum_j U[t][j] x[j]  (block per t)
template <typename TLU>
__global__ void k_u_x(const TLU* __restrict__ U, int64_t ldu, const double* __restrict__ x,
                      int64_t n, double* __restrict__ u) {
  __shared__ double red[256];
  const int t = blockIdx.x;
  double s = 0.0;
#pragma unroll 8
  for (int64_t j = threadIdx.x; j < n; j += 256) s = fma(to_d(U[(int64_t)t * ldu + j]), x[j], s);
  red[threadIdx.x] = s;
  __syncthreads();
  for (int off = 128; off > 0; off >>= 1) {
    if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) u[t] = red[0];
}

// y[i] = sum_t L[i][t] u[t]: 64 rows a block, four threads a row (every fourth t)
template <typename TLU>
__global__ void __launch_bounds__(256) k_l_u(ResidualArgs a, const double* __restrict__ u,
                                             double* __restrict__ y) {
  const TLU* __restrict__ L = static_cast<const TLU*>(a.L);
  __shared__ double red[4][64];
  const int r = threadIdx.x & 63, g = threadIdx.x >> 6;
  const int64_t i = blockIdx.x * 64ll + r;
  double s = 0.0;
  if (i < a.m)
#pragma unroll 4
    for (int t = g; t < a.k; t += 4) s = fma(to_d(L[(int64_t)t * a.ldl + i]), u[t], s);
  red[g][r] = s;
  __syncthreads();
  if (g == 0 && i < a.m) y[i] = (red[0][r] + red[1][r]) + (red[2][r] + red[3][r]);
}

// y[i] = sum_c A[P[i]][c] xq[c] - y[i]  (a warp per RB rows; xs: x's float parts)
template <typename TA, typename TLU, int RB, bool F32>
__global__ void __launch_bounds__(256) k_rows(ResidualArgs a, const double* __restrict__ xq,
                                              const float* __restrict__ xs,
                                              double* __restrict__ y,
                                              const uint32_t* __restrict__ mx) {
  const TA* __restrict__ A = static_cast<const TA*>(a.A);
  const int lane = threadIdx.x & 31;
  const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i0 = wid * RB; i0 < a.m; i0 += nw * RB) {
    const TA* row[RB];
    double s[RB];
#pragma unroll
    for (int b = 0; b < RB; ++b) row[b] = A + (int64_t)a.P[min(i0 + b, a.m - 1)] * a.lda;
    bool done = false;
    if constexpr (F32) {
      if (in_range(mx)) {
        Acc3 acc[RB];
#pragma unroll
        for (int b = 0; b < RB; ++b) acc[b] = Acc3{0.f, 0.f, 0.f};
        int64_t c = lane;
        for (; c + 96 < a.n; c += 128) {  // four columns in flight
          float av[RB][4], x1[4], x2[4], x3[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
#pragma unroll
            for (int b = 0; b < RB; ++b) av[b][q] = to_f(row[b][c + 32 * q]);
            x1[q] = xs[c + 32 * q];
            x2[q] = xs[a.n + c + 32 * q];
            x3[q] = xs[2 * a.n + c + 32 * q];
          }
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int b = 0; b < RB; ++b) acc[b].mac(av[b][q], x1[q], x2[q], x3[q]);
        }
        for (; c < a.n; c += 32)
#pragma unroll
          for (int b = 0; b < RB; ++b)
            acc[b].mac(to_f(row[b][c]), xs[c], xs[a.n + c], xs[2 * a.n + c]);
#pragma unroll
        for (int b = 0; b < RB; ++b) s[b] = acc[b].value();
        done = true;
      }
    }
    if (!done) {
#pragma unroll
      for (int b = 0; b < RB; ++b) s[b] = 0.0;
      for (int64_t c = lane; c < a.n; c += 32)
#pragma unroll
        for (int b = 0; b < RB; ++b) s[b] = fma(to_d(row[b][c]), xq[c], s[b]);
    }
#pragma unroll
    for (int b = 0; b < RB; ++b) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) s[b] += __shfl_xor_sync(0xffffffffu, s[b], off);
      if (lane == 0 && i0 + b < a.m) y[i0 + b] = s[b] - y[i0 + b];
    }
  }
}

// v[t] = sum_i L[i][t] y[i] (block per t)
template <typename TLU>
__global__ void k_lt_y(const TLU* __restrict__ L, int64_t ldl, const double* __restrict__ y,
                       int64_t m, double* __restrict__ v) {
  __shared__ double red[256];
  const int t = blockIdx.x;
  double s = 0.0;
#pragma unroll 8
  for (int64_t i = threadIdx.x; i < m; i += 256) s = fma(to_d(L[(int64_t)t * ldl + i]), y[i], s);
  red[threadIdx.x] = s;
  __syncthreads();
  for (int off = 128; off > 0; off >>= 1) {
    if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) v[t] = red[0];
}

// zpart[rb][c] = sum over rows i of chunk rb of A[P[i]][c] y[i]  (thread per column; the rows'
// offsets and y, with its float parts, staged in shared memory)
template <typename TA, typename TLU, bool F32>
__global__ void __launch_bounds__(256) k_cols(ResidualArgs a, const double* __restrict__ y,
                                              int64_t rows_per, double* __restrict__ zpart,
                                              const uint32_t* __restrict__ mx) {
  constexpr int CH = 128;
  __shared__ int64_t off[CH];
  __shared__ double yd[CH];
  __shared__ float4 yf[CH];
  const TA* __restrict__ A = static_cast<const TA*>(a.A);
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t rb = blockIdx.y;
  const int64_t i0 = rb * rows_per, i1 = min(a.m, i0 + rows_per);
  bool fast = false;
  if constexpr (F32) fast = in_range(mx);
  Acc3 acc{0.f, 0.f, 0.f};
  double s = 0.0;
  const TA* col = A + (c < a.n ? c : 0);
  for (int64_t ib = i0; ib < i1; ib += CH) {
    const int rows = (int)min((int64_t)CH, i1 - ib);
    for (int r = threadIdx.x; r < rows; r += 256) {
      off[r] = (int64_t)a.P[ib + r] * a.lda;
      yd[r] = y[ib + r];
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      split3(yd[r], v.x, v.y, v.z);
      yf[r] = v;
    }
    __syncthreads();
    if (fast) {
      int r = 0;
      for (; r + 3 < rows; r += 4) {
        float av[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) av[q] = to_f(col[off[r + q]]);
#pragma unroll
        for (int q = 0; q < 4; ++q) acc.mac(av[q], yf[r + q].x, yf[r + q].y, yf[r + q].z);
      }
      for (; r < rows; ++r) acc.mac(to_f(col[off[r]]), yf[r].x, yf[r].y, yf[r].z);
    } else {
      for (int r = 0; r < rows; ++r) s = fma(to_d(col[off[r]]), yd[r], s);
    }
    __syncthreads();
  }
  if (c < a.n) zpart[rb * a.n + c] = fast ? acc.value() : s;
}

// z[j] = sum_rb zpart[rb][Q[j]] - sum_t U[t][j] v[t]  (64 columns a block, eight threads
// a column, each every eighth rb and t); sq: each block's sum of squares
template <typename TLU>
__global__ void __launch_bounds__(512) k_finish_z(ResidualArgs a, const double* __restrict__ zpart,
                                                  int nrb, const double* __restrict__ v,
                                                  double* __restrict__ z, double* __restrict__ sq) {
  const TLU* __restrict__ U = static_cast<const TLU*>(a.U);
  __shared__ double red[8][64];
  const int tx = threadIdx.x & 63, g = threadIdx.x >> 6;
  const int64_t j = blockIdx.x * 64ll + tx;
  double s = 0.0;
  if (j < a.n) {
    const int64_t c = a.Q[j];
#pragma unroll 8
    for (int rb = g; rb < nrb; rb += 8) s += zpart[(int64_t)rb * a.n + c];
    double s2 = 0.0;
#pragma unroll 8
    for (int t = g; t < a.k; t += 8) s2 = fma(to_d(U[(int64_t)t * a.ldu + j]), v[t], s2);
    s -= s2;
  }
  red[g][tx] = s;
  __syncthreads();
  if (g > 0) return;
#pragma unroll
  for (int q = 1; q < 8; ++q) s += red[q][tx];
  if (j < a.n) z[j] = s;
  sum_sq64(j < a.n ? s : 0.0, sq + blockIdx.x);
}

__global__ void k_sqrt_into(const double* __restrict__ in, double* __restrict__ out) {
  out[0] = sqrt(in[0]);
}


size_t residual_workspace_bytes(int64_t m, int64_t n, int k) {
  const int64_t tiles = ceil_div(m, RS_BM) * ceil_div(n, RS_BN);
  const int64_t doubles = round_up(tiles, 32) + 4 * round_up(n, 32) + round_up(m, 32) +
                          2 * round_up(k, 32) + (int64_t)RS_RB * round_up(n, 32) + 32;
  return (size_t)doubles * sizeof(double);
}

template <typename TA, typename TLU, bool F32>
static int32_t residual_run(const ResidualArgs& a, double* err_fro, double* err_spec, int iters,
                            double* ws, cudaStream_t s) {
  const int64_t tx = ceil_div(a.n, RS_BN), ty = ceil_div(a.m, RS_BM);
  double* partial = ws;
  double* x = partial + round_up(tx * ty, 32);
  double* xq = x + round_up(a.n, 32);
  double* z = xq + round_up(a.n, 32);
  double* nrm = z + round_up(a.n, 32);  // 32 doubles of scalars
  double* y = nrm + 32;
  double* u = y + round_up(a.m, 32);
  double* v = u + round_up(a.k, 32);
  double* zpart = v + round_up(a.k, 32);
  uint32_t* mx = reinterpret_cast<uint32_t*>(nrm + 16);
  // x's float parts, dead before the transposed product writes zpart
  float* xs = reinterpret_cast<float*>(zpart);
  if (ty > 65535) return RLU_EUNSUPPORTED;
  if constexpr (F32) {
    RLU_CUDA_TRY(cudaMemsetAsync(mx, 0, 4 * sizeof(uint32_t), s));
    const RangeLimits lim = range_limits(a);
    k_range<TA, TLU><<<(unsigned)std::min<int64_t>(std::max<int64_t>(a.m, a.k), 16 * sm_count()), 256, 0, s>>>(
        a, lim.lu_exp, lim.top_exp, mx);
    RLU_TRY(last_launch_status());
  }
  k_residual_fro<TA, TLU, F32><<<dim3((unsigned)tx, (unsigned)ty), 256, 0, s>>>(a, partial, mx);
  RLU_TRY(last_launch_status());
  k_sum_sqrt<<<1, 256, 0, s>>>(partial, tx * ty, err_fro, true);
  RLU_TRY(last_launch_status());
  if (err_spec == nullptr) return RLU_OK;
  const int threads = 256;
  const unsigned gn = (unsigned)std::min<int64_t>(ceil_div(a.n, threads), 4096);
  // blocks of z, each with its sum of squares in place of the (at least as many) tile sums
  const unsigned gz = (unsigned)ceil_div(a.n, 64);
  double* sq = partial;
  // two rows a warp share their loads of x once that leaves 16 warps to every SM
  const int rbw = a.m >= 32 * (int64_t)sm_count() ? 2 : 1;
  const unsigned gm = (unsigned)std::min<int64_t>(ceil_div(ceil_div(a.m, rbw) * 32, threads), 8192);
  const int64_t rows_per = ceil_div(a.m, RS_RB);
  k_init_x<<<gz, 64, 0, s>>>(z, a.n, sq);
  RLU_TRY(last_launch_status());
  for (int it = 0; it < iters; ++it) {
    k_scatter_q<<<gn, threads, 0, s>>>(z, sq, gz, a.Q, a.n, x, xq, xs);
    k_u_x<TLU><<<a.k, 256, 0, s>>>(static_cast<const TLU*>(a.U), a.ldu, x, a.n, u);
    k_l_u<TLU><<<(unsigned)ceil_div(a.m, 64), 256, 0, s>>>(a, u, y);
    if (rbw == 2) k_rows<TA, TLU, 2, F32><<<gm, threads, 0, s>>>(a, xq, xs, y, mx);
    else k_rows<TA, TLU, 1, F32><<<gm, threads, 0, s>>>(a, xq, xs, y, mx);
    k_lt_y<TLU><<<a.k, 256, 0, s>>>(static_cast<const TLU*>(a.L), a.ldl, y, a.m, v);
    k_cols<TA, TLU, F32><<<dim3((unsigned)ceil_div(a.n, threads), RS_RB), threads, 0, s>>>(a, y, rows_per, zpart, mx);
    k_finish_z<TLU><<<gz, 512, 0, s>>>(a, zpart, RS_RB, v, z, sq);
    RLU_TRY(last_launch_status(7));
  }
  k_norm<<<1, 256, 0, s>>>(sq, gz, nrm);
  RLU_TRY(last_launch_status());
  // ||R^T R x|| with ||x|| = 1 converges to sigma_max^2
  k_sqrt_into<<<1, 1, 0, s>>>(nrm, err_spec);
  return last_launch_status();
}

// Up to one tile for every SM and one chunk of k, the FP64 form takes less than k_range, its
// memset and the FP32 form: ||R||_F alone, in a row of calls, 36-38 us against 41 at 300 x 300 to
// 700 x 700, k = 4 or 16; at k = 64 85 against 62, at 1000 x 1000, k = 16 54 against 51.
template <typename TA, typename TLU>
static int32_t residual_t(const ResidualArgs& a, double* err_fro, double* err_spec, int iters,
                          double* ws, cudaStream_t s) {
  if constexpr (has_f32<TA, TLU>()) {
    if (a.k > RS_BK || ceil_div(a.n, RS_BN) * ceil_div(a.m, RS_BM) > sm_count())
      return residual_run<TA, TLU, true>(a, err_fro, err_spec, iters, ws, s);
  }
  return residual_run<TA, TLU, false>(a, err_fro, err_spec, iters, ws, s);
}

int32_t residual_error(int32_t dtA, int32_t dtLU, const ResidualArgs& a, double* err_fro,
                       double* err_spec, int iters, double* ws, cudaStream_t s) {
  if (dtLU == RLU_F64) {
    if (dtA == RLU_F64) return residual_t<double, double>(a, err_fro, err_spec, iters, ws, s);
    if (dtA == RLU_F32) return residual_t<float, double>(a, err_fro, err_spec, iters, ws, s);
    if (dtA == RLU_BF16) return residual_t<__nv_bfloat16, double>(a, err_fro, err_spec, iters, ws, s);
  } else if (dtLU == RLU_F32) {
    if (dtA == RLU_F64) return residual_t<double, float>(a, err_fro, err_spec, iters, ws, s);
    if (dtA == RLU_F32) return residual_t<float, float>(a, err_fro, err_spec, iters, ws, s);
    if (dtA == RLU_BF16) return residual_t<__nv_bfloat16, float>(a, err_fro, err_spec, iters, ws, s);
  }
  return RLU_EUNSUPPORTED;
}

}  // namespace rlu
