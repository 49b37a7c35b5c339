// SIMT (CUDA-core) GEMMs for the plain FP32 and FP64 paths:
//   step 2  Y = A G,   step 5  C = L~^T A,  M = L~^T L~,  T = R^-T C,  B = R^-1 T,
//   step 7  L = L_y L_b.
// C(M x N) = A(M x K) * B(K x N). Each operand is either K-contiguous ("K-major") or
// contiguous along its other dimension; C is row- or column-major. Split-K writes dense
// row-major partial slices that a second kernel sums in a fixed order (deterministic).
//
// Tiling: BM x BN x BK tiles in double-buffered shared memory; each thread owns a
// (2*V) x (2*V) register micro-tile split into two V-wide column groups and two V-tall row
// groups (V = 16 bytes / sizeof(T)) so that shared-memory fragment reads are 16-byte vector
// loads without bank conflicts.
#include <algorithm>

#include "common.cuh"
#include "gemm_simt.cuh"
#include "umma.cuh"

namespace rlu {

template <typename T> struct GemmCfg;
template <> struct GemmCfg<float> {
  static constexpr int BM = 128, BN = 128, BK = 16, V = 4, TX = 16, TY = 16;
};
template <> struct GemmCfg<double> {
  static constexpr int BM = 64, BN = 64, BK = 16, V = 2, TX = 16, TY = 16;
};
// the smaller FP32 tile of the batched products (chosen per step by the autotuner)
struct GemmCfgF64x64 {
  static constexpr int BM = 64, BN = 64, BK = 16, V = 2, TX = 16, TY = 16;
};

// FP64 tiles for products with a short side (k or l columns): the FP64 multiply-adds bound
// these products (1/64 of the FP32 rate), so a tile's padding costs as much as its work.
template <int TBM, int TBN> struct GemmCfgF64 {
  // the smallest tiles take 2 x 2 elements a thread: the FP64 rate is per quarter of an SM, so
  // a CTA needs four warps to reach it
  static constexpr int BM = TBM, BN = TBN, BK = 16, V = TBM * TBN <= 1024 ? 1 : 2,
                       TX = TBN / (2 * V), TY = TBM / (2 * V);
};

// V consecutive elements of T as one vector load
template <typename T, int V> struct Vec;
template <> struct Vec<float, 4> { using type = float4; };
template <> struct Vec<float, 2> { using type = float2; };
template <> struct Vec<double, 2> { using type = double2; };
template <> struct Vec<double, 1> { using type = double; };

// One BM x BN output tile (bx, by) of K range slice bz; the output element type OutT may be
// wider than T (the batched Gram matrix is stored in FP64 for the LDL^T).
template <typename T, typename OutT, bool AK, bool BKM, bool CR, typename Cfg = GemmCfg<T>>
__device__ __forceinline__ void gemm_tile(const GemmArgs& p, int bx, int by, int bz) {
  constexpr int BM = Cfg::BM, BN = Cfg::BN, BK = Cfg::BK, V = Cfg::V;
  constexpr int NT = Cfg::TX * Cfg::TY;
  constexpr int PAD = V;
  constexpr int A_LD = (BM * BK + NT - 1) / NT, B_LD = (BN * BK + NT - 1) / NT;
  using VT = typename Vec<T, V>::type;

  __shared__ __align__(16) T As[2][BK][BM + PAD];
  __shared__ __align__(16) T Bs[2][BK][BN + PAD];

  const T* __restrict__ A = static_cast<const T*>(p.A);
  const T* __restrict__ Bm = static_cast<const T*>(p.B);
  const int tid = threadIdx.x;
  const int tx = tid % Cfg::TX, ty = tid / Cfg::TX;
  const int64_t m0 = (int64_t)by * BM, n0 = (int64_t)bx * BN;
  const int64_t kbeg = (int64_t)bz * p.kchunk;
  const int64_t kend = (kbeg + p.kchunk < p.K) ? kbeg + p.kchunk : p.K;

  T acc[2 * V][2 * V];
#pragma unroll
  for (int i = 0; i < 2 * V; ++i)
#pragma unroll
    for (int j = 0; j < 2 * V; ++j) acc[i][j] = T(0);

  T ra[A_LD], rb[B_LD];
  auto load_tile = [&](int64_t k0) {
#pragma unroll
    for (int i = 0; i < A_LD; ++i) {
      const int idx = tid + i * NT;
      const int r = AK ? idx / BK : idx % BM;
      const int kk = AK ? idx % BK : idx / BM;
      const int64_t gm = m0 + r, gk = k0 + kk;
      ra[i] = (gm < p.M && gk < kend && (BM * BK % NT == 0 || idx < BM * BK)) ? A[AK ? gm * p.lda + gk : gk * p.lda + gm] : T(0);
    }
#pragma unroll
    for (int i = 0; i < B_LD; ++i) {
      const int idx = tid + i * NT;
      const int c = BKM ? idx / BK : idx % BN;
      const int kk = BKM ? idx % BK : idx / BN;
      const int64_t gn = n0 + c, gk = k0 + kk;
      rb[i] = (gn < p.N && gk < kend && (BN * BK % NT == 0 || idx < BN * BK)) ? Bm[BKM ? gn * p.ldb + gk : gk * p.ldb + gn] : T(0);
    }
  };
  auto store_tile = [&](int buf) {
#pragma unroll
    for (int i = 0; i < A_LD; ++i) {
      const int idx = tid + i * NT;
      const int r = AK ? idx / BK : idx % BM;
      const int kk = AK ? idx % BK : idx / BM;
      if (BM * BK % NT == 0 || idx < BM * BK) As[buf][kk][r] = ra[i];
    }
#pragma unroll
    for (int i = 0; i < B_LD; ++i) {
      const int idx = tid + i * NT;
      const int c = BKM ? idx / BK : idx % BN;
      const int kk = BKM ? idx % BK : idx / BN;
      if (BN * BK % NT == 0 || idx < BN * BK) Bs[buf][kk][c] = rb[i];
    }
  };

  if (kbeg < kend) {
    load_tile(kbeg);
    store_tile(0);
  }
  __syncthreads();
  int buf = 0;
  for (int64_t k0 = kbeg; k0 < kend; k0 += BK) {
    const bool has_next = k0 + BK < kend;
    if (has_next) load_tile(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      T a[2 * V], b[2 * V];
      const VT a0 = *reinterpret_cast<const VT*>(&As[buf][kk][ty * V]);
      const VT a1 = *reinterpret_cast<const VT*>(&As[buf][kk][BM / 2 + ty * V]);
      const VT b0 = *reinterpret_cast<const VT*>(&Bs[buf][kk][tx * V]);
      const VT b1 = *reinterpret_cast<const VT*>(&Bs[buf][kk][BN / 2 + tx * V]);
      memcpy(&a[0], &a0, sizeof(VT));
      memcpy(&a[V], &a1, sizeof(VT));
      memcpy(&b[0], &b0, sizeof(VT));
      memcpy(&b[V], &b1, sizeof(VT));
#pragma unroll
      for (int i = 0; i < 2 * V; ++i)
#pragma unroll
        for (int j = 0; j < 2 * V; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    if (has_next) store_tile(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }

  OutT* __restrict__ Cm = static_cast<OutT*>(p.C) + (int64_t)bz * p.split_stride;
#pragma unroll
  for (int i = 0; i < 2 * V; ++i) {
    const int64_t gm = m0 + (i < V ? ty * V + i : BM / 2 + ty * V + (i - V));
    if (gm >= p.M) continue;
#pragma unroll
    for (int j = 0; j < 2 * V; ++j) {
      const int64_t gn = n0 + (j < V ? tx * V + j : BN / 2 + tx * V + (j - V));
      if (gn >= p.N) continue;
      const OutT v = (OutT)(p.alpha_neg ? -acc[i][j] : acc[i][j]);
      if (CR)
        Cm[gm * p.ldc + gn] = v;
      else
        Cm[gn * p.ldc + gm] = v;
    }
  }
}

template <typename T, bool AK, bool BKM, bool CR, typename Cfg = GemmCfg<T>>
__global__ void __launch_bounds__(Cfg::TX* Cfg::TY) k_gemm_simt(GemmArgs p) {
  gemm_tile<T, T, AK, BKM, CR, Cfg>(p, blockIdx.x, blockIdx.y, blockIdx.z);
}

// Batched form: problem blockIdx.z of the table, whole K range (no split); CTAs past the
// problem's own tile counts return at once.
template <typename T, typename OutT, bool AK, bool BKM, bool CR, typename Cfg>
__global__ void __launch_bounds__(256) k_gemm_simt_batched(const GemmArgs* __restrict__ table) {
  const GemmArgs p = table[blockIdx.z];
  if ((int64_t)blockIdx.y * Cfg::BM >= p.M || (int64_t)blockIdx.x * Cfg::BN >= p.N) return;
  gemm_tile<T, OutT, AK, BKM, CR, Cfg>(p, blockIdx.x, blockIdx.y, 0);
}

// Split-K reductions: out(i, j) = sum_z part[z][i][j], z ascending, accumulated and stored in
// OutT. What bounds them is the latency of the slices' loads, so a thread has eight slices in
// flight before it adds the first (one at a time, the 33 slices of the Gram matrix at
// 8192 x 200 took 12 us, of a 512 x 25 FP64 product 33 us), and for FP64 the rate of the FP64
// adds, so that its tiles are small enough to reach most SMs.
template <int R, typename T, typename OutT>
__device__ __forceinline__ void sum_slices(const T* __restrict__ p, int64_t slice, int splits,
                                           int64_t step, int rows, OutT (&s)[R]) {
  constexpr int ZB = 8;
#pragma unroll
  for (int r = 0; r < R; ++r) s[r] = OutT(0);
  for (int z0 = 0; z0 < splits; z0 += ZB) {
    T v[R][ZB];
#pragma unroll
    for (int u = 0; u < ZB; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (z0 + u < splits && r < rows) v[r][u] = p[(z0 + u) * slice + r * step];
#pragma unroll
    for (int u = 0; u < ZB; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (z0 + u < splits && r < rows) s[r] += (OutT)v[r][u];
  }
}

// FP32 slices with an FP64 sum (the Gram matrix): the FP64 units' conversion and add per slice
// (128 cycles a warp) bounded it, 20 us for 76 slices of 200 x 200, so the sum is kept exactly
// in FP32: three floats, the first two with the rounding error of every addition carried down.
__device__ __forceinline__ void two_sum32(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void sum_slices_exact(const float* __restrict__ p, int64_t slice,
                                                 int splits, double& sum) {
  constexpr int ZB = 16;
  float s1 = 0.f, s2 = 0.f, s3 = 0.f;
  for (int z0 = 0; z0 < splits; z0 += ZB) {
    float v[ZB];
#pragma unroll
    for (int u = 0; u < ZB; ++u) v[u] = z0 + u < splits ? p[(z0 + u) * slice] : 0.f;
#pragma unroll
    for (int u = 0; u < ZB; ++u) {
      float r, r2;
      two_sum32(s1, v[u], s1, r);
      two_sum32(s2, r, s2, r2);
      s3 = __fadd_rn(s3, r2);
    }
  }
  sum = (double)s1 + ((double)s2 + (double)s3);
}

template <typename T, typename OutT>
__global__ void __launch_bounds__(256) k_splitk_reduce(const T* __restrict__ part, int splits,
                                                       int64_t M, int64_t N, int64_t slice,
                                                       OutT* __restrict__ out, int64_t ldo,
                                                       bool out_rowmajor) {
  const int64_t total = M * N;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    OutT s[1];
    bool exact = false;
    if constexpr (std::is_same<T, float>::value && std::is_same<OutT, double>::value) {
      sum_slices_exact(part + e, slice, splits, s[0]);
      exact = isfinite(s[0]);  // infinities, NaN and sums past FLT_MAX take FP64
    }
    if (!exact) sum_slices<1>(part + e, slice, splits, 0, 1, s);
    const int64_t i = total < INT32_MAX ? (int64_t)((uint32_t)e / (uint32_t)N) : e / N;
    const int64_t j = e - i * N;
    if (out_rowmajor)
      out[i * ldo + j] = s[0];
    else
      out[j * ldo + i] = s[0];
  }
}

// For a column-major output (out(i, j) at out[j * ldo + i]): tiles of TR rows x 32 columns
// staged in shared memory, so that the partial slices are read along their rows and the
// output is written along its columns. TR = 32 in FP32 (both coalesced), 8 in FP64 (four times
// the SMs for its adds).
template <typename T, typename OutT, int TR>
__global__ void __launch_bounds__(256) k_splitk_reduce_t(const T* __restrict__ part, int splits,
                                                         int64_t M, int64_t N, int64_t slice,
                                                         OutT* __restrict__ out, int64_t ldo) {
  __shared__ OutT tile[TR][33];
  const int64_t i0 = (int64_t)blockIdx.y * TR, j0 = (int64_t)blockIdx.x * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 32 x 8
  constexpr int R = TR / 8;
  const int64_t ib = i0 + ty * R, j = j0 + tx;
  OutT s[R];
  const int64_t left = M - ib;
  const int rows = j < N ? (int)(left < R ? (left > 0 ? left : 0) : R) : 0;
  sum_slices<R>(part + ib * N + j, slice, splits, N, rows, s);
#pragma unroll
  for (int r = 0; r < R; ++r) tile[ty * R + r][tx] = s[r];
  __syncthreads();
  for (int e = threadIdx.x; e < TR * 32; e += 256) {
    const int64_t jj = j0 + e / TR, i = i0 + e % TR;
    if (i < M && jj < N) out[jj * ldo + i] = tile[e % TR][e / TR];
  }
}

template <typename T, typename OutT>
static int32_t splitk_reduce_t(const T* part, int splits, int64_t M, int64_t N, OutT* out,
                               int64_t ldo, cudaStream_t s) {
  constexpr int TR = sizeof(OutT) == 8 ? 8 : 32;
  const dim3 grid((unsigned)ceil_div(N, 32), (unsigned)ceil_div(M, TR));
  k_splitk_reduce_t<T, OutT, TR><<<grid, 256, 0, s>>>(part, splits, M, N, M * N, out, ldo);
  return last_launch_status();
}
// whether its grid holds the rows
template <typename OutT>
static bool splitk_reduce_t_fits(int64_t M) { return ceil_div(M, sizeof(OutT) == 8 ? 8 : 32) <= 65535; }

template <typename T, typename OutT>
static int32_t splitk_reduce(const T* part, int splits, int64_t M, int64_t N, OutT* out,
                             int64_t ldo, bool out_rowmajor, cudaStream_t s) {
  const int threads = sizeof(OutT) == 8 ? 64 : 256;  // (FP64: over more SMs)
  int64_t blocks = ceil_div(M * N, threads);
  if (blocks > (int64_t)sm_count() * 32) blocks = (int64_t)sm_count() * 32;
  k_splitk_reduce<T, OutT><<<(unsigned)blocks, threads, 0, s>>>(part, splits, M, N, M * N, out,
                                                               ldo, out_rowmajor);
  return last_launch_status();
}

template <typename T, typename Cfg>
static void launch_variant(const GemmArgs& a, bool AK, bool BKM, bool CR, int splits,
                           cudaStream_t s) {
  const dim3 grid((unsigned)ceil_div(a.N, Cfg::BN), (unsigned)ceil_div(a.M, Cfg::BM),
                  (unsigned)splits);
#define RLU_GEMM_CASE(x, y, z)                                                 \
  if (AK == x && BKM == y && CR == z) {                                       \
    k_gemm_simt<T, x, y, z, Cfg><<<grid, Cfg::TX * Cfg::TY, 0, s>>>(a);       \
    return;                                                                   \
  }
  RLU_GEMM_CASE(true, true, true)
  RLU_GEMM_CASE(true, true, false)
  RLU_GEMM_CASE(true, false, true)
  RLU_GEMM_CASE(true, false, false)
  RLU_GEMM_CASE(false, true, true)
  RLU_GEMM_CASE(false, true, false)
  RLU_GEMM_CASE(false, false, true)
  RLU_GEMM_CASE(false, false, false)
#undef RLU_GEMM_CASE
}

// FP64 tile of an M x N product: a side of at most 48 takes the smallest of 32 and 48 that
// holds it, every other side tiles of 64. A product that is not split along K (one slice)
// with at most 32 columns takes fewer rows a tile while its tiles are fewer than the SMs
// (L = L_y L_b at 512 x 20: 36 us on 8 tiles of 64 x 64).
static int f64_side(int64_t n) { return n <= 32 ? 32 : n <= 48 ? 48 : 64; }

template <typename T>
static void launch_tiles(const GemmArgs& a, bool AK, bool BKM, bool CR, int splits,
                         cudaStream_t s) {
  if constexpr (std::is_same<T, double>::value) {
    int bm = f64_side(a.M);
    const int bn = f64_side(a.N);
    if (splits == 1 && bn == 32)
      while (bm > 16 && ceil_div(a.M, bm) < sm_count()) bm = bm > 32 ? 32 : 16;
#define RLU_GEMM_TILE(x, y) \
  if (bm == x && bn == y) return launch_variant<T, GemmCfgF64<x, y>>(a, AK, BKM, CR, splits, s);
    RLU_GEMM_TILE(64, 48)
    RLU_GEMM_TILE(64, 32)
    RLU_GEMM_TILE(16, 32)
    RLU_GEMM_TILE(48, 64)
    RLU_GEMM_TILE(32, 64)
    if (bm < 64 && bn < 64) {
      if (bm == 32 && bn == 32)
        return launch_variant<T, GemmCfgF64<32, 32>>(a, AK, BKM, CR, splits, s);
      return launch_variant<T, GemmCfgF64<48, 48>>(a, AK, BKM, CR, splits, s);
    }
#undef RLU_GEMM_TILE
  }
  launch_variant<T, GemmCfg<T>>(a, AK, BKM, CR, splits, s);
}

int gemm_splits_f64(int64_t M, int64_t N, int64_t K) {
  const int bm = f64_side(M), bn = f64_side(N);
  const int64_t tiles = ceil_div(M, bm) * ceil_div(N, bn), sms = sm_count();
  // cycles: the busiest SM's k-steps of 16 at two multiply-adds a cycle, then the reduction's
  // launch and its chain of adds; a split needs at least one k-step
  const int64_t steps = ceil_div(K > 0 ? K : 1, 16);
  const int64_t most = std::min<int64_t>(steps, std::max<int64_t>(1, 8 * sms / tiles));
  int best = 1;
  double cost = 1e300;
  for (int64_t s = 1; s <= most; ++s) {
    const int64_t per = ceil_div(steps, s), n = ceil_div(steps, per);
    const double adds = 70.0 + (double)M * (double)N / (2.0 * (double)sms);
    const double c = (double)(ceil_div(tiles * n, sms) * per) * (8.0 * bm * bn + 300.0) +
                     (n > 1 ? 6000.0 + adds * (double)n : 0.0);
    if (c < cost) {
      cost = c;
      best = (int)n;
    }
  }
  return best;
}

template <typename T, typename OutT, typename Cfg>
static int32_t gemm_batched_cfg(const GemmArgs* table_dev, int count, int64_t max_m,
                                int64_t max_n, bool a_kmajor, bool b_kmajor, bool c_rowmajor,
                                cudaStream_t s) {
  const dim3 grid((unsigned)ceil_div(max_n, Cfg::BN), (unsigned)ceil_div(max_m, Cfg::BM),
                  (unsigned)count);
#define RLU_GEMM_BCASE(x, y, z)                                                        \
  if (a_kmajor == x && b_kmajor == y && c_rowmajor == z) {                             \
    k_gemm_simt_batched<T, OutT, x, y, z, Cfg><<<grid, 256, 0, s>>>(table_dev);        \
    return last_launch_status();                                                       \
  }
  RLU_GEMM_BCASE(true, true, true)
  RLU_GEMM_BCASE(true, true, false)
  RLU_GEMM_BCASE(true, false, true)
  RLU_GEMM_BCASE(true, false, false)
  RLU_GEMM_BCASE(false, true, true)
  RLU_GEMM_BCASE(false, true, false)
  RLU_GEMM_BCASE(false, false, true)
  RLU_GEMM_BCASE(false, false, false)
#undef RLU_GEMM_BCASE
  return RLU_EINVAL;
}

template <typename T, typename OutT>
int32_t gemm_simt_batched(const GemmArgs* table_dev, int count, int64_t max_m, int64_t max_n,
                          bool a_kmajor, bool b_kmajor, bool c_rowmajor, cudaStream_t s,
                          int tile) {
  if (count <= 0) return RLU_OK;
  if (count > 65535) return RLU_EINVAL;
  if (tile == 1)
    return gemm_batched_cfg<T, OutT, GemmCfgF64x64>(table_dev, count, max_m, max_n, a_kmajor,
                                                    b_kmajor, c_rowmajor, s);
  return gemm_batched_cfg<T, OutT, GemmCfg<T>>(table_dev, count, max_m, max_n, a_kmajor,
                                               b_kmajor, c_rowmajor, s);
}
template int32_t gemm_simt_batched<float, float>(const GemmArgs*, int, int64_t, int64_t, bool,
                                                 bool, bool, cudaStream_t, int);
template int32_t gemm_simt_batched<float, double>(const GemmArgs*, int, int64_t, int64_t, bool,
                                                  bool, bool, cudaStream_t, int);

template <typename T>
size_t gemm_partial_bytes(int64_t M, int64_t N, int splits) {
  return splits > 1 ? (size_t)splits * (size_t)M * (size_t)N * sizeof(T) : 0;
}

template <typename T, typename OutT>
int32_t gemm_simt(const GemmOp& op, cudaStream_t s) {
  using Cfg = GemmCfg<T>;
  if (op.M == 0 || op.N == 0) return RLU_OK;
  int splits = op.splits < 1 ? 1 : op.splits;
  int64_t kchunk = round_up(ceil_div(op.K > 0 ? op.K : 1, splits), Cfg::BK);
  splits = (int)ceil_div(op.K > 0 ? op.K : 1, kchunk);
  GemmArgs a;
  a.A = op.A; a.lda = op.lda;
  a.B = op.B; a.ldb = op.ldb;
  a.M = op.M; a.N = op.N; a.K = op.K;
  a.kchunk = kchunk;
  a.alpha_neg = op.negate;
  const bool direct = (splits == 1) && std::is_same<T, OutT>::value;
  if (direct) {
    a.C = op.C; a.ldc = op.ldc; a.split_stride = 0;
    launch_tiles<T>(a, op.a_kmajor, op.b_kmajor, op.c_rowmajor, splits, s);
    return last_launch_status();
  }
  if (op.partial == nullptr) return RLU_ENOMEM;
  a.C = op.partial; a.ldc = op.N; a.split_stride = op.M * op.N;
  launch_tiles<T>(a, op.a_kmajor, op.b_kmajor, true, splits, s);
  RLU_TRY(last_launch_status());  // the split-K product
  const T* part = static_cast<const T*>(op.partial);
  OutT* C = static_cast<OutT*>(op.C);
  if (!op.c_rowmajor && splitk_reduce_t_fits<OutT>(op.M))
    return splitk_reduce_t<T, OutT>(part, splits, op.M, op.N, C, op.ldc, s);
  return splitk_reduce<T, OutT>(part, splits, op.M, op.N, C, op.ldc, op.c_rowmajor, s);
}

template int32_t gemm_simt<float, float>(const GemmOp&, cudaStream_t);
template int32_t gemm_simt<float, double>(const GemmOp&, cudaStream_t);
template int32_t gemm_simt<double, double>(const GemmOp&, cudaStream_t);
template size_t gemm_partial_bytes<float>(int64_t, int64_t, int);
template size_t gemm_partial_bytes<double>(int64_t, int64_t, int);

int32_t splitk_reduce_f32(const float* part, int splits, int64_t M, int64_t N, float* out,
                          int64_t ldo, bool out_rowmajor, cudaStream_t s) {
  if (!out_rowmajor) {
    if (!splitk_reduce_t_fits<float>(M)) return RLU_EUNSUPPORTED;
    return splitk_reduce_t<float, float>(part, splits, M, N, out, ldo, s);
  }
  return splitk_reduce<float, float>(part, splits, M, N, out, ldo, true, s);
}

// Column-major slices and output: a column per grid row, four rows a thread (VEC: as one
// 16-byte access; M and ldo multiples of 4, bases aligned). One element at a time with its
// 64-bit division it took 10 us at 8192 x 210.
template <bool VEC>
__global__ void __launch_bounds__(256) k_splitk_reduce_cm(const float* __restrict__ part,
                                                          int splits, int64_t M, int64_t N,
                                                          float* __restrict__ out,
                                                          int64_t ldo) {
  const int64_t total = M * N, i = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 4;
  if (i >= M) return;
  for (int64_t j = blockIdx.y; j < N; j += gridDim.y) {
    const float* p = part + j * M + i;
    float* o = out + j * ldo + i;
    if constexpr (VEC) {
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
      for (int z = 0; z < splits; ++z) {
        const float4 v = *reinterpret_cast<const float4*>(p + z * total);
        s.x += v.x;
        s.y += v.y;
        s.z += v.z;
        s.w += v.w;
      }
      *reinterpret_cast<float4*>(o) = s;
    } else {
      const int rows = (int)(M - i < 4 ? M - i : 4);
      float s[4];
      sum_slices<4>(p, total, splits, 1, rows, s);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (r < rows) o[r] = s[r];
    }
  }
}

int32_t splitk_reduce_cm_f32(const float* part, int splits, int64_t M, int64_t N, float* out,
                             int64_t ldo, cudaStream_t s) {
  const dim3 grid((unsigned)ceil_div(M, 1024), (unsigned)(N < 65535 ? N : 65535));
  const bool vec = M % 4 == 0 && ldo % 4 == 0 && (((uintptr_t)part | (uintptr_t)out) & 15u) == 0;
  if (vec) k_splitk_reduce_cm<true><<<grid, 256, 0, s>>>(part, splits, M, N, out, ldo);
  else k_splitk_reduce_cm<false><<<grid, 256, 0, s>>>(part, splits, M, N, out, ldo);
  return last_launch_status();
}

int32_t splitk_reduce_f64(const float* part, int splits, int64_t M, int64_t N, double* out,
                          int64_t ldo, cudaStream_t s) {
  return splitk_reduce<float, double>(part, splits, M, N, out, ldo, true, s);
}

int gemm_tile_m(int32_t dtype) { return dtype == RLU_F64 ? GemmCfg<double>::BM : GemmCfg<float>::BM; }
int gemm_tile_n(int32_t dtype) { return dtype == RLU_F64 ? GemmCfg<double>::BN : GemmCfg<float>::BN; }

}  // namespace rlu
