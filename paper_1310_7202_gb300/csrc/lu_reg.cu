// Pivoted LU of a tall-skinny column-major X (R x C) on one thread-block cluster: the fast
// form of steps 3 (Doolittle, X = Y) and 6 (Crout, X = B^T) of Algorithm 1, with the same
// swap-free position bookkeeping and tie rule as panel_lu.cu (largest |value|, then smallest
// current position, which is getf2's choice). The element type is float, double or cf32
// (complex FP32, for the fast randomized LU of Algorithm 4, whose pivots go by |Re| + |Im|).
//
// One launch factors one panel; the positions of the rows persist in global memory between
// launches, and k_lu_trail (all SMs) applies each panel's update to the remaining columns.
// Narrow panels (tall X, whose rows leave little shared memory per column) are grouped into
// blocks of about 64 columns, a right-looking blocked LU: a panel's update reaches only the
// rest of its block, the block's last panel solves the block's pivot rows for the columns
// after it, and the block's update is applied to those once.
//
// What bounds it is the chain of one pivot step, C times: find the largest candidate, tell
// every CTA, update the next column. So a CTA's warps are split by role:
//   - Control warps own the rows (RT each thread). They hold the current inner block of 8
//     columns in registers, and a step touches nothing else: warp reduction on
//     order-preserving integer keys, one CTA barrier, one record (value, position, row, the
//     row's entries in the rest of the block: at most 48 bytes in FP32) per CTA pushed with
//     st.async into a receive slot of every CTA of the cluster, a wait on the CTA's own
//     mbarrier, the winner among the records, and the update of at most 7 columns.
//   - Update warps hold the rest of the panel in shared memory. While the control warps factor
//     the next block they solve the block's 8 pivot rows (published by their owners through
//     st.async at the end of the block) and apply its rank-8 update there, four rows of a
//     column to a thread, two to an instruction (fma.rn.f32x2).
// Every element sees the same multiply-adds in the same order as column-by-column elimination,
// so the inner blocks and the panel width change no bit of the result.
//
// Measured against the form it replaced (one row of the whole panel in each thread's
// registers, every step updating all its columns and sending the whole row, 3900 cycles a
// step at 8192 rows): LU of Y at 8192 x 210 391 -> 243 us and of B^T (8192 x 200) 385 -> 221,
// 3001 x 71 110 -> 60 us, 32768 x 532 1905 -> 1336 us. A step takes about 1900 cycles, of which
// the exchange between 16 CTAs alone takes 440 (measured in isolation), the warp reduction with
// its record and barrier 110. Tried and slower: 256 control threads with half the rows each
// (two warps a scheduler), one control warp with all rows (no CTA barrier), every warp sending
// its own record (the exchange pays for packets: 64 of them took 1.9x as long as 16), and
// eight unrolled steps (instruction-cache misses).
//
// A problem whose rows fit one CTA (SOLO) skips the exchange: the record of the winning warp is
// read from shared memory.
//
// Waits on an mbarrier give up after about one second (globaltimer); the kernel then
// records RLU_ETIMEOUT in the status word and keeps going without waiting, so every CTA
// still reaches the same cluster barriers and exits.
#include <cooperative_groups.h>
#include <type_traits>

#include "common.cuh"
#include "panel_lu.cuh"
#include "umma.cuh"

namespace cg = cooperative_groups;

namespace rlu {

static constexpr int LR_CH = 32;  // trailing-update column chunk

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
// Test for completion of the phase of the given parity; the warp may sleep in the
// instruction up to the hinted time (ns) instead of spinning on issue slots.
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n"
               " mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n"
               " selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(ok) : "r"(bar), "r"(parity), "r"(20000u) : "memory");
  return ok != 0;
}
// Predicated instructions instead of branches around them (a branch on the chain of a pivot
// step costs more than the instruction).
__device__ __forceinline__ void mbar_arm_if(bool p, uint32_t bar, uint32_t tx) {
  asm volatile("{\n .reg .b64 st;\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n"
               " @p mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n"
               ::"r"(bar), "r"(tx), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void sts16_if(bool p, uint32_t addr, uint4 v) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %5, 0;\n"
               " @p st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n}\n"
               ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void st_async16_if(bool p, uint32_t raddr, uint4 v, uint32_t rbar) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %6, 0;\n"
               " @p st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];\n}\n"
               ::"r"(raddr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(rbar), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void st_async_if(bool p, uint32_t raddr, float v, uint32_t rbar) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %3, 0;\n"
               " @p st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];\n}\n"
               ::"r"(raddr), "r"(__float_as_uint(v)), "r"(rbar), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void st_async_if(bool p, uint32_t raddr, double v, uint32_t rbar) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %3, 0;\n"
               " @p st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];\n}\n"
               ::"r"(raddr), "l"(__double_as_longlong(v)), "r"(rbar), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void st_async_if(bool p, uint32_t raddr, cf32 v, uint32_t rbar) {
  st_async_if(p, raddr, __hiloint2double(__float_as_int(v.y), __float_as_int(v.x)), rbar);
}
__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;\n" : "=l"(t));
  return t;
}

// Order-preserving integer key of |v| (complex FP32, the fast randomized LU of Algorithm 4:
// |Re| + |Im|). A NaN's key lies above inf_key; it counts as 0, so that a NaN never beats a
// number.
__device__ __forceinline__ uint32_t raw_key(float v) { return __float_as_uint(fabsf(v)); }
__device__ __forceinline__ uint64_t raw_key(double v) {
  return (uint64_t)__double_as_longlong(fabs(v));
}
__device__ __forceinline__ uint32_t raw_key(cf32 v) {
  return __float_as_uint(fabsf(v.x) + fabsf(v.y));
}
template <typename K> __device__ __forceinline__ constexpr K inf_key() {
  return sizeof(K) == 4 ? (K)0x7f800000u : (K)0x7ff0000000000000ull;
}
template <typename T> using key_t = decltype(raw_key(T(0)));

// v where the mask is all ones, else (positive) zero
__device__ __forceinline__ float and_mask(float v, uint32_t m) {
  return __uint_as_float(__float_as_uint(v) & m);
}
__device__ __forceinline__ double and_mask(double v, uint32_t m) {
  return __hiloint2double(__double2hiint(v) & (int)m, __double2loint(v) & (int)m);
}
__device__ __forceinline__ cf32 and_mask(cf32 v, uint32_t m) {
  return cf32(and_mask(v.x, m), and_mask(v.y, m));
}

// Reciprocal of a pivot: the hardware approximation refined by Newton-Raphson steps
// (y' = y + y (1 - p y)): one step in FP32 (within an ulp or so), two from the FP32 seed in
// FP64 (IEEE divide outside the FP32 exponent range). Multipliers are x * (1/pivot).
__device__ __forceinline__ float rcp_approx(float p) {
  float y;
  asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(p));
  return y;
}
__device__ __forceinline__ float rcp_piv(float p) {
  const float y = rcp_approx(p);
  const float z = fmaf(y, fmaf(-p, y, 1.0f), y);
  return isfinite(y) ? z : y;
}
// 1 / p with the larger of |Re p|, |Im p| scaled out first (no overflow of |p|^2)
__device__ __forceinline__ cf32 rcp_piv(cf32 p) {
  const float sc = fmaxf(fabsf(p.x), fabsf(p.y));
  const float qx = p.x / sc, qy = p.y / sc;
  const float den = (qx * qx + qy * qy) * sc;
  return cf32(qx / den, -qy / den);
}
__device__ __forceinline__ double rcp_piv(double p) {
  const double a = fabs(p);
  if (!(a > 1e-30 && a < 1e30)) return 1.0 / p;
  double y = (double)rcp_approx((float)p);
  double e = fma(-p, y, 1.0);
  y = fma(y, e, y);
  e = fma(-p, y, 1.0);
  return fma(y, e, y);
}

// Vector shared-memory access of 4 consecutive elements (16-byte aligned for float).
__device__ __forceinline__ void ld4(const float* p, float (&o)[4]) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void ld4(const double* p, double (&o)[4]) {
  const double2 a = *reinterpret_cast<const double2*>(p);
  const double2 b = *reinterpret_cast<const double2*>(p + 2);
  o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}
__device__ __forceinline__ void ld4(const cf32* p, cf32 (&o)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  const float4 b = *reinterpret_cast<const float4*>(p + 2);
  o[0] = cf32(a.x, a.y); o[1] = cf32(a.z, a.w); o[2] = cf32(b.x, b.y); o[3] = cf32(b.z, b.w);
}
// warp shuffle of one element
__device__ __forceinline__ float shfl_t(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ double shfl_t(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ cf32 shfl_t(cf32 v, int src) {
  return cf32(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// Asynchronous global -> shared copies (cp.async): 16 bytes, or one element.
__device__ __forceinline__ void lr_cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n"
               ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
template <int BYTES>
__device__ __forceinline__ void lr_cp(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n"
               ::"r"(smem_u32(dst)), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void lr_cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void lr_cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

static constexpr int kLuUpd = 128;  // threads of a CTA's update warps

// Pivot candidates and records. A record is the header chunk (value in the current column,
// packed position and row, FP32: also the values in the next two columns) and the
// candidate's values in the rest of the inner block, in 16-byte chunks.
static constexpr int LB = 8;                // columns of an inner block
static constexpr int kNone = 0x7fffffff;    // packed (position << 16 | row) of no candidate

template <typename T>
struct RecT {
  static constexpr int EPC = 16 / (int)sizeof(T);        // elements per 16-byte chunk
  static constexpr int E0 = sizeof(T) == 4 ? 2 : 0;      // block values in the header chunk
  static constexpr int MC = 1 + (LB - 1 - E0 + EPC - 1) / EPC;  // chunks of the longest record
  // chunks of the record of step i of an inner block
  static __device__ __forceinline__ int chunks(int i) { return 1 + (LB - i) / EPC; }
};

__device__ __forceinline__ uint4 pack_hdr(float v, int pr, float n1, float n2) {
  return make_uint4(__float_as_uint(v), (uint32_t)pr, __float_as_uint(n1), __float_as_uint(n2));
}
__device__ __forceinline__ uint4 pack_hdr(double v, int pr, double, double) {
  return make_uint4((uint32_t)__double2loint(v), (uint32_t)pr, (uint32_t)__double2hiint(v), 0u);
}
__device__ __forceinline__ uint4 pack_hdr(cf32 v, int pr, cf32, cf32) {
  return make_uint4(__float_as_uint(v.x), (uint32_t)pr, __float_as_uint(v.y), 0u);
}
__device__ __forceinline__ void unpack_hdr(uint4 h, float& v, float& n1, float& n2) {
  v = __uint_as_float(h.x); n1 = __uint_as_float(h.z); n2 = __uint_as_float(h.w);
}
__device__ __forceinline__ void unpack_hdr(uint4 h, double& v, double&, double&) {
  v = __hiloint2double((int)h.z, (int)h.x);
}
__device__ __forceinline__ void unpack_hdr(uint4 h, cf32& v, cf32&, cf32&) {
  v = cf32(__uint_as_float(h.x), __uint_as_float(h.z));
}
__device__ __forceinline__ uint4 pack_chunk(const float (&v)[4]) {
  return make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]),
                    __float_as_uint(v[3]));
}
__device__ __forceinline__ uint4 pack_chunk(const double (&v)[2]) {
  return make_uint4((uint32_t)__double2loint(v[0]), (uint32_t)__double2hiint(v[0]),
                    (uint32_t)__double2loint(v[1]), (uint32_t)__double2hiint(v[1]));
}
__device__ __forceinline__ uint4 pack_chunk(const cf32 (&v)[2]) {
  return make_uint4(__float_as_uint(v[0].x), __float_as_uint(v[0].y), __float_as_uint(v[1].x),
                    __float_as_uint(v[1].y));
}
__device__ __forceinline__ void unpack_chunk(uint4 h, float (&v)[4]) {
  v[0] = __uint_as_float(h.x); v[1] = __uint_as_float(h.y);
  v[2] = __uint_as_float(h.z); v[3] = __uint_as_float(h.w);
}
__device__ __forceinline__ void unpack_chunk(uint4 h, double (&v)[2]) {
  v[0] = __hiloint2double((int)h.y, (int)h.x);
  v[1] = __hiloint2double((int)h.w, (int)h.z);
}
__device__ __forceinline__ void unpack_chunk(uint4 h, cf32 (&v)[2]) {
  v[0] = cf32(__uint_as_float(h.x), __uint_as_float(h.y));
  v[1] = cf32(__uint_as_float(h.z), __uint_as_float(h.w));
}

__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ uint32_t warp_max(uint32_t v) { return __reduce_max_sync(0xffffffffu, v); }
__device__ __forceinline__ uint64_t warp_max(uint64_t v) {
  const uint32_t hi = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32));
  const uint32_t lo = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0u);
  return (uint64_t)hi << 32 | lo;
}

// Shared memory of one CTA: the fixed part, then (by the rows of a CTA and the panel width)
// the published pivot rows ub, the solved pivot rows us, the panel xs (a column's multipliers
// take its place once it is eliminated) and, where the launch solves the pivot rows of later
// columns, L11.
template <typename T, int NCW>
struct LrShared {
  static constexpr int MC = RecT<T>::MC;
  // records of even and odd steps, pivot rows of even and odd blocks, L11
  uint64_t mbar[5];
  int32_t err, nonfinite;
  alignas(16) T uc[NCW][LB][LB];   // per control warp: U of the next block's columns, by row
  // records in one piece (MC is odd: headers of consecutive records meet no bank twice)
  uint4 wrec[2][NCW][MC];          // the warps' candidates, by step parity
  alignas(16) key_t<T> wkey[2][NCW];  // their keys
  alignas(16) int32_t wpr[2][NCW];    // and packed positions and rows
  uint4 recv[2][16][MC];           // the cluster's
  // pivot rows of the column block whose last panel this is (a panel alone: its own), and
  // the reciprocals of their pivots (1 at a zero pivot)
  int32_t prows[96];
  T rp[96];
};

template <typename T>
struct LrLayout {  // byte offsets behind LrShared
  int rs;          // stride of an xs column (elements): rows padded by one 16-byte chunk
  int ubw;         // stride of a published row
  int ub, us, xs, l11, total;
  // pw: panel columns, tw: rows of the triangular solve at the end (0: none)
  __host__ __device__ LrLayout(int fixed, int rows, int pw, int tw) {
    constexpr int E = 16 / (int)sizeof(T);
    const int oc = pw > LB ? (pw - LB + E - 1) / E * E : 0;
    rs = rows + E;
    ubw = LB + oc;
    int at = (fixed + 15) / 16 * 16;
    ub = at;
    at += 2 * LB * ubw * (int)sizeof(T);
    us = at;
    at += oc * LB * (sizeof(T) == 4 ? 8 : (int)sizeof(T));
    xs = at;
    at += (pw > LB || tw > 0 ? LB + oc : 0) * rs * (int)sizeof(T);
    l11 = at;
    at += tw * (tw + 1) * (int)sizeof(T);
    total = at;
  }
};

// rank-8 update of one 16-byte chunk of rows of columns: x -= mm u (us holds -u)
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
template <typename T>
struct RankUpdate {  // double and cf32: two rows a chunk
  T m[LB][2];
  __device__ __forceinline__ void load(const T* mm, int rows, int row) {
#pragma unroll
    for (int q = 0; q < LB; ++q) {
      m[q][0] = mm[q * rows + row];
      m[q][1] = mm[q * rows + row + 1];
    }
  }
  // N columns dx apart, their U du apart: all loads before the first store
  template <int N>
  __device__ __forceinline__ void apply(T* x, int dx, const T* u, int du) const {
    T v[N][2];
#pragma unroll
    for (int n = 0; n < N; ++n) {
      v[n][0] = x[n * dx];
      v[n][1] = x[n * dx + 1];
    }
#pragma unroll
    for (int q = 0; q < LB; ++q)
#pragma unroll
      for (int n = 0; n < N; ++n) {
        const T uq = u[n * du + q];
        v[n][0] = fma(m[q][0], uq, v[n][0]);
        v[n][1] = fma(m[q][1], uq, v[n][1]);
      }
#pragma unroll
    for (int n = 0; n < N; ++n) {
      x[n * dx] = v[n][0];
      x[n * dx + 1] = v[n][1];
    }
  }
};
template <>
struct RankUpdate<float> {  // four rows a chunk, two to an instruction; u held twice
  ulonglong2 m[LB];
  __device__ __forceinline__ void load(const float* mm, int rows, int row) {
#pragma unroll
    for (int q = 0; q < LB; ++q) m[q] = *reinterpret_cast<const ulonglong2*>(mm + q * rows + row);
  }
  template <int N>
  __device__ __forceinline__ void apply(float* x, int dx, const float* u, int du) const {
    ulonglong2 v[N];
#pragma unroll
    for (int n = 0; n < N; ++n) v[n] = *reinterpret_cast<const ulonglong2*>(x + n * dx);
#pragma unroll
    for (int q = 0; q < LB; q += 2)
#pragma unroll
      for (int n = 0; n < N; ++n) {
        const ulonglong2 uq = *reinterpret_cast<const ulonglong2*>(u + n * du + 2 * q);
        v[n].x = fma2(m[q].x, uq.x, v[n].x);
        v[n].y = fma2(m[q].y, uq.x, v[n].y);
        v[n].x = fma2(m[q + 1].x, uq.y, v[n].x);
        v[n].y = fma2(m[q + 1].y, uq.y, v[n].y);
      }
#pragma unroll
    for (int n = 0; n < N; ++n) *reinterpret_cast<ulonglong2*>(x + n * dx) = v[n];
  }
};

// U of one column of the block's pivot rows: forward substitution with the published rows
template <typename T, bool CROUT>
__device__ __forceinline__ void solve_block(const T* ub, int ubw, const T* rp, int c, T (&u)[LB]) {
#pragma unroll
  for (int t = 0; t < LB; ++t) u[t] = ub[t * ubw + LB + c];
#pragma unroll
  for (int q = 0; q < LB; ++q) {
    if (CROUT) u[q] = u[q] * rp[q];
#pragma unroll
    for (int t = q + 1; t < LB; ++t) u[t] = fma(-ub[t * ubw + q], u[q], u[t]);
  }
}

template <typename T, bool CROUT, int RT, int NC, bool SOLO>
__device__ __forceinline__ void lu_reg_body(const LuArgs& a) {
  constexpr int NCW = NC / 32;
  constexpr int NT = NC + kLuUpd;
  constexpr int ROWS = NC * RT;  // rows of a CTA
  using RC = RecT<T>;
  constexpr int EPC = RC::EPC, E0 = RC::E0, MC = RC::MC;
  cg::cluster_group cl = cg::this_cluster();
  const int ncta = SOLO ? 1 : (int)cl.num_blocks();
  const int crank = SOLO ? 0 : (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = crank * ROWS;
  const int C = a.C, R = a.R;
  const int64_t ldx = a.ldx;
  const int p0 = a.p0, w = a.pw;
  const int cu = a.cu > 0 ? a.cu : C;
  const int o0 = a.o0, W = p0 + w - o0;  // the rows solved for the columns [p0 + w, cu)
  const bool tail = p0 + w < cu;
  T* __restrict__ X = static_cast<T*>(a.X);

  extern __shared__ __align__(16) unsigned char smem_raw[];
  using Sh = LrShared<T, NCW>;
  Sh& sh = *reinterpret_cast<Sh*>(smem_raw);
  const LrLayout<T> lay((int)sizeof(Sh), ROWS, a.nb, tail ? W : 0);
  T* const ub = reinterpret_cast<T*>(smem_raw + lay.ub);  // [2][LB][ubw]
  T* const us = reinterpret_cast<T*>(smem_raw + lay.us);  // [oc][LB], negated; FP32: every value twice
  T* const xs = reinterpret_cast<T*>(smem_raw + lay.xs);  // [panel columns][rs]
  const int ubw = lay.ubw, rs = lay.rs;

  if (tid == 0) {
    for (int i = 0; i < 5; ++i) mbar_init(smem_u32(&sh.mbar[i]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    sh.err = 0;
    sh.nonfinite = 0;
  }
  if (SOLO) __syncthreads();
  else cl.sync();

  const uint32_t mbar_a = smem_u32(&sh.mbar[0]);
  bool timed_out = false;
  auto wait = [&](uint32_t bar, uint32_t ph) {
    if (timed_out || mbar_try(bar, ph)) return;
    const uint64_t t0 = gtimer();
    while (!mbar_try(bar, ph)) {
      if (gtimer() - t0 > 1000000000ull) {
        timed_out = true;
        sh.err = 1;
        break;
      }
    }
  };
  int first_zero = -1;
  int pos[RT];  // positions of the thread's rows (-1: no such row)

  if (tid < NC) {
    // ================================ control warps ========================================
    // The step is one rolled loop body: the column index moves through the registers (the
    // update writes column c + 1 to place c), so that the body stays in the instruction caches
    // (eight unrolled steps waited for instructions a quarter of the time). Its chain is what
    // every CTA waits for, so it holds only what the next record needs: what a step stores
    // (multipliers, the pivot row's entries, its reciprocal) is written while the next step's
    // records are in flight, and what is rare (ties, zeros, Inf and NaN, the two rows whose
    // positions change) sits behind branches that are seldom taken.
    using K = key_t<T>;
    // FP64 multiply-adds (64 cycles each) are worth a branch around dead columns, where the
    // branches cost no spills
    constexpr bool kSlow = std::is_same<T, double>::value && RT <= 2;
    const uint32_t recv_a = smem_u32(&sh.recv[0][0][0]);
    const uint32_t ub_a = smem_u32(ub);
    T x[RT][LB];        // rows r0 + tid + s NC: the block's columns from the current one on
    uint32_t lm[RT];    // all ones while the row is to be eliminated, else 0
#pragma unroll
    for (int s = 0; s < RT; ++s) {
      const int row = r0 + tid + s * NC;
      pos[s] = row < R ? (p0 == 0 ? row : a.posg[row]) : -1;
      lm[s] = pos[s] >= p0 ? 0xffffffffu : 0u;
#pragma unroll
      for (int c = 0; c < LB; ++c)
        x[s][c] = (row < R && c < w) ? X[(int64_t)(p0 + c) * ldx + row] : T(0);
    }
    constexpr int LPR = MC <= 4 ? 4 : 8;  // lanes per destination of a record
    constexpr int RPW = 32 / LPR;
    const int ch = lane % LPR;
    // where this lane's chunk of the CTA's record and its completion go (first destination)
    const int rk = warp * RPW + lane / LPR;
    const uint32_t rdst = map_rank(recv_a + (uint32_t)((crank * MC + ch) * 16), rk < ncta ? rk : 0);
    const uint32_t rbar = map_rank(mbar_a, rk < ncta ? rk : 0);
    // lane r: where this CTA's mbarriers lie in the shared memory of the cluster's CTA r
    const uint32_t wbase = SOLO ? 0u : map_rank(mbar_a, lane < ncta ? lane : 0);
    bool nonfinite = false;
    T* Xj = X + (int64_t)p0 * ldx + r0 + tid;  // the step's column at the thread's first row
    // the step before, whose results are still to be stored
    T m[RT], P[LB + EPC + 2];
    T prp = T(1);
    int pwl = -1, pwrow = -1;
    bool pnz = false;
#pragma unroll
    for (int s = 0; s < RT; ++s) {
      m[s] = T(0);
    }
#pragma unroll
    for (int c = 0; c < LB + EPC + 2; ++c) P[c] = T(0);

    // stores of step jj (its column at Xc): the multipliers, to X and for the update warps, and
    // the pivot row's entries in the block's columns
    auto store_step = [&](int jj, T* Xc, bool keep) {
      const int i = jj & (LB - 1);
#pragma unroll
      for (int s = 0; s < RT; ++s) {
        if (lm[s] && pnz) Xc[s * NC] = m[s];
        if (keep) xs[jj * rs + tid + s * NC] = m[s];
      }
      if (tid == 0) {
        sh.prows[p0 - o0 + jj] = pwrow;
        sh.rp[p0 - o0 + jj] = prp;
      }
      if (warp == NCW - 1 && (uint32_t)pwl < (uint32_t)ROWS && (lane > 0 || pnz) &&
          lane < min(LB - i, w - jj)) {
        T v = P[0];
#pragma unroll
        for (int c = 1; c < LB; ++c) v = lane == c ? P[c] : v;
        Xc[(int64_t)lane * ldx + pwl - tid] = v;
      }
    };

    if (!SOLO) mbar_arm_if(tid == NC - 1, mbar_a, (uint32_t)(ncta * RC::chunks(0) * 16));
#pragma unroll 1
    for (int b0 = 0; b0 < w; b0 += LB) {
      const int bw = min(LB, w - b0);   // columns of the block
      const int rem = w - b0 - LB;      // panel columns after it (<= 0: last block)
      const int bp = b0 / LB & 1;       // its parity
      const int urow = (LB + rem + EPC - 1) / EPC;  // chunks of a published pivot row
      if (!SOLO && rem > 0)
        mbar_arm_if(tid == NC - 1, mbar_a + 16 + 8 * bp, (uint32_t)(LB * urow * 16));
#pragma unroll 1
      for (int i = 0; i < bw; ++i, Xj += ldx) {
        const int jj = b0 + i, j = p0 + jj;
        // records and mbarriers alternate by the step's parity (a block has an even number
        // of steps); the mbarriers start at phase 0 in every launch
        const int par = i & 1;
        // ---- the warp's candidate: its lane writes the record -------------------------------
        K kk[RT], key = 0;
#pragma unroll
        for (int s = 0; s < RT; ++s) {
          kk[s] = raw_key(and_mask(x[s][0], lm[s]));
          key = kk[s] > key ? kk[s] : key;
        }
        K wkey = warp_max(key);
        // the thread's best row, by a tree of selects; equal keys count as a tie below
        int kp = pos[0], krow = r0 + tid;
        T kv[LB];
        bool dup = false;
        {
          K tk[RT];
          int tp[RT], tr[RT];
          T tv[RT][LB];
#pragma unroll
          for (int s = 0; s < RT; ++s) {
            tk[s] = kk[s];
            tp[s] = pos[s];
            tr[s] = r0 + tid + s * NC;
#pragma unroll
            for (int c = 0; c < LB; ++c) tv[s][c] = x[s][c];
          }
#pragma unroll
          for (int h = 1; h < RT; h *= 2) {
#pragma unroll
            for (int s = 0; s + h < RT; s += 2 * h) {
              const bool take = tk[s + h] > tk[s];
              dup |= tk[s + h] == tk[s];
              tk[s] = take ? tk[s + h] : tk[s];
              tp[s] = take ? tp[s + h] : tp[s];
              tr[s] = take ? tr[s + h] : tr[s];
#pragma unroll
              for (int c = 0; c < LB; ++c) tv[s][c] = take ? tv[s + h][c] : tv[s][c];
            }
          }
          kp = tp[0];
          krow = tr[0];
#pragma unroll
          for (int c = 0; c < LB; ++c) kv[c] = tv[0][c];
        }
        uint32_t who = __ballot_sync(0xffffffffu, key == wkey);
        if (wkey >= inf_key<K>() || (who & (who - 1)) ||
            (RT > 1 && __any_sync(0xffffffffu, dup && key == wkey))) {
          // a tie, nothing but zeros, Inf or NaN: the smallest position among the largest
          nonfinite |= key >= inf_key<K>();
          key = 0;
#pragma unroll
          for (int s = 0; s < RT; ++s) {
            kk[s] = kk[s] > inf_key<K>() ? (K)0 : kk[s];
            key = kk[s] > key ? kk[s] : key;
          }
          wkey = warp_max(key);
          kp = kNone;
#pragma unroll
          for (int s = 0; s < RT; ++s) {
            const bool take = kk[s] == wkey && lm[s] && pos[s] < kp;
            kp = take ? pos[s] : kp;
            krow = take ? r0 + tid + s * NC : krow;
#pragma unroll
            for (int c = 0; c < LB; ++c) kv[c] = take ? x[s][c] : kv[c];
          }
          const int wp = (int)__reduce_min_sync(0xffffffffu, (uint32_t)kp);
          who = __ballot_sync(0xffffffffu, kp == wp);
          who &= 0u - who;
          if (wkey == 0) kv[0] = T(0);  // also in place of a NaN, which does not count
        }
        {
          const bool mine = who >> lane & 1u;
          const int kpr = kp == kNone ? kNone : kp << 16 | krow;
          const uint32_t rec = smem_u32(&sh.wrec[par][warp][0]);
          if (NCW > 1 && mine) {
            sh.wkey[par][warp] = wkey;
            sh.wpr[par][warp] = kpr;
          }
          sts16_if(mine, rec, pack_hdr(kv[0], kpr, kv[1], kv[2]));
#pragma unroll
          for (int q = 1; q < MC; ++q) {
            T v[EPC];
#pragma unroll
            for (int e = 0; e < EPC; ++e) {
              const int c = 1 + E0 + (q - 1) * EPC + e;
              v[e] = c < LB ? kv[c < LB ? c : 0] : T(0);
            }
            sts16_if(mine, rec + 16 * q, pack_chunk(v));
          }
        }
        if (NCW > 1) bar_sync(4, NC);
        else __syncwarp();
        // ---- the CTA's winner goes to every CTA of the cluster: a record is one piece, since
        // the cost of the exchange is its packets (a piece per destination) more than its bytes
        int ow = 0;
        if (NCW > 1 && (SOLO || warp * RPW < ncta)) {  // every lane compares the warps' keys
          K k[NCW], top = 0;
#pragma unroll
          for (int g = 0; g < NCW; ++g) {
            k[g] = sh.wkey[par][g];
            top = k[g] > top ? k[g] : top;
          }
          int ties = 0;
#pragma unroll
          for (int g = NCW - 1; g >= 0; --g) {
            ties += k[g] == top;
            ow = k[g] == top ? g : ow;
          }
          if (ties > 1) {
            int p = kNone;
#pragma unroll
            for (int g = 0; g < NCW; ++g) {
              const int pg = sh.wpr[par][g];
              const bool take = k[g] == top && pg < p;
              p = take ? pg : p;
              ow = take ? g : ow;
            }
          }
        }
        if (!SOLO && warp * RPW < ncta) {
          const uint4 v = sh.wrec[par][ow][ch < MC ? ch : 0];
          const int nch = RC::chunks(i);
          st_async16_if(ch < nch && rk < ncta, rdst + (uint32_t)(par * 16 * MC * 16), v,
                        rbar + 8 * par);
          if (NCW * RPW < 16)
            for (int r = rk + NCW * RPW; r < ncta; r += NCW * RPW)
              st_async16_if(ch < nch, map_rank(recv_a + (uint32_t)(((par * 16 + crank) * MC + ch) * 16), r),
                            v, map_rank(mbar_a + 8 * par, r));
        }
        // ---- meanwhile: the step before is stored, the next step's mbarrier armed ------------
        if (i > 0) store_step(jj - 1, Xj - ldx, rem > 0 || tail);
        if (!SOLO) {
          mbar_arm_if(tid == NC - 1 && jj + 1 < w, mbar_a + 8 * (par ^ 1),
                      (uint32_t)(ncta * RC::chunks((i + 1) & (LB - 1)) * 16));
          wait(mbar_a + 8 * par, (uint32_t)((i >> 1) & 1));
        }
        // ---- winner among the records, in every warp ----------------------------------------
        const uint4* recs = SOLO ? &sh.wrec[par][ow][0] : &sh.recv[par][0][0];
        T rp;  // reciprocal of the winner: every lane takes its own record's meanwhile
        if (!SOLO) {
          const uint4 h = recs[(lane < ncta ? lane : 0) * MC];
          T hv, n1, n2;
          unpack_hdr(h, hv, n1, n2);
          const K k = raw_key(hv);  // lanes past the records repeat the first
          const bool top = k == warp_max(k);
          rp = rcp_piv(hv);
          uint32_t wh = __ballot_sync(0xffffffffu, top && lane < ncta);
          if (wh & (wh - 1)) {
            const int p = (int)__reduce_min_sync(0xffffffffu, top ? h.y : (uint32_t)kNone);
            wh = __ballot_sync(0xffffffffu, top && lane < ncta && (int)h.y == p);
          }
          const int win = __ffs(wh) - 1;
          rp = shfl_t(rp, win);
          recs += win * MC;
        }
        int wpr;
        {
          const uint4 h = recs[0];
          unpack_hdr(h, P[0], P[1], P[2]);  // the pivot row in the block's columns
          wpr = (int)h.y;
#pragma unroll
          for (int q = 1; q < MC; ++q) {
            T v[EPC];
            unpack_chunk(recs[q], v);
#pragma unroll
            for (int e = 0; e < EPC; ++e) P[1 + E0 + (q - 1) * EPC + e] = v[e];
          }
        }
        if (timed_out) {  // the records may not have come: no pivot, positions stay as they are
          wpr = kNone;
          P[0] = T(0);
        }
        if (SOLO) rp = rcp_piv(P[0]);
        const bool nz = raw_key(P[0]) != (K)0;  // false too where there is no candidate
        prp = nz ? rp : T(1);
        pnz = nz;
        if (CROUT) {
#pragma unroll
          for (int c = 1; c < LB; ++c)
            if (!kSlow || c < LB - i) P[c] = P[c] * prp;
        }
        // positions after the exchange of positions j and the winner's
        const int wpos = wpr >> 16;
        pwrow = wpr & 0xffff;
        pwl = pwrow - r0;
        {
          bool any = (uint32_t)pwl < (uint32_t)ROWS && pwl % NC == tid;
#pragma unroll
          for (int s = 0; s < RT; ++s) any |= pos[s] == j;
          if (any && wpr != kNone) {
#pragma unroll
            for (int s = 0; s < RT; ++s) {
              if (pos[s] == wpos) {  // the winner's row
                pos[s] = j;
                lm[s] = 0;
                if (!nz) Xj[s * NC] = x[s][0];  // a zero (or NaN) pivot
              } else if (pos[s] == j) {
                pos[s] = wpos;
              }
            }
          }
        }
        // multipliers of the live rows; the update of the block's columns
#pragma unroll
        for (int s = 0; s < RT; ++s) {
          m[s] = and_mask(CROUT ? x[s][0] : x[s][0] * rp, lm[s]);
        }
        if (!nz) {  // nothing is eliminated; the column keeps its values
          if (first_zero < 0) first_zero = j;
          if (wpr == kNone) pwl = pwrow = -1;
#pragma unroll
          for (int s = 0; s < RT; ++s) {
            if (lm[s]) Xj[s * NC] = x[s][0];
            m[s] = T(0);
          }
        }
#pragma unroll
        for (int s = 0; s < RT; ++s) {
          x[s][0] = m[s] != T(0) ? fma(-m[s], P[1], x[s][1]) : x[s][1];
#pragma unroll
          for (int c = 1; c + 1 < LB; ++c)
            if (!kSlow || c + 1 < LB - i) x[s][c] = fma(-m[s], P[c + 1], x[s][c + 1]);
        }
      }
      store_step(b0 + bw - 1, Xj - ldx, rem > 0 || tail);
      if (rem > 0) {
        // ---- end of a block: its pivot rows go to every CTA ----------------------------------
        bar_sync(2, NT);  // xs holds the panel through the block before
        if (NCW > 1) bar_sync(4, NC);  // multipliers, prows, rp
        else __syncwarp();
        const T* xb = xs + b0 * rs;  // the block's multipliers, then the panel's later columns
        const int brow = lane < LB ? sh.prows[p0 - o0 + b0 + lane] - r0 : -1;
        uint32_t own = __ballot_sync(0xffffffffu, (uint32_t)brow < (uint32_t)ROWS);
        while (own) {
          const int t = __ffs(own) - 1;
          own &= own - 1;
          const int lr = __shfl_sync(0xffffffffu, brow, t);
          for (int ck = lane; ck < 32 * ((urow + 31) / 32); ck += 32) {
            constexpr uint32_t ckm = 0xffffffffu;
            T v[EPC];
#pragma unroll
            for (int e = 0; e < EPC; ++e) {
              const int c = ck * EPC + e;
              v[e] = c < LB + rem ? xb[c * rs + lr] : T(0);
            }
            const uint4 pv = pack_chunk(v);
            const uint32_t at = (uint32_t)(sizeof(T) * ((bp * LB + t) * ubw) + 16 * ck);
            if (SOLO) {
              if (warp == 0 && ck < urow)
                *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(ub) + at) = pv;
            } else {
#pragma unroll
              for (int k = 0; k < 16 / NCW; ++k) {
                const uint32_t peer = __shfl_sync(ckm, wbase, (warp + k * NCW) & 31);
                st_async16_if(ck < urow && warp + k * NCW < ncta, peer + (ub_a - mbar_a) + at, pv,
                              peer + 16 + 8 * bp);
              }
            }
          }
        }
        if (SOLO && NCW > 1) bar_sync(4, NC);
        else __syncwarp();
        bar_arrive(1, NT);
        // ---- the next block's columns: their U, then the rank-8 update of the rows ----------
#pragma unroll
        for (int s = 0; s < RT; ++s)
#pragma unroll
          for (int c = 0; c < LB; ++c)
            x[s][c] = c < rem ? xb[(LB + c) * rs + tid + s * NC] : T(0);
        if (!SOLO) wait(mbar_a + 16 + 8 * bp, (uint32_t)((b0 / LB >> 1) & 1));
        if (lane < LB) {
          T u[LB];
          solve_block<T, CROUT>(ub + bp * LB * ubw, ubw, sh.rp + (p0 - o0 + b0), lane, u);
#pragma unroll
          for (int q = 0; q < LB; ++q) sh.uc[warp][q][lane] = u[q];
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < LB; ++q) {
          T uv[LB];
#pragma unroll
          for (int c = 0; c < LB; c += EPC) {
            T v[EPC];
            unpack_chunk(*reinterpret_cast<const uint4*>(&sh.uc[warp][q][c]), v);
#pragma unroll
            for (int e = 0; e < EPC; ++e) uv[c + e] = v[e];
          }
#pragma unroll
          for (int s = 0; s < RT; ++s) {
            const T mq = xb[q * rs + tid + s * NC];
#pragma unroll
            for (int c = 0; c < LB; ++c)
              if (!kSlow || c < rem) x[s][c] = fma(-mq, uv[c], x[s][c]);
          }
        }
        __syncwarp();  // uc is free for the next block
      }
    }
    if (nonfinite) sh.nonfinite = 1;
    bar_sync(2, NT);
  } else {
    // ================================ update warps =========================================
    const int ut = tid - NC;
    // the panel's columns after the first block: every copy in flight at once (16-byte ones
    // where X's columns start on 16-byte boundaries; their padding rows are never used)
    if (((uintptr_t)X & 15u) == 0 && (ldx * (int64_t)sizeof(T)) % 16 == 0) {
      const int nq = min(ROWS, max(R - r0, 0) + EPC - 1) / EPC;
      for (int c = LB; c < w; ++c)
        for (int q = ut; q < nq; q += kLuUpd)
          lr_cp16(xs + c * rs + q * EPC, X + (int64_t)(p0 + c) * ldx + r0 + q * EPC);
    } else {
      for (int c = LB; c < w; ++c)
        for (int r = ut; r < ROWS && r0 + r < R; r += kLuUpd)
          lr_cp<(int)sizeof(T)>(xs + c * rs + r, X + (int64_t)(p0 + c) * ldx + r0 + r);
    }
    lr_cp_commit();
    lr_cp_wait<0>();
    bar_arrive(2, NT);
    for (int b = 0; w - b * LB - LB > 0; ++b) {
      const int rem = w - b * LB - LB, bp = b & 1, j0 = p0 + b * LB;
      bar_sync(1, NT);
      if (!SOLO) wait(mbar_a + 16 + 8 * bp, (uint32_t)((b >> 1) & 1));
      // U of the block's pivot rows in the panel's later columns, one thread per column
      for (int c = ut; c < rem; c += kLuUpd) {
        T u[LB];
        solve_block<T, CROUT>(ub + bp * LB * ubw, ubw, sh.rp + (p0 - o0 + b * LB), c, u);
#pragma unroll
        for (int q = 0; q < LB; ++q) {
          if (sizeof(T) == 4) us[(c * LB + q) * 2] = us[(c * LB + q) * 2 + 1] = -u[q];
          else us[c * LB + q] = -u[q];
        }
      }
      bar_sync(3, kLuUpd);
      constexpr int UQ = sizeof(T) == 4 ? 2 : 1;
      for (int t = crank; t < LB; t += ncta) {
        const int prow = sh.prows[p0 - o0 + b * LB + t];
        if (prow >= 0)
          for (int c = ut; c < rem; c += kLuUpd)
            X[(int64_t)(j0 + LB + c) * ldx + prow] = -us[(c * LB + t) * UQ];
      }
      // rank-8 update of the columns after the next block: a thread takes a chunk of rows
      // and every CG-th column
      constexpr int NQ = ROWS / EPC;                          // row chunks
      constexpr int CG = NQ >= kLuUpd ? 1 : kLuUpd / NQ;      // column groups
      for (int q = ut % (NQ < kLuUpd ? NQ : kLuUpd); q < NQ; q += kLuUpd) {
        RankUpdate<T> up;
        up.load(xs + b * LB * rs, rs, q * EPC);
        T* xq = xs + (b + 1) * LB * rs + q * EPC;
        int c = LB + (CG > 1 ? ut / NQ : 0);
        for (; c + 3 * CG < rem; c += 4 * CG)
          up.template apply<4>(xq + c * rs, CG * rs, us + c * LB * UQ, CG * LB * UQ);
        for (; c < rem; c += CG) up.template apply<1>(xq + c * rs, 0, us + c * LB * UQ, 0);
      }
      bar_arrive(2, NT);
    }
  }

  constexpr int NW = NT / 32;
  __syncthreads();
  const int32_t* prows = sh.prows;
  if (tail) {
    // ---- the pivot rows of the later columns: u = L11^-1 x (unit lower; Crout divides by the
    // pivots). Every CTA sends its own rows of L11 to the cluster: this panel's multipliers
    // from shared memory, those of the block's earlier panels from X.
    T* const L11 = reinterpret_cast<T*>(smem_raw + lay.l11);  // [W][LP], zero above
    const int LP = W + 1;
    if (!SOLO) mbar_arm_if(tid == 0, mbar_a + 32, (uint32_t)(W * W * sizeof(T)));
    for (int t = tid; t < p0 - o0; t += NT) {
      const int prow = a.psg[o0 + t];
      sh.prows[t] = prow;
      if (CROUT) {
        const T pv = prow >= 0 ? X[(int64_t)(o0 + t) * ldx + prow] : T(0);
        sh.rp[t] = raw_key(pv) != 0 ? rcp_piv(pv) : T(1);
      }
    }
    __syncthreads();
    const uint32_t wbase = SOLO ? 0u : map_rank(mbar_a, lane < ncta ? lane : 0);
    const uint32_t l11_a = smem_u32(L11) - mbar_a;
    for (int t = warp; t < W; t += NW) {
      const int lr = prows[t] - r0;
      if (prows[t] < 0 || (uint32_t)lr >= (uint32_t)ROWS) continue;
      for (int e = lane; e < (W + 31) / 32 * 32; e += 32) {
        T v = T(0);
        if (e < t) v = e < p0 - o0 ? X[(int64_t)(o0 + e) * ldx + prows[t]] : xs[(e - (p0 - o0)) * rs + lr];
        const uint32_t at = (uint32_t)((t * LP + e) * sizeof(T));
        if (SOLO) {
          if (e < W) L11[t * LP + e] = v;
        } else {
#pragma unroll 4
          for (int r = 0; r < 16; ++r) {
            const int to = (crank + r) & 15;  // each CTA starts at itself
            const uint32_t peer = __shfl_sync(0xffffffffu, wbase, to);
            st_async_if(e < W && to < ncta, peer + l11_a + at, v, peer + 32);
          }
        }
      }
    }
    if (SOLO) __syncthreads();
    else wait(mbar_a + 32, 0);
    // a warp takes two columns at once: two chains of shuffles and multiply-adds in flight
    constexpr int NQ = 3;  // W <= 96
    int prq[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) prq[q] = lane + 32 * q < W ? prows[lane + 32 * q] : -1;
    for (int c = p0 + w + crank * NW + warp; c < cu; c += 2 * ncta * NW) {
      const int c2 = c + ncta * NW;
      T u[2][NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        u[0][q] = prq[q] >= 0 ? X[(int64_t)c * ldx + prq[q]] : T(0);
        u[1][q] = prq[q] >= 0 && c2 < cu ? X[(int64_t)c2 * ldx + prq[q]] : T(0);
      }
      T fin[2][NQ];
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const T* lp[NQ];  // the lane's rows of L11 (lanes past W repeat the last)
#pragma unroll
        for (int qq = 0; qq < NQ; ++qq) lp[qq] = L11 + min(lane + 32 * qq, W - 1) * LP;
#pragma unroll 4
        for (int s = 32 * q; s < min(W, 32 * q + 32); ++s) {
          T u0 = shfl_t(u[0][q], s - 32 * q), u1 = shfl_t(u[1][q], s - 32 * q);
          if (CROUT) {
            const T r = sh.rp[s];
            u0 = u0 * r;
            u1 = u1 * r;
          }
          fin[0][q] = lane == s - 32 * q ? u0 : fin[0][q];
          fin[1][q] = lane == s - 32 * q ? u1 : fin[1][q];
#pragma unroll
          for (int qq = q; qq < NQ; ++qq) {  // rows up to s: times zero, and final already
            const T l = lp[qq][s];
            u[0][qq] = fma(-l, u0, u[0][qq]);
            u[1][qq] = fma(-l, u1, u[1][qq]);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const int t = lane + 32 * q;
        if (t < W) {
          T* d = static_cast<T*>(a.u12) + (int64_t)t * a.ldu;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int cc = h ? c2 : c;
            if (cc < cu) {
              if (prq[q] >= 0) X[(int64_t)cc * ldx + prq[q]] = fin[h][q];
              d[cc] = prq[q] >= 0 ? fin[h][q] : T(0);
            }
          }
        }
      }
    }
  }

  // persist the positions for the next panel; the last panel writes P (gather form)
  const bool last = (p0 + w >= C);
  if (tid < NC) {
#pragma unroll
    for (int s = 0; s < RT; ++s)
      if (pos[s] >= 0) a.posg[r0 + tid + s * NC] = pos[s];
  }
  if (crank == 0)
    for (int t = tid; t < w; t += NT) a.psg[p0 + t] = prows[p0 - o0 + t];
  if (last && tid < NC) {
#pragma unroll
    for (int s = 0; s < RT; ++s)
      if (pos[s] >= 0) a.perm[pos[s]] = r0 + tid + s * NC;
  }
  if (tid == 0) {
    if (crank == 0 && a.zero_step && first_zero >= 0) atomicCAS(a.zero_step, -1, first_zero);
    if (sh.nonfinite && a.nonfinite) atomicOr(a.nonfinite, 1);
    if (sh.err && a.status) atomicExch(a.status, RLU_ETIMEOUT);
  }
  if (!SOLO) cl.sync();
}

template <typename T, bool CROUT, int RT, int NC, bool SOLO>
__global__ void __launch_bounds__(NC + kLuUpd, 1) k_lu_reg(LuArgs a) {
  lu_reg_body<T, CROUT, RT, NC, SOLO>(a);
}

// Batched form: cluster c of the launch factors problem table[c] (one panel: pw = C).
template <typename T, bool CROUT, int RT, int NC, bool SOLO>
__global__ void __launch_bounds__(NC + kLuUpd, 2) k_lu_reg_batched(const LuArgs* __restrict__ table,
                                                                   int pw) {
  const int csize = (int)cg::this_cluster().num_blocks();
  LuArgs a = table[blockIdx.x / csize];
  a.nb = pw;
  lu_reg_body<T, CROUT, RT, NC, SOLO>(a);
}

// Rank-w update (w <= 96) of the columns [c_begin, c_end) of every row whose position is at
// least p0 + w: X[r][c] -= sum_s X[r][p0 + s] U[s][c], U = the solved pivot rows, dense in
// u12 (row s at u12 + s * ldu). A CTA takes 256 rows (128 threads, 2 rows each) and nch
// chunks of 32 columns. Its rows' multipliers are copied to shared memory once and each
// chunk of U while the previous chunk is computed (cp.async, many copies in flight); every
// thread keeps 2 x 32 accumulators in registers. vec: X's columns start on 16-byte
// boundaries, so the multipliers move in 16-byte copies.
static constexpr int TR_T = 128;
static constexpr int TR_R = 256;

template <typename T>
__global__ void __launch_bounds__(TR_T) k_lu_trail(T* __restrict__ X, int64_t ldx, int R,
                                                  int c_begin, int c_end, int p0, int w,
                                                  const int32_t* __restrict__ posg,
                                                  const T* __restrict__ u12, int64_t ldu,
                                                  int nch, bool vec) {
  extern __shared__ __align__(16) unsigned char tr_smem[];
  T* Ls = reinterpret_cast<T*>(tr_smem);  // [w][TR_R] multipliers of this CTA's rows
  T* Us = Ls + (size_t)w * TR_R;          // [2][w][LR_CH] chunks of U
  const int tid = threadIdx.x;
  const int rb = (int)blockIdx.x * TR_R;
  const int r0 = rb + tid, r1 = rb + tid + TR_T;
  const bool u0 = r0 < R && posg[r0] >= p0 + w;
  const bool u1 = r1 < R && posg[r1] >= p0 + w;
  // the multipliers: rows rb .. rb + 255 of columns p0 .. p0 + w - 1 (rows past the column's
  // storage, ldx, read as zero)
  constexpr int EPC = 16 / (int)sizeof(T);
  if (vec) {
    for (int e = tid; e < w * (TR_R / EPC); e += TR_T) {
      const int s = e / (TR_R / EPC), i = (e % (TR_R / EPC)) * EPC;
      T* d = Ls + (size_t)s * TR_R + i;
      if (rb + i + EPC <= ldx) {
        lr_cp16(d, X + (int64_t)(p0 + s) * ldx + rb + i);
      } else {
#pragma unroll
        for (int u = 0; u < EPC; ++u) d[u] = T(0);
      }
    }
  } else {
    for (int e = tid; e < w * TR_R; e += TR_T) {
      const int s = e / TR_R, i = e % TR_R;
      if (rb + i < ldx) lr_cp<sizeof(T)>(Ls + e, X + (int64_t)(p0 + s) * ldx + rb + i);
      else Ls[e] = T(0);
    }
  }
  const int cb = c_begin + (int)blockIdx.y * nch * LR_CH;
  int nc = (c_end - cb + LR_CH - 1) / LR_CH;
  nc = nc < nch ? nc : nch;
  auto issue = [&](int ch) {  // chunk ch of U into buffer ch & 1
    const int c0 = cb + ch * LR_CH, cw = min(LR_CH, c_end - c0);
    T* d = Us + (size_t)(ch & 1) * w * LR_CH;
    for (int e = tid; e < w * LR_CH; e += TR_T) {
      const int s = e / LR_CH, q = e % LR_CH;
      if (q < cw) lr_cp<sizeof(T)>(d + e, u12 + (int64_t)s * ldu + c0 + q);
      else d[e] = T(0);
    }
  };
  issue(0);
  lr_cp_commit();
  for (int ch = 0; ch < nc; ++ch) {
    const int c0 = cb + ch * LR_CH, cw = min(LR_CH, c_end - c0);
    if (ch + 1 < nc) issue(ch + 1);
    lr_cp_commit();
    T acc0[LR_CH], acc1[LR_CH];
#pragma unroll
    for (int q = 0; q < LR_CH; ++q) {
      acc0[q] = (u0 && q < cw) ? X[(int64_t)(c0 + q) * ldx + r0] : T(0);
      acc1[q] = (u1 && q < cw) ? X[(int64_t)(c0 + q) * ldx + r1] : T(0);
    }
    lr_cp_wait<1>();  // everything but the chunk just issued has landed
    __syncthreads();
    const T* U = Us + (size_t)(ch & 1) * w * LR_CH;
#pragma unroll 2
    for (int s = 0; s < w; ++s) {
      const T l0 = Ls[s * TR_R + tid], l1 = Ls[s * TR_R + tid + TR_T];
#pragma unroll
      for (int q = 0; q < LR_CH; q += 4) {
        T uv[4];
        ld4(&U[s * LR_CH + q], uv);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          acc0[q + v] = fma(-l0, uv[v], acc0[q + v]);
          acc1[q + v] = fma(-l1, uv[v], acc1[q + v]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < LR_CH; ++q) {
      if (u0 && q < cw) X[(int64_t)(c0 + q) * ldx + r0] = acc0[q];
      if (u1 && q < cw) X[(int64_t)(c0 + q) * ldx + r1] = acc1[q];
    }
    __syncthreads();  // buffer ch & 1 is free for chunk ch + 2
  }
  lr_cp_wait<0>();
}

// Launches k_lu_trail on the columns [c_begin, c_end): chunks of 32 columns are grouped
// per CTA only while the grid keeps at least two CTAs per SM.
template <typename T>
static int32_t launch_trail(T* X, int64_t ldx, int R, int c_begin, int c_end, int p0, int w,
                            const int32_t* posg, const T* u12, int64_t ldu, cudaStream_t s) {
  const int rows = (int)ceil_div(R, TR_R);
  const int chunks = (int)ceil_div(c_end - c_begin, LR_CH);
  int nch = 1;
  while (nch < 4 && (int64_t)rows * ceil_div(chunks, nch + 1) >= 2 * sm_count()) ++nch;
  const size_t smem = sizeof(T) * (size_t)w * (TR_R + 2 * LR_CH);
  RLU_TRY(allow_smem(k_lu_trail<T>));
  const bool vec = ((uintptr_t)X % 16 == 0) && (ldx * (int64_t)sizeof(T)) % 16 == 0;
  const dim3 grid((unsigned)rows, (unsigned)ceil_div(chunks, nch));
  k_lu_trail<T><<<grid, TR_T, smem, s>>>(X, ldx, R, c_begin, c_end, p0, w, posg, u12, ldu, nch,
                                         vec);
  return last_launch_status();
}

template <typename T, int RT, int NC>
static size_t lr_smem_bytes(int pw, int tw) {
  return (size_t)LrLayout<T>((int)sizeof(LrShared<T, NC / 32>), NC * RT, pw, tw).total;
}

// A rank-w trailing update: large ones (rank >= 64 over >= 128 columns) on the tensor cores
// (FP32 with scratch for U^T's TF32 parts), the others (and where that form does not apply)
// on the SIMT kernel, whose launch costs less than the tensor-core form's set-up.
template <typename T>
static int32_t trail(const LuArgs& in, T* X, int c_begin, int c_end, int p0, int w, T* U12,
                     cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    if (in.u12t && w >= 64 && c_end - c_begin >= 128) {
      const int32_t st = umma3_trail(X, in.ldx, in.R, c_begin, c_end, p0, w, in.posg, U12,
                                     in.ldu, static_cast<float*>(in.u12t), in.status, s);
      if (st != RLU_EUNSUPPORTED) return st;
    }
  }
  return launch_trail<T>(X, in.ldx, in.R, c_begin, c_end, p0, w, in.posg, U12, in.ldu, s);
}

template <typename T, bool CROUT, int RT, int NC, int pw_max, bool SOLO = false>
static int32_t try_launch(const LuArgs& in, cudaStream_t s, bool* launched) {
  *launched = false;
  const int ncta = (int)ceil_div(in.R, NC * RT);
  if (ncta > (SOLO ? 1 : 16)) return RLU_OK;
  int dev = 0;
  RLU_CUDA_TRY(cudaGetDevice(&dev));
  int optin = 0;
  RLU_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  // blocks of whole panels, about 64 columns (panels of 64 or more columns: each its own); the
  // last panel of a block solves the block's pivot rows (at most 96) for the columns after it
  const int pw = min(in.C, pw_max);
  int np = (64 + pw_max / 2) / pw_max;
  // complex: a two-panel block's 72-row pivot solve (complex shuffles and FMAs) costs more
  // than the trailing columns' extra reads save, so every panel is its own block (frlu_4096:
  // 2.52 -> 2.39 ms)
  if (np < 1 || std::is_same<T, cf32>::value) np = 1;
  const int wo = np * pw_max;
  const size_t bytes = lr_smem_bytes<T, RT, NC>(pw, in.C > wo ? wo : in.C > pw ? pw : 0);
  if (bytes > (size_t)optin) return RLU_OK;
  auto kern = k_lu_reg<T, CROUT, RT, NC, SOLO>;
  RLU_TRY(allow_smem(kern));
  RLU_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ncta;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(ncta);
  cfg.blockDim = dim3(NC + kLuUpd);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (ncta > 8) {
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) != cudaSuccess || nclusters < 1) {
      cudaGetLastError();
      return RLU_OK;
    }
  }
  // no position state or pivot-row buffer: the one-launch kernel takes the problem
  if (!in.posg || !in.psg || !in.u12) return RLU_OK;
  LuArgs a = in;
  a.nb = pw;
  T* X = static_cast<T*>(in.X);
  T* U12 = static_cast<T*>(in.u12);
  for (int o0 = 0; o0 < in.C; o0 += wo) {
    const int o1 = min(in.C, o0 + wo);
    for (int p0 = o0; p0 < o1; p0 += pw_max) {
      a.p0 = p0;
      a.pw = min(pw_max, o1 - p0);
      const int p1 = p0 + a.pw;
      const bool last = p1 == o1;  // the block's pivot rows for the columns after the block
      a.o0 = last && o1 < in.C ? o0 : p0;
      a.cu = last ? in.C : o1;     // else the panel's, for the rest of the block
      RLU_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, a));
      RLU_TRY(last_launch_status());
      *launched = true;
      if (p1 < a.cu) RLU_TRY(trail<T>(in, X, p1, a.cu, a.o0, p1 - a.o0, U12, s));
    }
  }
  return RLU_OK;
}

template <typename T, bool CROUT>
static int32_t launch_reg_t(const LuArgs& a, cudaStream_t s, bool* launched) {
  // threads per CTA, rows per thread and panel columns by the number of rows. The eight-row forms
  // of 8-byte elements spill (1.2 to 1.4 KB a thread) and still win over the ones they replaced:
  // FP64 factorizations of 20000 x 1000, k = 40, 6.6 -> 5.3 ms and 32768 x 600, k = 76, 14.0 ->
  // 12.1; fast randomized LUs of 20000 x 1000, k = 40, 1.48 -> 1.40 ms and 30000 x 1024, k = 60,
  // 1.80 -> 1.69.
  const int R = a.R;
  auto go = [&](int rows, auto f) -> int32_t {
    return (!*launched && R <= rows) ? f() : (int32_t)RLU_OK;
  };
#define RLU_LU_TRY(rows, ...) \
  RLU_TRY(go(rows, [&] { return try_launch<T, CROUT, __VA_ARGS__>(a, s, launched); }))
  if constexpr (std::is_same<T, float>::value) {
    RLU_LU_TRY(128, 1, 128, 76, true);
    RLU_LU_TRY(256, 2, 128, 76, true);
    RLU_LU_TRY(512, 4, 128, 76, true);
    RLU_LU_TRY(16 * 128, 1, 128, 76);
    RLU_LU_TRY(16 * 256, 2, 128, 76);
    RLU_LU_TRY(16 * 512, 4, 128, 76);
    RLU_LU_TRY(16 * 1024, 4, 256, 36);
    RLU_LU_TRY(16 * 2048, 8, 256, 24);
  } else {
    RLU_LU_TRY(16 * 32, 1, 32, 36);
    RLU_LU_TRY(16 * 64, 1, 64, 36);
    RLU_LU_TRY(16 * 128, 1, 128, 76);
    RLU_LU_TRY(16 * 256, 2, 128, 76);
    RLU_LU_TRY(16 * 512, 4, 128, 36);
    RLU_LU_TRY(16 * 1024, 4, 256, 18);
    RLU_LU_TRY(16 * 2048, 8, 256, 8);
  }
#undef RLU_LU_TRY
  return RLU_OK;
}

int32_t launch_lu_reg(int32_t dtype, bool crout, const LuArgs& a, cudaStream_t s, bool* launched) {
  *launched = false;
  if (dtype == RLU_F64) return crout ? launch_reg_t<double, true>(a, s, launched) : launch_reg_t<double, false>(a, s, launched);
  if (dtype == RLU_F32) return crout ? launch_reg_t<float, true>(a, s, launched) : launch_reg_t<float, false>(a, s, launched);
  if (dtype == kLuC64) return crout ? launch_reg_t<cf32, true>(a, s, launched) : launch_reg_t<cf32, false>(a, s, launched);
  return RLU_OK;
}

// Batched LUs of problems that fit one panel (C <= 76 FP32 columns, R <= 16 x rows_per_cta): the
// table on the device is grouped by cluster size (ceil(R / rows_per_cta) CTAs); group g starts at
// table entry first[g] and holds count[g] problems. rows_per_cta is 512 or 256 (twice as many
// CTAs per problem). A panel of 76 columns of 512 rows takes more than half an SM's shared
// memory, and a step of one CTA leaves its SM idle while it waits; the groups of 512-row CTAs are
// therefore launched in two parts, up to 48 columns (108 KB a CTA) and more, and no CTA takes
// more than 128 registers a thread, so that two share an SM. With the longest LUs of a group
// first, 512 problems (m <= 2048, k <= 64) 1239 -> 1168 us, of which 16 us are the order of the C
// product's tiles.
template <int RT>
static int32_t lu_batched_group(bool crout, const LuArgs* table_dev, int first, int count, int g,
                                int pw, cudaStream_t s) {
  using T = float;
  constexpr int NC = 128;
  int dev = 0;
  RLU_CUDA_TRY(cudaGetDevice(&dev));
  int optin = 0;
  RLU_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  const size_t bytes = lr_smem_bytes<T, RT, NC>(pw, 0);
  if (bytes > (size_t)optin) return RLU_EUNSUPPORTED;
  auto kern = g == 1 ? (crout ? k_lu_reg_batched<T, true, RT, NC, true>
                              : k_lu_reg_batched<T, false, RT, NC, true>)
                    : (crout ? k_lu_reg_batched<T, true, RT, NC, false>
                             : k_lu_reg_batched<T, false, RT, NC, false>);
  RLU_TRY(allow_smem(kern));
  RLU_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = g;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(g * count));
  cfg.blockDim = dim3(NC + kLuUpd);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  RLU_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, table_dev + first, pw));
  return last_launch_status();
}

int32_t launch_lu_reg_batched(bool crout, int rows_per_cta, const LuArgs* table_dev,
                              const int* first, const int* count, const int* wide,
                              cudaStream_t s, const LuFork* fork) {
  if (rows_per_cta != 512 && rows_per_cta != 256) return RLU_EINVAL;
  struct Part {
    int g, first, count, pw;
  } parts[2 * kLuGroups];
  int np = 0;
  auto add = [&](int g) {
    if (wide[g] > 0) parts[np++] = {g, first[g], wide[g], 76};
    if (count[g] > wide[g]) parts[np++] = {g, first[g] + wide[g], count[g] - wide[g], kLuNarrow};
  };
  for (int g = 16; g >= 1; --g) add(g);  // widest clusters first
  for (int g : {17, 18}) add(g);         // one CTA for small problems, several per SM
  const bool par = fork != nullptr && np > 1;
  if (par) RLU_CUDA_TRY(cudaEventRecord(fork->fork, s));
  int32_t st = RLU_OK;
  int used = 0;  // helper streams that wait for the fork
  for (int i = 0; i < np && st == RLU_OK; ++i) {
    const Part& p = parts[i];
    cudaStream_t gs = s;
    if (par) {
      gs = fork->hs[i % kLuSide];
      if (i < kLuSide) {
        if (cudaStreamWaitEvent(gs, fork->fork, 0) != cudaSuccess) {
          st = RLU_ECUDA;
          break;
        }
        ++used;
      }
    }
    if (p.g == 17)
      st = lu_batched_group<1>(crout, table_dev, p.first, p.count, 1, p.pw, gs);
    else if (p.g == 18)
      st = lu_batched_group<2>(crout, table_dev, p.first, p.count, 1, p.pw, gs);
    else if (rows_per_cta == 512)
      st = lu_batched_group<4>(crout, table_dev, p.first, p.count, p.g, p.pw, gs);
    else
      st = lu_batched_group<2>(crout, table_dev, p.first, p.count, p.g, p.pw, gs);
  }
  // joined also after an error: what follows on s comes after everything launched above
  for (int i = 0; i < used; ++i) {
    if (cudaEventRecord(fork->join[i], fork->hs[i]) != cudaSuccess ||
        cudaStreamWaitEvent(s, fork->join[i], 0) != cudaSuccess)
      st = st == RLU_OK ? (int32_t)RLU_ECUDA : st;
  }
  return st;
}

}  // namespace rlu
