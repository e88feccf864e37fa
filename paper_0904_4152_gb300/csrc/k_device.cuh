// Device code shared by the V-cycle kernels (k_*.cu): programmatic dependent
// launch, the debug build's index checks, precision policies and loads, the deterministic norm
// sums and the lagged convergence test, the transfer formulas, and the mbarrier / bulk-copy helpers.
#pragma once

#include <type_traits>

#include "hn_internal.h"
#include "k_convert.cuh"

namespace hn {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// Programmatic dependent launch: a kernel lets its successor in the stream launch as soon as all
// of its blocks are running (launch_dependents), and waits for its predecessor's completion and
// memory before touching any data (wait).  Both are no-ops for a normal launch.
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}
__device__ __forceinline__ void pdl_start() {
  pdl_trigger();
  pdl_wait();
}

// ------------------------------------------------------------ debug-build index checks
// With HN_DEBUG_CHECKS the kernels check every work-list item (problem slot, level, tile) and
// every one-problem level descriptor against the hierarchy's layout before touching memory; a
// failed check records the source line and the indices in the engine's error words (the first
// failure wins), skips the access and lets the launch finish.  Release builds compile the checks
// to nothing.
#ifndef HN_DEBUG_CHECKS
#define HN_DEBUG_CHECKS 0
#endif
// (a file with checks defines HN_SOURCE, its place among source_name's)
#define HN_HERE (HN_SOURCE << 16 | __LINE__)
__device__ __forceinline__ void dbg_fail(const EngineDev& E, int line, int a, int b) {
  if (atomicCAS(E.err, 0, 5) == 0) {
    E.err[1] = line;
    E.err[2] = a;
    E.err[3] = b;
  }
}
// problem p's tile `tile` of level lv (lv < 0: its finest level)
__device__ __forceinline__ bool dbg_item(const EngineDev& E, int p, int tile, int lv, int line) {
#if HN_DEBUG_CHECKS
  bool ok = p >= 0 && p < E.nprob;
  if (ok) {
    const ProblemDev& P = E.P[p];
    const int l = lv < 0 ? P.L : lv;
    ok = l >= P.coarse && l <= P.L && P.lev[l].n == (1 << l) + 1 && tile >= 0 &&
         (long long)(tile + 1) * kTile <= (long long)P.lev[l].pitch;
  }
  if (!ok) dbg_fail(E, line, p, tile);
  return ok;
#else
  (void)E; (void)p; (void)tile; (void)lv; (void)line;
  return true;
#endif
}
// a one-problem descriptor of level l serving `tiles` tiles
__device__ __forceinline__ bool dbg_level(const EngineDev& E, const LevelDev& d, int l, int tiles, int line) {
#if HN_DEBUG_CHECKS
  const bool ok = l >= HN_MIN_LEVEL && l <= kMaxLevel && d.n == (1 << l) + 1 && tiles >= 0 &&
                  (long long)tiles * kTile <= (long long)d.pitch;
  if (!ok) dbg_fail(E, line, l, tiles);
  return ok;
#else
  (void)E; (void)d; (void)l; (void)tiles; (void)line;
  return true;
#endif
}

// Ask L2 for a tile's 9 band slices ahead of their loads (one prefetch per lane and band).  The
// FP16-band kernels move 8 bytes per lane and band, half of what an FP32 lane moves, so with the
// same warps in flight they keep fewer bytes outstanding; prefetching the bands of the warp's next
// tile while it works on the current one lifts them from 0.81-0.86 to 0.87-0.89 of HBM at L = 12.
// (Further ahead, with the x rows as well, or in the FP32 / FP64 kernels, it measured slower.)
template <class Pol>
__device__ __forceinline__ void prefetch_bands(const LevelDev& d, long long i0) {
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const char* p = static_cast<const char*>(d.band[k]) + i0 * (long long)sizeof(typename Pol::B);
    asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p));
  }
}

// An engine of one problem skips a whole fine-level launch when its problem is not in the phase
// the kernel serves (otherwise every warp would walk its share of the work list to find that out:
// ~20 us per empty launch at L = 12)
__device__ __forceinline__ bool solo_idle(const EngineDev& E, int phase);

// -------------------------------------------------------------------- precision policies
struct F64 { using B = double; using V = double; using A = double; static constexpr int prec = P64; };
struct F32 { using B = float; using V = float; using A = float; static constexpr int prec = P32; };
struct F16 { using B = __half; using V = float; using A = float; static constexpr int prec = P16; };

// Load kinds: LD_NC reads global memory through the non-coherent path (data written by an
// earlier launch); LD_CG reads global memory from L2 (data written earlier in the same launch by
// other SMs of the cluster); LD_GEN is a plain generic load (data in shared memory).  Bands are
// never written by the solver: NC from global memory, GEN from shared memory.
// LD_EF: non-coherent, marked first to be evicted from L2 (data read once per outer step, such as
// the FP64 operator of the outer defect, which would otherwise push the inner cycles' working set
// out of L2).
enum { LD_NC = 0, LD_CG = 1, LD_GEN = 2, LD_EF = 3 };
template <int LK> __device__ __forceinline__ constexpr int band_kind() { return LK == LD_GEN ? LD_GEN : LD_NC; }

__device__ __forceinline__ unsigned long long l2_evict_first_policy() {
  unsigned long long pol;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ double2 ld_ef(const double2* p) {
  double2 v;
  asm volatile("ld.global.nc.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;"
               : "=d"(v.x), "=d"(v.y) : "l"(p), "l"(l2_evict_first_policy()));
  return v;
}
__device__ __forceinline__ double ld_ef(const double* p) {
  double v;
  asm volatile("ld.global.nc.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(p), "l"(l2_evict_first_policy()));
  return v;
}

template <int LK, class T> __device__ __forceinline__ T ldk(const T* p) {
  if constexpr (LK == LD_NC) return __ldg(p);
  else if constexpr (LK == LD_CG) return __ldcg(p);
  else if constexpr (LK == LD_EF) return ld_ef(p);
  else return *p;
}
template <int LK> __device__ __forceinline__ double ld1(const double* p) { return ldk<LK>(p); }
template <int LK> __device__ __forceinline__ float ld1(const float* p) { return ldk<LK>(p); }

template <int LK>
__device__ __forceinline__ void ld4(const double* p, double (&o)[4]) {
  const double2* q = reinterpret_cast<const double2*>(p);
  const double2 a = ldk<LK>(q);
  const double2 b = ldk<LK>(q + 1);
  o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}
template <int LK>
__device__ __forceinline__ void ld4(const float* p, float (&o)[4]) {
  const float4 a = ldk<LK>(reinterpret_cast<const float4*>(p));
  o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
}
__device__ __forceinline__ void st4(double* p, const double (&v)[4]) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void st4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
// plain (coherent) loads for data the same thread also writes
__device__ __forceinline__ void ld4c(const double* p, double (&o)[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0];
  const double2 b = reinterpret_cast<const double2*>(p)[1];
  o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}
__device__ __forceinline__ void ld4c(const float* p, float (&o)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
}

// products rounded on their own (never contracted into a following add or subtract)
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// 4 consecutive band values of band k at node i0, in the arithmetic type
template <class Pol, int LKB = LD_NC>
__device__ __forceinline__ void load_band(const void* band, float scale, long long i0,
                                          typename Pol::A (&o)[4]) {
  if constexpr (Pol::prec == P16) {
    const uint2 u = ldk<LKB>(reinterpret_cast<const uint2*>(static_cast<const __half*>(band) + i0));
    const __half2 h0 = *reinterpret_cast<const __half2*>(&u.x);
    const __half2 h1 = *reinterpret_cast<const __half2*>(&u.y);
    const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
    // each value rounded on its own (never contracted into a following add)
    o[0] = __fmul_rn(scale, f0.x); o[1] = __fmul_rn(scale, f0.y);
    o[2] = __fmul_rn(scale, f1.x); o[3] = __fmul_rn(scale, f1.y);
  } else {
    ld4<LKB>(static_cast<const typename Pol::B*>(band) + i0, o);
  }
}

// Row window around the lane's 4 nodes: w[o + 2] = v[a + o], o = -2..5, a aligned to 4.
template <class V, int LK>
__device__ __forceinline__ void load_row(const V* __restrict__ v, long long a, int lane, V (&w)[8]) {
  V c[4];
  ld4<LK>(v + a, c);
  V l2 = __shfl_up_sync(kFull, c[2], 1), l1 = __shfl_up_sync(kFull, c[3], 1);
  V r0 = __shfl_down_sync(kFull, c[0], 1), r1 = __shfl_down_sync(kFull, c[1], 1);
  if (lane == 0) { l2 = ld1<LK>(v + a - 2); l1 = ld1<LK>(v + a - 1); }
  if (lane == 31) { r0 = ld1<LK>(v + a + 4); r1 = ld1<LK>(v + a + 5); }
  w[0] = l2; w[1] = l1; w[2] = c[0]; w[3] = c[1]; w[4] = c[2]; w[5] = c[3]; w[6] = r0; w[7] = r1;
}

// The FP64 kernels form a defect b - A x as one FMA chain from b (b - a_0 x_0 - a_1 x_1 ...), one
// FP64 operation per node fewer than b - (A x): they are bound by the FP64 pipe on this part.  The
// FP32 and FP16-band kernels, bound by HBM, subtract the finished product.
template <class Pol> __device__ __forceinline__ constexpr bool def_chain() { return Pol::prec == P64; }

// acc[j] = sum_k band_k[i0+j] * x[i0+j+off_k] over the windows w (rows dy = -1, 0, 1), in band
// order k = 0..8; also the diagonal.  off_k = dy*n + dx = dy*shift + (dy + dx), shift = n - 1.
// DEF: acc enters holding b and leaves holding b - sum_k (same order).
template <class Pol, int LKB, bool DEF = false>
__device__ __forceinline__ void stencil_windows(const void* const* band, const float* scale,
                                                const typename Pol::V (&w)[3][8], long long i0,
                                                typename Pol::A (&acc)[4],
                                                typename Pol::A (&dg)[4]) {
  using A = typename Pol::A;
  if constexpr (!DEF) {
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j] = A(0);
  }
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int dy = k / 3 - 1, dx = k % 3 - 1;
    A b[4];
    load_band<Pol, LKB>(band[k], scale ? scale[k] : 1.0f, i0, b);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      acc[j] = DEF ? fma(-b[j], A(w[dy + 1][j + dy + dx + 2]), acc[j])
                   : fma(b[j], A(w[dy + 1][j + dy + dx + 2]), acc[j]);
    if (k == 4) {
#pragma unroll
      for (int j = 0; j < 4; ++j) dg[j] = b[j];
    }
  }
}

// FP16-band operator in row-sum form (array 4 holds the row sum rho):
// acc[j] = rho x_i + sum_{k != 4} a_k (x_{i+off_k} - x_i) in band order; dg[j] = rho - sum a_k.
// The nine 8-byte band loads of the lane are issued before any arithmetic (the FP16 kernels move
// half an FP32 lane's bytes per load, so more of them must be in flight: L = 12 Jacobi 0.88 ->
// 0.90 of HBM); each value is then scaled and used in band order as before.
template <int LKB>
__device__ __forceinline__ void stencil_windows_rowsum(const void* const* band, const float* scale,
                                                       const float (&w)[3][8], long long i0,
                                                       float (&acc)[4], float (&dg)[4]) {
  uint2 raw[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) raw[k] = ldk<LKB>(reinterpret_cast<const uint2*>(static_cast<const __half*>(band[k]) + i0));
  // 4 consecutive values of band k, each rounded on its own (never contracted into a following add)
  auto unpack = [&](int k, float (&o)[4]) {
    const __half2 h0 = *reinterpret_cast<const __half2*>(&raw[k].x);
    const __half2 h1 = *reinterpret_cast<const __half2*>(&raw[k].y);
    const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
    o[0] = __fmul_rn(scale[k], f0.x); o[1] = __fmul_rn(scale[k], f0.y);
    o[2] = __fmul_rn(scale[k], f1.x); o[3] = __fmul_rn(scale[k], f1.y);
  };
  float rho[4];
  unpack(4, rho);
#pragma unroll
  for (int j = 0; j < 4; ++j) { acc[j] = rho[j] * w[1][j + 2]; dg[j] = rho[j]; }
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    if (k == 4) continue;
    const int dy = k / 3 - 1, dx = k % 3 - 1;
    float b[4];
    unpack(k, b);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      acc[j] = fmaf(b[j], w[dy + 1][j + dy + dx + 2] - w[1][j + 2], acc[j]);
      dg[j] -= b[j];
    }
  }
}

// diagonal of the row-sum form without x (for the zero-guess Jacobi step)
template <int LKB>
__device__ __forceinline__ void diag_rowsum(const void* const* band, const float* scale,
                                            long long i0, float (&dg)[4]) {
  load_band<F16, LKB>(band[4], scale[4], i0, dg);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    if (k == 4) continue;
    float b[4];
    load_band<F16, LKB>(band[k], scale[k], i0, b);
#pragma unroll
    for (int j = 0; j < 4; ++j) dg[j] -= b[j];
  }
}

// y = A x at the lane's 4 nodes (x read with load kind LK); xc = x at the nodes, dg = diagonal.
// DEF (plain band form, not the FP16 row sums): acc enters holding b and leaves holding b - A x.
template <class Pol, int LK, bool DEF = false>
__device__ __forceinline__ void apply_op4(const LevelDev& d, const typename Pol::V* __restrict__ x,
                                          long long i0, long long ib, long long shift, int lane,
                                          typename Pol::A (&acc)[4], typename Pol::V (&xc)[4],
                                          typename Pol::A (&dg)[4]) {
  typename Pol::V w[3][8];
#pragma unroll
  for (int dy = -1; dy <= 1; ++dy) load_row<typename Pol::V, LK>(x, i0 + dy * shift, lane, w[dy + 1]);
#pragma unroll
  for (int j = 0; j < 4; ++j) xc[j] = w[1][j + 2];
  if constexpr (Pol::prec == P16) stencil_windows_rowsum<band_kind<LK>()>(d.band, d.scale, w, ib, acc, dg);
  else stencil_windows<Pol, band_kind<LK>(), DEF>(d.band, nullptr, w, ib, acc, dg);
}

// deterministic warp sum (butterfly; every lane ends with the same value)
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Tile partial of a residual norm: the sum over the warp of the squares of each lane's 4 values.
// FP64 values: squares and sums in FP64.  FP32 values: on the FP32 pipe in double-float
// arithmetic (each square exactly as p + e by an FMA, sums by TwoSum), within ~2^-46 of the exact
// sum of the non-negative terms; FP64 operations run at 1/74 of the FP32 rate on this part, and
// per node four of them (two conversions, a product, a sum) cost as much as the band kernel's
// memory traffic at L = 10.  Every lane gets the same value (each butterfly step is symmetric in
// its two operands).
__device__ __forceinline__ void df_add(float& hi, float& lo, float bh, float bl) {
  const float s = hi + bh;
  const float bb = s - hi;
  const float err = (hi - (s - bb)) + (bh - bb);  // TwoSum: hi + bh = s + err exactly
  const float t = err + (lo + bl);
  hi = s + t;                                      // FastTwoSum (|s| >= |t|)
  lo = t - (hi - s);
}
__device__ __forceinline__ double tile_sumsq(const double (&r)[4]) {
  double q = 0.0;
#pragma unroll
  for (int j = 0; j < 4; ++j) q += r[j] * r[j];
  return warp_sum(q);
}
// FP32: the pair (hi, lo) itself, stored in the partial's 8 bytes; every consumer of the partials
// of an FP32 / FP16 cycle sums them as pairs (problem_partial_sum with df)
__device__ __forceinline__ float2 lane_sumsq(const float (&r)[4]) {
  float hi = __fmul_rn(r[0], r[0]), lo = fmaf(r[0], r[0], -hi);
#pragma unroll
  for (int j = 1; j < 4; ++j) {
    const float p = __fmul_rn(r[j], r[j]);
    df_add(hi, lo, p, fmaf(r[j], r[j], -p));
  }
  return make_float2(hi, lo);
}
__device__ __forceinline__ float2 tile_sumsq(const float (&r)[4]) {
  const float2 q = lane_sumsq(r);
  float hi = q.x, lo = q.y;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float bh = __shfl_xor_sync(kFull, hi, o), bl = __shfl_xor_sync(kFull, lo, o);
    df_add(hi, lo, bh, bl);
  }
  return make_float2(hi, lo);
}
__device__ __forceinline__ void store_partial(double* slot, double q) { *slot = q; }
__device__ __forceinline__ void store_partial(double* slot, float2 q) { *reinterpret_cast<float2*>(slot) = q; }

// the same butterfly over the block (any multiple of 32 threads up to 1024); valid in warp 0.
// sh: 32 doubles of shared memory, used as 64 floats
__device__ double block_sum_df(float hi, float lo, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float bh = __shfl_xor_sync(kFull, hi, o), bl = __shfl_xor_sync(kFull, lo, o);
    df_add(hi, lo, bh, bl);
  }
  float* sf = reinterpret_cast<float*>(sh);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { sf[2 * w] = hi; sf[2 * w + 1] = lo; }
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    const bool in = lane < (int)(blockDim.x >> 5);
    float h = in ? sf[2 * lane] : 0.0f, l = in ? sf[2 * lane + 1] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float bh = __shfl_xor_sync(kFull, h, o), bl = __shfl_xor_sync(kFull, l, o);
      df_add(h, l, bh, bl);
    }
    t = double(h) + double(l);                    // exact (l is below half an ulp of h)
  }
  __syncthreads();
  return t;
}

// deterministic block sum of a per-thread value (256 threads)
__device__ double block_sum256(double v, double* sh) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
    t = warp_sum(t);
  }
  __syncthreads();
  return t;   // valid in warp 0
}

// Fixed-order sum of one problem's per-tile partials by one block of 256 threads: thread t adds
// slots t + 256 (4j + c) into chain c = 0..3 (in order of j), then (c0 + c1) + (c2 + c3), then
// the block tree.  Every caller uses this order, so a problem's norm does not depend on which
// kernel or batch computed it.  (Four chains: a dependent FP64 add costs ~64 cycles here.)
// Valid in thread 0.
// df: the partials are double-float pairs (an FP32 / FP16 cycle's), summed in the same order in
// double-float arithmetic on the FP32 pipe: one SM's FP64 rate (~1.7 operations per cycle) made
// the 8,209 FP64 additions of an L = 10 norm the longest part of its lagged check (~10 us).
//
// Not inlined, either of them: inlined, the loads of a batch are issued as the caller's registers allow (the control step
// after a check at L = 11 16.2 us as a call, 29.1 inlined; a cycle of k_span over level 4's 225 unknowns 92.6, 106.1).
__device__ __noinline__ double problem_partial_sum_df(const double* part, int ntiles, double* sh) {
  const float2* pp = reinterpret_cast<const float2*>(part);
  float h[4] = {0.0f, 0.0f, 0.0f, 0.0f}, l[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  if (threadIdx.x < 256) {
    int q = threadIdx.x;
    for (; q + 31 * 256 < ntiles; q += 32 * 256) {
      float2 v[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) v[k] = __ldcg(pp + q + k * 256);
#pragma unroll
      for (int k = 0; k < 32; k += 4)
#pragma unroll
        for (int c = 0; c < 4; ++c) df_add(h[c], l[c], v[k + c].x, v[k + c].y);
    }
    for (; q + 3 * 256 < ntiles; q += 4 * 256)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float2 v = __ldcg(pp + q + c * 256);
        df_add(h[c], l[c], v.x, v.y);
      }
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (q + c * 256 < ntiles) {
        const float2 v = __ldcg(pp + q + c * 256);
        df_add(h[c], l[c], v.x, v.y);
      }
  }
  df_add(h[0], l[0], h[1], l[1]);
  df_add(h[2], l[2], h[3], l[3]);
  df_add(h[0], l[0], h[2], l[2]);
  return block_sum_df(h[0], l[0], sh);
}

__device__ __noinline__ double problem_partial_sum(const double* part, int ntiles, double* sh, bool df = false) {
  if (df) return problem_partial_sum_df(part, ntiles, sh);
  double c0 = 0.0, c1 = 0.0, c2 = 0.0, c3 = 0.0;
  if (threadIdx.x < 256) {                    // larger blocks: the other threads add +0.0
    int q = threadIdx.x;
    // batches of 8 rounds: the 32 loads of a batch are issued before its adds (the adds keep
    // the order above), so L2 latency is paid once per batch rather than once per round
    for (; q + 31 * 256 < ntiles; q += 32 * 256) {
      double v[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) v[k] = __ldcg(part + q + k * 256);
#pragma unroll
      for (int k = 0; k < 32; k += 4) {
        c0 += v[k];
        c1 += v[k + 1];
        c2 += v[k + 2];
        c3 += v[k + 3];
      }
    }
    for (; q + 3 * 256 < ntiles; q += 4 * 256) {
      c0 += __ldcg(part + q);
      c1 += __ldcg(part + q + 256);
      c2 += __ldcg(part + q + 512);
      c3 += __ldcg(part + q + 768);
    }
    if (q < ntiles) c0 += __ldcg(part + q);
    if (q + 256 < ntiles) c1 += __ldcg(part + q + 256);
    if (q + 512 < ntiles) c2 += __ldcg(part + q + 512);
  }
  return block_sum256((c0 + c1) + (c2 + c3), sh);
}

// A problem's tiles are summed in groups of kSumGroup consecutive tiles when it has more than one
// group: each group by problem_partial_sum, then the group sums in group order.  (One block adding
// 131,072 FP64 partials at L = 12 is bound by one SM's FP64 rate, ~30 us; the control kernel
// gives each group its own block.)  Every path that forms a problem's norm uses this order.
__host__ __device__ inline int sum_groups(int ntiles) { return (ntiles + kSumGroup - 1) / kSumGroup; }

__device__ double group_partial_sum(const double* part, int ntiles, int j, double* sh, bool df = false) {
  const int lo = j * kSumGroup;
  return problem_partial_sum(part + lo, min(kSumGroup, ntiles - lo), sh, df);
}

// the same order in one block (valid in thread 0)
__device__ double problem_norm_sum(const double* part, int ntiles, double* sh, bool df = false) {
  const int ng = sum_groups(ntiles);
  if (ng == 1) return problem_partial_sum(part, ntiles, sh, df);
  double t = 0.0;
  for (int j = 0; j < ng; ++j) {
    const double g = group_partial_sum(part, ntiles, j, sh, df);
    if (threadIdx.x == 0) t += g;
  }
  return t;
}

__host__ __device__ inline int fine_tiles(int L) {
  const long long n = (1LL << L) + 1;
  return (int)((n * n + kTile - 1) / kTile);
}

// Lagged convergence test: the first smoothing step of a cycle from a nonzero iterate computes
// the residual of that iterate; nrm is its norm.  FP64 multigrid stops when relres <= tol (the
// iterate in buffer 0 is the result) or at the cycle cap; inner cycles of the defect correction
// stop at the inner tolerance or the inner caps (the correction goes to the update).  Otherwise
// the cycle proceeds and is counted.
__device__ __forceinline__ void cond_set(const CondDev& c, unsigned v) {
  if (!c.on) return;
  cudaGraphSetConditional(c.cycle, v);
  *c.taken = v;
}

__device__ void pre_check(ProbState& st, const Params& prm, double nrm) {
  if (!isfinite(nrm)) { st.status = HN_ERR_NONFINITE; st.phase = PH_DONE; return; }
  if (st.phase == PH_CYCLE) {
    st.dnorm = nrm;
    st.relres = nrm / st.bnorm;
    if (st.relres <= prm.tol) { st.status = HN_OK; st.phase = PH_DONE; }
    else if (st.cycles >= prm.max_cycles) { st.status = HN_ERR_NOT_CONVERGED; st.phase = PH_DONE; }
    else st.cycles += 1;
  } else {
    st.inner_res = nrm;
    if (nrm <= prm.inner_tol * st.inner_ref || st.inner_k >= prm.inner_max ||
        st.inner_cycles >= prm.max_cycles) {
      st.phase = PH_UPDATE;
    } else { st.inner_k += 1; st.inner_cycles += 1; st.cycles += 1; }
  }
}

__device__ __forceinline__ bool solo_idle(const EngineDev& E, int phase) {
  return E.nprob == 1 && E.S[0].phase != phase;
}

// Full-weighting restriction of the fine defect onto coarse node (I, J) (Dirichlet and padding
// nodes get 0).  Summation order: fine rows 2J-1, 2J, 2J+1, columns 2I-1, 2I, 2I+1, weights 1/4,
// 1/2, 1/4 x 1/4, 1/2, 1/4 (products by powers of two are exact); a fine node off the grid (next
// to a free Neumann side) contributes 0.  rd(y, x) reads fine node (x, y).
template <class V, class F>
__device__ __forceinline__ V restrict_value_xy(int I, int J, int nc, int nf, int bc, F rd) {
  if (I < 0 || J >= nc || is_dirichlet(I, J, nc, bc)) return V(0);
  const int fx = 2 * I, fy = 2 * J;
  auto R = [&](int dy, int dx) -> V {
    const int x = fx + dx, y = fy + dy;
    return (x >= 0 && y >= 0 && x < nf && y < nf) ? rd(y, x) : V(0);
  };
  const V q = V(0.25), h = V(0.5);
  V v = q * R(-1, -1);
  v = fma(h, R(-1, 0), v);
  v = fma(q, R(-1, 1), v);
  v = fma(h, R(0, -1), v);
  v = v + R(0, 0);
  v = fma(h, R(0, 1), v);
  v = fma(q, R(1, -1), v);
  v = fma(h, R(1, 0), v);
  v = fma(q, R(1, 1), v);
  return v;
}
// the same with rd(i) reading fine node i = y nf + x
template <class V, class F>
__device__ __forceinline__ V restrict_value(int I, int J, int nc, int nf, int bc, F rd) {
  return restrict_value_xy<V>(I, J, nc, nf, bc, [&](int y, int x) { return rd((long long)y * nf + x); });
}

// x_f[x_sel] += P e_c at fine node (ix, iy): bilinear interpolation of the coarse iterate, ec(cy, cx)
// reading coarse node (cx, cy); Dirichlet fine nodes are left unchanged (their coarse neighbours on
// the same side are Dirichlet too and hold 0).  Returns false for them, else the value added.
template <class V, class F>
__device__ __forceinline__ bool prolong_value_xy(int ix, int iy, int nf, int bc, F ec, V* add) {
  if (is_dirichlet(ix, iy, nf, bc)) return false;
  const int cx0 = ix >> 1, cx1 = (ix + 1) >> 1, cy0 = iy >> 1, cy1 = (iy + 1) >> 1;
  const bool ox = ix & 1, oy = iy & 1;
  if (!ox && !oy) *add = ec(cy0, cx0);
  else if (ox && !oy) *add = V(0.5) * (ec(cy0, cx0) + ec(cy0, cx1));
  else if (!ox && oy) *add = V(0.5) * (ec(cy0, cx0) + ec(cy1, cx0));
  else *add = V(0.25) * (((ec(cy0, cx0) + ec(cy0, cx1)) + ec(cy1, cx0)) + ec(cy1, cx1));
  return true;
}
// the same with ec(k) reading coarse node k = cy nc + cx
template <class V, class F>
__device__ __forceinline__ bool prolong_value(int ix, int iy, int nf, int nc, int bc, F ec, V* add) {
  return prolong_value_xy<V>(ix, iy, nf, bc, [&](int cy, int cx) { return ec(cy * nc + cx); }, add);
}

// node coordinates of flat index f in [0, n^2)
__device__ __forceinline__ void node_xy(int f, int L, int& x, int& y) {
  const int q = f >> L, c = f & ((1 << L) - 1), n = (1 << L) + 1;
  y = q;
  x = c - q;
  if (x < 0) { x += n; --y; }
  if (x < 0) { x += n; --y; }
}

// mbarrier and bulk-copy (TMA engine, 1D) helpers
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes,
                                         unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
// one bulk copy global -> this block's shared memory, accounted on bar (16-byte aligned, size a
// multiple of 16); issued by one thread, which arrives on bar once all its copies are issued
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, unsigned bytes,
                                          unsigned long long* bar) {
  if (bytes == 0) return;
  mbar_expect(bar, bytes);
  bulk_g2s(dst, src, bytes, bar);
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait for phase `parity` of an mbarrier; false if it did not complete in time
constexpr int kWaitTries = 1 << 22;
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity) {
  for (int i = 0; i < kWaitTries; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// true in the last block of the launch to get here (every block calls it once, after its work;
// the block's writes are visible to that block); the last block resets the ticket when done
__device__ bool solo_last_block(const EngineDev& E) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(E.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}

// The lagged check of an engine of one problem taken inside its first smoothing step (in place of
// a separate control launch, for problems whose norm is one group of partials): the last block to
// finish sums the tile partials in the fixed order and updates the state, and the cycle's IF value
// is set as the control kernel sets it (the problem is still in the cycle).  A uniform early
// return of every block (problem not in the phase) leaves the ticket at zero.
__device__ void solo_fused_check(const EngineDev& E, int level, bool checked, int want) {
  __shared__ double sh[32];
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();                              // this block's partials before its ticket
    s_last = atomicAdd(E.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  ProbState& st = E.S[0];
  double sum = 0.0;
  if (checked) sum = problem_norm_sum(E.partial, fine_tiles(level), sh, E.prm.prec != P64);
  if (threadIdx.x == 0) {
    if (checked) pre_check(st, E.prm, sqrt(sum));
    if (st.phase == want && (st.phase == PH_INNER || st.phase == PH_CYCLE)) cond_set(E.prm.cond, 1u);
    *E.ticket = 0u;                                 // ready for the next launch
  }
}

// The state transition of control step `kind` for problem state st, given the summed partials
// (thread 0 of one block; the control kernel, or the last block of a kernel that folds the step in)
__device__ void control_apply(const EngineDev& E, ProbState& st, int kind, double sum) {
  const int ph = st.phase;
  const Params& prm = E.prm;
  const double nrm = sqrt(sum);
  switch (kind) {
    case CTRL_INIT:
      if (st.status == HN_ERR_ARG) { st.phase = PH_DONE; break; }
      if (!isfinite(nrm)) { st.status = HN_ERR_NONFINITE; st.phase = PH_DONE; break; }
      if (nrm == 0.0) { st.bnorm = 0.0; st.relres = 0.0; st.status = HN_OK; st.phase = PH_DONE; break; }
      st.bnorm = nrm;
      st.s = 1.0 / nrm;
      st.inv_s = 1.0 / st.s;
      st.relres = 1.0;
      if (prm.prec == P64 && prm.solver != SOLVER_PCG) {
        // a zero initial guess starts its first cycle unchecked (relres 1); a given guess is
        // checked by the first smoothing step of its first cycle
        st.phase = PH_CYCLE;
        st.cycles = st.x_zero ? 1 : 0;
      } else {
        st.phase = PH_OUTER;
      }
      break;
    case CTRL_CHECK0:
      st.dnorm = nrm;
      st.relres = nrm / st.bnorm;
      if (!isfinite(nrm)) { st.status = HN_ERR_NONFINITE; st.phase = PH_DONE; }
      else if (st.relres <= prm.tol) { st.status = HN_OK; st.phase = PH_DONE; }
      else if (st.cycles >= prm.max_cycles) { st.status = HN_ERR_NOT_CONVERGED; st.phase = PH_DONE; }
      else st.phase = PH_CYCLE;
      break;
    case CTRL_OUTER:
      if (prm.solver == SOLVER_PCG) {
        // after the initial residual or a CG step: check, then precondition the new residual
        if (st.cycles > 0) st.outer_iters += 1;
        st.dnorm = nrm;
        st.relres = nrm / st.bnorm;
        if (!isfinite(nrm)) { st.status = HN_ERR_NONFINITE; st.phase = PH_DONE; }
        else if (st.relres <= prm.tol) { st.status = HN_OK; st.phase = PH_DONE; }
        else if (st.outer_iters >= prm.max_outer || st.cycles >= prm.max_cycles) {
          st.status = HN_ERR_NOT_CONVERGED; st.phase = PH_DONE;
        } else {
          st.phase = PH_PRECOND; st.zero_top = 1; st.cycles += 1;
          if (prm.prec != P64) st.inner_cycles += 1;
        }
        break;
      }
      st.dnorm = nrm;
      st.relres = nrm / st.bnorm;
      if (!isfinite(nrm)) { st.status = HN_ERR_NONFINITE; st.phase = PH_DONE; }
      else if (st.relres <= prm.tol) { st.status = HN_OK; st.phase = PH_DONE; }
      else if (st.outer_iters >= prm.max_outer || st.inner_cycles >= prm.max_cycles) {
        st.status = HN_ERR_NOT_CONVERGED; st.phase = PH_DONE;
      } else {
        // the first inner cycle starts from zero: it runs unchecked and is counted here
        st.phase = PH_INNER; st.zero_top = 1; st.inner_ref = st.s * nrm;
        st.inner_k = 1; st.inner_cycles += 1; st.cycles += 1;
      }
      break;
    case CTRL_PCG_ALPHA:
      // sum = (p, q); a breakdown (not positive: the preconditioned operator is not definite in
      // this arithmetic) stops the solve
      if (!isfinite(sum) || !(sum > 0.0)) { st.status = HN_ERR_NONFINITE; st.phase = PH_DONE; }
      else st.alpha = st.rho / sum;
      break;
    case CTRL_PCG_BETA: {
      // sum = (r, c) with z = c / s: rho' = (r, z); the first direction is z itself
      const double rho = sum / st.s;
      if (!isfinite(rho) || !(rho > 0.0)) { st.status = HN_ERR_NONFINITE; st.phase = PH_DONE; break; }
      st.beta = st.cycles > 1 ? rho / st.rho : 0.0;
      st.rho = rho;
      st.phase = PH_UPDATE;
      break;
    }
    case CTRL_POST: {
      if (prm.solver == SOLVER_PCG) {
        // the next cycle's right-hand side is scaled by 1 / ||r|| of this step
        if (st.dnorm > 0.0 && isfinite(st.dnorm)) { st.s = 1.0 / st.dnorm; st.inv_s = 1.0 / st.s; }
        st.phase = PH_OUTER;
        break;
      }
      st.outer_iters += 1;
      st.x_zero = 0;
      // scale for the next defect: the inner solve reduced the defect by about inner_res/inner_ref
      const double red = st.inner_ref > 0.0 ? st.inner_res / st.inner_ref : 1.0;
      const double pred = st.dnorm * fmax(red, 1e-7);
      if (pred > 0.0 && isfinite(pred)) { st.s = 1.0 / pred; st.inv_s = 1.0 / st.s; }
      st.phase = PH_OUTER;
      break;
    }
    default: break;
  }
}

// Count problems still running; publish to the host word and, inside a device-side loop, to the
// graph's while-condition.  Past the iteration limit every running problem is stopped as not
// converged, so a device-side loop always ends.
__device__ void summary_apply(const EngineDev& E, cudaGraphConditionalHandle h, int use_handle,
                              int end_of_iteration, double* sh) {
  __shared__ unsigned over;
  if (threadIdx.x == 0) {
    const unsigned it = E.iter ? (*E.iter += 1) : 0u;
    over = (E.iter && it > E.iter_limit) ? 1u : 0u;
  }
  __syncthreads();
  double c = 0.0;
  for (int p = threadIdx.x; p < E.nprob; p += blockDim.x) {
    ProbState& st = E.S[p];
    if (st.phase != PH_DONE && over) { st.status = HN_ERR_NOT_CONVERGED; st.phase = PH_DONE; }
    // after an iteration the finest-level iterate of a running cycle is no longer zero
    if (end_of_iteration && (st.phase == PH_INNER || st.phase == PH_CYCLE)) st.zero_top = 0;
    if (E.states_host) E.states_host[p] = st;
    c += st.phase != PH_DONE ? 1.0 : 0.0;
  }
  c = block_sum256(c, sh);
  if (threadIdx.x == 0) {
    const unsigned active = (unsigned)c;
    if (E.active_host) *E.active_host = active;
    if (use_handle) cudaGraphSetConditional(h, active > 0 ? 1u : 0u);
    const CondDev& cd = E.prm.cond;
    if (cd.on) {
      *cd.launches += cd.n_base + (*cd.taken ? cd.n_cycle : 0u);
      cond_set(cd, 0u);
    }
  }
}

// The problems of an engine that a launch serves: those of at most kListMax slots from `base` that on(state,
// finest level) chooses, in slot order, with the levels they are taken at (level, or 0: their own finest).
// The whole block; returns the number of problems.  Every block of a launch has to find the same list, so
// what `on` looks at must not change before every block has listed.
constexpr int kListMax = 1024;
struct Served {
  int slot[kListMax];                    // (a batch may have any number of problems)
  unsigned char level[kListMax];
  int start[kListMax + 1];
  int count[32];
};
template <class F>
__device__ int list_served(const EngineDev& E, Served& q, int base, int level, F&& chosen) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
  const int n = min(kListMax, E.nprob - base);
  // slots of a warp: a contiguous share, read in one go (the loads of a round do not depend on each other)
  const int share = (n + nw * 32 - 1) / (nw * 32);
  const int lo = warp * share * 32;
  unsigned take = 0;
  for (int k = 0; k < share; ++k) {
    const int p = lo + k * 32 + lane;
    const bool on = p < n && chosen(E.S[base + p], E.P[base + p].L);
    take |= on ? 1u << k : 0u;
  }
  int mine = 0;
  for (int k = 0; k < share; ++k) mine += __popc(__ballot_sync(kFull, (take >> k) & 1u));
  if (lane == 0) q.count[warp] = mine;
  __syncthreads();
  int at = 0, total = 0;
  for (int w = 0; w < nw; ++w) {
    if (w < warp) at += q.count[w];
    total += q.count[w];
  }
  for (int k = 0; k < share; ++k) {
    const bool on = (take >> k) & 1u;
    const unsigned m = __ballot_sync(kFull, on);
    if (on) {
      const int i = at + __popc(m & ((1u << lane) - 1u)), p = base + lo + k * 32 + lane;
      q.slot[i] = p;
      q.level[i] = (unsigned char)(level ? level : E.P[p].L);
    }
    at += __popc(m);
  }
  __syncthreads();
  return total;
}
// running numbers of the problems' work items (items: of a level; 32-bit arithmetic only: a round of 32
// problems is on every block's way to its first load); the whole block; returns their sum
template <class F>
__device__ int number_items(Served& q, int n, F&& items) {
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {
    int run = 0;
    for (int b = 0; b < n; b += 32) {
      const int c = b + lane < n ? items((int)q.level[b + lane]) : 0;
      int s = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, s, o);
        if (lane >= o) s += t;
      }
      if (b + lane < n) q.start[b + lane] = run + s - c;
      run += __shfl_sync(kFull, s, 31);
    }
    if (lane == 0) q.start[n] = run;
  }
  __syncthreads();
  return q.start[n];
}
// the problem of work item `it`
__device__ __forceinline__ int served_of(const Served& q, int n, int it) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (q.start[mid] <= it) lo = mid; else hi = mid - 1;
  }
  return lo;
}

}  // namespace

}  // namespace hn
