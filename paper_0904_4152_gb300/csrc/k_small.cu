// The V(2,2) cycle on the coarse levels of one problem inside one block's shared memory: levels
// coarse..T, T <= kSmallTop, of an FP32 or FP16-band hierarchy with the exact coarse solver.
//
// What bounds it: a chain of about 26 dependent steps (three smoothing steps, the defect and two
// transfers a level), each a few instructions per node on at most 1089 nodes, so the length of the
// instruction stream and the block barriers.  Level sizes are template constants: a node's neighbours,
// bands and vectors are fixed offsets from one register (the general kernel, k_tail, reads every array
// through a descriptor and generic addresses: 8 us of steps at levels 5..2).  The operator's bands
// towards smaller indices are those towards greater ones at the neighbour, bit for bit (see
// k_march.cu), so only five are staged: 82 KB in FP32, two blocks to an SM.  Measured per launch (levels
// 5..2, with the launch itself): 20.9 us before, 12.0 us; L = 7 solve 835 -> 738 us, L = 10 1.490 -> 1.457 ms,
// the 256-problem batch 20.8 -> 20.0 ms.  The constant data of an engine of one
// problem, whose descriptors come by value, are staged before the preceding launch ends.
//
// Every value is formed by the operations of the per-step kernels in their order (same bits).
#include <algorithm>

#include "k_device.cuh"

namespace hn {

namespace {

constexpr int kSmallThreads = 512;

// a level's arrays in shared memory: E elements, H of them before node 0 (zeros, as in memory)
template <int l>
struct Lev {
  static constexpr int n = (1 << l) + 1, N = n * n, pitch = (N + kTile - 1) / kTile * kTile;
  static constexpr int H = (n + 1 + 7) / 8 * 8, E = pitch + 2 * H;
};
constexpr int kElems = Lev<2>::E + Lev<3>::E + Lev<4>::E + Lev<5>::E;
template <int l> constexpr int elems_before() { return l <= 2 ? 0 : elems_before<(l > 2 ? l - 1 : 2)>() + Lev<(l > 2 ? l - 1 : 2)>::E; }

constexpr int kCinvDoubles = 25 * 25;    // a staged coarse inverse (level 2, free sides at most)

template <class Pol>
constexpr int small_smem() { return kElems * (5 * (int)sizeof(typename Pol::B) + 5 * 4) + kCinvDoubles * 8; }

// the arrays of level l: five bands (4..8), omega / D, right-hand side, iterate, its partner, defect
template <class Pol, int l>
struct Arr {
  using B = typename Pol::B;
  using G = Lev<l>;
  static constexpr int base_b = elems_before<l>() * 5, base_v = elems_before<l>() * 5;
  unsigned char* sm;
  __device__ __forceinline__ B* band(int k) const { return reinterpret_cast<B*>(sm) + base_b + k * G::E + G::H; }
  __device__ __forceinline__ float* vec(int k) const {
    return reinterpret_cast<float*>(sm + kElems * 5 * (int)sizeof(B)) + base_v + k * G::E + G::H;
  }
  __device__ __forceinline__ float* wd() const { return vec(0); }
  __device__ __forceinline__ float* rhs() const { return vec(1); }
  __device__ __forceinline__ float* x0() const { return vec(2); }
  __device__ __forceinline__ float* x1() const { return vec(3); }
  __device__ __forceinline__ float* r() const { return vec(4); }
};

// (A x) at node i, in the band order of stencil_node
template <class Pol, int l>
__device__ __forceinline__ float apply_node(const Arr<Pol, l>& a, const float* scale, const float* x, int i) {
  constexpr int n = Lev<l>::n;
  float band[9];
  auto get = [&](int k, int at) {                 // band k (4..8) at node `at`
    if constexpr (Pol::prec == P16) return __fmul_rn(scale[k - 4], __half2float(a.band(k - 4)[at]));
    else return a.band(k - 4)[at];
  };
  band[0] = get(8, i - n - 1); band[1] = get(7, i - n); band[2] = get(6, i - n + 1); band[3] = get(5, i - 1);
#pragma unroll
  for (int k = 4; k < 9; ++k) band[k] = get(k, i);
  float acc = 0.0f;
  if constexpr (Pol::prec == P16) {
    const float xi = x[i];
    acc = band[4] * xi;
#pragma unroll
    for (int k = 0; k < 9; ++k)
      if (k != 4) acc = fmaf(band[k], x[i + (k / 3 - 1) * n + (k % 3 - 1)] - xi, acc);
  } else {
#pragma unroll
    for (int k = 0; k < 9; ++k) acc = fmaf(band[k], x[i + (k / 3 - 1) * n + (k % 3 - 1)], acc);
  }
  return acc;
}

template <class F>
__device__ __forceinline__ void for_nodes(int count, F&& f) {
  for (int i = threadIdx.x; i < count; i += kSmallThreads) f(i);
}

// a Jacobi step from x to y
template <class Pol, int l>
__device__ __forceinline__ void jacobi(const Arr<Pol, l>& a, const float* scale, const float* x, float* y) {
  for_nodes(Lev<l>::N, [&](int i) { y[i] = fmaf(a.wd()[i], a.rhs()[i] - apply_node(a, scale, x, i), x[i]); });
  __syncthreads();
}

// what a block knows of its problem
struct Ctx {
  unsigned char* sm;
  const float (*scale)[5];               // per level
  double* sol;                           // kMaxCoarseM doubles each
  double* rd;
  double* sh;
  const double* cinv;
  int c, top, m, bc;
  int check;                             // the top level is the problem's finest and its iterate is not zero
  double* part;                          // its norm partials
};

// The lagged check of a problem whose finest level is here: the norm of the defect in a.r(), summed as
// every other path sums it.  False if the problem leaves the cycle.
template <class Pol, int l>
__device__ __forceinline__ bool check(const Ctx& k, const Arr<Pol, l>& a, const EngineDev& E, ProbState* st, int want) {
  const int lane = threadIdx.x & 31;
  for (int t = threadIdx.x >> 5; t < Lev<l>::pitch / kTile; t += kSmallThreads / 32) {
    float r[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) r[j] = a.r()[t * kTile + lane * 4 + j];
    const float2 q = tile_sumsq(r);
    if (lane == 0) store_partial(k.part + t, q);
  }
  __syncthreads();
  const double sum = problem_norm_sum(k.part, Lev<l>::pitch / kTile, k.sh, true);
  if (threadIdx.x == 0) pre_check(*st, E.prm, sqrt(sum));
  __syncthreads();
  return __ldcg(&st->phase) == want;
}

// pre-smoothing, defect and restriction of levels l..c + 1; false if the problem leaves the cycle
template <class Pol, int l>
__device__ __forceinline__ bool down(const Ctx& k, const EngineDev& E, ProbState* st, int want) {
  if constexpr (l > 2) {
    if (l <= k.top && l > k.c) {
      using G = Lev<l>;
      const Arr<Pol, l> a{k.sm};
      const Arr<Pol, l - 1> c{k.sm};
      const float* sc = k.scale[l];
      if (l == k.top && k.check) {                // from a nonzero iterate
        for_nodes(G::N, [&](int i) {
          const float r = a.rhs()[i] - apply_node(a, sc, a.x0(), i);
          a.r()[i] = r;
          a.x1()[i] = fmaf(a.wd()[i], r, a.x0()[i]);
        });
        __syncthreads();
        if (!check(k, a, E, st, want)) return false;
      } else {
        for_nodes(G::N, [&](int i) { a.x1()[i] = mul_rn(a.wd()[i], a.rhs()[i]); });
        __syncthreads();
      }
      jacobi(a, sc, a.x1(), a.x0());
      for_nodes(G::N, [&](int i) { a.r()[i] = a.rhs()[i] - apply_node(a, sc, a.x0(), i); });
      __syncthreads();
      for_nodes(Lev<l - 1>::N, [&](int i) {
        constexpr int nc = Lev<l - 1>::n;
        const int J = i / nc, I = i - J * nc;
        c.rhs()[i] = restrict_value<float>(I, J, nc, G::n, k.bc, [&](long long q) { return a.r()[(int)q]; });
      });
      __syncthreads();
    }
    return down<Pol, l - 1>(k, E, st, want);
  } else {
    return true;
  }
}

// prolongation and post-smoothing of levels c + 1..l
template <class Pol, int l>
__device__ __forceinline__ void up(const Ctx& k) {
  if constexpr (l > 2) {
    up<Pol, l - 1>(k);
    if (l <= k.top && l > k.c) {
      using G = Lev<l>;
      const Arr<Pol, l> a{k.sm};
      const Arr<Pol, l - 1> c{k.sm};
      for_nodes(G::N, [&](int i) {
        const int iy = i / G::n, ix = i - iy * G::n;
        float add;
        if (prolong_value<float>(ix, iy, G::n, Lev<l - 1>::n, k.bc, [&](int q) { return c.x0()[q]; }, &add)) a.x0()[i] = a.x0()[i] + add;
      });
      __syncthreads();
      jacobi(a, k.scale[l], a.x0(), a.x1());
      jacobi(a, k.scale[l], a.x1(), a.x0());
    }
  }
}

// the exact solve on the coarsest level (one thread per unknown, k_tail's sums)
template <class Pol, int l>
__device__ __forceinline__ bool coarse(const Ctx& k, const EngineDev& E, ProbState* st, int want) {
  if constexpr (l <= 4) {
    if (k.c == l) {
      using G = Lev<l>;
      const Arr<Pol, l> a{k.sm};
      if (k.top == l && k.check) {                // the problem is the coarsest level alone
        for_nodes(G::N, [&](int i) { a.r()[i] = a.rhs()[i] - apply_node(a, k.scale[l], a.x0(), i); });
        __syncthreads();
        if (!check(k, a, E, st, want)) return false;
      }
      const UnknownRect ur = unknown_rect(G::n, k.bc);
      const int m = k.m;
      for_nodes(m, [&](int v) { k.rd[v] = double(a.rhs()[(v / ur.nx + ur.y0) * G::n + (v % ur.nx + ur.x0)]); });
      __syncthreads();
      for_nodes(m, [&](int u) {
        const double* row = k.cinv + u * m;
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
        int v = 0;
        for (; v + 3 < m; v += 4) {
          a0 = fma(row[v], k.rd[v], a0);
          a1 = fma(row[v + 1], k.rd[v + 1], a1);
          a2 = fma(row[v + 2], k.rd[v + 2], a2);
          a3 = fma(row[v + 3], k.rd[v + 3], a3);
        }
        if (v < m) a0 = fma(row[v], k.rd[v], a0);
        if (v + 1 < m) a1 = fma(row[v + 1], k.rd[v + 1], a1);
        if (v + 2 < m) a2 = fma(row[v + 2], k.rd[v + 2], a2);
        k.sol[u] = (a0 + a1) + (a2 + a3);
      });
      __syncthreads();
      for_nodes(G::N, [&](int q) {
        const int iy = q / G::n - ur.y0, ix = q % G::n - ur.x0;
        a.x0()[q] = ix >= 0 && iy >= 0 && ix < ur.nx && iy < ur.ny ? float(k.sol[iy * ur.nx + ix]) : 0.0f;
      });
      __syncthreads();
    }
    if constexpr (l < 4) return coarse<Pol, l + 1>(k, E, st, want);
  }
  return true;
}

__device__ __forceinline__ void stage16(void* dst, const void* src, int bytes) {
  for (int q = threadIdx.x * 16; q < bytes; q += kSmallThreads * 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(static_cast<unsigned char*>(dst) + q)),
                 "l"(static_cast<const unsigned char*>(src) + q) : "memory");
}

// start the copies of level l's constant arrays, and of the levels below it
template <class Pol, int l>
__device__ __forceinline__ void stage(const Ctx& k, const LevelDev* lev) {
  using G = Lev<l>;
  if (l <= k.top && l >= k.c) {
    const Arr<Pol, l> a{k.sm};
    const LevelDev& d = lev[l];
#pragma unroll
    for (int b = 0; b < 5; ++b)
      stage16(a.band(b) - G::H, static_cast<const typename Pol::B*>(d.band[b + 4]) - G::H, G::E * (int)sizeof(typename Pol::B));
    stage16(a.wd() - G::H, d.wdf - G::H, G::E * 4);
  }
  if constexpr (l > 2) stage<Pol, l - 1>(k, lev);
}

// the top level's right-hand side (and nonzero iterate) in, its iterate out
template <class Pol, int l>
__device__ __forceinline__ void top_in(const Ctx& k, const LevelDev* lev) {
  if (l == k.top) {
    const Arr<Pol, l> a{k.sm};
    const float* b = static_cast<const float*>(lev[l].rhs);
    const float* x = static_cast<const float*>(lev[l].x[0]);
    for_nodes(Lev<l>::N, [&](int i) { a.rhs()[i] = __ldcg(b + i); });
    if (k.check) for_nodes(Lev<l>::N, [&](int i) { a.x0()[i] = __ldcg(x + i); });
  }
  if constexpr (l > 2) top_in<Pol, l - 1>(k, lev);
}
template <class Pol, int l>
__device__ __forceinline__ void top_out(const Ctx& k, const LevelDev* lev) {
  if (l == k.top) {
    const Arr<Pol, l> a{k.sm};
    float* x = static_cast<float*>(lev[l].x[0]);
    for_nodes(Lev<l>::N, [&](int i) { x[i] = a.x0()[i]; });
  }
  if constexpr (l > 2) top_out<Pol, l - 1>(k, lev);
}

template <class Pol>
__global__ void __launch_bounds__(kSmallThreads, 2) k_small(EngineDev E, SmallSolo solo, int T, int want) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ LevelDev lev[kSmallTop + 1];
  __shared__ float scale[kSmallTop + 1][5];
  __shared__ double sol[kMaxCoarseM], rd[kMaxCoarseM], sh[32];
  pdl_trigger();
  const int p = blockIdx.x;
  Ctx k;
  k.sm = smem;
  k.scale = scale;
  k.sol = sol;
  k.rd = rd;
  k.sh = sh;
  int L;
  const double* cinv_g;
  if (solo.L) {
    L = solo.L;
    k.c = solo.coarse;
    k.m = solo.m;
    cinv_g = solo.cinv;
  } else {
    pdl_wait();
    const ProblemDev& P = E.P[p];
    if (E.S[p].phase != want) return;
    L = P.L;
    if (L < HN_MIN_LEVEL) return;                 // an empty slot
    k.c = P.coarse;
    k.m = P.m;
    cinv_g = P.cinv;
  }
  k.top = min(L, T);
  {
    constexpr int words = (int)(sizeof(LevelDev) / 4);
    const unsigned* src = reinterpret_cast<const unsigned*>(solo.L ? &solo.lev[0] : &E.P[p].lev[2]);
    for (int q = threadIdx.x; q < words * (k.top - 1); q += kSmallThreads) reinterpret_cast<unsigned*>(&lev[2])[q] = src[q];
  }
  // vectors start as zeros (their halos and padding stay so)
  float4* z = reinterpret_cast<float4*>(smem + kElems * 5 * (int)sizeof(typename Pol::B));
  for (int q = threadIdx.x; q < kElems * 5 / 4; q += kSmallThreads) z[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  __syncthreads();
  k.bc = lev[k.top].bc;
  if (threadIdx.x < 5)
    for (int l = k.c; l <= k.top; ++l) scale[l][threadIdx.x] = lev[l].scale[threadIdx.x + 4];
  stage<Pol, kSmallTop>(k, lev);
  double* cinv_s = reinterpret_cast<double*>(smem + kElems * (5 * (int)sizeof(typename Pol::B) + 5 * 4));
  const bool staged = k.m * k.m <= kCinvDoubles;
  if (staged)
    for (int q = threadIdx.x; q < k.m * k.m; q += kSmallThreads) cinv_s[q] = __ldg(cinv_g + q);
  k.cinv = staged ? cinv_s : cinv_g;
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  if (solo.L) pdl_wait();
  ProbState* st = E.S + p;
  const bool go = !solo.L || __ldcg(&st->phase) == want;
  if (go) {
    k.check = L == k.top && !__ldcg(&st->zero_top) && E.prm.solver != SOLVER_PCG;
    k.part = E.partial + (solo.L ? 0 : E.fine_off[p]);
    top_in<Pol, kSmallTop>(k, lev);
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
  if (!go || !down<Pol, kSmallTop>(k, E, st, want) || !coarse<Pol, 2>(k, E, st, want)) return;
  up<Pol, kSmallTop>(k);
  top_out<Pol, kSmallTop>(k, lev);
}

template <class Pol>
cudaError_t launch_small_t(const EngineDev& E, const SmallSolo& solo, int T, int want, cudaStream_t s) {
  auto kern = k_small<Pol>;
  static const cudaError_t ready = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, small_smem<Pol>());
  if (ready != cudaSuccess) return ready;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)E.nprob, 1, 1);
  cfg.blockDim = dim3((unsigned)kSmallThreads, 1, 1);
  cfg.dynamicSmemBytes = (size_t)small_smem<Pol>();
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  if (pdl_launch(E.pdl, (int)cfg.gridDim.x)) {
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 1;
    cfg.attrs = attr;
  }
  return cudaLaunchKernelEx(&cfg, kern, E, solo, T, want);
}

}  // namespace

cudaError_t launch_small(const EngineDev& E, const SmallSolo& solo, int T, int want, cudaStream_t s) {
  if (E.prm.prec == P32) return launch_small_t<F32>(E, solo, T, want, s);
  if (E.prm.prec == P16) return launch_small_t<F16>(E, solo, T, want, s);
  return cudaErrorInvalidValue;
}

}  // namespace hn
