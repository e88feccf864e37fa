// The V(2,2) cycle of an FP32 or FP16-band hierarchy on the levels coarse..T, T <= kSpanTop, of one problem by a
// cluster of 16 blocks, with the exact coarse solver.
//
// What bounds it: some 40 dependent steps, each a barrier over the cluster or block and, on level 8, about 1,400 shared
// memory accesses a warp port (66,049 nodes on 16 SMs).  As one launch per level and direction these steps wait for
// launches, first loads and, between cycles, the graph's conditional nodes; here a level stays in shared memory.
// Levels 8 to 6 are spread over the cluster by rows: a thread marches down a few rows of one column, so that a node
// costs 11 shared-memory loads (three of the iterate, eight of the bands, of which the operator's symmetry
// leaves four arrays, bit for bit: see k_march.cu) in place of 18; a warp more takes the last column.  Diagonals,
// omega / D and right-hand sides stay in registers, first and last rows go to the neighbours' ghost rows as they
// are formed.  Two buffers a level do: no step writes what a neighbour may still read.  Levels 5 and below run in
// block 0 (spread out, level 5 would take a barrier a step for a quarter of its instructions).
//
// The lagged check (the problem's finest level is here, its iterate is not zero): the defects go through memory to the
// warps that sum the tiles, while the second smoothing step runs; an iterate is overwritten in shared memory only,
// the accepted one is in memory.  So a problem whose finest level is here runs all cycles of an inner solve in one
// launch.  Measured: L = 7 solve 715 -> 415 us, L = 8 796 -> 613 us (its straight-line form, each step's code its own,
// 639 us: a fifth of the stalls were instruction fetches).
//
// Every value is formed by the operations of the per-step kernels in their order (same bits).
#include <type_traits>
#include <cooperative_groups.h>

#include "k_device.cuh"

namespace cg = cooperative_groups;

namespace hn {

namespace {

constexpr int kBlocks = 16, kThreads = 512, kEdge = kThreads - 32;

// Level l's shape.  Cluster levels (l > 5): block r has rows h r .. h r + h - 1, the last one also the last row; its
// arrays hold the flat range of these rows, a row and a node more on each side, from a 16-byte boundary.
template <int l>
struct Lv {
  static constexpr int n = (1 << l) + 1, N = n * n;
  static constexpr bool wide = l > 5;
  static constexpr int h = wide ? (1 << l) / kBlocks : n;
  // a thread has K rows of one of the columns 0 .. 2^l - 1 and at most one node more: of the last column (the last
  // warp, lane by row) or of the last row (the last block)
  static constexpr int K = wide ? (h * (1 << l) + kThreads - 1) / kThreads : 0;
  static constexpr int strips = wide ? h / K : 0;
  static constexpr int E = ((wide ? (h + 3) * n + 10 : N + 2 * n + 10) + 3) / 4 * 4;
  __host__ __device__ static constexpr int start(int rank) { return ((wide ? (rank * h - 1) : -1) * n - 4) & ~3; }
};
// floats of level l's arrays (bands 5..8, two iterates) and of those before it
template <int l> constexpr int floats() { return 6 * Lv<l>::E; }
template <int l> constexpr int before() {
  if constexpr (l >= kSpanTop) return 0;
  else return before<l + 1>() + floats<l + 1>();
}
constexpr int kCinvDoubles = 25 * 25;
constexpr int kFloats = before<2>() + floats<2>();
constexpr int kLow = Lv<5>::N + Lv<4>::N + Lv<3>::N + Lv<2>::N;
struct Tail {                             // behind the levels
  double cinv[kCinvDoubles], rd[kMaxCoarseM], sh[32];
  float low[3][kLow];                     // block 0, levels 5..2: diagonal, omega / D, right-hand side
  float e5[4 * Lv<5>::n];                 // level 5's iterate: the four rows around this block's of level 6
  float scale[kSpanTop + 1][5];
  int go;
};
constexpr int kBytes = (kFloats * 4 + 15) / 16 * 16 + ((int)sizeof(Tail) + 15) / 16 * 16;

// what a thread keeps of its nodes of a cluster level: diagonal, omega / D, right-hand side
template <int l>
struct Own { float dg[Lv<l>::K + 1], wd[Lv<l>::K + 1], rhs[Lv<l>::K + 1]; };
struct Owns { Own<8> o8; Own<7> o7; Own<6> o6; };

struct Job {
  const EngineDev& E;
  const ProblemDev& P;
  ProbState* st;
  float* sm;                              // this block's shared memory, its neighbours', block 0's
  float *lo, *hi, *b0;
  int p, rank, top, c, bc, want;
  __device__ __forceinline__ static Tail& tail(float* sm) { return *reinterpret_cast<Tail*>(sm + (kFloats + 3) / 4 * 4); }
  __device__ __forceinline__ Tail& mine() const { return tail(sm); }
};

// array a of level l (0..3: bands 5..8, 4 and 5: iterates) of block `rank`, by node
template <int l>
__device__ __forceinline__ float* arr(float* sm, int rank, int a) { return sm + before<l>() + a * Lv<l>::E - Lv<l>::start(rank); }
template <int l>
__device__ __forceinline__ float* vec(const Job& j, int b) { return arr<l>(j.sm, j.rank, 4 + b); }

// coefficient a (0: diagonal, 1: omega / D, 2: right-hand side) of the thread's k-th node of level l, node i
template <int l>
__device__ __forceinline__ float& coef(const Job& j, Owns& o, int a, int k, int i) {
  auto of = [&](auto& w) -> float& { return a == 0 ? w.dg[k] : a == 1 ? w.wd[k] : w.rhs[k]; };
  if constexpr (l == 8) return of(o.o8);
  else if constexpr (l == 7) return of(o.o7);
  else if constexpr (l == 6) return of(o.o6);
  else return j.mine().low[a][(l < 5 ? Lv<5>::N : 0) + (l < 4 ? Lv<4>::N : 0) + (l < 3 ? Lv<3>::N : 0) + i];
}

template <int l>
__device__ __forceinline__ void level_sync() {
  if constexpr (Lv<l>::wide) cg::this_cluster().sync();
  else __syncthreads();
}

// The thread's nodes of level l: f(k, node).  Cluster levels: all nodes of the block's rows (Dirichlet nodes have identity
// rows); below: the unknowns (the other nodes stay zero).
template <int l, class F>
__device__ __forceinline__ void for_extra(const Job& j, F&& f) {
  using G = Lv<l>;
  const int tid = threadIdx.x, last = j.rank == kBlocks - 1;
  if (tid >= kEdge) {
    if (tid - kEdge < G::h + last) f(G::K, (j.rank * G::h + tid - kEdge) * G::n + G::n - 1);
  } else if (last && tid < (1 << l)) {
    f(G::K, (1 << l) * G::n + tid);
  }
}
template <int l, class F>
__device__ __forceinline__ void for_own(const Job& j, F&& f) {
  using G = Lv<l>;
  if constexpr (G::wide) {
    const int col = threadIdx.x & ((1 << l) - 1), s = threadIdx.x >> l;
    if (s < G::strips) {
#pragma unroll
      for (int k = 0; k < G::K; ++k) f(k, (j.rank * G::h + s * G::K + k) * G::n + col);
    }
    for_extra<l>(j, f);
  } else {
    const UnknownRect r = unknown_rect(G::n, j.bc);
    const int col = threadIdx.x & ((1 << l) - 1);
    for (int y = threadIdx.x >> l; y < r.ny; y += kThreads >> l)
      if (col < r.nx) f(0, (r.y0 + y) * G::n + r.x0 + col);
    if (r.nx > (1 << l) && (int)threadIdx.x < r.ny) f(0, (r.y0 + threadIdx.x) * G::n + r.x0 + (1 << l));
  }
}

// store v at node i (the thread's k-th) of iterate b, and in the neighbours' ghost rows
template <int l>
__device__ __forceinline__ void put(const Job& j, int b, int k, int i, float v) {
  using G = Lv<l>;
  vec<l>(j, b)[i] = v;
  if (G::wide && (k == 0 || k >= G::K - 1)) {
    const int R0 = j.rank * G::h * G::n, R1 = R0 + (G::h - 1) * G::n;      // first and last row
    if (i < R0 + G::n && j.rank > 0) arr<l>(j.lo, j.rank - 1, 4 + b)[i] = v;
    if (i >= R1 && j.rank < kBlocks - 1) arr<l>(j.hi, j.rank + 1, 4 + b)[i] = v;
  }
}

// A v at a node from its nine band entries and values, in the band order of every other kernel
template <class Pol>
__device__ __forceinline__ float apply9(const float (&b)[9], const float (&x)[9]) {
  float acc = 0.0f;
  if constexpr (Pol::prec == P16) {
    acc = b[4] * x[4];
#pragma unroll
    for (int k = 0; k < 9; ++k)
      if (k != 4) acc = fmaf(b[k], x[k] - x[4], acc);
  } else {
#pragma unroll
    for (int k = 0; k < 9; ++k) acc = fmaf(b[k], x[k], acc);
  }
  return acc;
}

// f(k, i, A v, v) at the thread's nodes of level l, v: iterate b
template <class Pol, int l, class F>
__device__ __forceinline__ void for_applied(const Job& j, Owns& o, int b, F&& f) {
  using G = Lv<l>;
  constexpr int n = G::n;
  const float* v = vec<l>(j, b);
  const float *b5 = arr<l>(j.sm, j.rank, 0), *b6 = arr<l>(j.sm, j.rank, 1), *b7 = arr<l>(j.sm, j.rank, 2), *b8 = arr<l>(j.sm, j.rank, 3);
  auto direct = [&](int k, int i) {
    const float bd[9] = {b8[i - n - 1], b7[i - n], b6[i - n + 1], b5[i - 1], coef<l>(j, o, 0, k, i), b5[i], b6[i], b7[i], b8[i]};
    float x[9];
#pragma unroll
    for (int m = 0; m < 9; ++m) x[m] = v[i + (m / 3 - 1) * n + (m % 3 - 1)];
    f(k, i, apply9<Pol>(bd, x), x[4]);
  };
  if constexpr (G::wide && G::K > 1) {
    const int col = threadIdx.x & ((1 << l) - 1), s = threadIdx.x >> l;
    const int at = (j.rank * G::h + s * G::K) * n + col;
    static_assert(G::strips << l == kThreads, "every thread has rows");
    float x[9], up[3];                                   // up: bands 8, 7 and 6 of the row before, towards this node
#pragma unroll
    for (int m = 0; m < 6; ++m) x[3 + m] = v[at + (m / 3 - 1) * n + (m % 3 - 1)];
    up[0] = b8[at - n - 1]; up[1] = b7[at - n]; up[2] = b6[at - n + 1];
#pragma unroll
    for (int k = 0; k < G::K; ++k) {
      const int i = at + k * n;
#pragma unroll
      for (int m = 0; m < 6; ++m) x[m] = x[m + 3];
#pragma unroll
      for (int m = 0; m < 3; ++m) x[6 + m] = v[i + n + m - 1];
      const float bd[9] = {up[0], up[1], up[2], b5[i - 1], coef<l>(j, o, 0, k, i), b5[i], b6[i], b7[i], b8[i]};
      up[0] = b8[i - 1]; up[1] = bd[7]; up[2] = b6[i + 1];
      f(k, i, apply9<Pol>(bd, x), x[4]);
    }
    for_extra<l>(j, direct);
  } else {
    for_own<l>(j, direct);
  }
}

// iterate 0 += P e on the block's rows and ghost rows, e: the coarse iterate by node
template <int l>
__device__ __forceinline__ void prolong(const Job& j, const float* e) {
  using G = Lv<l>;
  float* x = vec<l>(j, 0);
  const int a = G::wide ? max(j.rank * G::h - 1, 0) * G::n : 0;
  const int b = G::wide ? min((j.rank + 1) * G::h + 1, G::n) * G::n : G::N;
  for (int i = a + threadIdx.x; i < b; i += kThreads) {
    const int iy = i / G::n, ix = i - iy * G::n;
    float add;
    if (prolong_value<float>(ix, iy, G::n, Lv<l - 1>::n, j.bc, [&](int q) { return e[q]; }, &add)) x[i] = x[i] + add;
  }
  __syncthreads();
}

// Sums of the tiles of the defects in memory (d.r), to the problem's partials: the loads before, the sums after the
// second smoothing step's work
template <int l>
struct TileSums {
  static constexpr int tiles = (Lv<l>::N + kTile - 1) / kTile, per = (tiles + kBlocks * (kThreads / 32) - 1) / (kBlocks * (kThreads / 32));
  float r[per][4];
  __device__ __forceinline__ static int tile(const Job& j, int q) { return j.rank + kBlocks * ((int)(threadIdx.x >> 5) + q * (kThreads / 32)); }
  __device__ __forceinline__ void load(const Job& j) {
    const float* d = static_cast<const float*>(j.P.lev[l].r);
#pragma unroll
    for (int q = 0; q < per; ++q)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = tile(j, q) * kTile + (threadIdx.x & 31) * 4 + k;
        r[q][k] = i < Lv<l>::N ? __ldcg(d + i) : 0.0f;
      }
  }
  __device__ __forceinline__ void sum(const Job& j) {
#pragma unroll
    for (int q = 0; q < per; ++q) {
      const int t = tile(j, q);
      if (t >= tiles) break;
      const float2 v = tile_sumsq(r[q]);
      if ((threadIdx.x & 31) == 0) store_partial(j.E.partial + j.E.fine_off[j.p] + t, v);
    }
  }
};

template <class Pol, int l>
__device__ __forceinline__ void low(const Job& j, Owns& o);

// Level l from its right-hand side and its first smoothing step (in iterate 1; checked, the launch's top level: from
// iterate 0), to its result in iterate 0; false if the problem leaves.  One copy of the stencil code a level serves
// all its steps: as straight-line code they missed the instruction cache at every step.
template <class Pol, int l, bool TOP>
__device__ __forceinline__ bool level(const Job& j, Owns& o, bool checked) {
  using G = Lv<l>;
  enum { FIRST = 0, SECOND, DEFECT, POST1, POST2 };
#pragma unroll 1
  for (int step = TOP && checked ? FIRST : SECOND; step <= POST2; ++step) {
    const int b = step == SECOND || step == POST2;
    const bool sums = TOP && checked && step == SECOND;
    TileSums<TOP ? l : 6> t;
    if (sums) t.load(j);
    float* r = TOP ? static_cast<float*>(j.P.lev[l].r) : nullptr;
    for_applied<Pol, l>(j, o, b, [&](int k, int i, float ax, float x) {
      const float q = coef<l>(j, o, 2, k, i) - ax;
      if (TOP && step == FIRST) r[i] = q;
      put<l>(j, 1 - b, k, i, step == DEFECT ? q : fmaf(coef<l>(j, o, 1, k, i), q, x));
    });
    if (sums) t.sum(j);
    level_sync<l>();
    if (sums && j.rank == 0) {
      const double sum = problem_norm_sum(j.E.partial + j.E.fine_off[j.p], t.tiles, j.mine().sh, true);
      if (threadIdx.x < 32) {
        int go = 0;
        if (threadIdx.x == 0) {
          pre_check(*j.st, j.E.prm, sqrt(sum));
          go = *reinterpret_cast<volatile int*>(&j.st->phase) == j.want;
        }
        go = __shfl_sync(kFull, go, 0);
        if (threadIdx.x < kBlocks) Job::tail(cg::this_cluster().map_shared_rank(j.sm, threadIdx.x)).go = go;
      }
    }
    if (step != DEFECT) continue;
    if (TOP && checked && !j.mine().go) return false;
    // the restricted defect and the next level's first step
    const float* d = vec<l>(j, 1);
    auto restricted = [&](int i) {
      const int J = i / Lv<l - 1>::n, I = i - J * Lv<l - 1>::n;
      return restrict_value<float>(I, J, Lv<l - 1>::n, G::n, j.bc, [&](long long q) { return d[(int)q]; });
    };
    if constexpr (l == 6) {               // into block 0: level 5's rows of this block
      constexpr int nc = Lv<5>::n;
      const int a = j.rank * (G::h / 2) * nc, e = a + (G::h / 2 + (j.rank == kBlocks - 1)) * nc;
      for (int i = a + threadIdx.x; i < e; i += kThreads) Job::tail(j.b0).low[2][i] = restricted(i);
    } else {
      for_own<l - 1>(j, [&](int k, int i) {
        const float v = restricted(i);
        coef<l - 1>(j, o, 2, k, i) = v;
        put<l - 1>(j, 1, k, i, mul_rn(coef<l - 1>(j, o, 1, k, i), v));
      });
    }
    level_sync<l>();
    if constexpr (l == 6) {
      if (j.rank == 0) {
        for_own<5>(j, [&](int k, int i) { put<5>(j, 1, k, i, mul_rn(coef<5>(j, o, 1, k, i), coef<5>(j, o, 2, k, i))); });
        __syncthreads();
        low<Pol, 5>(j, o);
        // its result's rows to the blocks that prolong from them
        cg::cluster_group cl = cg::this_cluster();
        for_own<5>(j, [&](int, int i) {
          constexpr int n = Lv<5>::n;
          const int J = i / n;
          const float v = vec<5>(j, 0)[i];
          for (int q = max(0, (J - 1) / 2); q <= min(kBlocks - 1, (J + 1) / 2); ++q)     // rows 2 q - 1 .. 2 q + 2
            if (J <= 2 * q + 2 && J >= 2 * q - 1) Job::tail(cl.map_shared_rank(j.sm, q)).e5[i - (2 * q - 1) * n] = v;
        });
      }
      cg::this_cluster().sync();
      prolong<6>(j, j.mine().e5 - (2 * j.rank - 1) * Lv<5>::n);
    } else if constexpr (G::wide) {
      level<Pol, l - 1, false>(j, o, false);
      prolong<l>(j, vec<l - 1>(j, 0));
    } else {
      low<Pol, l - 1>(j, o);
      prolong<l>(j, vec<l - 1>(j, 0));
    }
  }
  return true;
}

// block 0: the levels l..c, l <= 5, from the first step of level l; the result in iterate 0
template <class Pol, int l>
__device__ __forceinline__ void low(const Job& j, Owns& o) {
  if (l == j.c) {
    if constexpr (l <= 4) {
      Tail& t = j.mine();
      const UnknownRect ur = unknown_rect(Lv<l>::n, j.bc);
      const int m = j.P.m, u = threadIdx.x;   // (at most kMaxCoarseM unknowns)
      const int iu = (u / ur.nx + ur.y0) * Lv<l>::n + u % ur.nx + ur.x0;
      if (u < m) t.rd[u] = double(coef<l>(j, o, 2, 0, iu));
      __syncthreads();
      if (u < m) {
        const double* row = (m * m <= kCinvDoubles ? t.cinv : j.P.cinv) + u * m;
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
        int v = 0;
        for (; v + 3 < m; v += 4) {
          a0 = fma(row[v], t.rd[v], a0);
          a1 = fma(row[v + 1], t.rd[v + 1], a1);
          a2 = fma(row[v + 2], t.rd[v + 2], a2);
          a3 = fma(row[v + 3], t.rd[v + 3], a3);
        }
        if (v < m) a0 = fma(row[v], t.rd[v], a0);
        if (v + 1 < m) a1 = fma(row[v + 1], t.rd[v + 1], a1);
        if (v + 2 < m) a2 = fma(row[v + 2], t.rd[v + 2], a2);
        vec<l>(j, 0)[iu] = float((a0 + a1) + (a2 + a3));
      }
      __syncthreads();
    }
    return;
  }
  if constexpr (l > 2) level<Pol, l, false>(j, o, false);
}

template <class Pol, int l>
__device__ __forceinline__ void run(const Job& j, Owns& o, bool checked, int loop) {
  using G = Lv<l>;
  const LevelDev& d = j.P.lev[l];
  {
    const float* b = static_cast<const float*>(d.rhs);
    for_own<l>(j, [&](int k, int i) { coef<l>(j, o, 2, k, i) = __ldcg(b + i); });
    if (checked) {
      const float* x = static_cast<const float*>(d.x[0]);
      const int a = max(j.rank * G::h - 1, 0) * G::n, e = min((j.rank + 1) * G::h + 1, G::n) * G::n;
      for (int i = a + threadIdx.x; i < e; i += kThreads) vec<l>(j, 0)[i] = __ldcg(x + i);
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  cg::this_cluster().sync();
  do {
    if (!checked) {
      for_own<l>(j, [&](int k, int i) { put<l>(j, 1, k, i, mul_rn(coef<l>(j, o, 1, k, i), coef<l>(j, o, 2, k, i))); });
      level_sync<l>();
    }
    if (!level<Pol, l, true>(j, o, checked)) return;
    float* x = static_cast<float*>(d.x[0]);
    for_own<l>(j, [&](int, int i) { x[i] = vec<l>(j, 0)[i]; });
    checked = true;
  } while (loop);
}

// start the copies of level l's constant data
template <class Pol, int l>
__device__ __forceinline__ void stage(const Job& j, Owns& o) {
  using G = Lv<l>;
  using B = typename Pol::B;
  if (l > j.top || l < j.c || (!G::wide && j.rank > 0)) return;
  const LevelDev& d = j.P.lev[l];
  const Tail& t = j.mine();
  const int a = G::start(j.rank);
  // rows to the last own one (the others' entries stay zero)
  const int end = G::wide ? (j.rank * G::h + G::h + (j.rank == kBlocks - 1)) * G::n : G::N;
  for (int k = 0; k < 4; ++k) {
    const B* src = static_cast<const B*>(d.band[5 + k]);
    float* dst = arr<l>(j.sm, j.rank, k);
    for (int i = a + 4 * (int)threadIdx.x; i < end; i += 4 * kThreads) {
      if constexpr (Pol::prec == P32) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst + i)), "l"(src + i) : "memory");
      } else {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(src + i));
        const float2 p = __half22float2(*reinterpret_cast<const __half2*>(&v.x)), q = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
        const float s = t.scale[l][k + 1];
        *reinterpret_cast<float4*>(dst + i) = make_float4(__fmul_rn(s, p.x), __fmul_rn(s, p.y), __fmul_rn(s, q.x), __fmul_rn(s, q.y));
      }
    }
  }
  for_own<l>(j, [&](int k, int i) {
    const B v = __ldg(static_cast<const B*>(d.band[4]) + i);
    if constexpr (Pol::prec == P32) coef<l>(j, o, 0, k, i) = v;
    else coef<l>(j, o, 0, k, i) = __fmul_rn(t.scale[l][0], __half2float(v));
    coef<l>(j, o, 1, k, i) = __ldg(d.wdf + i);
  });
}

template <class Pol>
__global__ void __launch_bounds__(kThreads, 1) k_span(const __grid_constant__ EngineDev E, int T, int want, int loop) {
  extern __shared__ __align__(128) float sm[];
  pdl_trigger();
  cg::cluster_group cl = cg::this_cluster();
  const int p = blockIdx.x / kBlocks, rank = (int)cl.block_rank();
  const ProblemDev& P = E.P[p];
  const int L = P.L, top = min(L, T);
  if (top <= 5) {                         // (not launched for such a problem; an empty slot)
    pdl_wait();
    return;
  }
  const Job j{E, P, E.S + p, sm, cl.map_shared_rank(sm, max(rank - 1, 0)), cl.map_shared_rank(sm, min(rank + 1, kBlocks - 1)),
              cl.map_shared_rank(sm, 0), p, rank, top, P.coarse, P.lev[top].bc, want};
  for (int i = threadIdx.x; i < kBytes / 16; i += kThreads) reinterpret_cast<float4*>(sm)[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  __syncthreads();
  Tail& t = j.mine();
  if (Pol::prec == P16) {
    for (int i = threadIdx.x; i < 5 * (top - j.c + 1); i += kThreads) t.scale[j.c + i / 5][i % 5] = P.lev[j.c + i / 5].scale[4 + i % 5];
    __syncthreads();
  }
  Owns o;
  stage<Pol, 8>(j, o);
  stage<Pol, 7>(j, o);
  stage<Pol, 6>(j, o);
  stage<Pol, 5>(j, o);
  stage<Pol, 4>(j, o);
  stage<Pol, 3>(j, o);
  stage<Pol, 2>(j, o);
  if (rank == 0 && P.m * P.m <= kCinvDoubles)
    for (int q = threadIdx.x; q < P.m * P.m; q += kThreads) t.cinv[q] = __ldg(P.cinv + q);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  pdl_wait();
  if (__ldcg(&j.st->phase) != want) {
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    return;
  }
  const bool checked = top == L && !__ldcg(&j.st->zero_top) && E.prm.solver != SOLVER_PCG;
  loop = loop && top == L && E.prm.solver != SOLVER_PCG;
  switch (top) {
    case 8: run<Pol, 8>(j, o, checked, loop); break;
    case 7: run<Pol, 7>(j, o, checked, loop); break;
    default: run<Pol, 6>(j, o, checked, loop); break;
  }
}

template <class Pol>
cudaError_t launch_span_t(const EngineDev& E, int T, int want, int loop, cudaStream_t s) {
  auto kern = k_span<Pol>;
  static const cudaError_t ready = [&] {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kBytes);
  }();
  if (ready != cudaSuccess) return ready;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(E.nprob * kBlocks), 1, 1);
  cfg.blockDim = dim3((unsigned)kThreads, 1, 1);
  cfg.dynamicSmemBytes = (size_t)kBytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)kBlocks;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.numAttrs = 1;
  if (pdl_launch(E.pdl, (int)cfg.gridDim.x)) {
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
  }
  cfg.attrs = attr;
  return cudaLaunchKernelEx(&cfg, kern, E, T, want, loop);
}

}  // namespace

cudaError_t launch_span(const EngineDev& E, int T, int want, int loop, cudaStream_t s) {
  if (E.prm.prec == P32) return launch_span_t<F32>(E, T, want, loop, s);
  if (E.prm.prec == P16) return launch_span_t<F16>(E, T, want, loop, s);
  return cudaErrorInvalidValue;
}

}  // namespace hn
