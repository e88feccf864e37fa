// The V(2,2) cycle in FP64 on the levels coarse..T, T <= kWideTop, of one problem by a cluster of 16 blocks, with
// the exact coarse solver.
//
// What bounds it: a chain of about 30 dependent steps, each the FP64 pipe's time for a warp's stencils (nine FMAs
// of some 70 cycles of a quarter of an SM each: 0.35 us for one warp, 0.7 us for two) and a barrier.  Levels 6 and 5
// are spread over the cluster by rows (a level-6 row set of 4 x 63 nodes is eight warps, two to a quarter SM), one
// thread a node; a thread keeps its node's bands, omega / D and right-hand side in registers for the whole
// launch, only the iterates and defects lie in shared memory, and a step stores its first and last row into the
// neighbours' ghost rows itself (three buffers a level: a step never writes what a neighbour may still read).
// Levels 4 to coarse run in block 0 alone.  The general kernel (k_tail) stages every array in shared memory, has
// block 0 do level 4 and 5 nodes in several rounds and, for a problem's own finest level, whose residual is
// checked, runs over L2.
//
// The lagged check (finest level here, iterate not zero) costs no barrier: the defects of a 128-node tile go to one
// block, its sum to block 0, and the decision is back with the barrier that ends the defect step; an iterate
// is overwritten in shared memory only, the accepted one is in memory.  So a problem whose finest level is here runs
// all its cycles in one launch.
//
// Measured: 92 -> 20.5 us a cycle at L = 6 (solve 890 -> 295 us), the tail below level 7 at L = 10 56.6 -> 37.9 us
// with its launch (the finer levels leave little of its data in L2; solve 2.67 -> 2.50 ms).
//
// Every value is formed by the operations of the per-step kernels in their order (same bits).
#include <type_traits>
#include <cooperative_groups.h>

#include "k_device.cuh"

namespace cg = cooperative_groups;

namespace hn {

namespace {

constexpr int kWideThreads = 352, kWideBlocks = 16;     // 65 x 5 nodes at most

// shared memory of a block; cluster levels: own rows with a ghost row and column on each side
template <int l> constexpr int wide_pitch() { return (1 << l) + 3; }
template <int l> constexpr int wide_rows() { return l > 4 ? (1 << l) / kWideBlocks + 3 : (1 << l) + 3; }
struct Wide {
  double v6[3][wide_rows<6>() * wide_pitch<6>()];
  double v5[3][wide_rows<5>() * wide_pitch<5>()];
  double v4[3][wide_rows<4>() * wide_pitch<4>()];     // block 0
  double v3[3][wide_rows<3>() * wide_pitch<3>()];
  double v2[3][wide_rows<2>() * wide_pitch<2>()];
  double e4[3 * wide_pitch<4>()];                     // level 4's iterate, the rows around this block's
  double b4[wide_rows<4>() * wide_pitch<4>()];        // block 0: level 4's right-hand side
  double tile[4][kTile];                              // defects of the tiles this block sums
  double tsum[64];                                    // block 0: sums of the tiles
  double rd[kMaxCoarseM], sh[32];
  int go;
};
template <int l>
__device__ __forceinline__ double (*vecs(Wide& s))[wide_rows<l>() * wide_pitch<l>()] {
  if constexpr (l == 6) return s.v6;
  else if constexpr (l == 5) return s.v5;
  else if constexpr (l == 4) return s.v4;
  else if constexpr (l == 3) return s.v3;
  else return s.v2;
}

// The block's nodes of level l: the rectangle `r` of its own rows, row by row, one thread each
template <int l>
struct Rows {
  static constexpr int n = (1 << l) + 1, W = wide_pitch<l>(), h = l > 4 ? (1 << l) / kWideBlocks : n;
  int R0, R1;                             // own rows
  UnknownRect r;
  __device__ __forceinline__ Rows(int rank, const UnknownRect& rect) : r(rect) {
    R0 = l > 4 ? rank * h : 0;
    R1 = l > 4 ? R0 + h + (rank == kWideBlocks - 1) : n;
  }
  __device__ __forceinline__ int at(int x, int y) const { return (y - R0 + 1) * W + x + 1; }
};

// a thread's node: its place in the block's arrays and what stays in registers
struct Node {
  int x, y, at;
  bool on, first, last;                   // first, last: in a row that is a neighbour's ghost row
  double a[9], wd, rhs;
};

template <int l>
__device__ __forceinline__ void node_init(Node& q, const Rows<l>& g, int rank, const LevelDev& d) {
  const int ya = max(g.R0, g.r.y0), yb = min(g.R1, g.r.y0 + g.r.ny), w = g.r.nx, i = threadIdx.x;
  q.on = i < (yb - ya) * w;
  q.y = ya + i / w;
  q.x = g.r.x0 + i % w;
  q.at = q.on ? g.at(q.x, q.y) : g.W + 1;
  q.first = l > 4 && q.on && q.y == g.R0 && rank > 0;
  q.last = l > 4 && q.on && q.y == g.R1 - 1 && rank < kWideBlocks - 1;
  q.rhs = 0.0;
  if (!q.on) return;
  const int f = q.y * g.n + q.x;
#pragma unroll
  for (int k = 0; k < 9; ++k) q.a[k] = __ldg(static_cast<const double*>(d.band[k]) + f);
  q.wd = __ldg(d.wdinv + f);
}

// b - A v at the node
template <int l>
__device__ __forceinline__ double defect(const Node& q, const double* v) {
  double acc = q.rhs;
#pragma unroll
  for (int k = 0; k < 9; ++k) acc = fma(-q.a[k], v[q.at + (k / 3 - 1) * wide_pitch<l>() + (k % 3 - 1)], acc);
  return acc;
}

// neighbours' shared memory (their own for the first and last block)
struct Peers {
  Wide *me, *lo, *hi, *b0;
};

template <int l>
__device__ __forceinline__ void put(const Peers& c, const Node& q, int k, double v) {
  if (!q.on) return;
  vecs<l>(*c.me)[k][q.at] = v;
  if constexpr (l > 4) {
    constexpr int shift = Rows<l>::h * wide_pitch<l>();
    if (q.first) vecs<l>(*c.lo)[k][q.at + shift] = v;
    if (q.last) vecs<l>(*c.hi)[k][q.at - shift] = v;
  }
}

template <int l>
__device__ __forceinline__ void step_sync() {
  if constexpr (l > 4) cg::this_cluster().sync();
  else __syncthreads();
}

// a smoothing step from buffer i to buffer o
template <int l>
__device__ __forceinline__ void smooth(const Peers& c, const Node& q, int i, int o) {
  const double* v = vecs<l>(*c.me)[i];
  if (q.on) put<l>(c, q, o, fma(q.wd, defect<l>(q, v), v[q.at]));
  step_sync<l>();
}

// the restricted defect (buffer 2 of level l) at the coarse node (I, J)
template <int l>
__device__ __forceinline__ double restricted(const Wide& s, const Rows<l>& g, int I, int J, int bc) {
  const double* r = vecs<l>(const_cast<Wide&>(s))[2];
  return restrict_value_xy<double>(I, J, Rows<l - 1>::n, g.n, bc, [&](int y, int x) { return r[g.at(x, y)]; });
}

// buffer 1 = buffer 0 + P e on the level's rows and ghost rows; e(cy, cx): the coarse iterate.  The sum that an odd
// row or column adds to is zero otherwise, so all nodes do the same four operations (the weights are exact).
template <int l, class F>
__device__ __forceinline__ void prolong(Wide& s, const Rows<l>& g, int bc, F&& e) {
  const int ya = max(g.R0 - (l > 4), g.r.y0), yb = min(g.R1 + (l > 4), g.r.y0 + g.r.ny), w = g.r.nx;
  for (int i = threadIdx.x; i < (yb - ya) * w; i += kWideThreads) {
    const int dy = i / w, y = ya + dy, x = g.r.x0 + i - dy * w, at = g.at(x, y);
    const bool ox = x & 1, oy = y & 1;
    const int cx = x >> 1, cy = y >> 1;
    const double a = e(cy, cx), b = ox ? e(cy, cx + 1) : 0.0, c = oy ? e(cy + 1, cx) : 0.0;
    const double d = ox && oy ? e(cy + 1, cx + 1) : 0.0, wt = ox == oy ? (ox ? 0.25 : 1.0) : 0.5;
    const double v = vecs<l>(s)[0][at];
    vecs<l>(s)[1][at] = is_dirichlet(x, y, g.n, bc) ? v : fma(wt, ((a + b) + c) + d, v);
  }
  __syncthreads();
}

struct Job {
  const EngineDev& E;
  const ProblemDev& P;
  ProbState* st;
  int p, rank, top, c, bc, want;
  bool full;                              // a given iterate: the top level's Dirichlet nodes take part
};

// The first smoothing step of the launch's top level l > 4, from a nonzero iterate in buffer 0 (checked) or from zero
template <int l>
__device__ __forceinline__ void first_step(const Job& j, const Peers& c, const Node& q, bool checked) {
  if (q.on) {
    if (checked) {
      const double* v = vecs<l>(*c.me)[0];
      const double r = defect<l>(q, v);
      put<l>(c, q, 1, fma(q.wd, r, v[q.at]));
      const int f = q.y * Rows<l>::n + q.x, t = f / kTile, o = min(t >> (l - 5), kWideBlocks - 1);
      cg::this_cluster().map_shared_rank(c.me, o)->tile[t - (o << (l - 5))][f % kTile] = r;
    } else {
      put<l>(c, q, 1, mul_rn(q.wd, q.rhs));
    }
  }
  cg::this_cluster().sync();
}

// The tiles' sums to block 0 (after the first step), and block 0's decision (after the second), which every block
// reads in s.go after the next barrier.
template <int l>
__device__ __forceinline__ void check_tiles(const Job& j, const Peers& c) {
  constexpr int n = Rows<l>::n, tiles = (n * n + kTile - 1) / kTile;
  const int lane = threadIdx.x & 31, k = (int)(threadIdx.x >> 5) - (kWideThreads / 32 - 4);   // the last warps
  const int t = (j.rank << (l - 5)) + k;
  const int mine = j.rank == kWideBlocks - 1 ? 4 : 1 << (l - 5);
  if (k < 0 || k >= mine || t >= tiles) return;
  double r[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) r[m] = c.me->tile[k][lane * 4 + m];
  const double v = tile_sumsq(r);
  if (lane == 0) c.b0->tsum[t] = v;
}
template <int l>
__device__ __forceinline__ void check_decide(const Job& j, const Peers& c) {
  constexpr int n = Rows<l>::n, tiles = (n * n + kTile - 1) / kTile;
  static_assert(tiles <= 64, "two tile sums a lane");
  if (j.rank != 0 || (threadIdx.x >> 5) != kWideThreads / 32 - 1) return;
  const int lane = threadIdx.x & 31;
  // problem_partial_sum's warps 0 and 1 (the others add zeros)
  double sum = warp_sum(lane < tiles ? c.me->tsum[lane] : 0.0);
  if (tiles > 32) sum += warp_sum(lane + 32 < tiles ? c.me->tsum[lane + 32] : 0.0);
  int go = 0;
  if (lane == 0) {
    pre_check(*j.st, j.E.prm, sqrt(sum));
    go = *reinterpret_cast<volatile int*>(&j.st->phase) == j.want;
  }
  go = __shfl_sync(kFull, go, 0);
  if (lane < kWideBlocks) cg::this_cluster().map_shared_rank(c.me, lane)->go = go;
}

// Level l's first smoothing step is done (buffer 1): the second, the defect, and its restriction into the next
// level's right-hand side, with that level's first smoothing step where its nodes are here.  checked: decide
// meanwhile (cluster levels); false if the problem leaves.
template <int l>
__device__ __forceinline__ bool down_rest(const Job& j, const Peers& c, const Rows<l>& g, const Node& q, Node& qc,
                                          bool checked) {
  if constexpr (l > 4)
    if (checked) check_tiles<l>(j, c);
  smooth<l>(c, q, 1, 0);
  if constexpr (l > 4)
    if (checked) check_decide<l>(j, c);
  if (q.on) put<l>(c, q, 2, defect<l>(q, vecs<l>(*c.me)[0]));
  step_sync<l>();
  if (l > 4 && checked && !c.me->go) return false;
  if constexpr (l == 5) {                 // into block 0
    const UnknownRect r4 = unknown_rect(Rows<4>::n, j.bc);
    const int ya = max(j.rank, r4.y0), yb = min(j.rank + 1 + (j.rank == kWideBlocks - 1), r4.y0 + r4.ny);
    const int i = threadIdx.x;
    if (i < (yb - ya) * r4.nx) {
      const int y = ya + i / r4.nx, x = r4.x0 + i % r4.nx;
      c.b0->b4[(y + 1) * wide_pitch<4>() + x + 1] = restricted<l>(*c.me, g, x, y, j.bc);
    }
  } else if (qc.on) {
    qc.rhs = restricted<l>(*c.me, g, qc.x, qc.y, j.bc);
    put<l - 1>(c, qc, 1, mul_rn(qc.wd, qc.rhs));
  }
  step_sync<l>();
  return true;
}

// The residual check of a problem whose finest level l <= 4 is block 0's: its defects in buffer 2
template <int l>
__device__ __forceinline__ bool check_low(const Job& j, Wide& s) {
  constexpr int n = Rows<l>::n, tiles = (n * n + kTile - 1) / kTile;
  const int lane = threadIdx.x & 31;
  double* part = j.E.partial + j.E.fine_off[j.p];
  for (int t = threadIdx.x >> 5; t < tiles; t += kWideThreads / 32) {
    double r[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int f = t * kTile + lane * 4 + k;
      r[k] = f < n * n ? vecs<l>(s)[2][(f / n + 1) * wide_pitch<l>() + f % n + 1] : 0.0;
    }
    const double v = tile_sumsq(r);
    if (lane == 0) part[t] = v;
  }
  __syncthreads();
  const double sum = problem_norm_sum(part, tiles, s.sh);
  if (threadIdx.x == 0) {
    pre_check(*j.st, j.E.prm, sqrt(sum));
    s.go = *reinterpret_cast<volatile int*>(&j.st->phase) == j.want;
  }
  __syncthreads();
  return s.go;
}

// The cycle on levels l..c (l <= 4) in block 0.  start: from l's right-hand side and, checked, its nonzero iterate
// in buffer 0 (the problem's finest level; false if the problem leaves); else l's first step is done.
template <int l>
__device__ __forceinline__ bool low(const Job& j, const Peers& c, Node* q, bool start, bool checked) {
  Node& me = q[l];
  const Rows<l> g(0, start && j.full ? UnknownRect{0, 0, Rows<l>::n, Rows<l>::n} : unknown_rect(Rows<l>::n, j.bc));
  if (checked) {
    const double* v = vecs<l>(*c.me)[0];
    if (me.on) {
      const double r = defect<l>(me, v);
      put<l>(c, me, 2, r);
      put<l>(c, me, 1, fma(me.wd, r, v[me.at]));
    }
    __syncthreads();
    if (!check_low<l>(j, *c.me)) return false;
  } else if (start && l > j.c) {
    if (me.on) put<l>(c, me, 1, mul_rn(me.wd, me.rhs));
    __syncthreads();
  }
  if (l == j.c) {
    // the exact solve, one thread per unknown
    const UnknownRect ur = unknown_rect(Rows<l>::n, j.bc);
    const int m = j.P.m, u = threadIdx.x;
    const int x = ur.x0 + u % ur.nx, y = ur.y0 + u / ur.nx;
    double* rd = c.me->rd;
    if (u < m) rd[u] = j.top == l ? __ldcg(static_cast<const double*>(j.P.lev[l].rhs) + y * Rows<l>::n + x) : me.rhs;
    __syncthreads();
    if (u < m) {
      const double* row = j.P.cinv + u * m;
      double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
      int v = 0;
      for (; v + 3 < m; v += 4) {
        a0 = fma(__ldg(row + v), rd[v], a0);
        a1 = fma(__ldg(row + v + 1), rd[v + 1], a1);
        a2 = fma(__ldg(row + v + 2), rd[v + 2], a2);
        a3 = fma(__ldg(row + v + 3), rd[v + 3], a3);
      }
      if (v < m) a0 = fma(__ldg(row + v), rd[v], a0);
      if (v + 1 < m) a1 = fma(__ldg(row + v + 1), rd[v + 1], a1);
      if (v + 2 < m) a2 = fma(__ldg(row + v + 2), rd[v + 2], a2);
      vecs<l>(*c.me)[0][g.at(x, y)] = (a0 + a1) + (a2 + a3);
    }
    if (start && j.full && me.on && is_dirichlet(me.x, me.y, Rows<l>::n, j.bc)) vecs<l>(*c.me)[0][me.at] = 0.0;
    __syncthreads();
    return true;
  }
  if constexpr (l > 2) {
    down_rest<l>(j, c, g, me, q[l - 1], false);
    low<l - 1>(j, c, q, false, false);
    const double* e = vecs<l - 1>(*c.me)[0];
    prolong<l>(*c.me, g, j.bc, [&](int cy, int cx) { return e[(cy + 1) * wide_pitch<l - 1>() + cx + 1]; });
    smooth<l>(c, me, 1, 2);
    smooth<l>(c, me, 2, 0);
  }
  return true;
}

// block 0's levels below the cluster's; its result's rows to the blocks that prolong from them
__device__ __forceinline__ void low_of_cluster(const Job& j, const Peers& c, Node* q) {
  if (j.rank == 0) {
    q[4].rhs = c.me->b4[q[4].at];
    low<4>(j, c, q, true, false);
    cg::cluster_group cl = cg::this_cluster();
    constexpr int W = wide_pitch<4>();
    if (q[4].on) {
      const double v = c.me->v4[0][q[4].at];
      for (int r = max(0, q[4].y - 1); r <= min(kWideBlocks - 1, q[4].y + 1); ++r)
        cl.map_shared_rank(c.me, r)->e4[(q[4].y - r + 1) * W + q[4].x + 1] = v;
    }
  }
  cg::this_cluster().sync();
}

// The cycle(s) of a launch whose top level is l: `loop`: until the problem leaves
template <int l>
__device__ __forceinline__ void run(const Job& j, const Peers& c, Node* q, bool checked, int loop) {
  constexpr int n = Rows<l>::n;
  const UnknownRect all{0, 0, n, n};
  const Rows<l> g(j.rank, j.full ? all : unknown_rect(n, j.bc));
  const LevelDev& d = j.P.lev[l];
  Node& me = q[l];
  if (j.full) node_init<l>(me, g, j.rank, d);
  if (me.on) me.rhs = __ldcg(static_cast<const double*>(d.rhs) + me.y * n + me.x);
  if (checked) {                          // own rows and ghost rows
    const int ya = max(g.R0 - 1, 0), yb = min(g.R1 + 1, n);
    for (int i = threadIdx.x; i < (yb - ya) * n; i += kWideThreads)
      vecs<l>(*c.me)[0][g.at(i % n, ya + i / n)] = __ldcg(static_cast<const double*>(d.x[0]) + ya * n + i);
  }
  // An iterate that another kernel reads is 0 on the Dirichlet nodes, whatever a caller has put there (hn_mg_apply takes
  // any vector); that of a solve's own cycles is so from the start, or `full`.
  if (!loop && !j.full)
    for (int i = threadIdx.x; i < (g.R1 - g.R0) * n; i += kWideThreads) {
      const int y = g.R0 + i / n, x = i % n;
      if (is_dirichlet(x, y, n, j.bc)) static_cast<double*>(d.x[0])[y * n + x] = 0.0;
    }
  step_sync<l>();
  for (;;) {
    if constexpr (l > 4) {
      first_step<l>(j, c, me, checked);
      if (!down_rest<l>(j, c, g, me, q[l - 1], checked)) return;
      const Rows<5> g5(j.rank, unknown_rect(Rows<5>::n, j.bc));
      if constexpr (l == 6) down_rest<5>(j, c, g5, q[5], q[4], false);
      low_of_cluster(j, c, q);
      auto e4 = [&](int cy, int cx) { return c.me->e4[(cy - j.rank + 1) * wide_pitch<4>() + cx + 1]; };
      if constexpr (l == 6) {
        prolong<5>(*c.me, g5, j.bc, e4);
        smooth<5>(c, q[5], 1, 2);
        smooth<5>(c, q[5], 2, 0);
        const double* e = c.me->v5[0];
        prolong<6>(*c.me, g, j.bc, [&](int cy, int cx) { return e[(cy - g5.R0 + 1) * wide_pitch<5>() + cx + 1]; });
      } else {
        prolong<5>(*c.me, g, j.bc, e4);
      }
      smooth<l>(c, me, 1, 2);
      smooth<l>(c, me, 2, 0);
    } else {
      if (!low<l>(j, c, q, true, checked)) return;
    }
    if (me.on) static_cast<double*>(d.x[0])[me.y * n + me.x] = vecs<l>(*c.me)[0][me.at];
    if (!loop) return;
    checked = true;
  }
}

__global__ void __launch_bounds__(kWideThreads, 1) k_wide(const __grid_constant__ EngineDev E, int T, int want, int loop) {
  __shared__ Wide s;
  pdl_trigger();
  cg::cluster_group cl = cg::this_cluster();
  const int p = blockIdx.x / kWideBlocks, rank = (int)cl.block_rank();
  // constant data before the wait for the preceding launch (descriptors change only between launches)
  const ProblemDev& P = E.P[p];
  const int L = P.L, top = min(L, T);
  if (L < HN_MIN_LEVEL || (rank > 0 && top <= 4)) return;
  Job j{E, P, E.S + p, p, rank, top, P.coarse, P.lev[top].bc, want, false};
  Node q[7];
  auto init = [&](auto level) {
    constexpr int l = decltype(level)::value;
    q[l].on = false;
    if (l <= top && l >= j.c && (l > 4 || rank == 0))
      node_init<l>(q[l], Rows<l>(rank, unknown_rect(Rows<l>::n, j.bc)), rank, P.lev[l]);
  };
  init(std::integral_constant<int, 6>{});
  init(std::integral_constant<int, 5>{});
  init(std::integral_constant<int, 4>{});
  init(std::integral_constant<int, 3>{});
  init(std::integral_constant<int, 2>{});
  for (int i = threadIdx.x; i < (int)(sizeof(Wide) / 8); i += kWideThreads) reinterpret_cast<double*>(&s)[i] = 0.0;
  const Peers c{&s, cl.map_shared_rank(&s, max(rank - 1, 0)), cl.map_shared_rank(&s, min(rank + 1, kWideBlocks - 1)),
                cl.map_shared_rank(&s, 0)};
  __syncthreads();
  pdl_wait();
  if (__ldcg(&j.st->phase) != want) return;
  const bool checked = top == L && !__ldcg(&j.st->zero_top) && E.prm.solver != SOLVER_PCG;
  j.full = top == L && !__ldcg(&j.st->x_zero);
  loop = loop && top == L && E.prm.solver != SOLVER_PCG;
  switch (top) {
    case 6: run<6>(j, c, q, checked, loop); break;
    case 5: run<5>(j, c, q, checked, loop); break;
    case 4: run<4>(j, c, q, checked, loop); break;
    case 3: run<3>(j, c, q, checked, loop); break;
    case 2: run<2>(j, c, q, checked, loop); break;
  }
}

}  // namespace

cudaError_t launch_wide(const EngineDev& E, int T, int want, int loop, cudaStream_t s) {
  auto kern = k_wide;
  static const cudaError_t ready = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (ready != cudaSuccess) return ready;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(E.nprob * kWideBlocks), 1, 1);
  cfg.blockDim = dim3((unsigned)kWideThreads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)kWideBlocks;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.numAttrs = 1;
  // programmatic at any size (unless off): the blocks fetch their nodes' bands while they wait (10 problems of L = 8 4028 us
  // by the rule, 3969 so; 14 of L = 6..9 5849, 5772)
  if (pdl_launch(E.pdl ? 1 : 0, (int)cfg.gridDim.x)) {
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
  }
  cfg.attrs = attr;
  return cudaLaunchKernelEx(&cfg, kern, E, T, want, loop);
}

}  // namespace hn
