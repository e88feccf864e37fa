// Vector steps on each problem's finest level, in FP64: ||b|| and the boundary check at the start of a
// solve, the outer defect and the update of the defect correction, and the steps of conjugate gradients
// with the V cycle as preconditioner (a solver plugged into another, Sec. 4.1).
//
// The 128-node tiles of a problem solved alone go to the warps in turn; those of several problems are shared in
// runs among the problems in the phase.  The stencil steps are bound by the FP64 pipe (the outer defect: 11
// operations per node, of 0.53 T a second), the others by it and by memory alike.
//
// A norm is summed in the order of problem_norm_sum.  Up to kSumGroup tiles the block that finishes a problem
// adds its tiles' sums.  More of them (131,080 at L = 12) would keep one SM's FP64 pipe busy for 40 us: there
// 32 consecutive tiles, a link, are one lane each of one of the sum's 32 independent warp-wide chains; the warp
// that finishes a chain adds it, the one that finishes a kSumGroup adds its 32 chains, and the one that
// finishes the problem adds those in order.  A block's warps share a link and sum their four tiles over the
// lanes together, 6 additions in place of 20 (eight tiles a warp leave one SM in five a third of the work more at
// L = 11).  The launch's last block takes all control steps, so that no control launch follows, whatever the
// number of problems, and no phase changes while blocks look for work.
//
// Against work lists of tiles and a control launch after each step: a solve in FP32 739 -> 715 us at L = 7,
// 1453 -> 1394 at L = 10, 2853 -> 2810 at L = 11, 7006 -> 6890 at L = 12; PCG at L = 11 4095 -> 4033 us; 256 problems
// of L = 3..9 in a batch 18.57 -> 18.22 ms.  Three blocks an SM for the stencil steps: four (64 registers)
// measured 1414 us at L = 10, two 7000 us at L = 12.
#include <algorithm>

#define HN_SOURCE 2
#include "k_device.cuh"

namespace hn {

namespace {

constexpr int kFineThreads = 256, kFineWarps = kFineThreads / 32;
constexpr int kLink = 32;                 // tiles of a link

enum FineOp { F_NORM_B = 0, F_OUTER, F_UPDATE, F_PCG_Q, F_PCG_X, F_PCG_DOT, F_PCG_P };

__device__ __forceinline__ bool fine_serves(int op, const ProbState& st, bool pcg) {
  switch (op) {
    case F_NORM_B: return st.phase == PH_INIT;
    case F_OUTER: return st.phase == PH_OUTER && !(pcg && st.cycles > 0);
    case F_PCG_Q:
    case F_PCG_X: return st.phase == PH_OUTER && st.cycles > 0;
    case F_PCG_DOT: return st.phase == PH_PRECOND;
    default: return st.phase == PH_UPDATE;
  }
}
__host__ __device__ constexpr int fine_control(int op) {
  return op == F_NORM_B ? CTRL_INIT : op == F_PCG_Q ? CTRL_PCG_ALPHA : op == F_PCG_DOT ? CTRL_PCG_BETA
       : op == F_UPDATE || op == F_PCG_P ? CTRL_POST : CTRL_OUTER;
}

__host__ __device__ constexpr bool fine_sums(int op) { return op != F_UPDATE && op != F_PCG_P; }

// A lane's term of ||b||^2 and of the outer defect's norm: one chain for both (x = 0 has ||r|| = ||b|| to the bit)
__device__ __forceinline__ double lane_norm(const double (&a)[4]) {
  return fma(a[3], a[3], fma(a[2], a[2], fma(a[0], a[0], a[1] * a[1])));
}

// One tile of a problem's finest level; returns the lane's term of the problem's sum.  V: the cycle's vector type.
template <int OP, class V>
__device__ __forceinline__ double fine_tile(const ProblemDev& P, ProbState& st, bool pcg, long long i0, int lane) {
  const LevelDev& top = P.lev[P.L];
  double q = 0.0;
  if constexpr (OP == F_NORM_B) {
    double b[4];
    ld4<LD_NC>(P.b64 + i0, b);
    const int n = top.n;
    bool bad = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = (int)i0 + j;
      if (b[j] != 0.0 && i < n * n) {             // a right-hand side has to be zero on the Dirichlet nodes
        int x, y;
        node_xy(i, P.L, x, y);
        bad = bad || is_dirichlet(x, y, n, top.bc);
      }
    }
    if (bad) atomicExch(&st.status, (int)HN_ERR_ARG);
    q = lane_norm(b);
  } else if constexpr (OP == F_OUTER) {
    // d = b - A x (x = 0: d = b), as V(d s) the inner right-hand side; CG: the initial residual, kept in FP64
    double b[4], r[4];
    ld4<LD_EF>(P.b64 + i0, b);
#pragma unroll
    for (int j = 0; j < 4; ++j) r[j] = b[j];
    if (!st.x_zero) {
      double w[3][8], dg[4];
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy) load_row<double, LD_NC>(P.x64, i0 + dy * (1LL << P.L), lane, w[dy + 1]);
      // r = b - A x as one chain from b
      stencil_windows<F64, LD_EF, true>(reinterpret_cast<const void* const*>(P.band64), nullptr, w, i0, r, dg);
    }
    const double s = st.s;
    V out[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) out[j] = from_f64<V>(r[j] * s);
    q = lane_norm(r);
    st4(static_cast<V*>(top.rhs) + i0, out);
    if (pcg) st4(P.r64 + i0, r);
  } else if constexpr (OP == F_UPDATE) {
    // x += c / s (c = the inner iterate, buffer 0)
    float c[4];
    double x[4];
    ld4<LD_NC>(static_cast<const float*>(top.x[0]) + i0, c);
    ld4c(P.x64 + i0, x);
    const double inv_s = st.inv_s;
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = fma(to_f64(c[j]), inv_s, x[j]);
    st4(P.x64 + i0, x);
  } else if constexpr (OP == F_PCG_Q) {
    // q = A p (p with zero halos) and (p, q)
    double w[3][8], acc[4], dg[4];
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) load_row<double, LD_NC>(P.p64, i0 + dy * (1LL << P.L), lane, w[dy + 1]);
    stencil_windows<F64, LD_NC>(reinterpret_cast<const void* const*>(P.band64), nullptr, w, i0, acc, dg);
    st4(P.q64 + i0, acc);
#pragma unroll
    for (int j = 0; j < 4; ++j) q = fma(w[1][j + 2], acc[j], q);
  } else if constexpr (OP == F_PCG_X) {
    // x += alpha p, r -= alpha q, ||r||^2; the next cycle's right-hand side V(s r)
    double x[4], r[4], pv[4], qv[4];
    ld4c(P.x64 + i0, x);
    ld4c(P.r64 + i0, r);
    ld4<LD_NC>(P.p64 + i0, pv);
    ld4<LD_NC>(P.q64 + i0, qv);
    const double alpha = st.alpha, s = st.s;
    V out[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[j] = fma(alpha, pv[j], x[j]);
      r[j] = fma(-alpha, qv[j], r[j]);
      q = fma(r[j], r[j], q);
      out[j] = from_f64<V>(r[j] * s);
    }
    st4(P.x64 + i0, x);
    st4(P.r64 + i0, r);
    st4(static_cast<V*>(top.rhs) + i0, out);
  } else if constexpr (OP == F_PCG_DOT) {
    // (r, c), c = the cycle's result (buffer 0; z = c / s)
    double r[4];
    V c[4];
    ld4<LD_NC>(P.r64 + i0, r);
    ld4<LD_NC>(static_cast<const V*>(top.x[0]) + i0, c);
#pragma unroll
    for (int j = 0; j < 4; ++j) q = fma(r[j], to_f64(c[j]), q);
  } else {
    // p = c / s + beta p (the new search direction)
    V c[4];
    double pv[4];
    ld4<LD_NC>(static_cast<const V*>(top.x[0]) + i0, c);
    ld4c(P.p64 + i0, pv);
    const double beta = st.beta, inv_s = st.inv_s;
#pragma unroll
    for (int j = 0; j < 4; ++j) pv[j] = fma(beta, pv[j], to_f64(c[j]) * inv_s);
    st4(P.p64 + i0, pv);
  }
  return q;
}

// The lanes' terms of N = 4 or 8 tiles summed over the warp, each in warp_sum's order (a step of that butterfly
// gives both halves of the lanes the same sum, so a step sums two tiles at once, half of the lanes keeping one,
// half the other).  Lane l ends with tile sum_tile<N>(l).  term(k): the lane's term of tile k.
template <int N>
__device__ __forceinline__ int sum_tile(int lane) {
  const int hi = ((lane >> 4) & 1) << 1 | ((lane >> 3) & 1);
  return N == 8 ? hi << 1 | ((lane >> 2) & 1) : hi;
}
__device__ __forceinline__ double sum_step2(double a, double b, int o) {      // a: kept by the lower half
  const bool up = threadIdx.x & o;
  const double keep = up ? b : a, give = up ? a : b;
  return keep + __shfl_xor_sync(kFull, give, o);
}
template <int N, class F>
__device__ __forceinline__ double sum_tiles(F&& term) {
  auto two = [&](int k) { const double a = term(k); return sum_step2(a, term(k + N / 2), 16); };
  auto four = [&](int k) { const double a = two(k); return sum_step2(a, two(k + N / 4), 8); };
  double v = four(0);
  if constexpr (N == 8) v = sum_step2(v, four(1), 4);
  else v += __shfl_xor_sync(kFull, v, 4);
  v += __shfl_xor_sync(kFull, v, 2);
  return v + __shfl_xor_sync(kFull, v, 1);
}

// true in the warp / block that makes the last of `all` counts on a ticket, which it resets (what the warp /
// block wrote before is visible to it)
__device__ __forceinline__ bool warp_counted(unsigned* ticket, unsigned all) {
  int last = 0;
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    __threadfence();
    last = atomicAdd(ticket, 1u) == all - 1u;
    if (last) *ticket = 0u;
  }
  last = __shfl_sync(kFull, last, 0);
  if (last) __threadfence();
  return last;
}
__device__ __forceinline__ bool block_counted(unsigned* ticket, unsigned count, unsigned all, int* s_last) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    *s_last = atomicAdd(ticket, count) == all - count;
    if (*s_last) *ticket = 0u;
  }
  __syncthreads();
  const bool last = *s_last;
  if (last) __threadfence();
  return last;
}

// A warp has the sums of its four tiles of link g of a problem of more than kSumGroup tiles in part: add
// whatever that finishes; the problem's norm sum goes to gsum[0].
__device__ void sum_link(const EngineDev& E, int p, double* part, int tiles, int g) {
  const int lane = threadIdx.x & 31;
  const int j = g * kLink / kSumGroup, lo = j * kSumGroup, hi = min(tiles, lo + kSumGroup);
  const int links = (hi - lo + kLink - 1) / kLink, mine = g - lo / kLink, chain = mine & 31;   // of this kSumGroup
  unsigned* ticket = E.gticket + (long long)p * ticket_words(E.ctl_groups);
  // the chain: tiles lo + 1024 i + 32 chain + lane, its sum in the place of its first
  const int counts = kFineWarps * ((links - chain + 31) / 32);
  if (!warp_counted(ticket + 2 + E.ctl_groups + j * 32 + chain, (unsigned)counts)) return;
  {
    const int first = lo + kLink * chain + lane;
    double c = 0.0, w[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) w[k] = first + k * 1024 < hi ? __ldcg(part + first + k * 1024) : 0.0;
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (first + k * 1024 < hi) c += w[k];
    if (first < hi) part[first] = c;
    __threadfence();
  }
  if (!warp_counted(ticket + 2 + j, (unsigned)min(32, links))) return;
  // the kSumGroup: problem_partial_sum's eight warps, each thread's four chains first
  double s = sum_tiles<8>([&](int k) {
    double c[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int q = lo + m * 256 + k * 32 + lane;
      c[m] = q < hi ? __ldcg(part + q) : 0.0;
    }
    return (c[0] + c[1]) + (c[2] + c[3]);
  });
  // lane l has warp sum_tile<8>(l); block_sum256's steps over the eight (lane w: warp w)
  s = __shfl_sync(kFull, s, ((lane >> 2) & 1) << 4 | ((lane >> 1) & 1) << 3 | (lane & 1) << 2);
  s += __shfl_xor_sync(kFull, s, 4);
  s += __shfl_xor_sync(kFull, s, 2);
  s += __shfl_xor_sync(kFull, s, 1);
  double* gsum = E.gsum + (long long)p * E.ctl_groups;
  const int all = sum_groups(tiles);
  if (lane == 0) gsum[j] = s;
  if (!warp_counted(ticket + 1, (unsigned)all)) return;
  double t = 0.0;
  for (int b = 0; b < all; b += 32) {
    const double v = b + lane < all ? __ldcg(gsum + b + lane) : 0.0;
    for (int k = 0; k < 32 && b + k < all; ++k) t += __shfl_sync(kFull, v, k);
  }
  if (lane == 0) gsum[0] = t;
}

// Tiles a, a + step, .. < b of problem p, their sums to its partial slots
template <int OP, class V>
__device__ __forceinline__ void fine_run(const EngineDev& E, int p, int a, int b, int step, bool pcg) {
  const int lane = threadIdx.x & 31;
  ProbState& st = E.S[p];
  const ProblemDev& P = E.P[p];
  double* part = E.partial + E.fine_off[p];
  for (int t = a; t < b; t += step) {
    double q = fine_tile<OP, V>(P, st, pcg, (long long)t * kTile + lane * kLaneNodes, lane);
    if constexpr (fine_sums(OP)) {
      q = warp_sum(q);
      if (lane == 0) part[t] = q;
    }
  }
}
// Links a, a + step, .. < b of a problem of more than kSumGroup tiles, the block's warps sharing each
template <int OP, class V>
__device__ __forceinline__ void fine_links(const EngineDev& E, int p, int a, int b, int step, bool pcg) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  ProbState& st = E.S[p];
  const ProblemDev& P = E.P[p];
  const int tiles = fine_tiles(P.L);
  double* part = E.partial + E.fine_off[p];
  for (int g = a; g < b; g += step) {
    const double v = sum_tiles<kLink / kFineWarps>([&](int k) {
      const int t = g * kLink + w + kFineWarps * k;
      return t < tiles ? fine_tile<OP, V>(P, st, pcg, (long long)t * kTile + lane * kLaneNodes, lane) : 0.0;
    });
    const int t = g * kLink + w + kFineWarps * sum_tile<kLink / kFineWarps>(lane);
    if ((lane & 7) == 0 && t < tiles) part[t] = v;
    sum_link(E, p, part, tiles, g);
  }
}

// summary: 1: the last block (of an engine of one problem with nothing to do: block 0) also ends the iteration
// (2: only counts it: the start of a solve).
enum FineForm { SOLO_TILES, SOLO_LINKS, GROUPS };   // (links: where the sum has more than kSumGroup tiles)
template <int OP, class V, int FORM>
__global__ void __launch_bounds__(kFineThreads, OP == F_OUTER || OP == F_PCG_Q ? 3 : 4)
    k_fine(EngineDev E, int solo_tiles, int summary, cudaGraphConditionalHandle h, int use_handle) {
  pdl_start();
  __shared__ double sh[32];
  __shared__ int s_last;
  const bool pcg = E.prm.solver == SOLVER_PCG;
  const int warp = threadIdx.x >> 5, G = (int)gridDim.x, blk = (int)blockIdx.x;
  if constexpr (FORM != GROUPS) {
    if (!fine_serves(OP, E.S[0], pcg)) {
      if (summary && blk == 0) summary_apply(E, h, use_handle, summary == 1, sh);
      return;
    }
    constexpr bool large = FORM == SOLO_LINKS;
    if constexpr (large) fine_links<OP, V>(E, 0, blk, (solo_tiles + kLink - 1) / kLink, G, pcg);
    else fine_run<OP, V>(E, 0, blk * kFineWarps + warp, solo_tiles, G * kFineWarps, pcg);
    if (!block_counted(E.ticket, 1u, (unsigned)G, &s_last)) return;
    double sum = 0.0;
    if (large) sum = __ldcg(E.gsum);
    else if (fine_sums(OP)) sum = problem_partial_sum(E.partial, solo_tiles, sh);
    if (threadIdx.x == 0) control_apply(E, E.S[0], fine_control(OP), sum);
    __syncthreads();
    if (summary) summary_apply(E, h, use_handle, summary == 1, sh);
  } else {
    __shared__ Served q;
    for (int base = 0; base < E.nprob; base += kListMax) {
      const int n = list_served(E, q, base, 0, [&](const ProbState& S, int L) {
        return L >= HN_MIN_LEVEL && fine_serves(OP, S, pcg);
      });
      if (n == 0) continue;
      const long long all = number_items(q, n, [](int l) { return fine_tiles(l); });
      const int lo = (int)(blk * all / G), hi = (int)((blk + 1) * all / G);     // the block's run of tiles
      for (int m = hi > lo ? served_of(q, n, lo) : n; m < n && q.start[m] < hi; ++m) {
        const int p = q.slot[m], tiles = fine_tiles(q.level[m]);
        if (!dbg_item(E, p, 0, -1, HN_HERE)) continue;
        const int a = max(0, lo - q.start[m]), b = min(tiles, hi - q.start[m]);
        if (fine_sums(OP) && tiles > kSumGroup) {   // (a link belongs to the block that has its first tile)
          fine_links<OP, V>(E, p, (a + kLink - 1) / kLink, (b + kLink - 1) / kLink, 1, pcg);
          continue;
        }
        fine_run<OP, V>(E, p, a + warp, b, kFineWarps, pcg);
        unsigned* ticket = E.gticket + (long long)p * ticket_words(E.ctl_groups) + 1;
        if (fine_sums(OP) && block_counted(ticket, (unsigned)(b - a), (unsigned)tiles, &s_last)) {
          const double sum = problem_partial_sum(E.partial + E.fine_off[p], tiles, sh);
          if (threadIdx.x == 0) E.gsum[(long long)p * E.ctl_groups] = sum;
        }
      }
      __syncthreads();
    }
    if (!block_counted(E.ticket, 1u, (unsigned)G, &s_last)) return;
    for (int p = threadIdx.x; p < E.nprob; p += kFineThreads) {
      ProbState& st = E.S[p];
      if (E.P[p].L >= HN_MIN_LEVEL && fine_serves(OP, st, pcg))
        control_apply(E, st, fine_control(OP), fine_sums(OP) ? __ldcg(E.gsum + (long long)p * E.ctl_groups) : 0.0);
    }
    __syncthreads();
    if (summary) summary_apply(E, h, use_handle, summary == 1, sh);
  }
}

template <int OP, class V, int FORM>
cudaError_t launch_fine_f(const EngineDev& E, const GroupSize& size, int solo_tiles, int summary, cudaGraphConditionalHandle h,
                          int use_handle, cudaStream_t s) {
  auto kern = k_fine<OP, V, FORM>;
  static const int per_sm = [&] {
    int b = 0;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, kFineThreads, 0) == cudaSuccess && b > 0 ? b : 1;
  }();
  cudaLaunchConfig_t cfg = {};
  // no more than one wave of blocks, nor than have work: a tile for each warp; a link for all warps, which share it.  The steps
  // of CG on several problems take a block for each tile: few problems leave SMs idle, and eight stencils on one
  // SM wait for its FP64 pipe (2 problems of L = 5 551 -> 489 us, of L = 5..7 823 -> 756; a whole wave 523, 773; as programmatic
  // launches, where the rule would have them so, 487, 774).  The defect correction's two steps a solve gain more
  // from a grid below that rule's line (4 problems of L = 5..7 1317 against 1352 us, a whole wave 1360).
  const bool by_tile = FORM == GROUPS && E.prm.solver == SOLVER_PCG;
  const long long tiles = FORM == GROUPS ? size.sum([](int l) { return fine_tiles(l); }) : solo_tiles;
  const int share = FORM == SOLO_LINKS ? kLink : by_tile ? 1 : kFineWarps;
  cfg.gridDim = dim3((unsigned)std::max<long long>(1, std::min<long long>(per_sm * sm_count(), (tiles + share - 1) / share)), 1, 1);
  cfg.blockDim = dim3((unsigned)kFineThreads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  if (!by_tile && pdl_launch(E.pdl, (int)cfg.gridDim.x)) {
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  return cudaLaunchKernelEx(&cfg, kern, E, solo_tiles, summary, h, use_handle);
}
template <int OP, class V>
cudaError_t launch_fine_t(const EngineDev& E, const GroupSize& size, int solo_tiles, int summary, cudaGraphConditionalHandle h,
                          int use_handle, cudaStream_t s) {
  if (!solo_tiles) return launch_fine_f<OP, V, GROUPS>(E, size, solo_tiles, summary, h, use_handle, s);
  if constexpr (fine_sums(OP))
    if (solo_tiles > kSumGroup) return launch_fine_f<OP, V, SOLO_LINKS>(E, size, solo_tiles, summary, h, use_handle, s);
  return launch_fine_f<OP, V, SOLO_TILES>(E, size, solo_tiles, summary, h, use_handle, s);
}
template <int OP>
cudaError_t launch_fine_p(const EngineDev& E, const GroupSize& size, int solo_tiles, int summary, cudaGraphConditionalHandle h,
                          int use_handle, cudaStream_t s) {
  return E.prm.prec == P64 ? launch_fine_t<OP, double>(E, size, solo_tiles, summary, h, use_handle, s)
                           : launch_fine_t<OP, float>(E, size, solo_tiles, summary, h, use_handle, s);
}

// A smoothing step or the defect of an FP64 level of a problem solved alone (k_band's step, same bits).  Bound by the
// FP64 pipe (10 operations a node, 20 us at L = 10) once the vectors come from L2: there the level and those below
// it (157 MB) are more than L2 holds, so from level 10 on the bands are marked to be evicted first and the
// vectors, which every step reads or writes, stay (solve at L = 10 2421 -> 2257 us, with all bands kept 2325 us;
// L = 11 6180 -> 5993).  Level 9 below them the same way, against fused sweeps of recomputed halos, which cost the
// FP64 pipe more than the launches saved: L = 10 2257 -> 2202 us, L = 11 5993 -> 5907; level 8 too is slower
// (2430 against 2350 us, bands kept).  Two, three, four blocks an SM: 2518 / 2432 / 2475 us (bands kept).
enum { LV_FIRST = 0, LV_SMOOTH, LV_DEFECT };
template <int OP, int LKB>
__global__ void __launch_bounds__(kFineThreads, 3)
    k_level64(EngineDev E, TileList tl, int level, int want, int in_sel, int fuse) {
  pdl_start();
  if (tl.solo_d.n == 0) return;
  const ProbState& st = E.S[0];
  if (st.phase != want) return;
  if (!dbg_level(E, tl.solo_d, level, tl.solo_tiles, HN_HERE)) return;
  const LevelDev& d = tl.solo_d;
  const bool zero = OP == LV_FIRST && (tl.solo_L > level || st.zero_top);
  const bool summed = OP == LV_FIRST && tl.solo_L == level && !zero;
  const int lane = threadIdx.x & 31, src = OP == LV_FIRST ? 0 : in_sel;
  const double* x = static_cast<const double*>(d.x[src]);
  double* out = static_cast<double*>(OP == LV_DEFECT ? d.r : d.x[1 - src]);
  const int step = (int)gridDim.x * kFineWarps;
  for (int t = (int)blockIdx.x * kFineWarps + (int)(threadIdx.x >> 5); t < tl.solo_tiles; t += step) {
    const long long i0 = (long long)t * kTile + lane * kLaneNodes;
    double r[4], v[4];
    ld4<LD_NC>(static_cast<const double*>(d.rhs) + i0, r);
    if (zero) {
      double wd[4];
      ld4<LKB>(d.wdinv + i0, wd);
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = wd[j] * r[j];
    } else {
      double w[3][8], dg[4];
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy) load_row<double, LD_NC>(x, i0 + dy * (1LL << level), lane, w[dy + 1]);
      stencil_windows<F64, LKB, true>(d.band, nullptr, w, i0, r, dg);
      if constexpr (OP == LV_DEFECT) {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = r[j];
      } else {
        double wd[4];
        ld4<LKB>(d.wdinv + i0, wd);
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = fma(wd[j], r[j], w[1][j + 2]);
      }
    }
    st4(out + i0, v);
    if (summed) {
      const double q = tile_sumsq(r);
      if (lane == 0) E.partial[t] = q;
    }
  }
  if (OP == LV_FIRST && fuse) solo_fused_check(E, level, summed, want);
}

template <int OP, int LKB>
cudaError_t launch_level64_t(const EngineDev& E, const TileList& tl, int level, int want, int in_sel, int fuse,
                             cudaStream_t s) {
  auto kern = k_level64<OP, LKB>;
  static const int per_sm = [&] {
    int b = 0;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, kFineThreads, 0) == cudaSuccess && b > 0 ? b : 1;
  }();
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::max(1, std::min(per_sm * sm_count(), (tl.solo_tiles + kFineWarps - 1) / kFineWarps)), 1, 1);
  cfg.blockDim = dim3((unsigned)kFineThreads, 1, 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  if (pdl_launch(E.pdl, (int)cfg.gridDim.x)) {
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  return cudaLaunchKernelEx(&cfg, kern, E, tl, level, want, in_sel, fuse);
}

}  // namespace

cudaError_t launch_level64(const EngineDev& E, const TileList& tl, int kind, int level, int want, int in_sel, int fuse,
                           cudaStream_t s) {
  const bool stream = level >= 10;
  if (kind == LV_FIRST) return stream ? launch_level64_t<LV_FIRST, LD_EF>(E, tl, level, want, in_sel, fuse, s)
                                      : launch_level64_t<LV_FIRST, LD_NC>(E, tl, level, want, in_sel, fuse, s);
  if (kind == LV_SMOOTH) return stream ? launch_level64_t<LV_SMOOTH, LD_EF>(E, tl, level, want, in_sel, fuse, s)
                                       : launch_level64_t<LV_SMOOTH, LD_NC>(E, tl, level, want, in_sel, fuse, s);
  return stream ? launch_level64_t<LV_DEFECT, LD_EF>(E, tl, level, want, in_sel, fuse, s)
                : launch_level64_t<LV_DEFECT, LD_NC>(E, tl, level, want, in_sel, fuse, s);
}

cudaError_t launch_fine(const EngineDev& E, const GroupSize& size, int kind, int solo_tiles, int summary, cudaGraphConditionalHandle h,
                        int use_handle, cudaStream_t s) {
  switch (kind) {
    case FINE_NORM_B: return launch_fine_t<F_NORM_B, float>(E, size, solo_tiles, summary, h, use_handle, s);
    case FINE_OUTER: return launch_fine_p<F_OUTER>(E, size, solo_tiles, summary, h, use_handle, s);
    case FINE_UPDATE: return launch_fine_t<F_UPDATE, float>(E, size, solo_tiles, summary, h, use_handle, s);
    case FINE_PCG_Q: return launch_fine_t<F_PCG_Q, float>(E, size, solo_tiles, summary, h, use_handle, s);
    case FINE_PCG_X: return launch_fine_p<F_PCG_X>(E, size, solo_tiles, summary, h, use_handle, s);
    case FINE_PCG_DOT: return launch_fine_p<F_PCG_DOT>(E, size, solo_tiles, summary, h, use_handle, s);
    case FINE_PCG_P: return launch_fine_p<F_PCG_P>(E, size, solo_tiles, summary, h, use_handle, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace hn
