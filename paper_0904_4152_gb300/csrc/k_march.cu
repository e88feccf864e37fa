// Marching sweeps: the down part of a level (both pre-smoothing steps, the squares of the lagged
// residual check, the defect and the restriction) and its up part (prolongation and both
// post-smoothing steps) as one pass over the level's memory each, for FP32 and FP16-band hierarchies
// with V(2,2) cycles.
//
// What bounds it.  One launch per step reads the nine bands five times a cycle (254 B per node in FP32,
// 164 with FP16 bands); the two passes here move 37 + 36 B (27 + 26).  Measured at L = 12 (16.8 M nodes,
// FP32): down 390 -> 107 us (5.8 TB/s), up 275 -> 115 us, of 93 us at the HBM rate; FP16 bands 280 -> 111
// and 195 -> 117 us of 68 us.  What is left is instruction latency: 230 registers allow two warps per
// scheduler (three, at 168, would spill), and an iteration is a chain of three stencils.
//
// Layout.  Node (x, y) has flat index y n + x = y W + (x + y) with W = 2^L, n = W + 1: seen as a matrix
// of row length W, the flat array has every row 16-byte aligned, and the stencil neighbour (dy, dx) of
// row r, column c is row r + dy, column c + dy + dx (beyond column W the flat array simply goes on in
// the next row).  A warp takes a strip of up to 128 columns, 8 of them on either side recomputed, and
// marches over a chunk of rows; lane l owns columns 4 l .. 4 l + 3 of the strip.  In iteration i it
// forms the first step on row i, the second on row i - 1, the defect on row i - 2 and the restriction
// around row i - 3: a row's bands stay in registers from the first use to the last, neighbouring
// columns come by shuffles, so a warp waits for no other.  The rows arrive by asynchronous copies into
// a ring of shared-memory slots (each lane reads what it copied itself).  Three more rows at either end
// of a chunk are recomputed; the arrays' zero halos (halo_of) cover every row and column read beyond
// the grid, where all values come out as zero.
//
// The operator is symmetric, bit for bit (a pair's two entries are formed from the same cells in the
// same order, and the FP16 scales of opposite bands are the maxima of the same values), so only the
// diagonal (FP16: the row sum) and the bands towards greater indices are read; the others are theirs
// at the neighbour.
//
// Every value is formed by the operations of the per-step kernels in their order, so the results have
// the same bits.
#include <algorithm>

#define HN_SOURCE 1
#include "k_device.cuh"

namespace hn {

namespace {

constexpr int kWarps = 2;                // independent warps of a block
constexpr int kSlots = 4;                // rows of the ring: one in use, three on their way
enum { DOWN_ZERO = 0, DOWN = 1, UP = 2 };

// a slot: five bands, omega / D, right-hand side, iterate, each 128 columns
template <class Pol> constexpr int band_bytes() { return kTile * (int)sizeof(typename Pol::B); }
template <class Pol> constexpr int slot_bytes() { return 5 * band_bytes<Pol>() + 3 * kTile * 4; }

// a row at the lane's columns: bands 4..8 (band[k - 4]; FP16: scaled, the first the row sum) and what
// the left neighbour holds of them: band 5 one column to the left, band 7 one, band 8 two
struct Bands {
  float v[5][4];
  float l5, l7, l8[2];
};
// a vector's two rows before the one that arrives: own columns, and the neighbour's column that the
// next product will need again (row -1: one to the left, row 0: one to the right)
struct Field {
  float m[4], c[4], ml, cr;
};

__device__ __forceinline__ void copy16(unsigned dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy8(unsigned dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N> __device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

__device__ __forceinline__ void lds4(const unsigned char* p, float (&o)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
}
// acc = (A x) at the lane's columns of the field's row 0, given its next row p, which then moves in: B the
// row's bands, S the bands of the row before it; in the band order of stencil_windows (FP16: of
// stencil_windows_rowsum).  Columns beyond the lane's own come from its neighbours (the strip's outermost
// columns get values that are never used).
template <class Pol>
__device__ __forceinline__ void apply_row(const Bands& B, const Bands& S, Field& F, const float (&p)[4], float (&acc)[4]) {
  const float pr0 = __shfl_down_sync(kFull, p[0], 1), pr1 = __shfl_down_sync(kFull, p[1], 1);
  const float cl = __shfl_up_sync(kFull, F.c[3], 1), mll = __shfl_up_sync(kFull, F.m[2], 1);
  const float wm[6] = {mll, F.ml, F.m[0], F.m[1], F.m[2], F.m[3]};     // columns -2 .. 3
  const float wc[6] = {cl, F.c[0], F.c[1], F.c[2], F.c[3], F.cr};      // columns -1 .. 4
  const float wp[6] = {p[0], p[1], p[2], p[3], pr0, pr1};              // columns 0 .. 5
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float band[9] = {j < 2 ? S.l8[j] : S.v[4][j - 2], j < 1 ? S.l7 : S.v[3][j - 1], S.v[2][j],
                           j < 1 ? B.l5 : B.v[1][j - 1], B.v[0][j], B.v[1][j], B.v[2][j], B.v[3][j], B.v[4][j]};
    const float xc = wc[j + 1];
    float a = Pol::prec == P16 ? band[4] * xc : 0.0f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const int o = j + k % 3;
      const float x = k < 3 ? wm[o] : (k < 6 ? wc[o] : wp[o]);
      if constexpr (Pol::prec == P16) {
        if (k != 4) a = fmaf(band[k], x - xc, a);
      } else {
        a = fmaf(band[k], x, a);
      }
    }
    acc[j] = a;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) { F.m[j] = F.c[j]; F.c[j] = p[j]; }
  F.ml = cl;
  F.cr = pr0;
}

__device__ __forceinline__ void band_edges(Bands& B) {
  B.l5 = __shfl_up_sync(kFull, B.v[1][3], 1);
  B.l7 = __shfl_up_sync(kFull, B.v[3][3], 1);
  B.l8[0] = __shfl_up_sync(kFull, B.v[4][2], 1);
  B.l8[1] = __shfl_up_sync(kFull, B.v[4][3], 1);
}
__device__ __forceinline__ void scale_halves(uint2 u, float s, float (&o)[4]) {
  const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
  const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
  o[0] = __fmul_rn(s, f0.x); o[1] = __fmul_rn(s, f0.y);
  o[2] = __fmul_rn(s, f1.x); o[3] = __fmul_rn(s, f1.y);
}
// a row's bands from its slot
template <class Pol>
__device__ __forceinline__ void load_bands(Bands& B, const unsigned char* slot, int lane, const float* scale) {
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const unsigned char* p = slot + k * band_bytes<Pol>();
    if constexpr (Pol::prec == P16) scale_halves(*reinterpret_cast<const uint2*>(p + lane * 8), scale[k], B.v[k]);
    else lds4(p + lane * 16, B.v[k]);
  }
  band_edges(B);
}

// What a warp works on: rows r0..r1-1 of the strip whose first own column is c0
struct Item {
  int c0, r0, r1;
};
// A level as the warps read it.  The strip's columns start `side` to the left of its own ones.
struct View {
  const unsigned char* band;             // band 4; bands 5..8 follow at `stride` bytes
  long long stride;
  const float *wd, *b, *x;               // omega / D, right-hand side, the iterate that is read
  float* out;                            // the iterate that is written
  float* coarse;                         // down: the coarse right-hand side, up: the coarse iterate (read)
  float* squares;                        // down: one pair per lane's four nodes (the lagged check), or null
  const float* scale;
  int L, n, pitch, bc;
};

// The copies of a lane, row by row into the ring's slots: the sources of the row that comes next
template <class Pol>
struct Cursor {
  static constexpr int BB = band_bytes<Pol>(), es = (int)sizeof(typename Pol::B);
  const unsigned char* band;
  const float *wd, *b, *x;
  // f, g: flat indices of the lane's first column in the first row, for the iterate in the row it is read from
  __device__ __forceinline__ void start(const View& v, int f, int g) {
    band = v.band + (long long)f * es;
    wd = v.wd + f;
    b = v.b + f;
    x = v.x + g;
  }
  __device__ __forceinline__ void next(int W) {
    band += (long long)W * es;
    wd += W;
    b += W;
    x += W;
  }
  __device__ __forceinline__ void constants(long long stride, unsigned slot, int lane) const {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      if constexpr (es == 4) copy16(slot + k * BB + lane * 16, band + k * stride);
      else copy8(slot + k * BB + lane * 8, band + k * stride);
    }
    copy16(slot + 5 * BB + lane * 16, wd);
  }
  __device__ __forceinline__ void vectors(unsigned slot, int lane, bool iterate) const {
    copy16(slot + 5 * BB + kTile * 4 + lane * 16, b);
    if (iterate) copy16(slot + 5 * BB + 2 * kTile * 4 + lane * 16, x);
  }
};

// a row's bands towards the row after it straight from memory (flat index f)
template <class Pol>
__device__ __forceinline__ void load_bands_ahead(Bands& B, const View& v, int f, bool live) {   // (f: a multiple of 4)
#pragma unroll
  for (int k = 2; k < 5; ++k) {
    if (!live) continue;
    if constexpr (Pol::prec == P16)
      scale_halves(__ldg(reinterpret_cast<const uint2*>(v.band + k * v.stride) + f / 4), v.scale[k], B.v[k]);
    else ld4<LD_NC>(reinterpret_cast<const float*>(v.band + k * v.stride) + f, B.v[k]);
  }
  band_edges(B);
}

// Full weighting onto the coarse nodes at the lane's columns 0 and 2 (those whose fine coordinates are
// even), as the defect's rows arrive: a row adds the last three terms of the nodes on the row before
// it, the middle three of the nodes on itself and the first three of the nodes on the next row, in
// restrict_value's order.  restrict_row(d: the defect on row r, x, y: the grid coordinates of the lane's
// first column there, store: row r - 1 is the warp's).
//
// Dirichlet sides only: the nodes that count lie inside the grid, where the rows of a column are
// alternately coarse rows (both coordinates even) and rows between two of them (both odd): one sum per
// column.  (zero_sides sets the others.)
struct RestrictInner {
  float s[2];
  __device__ __forceinline__ void row(const View& v, const float (&d)[4], int x, int y, int, bool store) {
    const float l1 = __shfl_up_sync(kFull, d[3], 1), l2 = __shfl_up_sync(kFull, d[2], 1);
    const float r1 = __shfl_down_sync(kFull, d[0], 1);
    const float w[7] = {l2, l1, d[0], d[1], d[2], d[3], r1};           // columns -2 .. 4
    const int n1 = v.n - 1;
    const float q = 0.25f, h = 0.5f;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float* c = w + 2 + 2 * e;
      if (e == 1) {
        x += 2;
        if (x > n1) { x -= n1 + 1; ++y; }
      }
      if (y & 1) {
        float u = fmaf(q, c[0], s[e]);
        u = fmaf(h, c[1], u);
        u = fmaf(q, c[2], u);
        // the node on row r - 1 is (x + 1, y - 1)
        if (store && x + 1 < n1 && y > 1 && y < n1) v.coarse[(y >> 1) * ((n1 >> 1) + 1) + ((x + 1) >> 1)] = u;
        s[e] = fmaf(q, c[0], fmaf(h, c[-1], q * c[-2]));
      } else {
        s[e] = fmaf(h, c[1], fmaf(h, c[-1], s[e]) + c[0]);
      }
    }
  }
};
// The coarse right-hand side on the sides, all Dirichlet: 0 in every cycle, whatever a caller has put there (hn_mg_apply
// takes any vector).  Coarse rows r0 / 2 .. r1 / 2 by the warp that has rows r0 .. r1 - 1 (of R) of the first strip.  (As stores
// of the restriction itself, a branch more in each row: L = 10 solve 1342 -> 1362 us, FP16 L = 12 8333 -> 8578.)
__device__ __forceinline__ void zero_sides(float* coarse, int n, int r0, int r1, int R, int lane) {
  const int nc = (n >> 1) + 1;
  for (int J = (r0 + 1) / 2 + lane; J < min((r1 + 1) / 2, nc); J += 32) coarse[J * nc] = coarse[J * nc + nc - 1] = 0.0f;
  if (r0 != 0 && r1 != R) return;
  for (int I = lane; I < nc; I += 32) {
    if (r0 == 0) coarse[I] = 0.0f;
    if (r1 == R) coarse[(nc - 1) * nc + I] = 0.0f;
  }
}
// Any sides: the sums and packed coordinates of the nodes on the row itself ([0]) and on the next one
// ([1]); a neighbour off the grid, next to a free side, adds 0.
struct RestrictAny {
  float s[2][2];
  int xy[2][2];
  __device__ __forceinline__ void row(const View& v, const float (&d)[4], int, int, int flat, bool store) {
    const float l1 = __shfl_up_sync(kFull, d[3], 1), l2 = __shfl_up_sync(kFull, d[2], 1);
    const float r1 = __shfl_down_sync(kFull, d[0], 1);
    const float w[7] = {l2, l1, d[0], d[1], d[2], d[3], r1};           // columns -2 .. 4
    const int n1 = v.n - 1, W = 1 << v.L;
    const float q = 0.25f, h = 0.5f;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float* c = w + 2 + 2 * e;
      {                                           // the nodes on row r - 1
        const int x = xy[0][e] & 0xffff, y = xy[0][e] >> 16;
        const bool t = y < n1;
        float u = s[0][e];
        u = fmaf(q, x > 0 && t ? c[0] : 0.0f, u);
        u = fmaf(h, t ? c[1] : 0.0f, u);
        u = fmaf(q, x < n1 && t ? c[2] : 0.0f, u);
        if (store && !((x | y) & 1) && y <= n1) {
          const int I = x >> 1, J = y >> 1, nc = (n1 >> 1) + 1;
          v.coarse[J * nc + I] = is_dirichlet(I, J, nc, v.bc) ? 0.0f : u;
        }
      }
      {                                           // the nodes on row r
        const int x = xy[1][e] & 0xffff;
        float u = s[1][e];
        u = fmaf(h, x > 0 ? c[-1] : 0.0f, u);
        u = u + c[0];
        u = fmaf(h, x < n1 ? c[1] : 0.0f, u);
        s[0][e] = u;
        xy[0][e] = xy[1][e];
      }
      {                                           // the nodes on row r + 1
        int x, y;
        node_xy(flat + W + 2 * e, v.L, x, y);
        const bool b = y > 0;
        float u = q * (x > 0 && b ? c[-2] : 0.0f);
        u = fmaf(h, b ? c[-1] : 0.0f, u);
        u = fmaf(q, x < n1 && b ? c[0] : 0.0f, u);
        s[1][e] = u;
        xy[1][e] = x | (y << 16);
      }
    }
  }
};

// The strip of a warp: `own` columns per strip, `side` more on either side
struct Strip {
  int own, side;
};

// The down part.  MODE DOWN_ZERO: the iterate is zero (x1 = omega D^-1 b without a stencil); DOWN: it is
// v.x, and the squares of its residual go to v.squares.  early: the bands of the first kSlots rows are
// on their way already (cur: the copies' cursor past them).
template <class Pol, int MODE, class Restrict>
__device__ void march_down(const View& v, const Strip& st, const Item& it, unsigned char* ring, bool early, int lane, bool live) {
  constexpr bool Z = MODE == DOWN_ZERO;
  constexpr int SB = slot_bytes<Pol>(), BB = band_bytes<Pol>();
  const int W = 1 << v.L;
  const int col = 4 * lane - st.side;                                  // relative to the strip's own columns
  const bool mine = col >= 0 && col < st.own && it.c0 + col < W;
  const int first = it.r0 - 3, last = it.r1 + 2;
  const unsigned ring_u = smem_u32(ring);
  int f = first * W + it.c0 + col;                // the lane's first node in row i
  Cursor<Pol> cur;
  cur.start(v, f, f + W);                         // (a slot holds the iterate of the row after its own)
#pragma unroll
  for (int q = 0; q < kSlots; ++q) {
    if (live && first + q <= last) {
      if (!early) cur.constants(v.stride, ring_u + q * SB, lane);
      cur.vectors(ring_u + q * SB, lane, !Z);
    }
    copy_commit();
    cur.next(W);
  }
  // the grid coordinates of the lane's first column on row i - 2, row by row (not used before the grid)
  int gx = 0, gy = 0;
  node_xy(f - 2 * W, v.L, gx, gy);
  Bands B0{}, B1{}, B2{}, B3{};                   // rows i, i - 1, i - 2, i - 3
  Field X0{}, X1{}, X2{};
  Restrict rs{};
  float b0[4] = {}, b1[4] = {}, b2[4] = {}, w0[4] = {}, w1[4] = {};
  if constexpr (!Z) {                             // rows i - 1 and i of the iterate, the bands of row i - 1
    load_bands_ahead<Pol>(B0, v, f - W, live);
    if (live) {
      ld4<LD_NC>(v.x + (f - W), X0.m);
      ld4<LD_NC>(v.x + f, X0.c);
    }
    X0.ml = __shfl_up_sync(kFull, X0.m[3], 1);
    X0.cr = __shfl_down_sync(kFull, X0.c[0], 1);
  }
  int i = first, s = 0;                           // the row and its slot
  auto step = [&]() __attribute__((always_inline)) {
    copy_wait<kSlots - 1>();
    const unsigned char* slot = ring + s * SB;
    B3 = B2; B2 = B1; B1 = B0;
#pragma unroll
    for (int m = 0; m < 4; ++m) { b2[m] = b1[m]; b1[m] = b0[m]; w1[m] = w0[m]; }
    load_bands<Pol>(B0, slot, lane, v.scale);
    lds4(slot + 5 * BB + lane * 16, w0);
    lds4(slot + 5 * BB + kTile * 4 + lane * 16, b0);
    float p[4], acc[4], x1[4];
    if constexpr (Z) {
#pragma unroll
      for (int m = 0; m < 4; ++m) x1[m] = mul_rn(w0[m], b0[m]);
    } else {
      lds4(slot + 5 * BB + 2 * kTile * 4 + lane * 16, p);              // row i + 1
      const float c[4] = {X0.c[0], X0.c[1], X0.c[2], X0.c[3]};
      apply_row<Pol>(B0, B1, X0, p, acc);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        acc[m] = b0[m] - acc[m];
        x1[m] = fmaf(w0[m], acc[m], c[m]);
      }
      if (v.squares && mine && i >= it.r0 && i < it.r1 && f < v.pitch) {
        const float2 q = lane_sumsq(acc);
        *reinterpret_cast<float2*>(v.squares + (f >> 1)) = q;
      }
    }
    if (live && i + kSlots <= last) {             // (the slot was read above)
      cur.constants(v.stride, ring_u + s * SB, lane);
      cur.vectors(ring_u + s * SB, lane, !Z);
      cur.next(W);
    }
    copy_commit();
    s = s + 1 == kSlots ? 0 : s + 1;
    {                                             // the second step on row i - 1
      const float c[4] = {X1.c[0], X1.c[1], X1.c[2], X1.c[3]};
      apply_row<Pol>(B1, B2, X1, x1, acc);
#pragma unroll
      for (int m = 0; m < 4; ++m) p[m] = fmaf(w1[m], b1[m] - acc[m], c[m]);
      if (mine && i - 1 >= it.r0 && i - 1 < it.r1 && f - W < v.pitch) st4(v.out + (f - W), p);
    }
    // the defect on row i - 2, and the restriction around row i - 3
    apply_row<Pol>(B2, B3, X2, p, acc);
#pragma unroll
    for (int m = 0; m < 4; ++m) acc[m] = b2[m] - acc[m];
    rs.row(v, acc, gx, gy, f - 2 * W, mine && i >= it.r0 + 3);
    if (--gx < 0) gx += v.n;
    else ++gy;
    ++i;
    f += W;
  };
  for (;;) {
    step();
    if (i > last) break;
    step();
    if (i > last) break;
    step();
    if (i > last) break;
    step();
    if (i > last) break;
  }
  copy_wait<0>();
}

// The coarse values that a lane's four nodes of a fine row interpolate from, loaded a row ahead: columns
// ex / 2 .. ex / 2 + 2 of coarse row ey / 2 and (odd ey) the next one; for nodes that wrap into the next
// fine row, also columns 0 and 1 of the coarse rows below that one's.
struct Coarse {
  float e[2][3], w[2][2];
  int x, y;                              // the first node
  int kind;                              // 0: off the grid, 1: one fine row, 2: wraps
};
__device__ __forceinline__ void load_coarse(const View& v, int f, bool live, Coarse& q) {
  const int n = v.n, nc = (n >> 1) + 1;
  q.kind = 0;
  if (!live || f < 0 || f >= n * n) return;
  node_xy(f, v.L, q.x, q.y);
  q.kind = q.x + 3 < n ? 1 : 2;
  const float* e = v.coarse + (q.y >> 1) * nc + (q.x >> 1);
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    q.e[0][m] = __ldg(e + m);
    q.e[1][m] = (q.y & 1) ? __ldg(e + nc + m) : 0.0f;
  }
  if (q.kind == 2) {                     // (beyond the last row of the grid: the array's halo, unused)
    const float* w = v.coarse + ((q.y + 1) >> 1) * nc;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      q.w[0][m] = __ldg(w + m);
      q.w[1][m] = ((q.y + 1) & 1) ? __ldg(w + nc + m) : 0.0f;
    }
  }
}
// y += P e at the lane's nodes, with prolong_tile's arithmetic.  (Column 4 l of the strip is even, so the
// coordinates of a lane's first node are both even or both odd.)
__device__ __forceinline__ void add_coarse(const View& v, const Coarse& q, float (&y)[4]) {
  if (q.kind == 0) return;
  const float (&e)[3] = q.e[0], (&g)[3] = q.e[1];
  float z[4];
  if (q.y & 1) {
    z[0] = fmaf(0.25f, ((e[0] + e[1]) + g[0]) + g[1], y[0]);
    z[1] = fmaf(0.5f, e[1] + g[1], y[1]);
    z[2] = fmaf(0.25f, ((e[1] + e[2]) + g[1]) + g[2], y[2]);
    z[3] = fmaf(0.5f, e[2] + g[2], y[3]);
  } else {
    z[0] = y[0] + e[0];
    z[1] = fmaf(0.5f, e[0] + e[1], y[1]);
    z[2] = y[2] + e[1];
    z[3] = fmaf(0.5f, e[1] + e[2], y[3]);
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    int px = q.x + m, py = q.y;
    if (q.kind == 2 && px >= v.n) {
      px -= v.n;
      ++py;
      if (py >= v.n) continue;
      const int a = px >> 1, b = (px + 1) >> 1;
      const bool ny = py & 1;
      const float a0 = a ? q.w[0][1] : q.w[0][0], a1 = a ? q.w[1][1] : q.w[1][0];
      const float b0 = b ? q.w[0][1] : q.w[0][0], b1 = b ? q.w[1][1] : q.w[1][0];
      if (px & 1) z[m] = ny ? fmaf(0.25f, ((a0 + b0) + a1) + b1, y[m]) : fmaf(0.5f, a0 + b0, y[m]);
      else z[m] = ny ? fmaf(0.5f, a0 + a1, y[m]) : y[m] + a0;
    }
    if (!is_dirichlet(px, py, v.n, v.bc)) y[m] = z[m];
  }
}

// The up part: y = x + P e on row i, the first step on row i - 1, the second on row i - 2
template <class Pol>
__device__ void march_up(const View& v, const Strip& st, const Item& it, unsigned char* ring, bool early, int lane, bool live) {
  constexpr int SB = slot_bytes<Pol>(), BB = band_bytes<Pol>();
  const int W = 1 << v.L;
  const int col = 4 * lane - st.side;
  const bool mine = col >= 0 && col < st.own && it.c0 + col < W;
  const int first = it.r0 - 2, last = it.r1 + 1;
  const unsigned ring_u = smem_u32(ring);
  int f = first * W + it.c0 + col;
  Cursor<Pol> cur;
  cur.start(v, f, f);
#pragma unroll
  for (int q = 0; q < kSlots; ++q) {
    if (live && first + q <= last) {
      if (!early) cur.constants(v.stride, ring_u + q * SB, lane);
      cur.vectors(ring_u + q * SB, lane, true);
    }
    copy_commit();
    cur.next(W);
  }
  Bands B0{}, B1{}, B2{}, B3{};
  Field Y{}, X1{};
  float b0[4] = {}, b1[4] = {}, b2[4] = {}, w0[4] = {}, w1[4] = {}, w2[4] = {};
  Coarse e;
  load_coarse(v, f, live, e);
  int i = first, s = 0;
  auto step = [&]() __attribute__((always_inline)) {
    copy_wait<kSlots - 1>();
    const unsigned char* slot = ring + s * SB;
    B3 = B2; B2 = B1; B1 = B0;
#pragma unroll
    for (int m = 0; m < 4; ++m) { b2[m] = b1[m]; b1[m] = b0[m]; w2[m] = w1[m]; w1[m] = w0[m]; }
    load_bands<Pol>(B0, slot, lane, v.scale);
    lds4(slot + 5 * BB + lane * 16, w0);
    lds4(slot + 5 * BB + kTile * 4 + lane * 16, b0);
    float y[4], acc[4], x1[4];
    lds4(slot + 5 * BB + 2 * kTile * 4 + lane * 16, y);
    add_coarse(v, e, y);
    load_coarse(v, f + W, live, e);
    if (live && i + kSlots <= last) {
      cur.constants(v.stride, ring_u + s * SB, lane);
      cur.vectors(ring_u + s * SB, lane, true);
      cur.next(W);
    }
    copy_commit();
    s = s + 1 == kSlots ? 0 : s + 1;
    {
      const float c[4] = {Y.c[0], Y.c[1], Y.c[2], Y.c[3]};
      apply_row<Pol>(B1, B2, Y, y, acc);
#pragma unroll
      for (int m = 0; m < 4; ++m) x1[m] = fmaf(w1[m], b1[m] - acc[m], c[m]);
    }
    {
      const float c[4] = {X1.c[0], X1.c[1], X1.c[2], X1.c[3]};
      apply_row<Pol>(B2, B3, X1, x1, acc);
#pragma unroll
      for (int m = 0; m < 4; ++m) acc[m] = fmaf(w2[m], b2[m] - acc[m], c[m]);
      if (mine && i >= it.r0 + 2 && f - 2 * W < v.pitch) st4(v.out + (f - 2 * W), acc);
    }
    ++i;
    f += W;
  };
  for (;;) {
    step();
    if (i > last) break;
    step();
    if (i > last) break;
    step();
    if (i > last) break;
    step();
    if (i > last) break;
  }
  copy_wait<0>();
}

// How a level is cut: strips of `own` columns, chunks of `rows` rows
struct Geom {
  int strips, own, chunks, rows, R;
};
constexpr int kLeastRows = 2;            // of a chunk, in a launch that serves several problems
__host__ __device__ inline Geom march_strips(int L, int up) {
  Geom g;
  const unsigned W = 1u << L, widest = kTile - 2 * (up ? 4 : 8);
  const long long n = W + 1, pitch = (n * n + kTile - 1) / kTile * kTile;
  g.strips = (int)((W + widest - 1) / widest);
  g.own = (int)((W / 4 + g.strips - 1) / g.strips * 4);
  g.R = (int)((pitch + W - 1) >> L);
  g.chunks = 1;
  g.rows = g.R;
  return g;
}
// Rows of a chunk so that S strips fill whole waves of G warps: a chunk of r rows costs r + 6 iterations
// and about 6 to start
inline void march_chunks(Geom& g, unsigned S, unsigned G) {
  unsigned best = 0xffffffffu;
  for (unsigned w = 1; w <= 3; ++w) {
    unsigned c = w * G / S;
    if (c < 1) continue;
    c = c > (unsigned)g.R / 2 ? (unsigned)g.R / 2 : c;
    const unsigned rows = ((unsigned)g.R + c - 1) / c, cost = w * (rows + 12);
    if (cost < best) { best = cost; g.rows = (int)rows; }
  }
  g.chunks = (g.R + g.rows - 1) / g.rows;
}

// (the whole warp, between two __syncwarp)
template <class Pol, bool UPWARD>
__device__ __forceinline__ void make_view(View& v, const LevelDev& d, const LevelDev& dc, int e_sel, float* scale,
                                          bool squares) {
  const int lane = threadIdx.x & 31;
  __syncwarp();                                   // the previous item's readers
  if (lane < 5) scale[lane] = d.scale[lane + 4];
  if (lane == 0) {
    v.band = static_cast<const unsigned char*>(d.band[4]);
    v.stride = static_cast<const unsigned char*>(d.band[5]) - v.band;   // the bands are equal arrays in a row
    v.wd = d.wdf;
    v.b = static_cast<const float*>(d.rhs);
    v.x = static_cast<const float*>(d.x[UPWARD ? 1 : 0]);
    v.out = static_cast<float*>(d.x[UPWARD ? 0 : 1]);
    v.coarse = static_cast<float*>(UPWARD ? (e_sel ? dc.x[1] : dc.x[0]) : dc.rhs);
    v.squares = squares ? static_cast<float*>(d.r) : nullptr;
    v.scale = scale;
    v.L = d.L;
    v.n = d.n;
    v.pitch = d.pitch;
    v.bc = d.bc;
  }
  __syncwarp();
}

__device__ __forceinline__ Item item_of(const Geom& g, int s) {
  const int ch = s / g.strips;
  Item it;
  it.c0 = (s - ch * g.strips) * g.own;
  it.r0 = ch * g.rows;
  it.r1 = min(g.R, it.r0 + g.rows);
  return it;
}
// the lane's columns belong to the widened strip (and to the level)
__device__ __forceinline__ bool live_lane(const Strip& st, const Item& it, int lane, int level) {
  return 4 * lane < st.own + 2 * st.side && it.c0 + 4 * lane < (1 << level) + 2 * st.side;
}

template <class Pol, bool UPWARD>
__device__ __forceinline__ void sweep(const View& v, const Strip& st, const Item& it, unsigned char* ring, bool early, bool zero,
                                      int lane, bool live) {
  if constexpr (UPWARD) march_up<Pol>(v, st, it, ring, early, lane, live);
  else if (v.bc == (int)HN_DIRICHLET_ALL) {
    if (it.c0 == 0) zero_sides(v.coarse, v.n, it.r0, it.r1, (v.pitch + (1 << v.L) - 1) >> v.L, lane);
    if (zero) march_down<Pol, DOWN_ZERO, RestrictInner>(v, st, it, ring, early, lane, live);
    else march_down<Pol, DOWN, RestrictInner>(v, st, it, ring, early, lane, live);
  } else {
    if (zero) march_down<Pol, DOWN_ZERO, RestrictAny>(v, st, it, ring, early, lane, live);
    else march_down<Pol, DOWN, RestrictAny>(v, st, it, ring, early, lane, live);
  }
}

// A level's down or up part for an engine of one problem, which passes its descriptors and the cut of the
// level by value.  e_sel (up): the coarse iterate's buffer.
template <class Pol, bool UPWARD>
__global__ void __launch_bounds__(kWarps * 32, 4) k_march(EngineDev E, TileList tl, int level, int want, int e_sel, Geom g) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ float scale[kWarps][8];
  __shared__ View views[kWarps];
  pdl_trigger();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* ring = smem + warp * kSlots * slot_bytes<Pol>();
  const int gw = (int)blockIdx.x * kWarps + warp, G = (int)gridDim.x * kWarps;
  View& v = views[warp];                          // (in shared memory: its pointers take no registers)
  // the coarsest level, or one that the problem does not have (a server's engine of one slot may be built for a
  // larger one): nothing to do, but the launch must not end before the one it follows, which the next one's wait
  // would then no longer cover
  if (tl.solo_c.n == 0 || !dbg_level(E, tl.solo_d, level, tl.solo_tiles, HN_HERE)) {
    pdl_wait();
    return;
  }
  // (a zero iterate leaves no squares)
  make_view<Pol, UPWARD>(v, tl.solo_d, tl.solo_c, e_sel, scale[warp], E.prm.solver != SOLVER_PCG);
  const int items = g.strips * g.chunks;
  if (gw >= items) return;
  const Strip st{g.own, UPWARD ? 4 : 8};
  Item it = item_of(g, gw);
  // the bands and omega / D of the first rows are constant: fetched before the preceding launch ends
  if (live_lane(st, it, lane, level)) {
    const int first = it.r0 - (UPWARD ? 2 : 3), last = it.r1 + (UPWARD ? 1 : 2);
    Cursor<Pol> cur;
    cur.start(v, (first << level) + it.c0 + 4 * lane - st.side, 0);
    for (int q = 0; q < kSlots && first + q <= last; ++q, cur.next(1 << level))
      cur.constants(v.stride, smem_u32(ring) + q * slot_bytes<Pol>(), lane);
  }
  pdl_wait();
  const ProbState& S = E.S[0];
  if (S.phase != want) {
    copy_commit();
    copy_wait<0>();
    return;
  }
  const bool zero = tl.solo_L > level || S.zero_top;
  for (int s = gw; s < items; s += G) {
    it = item_of(g, s);
    sweep<Pol, UPWARD>(v, st, it, ring, s == gw, zero, lane, live_lane(st, it, lane, level));
  }
}

// The down or up part of level `level` for the problems with a finer level, or (level 0) of every problem's
// own finest level above the tail level T, in one launch: the strips of all problems in the phase are cut
// into chunks of one height, so that they fill one wave of warps.
template <class Pol, bool UPWARD>
__global__ void __launch_bounds__(kWarps * 32, 4) k_march_group(EngineDev E, int level, int T, int want) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ float scale[kWarps][8];
  __shared__ View views[kWarps];
  __shared__ Served q;
  __shared__ int2 cut[kMaxLevel + 1];             // strips and rows of a level
  __shared__ int hist[kMaxLevel + 1], s_rows;
  pdl_trigger();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* ring = smem + warp * kSlots * slot_bytes<Pol>();
  const int gw = (int)blockIdx.x * kWarps + warp, G = (int)gridDim.x * kWarps;
  View& v = views[warp];
  if (threadIdx.x <= kMaxLevel) {
    const Geom g = march_strips((int)threadIdx.x, UPWARD);
    cut[threadIdx.x] = make_int2(g.strips, g.R);
  }
  pdl_wait();
  for (int base = 0; base < E.nprob; base += kListMax) {
    const int n = list_served(E, q, base, level, [&](const ProbState& S, int L) { return S.phase == want && L > (level ? level : T); });
    if (n == 0) continue;
    // one height for all chunks: the smallest of 32 candidates that takes no more items than warps
    if (threadIdx.x < kMaxLevel + 1) hist[threadIdx.x] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) atomicAdd(&hist[q.level[i]], 1);
    __syncthreads();
    if (threadIdx.x < 32) {
      int total = 0;
      for (int l = kMarchMinLevel; l <= kMaxLevel; ++l) total += hist[l] * cut[l].x * cut[l].y;
      const int least = max(kLeastRows, (total + G - 1) / G), rows = least + lane * max(1, least / 16);
      int items = 0;
      for (int l = kMarchMinLevel; l <= kMaxLevel; ++l)
        if (hist[l]) items += hist[l] * cut[l].x * ((cut[l].y + rows - 1) / rows);
      const unsigned fits = __ballot_sync(kFull, items <= G);
      const int best = fits ? __ffs(fits) - 1 : 31;
      if (lane == best) s_rows = rows;
    }
    __syncthreads();
    const int rows = s_rows;
    const int items = number_items(q, n, [&](int l) { return cut[l].x * ((cut[l].y + rows - 1) / rows); });
    for (int it = gw; it < items; it += G) {
      const int m = served_of(q, n, it), p = q.slot[m], l = q.level[m];
      if (!dbg_item(E, p, 0, l, HN_HERE)) continue;
      const ProblemDev& P = E.P[p];
      const bool zero = P.L > l || E.S[p].zero_top;
      make_view<Pol, UPWARD>(v, P.lev[l], P.lev[l - 1], 0, scale[warp], E.prm.solver != SOLVER_PCG);
      Geom g = march_strips(l, UPWARD);
      g.rows = rows;
      const Strip st{g.own, UPWARD ? 4 : 8};
      const Item t = item_of(g, it - q.start[m]);
      sweep<Pol, UPWARD>(v, st, t, ring, false, zero, lane, live_lane(st, t, lane, l));
    }
    __syncthreads();
  }
}

// The norm partials of a marching down sweep: the pairs of a 128-node tile's lanes (left in the level's
// defect array, which the sweep does not need) summed by the butterfly of tile_sumsq, for every problem
// whose finest level is `level` and whose iterate was not zero.  A warp takes 32 tiles: a step of the
// butterfly gives both halves of the lanes the same sum, so each step sums two tiles at once, half of the
// lanes keeping one, half the other, and lane t ends with tile t (31 pair sums in place of 160).
__device__ __forceinline__ float2 tile_pairs(const float* r, int tile0, int ntiles) {
  const int lane = threadIdx.x & 31;
  const float2* p = reinterpret_cast<const float2*>(r) + (long long)tile0 * 32 + lane;
  float2 q[32];
#pragma unroll
  for (int t = 0; t < 32; ++t) q[t] = tile0 + t < ntiles ? __ldcg(p + t * 32) : make_float2(0.0f, 0.0f);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int t = 0; t < o; ++t) {
      float2 keep = up ? q[t + o] : q[t];
      const float2 give = up ? q[t] : q[t + o];
      const float bh = __shfl_xor_sync(kFull, give.x, o), bl = __shfl_xor_sync(kFull, give.y, o);
      df_add(keep.x, keep.y, bh, bl);
      q[t] = keep;
    }
  }
  return q[0];
}

// The lagged check of problem p with finest level `level`, by the blocks that hold its squares: block `blk`
// of nb that serve group j of the problem's tiles sums its tiles; the last block of a group sums the
// group; the last group adds the groups in order and decides.  want: the phase of the cycle.
__device__ void check_part(const EngineDev& E, int p, const float* squares, int level, int j, int blk, int nb, int want, double* sh) {
  __shared__ int s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tiles = fine_tiles(level), groups = sum_groups(tiles);
  double* part = E.partial + E.fine_off[p];
  const int lo = j * kSumGroup, hi = min(tiles, lo + kSumGroup);
  for (int t = lo + (blk * 8 + warp) * 32; t < hi; t += nb * 256) {
    const float2 q = tile_pairs(squares, t, hi);
    if (t + lane < hi) store_partial(part + t + lane, q);
  }
  unsigned* ticket = E.gticket + (long long)p * ticket_words(E.ctl_groups);
  double* gsum = E.gsum + (long long)p * E.ctl_groups;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(ticket + 2 + j, 1u) == (unsigned)nb - 1u;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const double g = group_partial_sum(part, tiles, j, sh, true);
  __syncthreads();
  if (threadIdx.x == 0) {
    ticket[2 + j] = 0u;
    s_last = 1;
    if (groups > 1) {
      gsum[j] = g;
      __threadfence();
      s_last = atomicAdd(ticket + 1, 1u) == (unsigned)groups - 1u;
    }
  }
  __syncthreads();
  if (!s_last || threadIdx.x >= 32) return;
  double sum = g;
  if (groups > 1) {
    __threadfence();
    sum = 0.0;
    for (int b = 0; b < groups; b += 32) {        // group sums in group order, as problem_norm_sum
      const double mine = b + lane < groups ? __ldcg(gsum + b + lane) : 0.0;
      for (int k = 0; k < 32 && b + k < groups; ++k) sum += __shfl_sync(kFull, mine, k);
    }
  }
  if (threadIdx.x == 0) {
    ProbState& st = E.S[p];
    if (groups > 1) ticket[1] = 0u;
    pre_check(st, E.prm, sqrt(sum));
    if (st.phase == want) cond_set(E.prm.cond, 1u);
  }
}

// after the down part of the finest level: of an engine of one problem, nb blocks per group ...
__global__ void __launch_bounds__(256) k_march_check(EngineDev E, TileList tl, int level, int want, int nb) {
  pdl_start();
  __shared__ double sh[32];
  const ProbState& st = E.S[0];
  if (st.phase != want) return;
  if (tl.solo_L != level || st.zero_top) {        // nothing to check: the cycle goes on
    if (blockIdx.x == 0 && threadIdx.x == 0) cond_set(E.prm.cond, 1u);
    return;
  }
  check_part(E, 0, static_cast<const float*>(tl.solo_d.r), level, (int)blockIdx.x / nb, (int)blockIdx.x % nb, nb, want, sh);
}
// ... and of all problems whose finest level is above the tail, one block per 1024 tiles at most: the blocks of a problem
// (whole groups of kSumGroup tiles)
__host__ __device__ inline int check_blocks(int L, int T) {
  const int tiles = fine_tiles(L), first = tiles < kSumGroup ? tiles : kSumGroup;
  return L <= T ? 1 : sum_groups(tiles) * ((first + 1023) / 1024);
}
__global__ void __launch_bounds__(256) k_march_check_group(EngineDev E, int T, int want) {
  pdl_start();
  __shared__ double sh[32];
  __shared__ Served q;
  for (int base = 0; base < E.nprob; base += kListMax) {
    const int n = list_served(E, q, base, 0, [](const ProbState&, int L) { return L >= HN_MIN_LEVEL; });
    if (n == 0) continue;
    const int items = number_items(q, n, [T](int l) { return check_blocks(l, T); });
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
      const int m = served_of(q, n, it), p = q.slot[m], l = q.level[m], blk = it - q.start[m];
      // (a problem leaves the phase only after every block of its check has counted itself in)
      if (!dbg_item(E, p, 0, l, HN_HERE) || __ldcg(&E.S[p].phase) != want) continue;
      if (l <= T || E.S[p].zero_top) {            // no check (or the tail's own): the cycle goes on
        if (blk == 0 && threadIdx.x == 0) cond_set(E.prm.cond, 1u);
        continue;
      }
      const int nb = (min(fine_tiles(l), kSumGroup) + 1023) / 1024;
      check_part(E, p, static_cast<const float*>(E.P[p].lev[l].r), l, blk / nb, blk % nb, nb, want, sh);
      __syncthreads();
    }
    __syncthreads();
  }
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), int grid, int threads, size_t smem, cudaStream_t s, int pdl, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  if (pdl_launch(pdl, grid)) {
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 1;
    cfg.attrs = attr;
  }
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// resident blocks per SM of a marching kernel (its shared memory allowed on the first call); 0: none
template <class K>
int march_resident(K kern, int smem) {
  int b = 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, kWarps * 32, smem) != cudaSuccess)
    return 0;
  return b;
}

template <class Pol, bool UPWARD>
cudaError_t launch_march_t(const EngineDev& E, const TileList& tl, int level, int want, int e_sel, cudaStream_t s) {
  constexpr int smem = kWarps * kSlots * slot_bytes<Pol>();
  static const int per_sm = march_resident(k_march<Pol, UPWARD>, smem);
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  Geom g = march_strips(level, UPWARD ? 1 : 0);
  march_chunks(g, (unsigned)g.strips, (unsigned)(per_sm * sm_count() * kWarps));
  const int grid = std::min(per_sm * sm_count(), (g.strips * g.chunks + kWarps - 1) / kWarps);
  // programmatic at any size (unless off): the waiting blocks fetch their first rows' constant data meanwhile.  By the
  // rule (pdl_launch) the large levels' would not be: L = 10 solve 1344 -> 1383 us, L = 12 9300 -> 9524, FP16 9369 ->
  // 9687, CG at L = 11 3379 -> 3492.
  return launch_pdl(k_march<Pol, UPWARD>, grid, kWarps * 32, smem, s, E.pdl ? 1 : 0, E, tl, level, want, e_sel, g);
}

template <class Pol, bool UPWARD>
cudaError_t launch_group_t(const EngineDev& E, const GroupSize& size, int level, int T, int want, cudaStream_t s) {
  constexpr int smem = kWarps * kSlots * slot_bytes<Pol>();
  static const int per_sm = march_resident(k_march_group<Pol, UPWARD>, smem);
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // no more than one wave of blocks, nor than have work where every chunk has the least height
  const long long items = size.sum([&](int l) {
    if (l <= (level ? level : T)) return 0;
    const Geom g = march_strips(level ? level : l, UPWARD ? 1 : 0);
    return g.strips * ((g.R + kLeastRows - 1) / kLeastRows);
  });
  const int grid = (int)std::max<long long>(1, std::min<long long>(per_sm * sm_count(), (items + kWarps - 1) / kWarps));
  // never programmatic: what they can do before their predecessor ends is little, and blocks of 230 registers a thread
  // that wait on every SM hold up whatever else runs, such as a server's set-up of the next requests (24 requests of
  // L = 6..8, FP16 13.2 -> 10.4 ms, of L = 6..9 in FP32 11.1 -> 9.8; a batch of 64 6.26 -> 6.13; below the number of SMs
  // too: 2 problems of L = 5..7 1467 -> 1515 us)
  return launch_pdl(k_march_group<Pol, UPWARD>, grid, kWarps * 32, smem, s, 0, E, level, T, want);
}

}  // namespace

cudaError_t launch_march(const EngineDev& E, const TileList& tl, int level, int want, int up, int e_sel, cudaStream_t s) {
  if (level < kMarchMinLevel) return cudaErrorInvalidValue;
  if (E.prm.prec == P32)
    return up ? launch_march_t<F32, true>(E, tl, level, want, e_sel, s) : launch_march_t<F32, false>(E, tl, level, want, e_sel, s);
  if (E.prm.prec == P16)
    return up ? launch_march_t<F16, true>(E, tl, level, want, e_sel, s) : launch_march_t<F16, false>(E, tl, level, want, e_sel, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_march_group(const EngineDev& E, const GroupSize& size, int level, int T, int want, int up, cudaStream_t s) {
  if ((level ? level : T + 1) < kMarchMinLevel) return cudaErrorInvalidValue;
  if (E.prm.prec == P32)
    return up ? launch_group_t<F32, true>(E, size, level, T, want, s) : launch_group_t<F32, false>(E, size, level, T, want, s);
  if (E.prm.prec == P16)
    return up ? launch_group_t<F16, true>(E, size, level, T, want, s) : launch_group_t<F16, false>(E, size, level, T, want, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_march_check(const EngineDev& E, const TileList& tl, int level, int want, cudaStream_t s) {
  // 256 tiles a block, whole groups
  const int tiles = (int)(pitch_of(level) / kTile);
  const int groups = (tiles + kSumGroup - 1) / kSumGroup, nb = (std::min(tiles, kSumGroup) + 255) / 256;
  return launch_pdl(k_march_check, groups * nb, 256, 0, s, E.pdl, E, tl, level, want, nb);
}

cudaError_t launch_march_check_group(const EngineDev& E, const GroupSize& size, int T, int want, cudaStream_t s) {
  const long long items = size.sum([&](int l) { return check_blocks(l, T); });
  const int grid = (int)std::max<long long>(1, std::min<long long>(2 * sm_count(), items));
  return launch_pdl(k_march_check_group, grid, 256, 0, s, E.pdl, E, T, want);
}

}  // namespace hn
