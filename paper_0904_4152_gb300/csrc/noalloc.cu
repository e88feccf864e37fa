// Defect and norm of an assembled operator without any device allocation.
//
// hn_band_defect_norm_static computes r = b - A x and ||r||_2 for an operator built by
// hn_band_create, on caller-owned device vectors.  It exists for callers that cannot call
// cudaMalloc at that point: code that runs while another thread captures a CUDA graph in global
// mode (allocation is not permitted then), processes that hand out their whole device-memory plan
// up front, and latency-critical paths where cudaMalloc / cudaFree would synchronize the device.
// The only temporary, one partial sum of squares per strip of tiles, lives in the file-scope array
// below, so the call allocates nothing: every GPU that loads the library holds the array (29 KB)
// until the process exits.
#include <algorithm>
#include <mutex>

#include "engine.h"

namespace hn {
namespace {

constexpr long long kStaticMaxNodes = 65536LL * kTile;   // the largest operator that the contract takes (level 11)
// Strips of tiles, each with a partial sum in the array: three blocks of 8 warps on each of 152 SMs, also where the
// chip has another number (the order of the sum is fixed).
constexpr int kStrips = 3648;
constexpr unsigned kFullMask = 0xffffffffu;

// Scratch shared by every call on a device.  Each call writes its slots before reading
// them, so nothing has to start at zero; calls that overlap on the GPU race on it.
static __device__ __align__(256) double g_partials[kStrips];

// device address of g_partials, looked up once per device with that device current
constexpr int kMaxDevices = 64;
double* g_addr[kMaxDevices] = {};
std::mutex g_addr_mu;

hn_status scratch_for_current_device(double** out) {
  int dev = 0;
  HN_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return set_error(HN_ERR_ARG, "device ordinal %d unsupported", dev);
  std::lock_guard<std::mutex> lk(g_addr_mu);
  if (!g_addr[dev]) {
    void* p = nullptr;
    HN_CUDA(cudaGetSymbolAddress(&p, g_partials));
    g_addr[dev] = static_cast<double*>(p);
  }
  *out = g_addr[dev];
  return HN_OK;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFullMask, v, o);
  return v;
}

// Row window w[o + 2] = x[a + o], o = -2..5, of plain (unpadded) vectors: entries outside [0, N)
// read as 0 (their band entries are 0).  Warps whose windows lie inside use aligned vector loads
// and shuffles for the overhang, as the solver's kernel does; the first and last rows fall back
// to guarded scalar loads.
__device__ __forceinline__ void row_window(const double* __restrict__ x, long long a, long long N,
                                           int lane, double (&w)[8]) {
  const bool inside = __all_sync(kFullMask, a - 2 >= 0 && a + 5 < N);
  if (inside) {
    const double2 p = __ldg(reinterpret_cast<const double2*>(x + a));
    const double2 q = __ldg(reinterpret_cast<const double2*>(x + a) + 1);
    double l2 = __shfl_up_sync(kFullMask, q.x, 1), l1 = __shfl_up_sync(kFullMask, q.y, 1);
    double r0 = __shfl_down_sync(kFullMask, p.x, 1), r1 = __shfl_down_sync(kFullMask, p.y, 1);
    if (lane == 0) { l2 = __ldg(x + a - 2); l1 = __ldg(x + a - 1); }
    if (lane == 31) { r0 = __ldg(x + a + 4); r1 = __ldg(x + a + 5); }
    w[0] = l2; w[1] = l1; w[2] = p.x; w[3] = p.y; w[4] = q.x; w[5] = q.y; w[6] = r0; w[7] = r1;
  } else {
#pragma unroll
    for (int o = -2; o <= 5; ++o) {
      const long long j = a + o;
      w[o + 2] = (j >= 0 && j < N) ? __ldg(x + j) : 0.0;
    }
  }
}

// r = b - A x on 128-node warp-tiles of [0, N) (the last one ragged), as one chain from b.  Strip v of `strips` holds
// the tiles v, v + strips, ..; slot v of the scratch gets its sum of r^2 (a lane adds its nodes in order, then the
// lanes in a fixed tree).  Bands are the operator's pitch-padded FP64 arrays.
//
// Bound by the FP64 pipe (10 operations a node, 80 us at L = 11, where the bytes take 60): so the defect's subtraction
// is part of the chain and the lanes add up once a strip, not once a tile (11 + 5/4 operations a node before).  With
// the sum of 32,801 tiles by one block after it, L = 11 took 157 us, now 85; L = 10 43, now 29.
__global__ void __launch_bounds__(256, 3) k_defect_static(BandPtrs64c band, int L, long long N,
                                                          const double* __restrict__ x,
                                                          const double* __restrict__ b,
                                                          double* __restrict__ r, double* partials,
                                                          int tiles, int strips) {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  const int lane = threadIdx.x & 31;
  const int v = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (v >= strips) return;
  const long long shift = 1LL << L;
  double s = 0.0;
  for (int t = v; t < tiles; t += strips) {
    const long long i0 = (long long)t * kTile + lane * kLaneNodes;
    const bool whole = i0 + 3 < N;
    double acc[4];
    if (whole) {
      const double2 p = __ldg(reinterpret_cast<const double2*>(b + i0));
      const double2 q = __ldg(reinterpret_cast<const double2*>(b + i0) + 1);
      acc[0] = p.x; acc[1] = p.y; acc[2] = q.x; acc[3] = q.y;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[j] = i0 + j < N ? __ldg(b + i0 + j) : 0.0;
    }
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
      double w[8];
      row_window(x, i0 + dy * shift, N, lane, w);
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) {
        const int k = (dy + 1) * 3 + (dx + 1);
        const double2 p = __ldg(reinterpret_cast<const double2*>(band.p[k] + i0));
        const double2 q = __ldg(reinterpret_cast<const double2*>(band.p[k] + i0) + 1);
        const double bk[4] = {p.x, p.y, q.x, q.y};
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j] = fma(-bk[j], w[j + dy + dx + 2], acc[j]);
      }
    }
    if (whole) {
      reinterpret_cast<double2*>(r + i0)[0] = make_double2(acc[0], acc[1]);
      reinterpret_cast<double2*>(r + i0)[1] = make_double2(acc[2], acc[3]);
#pragma unroll
      for (int j = 0; j < 4; ++j) s = fma(acc[j], acc[j], s);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (i0 + j < N) {
          r[i0 + j] = acc[j];
          s = fma(acc[j], acc[j], s);
        }
    }
  }
  s = warp_sum_d(s);
  if (lane == 0) partials[v] = s;
}

// ||r|| = sqrt of the strips' sums added in a fixed order (one block), its launch overlapping the first kernel's end
__global__ void __launch_bounds__(256) k_sum_partials(const double* partials, int strips,
                                                      double* norm) {
  __shared__ double sh[8];
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  constexpr int kRounds = (kStrips + 255) / 256;
  double v[kRounds], t = 0.0;
#pragma unroll
  for (int k = 0; k < kRounds; ++k) {
    const int q = threadIdx.x + k * 256;
    v[k] = q < strips ? __ldcg(partials + q) : 0.0;
  }
#pragma unroll
  for (int k = 0; k < kRounds; ++k) t += v[k];
  t = warp_sum_d(t);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x < 32) {
    double u = threadIdx.x < 8 ? sh[threadIdx.x] : 0.0;
    u = warp_sum_d(u);
    if (threadIdx.x == 0) *norm = sqrt(u);
  }
}

}  // namespace
}  // namespace hn

using namespace hn;

extern "C" hn_status hn_band_defect_norm_static(const hn_band* A, const double* x, const double* b,
                                                double* r, double* norm, void* stream) {
  clear_error();
  if (!A || !x || !b || !r || !norm) return set_error(HN_ERR_ARG, "null argument");
  if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(b) |
       reinterpret_cast<uintptr_t>(r)) & 15)
    return set_error(HN_ERR_ARG, "x, b and r must be 16-byte aligned device pointers");
  if ((reinterpret_cast<uintptr_t>(norm) & 7))
    return set_error(HN_ERR_ARG, "norm must be an 8-byte aligned device pointer");
  {   // r is written while neighbouring warps still read x and b over the stencil's reach
    const uintptr_t r0 = reinterpret_cast<uintptr_t>(r), r1 = r0 + (uintptr_t)A->N * 8;
    for (const double* v : {x, b}) {
      const uintptr_t v0 = reinterpret_cast<uintptr_t>(v), v1 = v0 + (uintptr_t)A->N * 8;
      if (r0 < v1 && v0 < r1) return set_error(HN_ERR_ARG, "r must not overlap x or b");
    }
  }
  {
    int dev = 0;
    HN_CUDA(cudaGetDevice(&dev));
    if (dev != A->device)
      return set_error(HN_ERR_ARG, "the operator lives on device %d, the current device is %d",
                       A->device, dev);
  }
  if (A->N > kStaticMaxNodes)
    return set_error(HN_ERR_ARG,
                     "%lld nodes exceed the static scratch of this entry point (at most %lld nodes, "
                     "level 11); use hn_mg_apply",
                     A->N, kStaticMaxNodes);
  double* scratch = nullptr;
  HN_TRY(scratch_for_current_device(&scratch));
  const int tiles = (int)((A->N + kTile - 1) / kTile);
  BandPtrs64c bp{};
  for (int k = 0; k < 9; ++k) bp.p[k] = A->band[k];
  const int strips = std::min(tiles, kStrips);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  k_defect_static<<<(strips + 7) / 8, 256, 0, s>>>(bp, A->L, A->N, x, b, r, scratch, tiles, strips);
  HN_CUDA(cudaGetLastError());
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute overlap;
  overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  overlap.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &overlap;
  cfg.numAttrs = 1;
  HN_CUDA(cudaLaunchKernelEx(&cfg, k_sum_partials, static_cast<const double*>(scratch), strips, norm));
  return HN_OK;
}
