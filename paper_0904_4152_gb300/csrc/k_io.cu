// The start and the end of a solve as one kernel each: the right-hand sides (and given iterates) in, the states and
// counters reset; the results out, the states and counters to mapped host memory.
//
// As copies, fills and reads of their own these were 12 operations and four waits for one problem (~75 us of an
// L = 6 solve) and some 1,000 operations for a batch of 256 (~2 ms); the kernels move the same bytes at memory
// speed in one launch for up to kIoMax problems.  A vector that the caller did not put in this device's
// memory is copied by the runtime instead (engine.cu).
#include <algorithm>

#include "k_device.cuh"

namespace hn {

namespace {

// n doubles from src (null: zeros) to dst and, if it is there, to dst2; all 16-byte aligned
__device__ __forceinline__ void move(double* dst, double* dst2, const double* src, long long n) {
  const long long m = n / 2, step = (long long)gridDim.x * blockDim.x;
  double2* d = reinterpret_cast<double2*>(dst);
  double2* d2 = reinterpret_cast<double2*>(dst2);
  const double2* s = reinterpret_cast<const double2*>(src);
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (long long i = t; i < m; i += 4 * step) {
    double2 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = src && i + k * step < m ? s[i + k * step] : make_double2(0.0, 0.0);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i + k * step < m) {
        d[i + k * step] = v[k];
        if (d2) d2[i + k * step] = v[k];
      }
  }
  if (t == 0 && (n & 1)) {
    dst[n - 1] = src ? src[n - 1] : 0.0;
    if (dst2) dst2[n - 1] = dst[n - 1];
  }
}

__device__ __forceinline__ long long nodes(int L) { const long long n = (1LL << L) + 1; return n * n; }

__global__ void __launch_bounds__(256) k_begin(const __grid_constant__ EngineDev E, const __grid_constant__ IoBatch io,
                                               unsigned* taken, unsigned long long* launches) {
  const IoItem& it = io.item[blockIdx.y];
  const ProblemDev& P = E.P[it.slot];
  if (it.b) move(P.b64, nullptr, it.b, nodes(P.L));
  if (it.x || it.clear) move(P.x64, nullptr, it.x, nodes(P.L));
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  ProbState st{};
  st.phase = PH_INIT;
  st.status = HN_PENDING;
  st.zero_top = st.x_zero = !it.guess;
  st.s = st.inv_s = 1.0;
  E.S[it.slot] = st;
  if (blockIdx.y != 0 || !io.first) return;
  // the iteration counter restarts with every closed-world solve (serving keeps counting and relies on
  // per-problem caps; its limit is set out of reach)
  *E.iter = 0u;
  for (int k = 0; k < 4; ++k) E.err[k] = 0;
  for (int k = 0; k < 3; ++k) E.gbar[k] = 0ull;
  *E.ticket = 0u;
  // the mirror of the IF node's value as the closed-world graph sets it at its launch
  *taken = 0u;
  *launches = 0ull;
}

__global__ void __launch_bounds__(256) k_finish(const __grid_constant__ EngineDev E, const __grid_constant__ IoBatch io,
                                                const unsigned long long* launches, ProbState* states, IoResult* result) {
  const IoItem& it = io.item[blockIdx.y];
  const ProblemDev& P = E.P[it.slot];
  const ProbState& st = E.S[it.slot];
  if (*E.err == 0 && st.status != HN_ERR_ARG) {
    // a zero right-hand side has the solution zero, whatever the first iterate
    const bool zero = st.status == HN_OK && st.bnorm == 0.0;
    double* x = const_cast<double*>(it.x);
    if (zero) move(P.x64, x, nullptr, nodes(P.L));
    else if (x) move(x, nullptr, P.x64, nodes(P.L));
  }
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  states[it.slot] = st;
  if (blockIdx.y != 0 || !io.first) return;
  result->iterations = *E.iter;
  result->launches = *launches;
  for (int k = 0; k < 4; ++k) result->err[k] = E.err[k];
}

// blocks a problem: eight rounds of a block's 2,048 doubles, and no more than fills the chip once
unsigned io_blocks(const IoBatch& io, long long most) {
  const long long fill = std::max(1, 8 * sm_count() / std::max(1, io.n));
  return (unsigned)std::min(std::max<long long>(1, most / 2048), fill);
}

}  // namespace

cudaError_t launch_begin(const EngineDev& E, const IoBatch& io, long long most, unsigned* taken, unsigned long long* launches,
                         cudaStream_t s) {
  k_begin<<<dim3(io_blocks(io, most), (unsigned)io.n), 256, 0, s>>>(E, io, taken, launches);
  return cudaGetLastError();
}

cudaError_t launch_finish(const EngineDev& E, const IoBatch& io, long long most, const unsigned long long* launches,
                          ProbState* states, IoResult* result, cudaStream_t s) {
  k_finish<<<dim3(io_blocks(io, most), (unsigned)io.n), 256, 0, s>>>(E, io, launches, states, result);
  return cudaGetLastError();
}

}  // namespace hn
