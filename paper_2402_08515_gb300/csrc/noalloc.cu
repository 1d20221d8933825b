// Allocation-free variant of the FP64 filter application.
//
// Some callers cannot call cudaMalloc at all: a host program that reserves
// every byte of device memory it may use when it starts and forbids any later
// allocation (a long-running service with a fixed memory budget, or a plugin
// whose host owns the device heap), so that a mid-run allocation can neither
// fail nor fragment memory. kes_create allocates its own state, so those
// callers get this entry point instead: they pass every input and the output
// in device memory they already own, and the two leapfrog state vectors live
// in the fixed array below, a file-scope __device__ array of this module.
//
// The array takes 2 * KES_NOALLOC_MAX_N doubles (16 MiB) on every device where
// this module is loaded, until the process exits. Under CUDA's default lazy
// module loading the module (and so the array) is loaded on a device by the
// first call there, when the set-up looks up the array's address: a caller that
// reserves all of its device memory must make one call first (or run with
// CUDA_MODULE_LOADING=EAGER, which loads every module with the context).
// Every call shares the array and it keeps the previous call's contents; calls
// whose GPU work overlaps (two streams, two host threads) race on it and must
// be serialised by the caller. Nothing has to start at zero: each call writes
// every state entry it reads.
#include <cuda_runtime.h>

#include <mutex>

#include "kes_internal.h"

static __device__ __align__(256) double kes_noalloc_state[2 * KES_NOALLOC_MAX_N];

namespace {

constexpr int kThreads = 128;          // rows of a block, one per thread
constexpr int kChunk = 16 * kThreads;  // entries staged at a time
constexpr int kMaxDevices = 64;

// One fused leapfrog step on CSR:
//   out = 2 x - prev - tau2m .* (S x);  acc = acc + alpha[step+1] * out
// first: prev = x and acc = alpha[0] * x + alpha[1] * out; last: out is not stored.
//
// The FP64 pipe and latency bound it. A row belongs to one thread, which adds its entries up in
// four sums: 21 FP64 operations for 15 entries. (Eight lanes a row, as before, leave most lanes of
// every FP64 instruction idle and add their sums with three more: 64 per row.) Its entries lie
// side by side in memory, so the block copies the values and columns of its rows to shared
// memory first, coalesced, a chunk at a time; what a launch reads of them does not wait for the
// step before (programmatic launch). An entry's place in shared memory is i + i / 16, so that
// rows of even length meet different banks too. 103,823 rows: 20.1 -> 10.7 us a step.
__device__ __forceinline__ int place(int i) { return i + (i >> 4); }

template <bool FIRST, bool LAST>
__global__ void __launch_bounds__(kThreads) k_step_csr_f64(int64_t n, const int64_t* __restrict__ row_ptr,
                                                           const int32_t* __restrict__ col,
                                                           const double* __restrict__ val,
                                                           const double* __restrict__ tau2m, const double* x,
                                                           const double* prev, double* out, double* acc,
                                                           const double* __restrict__ alpha, int step) {
  __shared__ double s_val[kChunk + kChunk / 16];
  __shared__ int32_t s_col[kChunk + kChunk / 16];
  const int64_t row0 = static_cast<int64_t>(blockIdx.x) * kThreads, row = row0 + threadIdx.x;
  const int64_t end = row_ptr[row0 + kThreads < n ? row0 + kThreads : n];
  const int64_t first = row < n ? row_ptr[row] : end, stop = row < n ? row_ptr[row + 1] : end;
  double sum[4] = {0.0, 0.0, 0.0, 0.0};
  for (int64_t c0 = row_ptr[row0], begin = c0; c0 < end || c0 == begin; c0 += kChunk) {
    const int count = static_cast<int>(end - c0 < kChunk ? end - c0 : kChunk);
    if (c0 != begin) __syncthreads();
#pragma unroll 8
    for (int i = threadIdx.x; i < count; i += kThreads) {
      s_val[place(i)] = __ldcs(val + c0 + i);
      s_col[place(i)] = __ldcs(col + c0 + i);
    }
    if (c0 == begin) {
      // the next step may start (and read its matrix) once the one before this has finished
      asm volatile("griddepcontrol.wait;" ::: "memory");
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    __syncthreads();
    int k = static_cast<int>((first > c0 ? first : c0) - c0);
    const int64_t to = stop - c0;
    const int ke = static_cast<int>(to < count ? to : count);
    for (; k + 4 <= ke; k += 4) {
      double v[4], y[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        v[j] = s_val[place(k + j)];
        y[j] = x[s_col[place(k + j)]];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) sum[j] = fma(v[j], y[j], sum[j]);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j)
      if (k + j < ke) sum[j] = fma(s_val[place(k + j)], x[s_col[place(k + j)]], sum[j]);
  }
  if (row < n) {
    const double xi = x[row];
    const double pi = FIRST ? xi : prev[row];
    const double un = fma(-tau2m[row], (sum[0] + sum[2]) + (sum[1] + sum[3]), 2.0 * xi - pi);
    if (!LAST) out[row] = un;
    acc[row] = fma(alpha[step + 1], un, FIRST ? alpha[0] * xi : acc[row]);
  }
}

template <bool FIRST, bool LAST>
cudaError_t launch_step(int64_t n, cudaStream_t st, const int64_t* row_ptr, const int32_t* col, const double* val,
                        const double* tau2m, const double* x, const double* prev, double* out, double* acc,
                        const double* alpha, int step) {
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(static_cast<unsigned>((n + kThreads - 1) / kThreads));
  c.blockDim = dim3(kThreads);
  c.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = FIRST ? 0 : 1;  // the first step follows the caller's own work
  return cudaLaunchKernelEx(&c, k_step_csr_f64<FIRST, LAST>, n, row_ptr, col, val, tau2m, x, prev, out, acc, alpha,
                            step);
}

std::mutex g_setup_mu;
double* g_state[kMaxDevices] = {};

// Device address of the scratch array on the current device, looked up once per device.
cudaError_t state_for_current_device(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_setup_mu);
  if (!g_state[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, kes_noalloc_state);
    if (e != cudaSuccess) return e;
    g_state[dev] = static_cast<double*>(p);
  }
  *out = g_state[dev];
  return cudaSuccess;
}

}  // namespace

extern "C" kes_status kes_filter_apply_noalloc(int64_t n, const int64_t* row_ptr, const int32_t* col,
                                               const double* val, const double* tau2m, const double* alpha,
                                               int32_t L, const double* r_in, double* r_out, void* stream) {
  if (n < 1 || n > KES_NOALLOC_MAX_N || L < 1 || !row_ptr || !col || !val || !tau2m || !alpha || !r_in || !r_out)
    return KES_ERR_ARG;
  double* state = nullptr;
  if (state_for_current_device(&state) != cudaSuccess) {
    cudaGetLastError();
    return KES_ERR_CUDA;
  }
  double* U[2] = {state, state + KES_NOALLOC_MAX_N};
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  for (int s = 0; s < L; ++s) {
    const bool first = s == 0, last = s == L - 1;
    const double* x = s == 0 ? r_in : U[(s - 1) & 1];
    const double* prev = s <= 1 ? r_in : U[s & 1];
    double* out = U[s & 1];
    const auto go = first ? (last ? launch_step<true, true> : launch_step<true, false>)
                          : (last ? launch_step<false, true> : launch_step<false, false>);
    if (go(n, st, row_ptr, col, val, tau2m, x, prev, out, r_out, alpha, s) != cudaSuccess) {
      cudaGetLastError();
      return KES_ERR_CUDA;
    }
  }
  return cudaGetLastError() == cudaSuccess ? KES_OK : KES_ERR_CUDA;
}
