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

constexpr int kThreads = 128;          // rows of a group, and threads of a block
constexpr int kChunk = 16 * kThreads;  // entries staged at a time
constexpr int kThreadRow = 40;         // the most entries that one thread adds up
constexpr int kRowLanes = 8;           // lanes of a row of a matrix known to be wide: from
constexpr int kWideEntries = 48;       // so many entries a row on average and
constexpr int kWideRows = 20000;       // so many rows on (with fewer the groups are divided over more blocks)
constexpr int kMaxSplit = 8;           // blocks of a group of wide rows: at least 16 rows each
constexpr int kBlocks = 4 * 152;       // no more blocks than this for the sake of the split
constexpr int kMaxDevices = 64;

// One fused leapfrog step on CSR:
//   out = 2 x - prev - tau2m .* (S x);  acc = acc + alpha[step+1] * out
// first: prev = x and acc = alpha[0] * x + alpha[1] * out; last: out is not stored.
//
// The FP64 pipe and latency bound it. A group's entries lie side by side in memory, so a block copies
// the values and columns of its rows to shared memory first, coalesced, a chunk at a time; what a launch
// reads of them does not wait for the step before (programmatic launch). An entry's place in shared
// memory is i + i / 16, so that rows of even length meet different banks too. How a chunk is added up
// depends on the group's rows alone:
//
// Rows of up to kThreadRow entries (or a group of one chunk): a row per thread, in four sums: 21 FP64
// operations for 15 entries. (Eight lanes a row leave most lanes of every FP64 instruction idle and add
// their sums with three more: 64 per row.) A longer row among them is added up by its whole warp.
//
// Wider rows: a chunk holds rows for a few threads only, so as many threads share a row as a chunk's rows
// leave (a power of two up to 32: they lie in one warp), each with a part of its entries, and the group's rows
// are divided over gridDim.y blocks where the groups alone do not occupy the SMs. The other blocks of a group of
// the first kind leave at once; they come last in the grid and take the slots that are free.
//
// Us a step, eight lanes a row for all rows -> this: 103,823 rows of 15 entries 20.1 -> 10.7; 50 thousand rows of
// 27 entries 14.6 -> 8.8, of 41 entries 14.6 -> 13.0; 5 thousand rows of 125 entries 10.5 -> 5.7; 7 entries, but for
// 10 rows of 25 thousand, 988 -> 321.
__device__ __forceinline__ int place(int i) { return i + (i >> 4); }

// The sum over the staged entries [k, ke) of a thread, in four sums (folded to s[0] + s[2] and s[1] + s[3] by the
// caller); ranges too long for one thread are added up by the warp. All threads of a warp come here.
__device__ __forceinline__ void add_range(double (&s)[4], int k, int ke, const double* s_val, const int32_t* s_col,
                                          const double* x) {
  for (unsigned rest = __ballot_sync(0xffffffffu, ke - k > kThreadRow); rest; rest &= rest - 1) {
    const int lane = threadIdx.x % 32, of = __ffs(rest) - 1;
    const int a = __shfl_sync(0xffffffffu, k, of), b = __shfl_sync(0xffffffffu, ke, of);
    double part = 0.0;
#pragma unroll 4
    for (int i = a + lane; i < b; i += 32) part = fma(s_val[place(i)], x[s_col[place(i)]], part);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == of) {
      s[0] += part;
      k = ke;
    }
  }
  for (; k + 4 <= ke; k += 4) {
    double v[4], y[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[j] = s_val[place(k + j)];
      y[j] = x[s_col[place(k + j)]];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = fma(v[j], y[j], s[j]);
  }
#pragma unroll
  for (int j = 0; j < 3; ++j)
    if (k + j < ke) s[j] = fma(s_val[place(k + j)], x[s_col[place(k + j)]], s[j]);
}

// AHEAD: entries of a thread whose copies are under way together. Eight where the rows are short and the grid has
// no blocks that wait for a place, four elsewhere (us a step, four / eight: 15 entries a row, 29,791 rows 3.72 / 3.67,
// 64 thousand 6.29 / 6.10, 405 thousand 34.8 / 36.4; 27 entries, 27 thousand rows 7.5 / 7.9).
template <bool FIRST, bool LAST, int AHEAD>
__global__ void __launch_bounds__(kThreads, 8) k_step_csr_f64(int64_t n, const int64_t* __restrict__ row_ptr,
                                                              const int32_t* __restrict__ col,
                                                              const double* __restrict__ val,
                                                              const double* __restrict__ tau2m, const double* x,
                                                              const double* prev, double* out, double* acc,
                                                              const double* __restrict__ alpha, int step) {
  __shared__ double s_val[kChunk + kChunk / 16];
  __shared__ int32_t s_col[kChunk + kChunk / 16];
  const int tid = threadIdx.x;
  const int64_t row0 = static_cast<int64_t>(blockIdx.x) * kThreads, row = row0 + tid;
  const int64_t begin = row_ptr[row0], end = row_ptr[row0 + kThreads < n ? row0 + kThreads : n];
  const bool chunks = end - begin > kChunk;
  if (blockIdx.y > 0 && !chunks) return;
  const int64_t first = row < n ? row_ptr[row] : end, stop = row < n ? row_ptr[row + 1] : end;
  auto stage = [&](int64_t c0, int count) {
#pragma unroll AHEAD
    for (int i = tid; i < count; i += kThreads) {
      s_val[place(i)] = __ldcs(val + c0 + i);
      s_col[place(i)] = __ldcs(col + c0 + i);
    }
  };
  // the next step may start (and read its matrix) once the one before this has finished
  auto after_last_step = [&]() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  };
  auto finish = [&](int64_t r, double sum) {
    const double xi = x[r];
    const double pi = FIRST ? xi : prev[r];
    const double un = fma(-tau2m[r], sum, 2.0 * xi - pi);
    if (!LAST) out[r] = un;
    acc[r] = fma(alpha[step + 1], un, FIRST ? alpha[0] * xi : acc[r]);
  };

  const bool wide = chunks && end - begin < (int64_t(1) << 31);  // for 32-bit places (else: rows that repeat columns)
  if (wide && __syncthreads_or(gridDim.y == kMaxSplit || stop - first > kThreadRow)) {
    __shared__ int32_t s_first[kThreads];  // of the group's rows, counted from its first entry
    const int rows = kThreads / static_cast<int>(gridDim.y), r0 = static_cast<int>(blockIdx.y) * rows;
    const int32_t size = static_cast<int32_t>(end - begin), mine = static_cast<int32_t>(first - begin),
                  after = static_cast<int32_t>(stop - begin);
    s_first[tid] = mine;
    double* const s_sum = s_val + 16;  // of row r at 17 r: the places that place() skips
    s_sum[17 * tid] = 0.0;
    __syncthreads();
    auto first_of = [&](int r) { return r < kThreads ? s_first[r] : size; };
    const int32_t from = first_of(r0), to = first_of(r0 + rows);
    const bool own = tid >= r0 && tid < r0 + rows;  // this thread's row is one of the block's
    for (int32_t c0 = from;;) {  // once for a block without entries, else until they are used up
      const int count = min(to - c0, kChunk), c1 = c0 + count;
      stage(begin + c0, count);
      if (c0 == from) after_last_step();
      const int done = __syncthreads_count(own && after <= c0);  // rows that end before this chunk,
      const int m = __syncthreads_count(own && mine < c1) - done;  // and rows that lie in it
      // threads of a row: a power of two, so that they lie in one warp
      int each = 1;
      while (each < 32 && 2 * each * m <= kThreads) each *= 2;
      const int r = r0 + done + tid / each, part = tid % each;
      double sum[4] = {0.0, 0.0, 0.0, 0.0};
      int k = 0, ke = 0;
      if (tid / each < m) {
        const int lo = max(s_first[r] - c0, 0), w = min(first_of(r + 1) - c0, count) - lo;
        k = lo + w * part / each;
        ke = lo + w * (part + 1) / each;
      }
      add_range(sum, k, ke, s_val, s_col, x);
      double total = (sum[0] + sum[2]) + (sum[1] + sum[3]);
      for (int o = each / 2; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
      if (tid / each < m && part == 0) s_sum[17 * r] += total;
      __syncthreads();
      if (c1 >= to) break;
      c0 = c1;
    }
    if (own && row < n) finish(row, s_sum[17 * tid]);
    return;
  }
  if (blockIdx.y > 0) return;

  double sum[4] = {0.0, 0.0, 0.0, 0.0};
  for (int64_t c0 = begin; c0 < end || c0 == begin; c0 += kChunk) {
    const int count = static_cast<int>(end - c0 < kChunk ? end - c0 : kChunk);
    if (c0 != begin) __syncthreads();
    stage(c0, count);
    if (c0 == begin) after_last_step();
    __syncthreads();
    const int64_t to = stop - c0;
    add_range(sum, static_cast<int>((first > c0 ? first : c0) - c0), static_cast<int>(to < count ? to : count), s_val,
              s_col, x);
  }
  if (row < n) finish(row, (sum[0] + sum[2]) + (sum[1] + sum[3]));
}

// The same step for a matrix of wide rows, where the caller says that it is one: eight lanes a row straight from
// memory, with all of L1 for the gathers and twice the threads that shared memory leaves above (81 entries a row,
// us a step, shared rows above / this: 50 thousand rows 27.0 / 15.6, 150 thousand 60.2 / 46.6; 121 entries, 300
// thousand rows 179.6 / 112.0). The lanes' loop is not unrolled: four entries of a lane at a time lie in other lines than
// the ones at hand, which its neighbours still read (112.0 us against 157.4).
template <bool FIRST, bool LAST>
__global__ void __launch_bounds__(256) k_step_csr_wide_f64(int64_t n, const int64_t* __restrict__ row_ptr,
                                                           const int32_t* __restrict__ col,
                                                           const double* __restrict__ val,
                                                           const double* __restrict__ tau2m, const double* x,
                                                           const double* prev, double* out, double* acc,
                                                           const double* __restrict__ alpha, int step) {
  const int lane = threadIdx.x % kRowLanes;
  const int64_t row = (static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x) / kRowLanes;
  const int64_t first = row < n ? row_ptr[row] : 0, stop = row < n ? row_ptr[row + 1] : 0;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  double sum = 0.0;
#pragma unroll 1
  for (int64_t p = first + lane; p < stop; p += kRowLanes) sum = fma(val[p], x[col[p]], sum);
#pragma unroll
  for (int o = kRowLanes / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o, kRowLanes);
  if (lane == 0 && row < n) {
    const double xi = x[row];
    const double pi = FIRST ? xi : prev[row];
    const double un = fma(-tau2m[row], sum, 2.0 * xi - pi);
    if (!LAST) out[row] = un;
    acc[row] = fma(alpha[step + 1], un, FIRST ? alpha[0] * xi : acc[row]);
  }
}

enum Kernel { kShort, kStaged, kWide };  // of a call's steps

template <bool FIRST, bool LAST>
auto kernel_of(Kernel k) {
  return k == kWide ? k_step_csr_wide_f64<FIRST, LAST>
                    : k == kShort ? k_step_csr_f64<FIRST, LAST, 8> : k_step_csr_f64<FIRST, LAST, 4>;
}

template <bool FIRST, bool LAST>
cudaError_t launch_step(Kernel k, unsigned split, int64_t n, cudaStream_t st, const int64_t* row_ptr,
                        const int32_t* col, const double* val, const double* tau2m, const double* x,
                        const double* prev, double* out, double* acc, const double* alpha, int step) {
  const unsigned groups = static_cast<unsigned>((n + kThreads - 1) / kThreads);
  cudaLaunchConfig_t c{};
  c.gridDim = k == kWide ? dim3(static_cast<unsigned>((n * kRowLanes + 255) / 256)) : dim3(groups, split);
  c.blockDim = dim3(k == kWide ? 256 : kThreads);
  c.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = FIRST ? 0 : 1;  // the first step follows the caller's own work
  return cudaLaunchKernelEx(&c, kernel_of<FIRST, LAST>(k), n, row_ptr, col, val, tau2m, x, prev, out, acc, alpha, step);
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
  return kes_filter_apply_noalloc_sized(n, -1, row_ptr, col, val, tau2m, alpha, L, r_in, r_out, stream);
}

extern "C" kes_status kes_filter_apply_noalloc_sized(int64_t n, int64_t nnz, const int64_t* row_ptr,
                                                     const int32_t* col, const double* val, const double* tau2m,
                                                     const double* alpha, int32_t L, const double* r_in, double* r_out,
                                                     void* stream) {
  if (n < 1 || n > KES_NOALLOC_MAX_N || L < 1 || !row_ptr || !col || !val || !tau2m || !alpha || !r_in || !r_out)
    return KES_ERR_ARG;
  double* state = nullptr;
  if (state_for_current_device(&state) != cudaSuccess) {
    cudaGetLastError();
    return KES_ERR_CUDA;
  }
  double* U[2] = {state, state + KES_NOALLOC_MAX_N};
  const int64_t groups = (n + kThreads - 1) / kThreads;
  const bool narrow = nnz >= 0 && nnz <= 16 * n;  // a row on average fills no more than its share of a chunk
  const Kernel kernel = n >= kWideRows && nnz / n >= kWideEntries ? kWide
                        : narrow && groups <= 2 * kBlocks         ? kShort
                                                                  : kStaged;
  // blocks of a group: not where the rows are known to be short on average (the blocks that leave at once cost a small
  // matrix 4% of a step)
  unsigned split = narrow ? 1 : kMaxSplit;
  while (split > 1 && groups * split > kBlocks) split /= 2;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  for (int s = 0; s < L; ++s) {
    const bool first = s == 0, last = s == L - 1;
    const double* x = s == 0 ? r_in : U[(s - 1) & 1];
    const double* prev = s <= 1 ? r_in : U[s & 1];
    double* out = U[s & 1];
    const auto go = first ? (last ? launch_step<true, true> : launch_step<true, false>)
                          : (last ? launch_step<false, true> : launch_step<false, false>);
    if (go(kernel, split, n, st, row_ptr, col, val, tau2m, x, prev, out, r_out, alpha, s) != cudaSuccess) {
      cudaGetLastError();
      return KES_ERR_CUDA;
    }
  }
  return cudaGetLastError() == cudaSuccess ? KES_OK : KES_ERR_CUDA;
}
