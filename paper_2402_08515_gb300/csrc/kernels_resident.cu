// A whole filter application in one kernel, for matrices that fit the shared memory of one
// cluster of 16 blocks (Sec. 2.3, eq. 2stepmethod and eq. disc_filtercoeff).
//
// What bounds it: a step of a small matrix is a microsecond of work or less behind about two
// of launching and of reading the last step's state back from L2. Here a cluster keeps the
// matrix, u_n, u_{n-1} and the accumulators in the shared memory of its blocks for all L steps.
// A block owns a run of slices and holds u_n on the range of rows that its columns lie in; a
// warp that has a slice's u_{n+1} writes it to its own block and into the ranges of the other
// blocks that hold these rows (st.shared::cluster), and one cluster barrier ends the step, its
// wait behind the accumulators' update. The columns of a block are independent: each has a
// cluster of its own. No block waits for another except in the hardware's cluster barrier.
//
// Microseconds a step, chain of launches -> resident: 64^2 cells (3,969 rows) FP64 2.4 -> 1.02, 8
// columns 5.0 -> 1.5; FP32 2.3 -> 0.74, 8 columns 2.5 -> 0.82; 24^3 cells FP32 2.5 -> 1.43. (With
// the weights read from global memory 1.45 instead of 1.02: every step's came from L2.)
//
// Row sums, seeds and weighted terms are formed like those of the other step kernels, one FMA
// chain per row in entry order and one term per step in index order: the same bits.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "kes_internal.h"

namespace kes {
namespace {

constexpr int kResidentSmem = 220 * 1024;

struct ResidentArgs {
  SellDev A;
  const int2* range;    // per block: first row its columns lie in, and the row after the last
  const double* tau2m;
  const double* r;      // n_pad x NB row-major
  double* out;          // F x (n_pad x NB)
  int64_t out_stride;
  const double* alpha;  // [mesh][F][L + 1]
  const float* ahi;
  const float* alo;
  int blocks, slices, NB, F, Lp1, steps, cpt;  // slices: owned by each block but the last ones
  int off_val, off_idx, off_acc, off_rec, off_alpha;
  int meshes;
  int xrows;            // rows of the longest range
  int* flag;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t remote_addr(uint32_t addr, int block) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(block));
  return r;
}
__device__ __forceinline__ void st_remote(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ double neg(double x) {  // -x without the FP64 pipe
  asm("{\n\t.reg .b32 lo, hi;\n\tmov.b64 {lo, hi}, %0;\n\txor.b32 hi, hi, 0x80000000;\n\tmov.b64 %0, {lo, hi};\n\t}"
      : "+d"(x));
  return x;
}
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& t) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  const float ap = __fsub_rn(s, bp);
  t = __fadd_rn(__fsub_rn(a, ap), __fsub_rn(b, bp));
}

template <typename T, bool FOLD>
__global__ void __launch_bounds__(1024, 1) k_resident(const __grid_constant__ ResidentArgs a) {
  constexpr bool kF64 = std::is_same<T, double>::value;
  extern __shared__ __align__(128) unsigned char smem[];
  T* xb = reinterpret_cast<T*>(smem);                                 // [2][xrows]
  T* val = reinterpret_cast<T*>(smem + a.off_val);                    // per slice [w][32]
  uint32_t* idx = reinterpret_cast<uint32_t*>(smem + a.off_idx);      // per slice [(w + 1) / 2][32], two places each
  T* acc = reinterpret_cast<T*>(smem + a.off_acc);                    // [tables][FP32: s, c][slices][32]
  int4* rec = reinterpret_cast<int4*>(smem + a.off_rec);              // per slice {first value / 32, w, mesh, blocks}
  // the weights of this column's tables, [mesh][table][steps + 1] (FP32: hi, lo): a barrier's
  // acquire empties L1, so anything read from global memory in a step would come from L2
  double* weights = reinterpret_cast<double*>(smem + a.off_alpha);
  __shared__ int2 ranges[kResidentBlocks];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int rank = blockIdx.x % a.blocks, col = blockIdx.x / a.blocks;
  const int64_t s0 = static_cast<int64_t>(rank) * a.slices;
  const int own = static_cast<int>(max(int64_t(0), min(static_cast<int64_t>(a.slices), a.A.n_slices - s0)));
  const int nacc = a.cpt ? 1 : a.F;
  const int table0 = a.cpt ? min(col / a.cpt, a.F - 1) : 0;
  const int rows = a.slices * kSliceC;                                // rows of an accumulator
  const int2 mine = __ldg(a.range + rank);
  const int64_t beg0 = own > 0 ? a.A.slice_ptr[s0] : 0;
  const int n1 = a.steps + 1;
  if (threadIdx.x < a.blocks) ranges[threadIdx.x] = __ldg(a.range + threadIdx.x);
  for (int i = threadIdx.x; i < a.meshes * nacc * n1; i += blockDim.x) {
    const int m = i / (nacc * n1), f = i / n1 % nacc;
    const int64_t ai = (static_cast<int64_t>(m) * a.F + (a.cpt ? table0 : f)) * a.Lp1 + i % n1;
    if constexpr (kF64) weights[i] = a.alpha[ai];
    else reinterpret_cast<float2*>(weights)[i] = make_float2(a.ahi[ai], a.alo[ai]);
  }

  for (int i = mine.x + threadIdx.x; i < mine.y; i += blockDim.x)
    xb[i - mine.x] = static_cast<T>(a.r[static_cast<int64_t>(i) * a.NB + col]);
  for (int s = warp; s < own; s += warps) {
    const int64_t beg = a.A.slice_ptr[s0 + s];
    const int w = static_cast<int>((a.A.slice_ptr[s0 + s + 1] - beg) >> 5);
    const int v0 = static_cast<int>((beg - beg0) >> 5);
    const int64_t row = (s0 + s) * kSliceC + lane;
    const int mesh = a.A.slice_mesh ? a.A.slice_mesh[s0 + s] : 0;
    if (lane == 0) {
      int blocks = 0;
      for (int c = 0; c < a.blocks; ++c) {
        const int2 q = __ldg(a.range + c);
        if (c != rank && q.x < row + kSliceC && q.y > row) blocks |= 1 << c;
      }
      rec[s] = make_int4(v0, w, mesh, blocks);
    }
    // the step values A = -tau^2 M^{-1} S (FOLD: A + 2I) as k_scale_tiles forms them
    const double t = -a.tau2m[row];
    bool diag_done = false;
    uint32_t pair = 0;
    for (int k = 0; k < w; ++k) {
      const int64_t e = beg + static_cast<int64_t>(k) * kSliceC + lane;
      double v = t * a.A.val64[e];
      const int c = a.A.col[e];
      if (FOLD && !diag_done && c == row) {
        v += 2.0;
        diag_done = true;
      }
      val[(v0 + k) * kSliceC + lane] = static_cast<T>(v);
      const uint32_t place = static_cast<uint32_t>(c - mine.x);
      if (k & 1) pair |= place << 16;
      else pair = place;
      if ((k & 1) || k == w - 1) idx[((v0 + s) / 2 + s + (k >> 1)) * kSliceC + lane] = pair;
    }
    const double r0 = a.r[row * a.NB + col];
    for (int f = 0; f < nacc; ++f) {
      const double first = a.alpha[(static_cast<int64_t>(mesh) * a.F + (a.cpt ? table0 : f)) * a.Lp1] * r0;
      if constexpr (kF64) {
        acc[f * rows + s * kSliceC + lane] = first;
      } else {
        const float h = static_cast<float>(first);
        acc[2 * f * rows + s * kSliceC + lane] = h;
        acc[(2 * f + 1) * rows + s * kSliceC + lane] = static_cast<float>(first - static_cast<double>(h));
      }
    }
  }
  __syncthreads();
  cluster_arrive();  // no block writes into another's range before that one has its own start there
  cluster_wait();

  for (int step = 0; step < a.steps; ++step) {
    const T* x = xb + (step & 1) * a.xrows;
    T* next = xb + ((step + 1) & 1) * a.xrows;
    const bool last = step == a.steps - 1;
    for (int s = warp; s < own; s += warps) {
      const int4 q = rec[s];
      const int row = static_cast<int>(s0 + s) * kSliceC + lane;
      const int at = row - mine.x;
      const T xi = x[at];
      const T pi = step == 0 ? xi : next[at];
      T un;
      if constexpr (kF64) un = FOLD ? neg(pi) : 2.0 * xi - pi;
      else un = __fsub_rn(__fmul_rn(2.0f, xi), pi);
      const T* v = val + q.x * kSliceC + lane;
      const uint32_t* p = idx + ((q.x + s) / 2 + s) * kSliceC + lane;
      int k = 0;
#pragma unroll 2
      for (; k + 4 <= q.y; k += 4) {
        const uint32_t c0 = p[(k >> 1) * kSliceC], c1 = p[((k >> 1) + 1) * kSliceC];
        const T v0 = v[k * kSliceC], v1 = v[(k + 1) * kSliceC], v2 = v[(k + 2) * kSliceC], v3 = v[(k + 3) * kSliceC];
        const T x0 = x[c0 & 0xffff], x1 = x[c0 >> 16], x2 = x[c1 & 0xffff], x3 = x[c1 >> 16];
        un = fma(v3, x3, fma(v2, x2, fma(v1, x1, fma(v0, x0, un))));
      }
      if (q.y & 2) {
        const uint32_t c0 = p[(k >> 1) * kSliceC];
        const T v0 = v[k * kSliceC], v1 = v[(k + 1) * kSliceC];
        un = fma(v1, x[c0 >> 16], fma(v0, x[c0 & 0xffff], un));
        k += 2;
      }
      if (q.y & 1) un = fma(v[k * kSliceC], x[p[(k >> 1) * kSliceC] & 0xffff], un);
      next[at] = un;
      if (!last) {
        for (unsigned b = q.w; b != 0; b &= b - 1) {
          const int c = __ffs(b) - 1;
          const int2 o = ranges[c];
          if (row >= o.x && row < o.y) st_remote(remote_addr(smem_addr(next + (row - o.x)), c), un);
        }
      }
    }
    __syncwarp();
    cluster_arrive();
    for (int s = warp; s < own; s += warps) {  // while the others arrive: the weighted term
      const int4 q = rec[s];
      const T un = next[static_cast<int>(s0 + s) * kSliceC + lane - mine.x];  // this thread's own
      for (int f = 0; f < nacc; ++f) {
        const int ai = (q.z * nacc + f) * n1 + step + 1;
        if constexpr (kF64) {
          T* d = acc + f * rows + s * kSliceC + lane;
          *d = fma(weights[ai], un, *d);
        } else {
          float* ds = acc + 2 * f * rows + s * kSliceC + lane;
          float* dc = ds + rows;
          const float2 hl = reinterpret_cast<const float2*>(weights)[ai];
          const float h = hl.x, l = hl.y;
          // alpha u = p + pe, p = fl(hi u), pe = (hi u - p) + lo u
          const float pr = __fmul_rn(h, un);
          const float pe = fmaf(l, un, fmaf(h, un, -pr));
          float sn, e;
          two_sum(*ds, pr, sn, e);
          *dc = __fadd_rn(*dc, __fadd_rn(e, pe));
          *ds = sn;
        }
      }
    }
    __syncwarp();
    cluster_wait();
  }

  bool bad = false;
  for (int s = warp; s < own; s += warps) {
    const int64_t row = (s0 + s) * kSliceC + lane;
    for (int f = 0; f < nacc; ++f) {
      double v;
      if constexpr (kF64) {
        v = acc[f * rows + s * kSliceC + lane];
      } else {
        const float* ds = acc + 2 * f * rows + s * kSliceC + lane;
        v = static_cast<double>(ds[0]) + static_cast<double>(ds[rows]);
      }
      bad |= !isfinite(v);
      a.out[f * a.out_stride + row * a.NB + col] = v;
    }
  }
  if (bad) atomicOr(a.flag, 1);
}

struct ResidentFit {
  int off_val, off_idx, off_acc, off_rec, off_alpha, bytes;
};
ResidentFit resident_fit(const ResidentPlan& p, int size, int tables, int meshes, int steps) {
  auto up = [](int64_t v) { return (v + 127) & ~int64_t(127); };
  int64_t at = up(int64_t(2) * p.xrows * size);
  ResidentFit f;
  f.off_val = static_cast<int>(at);
  at += up(int64_t(p.entries) * size);
  f.off_idx = static_cast<int>(at);
  at += up(int64_t(p.entries) * 2 + int64_t(p.slices) * 256);
  f.off_acc = static_cast<int>(at);
  at += up(int64_t(tables) * 8 * p.slices * kSliceC);
  f.off_rec = static_cast<int>(at);
  at += up(int64_t(p.slices) * 16);
  f.off_alpha = static_cast<int>(std::min<int64_t>(at, kResidentSmem));
  at += up(int64_t(tables) * meshes * (steps + 1) * 8);
  f.bytes = at > kResidentSmem ? kResidentSmem + 1 : static_cast<int>(at);
  return f;
}

template <typename T, bool FOLD>
void launch_one(const ResidentArgs& a, int bytes, int warps, cudaStream_t st) {
  cudaFuncSetAttribute(k_resident<T, FOLD>, cudaFuncAttributeMaxDynamicSharedMemorySize, kResidentSmem);
  cudaFuncSetAttribute(k_resident<T, FOLD>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(a.blocks * a.NB);
  c.blockDim = dim3(32 * warps);
  c.dynamicSmemBytes = bytes;
  c.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = a.blocks;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, k_resident<T, FOLD>, a);
}

}  // namespace

// Whether the device can hold a cluster of that many blocks with all of that shared memory.
bool resident_available() {
  int n = 0;
  bool ok = true;
  auto ask = [&](auto kernel) {
    ok = ok && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kResidentSmem) == cudaSuccess &&
         cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(kResidentBlocks);
    c.blockDim = dim3(1024);
    c.dynamicSmemBytes = kResidentSmem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kResidentBlocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    c.attrs = at;
    c.numAttrs = 1;
    ok = ok && cudaOccupancyMaxActiveClusters(&n, kernel, &c) == cudaSuccess && n > 0;
  };
  ask(k_resident<float, false>);
  ask(k_resident<double, true>);
  ask(k_resident<double, false>);
  if (!ok) cudaGetLastError();
  return ok;
}

bool resident_fits(const ResidentPlan& p, bool fp64, int tables, int meshes, int steps) {
  return p.slices > 0 && resident_fit(p, fp64 ? 8 : 4, tables, meshes, steps).bytes <= kResidentSmem;
}

void launch_resident(const SellDev& A, const ResidentPlan& p, const int2* range, bool fp64, bool fold2,
                     cudaStream_t st, int NB, const double* tau2m, const double* r, double* out, int F,
                     const double* alpha, const float* ahi, const float* alo, int L, int steps, int cpt, int meshes, int* flag) {
  const ResidentFit f = resident_fit(p, fp64 ? 8 : 4, cpt ? 1 : F, meshes, steps);
  ResidentArgs a{};
  a.A = A;
  a.range = range;
  a.tau2m = tau2m;
  a.r = r;
  a.out = out;
  a.out_stride = A.n_pad * NB;
  a.alpha = alpha;
  a.ahi = ahi;
  a.alo = alo;
  a.blocks = p.blocks;
  a.slices = p.slices;
  a.NB = NB;
  a.F = F;
  a.Lp1 = L + 1;
  a.steps = steps;
  a.cpt = cpt;
  a.off_val = f.off_val;
  a.off_idx = f.off_idx;
  a.off_acc = f.off_acc;
  a.off_rec = f.off_rec;
  a.off_alpha = f.off_alpha;
  a.meshes = meshes;
  a.xrows = p.xrows;
  a.flag = flag;
  const int warps = std::max(4, std::min(32, p.slices));
  if (!fp64) launch_one<float, false>(a, f.bytes, warps, st);
  else if (fold2) launch_one<double, true>(a, f.bytes, warps, st);
  else launch_one<double, false>(a, f.bytes, warps, st);
  g_launches += steps;  // the statistics count its steps one by one, like a graph's nodes
}

}  // namespace kes
