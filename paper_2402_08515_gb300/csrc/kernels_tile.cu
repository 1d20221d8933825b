// Staged step kernels: the fused leapfrog step (Sec. 2.3, eq. 2stepmethod and
// eq. disc_filtercoeff) with everything a tile of rows needs copied to shared memory ahead of
// the arithmetic, for one to eight columns, in FP64, FP32 and FP32 pairs.
//
// What bounds it: a register-staged step (kernels_step.cu, kernels_block.cu) waits for memory:
// a warp has one slice in flight, its loads depend on one another (columns, then gathers), and
// a gather spends about ten instructions on every stored entry. Here one warp per block copies
// whole tiles with bulk copies (cp.async.bulk, one mbarrier per stage of a ring): the tile's
// matrix values, its rows of u_{n-1} and of the accumulators, and the few contiguous runs of
// rows of u_n that its columns lie in (on a tensor grid the three planes around the tile), so
// that the bytes in flight do not depend on registers or resident warps. The other warps read
// shared memory only: an entry costs one load of u_n, the FMAs of its columns, and a quarter
// of a value load and of an address. Entries of a tile whose rows are shifted copies of one
// another have no stored columns at all (kind 0, see TileSet); others have 16-bit places.
//
// Every row and column is the same FMA chain in entry order as in the other step kernels, so
// the results are the same to the bit: a zero entry, which a row of kind 0 holds for a coupling that it lacks, adds
// nothing to a finite sum. Once a value is not finite, more rows of its mesh and column are lost than the
// couplings alone would reach (no pattern leads out of a mesh); the call is unstable then and its result is none.
// Keeping the couplings' reach (summing such rows again from the stored matrix, or a switch to it) cost every FP32
// step 2 to 5%.
//
// Steps are launched programmatically one after the other (griddepcontrol): a block starts when
// the step before leaves its SM and reads its first tiles' matrix while that one ends, 3.6 us
// less a step at 128^3 cells and 1.0 us at 64^3 (FP32, one column).
//
// Microseconds a step, register-staged -> staged (cubes of n^3 cells): one column, 128^3: FP32
// 36.0 -> 22.7 (the 158 MB an average step cannot do without at 7.0 TB/s), FP64 67.8 -> 59.2 (FP64
// pipe); 64^3: FP32 6.0 -> 4.5, FP64 11.1 -> 9.9, fourth order 27.6 -> 19.6. FP32, 128^3: 2
// columns 44.8 -> 30.4, 4 62.3 -> 43.0, 8 84.8 -> 78.6 (shared memory and DRAM). FP64, 96^3: 2
// columns 55.3 -> 49.9, 4 104.7 -> 94.9, 8 204.9 -> 186.8 (FP64 pipe 97% busy).
// FP32 pairs (refinement sweeps): 250 thousand rows 2 columns 22.8 -> 10.5, 4 27.2 -> 14.1; 850 thousand rows 59.0 ->
// 29.5 and 78.2 -> 43.3.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "kes_internal.h"

namespace kes {
namespace {

constexpr int kGroupWarps = 8;      // warps that share a tile
constexpr int kMaxStages = 6;
constexpr int kTileSmem = 220 * 1024;  // bytes of shared memory a block may take
// Polls of a wait before it gives up: 1.5 us each on GB300 (the hardware suspends the warp), 1.5 seconds in all.
constexpr int kWaitLimit = 1 << 20;

struct TileArgs {
  TileSet ts;
  const void* val;
  const void* x;      // u_n
  const void* g;      // what the row sums gather from: u_n, or the fourth-order stage
  const void* prev;
  void* out;
  void* acc_s;        // FP64: the accumulator; else the compensated pair's s
  void* acc_c;
  double* acc64;
  int64_t acc_stride;
  const void* ahi;
  const void* alo;
  int F, Lp1, step, cpt;
  uint32_t coltab;
  int nterm, init, last, fold2;
  int keep, chained;
  int stages, stage_bytes, off_prev, off_own, off_acc, off_val, off_head;
  int* flag;
  int fail;           // the copying warps give up at their first wait
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, int bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Waits for the phase of that parity to complete; false once the limit is reached. (The limit is a constant: as a
// kernel parameter it cost the FP32 steps 1 to 2%.)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < kWaitLimit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
// bytes and both addresses: multiples of 16
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, int bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// With an L2 policy: matrix values are read once per step, so the first to leave L2 unless a
// whole step stays there.
__device__ __forceinline__ void bulk_copy_stream(uint32_t dst, const void* src, int bytes, uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(pol)
      : "memory");
}

// -x without the FP64 pipe: the compiler makes an FP64 instruction of every other form of it.
__device__ __forceinline__ double neg(double x) {
  asm("{\n\t.reg .b32 lo, hi;\n\tmov.b64 {lo, hi}, %0;\n\txor.b32 hi, hi, 0x80000000;\n\tmov.b64 %0, {lo, hi};\n\t}" : "+d"(x));
  return x;
}
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& t) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  const float ap = __fsub_rn(s, bp);
  t = __fadd_rn(__fsub_rn(a, ap), __fsub_rn(b, bp));
}

// N adjacent values, as wide as their bytes (N * sizeof(T) = 4, 8, 16 or 32)
template <typename T, int N>
struct alignas(sizeof(T) * N < 16 ? sizeof(T) * N : 16) Vec {
  T v[N];
};
template <typename T, int N>
__device__ __forceinline__ Vec<T, N> ld_vec(const T* p) {
  return *reinterpret_cast<const Vec<T, N>*>(p);
}
template <typename T, int N>
__device__ __forceinline__ void st_vec(T* p, const Vec<T, N>& v) {
  *reinterpret_cast<Vec<T, N>*>(p) = v;
}

// (sh, sl) += (ah + al)(xh + xl), the product's low-order terms and the sum's rounding error
// into sl
__device__ __forceinline__ void pair_fma(float ah, float al, float xh, float xl, float& sh, float& sl) {
  const float ph = __fmul_rn(ah, xh);
  float pe = fmaf(ah, xh, -ph);
  pe = fmaf(ah, xl, pe);
  pe = fmaf(al, xh, pe);
  float t, e;
  two_sum(sh, ph, t, e);
  sh = t;
  sl = __fadd_rn(sl, __fadd_rn(e, pe));
}

// The running sum of one row and column.
template <typename T> struct Sum {
  T s;
  __device__ __forceinline__ void add(T a, T x) { s = fma(a, x, s); }
};
template <> struct Sum<float2> {
  float h, l;
  __device__ __forceinline__ void add(float2 a, float2 x) { pair_fma(a.x, a.y, x.x, x.y, h, l); }
};

// Values of entries k .. k + 3 of a lane's row (FP32: quads; 8-byte values: pairs).
__device__ __forceinline__ void quad(const float* v, int k, int lr, float (&y)[4]) {
  const auto t = ld_vec<float, 4>(v + k * kSliceC + 4 * lr);
#pragma unroll
  for (int j = 0; j < 4; ++j) y[j] = t.v[j];
}
template <typename T>
__device__ __forceinline__ void quad(const T* v, int k, int lr, T (&y)[4]) {
  const auto a = ld_vec<T, 2>(v + k * kSliceC + 2 * lr), b = ld_vec<T, 2>(v + (k + 2) * kSliceC + 2 * lr);
  y[0] = a.v[0];
  y[1] = a.v[1];
  y[2] = b.v[0];
  y[3] = b.v[1];
}

// MODE 0: the step; 1: the stage v = u + A u / 12 of the fourth-order scheme (Remark 2.4). FOLD
// (FP64): the values hold A + 2I; a parameter of the kernel, since a condition in it costs the
// FP64 pipe one more operation a row (128^3 cells, one column: 62.7 -> 59.2 us a step).
template <typename T, int NB, int MODE, int GROUPS, bool FOLD>
__global__ void __launch_bounds__(32 * (kGroupWarps + 2) * GROUPS, 1) k_tile(const __grid_constant__ TileArgs a) {
  using S = typename std::conditional<std::is_same<T, double>::value, double, float>::type;  // accumulators, weights
  constexpr bool kPair = std::is_same<T, float2>::value, kF64 = std::is_same<T, double>::value;
  constexpr int CPL = NB < static_cast<int>(16 / sizeof(T)) ? NB : static_cast<int>(16 / sizeof(T));  // columns per lane
  constexpr int LPR = NB / CPL;           // lanes per row
  constexpr int RPU = kSliceC / LPR;      // rows per warp pass
  // weight tables' accumulators read ahead, besides the staged first one's, as registers allow
  constexpr int kAhead = GROUPS == 2 ? 3 : NB <= 2 ? 1 : 0;
  constexpr int kRowBytes = NB * static_cast<int>(sizeof(T));
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t bars[2 * kMaxStages];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stages = a.stages;
  if (threadIdx.x == 0) {
    for (int i = 0; i < stages; ++i) {
      mbar_init(smem_addr(&bars[i]), 2);
      mbar_init(smem_addr(&bars[kMaxStages + i]), kGroupWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // Programmatic launch: this step's blocks start as the previous step's end, and what no step
  // writes (the matrix, the tiles' descriptions) is read before that step has finished.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int first = blockIdx.x, stride = gridDim.x;
  const bool accs = MODE == 0 && a.nterm > 0 && !(kF64 && a.init);  // this step reads accumulators

  const int mine = (a.ts.n_tiles - first + stride - 1) / stride;  // this block's tiles (first < n_tiles)

  if (warp >= kGroupWarps * GROUPS) {
    // ------------------------------------------------------------ the copying warps
    // One copies state rows: lane l the tile's run l of what the sums gather, the last lanes the
    // tile's own rows of u_{n-1}, of u_n where the sums gather from something else, and of the
    // accumulators. The other copies the matrix. What they read to do so is read two tiles ahead.
    // Two roles with GROUPS warps each, a warp to every GROUPS-th tile: a bulk copy takes its
    // operands from one thread, and a warp works through its lanes' copies one after the other.
    const int part = (warp - kGroupWarps * GROUPS) >> 1;
    int n = part, st = part;
    uint32_t phase = 0;
    bool ok = true;
    auto next_stage = [&]() {
      st += GROUPS;
      if (st >= stages) {
        st -= stages;
        phase ^= 1;
      }
    };
    auto wait_empty = [&]() {
      return n < stages || (!a.fail && mbar_wait(smem_addr(&bars[kMaxStages + st]), phase ^ 1));
    };
    const int M = a.ts.max_runs + 2;
    if (((warp - kGroupWarps * GROUPS) & 1) == 0) {
      const bool own = MODE == 0 && a.g != a.x;
      const unsigned char* src = static_cast<const unsigned char*>(a.g);
      int row_bytes = kRowBytes, off = 0, slot = lane;
      bool active = lane < a.ts.max_runs;
      if (MODE == 0 && lane >= 28) {
        slot = a.ts.max_runs;
        active = true;
        if (lane == 31) {
          src = static_cast<const unsigned char*>(a.prev);
          off = a.off_prev;
        } else if (lane == 30) {
          active = own;
          src = static_cast<const unsigned char*>(a.x);
          off = a.off_own;
        } else {
          active = accs && (lane == 29 || !kF64);
          src = static_cast<const unsigned char*>(lane == 29 ? a.acc_s : a.acc_c);
          row_bytes = NB * static_cast<int>(sizeof(S));
          off = a.off_acc + (lane == 29 ? 0 : a.ts.R * row_bytes);
        }
      }
      const int4* p = a.ts.seg + static_cast<int64_t>(first) * M + slot;
      const int64_t pstep = static_cast<int64_t>(stride) * M;
      auto run_of = [&](int i) { return active && i < mine ? __ldg(p + i * pstep) : make_int4(0, 0, 0, 0); };
      int4 g0 = run_of(n), g1 = run_of(n + GROUPS);
      asm volatile("griddepcontrol.wait;" ::: "memory");
      for (; n < mine; n += GROUPS, next_stage()) {
        const int4 g = g0;
        g0 = g1;
        g1 = run_of(n + 2 * GROUPS);
        const int bytes = g.y * row_bytes;
        const int total = __reduce_add_sync(~0u, bytes);
        if (!(ok = wait_empty())) break;
        const uint32_t full = smem_addr(&bars[st]);
        if (lane == 0) mbar_expect(full, total);
        __syncwarp();
        if (bytes > 0)
          bulk_copy(smem_addr(smem) + static_cast<uint32_t>(st * a.stage_bytes + off + g.z * row_bytes),
                    src + static_cast<int64_t>(g.x) * row_bytes, bytes, full);
      }
    } else {
      uint64_t pol;
      if (a.keep) asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
      else asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
      const int4* p = a.ts.seg + static_cast<int64_t>(first) * M + M - 1;
      const int64_t pstep = static_cast<int64_t>(stride) * M;
      auto next_of = [&](int i) { return __ldg(p + min(i, mine - 1) * pstep); };
      int4 g0 = next_of(n), g1 = next_of(n + GROUPS);
      for (; n < mine; n += GROUPS, next_stage()) {
        const int4 g = g0;
        g0 = g1;
        g1 = next_of(n + 2 * GROUPS);
        const int val_bytes = g.y * static_cast<int>(sizeof(T));
        if (!(ok = wait_empty())) break;
        const uint32_t full = smem_addr(&bars[st]);
        const uint32_t base = smem_addr(smem) + static_cast<uint32_t>(st * a.stage_bytes);
        if (lane == 0) {
          mbar_expect(full, val_bytes + g.w);
          if (val_bytes > 0)
            bulk_copy_stream(base + a.off_val, static_cast<const T*>(a.val) + static_cast<int64_t>(g.x) * kSliceC,
                             val_bytes, full, pol);
          bulk_copy(base + a.off_head, a.ts.head + g.z, g.w, full);
        }
      }
    }
    if (!ok && lane == 0) atomicOr(a.flag, 2);
    // the copies still in flight write this block's shared memory
    for (int i = n - GROUPS; i >= 0 && i >= n - stages; i -= GROUPS)
      mbar_wait(smem_addr(&bars[i % stages]), (i / stages) & 1);
    return;
  }

  // -------------------------------------------------------------- the computing warps
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int grp = warp / kGroupWarps, wg = warp % kGroupWarps;
  const int sub = lane / LPR, co = (lane % LPR) * CPL;  // row of a pass, first column
  const int nacc = a.cpt ? 1 : a.F;
  bool bad = false;
  int st = grp;  // stages >= GROUPS
  uint32_t phase = 0;
  for (int n = grp; n < mine; n += GROUPS) {
    if (!mbar_wait(smem_addr(&bars[st]), phase)) {
      if (lane == 0) atomicOr(a.flag, 2);
      break;
    }
    const unsigned char* sp = smem + st * a.stage_bytes;
    const T* xs = reinterpret_cast<const T*>(sp);
    const T* vs = reinterpret_cast<const T*>(sp + a.off_val);
    const int4* head = reinterpret_cast<const int4*>(sp + a.off_head);
    const int w = head[0].x, kind = head[0].y;
    const int4 r1 = head[1];  // first row, rows, mesh, staged row of the first row
    const int units = r1.y / RPU;
    const int body = w & ~3, rest = w & 3;
    for (int u = wg; u < units; u += kGroupWarps) {
      const int r = u * RPU + sub, lr = r % kSliceC;
      const int at = r * NB + co;
      Vec<T, CPL> xi, pi;
      if (MODE == 0 && a.g != a.x) xi = ld_vec<T, CPL>(reinterpret_cast<const T*>(sp + a.off_own) + at);
      else xi = ld_vec<T, CPL>(xs + (r1.w + r) * NB + co);
      if (MODE == 0) pi = ld_vec<T, CPL>(reinterpret_cast<const T*>(sp + a.off_prev) + at);
      // the row's seed: -u_{n-1} when the values hold A + 2I, else 2 u_n - u_{n-1}
      Sum<T> un[CPL];
#pragma unroll
      for (int j = 0; j < CPL; ++j) {
        if constexpr (MODE == 1) {
          un[j].s = T(0);
        } else if constexpr (kPair) {
          if (a.fold2) {
            un[j].h = -pi.v[j].x;
            un[j].l = -pi.v[j].y;
          } else {
            float h, e;
            two_sum(__fmul_rn(2.0f, xi.v[j].x), -pi.v[j].x, h, e);
            un[j].h = h;
            un[j].l = __fadd_rn(e, __fsub_rn(__fmul_rn(2.0f, xi.v[j].y), pi.v[j].y));
          }
        } else if constexpr (kF64) {
          un[j].s = neg(pi.v[j]);
          if constexpr (!FOLD) un[j].s = fma(2.0, xi.v[j], un[j].s);
        } else {
          un[j].s = __fsub_rn(__fmul_rn(2.0f, xi.v[j]), pi.v[j]);
        }
      }
      const int64_t go = static_cast<int64_t>(r1.x) * NB + at;  // this lane's values in a row-major block
      // the accumulators of more tables than the staged one, read ahead of the row sums (96^3 cells,
      // 8 columns, 4 tables, FP32 67.5 -> 64.5 us a step; one column, 128^3, 46.5 -> 34.6)
      Vec<S, CPL> more_s[kAhead + 1], more_c[kAhead + 1];
      auto load_acc = [&](int f, int64_t go, Vec<S, CPL>& s_, Vec<S, CPL>& c_) {
        s_ = ld_vec<S, CPL>(static_cast<const S*>(a.acc_s) + f * a.acc_stride + go);
        if (!kF64) c_ = ld_vec<S, CPL>(static_cast<const S*>(a.acc_c) + f * a.acc_stride + go);
      };
      if (accs && nacc > 1) {
#pragma unroll
        for (int q = 0; q < kAhead; ++q)
          if (q + 1 < nacc) load_acc(q + 1, go, more_s[q], more_c[q]);
      }
      const T* v = vs + (r / kSliceC) * kSliceC * w;
      auto row_at = [&](int row) { return ld_vec<T, CPL>(xs + row * NB + co); };
      auto add = [&](T y, const Vec<T, CPL>& xv) {
#pragma unroll
        for (int j = 0; j < CPL; ++j) un[j].add(y, xv.v[j]);
      };
      if (kind == 0) {  // the pattern's entry k of every row: row base[k] + r of the staged ones
        const int* b = reinterpret_cast<const int*>(head + 2);
#pragma unroll 2
        for (int k = 0; k < body; k += 4) {
          T y[4];
          quad(v, k, lr, y);
          const int4 o = *reinterpret_cast<const int4*>(b + k);
          const Vec<T, CPL> x0 = row_at(o.x + r), x1 = row_at(o.y + r), x2 = row_at(o.z + r), x3 = row_at(o.w + r);
          add(y[0], x0);
          add(y[1], x1);
          add(y[2], x2);
          add(y[3], x3);
        }
        if (rest & 2) {
          const auto y = ld_vec<T, 2>(v + body * kSliceC + 2 * lr);
          const Vec<T, CPL> x0 = row_at(b[body] + r), x1 = row_at(b[body + 1] + r);
          add(y.v[0], x0);
          add(y.v[1], x1);
        }
        if (rest & 1) add(v[(w - 1) * kSliceC + lr], row_at(b[w - 1] + r));
      } else {  // each entry's own place
        const uint16_t* q = reinterpret_cast<const uint16_t*>(head + 2) + (r / kSliceC) * kSliceC * w;
#pragma unroll 2
        for (int k = 0; k < body; k += 4) {
          T y[4];
          quad(v, k, lr, y);
          const uint2 o = *reinterpret_cast<const uint2*>(q + k * kSliceC + 4 * lr);
          const Vec<T, CPL> x0 = row_at(o.x & 0xffff), x1 = row_at(o.x >> 16), x2 = row_at(o.y & 0xffff),
                            x3 = row_at(o.y >> 16);
          add(y[0], x0);
          add(y[1], x1);
          add(y[2], x2);
          add(y[3], x3);
        }
        if (rest & 2) {
          const auto y = ld_vec<T, 2>(v + body * kSliceC + 2 * lr);
          const uint32_t o = *reinterpret_cast<const uint32_t*>(q + body * kSliceC + 2 * lr);
          const Vec<T, CPL> x0 = row_at(o & 0xffff), x1 = row_at(o >> 16);
          add(y.v[0], x0);
          add(y.v[1], x1);
        }
        if (rest & 1) add(v[(w - 1) * kSliceC + lr], row_at(q[(w - 1) * kSliceC + lr]));
      }
      Vec<T, CPL> res;
#pragma unroll
      for (int j = 0; j < CPL; ++j) {
        if constexpr (MODE == 1) res.v[j] = fma(un[j].s, T(1) / T(12), xi.v[j]);
        else if constexpr (kPair) two_sum(un[j].h, un[j].l, res.v[j].x, res.v[j].y);
        else res.v[j] = un[j].s;
      }
      if (MODE == 1 || !a.last) st_vec<T, CPL>(static_cast<T*>(a.out) + go, res);
      if constexpr (MODE == 0) {
        // the last nterm of alpha_{n-1} u_{n-1}, alpha_n u_n, alpha_{n+1} u_{n+1}, in that order
        if (a.nterm > 0) {
          auto add_terms = [&](int f, Vec<S, CPL>& as, Vec<S, CPL>& ac) {
            const int64_t ga = f * a.acc_stride + go;
            if (kF64 && a.init) {  // it starts at the first term's product: fma(h, u, -0) = h u to the bit
#pragma unroll
              for (int j = 0; j < CPL; ++j) as.v[j] = static_cast<S>(-0.0);
            }
            auto term = [&](int q, const Vec<T, CPL>& uu) {
#pragma unroll
              for (int j = 0; j < CPL; ++j) {
                const int table = a.cpt ? static_cast<int>((a.coltab >> (4 * (co + j))) & 15u) : f;
                const int64_t ai = (static_cast<int64_t>(r1.z) * a.F + table) * a.Lp1 + a.step - 1 + q;
                const S h = __ldg(static_cast<const S*>(a.ahi) + ai);
                if constexpr (kF64) {
                  as.v[j] = fma(h, uu.v[j], as.v[j]);
                } else {
                  const float l = __ldg(static_cast<const float*>(a.alo) + ai);
                  if constexpr (kPair) {
                    pair_fma(h, l, uu.v[j].x, uu.v[j].y, as.v[j], ac.v[j]);
                  } else {
                    // alpha u = p + pe, p = fl(hi u), pe = (hi u - p) + lo u
                    const float p = __fmul_rn(h, uu.v[j]);
                    const float pe = fmaf(l, uu.v[j], fmaf(h, uu.v[j], -p));
                    float sn, e;
                    two_sum(as.v[j], p, sn, e);
                    ac.v[j] = __fadd_rn(ac.v[j], __fadd_rn(e, pe));
                    as.v[j] = sn;
                  }
                }
              }
            };
            if (a.nterm >= 3) term(0, pi);
            if (a.nterm >= 2) term(1, xi);
            term(2, res);
            if constexpr (kF64) {
              st_vec<S, CPL>(static_cast<S*>(a.acc_s) + ga, as);
              if (a.last)
#pragma unroll
                for (int j = 0; j < CPL; ++j) bad |= !isfinite(as.v[j]);
            } else if (a.last) {
#pragma unroll
              for (int j = 0; j < CPL; ++j) {
                const double v64 = static_cast<double>(as.v[j]) + static_cast<double>(ac.v[j]);
                bad |= !isfinite(v64);
                a.acc64[ga + j] = v64;
              }
            } else {
              st_vec<S, CPL>(static_cast<S*>(a.acc_s) + ga, as);
              st_vec<S, CPL>(static_cast<S*>(a.acc_c) + ga, ac);
            }
          };
          Vec<S, CPL> as, ac;
          if (accs) {
            as = ld_vec<S, CPL>(reinterpret_cast<const S*>(sp + a.off_acc) + at);
            if (!kF64) ac = ld_vec<S, CPL>(reinterpret_cast<const S*>(sp + a.off_acc) + a.ts.R * NB + at);
          }
          add_terms(0, as, ac);
          if (nacc > 1) {
#pragma unroll
            for (int q = 0; q < kAhead; ++q)
              if (q + 1 < nacc) add_terms(q + 1, more_s[q], more_c[q]);
            for (int f = kAhead + 1; f < nacc; ++f) {
              load_acc(f, go, as, ac);
              add_terms(f, as, ac);
            }
          }
        }
      }
    }
    // everything read from the stage has been used by now: the copies that follow may overwrite it
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_addr(&bars[kMaxStages + st]));
    st += GROUPS;
    if (st >= stages) {
      st -= stages;
      phase ^= 1;
    }
  }
  if (MODE == 0 && a.last && bad) atomicOr(a.flag, 1);
}

// ---------------------------------------------------------------- values
// Place of entry k of a lane: FP32 as quad_pos; 8-byte values in pairs.
__device__ __forceinline__ int64_t quad_place(int w, int k, int lane) {
  const int body = w & ~3;
  if (k < body) return static_cast<int64_t>(k >> 2) * 4 * kSliceC + 4 * lane + (k & 3);
  const int64_t at = static_cast<int64_t>(body) * kSliceC;
  if (!(w & 2)) return at + lane;
  return k - body < 2 ? at + 2 * lane + (k - body) : at + 2 * kSliceC + lane;
}
__device__ __forceinline__ int64_t pair_place(int w, int k, int lane) {
  if (k < (w & ~1)) return static_cast<int64_t>(k >> 1) * 2 * kSliceC + 2 * lane + (k & 1);
  return static_cast<int64_t>(k) * kSliceC + lane;
}

// Step values A = -tau^2 M^{-1} S in the order of the tiles: a = -tau2m[row] * val64[e]; q64 gets
// 2 added at the first entry at the row's own column when fold2 (A + 2I). What a row lacks of
// its pattern keeps the zero it was allocated with.
__global__ void k_scale_tiles(SellDev A, const int4* __restrict__ slice_rec, const int32_t* __restrict__ pat,
                              const double* __restrict__ tau2m, double* __restrict__ q64, float* __restrict__ q32,
                              int fold2) {
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  for (int64_t s = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; s < A.n_slices;
       s += nwarps) {
    const int64_t beg = A.slice_ptr[s], end = A.slice_ptr[s + 1];
    const int64_t row = s * kSliceC + lane;
    const double t = -tau2m[row];
    const int4 r = __ldg(slice_rec + s);
    bool diag_done = false;
    int k = 0, at = 0;   // at: the pattern's next difference
    int64_t last = -1;   // the row's last stored column: entries that do not pass it are padding
    for (int64_t e = beg + lane; e < end; e += kSliceC, ++k) {
      const double a = t * A.val64[e];
      const int64_t c = A.col[e];
      int pos = k;
      if (r.z == 0) {
        if (c <= last) continue;
        last = c;
        while (at < r.y && pat[r.w + at] != c - row) ++at;
        if (at == r.y) continue;  // only the zeros of rows past the mesh's last one
        pos = at;
      }
      const bool fold = fold2 && !diag_done && c == row;
      diag_done |= fold;
      const int64_t b = static_cast<int64_t>(r.x) * kSliceC;
      if (q64) q64[b + pair_place(r.y, pos, lane)] = fold ? a + 2.0 : a;
      if (q32) q32[b + quad_place(r.y, pos, lane)] = static_cast<float>(a);
    }
  }
}

struct Fit {
  int stages = 0, bytes = 0, off_prev = 0, off_own = 0, off_acc = 0, off_val = 0, off_head = 0;
};
// The stage's parts and how many stages fit.
Fit fit_stage(int R, int max_xrows, int max_w, int max_head, int row_bytes, int value_bytes, int NB, bool ho,
              int budget) {
  Fit f;
  int at = max_xrows * row_bytes;
  f.off_prev = at;
  at += R * row_bytes;
  f.off_own = at;
  if (ho) at += R * row_bytes;
  f.off_acc = at;
  at += R * NB * 8;
  f.off_val = at;
  at += R * max_w * value_bytes;
  f.off_head = at;
  at += max_head;
  f.bytes = (at + 127) & ~127;
  const int n = budget / f.bytes;
  f.stages = n >= 6 ? 6 : n >= 4 ? 4 : n >= 2 ? 2 : 0;  // a multiple of the groups of warps
  return f;
}

template <typename T, int NB, int MODE, int GROUPS, bool FOLD>
void launch_groups(TileArgs a, int grid, cudaStream_t st) {
  // The stages are a multiple of the groups, so a stage is used by one group and one copying
  // warp of each role only: whoever waits for its next use has seen the last one, and cannot
  // take the phase before that for the one it waits for.
  // the limit is the same for every context: another thread's launch never lowers it
  cudaFuncSetAttribute(k_tile<T, NB, MODE, GROUPS, FOLD>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmem);
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(32 * (kGroupWarps + 2) * GROUPS);
  c.dynamicSmemBytes = a.stages * a.stage_bytes;
  c.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = a.chained ? 1 : 0;
  cudaLaunchKernelEx(&c, k_tile<T, NB, MODE, GROUPS, FOLD>, a);
}
// Three groups of warps where two stages for each fit, else two (128^3 cells, one column: FP32,
// six stages, 22.7 us a step with three and 23.8 us with two; FP64, four stages of 45 KB, 59.2 us
// with two groups; three (78 us when two took 62.7) leave none to be filled while the others are in use).
// Four FP32 columns take two groups all the same: with three, 64 registers a thread hold a row's sums
// and loads only with spills (300 thousand rows, us a step with three / two groups: 7 entries a row in 2D
// 9.5 / 7.6, 25 entries 15.9 / 13.1; 970 thousand rows of a tube 34.4 / 29.5).
constexpr int groups_of(int stages, int value_bytes, int NB) {
  return stages >= 6 && !(value_bytes == 4 && NB == 4) ? 3 : 2;
}
template <typename T, int NB, int MODE>
void launch_one(const TileArgs& a, int grid, cudaStream_t st) {
  if constexpr (std::is_same<T, double>::value && MODE == 0) {
    if (a.fold2) {
      if (groups_of(a.stages, sizeof(T), NB) == 3) launch_groups<T, NB, MODE, 3, true>(a, grid, st);
      else launch_groups<T, NB, MODE, 2, true>(a, grid, st);
      return;
    }
  }
  if constexpr (groups_of(6, sizeof(T), NB) == 3) {
    if (a.stages >= 6) {
      launch_groups<T, NB, MODE, 3, false>(a, grid, st);
      return;
    }
  }
  launch_groups<T, NB, MODE, 2, false>(a, grid, st);
}

template <typename T, int MODE>
bool launch_nb(const TileArgs& a, int NB, int grid, cudaStream_t st) {
  if constexpr (!std::is_same<T, float2>::value)
    if (NB == 1) {
      launch_one<T, 1, MODE>(a, grid, st);
      return true;
    }
  if (NB == 2) launch_one<T, 2, MODE>(a, grid, st);
  else if (NB == 4) launch_one<T, 4, MODE>(a, grid, st);
  else if (NB == 8) launch_one<T, 8, MODE>(a, grid, st);
  else return false;
  return true;
}

// Whether the values stay in L2 (129 MB) with the rest of what a step reads and writes. 96^3
// cells in FP32 (62 MB): 10.4 us a step if so, 11.3 us with values that leave first; in FP64
// (123 MB) 29.0 and 28.2 us, 128^3 in FP32 (147 MB) 25.9 and 22.7 us.
bool keep_in_l2(const TileStep& p, int size) {
  const int64_t state = p.acc_stride * (3 * size + 8 * p.F);
  return p.n_values * size + state <= int64_t(80) << 20;
}

}  // namespace

int tile_stages(int R, int max_xrows, int max_w, int max_head, int row_bytes, int value_bytes, int NB, bool ho) {
  return fit_stage(R, max_xrows, max_w, max_head, row_bytes, value_bytes, NB, ho, kTileSmem).stages;
}

int tile_busy_warps(int R, int stages, int value_bytes, int NB) {
  const int columns = std::min(NB, 16 / value_bytes);  // of a lane (CPL)
  const int passes = R * (NB / columns) / kSliceC;     // of a warp over the tile's rows
  return std::min(kGroupWarps, passes) * groups_of(stages, value_bytes, NB);
}

void launch_tile_step(const TileStep& p, cudaStream_t st) {
  TileArgs a{};
  const int size = p.type == kTileF32 ? 4 : 8;
  const Fit f = fit_stage(p.ts.R, p.ts.max_xrows, p.ts.max_w, p.ts.max_head, size * p.NB, size, p.NB, p.g != p.x,
                          kTileSmem);
  a.ts = p.ts;
  a.val = p.val;
  a.x = p.x;
  a.g = p.g;
  a.prev = p.prev;
  a.out = p.out;
  a.acc_s = p.acc_s;
  a.acc_c = p.acc_c;
  a.acc64 = p.acc64;
  a.acc_stride = p.acc_stride;
  a.ahi = p.ahi;
  a.alo = p.alo;
  a.F = p.F;
  a.Lp1 = p.L + 1;
  a.step = p.step;
  a.cpt = p.cpt;
  if (p.cpt > 0)
    for (int c = 0; c < p.NB; ++c) a.coltab |= static_cast<uint32_t>(std::min(c / p.cpt, p.F - 1)) << (4 * c);
  a.nterm = p.nterm;
  a.init = p.init;
  a.last = p.last;
  a.fold2 = p.fold2;
  a.flag = p.flag;
  a.fail = p.fail;
  a.stages = f.stages;
  a.chained = p.chained;
  a.keep = keep_in_l2(p, size);
  a.stage_bytes = f.bytes;
  a.off_prev = f.off_prev;
  a.off_own = f.off_own;
  a.off_acc = f.off_acc;
  a.off_val = f.off_val;
  a.off_head = f.off_head;
  const int grid = std::min(p.ts.n_tiles, p.n_sm);
  if (p.stage4) {
    if (p.type == kTileF64) launch_nb<double, 1>(a, p.NB, grid, st);
    else launch_nb<float, 1>(a, p.NB, grid, st);
  } else if (p.type == kTileF64) {
    launch_nb<double, 0>(a, p.NB, grid, st);
  } else if (p.type == kTileF32) {
    launch_nb<float, 0>(a, p.NB, grid, st);
  } else {
    launch_nb<float2, 0>(a, p.NB, grid, st);
  }
  ++g_launches;
}

void launch_scale_tiles(const SellDev& A, const int4* slice_rec, const int32_t* pat, int n_sm, cudaStream_t st,
                        const double* tau2m, double* q64, float* q32, bool fold2) {
  const int64_t need = (A.n_slices + 7) / 8;
  const int64_t cap = static_cast<int64_t>(n_sm) * 8;
  k_scale_tiles<<<static_cast<int>(std::max<int64_t>(1, std::min(need, cap))), 256, 0, st>>>(A, slice_rec, pat, tau2m,
                                                                                           q64, q32, fold2 ? 1 : 0);
  ++g_launches;
}

}  // namespace kes
