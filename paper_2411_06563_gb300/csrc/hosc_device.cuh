// Device helpers shared by the kernels of libhosc.so: indexing, one-sided / central gradients,
// block reductions and the last-block reduction of per-block partials.
#pragma once

// Loads of arrays that a kernel only reads. A kernel launch reads them through the read-only
// (non-coherent) cache with restrict-qualified pointers. The persistent round kernel of the pool
// (hosc_round.cu, built with HOSC_PERSISTENT_BUILD) writes these arrays in one phase and reads
// them in a later one of the same launch, so there they are plain loads cached in L2 only
// (coherent across SMs), and pointers are not restrict-qualified.
#ifdef HOSC_PERSISTENT_BUILD
#define HOSC_RESTRICT
#define HOSC_LDG(p) __ldcg(p)
#else
#define HOSC_RESTRICT __restrict__
#define HOSC_LDG(p) __ldg(p)
#endif


#include <cuda_runtime.h>

#include "hosc_internal.h"

namespace hosc {

__device__ __forceinline__ long node(int i, int j, int k, int N) {
  return (long)i + (long)N * ((long)j + (long)N * (long)k);
}

// Derivative along one axis at a node whose coordinate along that axis is a (0..N-1); st is the
// memory stride of that axis. Central inside, second-order one-sided at the two walls.
__device__ __forceinline__ double grad_axis(const double* HOSC_RESTRICT f, long c, int a, int N,
                                            long st, double inv2h) {
  if (a == 0) return (-3.0 * f[c] + 4.0 * f[c + st] - f[c + 2 * st]) * inv2h;
  if (a == N - 1) return (3.0 * f[c] - 4.0 * f[c - st] + f[c - 2 * st]) * inv2h;
  return (f[c + st] - f[c - st]) * inv2h;
}

struct Grad9 {
  double ux, uy, uz, vx, vy, vz, wx, wy, wz;
};

// The nine velocity gradients at node (i, j, k); ix, iy, iz = 1/(2 h_d) of the three directions.
__device__ __forceinline__ Grad9 velocity_gradients(const double* HOSC_RESTRICT u,
                                                    const double* HOSC_RESTRICT v,
                                                    const double* HOSC_RESTRICT w, int i, int j,
                                                    int k, int N, double ix, double iy,
                                                    double iz) {
  const long c = node(i, j, k, N);
  const long sy = N, sz = (long)N * N;
  Grad9 g;
  g.ux = grad_axis(u, c, i, N, 1, ix);
  g.uy = grad_axis(u, c, j, N, sy, iy);
  g.uz = grad_axis(u, c, k, N, sz, iz);
  g.vx = grad_axis(v, c, i, N, 1, ix);
  g.vy = grad_axis(v, c, j, N, sy, iy);
  g.vz = grad_axis(v, c, k, N, sz, iz);
  g.wx = grad_axis(w, c, i, N, 1, ix);
  g.wy = grad_axis(w, c, j, N, sy, iy);
  g.wz = grad_axis(w, c, k, N, sz, iz);
  return g;
}

// Second invariant of the strain-rate tensor, Eq. (8).
__device__ __forceinline__ double second_invariant(const Grad9& g) {
  const double a = g.uz + g.wx, b = g.uy + g.vx, c = g.vz + g.wy;
  return 2.0 * (g.ux * g.ux + g.vy * g.vy + g.wz * g.wz) + a * a + b * b + c * c;
}

// Programmatic dependent launch: the kernels of a step are launched so that each may start while the
// previous one is finishing (its blocks take SMs as the previous kernel's blocks leave); a kernel
// waits for the previous grid's completion and memory before its first access, and lets the next
// kernel launch at once.
__device__ __forceinline__ void pdl_wait_and_release() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launch of a kernel that starts with pdl_wait_and_release; in a captured step such kernels chain
// with programmatic edges.
template <class... K, class... A>
inline void launch_pdl(void (*kern)(K...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                       const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, K(args)...);
}

// ----------------------------------------------------------------------------- reductions

// Larger of two non-negative doubles (+inf allowed). For such values the IEEE order is the order
// of their bit patterns as integers, so the comparison runs on the integer units: GB300 issues
// FP64 instructions at a small fraction of its integer rate. Every max-reduction here reduces
// magnitudes.
__device__ __forceinline__ double max_nonneg(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return __longlong_as_double(x > y ? x : y);
}

// What a reduction does with two values of its type V, and the double it ends in.
struct SumD {
  using V = double;
  using Total = SumD;   // the operation on the doubles of the blocks
  static __device__ __forceinline__ V zero() { return 0.0; }
  static __device__ __forceinline__ V add(V a, V b) { return a + b; }
  static __device__ __forceinline__ V shfl_xor(V a, int m) {
    return __shfl_xor_sync(0xffffffffu, a, m);
  }
  static __device__ __forceinline__ double value(V a) { return a; }
};
struct MaxD : SumD {   // of non-negative values
  using Total = MaxD;
  static __device__ __forceinline__ V add(V a, V b) { return max_nonneg(a, b); }
};

__host__ __device__ constexpr int pow2_at_least(int m) {
  return m <= 1 ? 1 : 2 * pow2_at_least((m + 1) / 2);
}

// Reduce Mp values (a power of two) over a warp by halving: at stage k a lane keeps one half of its
// values and gives the other half to the lane that differs in bit k, so that Mp - 1 + log2(32/Mp)
// additions take the place of 5 Mp. Every lane ends with the total of value fold_slot<Mp>(lane).
// What this saves: GB300 issues an FP64 instruction of a warp in 16 cycles of the SM's one FP64
// pipe, and a float-float addition is 10 float instructions, so the 20 to 40 additions per thread
// of a plain shuffle tree of 4 to 8 values cost more than the stencil arithmetic they followed.
// Measured per launch, with the ends of the Krylov kernels one thread a system (hosc_krylov4.cuh):
// x/r at 41^3 mixed 20.4 -> 10.0 us, at 101^3 mixed 33.1 -> 21.4 us, at 91^3 FP64 128 -> 75 us; p/v
// 13.7 -> 9.3, 45.2 -> 39.8 and 164 -> 138 us.
template <class Op, int Mp>
__device__ __forceinline__ typename Op::V warp_fold(typename Op::V (&v)[Mp]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; (Mp >> k) > 1; ++k) {
    const int h = Mp >> (k + 1);
    const bool up = (lane >> k) & 1;
#pragma unroll
    for (int q = 0; q < h; ++q) {
      const typename Op::V give = up ? v[q] : v[q + h], keep = up ? v[q + h] : v[q];
      v[q] = Op::add(keep, Op::shfl_xor(give, 1 << k));
    }
  }
  typename Op::V r = v[0];
#pragma unroll
  for (int off = Mp; off < 32; off <<= 1) r = Op::add(r, Op::shfl_xor(r, off));
  return r;
}
template <int Mp>
__device__ __forceinline__ int fold_slot(int lane) {
  int m = 0;
#pragma unroll
  for (int k = 0; (Mp >> k) > 1; ++k) m |= ((lane >> k) & 1) ? Mp >> (k + 1) : 0;
  return m;
}

// Warp 0: totals over the block's warps of s[warp * Mp + m]; lane m (m < Mp) gets value m.
template <class Op, int Mp>
__device__ __forceinline__ typename Op::V cross_warps(const typename Op::V* s) {
  const int lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  typename Op::V r = Op::zero();
  for (int w = lane / Mp; w < nw; w += 32 / Mp) r = Op::add(r, s[w * Mp + lane % Mp]);
  const int used = min(32, nw * Mp);   // the lanes past it hold zeros
  for (int off = Mp; off < used; off <<= 1) r = Op::add(r, Op::shfl_xor(r, off));
  return r;
}

constexpr int kMaxWarps = 16;   // warps of a block that reduces

// Sum (or max, of non-negative values) of M values over the block; thread m < M returns value m.
// Fixed order, so the result is the same run to run for the same launch shape.
template <class Op, int M>
__device__ __forceinline__ typename Op::V block_total(const typename Op::V (&v)[M]) {
  using V = typename Op::V;
  constexpr int Mp = pow2_at_least(M);
  static_assert(Mp <= 32, "at most 32 values");
  __shared__ V s_w[kMaxWarps * Mp];
  V x[Mp];
#pragma unroll
  for (int m = 0; m < Mp; ++m) x[m] = m < M ? v[m < M ? m : 0] : Op::zero();
  const V r = warp_fold<Op, Mp>(x);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane < Mp) s_w[wid * Mp + fold_slot<Mp>(lane)] = r;
  __syncthreads();
  return wid == 0 ? cross_warps<Op, Mp>(s_w) : Op::zero();
}

// Doubles per row of the partials buffer for M values per block: kRedSlots, 2 kRedSlots for
// 8 < M <= 16, 4 kRedSlots for 16 < M <= 32 (one row then spans two or four rows of kRedSlots;
// the kernels with more than 16 values have few enough blocks).
template <int M>
__host__ __device__ constexpr int row_stride() {
  return M > 2 * kRedSlots ? 4 * kRedSlots : (M > kRedSlots ? 2 * kRedSlots : kRedSlots);
}

// Sum of nr rows of M slots in an order that does not depend on the block's size, so that every kernel
// that forms the same rows gets the same bits: group g of G adds rows g, g + G, ... one after another
// (four loads in flight), then the groups combine in a tree. load(row, slot); the totals are left in
// tot (shared), valid for every thread. blockDim.x must be a multiple of 32.
template <int Mp>
constexpr int row_groups() { return Mp <= 8 ? 64 : 512 / Mp; }

// The totals of M slots over the groups of s_g[group * Mp + slot] into tot, a warp a slot.
template <class T, int M, int G = row_groups<pow2_at_least(M)>()>
__device__ __forceinline__ void sum_groups(const double* s_g, double* tot) {
  constexpr int Mp = pow2_at_least(M);
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int m = threadIdx.x >> 5; m < M; m += nw) {
    double a = lane < G ? s_g[lane * Mp + m] : 0.0;
    if (G > 32) a = T::add(a, s_g[(lane + 32) % G * Mp + m]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) a = T::add(a, T::shfl_xor(a, off));
    if (lane == 0) tot[m] = a;
  }
}

template <class T, int M, class Load>
__device__ __forceinline__ void sum_rows(int nr, Load load, double* tot) {
  constexpr int Mp = pow2_at_least(M);
  constexpr int G = row_groups<Mp>();
  __shared__ double s_g[Mp * G];
  const int t = threadIdx.x, bd = blockDim.x;
  for (int w = t; w < Mp * G; w += bd) {
    const int m = w % Mp;
    double acc = 0.0;
    int r = m < M ? w / Mp : nr;   // the slots past the M values stay zero
    for (; r + 3 * G < nr; r += 4 * G) {
      const double a0 = load(r, m), a1 = load(r + G, m), a2 = load(r + 2 * G, m),
                   a3 = load(r + 3 * G, m);
      acc = T::add(T::add(T::add(T::add(acc, a0), a1), a2), a3);
    }
    for (; r < nr; r += G) acc = T::add(acc, load(r, m));
    s_g[w] = acc;
  }
  __syncthreads();
  sum_groups<T, M>(s_g, tot);
  __syncthreads();
}

// A ticket of the `tickets` given out at counter, taken after warp 0's writes; true in the block that
// takes the last one (no block waits for another), which leaves the counter at zero for the next
// kernel and sees what the others wrote.
__device__ __forceinline__ bool last_ticket(unsigned int* counter, unsigned int tickets) {
  __shared__ int s_last;
  if (threadIdx.x < 32) {
    __syncwarp();
    if (threadIdx.x == 0) {
      __threadfence();
      s_last = atomicAdd(counter, 1u) == tickets - 1;
    }
  }
  __syncthreads();
  const bool last = s_last;
  if (last) {
    __threadfence();
    if (threadIdx.x == 0) *counter = 0u;
  }
  return last;
}

// Second half of a reduction over the grid, called by every block once its warp 0 has written values to
// row `row` of the nr rows of M slots (per_row blocks write a row): the last block returns the totals
// in shared memory, valid for its every thread; the others return null. Above kFlatRows rows the sum
// has two levels: one block summing the 8 000 rows of a 257^3 launch took 50 to 75 us of each kernel
// (x/r 384 -> 318 us, p/v 510 -> 448 us, s/t 369 -> 300 us).
template <class T, int M>
__device__ __forceinline__ const double* last_block_total(const RedBuf& b, unsigned int row,
                                                          unsigned int nr, unsigned int per_row) {
  constexpr long S = row_stride<M>();
  __shared__ double s_tot[pow2_at_least(M)];
  const double* rows = b.red;
  unsigned int tickets = nr * per_row;
  if (nr > kFlatRows) {
    const unsigned int g = row / kGroupRows, r0 = g * kGroupRows, n = min(kGroupRows, nr - r0);
    if (!last_ticket(b.counter + 1 + g, n * per_row)) return nullptr;
    rows = b.red + r0 * S;
    sum_rows<T, M>((int)n, [&](int r, int m) { return __ldcg(rows + r * S + m); }, s_tot);
    if (threadIdx.x < M) b.red2[g * S + threadIdx.x] = s_tot[threadIdx.x];
    rows = b.red2;
    tickets = nr = (nr + kGroupRows - 1) / kGroupRows;
  }
  if (!last_ticket(b.counter, tickets)) return nullptr;
  sum_rows<T, M>((int)nr, [&](int r, int m) { return __ldcg(rows + r * S + m); }, s_tot);
  return s_tot;
}

// Reduction over the grid of M values per thread: block b of nb writes its totals to its row;
// the last block returns the totals (see last_block_total), the others null.
template <class Op, int M>
__device__ __forceinline__ const double* grid_total(const typename Op::V (&v)[M], const RedBuf& buf,
                                                    unsigned int b, unsigned int nb) {
  const typename Op::V mine = block_total<Op, M>(v);
  if (threadIdx.x < M) buf.red[(long)b * row_stride<M>() + threadIdx.x] = Op::value(mine);
  return last_block_total<typename Op::Total, M>(buf, b, nb, 1u);
}

}  // namespace hosc
