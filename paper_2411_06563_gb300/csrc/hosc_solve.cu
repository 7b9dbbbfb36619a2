// The BiCGSTAB solve of one step as one launch, for grids whose unknowns fit on the chip (Punia & Ray,
// arXiv:2411.06563, Sec. 2.2: unpreconditioned BiCGSTAB on the four level-(n+1) systems of Eq. 5).
//
// On small grids an iteration's three launches cost 5 to 15 us each whatever the size: the launch
// itself, the scalars' read, the first loads, the ticket, the last block's sum of the partials and its
// divisions. Here the grid is cooperative (every block resident); a block keeps its nodes' vectors in
// registers and their operator rows in shared memory from the first iteration to the last, and a phase
// (p/v, s/t, x/r) ends in one exchange: each block puts its partial sums in its row of a buffer, and
// every block reads all rows, adds them in the same order and computes the scalars itself. A value
// travels as two 8-byte words that each carry 4 bytes of it and the exchange's number, so that a
// reader needs no other flag; two buffers alternate, since a block that has finished exchange e has
// every row of it, and so nobody still reads exchange e - 1. The vectors that other blocks need at the
// borders of a block (v after p/v; r and p - omega v after x/r) are written to memory before the
// exchange and read through L2 after it.
//
// The arithmetic of a node, the partial sums of a block and the order of the rows' sum are those of
// the kernels that run an iteration in three launches (hosc_krylov.cu) with the same block shape: the
// same bits.
//
// Every wait is bounded (kWaitNs on the GPU timer): a block whose wait runs out leaves the solve, the
// others follow when theirs do, and the step reports HOSC_ECUDA. No wait runs while some blocks cannot
// start: a cooperative grid starts whole, after other kernels have left it the room.
//
// Spills (-Xptxas -v): 32 bytes stored and 44 loaded a thread in k_solve_planar<1> (held to 64 registers),
// 22 and 12 in k_solve_mixed<4>, none in the other forms.
//
// Measured against an iteration in three launches: FP64 21^3 25.4 -> 12.1 us, 31^3 35 -> 18.1 us, 41^3
// 49 -> 24.2 us (there half of it FP64 instructions); mixed step at 41^3 226 -> 133 us, at 64^3
// 348 -> 232 us. An iteration at 21^3 spends about 3 x 1.2 us on the exchanges' trip through L2, 3 x 0.5 us
// on the writes before them becoming visible, 1.5 us on divisions; the rest is FP64 work and barriers.

#include <math.h>

#include <type_traits>

#include "hosc_device.cuh"
#include "hosc_internal.h"
#include "hosc_krylov4.cuh"

namespace hosc {

namespace {

constexpr unsigned long long kWaitNs = 2000000000ull;   // 2 s

__device__ __forceinline__ unsigned long long solve_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// One value of an exchange: two words of (4 bytes of the value, the exchange's number): data and flag in
// one store, as the low-latency protocols of collective libraries send it.
__device__ __forceinline__ void put_value(ulonglong2* p, double v, unsigned e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned long long f = (unsigned long long)e << 32;
  asm volatile("st.volatile.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"((b & 0xffffffffull) | f),
               "l"((b >> 32) | f)
               : "memory");
}
// An acquire: what the writer wrote before its row is visible to this thread, and to the block after its
// next barrier.
__device__ __forceinline__ bool get_value(const ulonglong2* p, unsigned e, double& v) {
  unsigned long long a, b;
  asm volatile("ld.acquire.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  v = __longlong_as_double((long long)((a & 0xffffffffull) | (b << 32)));
  return (unsigned)(a >> 32) == e && (unsigned)(b >> 32) == e;
}

// The blocks that exchange with one another: rows of `stride` values, two buffers.
struct Exchange {
  ulonglong2* rows;
  int nr, stride, mine;   // number of rows, values a row, this block's row
  unsigned e;             // number of the last exchange
  int* failed;            // shared: a wait of this block has run out
};

// Thread m < M of the block puts its value of the block's row and the block gathers the totals of all
// rows, in the order of sum_rows, in tot (shared), K rows of a sum in flight. A function of its own:
// inlined, its loops cost the callers the registers that hold their vectors; what it uses itself they
// have to keep clear of all the same, so K is small (a step with K = 4, 2 and 1: 21^3 FP64 351, 331 and
// 327 us, 64^3 mixed 244, 232 and 236; two sums side by side, eight in flight: 398 and 286).
template <class T, int M, int G, int K>
__device__ __noinline__ bool gather(ulonglong2* rows, int nr, int stride, int row, unsigned e,
                                    double mine, double* tot, int* failed) {
  constexpr int Mp = pow2_at_least(M);
  __shared__ double s_g[Mp * G];
  rows += (size_t)(e & 1u) * nr * stride;
  const int t = threadIdx.x;
  if (t < M) {
    fence_gpu();   // the block's writes to memory come before its row
    put_value(rows + row * stride + t, mine, e);
  }
  for (int w = t; w < Mp * G; w += blockDim.x) {
    const int m = w % Mp;
    double acc = 0.0;
    if (m < M) {
      for (int r = w / Mp; r < nr; r += K * G) {
        const int n = min(K, (nr - r + G - 1) / G);   // rows r, r + G, ... of this pass
        double a[K];
        unsigned long long t0 = 0;
        for (unsigned spin = 0;; ++spin) {
          bool ok = true;
#pragma unroll
          for (int q = 0; q < K; ++q)
            if (q < n) ok &= get_value(rows + (r + q * G) * stride + m, e, a[q]);
          if (ok) break;
          if ((spin & 255u) == 255u) {
            const unsigned long long now = solve_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > kWaitNs || *(volatile int*)failed) {
              *(volatile int*)failed = 1;
              break;
            }
          }
        }
#pragma unroll
        for (int q = 0; q < K; ++q)
          if (q < n) acc = T::add(acc, a[q]);
      }
    }
    s_g[w] = acc;
  }
  __syncthreads();
  sum_groups<T, M, G>(s_g, tot);
  __syncthreads();
  return *(volatile int*)failed == 0;
}

// The totals of M values per thread over all blocks of the exchange, in tot (shared). Orders the
// block's earlier writes to memory before the others' reads that follow. False when a wait ran out
// (uniform over the block).
template <class Op, int M, int G = row_groups<pow2_at_least(M)>()>
__device__ __forceinline__ bool exchange(Exchange& x, const typename Op::V (&v)[M], double* tot) {
  x.e += 1;
  const typename Op::V mine = block_total<Op, M>(v);
    // the FP64 shapes mostly have no more rows than groups, the mixed ones up to four times as many
  constexpr int K = std::is_same<Op, typename Op::Total>::value ? 1 : 2;
  return gather<typename Op::Total, M, G, K>(x.rows, x.nr, x.stride, x.mine, x.e, Op::value(mine), tot,
                                       x.failed);
}

// xr_scalars for S systems at ks, its three serial chains side by side: the two quotients of beta in two
// groups of S lanes (one division's time), the square root and the tests in another warp.
template <int S>
__device__ __forceinline__ void split_xr_scalars(const DevParams& P, KrylovScalars* ks,
                                                 const double* tot) {
  const int t = threadIdx.x, s = t % S;
  if (t < 2 * S) {
    const bool lo = t < S;
    const double q = (lo ? tot[s] : ks[s].alpha) / (lo ? ks[s].rho : ks[s].omega);
    const double q2 = __shfl_down_sync((1u << (2 * S)) - 1u, q, S);
    if (lo) {   // not read where the system is done
      ks[s].beta = q * q2;
      ks[s].rho = tot[s];
    }
  } else if (t >= 32 && t < 32 + S && !ks[s].done) {
    const double rnorm = sqrt(tot[S + s]);
    const int iters = ks[s].iters + 1;
    ks[s].rnorm = rnorm;
    ks[s].iters = iters;
    const bool conv = rnorm <= P.tol_lin * ks[s].r0norm;
    if (conv || !isfinite(rnorm) || iters >= P.max_lin_iter || tot[s] == 0.0 || ks[s].omega == 0.0) {
      ks[s].done = 1;
      ks[s].status = conv ? 0 : HOSC_ENOCONV;
    }
  }
}

// ------------------------------------------------------------------ FP64 (planar)
//
// A block has one system, as many consecutive nodes of the plane (i + N j, walls included) as threads
// and up to KZ planes; a system's blocks exchange among themselves and leave when it is done.

template <int KZ>
size_t planar_state(int N, int B) {   // operator rows and rhs, then KZ planes of B + 2 N values
  return sizeof(double) * ((size_t)8 * KZ * B + (size_t)KZ * (B + 2 * N));
}

// Most threads of the BiCGSTAB(2) form: seven vectors of KZ planes in registers.
constexpr int b2_threads(int KZ) { return KZ <= 2 ? kPlanarMost : KZ == 4 ? 384 : 256; }

static_assert(4 * 2 * 5 * kSolveRows <= kExchValues, "the rows of five values exceed the buffer");

// A thread's nodes of its block's planes, with the operator rows, rhs and the planes in shared memory.
template <int KZ>
struct Slab {
  int s, N, N2, B, w, t, c0, k0, nk, hs, hc;
  bool in, has_halo, hin, below, above;
  double* a;        // weight q of plane kk: a[(8 kk + q) B + t]; rhs at q = 7
  double* planes;   // plane kk: nodes l0 - N .. l0 + B + N

  __device__ __forceinline__ Slab(const DevParams& P, double* sh) {
    s = (int)(blockIdx.x & 3u), t = threadIdx.x;
    N = P.N, N2 = N * N, B = blockDim.x, w = B + 2 * N;
    const int l0 = (int)(blockIdx.x >> 2) * B, l = l0 + t;
    k0 = 1 + (int)blockIdx.y * P.pkz, nk = min(P.pkz, N - 1 - k0);
    // the node before or after the chunk whose value this thread fetches (2 N <= B)
    const int hl = t < N ? l0 - N + t : l0 + B + (t - N);
    hs = t < N ? t : B + t;
    in = inside(l);
    has_halo = t < 2 * N, hin = has_halo && inside(hl);
    below = in && k0 > 1, above = in && k0 + nk < N - 1;
    c0 = l + N2 * k0, hc = hl + N2 * k0;
    a = sh;
    planes = sh + 8 * KZ * B;
  }
  __device__ __forceinline__ bool inside(int q) const {   // node q of the plane lies inside the walls
    if (q < 0 || q >= N2) return false;
    const int j = q / N, i = q - j * N;
    return i > 0 && i < N - 1 && j > 0 && j < N - 1;
  }
  __device__ __forceinline__ Exchange rows(const Fields& F, int stride, int* failed) const {
    const unsigned chunks = gridDim.x >> 2;
    Exchange x;
    x.nr = (int)(chunks * gridDim.y);
    x.stride = stride;
    x.mine = (int)((blockIdx.x >> 2) + chunks * blockIdx.y);
    x.rows = F.exch + (size_t)s * 2 * x.nr * x.stride;
    x.e = 0;
    x.failed = failed;
    return x;
  }
  __device__ __forceinline__ bool mine(int kk) const { return in && kk < nk; }
  __device__ __forceinline__ int c(int kk) const { return c0 + N2 * kk; }
  __device__ __forceinline__ double r0(int kk) const { return a[(8 * kk + 7) * B + t]; }
  // rhs into r (zero elsewhere), operator rows and rhs into shared memory
  __device__ __forceinline__ void load(const Fields& F, double (&r)[KZ]) {
    const double* rhs = F.rhs[s];
    const double* const* A = s < 3 ? F.Am : F.Ae;
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) {
      r[kk] = 0.0;
      if (mine(kk)) {
        r[kk] = rhs[c(kk)];
        a[(8 * kk + 7) * B + t] = r[kk];
#pragma unroll
        for (int q = 0; q < 7; ++q) a[(8 * kk + q) * B + t] = A[q][c(kk)];
      }
    }
  }
  // the operator on own values f (registers) and the others' values val(c): y of each plane
  template <class Val>
  __device__ __forceinline__ void apply(const double (&f)[KZ], double (&y)[KZ], Val val) const {
    const double lo = below ? val(c0 - N2) : 0.0, hi = above ? val(c0 + N2 * nk) : 0.0;
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) {
      const double h = hin && kk < nk ? val(hc + N2 * kk) : 0.0;
      planes[kk * w + N + t] = f[kk];   // zero on the walls
      if (has_halo) planes[kk * w + hs] = h;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) {
      if (!mine(kk)) continue;
      const double* o = planes + kk * w + N + t;
      const double* ak = a + 8 * kk * B + t;
      const double zp = kk + 1 < nk && kk + 1 < KZ ? f[kk + 1 < KZ ? kk + 1 : kk] : hi;
      const double zm = kk > 0 ? f[kk > 0 ? kk - 1 : 0] : lo;
      y[kk] = planar_row(ak[0], ak[B], ak[2 * B], ak[3 * B], ak[4 * B], ak[5 * B], ak[6 * B], f[kk],
                         o[1], o[-1], o[N], o[-N], zp, zm);
    }
  }
  // the end of a solve: the increments, the scalars and the algorithmic bytes, from the words an
  // iteration of the three kernel classes (pvw, stw: of weights, the momentum ones counted once)
  __device__ __forceinline__ void store(const Fields& F, const double (&xi)[KZ], KrylovScalars& k,
                                        bool ok, bool first_row, double iters, double pv, double pvw,
                                        double st, double stw, double xr) const {
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk)
      if (mine(kk)) F.x[s][c(kk)] = xi[kk];
    if (!ok && t == 0) {
      k.done = 1;
      k.status = HOSC_ECUDA;
    }
    if (t == 0 && (first_row || !ok)) {
      F.ks[s] = k;
      const double ni = N - 2, n3 = 8.0 * ni * ni * ni * iters, wt = s == 0 || s == 3 ? 1.0 : 0.0;
      atomicAdd(F.alg_bytes + HOSC_K_BICG_PV, n3 * (pv + wt * pvw));
      atomicAdd(F.alg_bytes + HOSC_K_BICG_ST, n3 * (st + wt * stw));
      atomicAdd(F.alg_bytes + HOSC_K_BICG_XR, n3 * xr);
    }
  }
};

template <int KZ>
__global__ void __launch_bounds__(KZ <= 4 ? kPlanarMost : kPlanarMost / 2)
    k_solve_planar(DevParams P, Fields F) {
  extern __shared__ double sh[];
  __shared__ KrylovScalars k;
  __shared__ double tot[2];
  __shared__ int failed;
  if (*F.halt) return;   // the same for every block
  Slab<KZ> b(P, sh);
  Exchange x = b.rows(F, 2, &failed);
  const int t = b.t, s = b.s;
  const double* rhs = F.rhs[s];
  double *R = F.r[s], *Q = F.pk[0][s], *V = F.vk[0][s];
  double r[KZ], xi[KZ], p[KZ], v[KZ], tv[KZ];
  b.load(F, r);
#pragma unroll
  for (int kk = 0; kk < KZ; ++kk) {
    p[kk] = r[kk];
    xi[kk] = v[kk] = tv[kk] = 0.0;
  }
  if (t == 0) {
    k = F.ks[s];
    failed = 0;
  }
  __syncthreads();
  bool ok = true;
  for (int it = 0; !k.done; ++it) {
    // p = r + beta (p - omega v), v = A p
    const bool first = it == 0;
    const double beta = k.beta;
    double d2[2] = {0.0, 0.0};
    if (first) {
      b.apply(p, v, [&](int c) { return rhs[c]; });
    } else {
#pragma unroll
      for (int kk = 0; kk < KZ; ++kk) p[kk] = fma(beta, p[kk], r[kk]);
      b.apply(p, v, [&](int c) { return fma(beta, __ldcg(Q + c), __ldcg(R + c)); });
    }
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk)
      if (b.mine(kk)) {
        V[b.c(kk)] = v[kk];
        const double r0 = b.r0(kk);
        d2[0] = fma(r0, v[kk], d2[0]);
        if (first) d2[1] = fma(r0, r0, d2[1]);
      }
    if (first) {
      ok = exchange<SumD, 2>(x, d2, tot);
    } else {
      double d1[1] = {d2[0]};
      ok = exchange<SumD, 1>(x, d1, tot);
    }
    if (!ok) break;
    if (t == 0) pv_scalars(k, tot[0], first ? tot[1] : 0.0, first);
    __syncthreads();
    if (k.done) break;
    // s = r - alpha v (kept in r), t = A s
    const double alpha = k.alpha;
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) r[kk] = fma(-alpha, v[kk], r[kk]);
    if (first)
      b.apply(r, tv, [&](int c) { return fma(-alpha, __ldcg(V + c), rhs[c]); });
    else
      b.apply(r, tv, [&](int c) { return fma(-alpha, __ldcg(V + c), __ldcg(R + c)); });
    double ds[2] = {0.0, 0.0};
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk)
      if (b.mine(kk)) {
        ds[0] = fma(tv[kk], r[kk], ds[0]);
        ds[1] = fma(tv[kk], tv[kk], ds[1]);
      }
    ok = exchange<SumD, 2>(x, ds, tot);
    if (!ok) break;
    if (t == 0) st_scalars(k, tot[0], tot[1]);
    __syncthreads();
    // x += alpha p + omega s, r = s - omega t; p - omega v for the next p
    const double omega = k.omega;
    double dr[2] = {0.0, 0.0};
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk)
      if (b.mine(kk)) {
        const int c = b.c(kk);
        xi[kk] = fma(omega, r[kk], fma(alpha, p[kk], xi[kk]));
        r[kk] = fma(-omega, tv[kk], r[kk]);
        p[kk] = fma(-omega, v[kk], p[kk]);
        R[c] = r[kk];
        Q[c] = p[kk];
        dr[0] = fma(b.r0(kk), r[kk], dr[0]);
        dr[1] = fma(r[kk], r[kk], dr[1]);
      }
    ok = exchange<SumD, 2>(x, dr, tot);
    if (!ok) break;
    split_xr_scalars<1>(P, &k, tot);
    __syncthreads();
  }
  b.store(F, xi, k, ok, x.mine == 0, k.iters, 6.0, 7.0, 3.0, 7.0, 8.0);
}

// BiCGSTAB(2): the five phases of a cycle (see the kernels of hosc_krylov.cu, whose arithmetic this is). A
// neighbour's value is r_0 - beta u_0 in U1, r_0 - alpha u_1 in R1, r_1 - beta u_1 in U2 and r_1 -
// alpha u_2 in R2, so that r_0 and u_0 are written after MR, u_1 after U1, r_1 after R1, u_2 after U2.
// A 34^3 box (9 cycles' iterations a step): 467 us a step with five launches a cycle, 308 so.
template <int KZ>
__global__ void __launch_bounds__(b2_threads(KZ)) k_solve_b2(DevParams P, Fields F) {
  extern __shared__ double sh[];
  __shared__ KrylovScalars k;
  __shared__ double tot[5];
  __shared__ int failed;
  if (*F.halt) return;   // the same for every block
  Slab<KZ> b(P, sh);
  Exchange x = b.rows(F, 5, &failed);
  const int t = b.t, s = b.s;
  const double* rhs = F.rhs[s];
  double *R0 = F.r[s], *R1 = F.pk[0][s], *U0 = F.u0[s], *U1 = F.vk[0][s], *U2 = F.u2[s];
  double r0[KZ], r1[KZ], r2[KZ], u0[KZ], u1[KZ], u2[KZ], xi[KZ];
  b.load(F, r0);
#pragma unroll
  for (int kk = 0; kk < KZ; ++kk) {
    u0[kk] = r0[kk];
    r1[kk] = r2[kk] = u1[kk] = u2[kk] = xi[kk] = 0.0;
  }
  if (t == 0) {
    k = F.ks[s];
    failed = 0;
  }
  __syncthreads();
  bool ok = true;
  for (int it = 0; !k.done; ++it) {
    const bool first = it == 0;
    {   // U1: u_0 = r_0 - beta u_0, u_1 = A u_0
      const double beta = k.beta;
      double d2[2] = {0.0, 0.0};
      if (first) {
        b.apply(u0, u1, [&](int c) { return rhs[c]; });
      } else {
#pragma unroll
        for (int kk = 0; kk < KZ; ++kk) u0[kk] = fma(-beta, u0[kk], r0[kk]);
        b.apply(u0, u1, [&](int c) { return fma(-beta, __ldcg(U0 + c), __ldcg(R0 + c)); });
      }
#pragma unroll
      for (int kk = 0; kk < KZ; ++kk)
        if (b.mine(kk)) {
          U1[b.c(kk)] = u1[kk];
          const double rt = b.r0(kk);
          d2[0] = fma(rt, u1[kk], d2[0]);
          if (first) d2[1] = fma(rt, rt, d2[1]);
        }
      if (first) {
        ok = exchange<SumD, 2>(x, d2, tot);
      } else {
        double d1[1] = {d2[0]};
        ok = exchange<SumD, 1>(x, d1, tot);
      }
      if (!ok) break;
      if (t == 0) pv_scalars(k, tot[0], first ? tot[1] : 0.0, first);
      __syncthreads();
      if (k.done) break;
    }
    {   // R1: r_0 -= alpha u_1, r_1 = A r_0; x += alpha u_0
      const double alpha = k.alpha;
      double d1[1] = {0.0};
#pragma unroll
      for (int kk = 0; kk < KZ; ++kk) {
        r0[kk] = fma(-alpha, u1[kk], r0[kk]);
        xi[kk] = fma(alpha, u0[kk], xi[kk]);
      }
      if (first)
        b.apply(r0, r1, [&](int c) { return fma(-alpha, __ldcg(U1 + c), rhs[c]); });
      else
        b.apply(r0, r1, [&](int c) { return fma(-alpha, __ldcg(U1 + c), __ldcg(R0 + c)); });
#pragma unroll
      for (int kk = 0; kk < KZ; ++kk)
        if (b.mine(kk)) {
          R1[b.c(kk)] = r1[kk];
          d1[0] = fma(b.r0(kk), r1[kk], d1[0]);
        }
      ok = exchange<SumD, 1>(x, d1, tot);
      if (!ok) break;
      if (t == 0) b2_r1_scalars(k, tot[0]);
      __syncthreads();
      if (k.done) break;
    }
    {   // U2: u_0 = r_0 - beta u_0, u_1 = r_1 - beta u_1, u_2 = A u_1
      const double beta = k.beta;
      double d1[1] = {0.0};
#pragma unroll
      for (int kk = 0; kk < KZ; ++kk) {
        u0[kk] = fma(-beta, u0[kk], r0[kk]);
        u1[kk] = fma(-beta, u1[kk], r1[kk]);
      }
      b.apply(u1, u2, [&](int c) { return fma(-beta, __ldcg(U1 + c), __ldcg(R1 + c)); });
#pragma unroll
      for (int kk = 0; kk < KZ; ++kk)
        if (b.mine(kk)) {
          U2[b.c(kk)] = u2[kk];
          d1[0] = fma(b.r0(kk), u2[kk], d1[0]);
        }
      ok = exchange<SumD, 1>(x, d1, tot);
      if (!ok) break;
      if (t == 0) pv_scalars(k, tot[0], 0.0, false);
      __syncthreads();
      if (k.done) break;
    }
    {   // R2: r_0 -= alpha u_1, r_1 -= alpha u_2, r_2 = A r_1; x += alpha u_0
      const double alpha = k.alpha;
      double d[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int kk = 0; kk < KZ; ++kk) {
        r0[kk] = fma(-alpha, u1[kk], r0[kk]);
        r1[kk] = fma(-alpha, u2[kk], r1[kk]);
        xi[kk] = fma(alpha, u0[kk], xi[kk]);
      }
      b.apply(r1, r2, [&](int c) { return fma(-alpha, __ldcg(U2 + c), __ldcg(R1 + c)); });
#pragma unroll
      for (int kk = 0; kk < KZ; ++kk)
        if (b.mine(kk)) {
          d[0] = fma(r1[kk], r1[kk], d[0]);
          d[1] = fma(r1[kk], r2[kk], d[1]);
          d[2] = fma(r2[kk], r2[kk], d[2]);
          d[3] = fma(r0[kk], r1[kk], d[3]);
          d[4] = fma(r0[kk], r2[kk], d[4]);
        }
      // the rows of the kernel have 20 slots: 16 groups
      ok = exchange<SumD, 5, row_groups<32>()>(x, d, tot);
      if (!ok) break;
      if (t == 0) b2_r2_scalars(k, tot);
      __syncthreads();
      if (k.done) break;
    }
    {   // MR
      const double g1 = k.g1, g2 = k.g2;
      double dr[2] = {0.0, 0.0};
#pragma unroll
      for (int kk = 0; kk < KZ; ++kk)
        if (b.mine(kk)) {
          xi[kk] = fma(g2, r1[kk], fma(g1, r0[kk], xi[kk]));
          r0[kk] = fma(-g2, r2[kk], fma(-g1, r1[kk], r0[kk]));
          u0[kk] = fma(-g2, u2[kk], fma(-g1, u1[kk], u0[kk]));
          R0[b.c(kk)] = r0[kk];
          U0[b.c(kk)] = u0[kk];
          dr[0] = fma(b.r0(kk), r0[kk], dr[0]);
          dr[1] = fma(r0[kk], r0[kk], dr[1]);
        }
      ok = exchange<SumD, 2>(x, dr, tot);
      if (!ok) break;
      if (t == 0) b2_mr_scalars(P, k, tot[0], tot[1]);
      __syncthreads();
    }
  }
  b.store(F, xi, k, ok, x.mine == 0, 0.5 * k.iters, 12.0, 14.0, 19.0, 14.0, 11.0);
}

// ------------------------------------------------------------------ mixed (interleaved float)
//
// A block has 256 interior columns (in the order of the register kernels) and up to KZ planes, with
// all four systems of a node in one float4.

constexpr int kSolveBlock = 256;

template <int KZ>
constexpr size_t mixed_state(int N) {   // operators, r_0, v, then KZ planes of 256 + 2 (N - 2) float4
  return 16 * ((size_t)4 * KZ * kSolveBlock + (size_t)KZ * (kSolveBlock + 2 * (N - 2))) +
         4 * (size_t)KZ * kSolveBlock;
}

template <int KZ>
__global__ void __launch_bounds__(kSolveBlock, 2) k_solve_mixed(DevParams P, Fields F) {
  constexpr int B = kSolveBlock;
  extern __shared__ float4 sh4[];
  __shared__ KrylovScalars ks[4];
  __shared__ Scal4 sc;
  __shared__ double tot[8];
  __shared__ int failed;
  if (*F.halt) return;   // the same for every block
  const int t = threadIdx.x, N = P.N, N2 = N * N, ni = N - 2, w = B + 2 * ni;
  const int q0 = (int)blockIdx.x * B, q = q0 + t;
  const int k0 = 1 + (int)blockIdx.y * P.ckz, nk = min(P.ckz, N - 1 - k0);
  Exchange x;
  x.nr = (int)(gridDim.x * gridDim.y);
  x.stride = 8;
  x.mine = (int)(blockIdx.x + gridDim.x * blockIdx.y);
  x.rows = F.exch;
  x.e = 0;
  x.failed = &failed;
  auto column_of = [&](int c) {   // node (i, j, 0) of interior column c
    const int j = c / ni;
    return 1 + c - j * ni + N * (j + 1);
  };
  const bool in = q < ni * ni;
  const int i = q % ni, c0 = (in ? column_of(q) : 0) + N2 * k0;
  const bool has_xp = i < ni - 1, has_xm = i > 0;
  // the column before or after the chunk whose value this thread fetches (2 ni <= B)
  const int hq = t < ni ? q0 - ni + t : q0 + B + (t - ni), hs = t < ni ? t : B + t;
  const bool has_halo = t < 2 * ni, hin = has_halo && hq >= 0 && hq < ni * ni;
  const int hc = (hin ? column_of(hq) : 0) + N2 * k0;
  const bool below = in && k0 > 1, above = in && k0 + nk < N - 1;
  float4* om = sh4;                 // operators, r_0 and v of plane kk at kk B + t
  float4* oe = om + KZ * B;
  float4* r0 = oe + KZ * B;
  float4* vs = r0 + KZ * B;
  float4* planes = vs + KZ * B;     // plane kk: columns q0 - ni .. q0 + B + ni
  float* ol = (float*)(planes + KZ * w);
  const float4 zero = f4(0.f);
  float4 r[KZ], p[KZ], tv[KZ];
#pragma unroll
  for (int kk = 0; kk < KZ; ++kk) {
    r[kk] = p[kk] = tv[kk] = zero;
    if (in && kk < nk) {
      const int c = c0 + N2 * kk;
      r[kk] = p[kk] = F.kr0[c];
      r0[kk * B + t] = r[kk];
      om[kk * B + t] = F.kwm[c];
      oe[kk * B + t] = F.kwe[c];
      ol[kk * B + t] = F.kL[c];
    }
  }
  if (t < 4) ks[t] = F.ks[t];
  if (t == 0) failed = 0;
  __syncthreads();
  // the operators on own values f (registers) and the others' values val(c): out(kk, y) of each plane
  auto stencil = [&](const float4 (&f)[KZ], bool ene, auto val, auto out) {
    const float4 lo = below ? val(c0 - N2) : zero, hi = above ? val(c0 + N2 * nk) : zero;
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) {
      const float4 h = hin && kk < nk ? val(hc + N2 * kk) : zero;
      planes[kk * w + ni + t] = f[kk];   // zero past the last column
      if (has_halo) planes[kk * w + hs] = h;
      if (KZ > 2 && kk % 2) asm volatile("" ::: "memory");
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) {
      if (!in || kk >= nk) continue;
      const float4* o = planes + kk * w + ni + t;
      Op4 op;
      op.m = om[kk * B + t];
      op.e = ene ? oe[kk * B + t] : zero;
      op.L = ol[kk * B + t];
      const float4 zp = kk + 1 < nk && kk + 1 < KZ ? f[kk + 1 < KZ ? kk + 1 : kk] : hi;
      const float4 zm = kk > 0 ? f[kk > 0 ? kk - 1 : 0] : lo;
      out(kk, apply_op(P, op, f[kk], has_xp ? o[1] : zero, has_xm ? o[-1] : zero, o[ni], o[-ni],
                       zp, zm));
      asm volatile("" ::: "memory");   // one plane's operands in registers at a time
    }
  };
  double bytes[3] = {0.0, 0.0, 0.0};
  bool ok = true;
  bool any = false;   // an iterate has been written
  for (int it = 0;; ++it) {
    const bool first = it == 0;
    load_scalars(ks, sc);
    if (sc.all_done) break;
    // p = r + beta (p - omega v), v = A p
    bool ene = !sc.done[3];
    {
      const float4 b = sc.b;
      FF acc[8] = {};
      auto out = [&](int kk, const float4& y) {
        F.kv[0][c0 + N2 * kk] = y;
        vs[kk * B + t] = y;
        const float4 z = r0[kk * B + t];
        ff_dot4(acc, z, y);
        if (first) ff_dot4(acc + 4, z, z);
      };
      if (first) {
        stencil(p, ene, [&](int c) { return F.kr0[c]; }, out);
      } else {
#pragma unroll
        for (int kk = 0; kk < KZ; ++kk) p[kk] = fma4(b, p[kk], r[kk]);
        stencil(p, ene, [&](int c) { return fma4(b, __ldcg(F.kp[0] + c), __ldcg(F.kr + c)); }, out);
      }
      bytes[0] += (first ? 3.0 : 6.0) + op_words(ene);
      if (first) {
        ok = exchange<SumFF, 8>(x, acc, tot);
      } else {
        FF a4[4] = {acc[0], acc[1], acc[2], acc[3]};
        ok = exchange<SumFF, 4>(x, a4, tot);
      }
      if (!ok) break;
      finish_pv(ks, tot, first);
    }
    load_scalars(ks, sc);
    if (sc.all_done) break;
    // s = r - alpha v (kept in r), t = A s
    ene = !sc.done[3];
    {
      const float4 ma = neg4(sc.a);
      FF acc[8] = {};
#pragma unroll
      for (int kk = 0; kk < KZ; ++kk)
        if (in && kk < nk) r[kk] = fma4(ma, vs[kk * B + t], r[kk]);
      const float4* R = first ? F.kr0 : F.kr;
      stencil(r, ene, [&](int c) { return fma4(ma, __ldcg(F.kv[0] + c), __ldcg(R + c)); },
              [&](int kk, const float4& y) {
                tv[kk] = y;
                ff_dot4(acc, y, r[kk]);
                ff_dot4(acc + 4, y, y);
              });
      bytes[1] += 3.0 + op_words(ene);
      ok = exchange<SumFF, 8>(x, acc, tot);
      if (!ok) break;
      finish_st(ks, tot);
    }
    load_scalars(ks, sc);
    // x += alpha p + omega s, r = s - omega t; p - omega v for the next p
    {
      const float4 a = sc.a, o = sc.om, mo = neg4(sc.om);
      FF acc[8] = {};
      bytes[2] += first ? 6.0 : 8.0;
      any = true;
#pragma unroll
      for (int kk = 0; kk < KZ; ++kk)
        if (in && kk < nk) {
          const int c = c0 + N2 * kk;
          F.kx[c] = fma4(o, r[kk], fma4(a, p[kk], first ? zero : F.kx[c]));
          r[kk] = fma4(mo, tv[kk], r[kk]);
          p[kk] = fma4(mo, vs[kk * B + t], p[kk]);
          F.kr[c] = r[kk];
          F.kp[0][c] = p[kk];
          ff_dot4(acc, r0[kk * B + t], r[kk]);
          ff_dot4(acc + 4, r[kk], r[kk]);
        }
      ok = exchange<SumFF, 8>(x, acc, tot);
      if (!ok) break;
      split_xr_scalars<4>(P, ks, tot);
    }
    __syncthreads();   // two warps write the scalars
  }
  if (!any && in)   // every right-hand side is zero (or none to solve): zero increments
    for (int kk = 0; kk < nk; ++kk) F.kx[c0 + N2 * kk] = zero;
  if (!ok && t < 4) {
    ks[t].done = 1;
    ks[t].status = HOSC_ECUDA;
  }
  if (x.mine == 0 || !ok) {
    if (t < 4) F.ks[t] = ks[t];
    if (t < 3) atomicAdd(F.alg_bytes + HOSC_K_BICG_PV + t, bytes4(P, bytes[t]));
  }
}

// ------------------------------------------------------------------ host

typedef void (*SolveFn)(DevParams, Fields);

int template_planes(int z) { return z <= 1 ? 1 : z <= 2 ? 2 : z <= 4 ? 4 : 8; }

SolveFn planar_fn(int solver, int B, int z, int N, size_t* smem) {
  const int KZ = template_planes(z);
  *smem = KZ == 1 ? planar_state<1>(N, B) : KZ == 2 ? planar_state<2>(N, B)
          : KZ == 4 ? planar_state<4>(N, B) : planar_state<8>(N, B);
  if (solver == 1) {
    if (B > b2_threads(KZ)) return nullptr;
    return KZ == 1 ? k_solve_b2<1> : KZ == 2 ? k_solve_b2<2>
           : KZ == 4 ? k_solve_b2<4> : k_solve_b2<8>;
  }
  // eight planes: registers for 256 threads; fewer than 160 leave the FP64 pipe idle (31^3 with 128: 20.7
  // us an iteration, with 160 18.8)
  if (KZ > 4 && (B > kPlanarMost / 2 || B < 160)) return nullptr;
  return KZ == 1 ? k_solve_planar<1> : KZ == 2 ? k_solve_planar<2>
         : KZ == 4 ? k_solve_planar<4> : k_solve_planar<8>;
}
SolveFn mixed_fn(int KZ, int N, size_t* smem) {
  *smem = KZ == 1 ? mixed_state<1>(N) : KZ == 2 ? mixed_state<2>(N) : mixed_state<4>(N);
  return KZ == 1 ? k_solve_mixed<1> : KZ == 2 ? k_solve_mixed<2> : KZ == 4 ? k_solve_mixed<4> : nullptr;
}

// Blocks of fn that are resident at once, 0 when it cannot run so.
long resident(SolveFn fn, int threads, size_t smem) {
  if (!fn || smem > 200 * 1024) return 0;
  int occ = 0;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return (long)occ * device_sms();
}

void launch_cooperative(SolveFn fn, dim3 grid, int threads, size_t smem, cudaStream_t s,
                        const DevParams& P, const Fields& F) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, fn, P, F);
}

}  // namespace

// Shapes of the one-launch solves: the least modelled time of an iteration among the shapes whose
// blocks are all resident. False when none is: the vectors do not fit on the chip.
//
// FP64: microseconds of the busiest SM's FP64 instructions and of the exchange's rows, and what a form
// of KZ planes costs beside them (one plane: both neighbours of every node come from memory; more than
// two: registers). Fitted to every shape from 64 to 512 threads at 9^3 to 41^3; the chosen shape is
// the fastest there or within 0.8 us of it. 21^3 (128, 3) -> (160, 2): 14.4 -> 12.5 us an iteration,
// 25^3 (128, 4) -> (224, 2): 16.8 -> 13.8, 37^3 (256, 5) -> (352, 4): 23.1 -> 21.4. Mixed precision:
// planes of the busiest SM and rows.
bool solve_shape_planar(int N, int solver, int* pb, int* pkz) {
  // the answer for the last grid and device of this thread: asked at every set-up and every
  // allocation-free solve
  static thread_local struct Last { int N, device, pb, pkz; } of[2] = {{0, -1, 0, 0}, {0, -1, 0, 0}};
  Last& last = of[solver];
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess) return false;
  if (last.N == N && last.device == device) {
    *pb = last.pb;
    *pkz = last.pkz;
    return last.pb > 0;
  }
  const int sms = device_sms(), ni = N - 2;
  double best = 1e300;
  last = {N, device, 0, 0};
  for (int B = 64; B <= kPlanarMost; B += 32) {
    if (2 * N > B) continue;
    const long chunks = (N * (long)N + B - 1) / B;
    for (int z = 1; z <= 8 && z <= ni; ++z) {
      const long rows = chunks * ((ni + z - 1) / z);
      if (rows > kSolveRows) continue;
      const int KZ = template_planes(z);
      const double work = B / 32.0 * (12.0 * z + 20.0) + 2.0 * ((2 * N + 31) / 32) * z;
      const double cost = 0.0094 * work * (double)((4 * rows + sms - 1) / sms) + 0.06 * rows +
                          (KZ == 1 ? 0.7 : KZ == 2 ? 0.0 : KZ == 4 ? 1.2 : 1.6);
      if (cost >= best) continue;
      size_t smem = 0;
      const SolveFn fn = planar_fn(solver, B, z, N, &smem);
      if (resident(fn, B, smem) < 4 * rows) continue;
      best = cost;
      last.pb = *pb = B;
      last.pkz = *pkz = z;
    }
  }
  return best < 1e300;
}

bool solve_shape_mixed(int N, int* kblock, int* kz) {
  static thread_local struct { int N, device, kblock, kz; } last = {0, -1, 0, 0};
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess) return false;
  if (last.N == N && last.device == device) {
    *kblock = last.kblock;
    *kz = last.kz;
    return last.kz > 0;
  }
  last = {N, device, 0, 0};
  const int sms = device_sms(), ni = N - 2;
  if (2 * ni > kSolveBlock) return false;
  const long chunks = ((long)ni * ni + kSolveBlock - 1) / kSolveBlock;
  double best = 1e300;
  for (int z = 1; z <= 4 && z <= ni; ++z) {
    const long rows = chunks * ((ni + z - 1) / z);
    if (rows * 2 * 8 > kExchValues) continue;
    const double cost = (z + 1.5) * (double)((rows + sms - 1) / sms) + 0.004 * rows;
    if (cost >= best) continue;
    size_t smem = 0;
    const SolveFn fn = mixed_fn(template_planes(z), N, &smem);
    if (resident(fn, kSolveBlock, smem) < rows) continue;
    best = cost;
    last.kblock = *kblock = kSolveBlock;
    last.kz = *kz = z;
  }
  return best < 1e300;
}

void launch_solve(const DevParams& P, const Fields& F, cudaStream_t s) {
  const int ni = P.N - 2;
  size_t smem = 0;
  if (P.krylov_fp32) {
    const SolveFn fn = mixed_fn(template_planes(P.ckz), P.N, &smem);
    const dim3 g((ni * ni + kSolveBlock - 1) / kSolveBlock, (ni + P.ckz - 1) / P.ckz);
    launch_cooperative(fn, g, kSolveBlock, smem, s, P, F);
  } else {
    const SolveFn fn = planar_fn(P.solver, P.pb, P.pkz, P.N, &smem);
    const dim3 g(4u * ((P.N * P.N + P.pb - 1) / P.pb), (ni + P.pkz - 1) / P.pkz);
    launch_cooperative(fn, g, P.pb, smem, s, P, F);
  }
}

}  // namespace hosc
