// Unpreconditioned BiCGSTAB (van der Vorst) on the four HOSC systems of one step (Punia & Ray,
// arXiv:2411.06563, Sec. 2.2: the implicit seven-point systems are solved with BiCGSTAB without
// preconditioning).
//
// The four systems (u, v, w with the shared momentum operator, theta with the energy operator)
// advance together, each with its own scalars. The operator is applied matrix-free from the seven
// weights per node written by the right-hand-side kernel. Unknown is the increment
// x = chi^{n+1} - chi^n, zero on the walls, started at x = 0, so r_0 = dt (R - B chi^n); the
// shadow residual is r_0 (kept in rhs[]). Stop when ||r_k||_2 <= tol ||r_0||_2.
//
// One iteration = three kernels; each ends with a last-block reduction that finalises the scalar
// the next kernel needs (alpha, omega, beta / convergence). No kernel waits on another block.
//
// Two storage forms. FP64 (planar): one array per system and per weight; a block takes one system.
// Mixed precision (interleaved, float): one float4 per node holds the four systems, and a thread owns
// one interior (i, j) column over a segment of kz planes, keeping the z-neighbours in registers as
// it marches; its dot-product terms accumulate in float-float over the segment before the block
// reduction.

#include <math.h>

#include "hosc_device.cuh"
#include "hosc_internal.h"
#include "hosc_krylov4.cuh"

namespace hosc {

namespace {

// Algorithmic bytes of one launch: every array element the active systems touch, once.
__device__ __forceinline__ double launch_bytes(const DevParams& P, const int done[4],
                                               double per_system_words, double coeff_words,
                                               double word_bytes) {
  const double ni = (double)(P.N - 2);
  const int nm = !done[0] + !done[1] + !done[2], ne = !done[3];
  const double words = per_system_words * (nm + ne) + coeff_words * ((nm > 0) + ne);
  return word_bytes * ni * ni * ni * words;
}

// End of one pass of the captured BiCGSTAB loop body: continue while a system is iterating.
// Bounded: a system is done at max_lin_iter at the latest. A launch of its own: with the call in the
// iteration's last kernel a pass took about 5 us longer (41^3 FP64 step 976 -> 1030 us).
__global__ void k_loop_cond(const KrylovScalars* ks, cudaGraphConditionalHandle handle) {
  const int done = threadIdx.x < 4 ? ks[threadIdx.x].done : 1;
  const int all = __all_sync(0xffffffffu, done);
  if (threadIdx.x == 0) cudaGraphSetConditional(handle, !all);
}

// ------------------------------------------------------------------ planar FP64 solve
//
// GB300's FP64 pipe takes 16 cycles of an SM for a warp's instruction, so these kernels are bound by
// the number of FP64 instructions a node, not by bytes. A kernel that applies an operator to a vector
// combined on the fly (r + beta (p - omega v), r - alpha v, ...) evaluated that vector at all seven
// points of every node: 14 instructions beside the operator's 7 for p/v. Here a block takes one system,
// B consecutive nodes of the plane (i + N j, walls included: they are zero) and pkz planes; it
// evaluates the vector once at its nodes and at the N nodes before and after them, puts the plane in
// shared memory (two planes, one barrier a plane) and keeps the planes above and below in registers:
// 2 (1 + 2N/B) + 7 + 1 instructions for p/v. One system a block spreads the small grids over four
// times the SMs; the three momentum blocks of a chunk are neighbours in the grid, so their weights
// come from L2. A block's partial goes to its row's slot of its system; the last block of the launch
// sums all rows. The shape (B, pkz) has the least modelled load of the busiest SM (planar_shape).
// Measured, alone: p/v 137 -> 82.1 us, s/t 117 -> 71.6, x/r 74.5 -> 45.7 at 91^3; 14.4 -> 8.6, 14.2 ->
// 7.4, 12.3 -> 9.3 at 21^3.
//
// BiCGSTAB (solver = 0): p/v, s/t, x/r. BiCGSTAB(2) (Sleijpen and Fokkema's BiCGSTAB(ell) with
// ell = 2; shadow residual rt = r_0 = rhs), one cycle in five kernels:
//   U1  u_0 <- r_0 - beta u_0 (on the fly at the stencil), u_1 = A u_0;       alpha = rho/(rt.u_1)
//   R1  r_0 <- r_0 - alpha u_1 (on the fly), r_1 = A r_0; u_0 <- r_0 - beta u_0 and x += alpha u_0
//       (pointwise, with the r_0 of U1);                   rho_1 = rt.r_1, beta = alpha rho_1/rho
//   U2  u_0 <- r_0 - beta u_0 (pointwise); u_1 <- r_1 - beta u_1 (on the fly), u_2 = A u_1;
//                                                          alpha = rho/(rt.u_2)
//   R2  r_0 -= alpha u_1 (pointwise); r_1 <- r_1 - alpha u_2 (on the fly), r_2 = A r_1;
//       x += alpha u_0; the five inner products of r_0, r_1, r_2 give the minimal-residual
//       coefficients: tau = (r_1.r_2)/(r_1.r_1), gamma'_1 = (r_0.r_1)/(r_1.r_1), gamma_2 =
//       gamma'_2 = (r_0.r_2 - tau r_0.r_1)/(r_2.r_2 - tau r_1.r_2), gamma_1 = gamma'_1 - tau gamma_2
//   MR  x += gamma_1 r_0 + gamma_2 r_1; r_0 -= gamma_1 r_1 + gamma_2 r_2; u_0 -= gamma_1 u_1 +
//       gamma_2 u_2 (the Gram-Schmidt step folded into the coefficients); rho <- -omega rho,
//       rho_1 = rt.r_0, beta = alpha rho_1/rho, rho = rho_1, convergence on ||r_0||.
// Buffers per system: r_0 in r / t (ping-pong by cycle: R1 reads one and writes the other, the
// stencil reads the old r_0 at the neighbours), r_1 in pk[0] (R1) then pk[1] (R2), u_1 in vk[0]
// (U1) then vk[1] (U2), u_0, r_2, u_2 in their own arrays. A kernel writes no array that it reads
// at a neighbour.
//
// The first iteration (FIRST) reads rhs for the residual, no search direction and no iterate, so that
// nothing has to be initialised. Where the walls of rhs are not known to be zero
// (rhs_copied: the caller's arrays of the allocation-free solve) the residual is a copy.

enum { PL_PV, PL_ST, PL_U1, PL_R1, PL_U2, PL_R2, PL_XR, PL_MR };

// Dot products of a launch, per system, and the slots of a row of partials.
// (p/v and U1: r_0 . r_0 beside r_0 . v, used in the first iteration)
constexpr int pl_dots(int kind, bool first) {
  return kind == PL_R2 ? 5 : kind == PL_ST || kind >= PL_XR ? 2 : kind <= PL_U1 && first ? 2 : 1;
}
constexpr int pl_slots(int kind, bool first) {
  return kind == PL_R2 ? 20 : 4 * pl_dots(kind, first);
}

// The scalars that a launch of this kind leaves, and its algorithmic bytes.
template <int KIND>
__device__ __forceinline__ void planar_finish(const DevParams& P, const Fields& F,
                                              const double* tot, bool first,
                                              const int (&done)[4]) {
  if (KIND == PL_PV || KIND == PL_U1) finish_pv(F.ks, tot, first);
  if (KIND == PL_U2) finish_pv(F.ks, tot, false);
  if (KIND == PL_ST) finish_st(F.ks, tot);
  if (KIND == PL_XR) finish_xr(P, F.ks, tot);
  const int q = threadIdx.x;
  if (KIND == PL_R1 && q < 4) b2_r1_scalars(F.ks[q], tot[q]);
  if (KIND == PL_R2 && q < 4) b2_r2_scalars(F.ks[q], tot + 5 * q);
  if (KIND == PL_MR && q < 4) b2_mr_scalars(P, F.ks[q], tot[q], tot[4 + q]);
  constexpr int cls = KIND == PL_PV || KIND == PL_U1 || KIND == PL_U2 ? HOSC_K_BICG_PV
                      : KIND >= PL_XR                                 ? HOSC_K_BICG_XR
                                                                      : HOSC_K_BICG_ST;
  constexpr double words[8] = {6.0, 3.0, 4.0, 9.0, 8.0, 10.0, 8.0, 11.0};
  count_bytes(F, cls, launch_bytes(P, done, words[KIND], KIND >= PL_XR ? 0.0 : 7.0,
                                   sizeof(double)));
}

// What every planar kernel starts with: which system, chunk and planes this block has.
struct Planar {
  int s;          // system
  bool live;      // it still iterates
  int l;          // this thread's node of the plane, i + N j
  bool inner;     // inside the walls of the plane
  int k0, k1;     // planes
  unsigned row, rows;
};

// False when every system is done (the same for every block). The kernels that write x run in the
// first iteration all the same unless the sequence has been halted: a system with a zero right-hand
// side gets its zero increment.
template <int KIND, bool FIRST>
__device__ __forceinline__ bool planar_block(const DevParams& P, const Fields& F, Planar& b,
                                             int (&done)[4]) {
  b.s = (int)(blockIdx.x & 3u);
#pragma unroll
  for (int q = 0; q < 4; ++q) done[q] = F.ks[q].done;
  if (done[0] & done[1] & done[2] & done[3]) {
    if (!(FIRST && (KIND == PL_XR || KIND == PL_R1)) || *F.halt) return false;
  }
  b.live = !(b.s == 0 ? done[0] : b.s == 1 ? done[1] : b.s == 2 ? done[2] : done[3]);
  const int N = P.N;
  b.l = (int)(blockIdx.x >> 2) * (int)blockDim.x + (int)threadIdx.x;
  const int j = b.l / N, i = b.l - j * N;
  b.inner = i > 0 && i < N - 1 && j > 0 && j < N - 1;
  b.k0 = 1 + (int)blockIdx.y * P.pkz;
  b.k1 = min(b.k0 + P.pkz, N - 1);
  b.row = (blockIdx.x >> 2) + (gridDim.x >> 2) * blockIdx.y;
  b.rows = (gridDim.x >> 2) * gridDim.y;
  return true;
}

template <int KIND, bool FIRST>
__device__ __forceinline__ void planar_end(const DevParams& P, const Fields& F, const Planar& b,
                                           const double (&dot)[pl_dots(KIND, FIRST)],
                                           const int (&done)[4]) {
  constexpr int M = pl_dots(KIND, FIRST), S = pl_slots(KIND, FIRST);
  const double mine = block_total<SumD, M>(dot);
  if (threadIdx.x < M) {
    const int slot = M == 5 ? 5 * b.s + (int)threadIdx.x : b.s + 4 * (int)threadIdx.x;
    F.rb.red[(long)b.row * row_stride<S>() + slot] = mine;
  }
  if (const double* tot = last_block_total<SumD, S>(F.rb, b.row, b.rows, 4u))
    planar_finish<KIND>(P, F, tot, FIRST, done);
}

// The planar kernels that apply an operator. pp: parity of the iteration (BiCGSTAB) or cycle.
template <int KIND, bool FIRST>
__global__ void __launch_bounds__(kPlanarMost, 2) k_planar(DevParams P, Fields F, int pp) {
  extern __shared__ double planes[];   // two planes of N + B + N values
  pdl_wait_and_release();
  Planar b;
  int done[4];
  if (!planar_block<KIND, FIRST>(P, F, b, done)) return;
  constexpr int L = pl_dots(KIND, FIRST) - 1;
  double dot[L + 1] = {};
  if (b.live) {   // the same for the whole block
    const int s = b.s, N = P.N, N2 = N * N, t = threadIdx.x, B = blockDim.x, w = B + 2 * N;
    const double alpha = F.ks[s].alpha, beta = F.ks[s].beta, omega = F.ks[s].omega;
    const double* rhs = F.rhs[s];
    // the vector that the operator is applied to: X - q Y (p/v: X + beta (Z - omega Y))
    const double *X, *Y, *Z = nullptr;
    double q;
    if (KIND == PL_PV) { X = F.r[s]; Y = F.vk[pp][s]; Z = F.pk[pp][s]; q = omega; }
    if (KIND == PL_ST) { X = F.r[s]; Y = F.vk[1 - pp][s]; q = alpha; }
    if (KIND == PL_U1) { X = pp ? F.t[s] : F.r[s]; Y = F.u0[s]; q = beta; }
    if (KIND == PL_R1) { X = pp ? F.t[s] : F.r[s]; Y = F.vk[0][s]; q = alpha; }
    if (KIND == PL_U2) { X = F.pk[0][s]; Y = F.vk[0][s]; q = beta; }
    if (KIND == PL_R2) { X = F.pk[0][s]; Y = F.u2[s]; q = alpha; }
    if (FIRST && KIND <= PL_R1 && !P.rhs_copied) X = rhs;   // a copy in r otherwise
    constexpr bool plain = FIRST && (KIND == PL_PV || KIND == PL_U1);   // no search direction yet
    auto value = [&](int c) {
      const double x = X[c];
      if (plain) return x;
      if (KIND == PL_PV) return fma(beta, fma(-q, Y[c], Z[c]), x);
      return fma(-q, Y[c], x);
    };
    const double* const* A = s < 3 ? F.Am : F.Ae;
    const double *a0 = A[0], *a1 = A[1], *a2 = A[2], *a3 = A[3], *a4 = A[4], *a5 = A[5], *a6 = A[6];
    const bool mine = b.l < N2;
    const int l0 = b.l - t;
    double lo = mine ? value(b.l + N2 * (b.k0 - 1)) : 0.0;
    double mid = mine ? value(b.l + N2 * b.k0) : 0.0;
    for (int k = b.k0; k < b.k1; ++k) {
      const int c = b.l + N2 * k;
      double* pl = planes + (k & 1) * w;
      pl[N + t] = mid;
      for (int h = t; h < 2 * N; h += B) {   // the N nodes before the chunk and after it
        const int hl = h < N ? l0 - N + h : l0 + B + (h - N);
        pl[h < N ? h : B + h] = hl >= 0 && hl < N2 ? value(hl + N2 * k) : 0.0;
      }
      const double hi = mine ? value(c + N2) : 0.0;
      // the weights' loads in flight with the halo's, before the barrier: p/v and s/t at 91^3 together
      // 159.4 -> 154.8 us
      double e0 = 0.0, e1 = 0.0, e2 = 0.0, e3 = 0.0, e4 = 0.0, e5 = 0.0, e6 = 0.0;
      if (b.inner) {
        e0 = a0[c], e1 = a1[c], e2 = a2[c], e3 = a3[c], e4 = a4[c], e5 = a5[c], e6 = a6[c];
      }
      __syncthreads();
      if (b.inner) {
        const double* o = pl + N + t;
        const double y = planar_row(e0, e1, e2, e3, e4, e5, e6, mid, o[1], o[-1], o[N], o[-N], hi, lo);
        if (KIND == PL_PV) {
          F.pk[1 - pp][s][c] = mid;
          F.vk[1 - pp][s][c] = y;
          const double r0 = rhs[c];
          dot[0] = fma(r0, y, dot[0]);
          if (FIRST) dot[L] = fma(r0, r0, dot[L]);
        } else if (KIND == PL_ST) {
          F.t[s][c] = y;
          dot[0] = fma(y, mid, dot[0]);
          dot[L] = fma(y, y, dot[L]);
        } else if (KIND == PL_U1) {
          F.vk[0][s][c] = y;
          const double r0 = rhs[c];
          dot[0] = fma(r0, y, dot[0]);
          if (FIRST) dot[L] = fma(r0, r0, dot[L]);
        } else if (KIND == PL_R1) {
          (pp ? F.r[s] : F.t[s])[c] = mid;
          F.pk[0][s][c] = y;
          const double r0 = X[c], u0 = FIRST ? r0 : fma(-beta, F.u0[s][c], r0);
          F.u0[s][c] = u0;
          F.x[s][c] = fma(alpha, u0, FIRST ? 0.0 : F.x[s][c]);
          dot[0] = fma(rhs[c], y, dot[0]);
        } else if (KIND == PL_U2) {
          const double* r0 = pp ? F.r[s] : F.t[s];   // written by R1
          F.u0[s][c] = fma(-beta, F.u0[s][c], r0[c]);
          F.vk[1][s][c] = mid;
          F.u2[s][c] = y;
          dot[0] = fma(rhs[c], y, dot[0]);
        } else {
          double* r0 = pp ? F.r[s] : F.t[s];
          const double r0c = fma(-alpha, F.vk[1][s][c], r0[c]);
          r0[c] = r0c;
          F.pk[1][s][c] = mid;
          F.r2[s][c] = y;
          F.x[s][c] = fma(alpha, F.u0[s][c], F.x[s][c]);
          dot[0] = fma(mid, mid, dot[0]);   // L = 4 here
          dot[L / 4] = fma(mid, y, dot[L / 4]);
          dot[L / 2] = fma(y, y, dot[L / 2]);
          dot[3 * L / 4] = fma(r0c, mid, dot[3 * L / 4]);
          dot[L] = fma(r0c, y, dot[L]);
        }
      }
      lo = mid;
      mid = hi;
    }
  } else if (KIND == PL_R1 && FIRST && b.inner) {
    for (int k = b.k0; k < b.k1; ++k) F.x[b.s][b.l + P.N * P.N * k] = 0.0;
  }
  planar_end<KIND, FIRST>(P, F, b, dot, done);
}

// The pointwise ends: x/r (s = r - alpha v; x += alpha p + omega s; r = s - omega t; r0.r, r.r) and MR.
template <int KIND, bool FIRST>
__global__ void __launch_bounds__(kPlanarMost) k_planar_end(DevParams P, Fields F, int pp) {
  pdl_wait_and_release();
  Planar b;
  int done[4];
  if (!planar_block<KIND, FIRST>(P, F, b, done)) return;
  double dot[2] = {};
  if (b.live && b.inner) {
    const int s = b.s, N2 = P.N * P.N;
    const double* rhs = F.rhs[s];
    double* x = F.x[s];
    if (KIND == PL_XR) {
      const double a = F.ks[s].alpha, om = F.ks[s].omega;
      const double *v = F.vk[1 - pp][s], *p = F.pk[1 - pp][s], *tv = F.t[s];
      const double* ro = FIRST ? rhs : F.r[s];
      double* r = F.r[s];
#pragma unroll 2
      for (int k = b.k0; k < b.k1; ++k) {
        const int c = b.l + N2 * k;
        const double sv = fma(-a, v[c], ro[c]);
        x[c] = fma(om, sv, fma(a, p[c], FIRST ? 0.0 : x[c]));
        const double rn = fma(-om, tv[c], sv);
        r[c] = rn;
        dot[0] = fma(rhs[c], rn, dot[0]);
        dot[1] = fma(rn, rn, dot[1]);
      }
    } else {
      const double g1 = F.ks[s].g1, g2 = F.ks[s].g2;
      double *r0 = pp ? F.r[s] : F.t[s], *u0 = F.u0[s];
      const double *r1 = F.pk[1][s], *r2 = F.r2[s], *u1 = F.vk[1][s], *u2 = F.u2[s];
#pragma unroll 2
      for (int k = b.k0; k < b.k1; ++k) {
        const int c = b.l + N2 * k;
        const double r0c = r0[c], r1c = r1[c];
        x[c] = fma(g2, r1c, fma(g1, r0c, x[c]));
        const double rn = fma(-g2, r2[c], fma(-g1, r1c, r0c));
        r0[c] = rn;
        u0[c] = fma(-g2, u2[c], fma(-g1, u1[c], u0[c]));
        dot[0] = fma(rhs[c], rn, dot[0]);
        dot[1] = fma(rn, rn, dot[1]);
      }
    }
  } else if (KIND == PL_XR && FIRST && b.inner) {
    for (int k = b.k0; k < b.k1; ++k) F.x[b.s][b.l + P.N * P.N * k] = 0.0;
  }
  planar_end<KIND, FIRST>(P, F, b, dot, done);
}

// Start of a solve whose right-hand sides no kernel of this library wrote: the scalars, and the copy of
// rhs that the first residual is read from.
__global__ void __launch_bounds__(kThreads) k_planar_start(DevParams P, Fields F) {
  const int N = P.N, ni = N - 2, t = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (t < 4) start_system(P, F, t);
  if (t >= ni * ni * ni) return;
  const int q = t / ni, c = 1 + t - q * ni + N * (1 + q % ni + N * (1 + q / ni));
#pragma unroll
  for (int s = 0; s < 4; ++s) F.r[s][c] = F.rhs[s][c];
}

// ------------------------------------------------------------- merged iteration (two kernels)
//
// The same BiCGSTAB with two kernels per iteration i. k6_a applies the end of iteration i-1
// (s = r - alpha v, x += alpha p + omega s, r_i = s - omega t) and the start of iteration i
// (p_i = r_i + beta (p - omega v), v_i = A p_i) in one pass, recomputing r_i and p_i at the
// stencil's nodes; its partials give rho_i = r_0 . r_i, alpha_i = rho_i / (r_0 . v_i) and the
// true ||r_i|| (the convergence test, one kernel later than in the three-kernel form). k6_b
// computes s, t = A s and the dot products t.s, t.t, r_0.s, r_0.t, from which
// omega_i = t.s / t.t and r_0 . r_{i+1} = r_0.s - omega_i r_0.t follow without another pass;
// then beta_{i+1} = (r_0 . r_{i+1} / rho_i)(alpha_i / omega_i). The residual ping-pongs
// (kr, kr1) since k6_a reads it at the neighbours while writing it.

__global__ void __launch_bounds__(kThreads) k6_init(DevParams P, Fields F) {
  const int N = P.N;
  const int n3 = N * N * N;
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  FF acc[4] = {};
  if (c < n3) {
    const int i = c % N, j = (c / N) % N, k = c / (N * N);
    const bool inner = i > 0 && j > 0 && k > 0 && i < N - 1 && j < N - 1 && k < N - 1;
    const float4 z = f4(0.f);
    const float4 r = inner ? F.kr0[c] : z;
    F.kr[c] = r;
    F.kr1[c] = z;
    F.kx[c] = z;
    F.kt[c] = z;
    F.kp[0][c] = z;
    F.kp[1][c] = z;
    F.kv[0][c] = z;
    F.kv[1][c] = z;
    ff_dot4(acc, r, r);
  }
  if (const double* tot = grid_total<SumFF, 4>(acc, F.rb, blockIdx.x, gridDim.x))
    finish_init(P, F, tot);
}

template <int MinB>
__global__ void __launch_bounds__(256, MinB) k6_a(DevParams P, Fields F, int pp) {
  __shared__ Scal4 sc;
  load_scalars(F.ks, sc);
  if (sc.all_done) return;   // uniform over the grid
  const bool ene = !sc.done[3];   // the energy system still iterates (uniform)
  const int N = P.N, N2 = N * N;
  const float4 a = sc.a, ma = neg4(sc.a), om = sc.om, mom = neg4(sc.om), b = sc.b;
  const float4* __restrict__ Ro = pp ? F.kr1 : F.kr;
  float4* __restrict__ Rn = pp ? F.kr : F.kr1;
  const float4* __restrict__ Vo = F.kv[pp];
  const float4* __restrict__ Po = F.kp[pp];
  const float4* __restrict__ T = F.kt;
  auto pnew = [&](int c) {
    const float4 v = __ldg(Vo + c);
    const float4 rn = fma4(mom, __ldg(T + c), fma4(ma, v, __ldg(Ro + c)));
    return fma4(b, fma4(mom, v, __ldg(Po + c)), rn);
  };
  FF acc[12] = {};
  Column col;
  if (column(P, col)) {
    float4 pm = pnew(col.cb + N2 * (col.k0 - 1));
    float4 pc = pnew(col.cb + N2 * col.k0);
    for (int k = col.k0; k < col.k1; ++k) {
      const int c = col.cb + N2 * k;
      const float4 pz = pnew(c + N2);
      const float4 vn = apply_op(P, load_op(F, c, ene), pc, pnew(c + 1), pnew(c - 1),
                                 pnew(c + N), pnew(c - N), pz, pm);
      const float4 r = __ldg(Ro + c), v = __ldg(Vo + c), p = __ldg(Po + c);
      const float4 sv = fma4(ma, v, r);
      const float4 rn = fma4(mom, __ldg(T + c), sv);
      F.kx[c] = fma4(om, sv, fma4(a, p, F.kx[c]));
      Rn[c] = rn;
      F.kp[1 - pp][c] = pc;
      F.kv[1 - pp][c] = vn;
      const float4 r0 = __ldg(F.kr0 + c);
      ff_dot4(acc, r0, vn);
      ff_dot4(acc + 4, rn, rn);
      ff_dot4(acc + 8, r0, rn);
      pm = pc;
      pc = pz;
    }
  }
  if (const double* tot =
          grid_total<SumFF, 12>(acc, F.rb, block_id(), block_count())) {
    if (threadIdx.x < 4) {
      const int s = threadIdx.x;
      KrylovScalars& k = F.ks[s];
      if (!k.done) {
        k.rnorm = sqrt(tot[4 + s]);
        if (k.pad) k.iters += 1;
        k.pad = 1;
        if (k.rnorm <= P.tol_lin * k.r0norm) {
          k.done = 1;
          k.status = 0;
        } else if (!isfinite(k.rnorm) || k.iters >= P.max_lin_iter || tot[s] == 0.0 ||
                   !isfinite(tot[s])) {
          k.done = 1;
          k.status = HOSC_ENOCONV;
        } else {
          k.rho = tot[8 + s];   // rho_i = r_0 . r_i from the stored r_i
          k.alpha = k.rho / tot[s];
        }
      }
    }
    // r p v t x r0 in, x r p v out, the compact operators
    count_bytes(F, HOSC_K_BICG_PV, bytes4(P, 10.0 + op_words(ene)));
  }
}

template <int MinB>
__global__ void __launch_bounds__(256, MinB) k6_b(DevParams P, Fields F, int pp) {
  __shared__ Scal4 sc;
  load_scalars(F.ks, sc);
  if (sc.all_done) return;
  const bool ene = !sc.done[3];   // the energy system still iterates (uniform)
  const int N = P.N, N2 = N * N;
  const float4 ma = neg4(sc.a);
  const float4* __restrict__ R = pp ? F.kr : F.kr1;   // r_i, written by k6_a
  const float4* __restrict__ V = F.kv[1 - pp];
  auto sval = [&](int c) { return fma4(ma, __ldg(V + c), __ldg(R + c)); };
  FF acc[16] = {};
  Column col;
  if (column(P, col)) {
    float4 sm = sval(col.cb + N2 * (col.k0 - 1));
    float4 sc0 = sval(col.cb + N2 * col.k0);
    for (int k = col.k0; k < col.k1; ++k) {
      const int c = col.cb + N2 * k;
      const float4 sz = sval(c + N2);
      const float4 tv = apply_op(P, load_op(F, c, ene), sc0, sval(c + 1), sval(c - 1),
                                 sval(c + N), sval(c - N), sz, sm);
      F.kt[c] = tv;
      const float4 r0 = __ldg(F.kr0 + c);
      ff_dot4(acc, tv, sc0);
      ff_dot4(acc + 4, tv, tv);
      ff_dot4(acc + 8, r0, sc0);
      ff_dot4(acc + 12, r0, tv);
      sm = sc0;
      sc0 = sz;
    }
  }
  if (const double* tot =
          grid_total<SumFF, 16>(acc, F.rb, block_id(), block_count())) {
    if (threadIdx.x < 4) {
      const int s = threadIdx.x;
      KrylovScalars& k = F.ks[s];
      const double ts = tot[s], tt = tot[4 + s], r0s = tot[8 + s], r0t = tot[12 + s];
      const double om = tt > 0.0 ? ts / tt : 0.0;
      const double rho_next = r0s - om * r0t;   // r_0 . (s - omega t) = r_0 . r_{i+1}
      if (!k.done) {
        if (om == 0.0 || rho_next == 0.0 || !isfinite(rho_next)) {
          k.done = 1;
          k.status = HOSC_ENOCONV;
        } else {
          // k6_a recomputes rho_{i+1} from the stored r_{i+1}; this value only sets beta
          k.beta = (rho_next / k.rho) * (k.alpha / om);
          k.omega = om;
        }
      }
    }
    // r v r0 in, t out, the compact operators
    count_bytes(F, HOSC_K_BICG_ST, bytes4(P, 4.0 + op_words(ene)));
  }
}

// ------------------------------------------------------- shared-plane stencil kernels
//
// p/v and s/t of the three-kernel form, the default above the grids of the one-launch solve. A block
// has a tile of ptx * pty interior columns (one thread each) and pkz planes. The vector that the
// operator is applied to (r + beta (p - omega v), r - alpha v) is evaluated once at each node of the tile
// and of the ring around it and put in shared memory (two planes, one barrier a plane); the planes above
// and below stay in registers. A thread then reads 3 vectors (2 for s/t) and its operator row a plane
// where the register kernels read 21 (14) and the row; and the loads of the next plane are issued before
// the barrier, so that a plane's arithmetic covers them (the register kernels wait for a plane's 19
// dependent loads: 24 warps an SM at half of the copy bandwidth). Walls are read as the zeros they hold.
// Same arithmetic of a node as the register kernels. Measured, alone, register -> shared plane: s/t
// 301 -> 262 us at 257^3, 81.5 -> 71.5 at 161^3, 44.4 -> 42.4 at 129^3, 19.9 -> 22.4 at 101^3; p/v 450 -> 439,
// 121 -> 117.5, 69.1 -> 67.1, 36.9 -> 35.3 (step at 101^3 891 against 883 us, 81^3 561 against 587): used
// from kPlaneMinN up, where a launch is several waves of blocks.
// The p/v form holds the next plane's three vectors, operator row, r_0 and ring node beside its own
// plane in 80 registers and spills (120 bytes stored and 84 loaded a thread; s/t 32 and 32), which is why it
// gains 2-3 % where s/t gains 13 %.

constexpr int kPlaneThreads = 384;

template <bool PV, bool FIRST>
__global__ void __launch_bounds__(kPlaneThreads, 2) k_plane(DevParams P, Fields F, int pp) {
  constexpr int M = PV && !FIRST ? 4 : 8;
  extern __shared__ float4 plane_sh[];
  __shared__ Scal4 sc;
  pdl_wait_and_release();
  load_scalars(F.ks, sc);
  if (sc.all_done) return;   // uniform over the grid
  const bool ene = !sc.done[3];
  const int N = P.N, N2 = N * N, tx = P.ptx, ty = P.pty, w = tx + 2, t = threadIdx.x;
  const int i0 = 1 + (int)blockIdx.x * tx, j0 = 1 + (int)blockIdx.y * ty;
  const int k0 = 1 + (int)blockIdx.z * P.plz, k1 = min(k0 + P.plz, N - 1);
  const int np = 1 - pp;
  const float4 b = sc.b, mom = neg4(sc.om), ma = neg4(sc.a);
  const float4* __restrict__ R = FIRST ? F.kr0 : F.kr;
  const float4* __restrict__ Y = PV ? F.kp[pp] : F.kv[np];
  const float4* __restrict__ Z = F.kv[pp];
  struct Raw {
    float4 r, y, z;
  };
  auto load = [&](int c) {
    Raw a;
    a.r = __ldg(R + c);
    if (!(PV && FIRST)) a.y = __ldg(Y + c);
    if (PV && !FIRST) a.z = __ldg(Z + c);
    return a;
  };
  auto value = [&](const Raw& a) {
    if (PV && FIRST) return a.r;
    if (PV) return fma4(b, fma4(mom, a.z, a.y), a.r);
    return fma4(ma, a.y, a.r);
  };
  // this thread's column, and its node of the ring (the tile's 2 (tx + ty) neighbours)
  const int cy = t / tx, cx = t - cy * tx;
  const bool in = t < tx * ty && i0 + cx <= N - 2 && j0 + cy <= N - 2;
  const int c0 = in ? i0 + cx + N * (j0 + cy) : 0, h = (cy + 1) * w + cx + 1;
  int rx = 0, ry = 0;
  if (t < tx) rx = t + 1;
  else if (t < 2 * tx) rx = t - tx + 1, ry = ty + 1;
  else if (t < 2 * tx + ty) ry = t - 2 * tx + 1;
  else rx = tx + 1, ry = t - 2 * tx - ty + 1;
  const int gi = i0 - 1 + rx, gj = j0 - 1 + ry;
  const bool ring = t < 2 * (tx + ty), rin = ring && gi <= N - 1 && gj <= N - 1;
  const int rc = rin ? gi + N * gj : 0, hr = ry * w + rx;
  const float4 zero = f4(0.f);
  Raw own = {zero, zero, zero}, rim = {zero, zero, zero};
  float4 pm = zero, pc = zero, q = zero;
  Op4 op = {zero, zero, 0.f};
  if (in) {
    pm = value(load(c0 + N2 * (k0 - 1)));
    pc = value(load(c0 + N2 * k0));
    own = load(c0 + N2 * (k0 + 1));
    op = load_op(F, c0 + N2 * k0, ene);
    if (PV && !FIRST) q = __ldg(F.kr0 + c0 + N2 * k0);
  }
  if (rin) rim = load(rc + N2 * k0);
  FF acc[M] = {};
  for (int k = k0; k < k1; ++k) {
    float4* s = plane_sh + (k & 1) * w * (ty + 2);
    const bool more = k + 1 < k1;
    if (t < tx * ty) s[h] = pc;   // zero past the interior
    if (ring) s[hr] = rin ? value(rim) : zero;
    const float4 pz = in ? value(own) : zero;
    const Op4 o = op;
    const float4 z = q;
    if (more && in) {   // the next plane's operands, in flight over this plane's arithmetic
      const int cn = c0 + N2 * (k + 1);
      own = load(cn + N2);
      op = load_op(F, cn, ene);
      if (PV && !FIRST) q = __ldg(F.kr0 + cn);
    }
    if (more && rin) rim = load(rc + N2 * (k + 1));
    __syncthreads();
    if (in) {
      const int c = c0 + N2 * k;
      const float4 y = apply_op(P, o, pc, s[h + 1], s[h - 1], s[h + w], s[h - w], pz, pm);
      if (PV) {
        F.kp[np][c] = pc;
        F.kv[np][c] = y;
        ff_dot4(acc, FIRST ? pc : z, y);
        if (FIRST) ff_dot4(acc + M - 4, pc, pc);
      } else {
        F.kt[c] = y;
        ff_dot4(acc, y, pc);
        ff_dot4(acc + M - 4, y, y);
      }
    }
    pm = pc;
    pc = pz;
  }
  const unsigned bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  const unsigned nb = gridDim.x * gridDim.y * gridDim.z;
  if (const double* tot = grid_total<SumFF, M>(acc, F.rb, bid, nb)) {
    if (PV) {
      finish_pv(F.ks, tot, FIRST);
      count_bytes(F, HOSC_K_BICG_PV, bytes4(P, (FIRST ? 3.0 : 6.0) + op_words(ene)));
    } else {
      finish_st(F.ks, tot);
      count_bytes(F, HOSC_K_BICG_ST, bytes4(P, 3.0 + op_words(ene)));
    }
  }
}

dim3 plane_grid(const DevParams& P) {
  const int ni = P.N - 2;
  return dim3((ni + P.ptx - 1) / P.ptx, (ni + P.pty - 1) / P.pty, (ni + P.plz - 1) / P.plz);
}

template <bool PV>
void launch_plane(const DevParams& P, const Fields& F, int pp, bool first, cudaStream_t s) {
  const size_t smem = 2 * sizeof(float4) * (size_t)(P.ptx + 2) * (P.pty + 2);
  if (first) launch_pdl(k_plane<PV, true>, plane_grid(P), kPlaneThreads, smem, s, P, F, pp);
  else launch_pdl(k_plane<PV, false>, plane_grid(P), kPlaneThreads, smem, s, P, F, pp);
}

// ------------------------------------------------------- staged stencil kernels (cp.async)
//
// The p/v and s/t kernels again, with their reads staged through shared memory. A block owns a
// tile of sx * sy interior columns (one thread each) and a segment of skz planes. The planes it
// needs (the haloed tile of each stencil vector, and the weights and r_0 at the tile's nodes)
// stream through a ring of kStages shared-memory stages with cp.async: 16-byte copies from global
// to shared memory that hold no registers while in flight. While plane k is computed (from the
// stages of planes k and k+1; plane k-1 is held in registers), planes k+2 and k+3 are in flight.
// The stencil reads shared memory only.

constexpr int kStages = 4;

__device__ __forceinline__ void cp_async16(float4* smem_dst, const float4* gsrc, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  const int n = valid ? 16 : 0;   // 0: write zeros, read nothing
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(gsrc), "r"(n)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_wait_two() {   // all but the two newest groups have landed
  asm volatile("cp.async.wait_group 2;\n" ::: "memory");
}

__device__ __forceinline__ void cp_async4(float* smem_dst, const float* gsrc, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  const int n = valid ? 4 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(gsrc), "r"(n)
               : "memory");
}

// Shared-memory layout of one stage, in float4: NV haloed vectors ((sx+2)(sy+2) each), then the
// compact operators of the tile's nodes (momentum float4s, energy float4s, then L as floats in
// ceil(sx*sy/4) float4 slots), then (p/v only) r_0 of the tile.
struct StageLayout {
  int hx, halo, tile, nv, lslots, per_stage;
  __host__ __device__ StageLayout(int sx, int sy, int nvec, bool with_r0) {
    hx = sx + 2;
    halo = (sx + 2) * (sy + 2);
    tile = sx * sy;
    nv = nvec;
    lslots = (tile + 3) / 4;
    per_stage = nv * halo + 2 * tile + lslots + (with_r0 ? tile : 0);
  }
  __host__ __device__ int op_m() const { return nv * halo; }
  __host__ __device__ int op_e() const { return nv * halo + tile; }
  __host__ __device__ int op_l() const { return nv * halo + 2 * tile; }
  __host__ __device__ int r0() const { return nv * halo + 2 * tile + lslots; }
};

// Copy plane q (if it exists for this block) into stage buffer st: the haloed tile of each
// stencil vector, then the compact operators (and r_0) at the tile's interior nodes; the energy
// operator only while that system iterates. Positions outside the grid are zero-filled without
// a read; the data of this plane form one commit group.
template <int NV, bool R0>
__device__ __forceinline__ void stage_plane(float4* st, const StageLayout& L, int N, int i0,
                                            int j0, int q, bool live,
                                            const float4* const (&vecs)[NV], const Fields& F,
                                            bool ene, int sx) {
  if (live) {
    const int nthr = blockDim.x;
    for (int idx = threadIdx.x; idx < L.halo; idx += nthr) {
      const int hy = idx / L.hx, hx = idx - hy * L.hx;
      const int gi = i0 - 1 + hx, gj = j0 - 1 + hy;
      const bool ok = gi <= N - 1 && gj <= N - 1;
      const int off = ok ? gi + N * (gj + N * q) : 0;
#pragma unroll
      for (int v = 0; v < NV; ++v) cp_async16(st + v * L.halo + idx, vecs[v] + off, ok);
    }
    const bool inner_plane = q >= 1 && q <= N - 2;
    for (int e = threadIdx.x; e < L.tile; e += nthr) {
      const int ty = e / sx, tx = e - ty * sx;
      const int gi = i0 + tx, gj = j0 + ty;
      const bool ok = inner_plane && gi <= N - 2 && gj <= N - 2;
      const int off = ok ? gi + N * (gj + N * q) : 0;
      cp_async16(st + L.op_m() + e, F.kwm + off, ok);
      cp_async16(st + L.op_e() + e, F.kwe + off, ok && ene);
      cp_async4((float*)(st + L.op_l()) + e, F.kL + off, ok);
      if (R0) cp_async16(st + L.r0() + e, F.kr0 + off, ok);
    }
  }
  cp_commit();   // one group per plane, empty past the segment
}

__device__ __forceinline__ Op4 staged_op(const float4* sq, const StageLayout& L, int t) {
  Op4 op;
  op.m = sq[L.op_m() + t];
  op.e = sq[L.op_e() + t];
  op.L = ((const float*)(sq + L.op_l()))[t];
  return op;
}

// Staged p/v kernel (same arithmetic as k4_pv).
__global__ void __launch_bounds__(256) k5_pv(DevParams P, Fields F, int pp) {
  extern __shared__ float4 ring[];
  __shared__ Scal4 sc;
  load_scalars(F.ks, sc);
  if (sc.all_done) return;
  const int N = P.N, N2 = N * N, sx = P.sx;
  const StageLayout L(sx, P.sy, 3, true);
  const int i0 = 1 + blockIdx.x * sx, j0 = 1 + blockIdx.y * P.sy;
  const int k0 = 1 + blockIdx.z * P.skz, k1 = min(k0 + P.skz, N - 1);
  const int t = threadIdx.x, ty = t / sx, tx = t - ty * sx;
  const bool mine = ty < P.sy && i0 + tx <= N - 2 && j0 + ty <= N - 2;
  const int h = (ty + 1) * L.hx + (tx + 1);
  const float4 b = sc.b, mom = neg4(sc.om);
  const float4* const vecs[3] = {F.kr, F.kp[pp], F.kv[pp]};
  const bool ene = !sc.done[3];
  auto stage_of = [&](int q) { return ring + ((q - (k0 - 1)) % kStages) * L.per_stage; };
  auto pnew = [&](const float4* st, int idx) {
    return fma4(b, fma4(mom, st[2 * L.halo + idx], st[L.halo + idx]), st[idx]);
  };
  // planes k0-1 .. k0+2 in flight; wait for the first two
  for (int q = k0 - 1; q <= k0 + 2; ++q)
    stage_plane<3, true>(stage_of(q), L, N, i0, j0, q, q <= k1, vecs, F, ene, sx);
  cp_wait_two();
  __syncthreads();
  float4 pm = pnew(stage_of(k0 - 1), h), pc = pnew(stage_of(k0), h);
  __syncthreads();   // the stage of plane k0-1 is free for plane k0+3
  FF acc[4] = {};
  for (int k = k0; k < k1; ++k) {
    stage_plane<3, true>(stage_of(k + 3), L, N, i0, j0, k + 3, k + 3 <= k1, vecs, F, ene, sx);
    cp_wait_two();   // plane k+1 has landed
    __syncthreads();
    const float4* sq = stage_of(k);
    const float4 pz = pnew(stage_of(k + 1), h);
    if (mine) {
      const float4 vn = apply_op(P, staged_op(sq, L, t), pc, pnew(sq, h + 1), pnew(sq, h - 1),
                                 pnew(sq, h + L.hx), pnew(sq, h - L.hx), pz, pm);
      const int c = (i0 + tx) + N * (j0 + ty) + N2 * k;
      F.kp[1 - pp][c] = pc;
      F.kv[1 - pp][c] = vn;
      ff_dot4(acc, sq[L.r0() + t], vn);
    }
    pm = pc;
    pc = pz;
    __syncthreads();   // the stage of plane k is free for plane k+4
  }
  const unsigned bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  const unsigned nb = gridDim.x * gridDim.y * gridDim.z;
  if (const double* tot = grid_total<SumFF, 4>(acc, F.rb, bid, nb)) {
    finish_pv(F.ks, tot, false);
    count_bytes(F, HOSC_K_BICG_PV, bytes4(P, 6.0 + op_words(ene)));
  }
}

// Staged s/t kernel (same arithmetic as k4_st).
__global__ void __launch_bounds__(256) k5_st(DevParams P, Fields F, int pp) {
  extern __shared__ float4 ring[];
  __shared__ Scal4 sc;
  load_scalars(F.ks, sc);
  if (sc.all_done) return;
  const int N = P.N, N2 = N * N, sx = P.sx;
  const StageLayout L(sx, P.sy, 2, false);
  const int i0 = 1 + blockIdx.x * sx, j0 = 1 + blockIdx.y * P.sy;
  const int k0 = 1 + blockIdx.z * P.skz, k1 = min(k0 + P.skz, N - 1);
  const int t = threadIdx.x, ty = t / sx, tx = t - ty * sx;
  const bool mine = ty < P.sy && i0 + tx <= N - 2 && j0 + ty <= N - 2;
  const int h = (ty + 1) * L.hx + (tx + 1);
  const float4 ma = neg4(sc.a);
  const float4* const vecs[2] = {F.kr, F.kv[1 - pp]};
  const bool ene = !sc.done[3];
  auto stage_of = [&](int q) { return ring + ((q - (k0 - 1)) % kStages) * L.per_stage; };
  auto sval = [&](const float4* st, int idx) { return fma4(ma, st[L.halo + idx], st[idx]); };
  for (int q = k0 - 1; q <= k0 + 2; ++q)
    stage_plane<2, false>(stage_of(q), L, N, i0, j0, q, q <= k1, vecs, F, ene, sx);
  cp_wait_two();
  __syncthreads();
  float4 sm = sval(stage_of(k0 - 1), h), sc0 = sval(stage_of(k0), h);
  __syncthreads();
  FF acc[8] = {};
  for (int k = k0; k < k1; ++k) {
    stage_plane<2, false>(stage_of(k + 3), L, N, i0, j0, k + 3, k + 3 <= k1, vecs, F, ene, sx);
    cp_wait_two();
    __syncthreads();
    const float4* sq = stage_of(k);
    const float4 sz = sval(stage_of(k + 1), h);
    if (mine) {
      const float4 tv = apply_op(P, staged_op(sq, L, t), sc0, sval(sq, h + 1), sval(sq, h - 1),
                                 sval(sq, h + L.hx), sval(sq, h - L.hx), sz, sm);
      const int c = (i0 + tx) + N * (j0 + ty) + N2 * k;
      F.kt[c] = tv;
      ff_dot4(acc, tv, sc0);
      ff_dot4(acc + 4, tv, tv);
    }
    sm = sc0;
    sc0 = sz;
    __syncthreads();
  }
  const unsigned bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  const unsigned nb = gridDim.x * gridDim.y * gridDim.z;
  if (const double* tot = grid_total<SumFF, 8>(acc, F.rb, bid, nb)) {
    finish_st(F.ks, tot);
    count_bytes(F, HOSC_K_BICG_ST, bytes4(P, 3.0 + op_words(ene)));
  }
}

dim3 grid5(const DevParams& P) {
  const int ni = P.N - 2;
  return dim3((unsigned)((ni + P.sx - 1) / P.sx), (unsigned)((ni + P.sy - 1) / P.sy),
              (unsigned)((ni + P.skz - 1) / P.skz));
}

dim3 grid4(const DevParams& P) {
  const int ni = P.N - 2;
  return dim3((unsigned)((ni * ni + P.kblock - 1) / P.kblock), (unsigned)((ni + P.kz - 1) / P.kz));
}

}  // namespace

namespace {
__global__ void k_krylov_activate(KrylovScalars* ks) {
  if (threadIdx.x < 4) {
    ks[threadIdx.x].done = 0;
    ks[threadIdx.x].iters = 1;   // not the first iteration, which reads less
    ks[threadIdx.x].status = 0;
  }
}
}  // namespace

void launch_krylov_activate(const Fields& F, cudaStream_t s) {
  k_krylov_activate<<<1, 32, 0, s>>>(F.ks);
}

dim3 planar_grid(const DevParams& P) {
  const int ni = P.N - 2;
  return dim3(4u * (unsigned)((P.N * P.N + P.pb - 1) / P.pb), (unsigned)((ni + P.pkz - 1) / P.pkz));
}

// Threads a block and planes a block of the planar kernels: the least load of the busiest SM in
// cycles, from the FP64 instructions of p/v (16 cycles a warp), and the chain of a block's planes
// (a barrier and the loads behind it). At most red_rows(N^3)/4 rows of partials.
void planar_shape(int N, int* pb, int* pkz) {
  const int sms = device_sms(), ni = N - 2;
  const long most = red_rows((long)N * N * N) / 4;
  double best = 1e300;
  *pb = 512;
  *pkz = ni;
  for (int B = kPlanarLeast; B <= kPlanarMost; B *= 2) {
    const long chunks = (N * (long)N + B - 1) / B;
    for (int z = 1; z <= ni; ++z) {
      const long rows = chunks * ((ni + z - 1) / z);
      if (rows > most) continue;
      const double warps = B / 32.0, halo = (2 * N + 31) / 32;
      const double work = warps * (2.0 * (z + 2) + 8.0 * z + 10.0) + 2.0 * halo * z;
      const double cost = 16.0 * work * (double)((4 * rows + sms - 1) / sms) + 900.0 * z;
      if (cost < best) {
        best = cost;
        *pb = B;
        *pkz = z;
      }
    }
  }
}

void launch_bicg_init(const DevParams& P, const Fields& F, cudaStream_t s) {
  if (P.krylov_fp32 && P.merged) {
    const long n3 = (long)P.N * P.N * P.N;
    k6_init<<<red_blocks(n3), kThreads, 0, s>>>(P, F);
    return;
  }
  if (P.krylov_fp32) {
    const long n3 = (long)P.N * P.N * P.N;
    const int most = 8 * device_sms();   // resident blocks of one wave
    const int b = red_blocks(n3) < most ? red_blocks(n3) : most;
    k4_init<<<b, kThreads, 0, s>>>(P, F);
    return;
  }
  const long ni = P.N - 2;
  k_planar_start<<<red_blocks(ni * ni * ni), kThreads, 0, s>>>(P, F);
}

// x/r as one flat stream: every node of the interior planes, the i and j walls included (every
// vector is zero there: the workspace is zeroed at creation and no kernel writes other wall entries
// than these zeros), in a grid-stride loop that
// issues the loads of U nodes before their arithmetic, so that a thread keeps 6 U float4 loads in
// flight. Same arithmetic and float-float partials as k4_xr; one block partial per block. With a scalar
// beyond float or not finite (a solve that fails) 0 times it is no zero: the walls are then left out, one
// node at a time, since later solves read them.
template <int U, bool FIRST>
__global__ void __launch_bounds__(256) k8_xr(DevParams P, Fields F, int pp) {
  __shared__ Scal4 sc;
  pdl_wait_and_release();
  load_scalars(F.ks, sc);
  if (sc.all_done && (!FIRST || *F.halt)) return;
  const int np = 1 - pp;
  const float4 a = sc.a, om = sc.om, ma = neg4(sc.a), mom = neg4(sc.om);
  const float4* __restrict__ V = F.kv[np];
  const float4* __restrict__ Pv = F.kp[np];
  const float4* __restrict__ T = F.kt;
  const float4* __restrict__ R0 = F.kr0;
  float4* __restrict__ X = F.kx;
  float4* __restrict__ R = F.kr;
  const unsigned N2 = (unsigned)P.N * (unsigned)P.N, hi = N2 * (unsigned)(P.N - 1);
  const unsigned stride = gridDim.x * blockDim.x;
  auto finite = [](float4 q) {
    return isfinite(q.x) && isfinite(q.y) && isfinite(q.z) && isfinite(q.w);
  };
  const bool wild = !finite(a) || !finite(om);   // the same for every thread
  FF acc[8] = {};
  unsigned c = N2 + blockIdx.x * blockDim.x + threadIdx.x;
  for (; !wild && c + (U - 1) * stride < hi; c += U * stride) {
    float4 r[U], v[U], p[U], t[U], r0[U], x[U];
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const unsigned e = c + q * stride;
      r0[q] = __ldg(R0 + e);
      r[q] = FIRST ? r0[q] : R[e];
      x[q] = FIRST ? f4(0.f) : X[e];
      v[q] = __ldg(V + e);
      p[q] = __ldg(Pv + e);
      t[q] = __ldg(T + e);
    }
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const unsigned e = c + q * stride;
      const float4 sv = fma4(ma, v[q], r[q]);
      X[e] = fma4(om, sv, fma4(a, p[q], x[q]));
      const float4 rn = fma4(mom, t[q], sv);
      R[e] = rn;
      ff_dot4(acc, r0[q], rn);
      ff_dot4(acc + 4, rn, rn);
    }
  }
  for (; c < hi; c += stride) {
    if (wild) {
      const unsigned N = P.N, i = c % N, j = c / N % N;
      if (i == 0 || i == N - 1 || j == 0 || j == N - 1) continue;
    }
    const float4 r0 = __ldg(R0 + c);
    const float4 sv = fma4(ma, __ldg(V + c), FIRST ? r0 : R[c]);
    X[c] = fma4(om, sv, fma4(a, __ldg(Pv + c), FIRST ? f4(0.f) : X[c]));
    const float4 rn = fma4(mom, __ldg(T + c), sv);
    R[c] = rn;
    ff_dot4(acc, r0, rn);
    ff_dot4(acc + 4, rn, rn);
  }
  if (const double* tot = grid_total<SumFF, 8>(acc, F.rb, blockIdx.x, gridDim.x)) {
    finish_xr(P, F.ks, tot);
    // r v p x t r0 in, x r out
    count_bytes(F, HOSC_K_BICG_XR, bytes4(P, FIRST ? 6.0 : 8.0));
  }
}

// Blocks of the flat x/r kernel: resident blocks of one wave.
int xr_flat_blocks() {
  static int occ = 0;
  if (occ == 0) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k8_xr<4, false>, 256, 0) != cudaSuccess ||
        occ < 1) {
      cudaGetLastError();
      occ = 4;
    }
  }
  return occ * device_sms();
}


template <int KIND, bool FIRST>
void launch_planar_f(const DevParams& P, const Fields& F, int pp, cudaStream_t s) {
  if constexpr (KIND >= PL_XR)
    launch_pdl(k_planar_end<KIND, FIRST>, planar_grid(P), P.pb, 0, s, P, F, pp);
  else   // two planes of N + pb + N doubles: 41 KB at N = 1025
    launch_pdl(k_planar<KIND, FIRST>, planar_grid(P), P.pb, 16 * (size_t)(P.pb + 2 * P.N), s, P, F,
               pp);
}
template <int KIND>
void launch_planar(const DevParams& P, const Fields& F, int pp, bool first,
                   cudaStream_t s) {
  constexpr bool has_first = KIND <= PL_R1 || KIND == PL_XR;
  if (first && has_first) launch_planar_f<KIND, has_first>(P, F, pp, s);
  else launch_planar_f<KIND, false>(P, F, pp, s);
}

void launch_bicg_pv(const DevParams& P, const Fields& F, int pp, bool first, cudaStream_t s) {
  if (!P.krylov_fp32) return launch_planar<PL_PV>(P, F, pp, first, s);
  if (P.merged) {   // x, r update of the previous iteration, then p, v
    if (P.narrow) k6_a<4><<<grid4(P), P.kblock, 0, s>>>(P, F, pp);
    else k6_a<2><<<grid4(P), P.kblock, 0, s>>>(P, F, pp);
  } else if (P.tty > 0 && (P.tkernels & 1)) {
    launch_tma_pv(P, F, pp, s);
  } else if (P.sx > 0) {
    k5_pv<<<grid5(P), P.sx * P.sy, staged_smem_bytes(P.sx, P.sy, true), s>>>(P, F, pp);
  } else if (P.plane) {
    launch_plane<true>(P, F, pp, first, s);
  } else if (first && P.lean) {
    if (P.narrow) launch_pdl(k4_pv<4, true>, grid4(P), P.kblock, 0, s, P, F, pp);
    else launch_pdl(k4_pv<2, true>, grid4(P), P.kblock, 0, s, P, F, pp);
  } else {
    if (P.narrow) launch_pdl(k4_pv<4, false>, grid4(P), P.kblock, 0, s, P, F, pp);
    else launch_pdl(k4_pv<2, false>, grid4(P), P.kblock, 0, s, P, F, pp);
  }
}

void launch_bicg_st(const DevParams& P, const Fields& F, int pp, bool first, cudaStream_t s) {
  if (!P.krylov_fp32) return launch_planar<PL_ST>(P, F, pp, first, s);
  if (P.merged) {
    if (P.narrow) k6_b<4><<<grid4(P), P.kblock, 0, s>>>(P, F, pp);
    else k6_b<2><<<grid4(P), P.kblock, 0, s>>>(P, F, pp);
  } else if (P.tty > 0 && (P.tkernels & 2)) {
    launch_tma_st(P, F, pp, s);
  } else if (P.sx > 0) {
    k5_st<<<grid5(P), P.sx * P.sy, staged_smem_bytes(P.sx, P.sy, false), s>>>(P, F, pp);
  } else if (P.plane) {
    launch_plane<false>(P, F, pp, first, s);
  } else {
    const int f = first && P.lean;
    if (P.narrow) launch_pdl(k4_st<4>, grid4(P), P.kblock, 0, s, P, F, pp, f);
    else launch_pdl(k4_st<2>, grid4(P), P.kblock, 0, s, P, F, pp, f);
  }
}

template <bool FIRST>
void launch_xr4(const DevParams& P, const Fields& F, int pp, cudaStream_t s) {
  if (P.xr_flat) launch_pdl(k8_xr<4, FIRST>, dim3(xr_flat_blocks()), 256, 0, s, P, F, pp);
  else if (P.narrow) launch_pdl(k4_xr<4, FIRST>, grid4(P), P.kblock, 0, s, P, F, pp);
  else launch_pdl(k4_xr<2, FIRST>, grid4(P), P.kblock, 0, s, P, F, pp);
}

void launch_bicg_xr(const DevParams& P, const Fields& F, int pp, bool first, cudaStream_t s) {
  if (!P.krylov_fp32) return launch_planar<PL_XR>(P, F, pp, first, s);
  if (P.merged) return;   // folded into the next k6_a
  if (first && P.lean) launch_xr4<true>(P, F, pp, s);
  else launch_xr4<false>(P, F, pp, s);
}

void launch_loop_cond(const Fields& F, unsigned long long handle, cudaStream_t s) {
  k_loop_cond<<<1, 32, 0, s>>>(F.ks, (cudaGraphConditionalHandle)handle);
}

void launch_b2(int kernel, const DevParams& P, const Fields& F, int cp, bool first,
               cudaStream_t s) {
  switch (kernel) {
    case 0: launch_planar<PL_U1>(P, F, cp, first, s); break;
    case 1: launch_planar<PL_R1>(P, F, cp, first, s); break;
    case 2: launch_planar<PL_U2>(P, F, cp, false, s); break;
    case 3: launch_planar<PL_R2>(P, F, cp, false, s); break;
    default: launch_planar<PL_MR>(P, F, cp, false, s); break;
  }
}

long krylov4_blocks(const DevParams& P) {
  const dim3 g = grid4(P);
  long nb = (long)g.x * g.y;
  if (P.sx > 0) {
    const dim3 g5 = grid5(P);
    const long n5 = (long)g5.x * g5.y * g5.z;
    nb = n5 > nb ? n5 : nb;
  }
  const long n7 = tma_blocks(P);
  return n7 > nb ? n7 : nb;
}

size_t staged_smem_bytes(int sx, int sy, bool pv) {
  const StageLayout L(sx, sy, pv ? 3 : 2, pv);
  return (size_t)kStages * L.per_stage * sizeof(float4);
}

// Opt the staged kernels in to large dynamic shared memory (once per device and process).
bool staged_smem_ready() {
  static int done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  if (!done[dev]) {
    const int cap = 200 * 1024;
    if (cudaFuncSetAttribute(k5_pv, cudaFuncAttributeMaxDynamicSharedMemorySize, cap) !=
            cudaSuccess ||
        cudaFuncSetAttribute(k5_st, cudaFuncAttributeMaxDynamicSharedMemorySize, cap) !=
            cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    done[dev] = 1;
  }
  return true;
}

double staged_wave_cost(int N, int sx, int sy, int skz, int sms) {
  if (!staged_smem_ready()) return 1e300;
  const size_t smem = staged_smem_bytes(sx, sy, true);
  if (smem > 200 * 1024) return 1e300;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k5_pv, sx * sy, smem) != cudaSuccess ||
      occ < 1) {
    cudaGetLastError();
    return 1e300;
  }
  const long ni = N - 2;
  const long items = ((ni + sx - 1) / sx) * ((ni + sy - 1) / sy) * ((ni + skz - 1) / skz);
  const long slots = (long)occ * sms;
  const long waves = (items + slots - 1) / slots;
  return (double)waves * (skz + 2);
}

int krylov4_occupancy(int kblock, int narrow, int merged) {
  int occ = 0;
  cudaError_t e;
  if (merged)
    e = narrow ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k6_a<4>, kblock, 0)
               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k6_a<2>, kblock, 0);
  else
    e = narrow ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k4_pv<4, false>, kblock, 0)
               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k4_pv<2, false>, kblock, 0);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return occ > 0 ? occ : 1;
}

int device_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return 152;
  }
  return sms > 0 ? sms : 152;
}

double krylov4_wave_cost(int N, int kblock, int kz, int narrow, int merged, int sms) {
  const long ni = N - 2;
  const long items = ((ni * ni + kblock - 1) / kblock) * ((ni + kz - 1) / kz);
  const long slots = (long)krylov4_occupancy(kblock, narrow, merged) * sms;
  const long waves = (items + slots - 1) / slots;
  // every resident block streams kz planes plus the two it reads around its segment
  return (double)waves * (kz + 2);
}

// Tile and planes of the shared-plane kernels: the least modelled time, waves of the two resident blocks
// an SM times the planes a block streams times the nodes it reads a plane (tile and ring), among tiles
// that cut the interior evenly and fit a block's threads.
bool plane_shape(int N, int* ptx, int* pty, int* plz) {
  if (N < kPlaneMinN) return false;
  const int sms = device_sms(), ni = N - 2;
  double best = 1e300;
  *ptx = *pty = *plz = 1;
  for (int nx = 1; nx <= ni; ++nx) {
    const int tx = (ni + nx - 1) / nx;
    if (tx > 128) continue;
    if (tx < 16 && nx > 1) break;
    int ty = kPlaneThreads / tx < ni ? kPlaneThreads / tx : ni;
    const int ny = (ni + ty - 1) / ty;
    ty = (ni + ny - 1) / ny;
    if (2 * (tx + ty) > kPlaneThreads) continue;
    for (int z = 1; z <= ni && z <= 64; ++z) {
      const long blocks = (long)((ni + tx - 1) / tx) * ny * ((ni + z - 1) / z);
      const double waves = (double)((blocks + 2 * sms - 1) / (2 * sms));
      const double cost = waves * (z + 2) * (kPlaneThreads + 2.0 * (tx + ty));
      if (cost < best) {
        best = cost;
        *ptx = tx;
        *pty = ty;
        *plz = z;
      }
    }
  }
  return best < 1e300;
}

// Blocks of 384 threads: with the same bytes in flight as three blocks of 128 a launch leaves a third
// of the partials (sum of the three kernels at 71^3 43 -> 35 us, 81^3 47 -> 43.5, 101^3 77.3 -> 70.8,
// 161^3 and 257^3 within 1 %); the planes a block by the wave model.
void default_tiles(int N, int* kblock, int* kz) {
  const int sms = device_sms();
  const int ni = N - 2;
  double best = 1e300;
  *kblock = 384;
  *kz = 1;
  const long slots = (long)krylov4_occupancy(384, 0, 0) * sms, chunks = ((long)ni * ni + 383) / 384;
  for (int z = 1; z <= (ni < 33 ? ni : 33); ++z) {
    const long items = chunks * ((ni + z - 1) / z);
    const double c = (double)((items + slots - 1) / slots) * (z + 2);
    if (c < best) {
      best = c;
      *kz = z;
    }
  }
}

}  // namespace hosc
