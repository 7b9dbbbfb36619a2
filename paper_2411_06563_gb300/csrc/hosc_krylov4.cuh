// Device code of the interleaved FP32 BiCGSTAB of the mixed-precision solve (Punia & Ray,
// arXiv:2411.06563, Sec. 2.2: unpreconditioned BiCGSTAB on the four level-(n+1) systems): one
// float4 per node holds the u, v, w, theta values of a vector, the operators are the compact
// float forms written by the right-hand-side kernel, and a thread owns one interior (i, j) column
// over a segment of kz planes, keeping the z-neighbours in registers as it marches; dot-product
// terms accumulate in float-float over the segment before the block reduction, and the last
// block of a launch (a ticket counter) finalises the scalars the next kernel needs.
//
// The kernels are device bodies taking the block's (virtual) position in the grid of column chunks
// and plane segments, so that the per-kernel launches (hosc_krylov.cu) and the persistent round
// kernel of the pool (hosc_round.cu) run the same code.
#pragma once

#include <math.h>

#include "hosc_device.cuh"
#include "hosc_internal.h"

namespace hosc {

namespace {

// Float-float ("double-float") numbers: an unevaluated sum hi + lo of two floats. Knuth's TwoSum
// and an FMA-based exact product give sums with about 44 significant bits using float
// instructions only, which GB300 issues at 64x the rate of double instructions.
struct FF {
  float hi, lo;
};

__device__ __forceinline__ FF ff_prod(float a, float b) {
  FF r;
  r.hi = __fmul_rn(a, b);     // never fused into a sum
  r.lo = fmaf(a, b, -r.hi);   // exact rounding error of the product
  return r;
}

__device__ __forceinline__ FF ff_add(FF a, FF b) {
  const float s = a.hi + b.hi;
  const float bb = s - a.hi;
  const float err = (a.hi - (s - bb)) + (b.hi - bb);   // TwoSum: s + err == a.hi + b.hi exactly
  const float lo = err + a.lo + b.lo;
  FF r;
  r.hi = s + lo;
  r.lo = lo - (r.hi - s);
  return r;
}

// Sums of float-float values; the blocks' totals are added in double.
struct SumFF {
  using V = FF;
  using Total = SumD;
  static __device__ __forceinline__ V zero() { return FF{0.0f, 0.0f}; }
  static __device__ __forceinline__ V add(V a, V b) { return ff_add(a, b); }
  static __device__ __forceinline__ V shfl_xor(V a, int m) {
    return FF{__shfl_xor_sync(0xffffffffu, a.hi, m), __shfl_xor_sync(0xffffffffu, a.lo, m)};
  }
  static __device__ __forceinline__ double value(V a) { return (double)a.hi + (double)a.lo; }
};

// ------------------------------------------------------------------ interleaved FP32 solve

__device__ __forceinline__ float4 f4(float a) { return make_float4(a, a, a, a); }

// a + b * c per component
__device__ __forceinline__ float4 fma4(float4 b, float4 c, float4 a) {
  return make_float4(fmaf(b.x, c.x, a.x), fmaf(b.y, c.y, a.y), fmaf(b.z, c.z, a.z),
                     fmaf(b.w, c.w, a.w));
}
__device__ __forceinline__ float4 neg4(float4 a) { return make_float4(-a.x, -a.y, -a.z, -a.w); }

// acc[m0 + s] += a_s * b_s for the four systems s
__device__ __forceinline__ void ff_dot4(FF* acc, float4 a, float4 b) {
  acc[0] = ff_add(acc[0], ff_prod(a.x, b.x));
  acc[1] = ff_add(acc[1], ff_prod(a.y, b.y));
  acc[2] = ff_add(acc[2], ff_prod(a.z, b.z));
  acc[3] = ff_add(acc[3], ff_prod(a.w, b.w));
}

// The seven-point operators of the four systems at node c, from the compact operators: along
// direction d the +d and -d neighbours weigh S_d - B_d and S_d + B_d, so the product is
// D o + sum_d S_d (o_{+d} + o_{-d}) - B_d (o_{+d} - o_{-d}). Momentum (u, v, w lanes): B and D from
// kwm, S_d = -dt/(2 h_d^2) + L/12. Energy (theta lane): B and D from kwe, S_d = -dt/(2 h_d^2) +
// 1/12; with ene false (the energy system has converged) its weights are not read and the lane
// is zero. With Jacobi row scaling (precond) each row is divided by its diagonal D.
struct Op4 {
  float4 m, e;   // (B_x, B_y, B_z, D) of momentum and of energy
  float L;       // L of the momentum row
};

__device__ __forceinline__ Op4 load_op(const Fields& F, int c, bool ene) {
  Op4 op;
  op.m = HOSC_LDG(F.kwm + c);
  op.L = HOSC_LDG(F.kL + c);
  op.e = ene ? HOSC_LDG(F.kwe + c) : make_float4(0.f, 0.f, 0.f, 0.f);
  return op;
}

__device__ __forceinline__ float4 apply_op(const DevParams& P, const Op4& op, float4 o, float4 xp,
                                           float4 xm, float4 yp, float4 ym, float4 zp,
                                           float4 zm) {
  // momentum weights of the six neighbours, shared by the u, v, w lanes
  const float c12 = 1.f / 12.f;
  const float Sx = fmaf(op.L, c12, P.csf[0]), Sy = fmaf(op.L, c12, P.csf[1]),
              Sz = fmaf(op.L, c12, P.csf[2]);
  const float4 m = op.m, e = op.e;
  const float a1 = Sx - m.x, a2 = Sx + m.x, a3 = Sy - m.y, a4 = Sy + m.y, a5 = Sz - m.z,
              a6 = Sz + m.z;
  // one explicit order of the sums and fused multiply-adds, so that every kernel that applies the
  // operator gets the same bits
  auto row = [&](float c, float cp, float cm, float yp_, float ym_, float zp_, float zm_) {
    return fmaf(a6, zm_, fmaf(a5, zp_, fmaf(a4, ym_, fmaf(a3, yp_, fmaf(a2, cm, fmaf(m.w, c,
                __fmul_rn(a1, cp)))))));
  };
  float4 y;
  y.x = row(o.x, xp.x, xm.x, yp.x, ym.x, zp.x, zm.x);
  y.y = row(o.y, xp.y, xm.y, yp.y, ym.y, zp.y, zm.y);
  y.z = row(o.z, xp.z, xm.z, yp.z, ym.z, zp.z, zm.z);
  const float ex = P.csf[0] + c12, ey = P.csf[1] + c12, ez = P.csf[2] + c12;
  y.w = fmaf(ez + e.z, zm.w, fmaf(ez - e.z, zp.w, fmaf(ey + e.y, ym.w, fmaf(ey - e.y, yp.w,
        fmaf(ex + e.x, xm.w, fmaf(e.w, o.w, __fmul_rn(ex - e.x, xp.w)))))));
  if (P.precond) {
    const float im = 1.f / m.w;
    y.x *= im;
    y.y *= im;
    y.z *= im;
    y.w = e.w != 0.f ? y.w / e.w : 0.f;
  }
  return y;
}

// A row of the planar FP64 operator, in one explicit order for the same reason.
__device__ __forceinline__ double planar_row(double a0, double a1, double a2, double a3, double a4,
                                             double a5, double a6, double c, double xp, double xm,
                                             double yp, double ym, double zp, double zm) {
  return fma(a6, zm, fma(a5, zp, fma(a4, ym, fma(a3, yp, fma(a2, xm, fma(a0, c,
             __dmul_rn(a1, xp)))))));
}

// Float4 words per interior node of the compact operators a launch reads: kwm and kL, and kwe
// while the energy system iterates.
__device__ __forceinline__ double op_words(bool ene) { return 1.25 + (ene ? 1.0 : 0.0); }

// Thread -> interior column (i, j) and its segment [k0, k1) of planes. False for the threads
// past the last column of the plane (they still take part in the block reduction).
struct Column {
  int cb;      // node index of (i, j, 0)
  int k0, k1;  // planes of the segment
};
// A block's index in a two-dimensional grid of (column chunks) x (plane segments), and the grid's
// size: the hardware indices of a launch, or those a persistent kernel assigns.
struct VGrid {
  unsigned x, y, nx, ny;
};
__device__ __forceinline__ VGrid hw_grid() { return {blockIdx.x, blockIdx.y, gridDim.x, gridDim.y}; }

__device__ __forceinline__ bool column(const DevParams& P, Column& col, const VGrid& g) {
  const int N = P.N, ni = N - 2;
  const int q = (int)g.x * blockDim.x + threadIdx.x;
  if (q >= ni * ni) return false;
  const int j = q / ni, i = q - j * ni;
  col.cb = (i + 1) + N * (j + 1);
  col.k0 = 1 + (int)g.y * P.kz;
  col.k1 = min(col.k0 + P.kz, N - 1);
  return true;
}
__device__ __forceinline__ bool column(const DevParams& P, Column& col) {
  return column(P, col, hw_grid());
}

__device__ __forceinline__ unsigned block_id(const VGrid& g) { return g.x + g.nx * g.y; }
__device__ __forceinline__ unsigned block_count(const VGrid& g) { return g.nx * g.ny; }
__device__ __forceinline__ unsigned block_id() { return block_id(hw_grid()); }
__device__ __forceinline__ unsigned block_count() { return block_count(hw_grid()); }

// Per-system scalars of the interleaved kernels, zero for a finished system so that its vectors
// stay as they are (x += 0, r = r - 0).
struct Scal4 {
  float4 a, b, om;
  int done[4];
  int all_done;
};

// The first warp reads the four systems' scalars, one lane a system.
__device__ __forceinline__ void load_scalars(const KrylovScalars* ks, Scal4& sc) {
  if (threadIdx.x < 32) {
    __syncwarp();
    const int s = threadIdx.x;
    int d = 1;
    if (s < 4) {
      const double a = ks[s].alpha, b = ks[s].beta, om = ks[s].omega;
      d = ks[s].done;
      sc.done[s] = d;
      (&sc.a.x)[s] = d ? 0.f : (float)a;
      (&sc.b.x)[s] = d ? 0.f : (float)b;
      (&sc.om.x)[s] = d ? 0.f : (float)om;
    }
    const int all = __all_sync(0xffffffffu, d != 0);
    if (s == 0) sc.all_done = all;
  }
  __syncthreads();
}

// ---- ends of the Krylov kernels: the last block of a launch sets the scalars the next kernel
// needs from the launch's totals, one thread a system (each an FP64 divide or square root and a few
// dependent reads: one after another they took 4 us of a 20 us launch on a 41^3 grid).

// A system before its first iteration, set by the right-hand sides' kernel: the first p/v of the
// lean forms (no initialisation kernel) then finds ||r_0||.
__device__ __forceinline__ void start_system(const DevParams& P, const Fields& F, int s) {
  KrylovScalars& k = F.ks[s];
  k.rho = k.r0norm = k.rnorm = 0.0;
  k.alpha = 0.0;
  k.omega = 1.0;
  k.beta = 0.0;
  k.g1 = k.g2 = 0.0;
  k.iters = 0;
  k.pad = 0;
  k.status = 0;
  k.done = s == 3 && P.inner_pass;   // an inner pressure pass solves the momentum systems only
}

// r_0 . r_0 of each system: the solve starts (forms that are not lean).
__device__ __forceinline__ void finish_init(const DevParams& P, const Fields& F, const double* tot) {
  if (threadIdx.x >= 4) return;
  const int s = threadIdx.x;
  KrylovScalars& k = F.ks[s];
  const int halt = *F.halt;
  const double norm = sqrt(tot[s]);
  k.r0norm = norm;
  k.rnorm = norm;
  k.rho = tot[s];
  // the first kernel of the merged form then leaves x = 0, r = r_0 and sets p = r_0
  k.alpha = P.merged ? 0.0 : 1.0;
  k.omega = P.merged ? 0.0 : 1.0;
  k.beta = 0.0;
  k.g1 = k.g2 = 0.0;
  k.iters = 0;
  k.pad = 0;
  k.status = 0;
  // an inner pressure pass solves the momentum systems only
  k.done = (norm == 0.0 || halt || (s == 3 && P.inner_pass)) ? 1 : 0;
}

// One system's scalars from r_0 . v = d: alpha = rho / d. In the first iteration of a lean form r_0 .
// r_0 = rr too, which is rho; a system whose right-hand side is zero is then done.
__device__ __forceinline__ void pv_scalars(KrylovScalars& k, double d, double rr, bool first) {
  const int done = k.done;
  double rho = k.rho;
  if (done) return;
  if (first) {
    rho = rr;
    const double norm = sqrt(rr);
    k.rho = rho;
    k.r0norm = norm;
    k.rnorm = norm;
    if (norm == 0.0) {
      k.done = 1;
      return;
    }
  }
  if (d == 0.0 || !isfinite(d)) {
    k.done = 1;
    k.status = HOSC_ENOCONV;
  } else {
    k.alpha = rho / d;
  }
}

// omega = (t . s) / (t . t), 0 when t = 0.
__device__ __forceinline__ void st_scalars(KrylovScalars& k, double ts, double tt) {
  if (!k.done) k.omega = tt > 0.0 ? ts / tt : 0.0;
}

// r_0 . r = rho_new and r . r = rr: the convergence and breakdown tests, beta and rho of the next
// iteration.
__device__ __forceinline__ void xr_scalars(const DevParams& P, KrylovScalars& k, double rho_new,
                                           double rr) {
  const int done = k.done, iters = k.iters + 1;
  const double rho = k.rho, alpha = k.alpha, omega = k.omega, r0norm = k.r0norm;
  if (done) return;
  const double rnorm = sqrt(rr);
  k.rnorm = rnorm;
  k.iters = iters;
  if (rnorm <= P.tol_lin * r0norm) {
    k.done = 1;
    k.status = 0;
  } else if (!isfinite(rnorm) || iters >= P.max_lin_iter || rho_new == 0.0 || omega == 0.0) {
    k.done = 1;
    k.status = HOSC_ENOCONV;
  } else {
    k.beta = (rho_new / rho) * (alpha / omega);
    k.rho = rho_new;
  }
}

// BiCGSTAB(2): rho_1 = rt.r_1 and beta after R1.
__device__ __forceinline__ void b2_fail(KrylovScalars& k) {
  k.done = 1;
  k.status = HOSC_ENOCONV;
}
__device__ __forceinline__ void b2_r1_scalars(KrylovScalars& k, double rho1) {
  if (k.done) return;
  if (k.rho == 0.0 || !isfinite(rho1)) {
    b2_fail(k);
  } else {
    k.beta = k.alpha * rho1 / k.rho;
    k.rho = rho1;
  }
}

// The minimal-residual coefficients from d = r_1.r_1, r_1.r_2, r_2.r_2, r_0.r_1, r_0.r_2.
__device__ __forceinline__ void b2_r2_scalars(KrylovScalars& k, const double* d) {
  if (k.done) return;
  const double sig1 = d[0];
  const double tau = sig1 > 0.0 ? d[1] / sig1 : 0.0;
  const double sig2 = d[2] - tau * d[1];   // |r_2 - tau r_1|^2
  if (!(sig1 > 0.0) || !(sig2 > 0.0) || !isfinite(sig2)) {
    b2_fail(k);
  } else {
    const double gp1 = d[3] / sig1, g2 = (d[4] - tau * d[3]) / sig2;
    k.g2 = g2;
    k.g1 = gp1 - tau * g2;
    k.omega = g2;
  }
}

// The end of a cycle from rho_1 = rt.r_0 and rr = r_0.r_0.
__device__ __forceinline__ void b2_mr_scalars(const DevParams& P, KrylovScalars& k, double rho1,
                                              double rr) {
  if (k.done) return;
  const double rnorm = sqrt(rr);
  k.rnorm = rnorm;
  k.iters += 2;
  const double rho0 = -k.omega * k.rho;
  if (rnorm <= P.tol_lin * k.r0norm) {
    k.done = 1;
    k.status = 0;
  } else if (!isfinite(rnorm) || k.iters >= P.max_lin_iter || rho0 == 0.0) {
    b2_fail(k);
  } else {
    k.beta = k.alpha * rho1 / rho0;
    k.rho = rho1;
  }
}

// The same for the four systems at ks from the totals of a launch: slots 0..3 and 4..7.
__device__ __forceinline__ void finish_pv(KrylovScalars* ks, const double* tot, bool first) {
  const int s = threadIdx.x;
  if (s < 4) pv_scalars(ks[s], tot[s], first ? tot[4 + s] : 0.0, first);
}
__device__ __forceinline__ void finish_st(KrylovScalars* ks, const double* tot) {
  if (threadIdx.x < 4) st_scalars(ks[threadIdx.x], tot[threadIdx.x], tot[4 + threadIdx.x]);
}
__device__ __forceinline__ void finish_xr(const DevParams& P, KrylovScalars* ks, const double* tot) {
  if (threadIdx.x < 4) xr_scalars(P, ks[threadIdx.x], tot[threadIdx.x], tot[4 + threadIdx.x]);
}

// Add a launch's algorithmic bytes (a thread that takes no part in the ends above).
__device__ __forceinline__ void count_bytes(const Fields& F, int kid, double bytes) {
  if (threadIdx.x == blockDim.x - 1) atomicAdd(F.alg_bytes + kid, bytes);
}

// Algorithmic bytes of one interleaved launch: words (float4 per interior node) moved.
__device__ __forceinline__ double bytes4(const DevParams& P, double float4_words) {
  const double ni = (double)(P.N - 2);
  return 16.0 * float4_words * ni * ni * ni;
}

// r = r_0, x = 0, p = v = 0 at interior nodes, every vector zero on the walls; ||r_0||^2.
// Grid-stride over all N^3 nodes: each thread sums several nodes before the one block reduction.
// Returns true in the block that finished the launch's reduction (its scalars are then final).
__device__ __forceinline__ bool k4_init_body(const DevParams& P, const Fields& F, unsigned vbx,
                                             unsigned vnb) {
  const unsigned N = P.N;
  const unsigned n3 = N * N * N;
  FF acc[4] = {};
  for (unsigned c = vbx * blockDim.x + threadIdx.x; c < n3; c += vnb * blockDim.x) {
    const unsigned q = c / N;
    const unsigned i = c - q * N, j = q % N, k = q / N;
    const bool inner = i > 0 && j > 0 && k > 0 && i < N - 1 && j < N - 1 && k < N - 1;
    const float4 z = f4(0.f);
    const float4 r = inner ? F.kr0[c] : z;
    F.kr[c] = r;
    // t needs no zeros: inside, k4_st writes it before k4_xr reads it; its wall entries (and those
    // of r_0) are zero from the workspace's zeroing at creation, and no kernel writes them
    F.kx[c] = z;
    F.kp[0][c] = z;
    F.kp[1][c] = z;
    F.kv[0][c] = z;
    F.kv[1][c] = z;
    ff_dot4(acc, r, r);
  }
  const double* tot = grid_total<SumFF, 4>(acc, F.rb, vbx, vnb);
  if (!tot) return false;
  finish_init(P, F, tot);
  return true;
}

__global__ void __launch_bounds__(kThreads) k4_init(DevParams P, Fields F) {
  k4_init_body(P, F, blockIdx.x, gridDim.x);
}

// The kernels of a solve's first iteration are forms of their own (FIRST): the residual is r_0, there
// is no search direction and no iterate, so they read less (p/v 3 of 6 vectors, x/r 4 of 6) and no
// initialisation kernel has to write seven vectors (26 us of a step at 101^3). As a branch inside the
// kernels the same cost registers in the loop: p/v 39.9 -> 48.2 us at 101^3.
//
// p_new = r + beta (p_old - omega v_old) at the seven stencil nodes, v_new = A p_new, partial
// r_0 . v_new; last block: alpha = rho / (r_0 . v_new). FIRST: p_new = r_0, and the partial r_0 . r_0
// gives rho and ||r_0||.
template <bool FIRST>
__device__ __forceinline__ void k4_pv_body(const DevParams& P, const Fields& F, int pp,
                                            const VGrid& vg) {
  constexpr int M = FIRST ? 8 : 4;
  __shared__ Scal4 sc;
  load_scalars(F.ks, sc);
  if (sc.all_done) return;   // uniform over the grid
  const bool ene = !sc.done[3];   // the energy system still iterates (uniform)
  const int N = P.N, N2 = N * N;
  const float4 b = sc.b, mom = neg4(sc.om);
  const float4* HOSC_RESTRICT R = FIRST ? F.kr0 : F.kr;
  const float4* HOSC_RESTRICT Po = F.kp[pp];
  const float4* HOSC_RESTRICT Vo = F.kv[pp];
  float4* HOSC_RESTRICT Pn = F.kp[1 - pp];
  float4* HOSC_RESTRICT Vn = F.kv[1 - pp];
  auto pnew = [&](int c) {
    const float4 r = HOSC_LDG(R + c);
    if (FIRST) return r;
    const float4 p = HOSC_LDG(Po + c), v = HOSC_LDG(Vo + c);
    return fma4(b, fma4(mom, v, p), r);
  };
  FF acc[M] = {};
  Column col;
  if (column(P, col, vg)) {
    float4 pm = pnew(col.cb + N2 * (col.k0 - 1));
    float4 pc = pnew(col.cb + N2 * col.k0);
    for (int k = col.k0; k < col.k1; ++k) {
      const int c = col.cb + N2 * k;
      const float4 pz = pnew(c + N2);
      const float4 vn = apply_op(P, load_op(F, c, ene), pc, pnew(c + 1), pnew(c - 1),
                                 pnew(c + N), pnew(c - N), pz, pm);
      Pn[c] = pc;
      Vn[c] = vn;
      ff_dot4(acc, FIRST ? pc : HOSC_LDG(F.kr0 + c), vn);
      if (FIRST) ff_dot4(acc + M - 4, pc, pc);
      pm = pc;
      pc = pz;
    }
  }
  if (const double* tot =
          grid_total<SumFF, M>(acc, F.rb, block_id(vg), block_count(vg))) {
    finish_pv(F.ks, tot, FIRST);
    // r p v r0 in, p v out, the compact operators
    count_bytes(F, HOSC_K_BICG_PV, bytes4(P, (FIRST ? 3.0 : 6.0) + op_words(ene)));
  }
}

template <int MinB, bool FIRST>
__global__ void __launch_bounds__(MinB == 2 ? 384 : 256, MinB)
    k4_pv(DevParams P, Fields F, int pp) {
  pdl_wait_and_release();
  k4_pv_body<FIRST>(P, F, pp, hw_grid());
}

// s = r - alpha v at the seven stencil nodes, t = A s, partials (t . s, t . t); last block:
// omega = (t . s) / (t . t) (0 when t = 0).
__device__ __forceinline__ void k4_st_body(const DevParams& P, const Fields& F, int pp, int first,
                                            const VGrid& vg) {
  __shared__ Scal4 sc;
  load_scalars(F.ks, sc);
  if (sc.all_done) return;
  const bool ene = !sc.done[3];   // the energy system still iterates (uniform)
  const int N = P.N, N2 = N * N;
  const int np = 1 - pp;   // written by k4_pv of this iteration
  const float4 ma = neg4(sc.a);
  const float4* HOSC_RESTRICT R = first ? F.kr0 : F.kr;
  const float4* HOSC_RESTRICT V = F.kv[np];
  float4* HOSC_RESTRICT T = F.kt;
  auto sval = [&](int c) { return fma4(ma, HOSC_LDG(V + c), HOSC_LDG(R + c)); };
  FF acc[8] = {};
  Column col;
  if (column(P, col, vg)) {
    float4 sm = sval(col.cb + N2 * (col.k0 - 1));
    float4 sc0 = sval(col.cb + N2 * col.k0);
    for (int k = col.k0; k < col.k1; ++k) {
      const int c = col.cb + N2 * k;
      const float4 sz = sval(c + N2);
      const float4 tv = apply_op(P, load_op(F, c, ene), sc0, sval(c + 1), sval(c - 1),
                                 sval(c + N), sval(c - N), sz, sm);
      T[c] = tv;
      ff_dot4(acc, tv, sc0);
      ff_dot4(acc + 4, tv, tv);
      sm = sc0;
      sc0 = sz;
    }
  }
  if (const double* tot =
          grid_total<SumFF, 8>(acc, F.rb, block_id(vg), block_count(vg))) {
    finish_st(F.ks, tot);
    // r v in, t out, the compact operators
    count_bytes(F, HOSC_K_BICG_ST, bytes4(P, 3.0 + op_words(ene)));
  }
}

template <int MinB>
__global__ void __launch_bounds__(MinB == 2 ? 384 : 256, MinB)
    k4_st(DevParams P, Fields F, int pp, int first) {
  pdl_wait_and_release();
  k4_st_body(P, F, pp, first, hw_grid());
}

// s = r - alpha v; x += alpha p + omega s; r = s - omega t; partials (r_0 . r, r . r); last block:
// convergence and breakdown tests, beta and rho of the next iteration.
template <bool FIRST>
__device__ __forceinline__ void k4_xr_body(const DevParams& P, const Fields& F, int pp,
                                            const VGrid& vg) {
  __shared__ Scal4 sc;
  load_scalars(F.ks, sc);
  // FIRST runs with every right-hand side zero too (the increments are then zero), not when halted
  if (sc.all_done && (!FIRST || *F.halt)) return;
  const int N2 = P.N * P.N;
  const int np = 1 - pp;
  const float4 a = sc.a, om = sc.om, ma = neg4(sc.a), mom = neg4(sc.om);
  FF acc[8] = {};
  Column col;
  if (column(P, col, vg)) {
    for (int k = col.k0; k < col.k1; ++k) {
      const int c = col.cb + N2 * k;
      const float4 r0 = HOSC_LDG(F.kr0 + c);
      const float4 r = FIRST ? r0 : F.kr[c], x = FIRST ? f4(0.f) : F.kx[c];
      const float4 v = HOSC_LDG(F.kv[np] + c), p = HOSC_LDG(F.kp[np] + c);
      const float4 t = HOSC_LDG(F.kt + c);
      const float4 sv = fma4(ma, v, r);
      F.kx[c] = fma4(om, sv, fma4(a, p, x));
      const float4 rn = fma4(mom, t, sv);
      F.kr[c] = rn;
      ff_dot4(acc, r0, rn);
      ff_dot4(acc + 4, rn, rn);
    }
  }
  const double* tot =
      grid_total<SumFF, 8>(acc, F.rb, block_id(vg), block_count(vg));
  if (!tot) return;
  finish_xr(P, F.ks, tot);
  count_bytes(F, HOSC_K_BICG_XR, bytes4(P, FIRST ? 6.0 : 8.0));   // r v p x t r0 in, x r out
}

template <int MinB, bool FIRST>
__global__ void __launch_bounds__(MinB == 2 ? 384 : 256, MinB)
    k4_xr(DevParams P, Fields F, int pp) {
  pdl_wait_and_release();
  k4_xr_body<FIRST>(P, F, pp, hw_grid());
}

}  // namespace

}  // namespace hosc
