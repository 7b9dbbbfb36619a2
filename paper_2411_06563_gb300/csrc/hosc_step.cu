// Launchers of the step kernels other than the Krylov solver (Punia & Ray, arXiv:2411.06563,
// Sec. 2.2): viscosity (S1), momentum sources (S2), compact right-hand sides and level-(n+1)
// operator weights (S3/S4), increments, wall conditions, divergence and the modified
// artificial-compressibility pressure correction (S6-S8). The device code is in
// hosc_step_dev.cuh; one thread per node.

#include <math.h>

#include "hosc_step_dev.cuh"

namespace hosc {

void launch_arm(const Fields& F, int stop_steady, cudaStream_t s) {
  k_arm<<<1, 32, 0, s>>>(F.halt, F.ring_pos, F.steady_stop, stop_steady);
}

int red_blocks(long count, int threads) { return (int)((count + threads - 1) / threads); }


void launch_shadow(const DevParams& P, const Fields& F, int cur, int both, cudaStream_t s) {
  const int n3 = P.N * P.N * P.N;
  k_shadow<<<red_blocks(n3), kThreads, 0, s>>>(n3, F.u[cur], F.v[cur], F.w[cur], F.th, F.p,
                                               F.us[cur], F.vs[cur], F.ws[cur], F.ths, F.ps, F.halt);
  if (both) {
    const int o = 1 - cur;
    k_shadow<<<red_blocks(n3), kThreads, 0, s>>>(n3, F.u[o], F.v[o], F.w[o], nullptr, nullptr,
                                                 F.us[o], F.vs[o], F.ws[o], nullptr, nullptr,
                                                 F.halt);
  }
}

// Grid of a sweep over all nodes: the interior nodes' blocks, then the boundary nodes'.
struct SweepGrid {
  int threads;
  unsigned nbi, nb;
};
static SweepGrid sweep_grid(const DevParams& P) {
  const long n3 = (long)P.N * P.N * P.N, ni = P.N - 2, ni3 = ni * ni * ni;
  SweepGrid g;
  g.threads = P.sweep_fp32 ? kThreads : kFp64Threads;
  g.nbi = red_blocks(ni3, g.threads);
  g.nb = g.nbi + red_blocks(n3 - ni3, g.threads);
  return g;
}

void launch_viscosity(const DevParams& P, const Fields& F, int cur, cudaStream_t s) {
  const SweepGrid g = sweep_grid(P);
  if (P.sweep_fp32)
    launch_pdl(k_viscosity<float>, g.nb, g.threads, 0, s, P, F.us[cur], F.vs[cur], F.ws[cur],
               reinterpret_cast<float*>(F.eta), reinterpret_cast<float*>(F.L[cur]), F.halt, g.nbi);
  else
    launch_pdl(k_viscosity<double>, g.nb, g.threads, 0, s, P, F.u[cur], F.v[cur], F.w[cur], F.eta,
               F.L[cur], F.halt, g.nbi);
}

void launch_sources(const DevParams& P, const Fields& F, int cur, cudaStream_t s) {
  ulonglong2* exch = P.coop ? F.exch : nullptr;
  const SweepGrid g = sweep_grid(P);
  if (P.sweep_fp32)
    launch_pdl(k_sources<float>, g.nb, g.threads, 0, s, P, F.us[cur], F.vs[cur], F.ws[cur], F.ths,
               F.ps, reinterpret_cast<const float*>(F.eta), reinterpret_cast<float*>(F.Eu[cur]),
               reinterpret_cast<float*>(F.Ev[cur]), reinterpret_cast<float*>(F.Ew[cur]), F.halt,
               g.nbi, exch);
  else
    launch_pdl(k_sources<double>, g.nb, g.threads, 0, s, P, F.u[cur], F.v[cur], F.w[cur], F.th, F.p,
               F.eta, F.Eu[cur], F.Ev[cur], F.Ew[cur], F.halt, g.nbi, exch);
}

template <class Tc, class Ts>
static void rhs_t(const DevParams& P, const Fields& F, int cur, cudaStream_t s) {
  const long ni = P.N - 2;
  const int o = 1 - cur;
  auto T = [](double* p) { return reinterpret_cast<const Tc*>(p); };
  // the state: float copies for FP32 sweeps, the double arrays otherwise
  const Tc *u, *v, *w, *th, *up, *vp, *wp;
  if (sizeof(Tc) == sizeof(float)) {
    u = (const Tc*)F.us[cur]; v = (const Tc*)F.vs[cur]; w = (const Tc*)F.ws[cur];
    th = (const Tc*)F.ths;
    up = (const Tc*)F.us[o]; vp = (const Tc*)F.vs[o]; wp = (const Tc*)F.ws[o];
  } else {
    u = (const Tc*)F.u[cur]; v = (const Tc*)F.v[cur]; w = (const Tc*)F.w[cur];
    th = (const Tc*)F.th;
    up = (const Tc*)F.u[o]; vp = (const Tc*)F.v[o]; wp = (const Tc*)F.w[o];
  }
  const int threads = sizeof(Tc) == sizeof(float) ? kThreads : kFp64Threads;
  launch_pdl(k_rhs<Tc, Ts>, red_blocks(ni * ni * ni, threads), threads, 0, s, P, u, v, w, th,
             T(F.L[cur]), T(F.Eu[cur]), T(F.Ev[cur]), T(F.Ew[cur]), T(F.L[o]), up, vp, wp,
             T(F.Eu[o]), T(F.Ev[o]), T(F.Ew[o]), F);
}

void launch_rhs(const DevParams& P, const Fields& F, int cur, cudaStream_t s) {
  if (P.sweep_fp32)
    rhs_t<float, float>(P, F, cur, s);
  else if (P.krylov_fp32)
    rhs_t<double, float>(P, F, cur, s);
  else
    rhs_t<double, double>(P, F, cur, s);
}

void launch_finish(const DevParams& P, const Fields& F, cudaStream_t s) {
  k_finish_record<<<1, 32, 0, s>>>(P, F);
}

void launch_update(const DevParams& P, const Fields& F, int cur, int record, cudaStream_t s) {
  const long N = P.N, n3 = N * N * N, ni = N - 2;
  const int b_all = red_blocks(n3), b_int = red_blocks(ni * ni * ni);
  const int b_div = b_int + red_blocks(2 * ni * N + 2 * ni * ni);
  const int b_walls = red_blocks(n3 - ni * ni * ni);
  // the first follows the conditional node of a captured step: a plain launch
  if (P.krylov_fp32) k_increment<float><<<b_all, kThreads, 0, s>>>(P, F, cur, b_all);
  else k_increment<double><<<b_all, kThreads, 0, s>>>(P, F, cur, b_all);
  launch_pdl(k_div_walls, b_div, kThreads, 0, s, P, F, 1 - cur, b_int, b_div);
  launch_pdl(k_pressure_correct, b_int, kThreads, 0, s, P, F);
  launch_pdl(k_pressure_walls, b_walls, kThreads, 0, s, P, F, record, b_walls);
}

}  // namespace hosc
