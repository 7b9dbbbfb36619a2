// Device code of the step kernels other than the Krylov solver: S1 viscosity, S2 momentum sources,
// S3/S4 compact right-hand sides and operator weights, S6-S8 increments, wall conditions,
// divergence, pressure correction, the step record, and the float state copies (Punia & Ray,
// arXiv:2411.06563, Sec. 2.2). Each kernel is a device body taking its (virtual) block index, so
// that the one-launch-per-kernel path (hosc_step.cu) and the persistent round kernel of the pool
// (hosc_round.cu) run the same code; the __global__ wrappers launch one block per index.
//
// Layout: every field is N^3 doubles, x fastest (node (i,j,k) at i + N*(j + N*k)). One thread per
// node; node-linear thread indexing keeps consecutive threads on consecutive x.
#pragma once

#include <math.h>

#include <type_traits>

#include "hosc_device.cuh"
#include "hosc_internal.h"
#include "hosc_krylov4.cuh"

namespace hosc {

namespace {

// |x|, or +inf when x is not finite, on the integer units (see max_nonneg).
__device__ __forceinline__ double absfin(double x) {
  const long long b = __double_as_longlong(x) & 0x7fffffffffffffffLL;
  return b < 0x7ff0000000000000LL ? __longlong_as_double(b) : INFINITY;
}
__device__ __forceinline__ float absfinf(float x) {
  const int b = __float_as_int(x) & 0x7fffffff;
  return b < 0x7f800000 ? __int_as_float(b) : INFINITY;
}
__device__ __forceinline__ int inward(int a, int N) { return a == 0 ? 1 : (a == N - 1 ? N - 2 : a); }
__device__ __forceinline__ int on_wall(int a, int N) { return (a == 0) | (a == N - 1); }

// Arithmetic type helpers: the sweeps run in T = double (FP64 path, mixed-precision defect
// steps) or T = float (mixed-precision sweeps: the double state is rounded to float as it is
// loaded; the rounding noise this leaves in the right-hand side is what the FP64 defect sweeps
// remove near the steady state).
template <class T> __device__ __forceinline__ T tpow(T x, T y);
template <> __device__ __forceinline__ double tpow<double>(double x, double y) { return pow(x, y); }
template <> __device__ __forceinline__ float tpow<float>(float x, float y) { return powf(x, y); }


// A scalar parameter in the arithmetic type T: the double, or its float copy made on the host.
template <class T>
__device__ __forceinline__ T par(double d, float f) {
  if constexpr (sizeof(T) == sizeof(float)) return f;
  else return d;
}

__device__ __forceinline__ int node32(int i, int j, int k, int N) { return i + N * (j + N * k); }

// Node number t of the y faces (x interior, all z), then of the z faces (x, y interior):
// 0 <= t < 2 (N-2) N + 2 (N-2)^2, x fastest.
__device__ __forceinline__ void boundary_yz(int t, int N, int& i, int& j, int& k) {
  const int ni = N - 2;
  if (t < 2 * ni * N) {
    const int side = t / (ni * N), r = t - side * ni * N;
    const int q = r / ni;
    i = 1 + (r - q * ni);
    k = q;
    j = side ? N - 1 : 0;
  } else {
    const int u = t - 2 * ni * N;
    const int side = u / (ni * ni), r = u - side * ni * ni;
    const int q = r / ni;
    i = 1 + (r - q * ni);
    j = 1 + q;
    k = side ? N - 1 : 0;
  }
}

// Node number t of the cube's boundary, 0 <= t < N^3 - (N-2)^3: the x faces, then the y and z
// faces as in boundary_yz.
__device__ __forceinline__ void boundary_node(int t, int N, int& i, int& j, int& k) {
  const int N2 = N * N;
  if (t < 2 * N2) {
    const int side = t / N2, r = t - side * N2;
    const int q = r / N;
    j = r - q * N;
    k = q;
    i = side ? N - 1 : 0;
  } else {
    boundary_yz(t - 2 * N2, N, i, j, k);
  }
}

template <class T>
struct Grad9T {
  T ux, uy, uz, vx, vy, vz, wx, wy, wz;
};

// 1/(2 h_d) of the directions in the arithmetic type T.
template <class T>
struct Inv2h {
  T x, y, z;
};
template <class T>
__device__ __forceinline__ Inv2h<T> inv2h(const DevParams& P) {
  if constexpr (sizeof(T) == sizeof(float)) return {P.inv2f[0], P.inv2f[1], P.inv2f[2]};
  else return {P.inv2[0], P.inv2[1], P.inv2[2]};
}
// The constants of the right-hand sides in the arithmetic type T.
template <class T>
__device__ __forceinline__ const RhsC<T>& rhs_constants(const DevParams& P) {
  if constexpr (sizeof(T) == sizeof(float)) return P.rcf;
  else return P.rc;
}

// Derivative along an axis with memory stride st at a node of coordinate a along it. WALL: the node
// may lie on a wall of that axis (second-order one-sided there); otherwise central.
template <bool WALL, class T>
__device__ __forceinline__ T grad_axis_t(const T* HOSC_RESTRICT f, int c, int a, int N, int st,
                                         T inv2h) {
  if constexpr (WALL) {
    if (a == 0) return (T(-3) * f[c] + T(4) * f[c + st] - f[c + 2 * st]) * inv2h;
    if (a == N - 1) return (T(3) * f[c] - T(4) * f[c - st] + f[c - 2 * st]) * inv2h;
  }
  return (f[c + st] - f[c - st]) * inv2h;
}

template <bool WALL, class T>
__device__ __forceinline__ Grad9T<T> velocity_gradients_t(const T* HOSC_RESTRICT u,
                                                          const T* HOSC_RESTRICT v,
                                                          const T* HOSC_RESTRICT w, int i, int j,
                                                          int k, int N, const Inv2h<T>& i2) {
  const int sy = N, sz = N * N, c = node32(i, j, k, N);
  Grad9T<T> g;
  g.ux = grad_axis_t<WALL>(u, c, i, N, 1, i2.x);
  g.uy = grad_axis_t<WALL>(u, c, j, N, sy, i2.y);
  g.uz = grad_axis_t<WALL>(u, c, k, N, sz, i2.z);
  g.vx = grad_axis_t<WALL>(v, c, i, N, 1, i2.x);
  g.vy = grad_axis_t<WALL>(v, c, j, N, sy, i2.y);
  g.vz = grad_axis_t<WALL>(v, c, k, N, sz, i2.z);
  g.wx = grad_axis_t<WALL>(w, c, i, N, 1, i2.x);
  g.wy = grad_axis_t<WALL>(w, c, j, N, sy, i2.y);
  g.wz = grad_axis_t<WALL>(w, c, k, N, sz, i2.z);
  return g;
}

// The sweeps over all nodes (S1, S2) run the interior nodes in their first nbi blocks and the
// boundary nodes in the others: with both in one warp (an x row has a wall node at either end)
// every third warp went through the one-sided forms of each derivative beside the central ones.
// Measured with the split: S1 in float 249 -> 146 us at 257^3 and 17.2 -> 14.4 us at 101^3, S2 in
// float 354 -> 198 and 20.9 -> 16.6 us, S2 in double 236 -> 123 us at 101^3.
// Calls f(WALL, i, j, k) for this thread's node.
template <class Fn>
__device__ __forceinline__ void sweep_node(int N, unsigned vbx, unsigned nbi, Fn f) {
  const int ni = N - 2;
  if (vbx < nbi) {
    const int t = (int)(vbx * blockDim.x + threadIdx.x);
    if (t >= ni * ni * ni) return;
    const int q = t / ni;
    f(std::false_type(), 1 + t - q * ni, 1 + q % ni, 1 + q / ni);
  } else {
    const int t = (int)((vbx - nbi) * blockDim.x + threadIdx.x);
    if (t >= N * N * N - ni * ni * ni) return;
    int i, j, k;
    boundary_node(t, N, i, j, k);
    f(std::true_type(), i, j, k);
  }
}

// ------------------------------------------------------------------------------------ S1

// x^(-(1 - e)/m) for an integer m in 2..64 and an e of rounding size: a float estimate y of 1e-6 and one
// third-order step of Newton's iteration on y^-m = x^(1 - e), y (1 - r)^(-1/m) to r^2 with r = x^e - x y^m
// (the r^3 term is below 1e-16 of y); y^m by squaring. Largest error found against 200-bit arithmetic
// over 20 000 x in [1e-12, 1e12] with e = 0: 0.75 units in the last place (m = 8), 0.79 (m = 64); about
// 15 FP64 instructions against some 130 of pow(). A rounded n leaves an e (n = 1 + 2/3 missed the power
// by 14 units at 1e18 without it): x^e = 1 + e ln x to first order, e ln x = e2 log2(x) below 1e-13, is
// put together on the integer units (as an FP64 sum it cost the sweep 3.5 % at 101^3).
__device__ __forceinline__ double inverse_root(double x, int m, float e2) {
  const float a = 1.0f / (float)m, lx = log2f((float)x);
  const double y = (double)exp2f(-a * lx);
  double p = 1.0, b = y;
  for (int e = m;;) {   // m is the same for every thread
    if (e & 1) p *= b;
    if ((e >>= 1) == 0) break;
    b *= b;
  }
  const float d = e2 * lx;
  // 1 + d: doubles lie 2^-52 apart above 1 and 2^-53 below
  const long long k = __float2int_rn(d * (d < 0.0f ? 9007199254740992.0f : 4503599627370496.0f));
  const double r = fma(-x, p, __longlong_as_double(0x3ff0000000000000LL + k));
  const float c2 = 0.5f * a * (1.0f + a);
  return fma(y, r * fma((double)c2, r, 1.0 / (double)m), y);
}

// eta = (I2 + eps)^((n-1)/2) (Eqs. 7-8), eta == 1 for n == 1; L = 1/(Pr eta) (Sec. 2.2 momentum
// coefficients). On cube edges and corners, where the one-sided strain rates of two or three
// no-slip walls vanish identically, I2 is taken at the node one step inward along each of those
// wall normals. In double, where 2/|n-1| is an integer m (n = 0.75 and 1.25: 8), the power is
// inverse_root: 303 -> 120 us per sweep at 101^3 with the split of sweep_node (FP64-bound); pow()
// for other indices and outside [1e-30, 1e30].
template <class T>
__device__ __forceinline__ void k_viscosity_body(const DevParams& P, const T* HOSC_RESTRICT u,
                                                 const T* HOSC_RESTRICT v, const T* HOSC_RESTRICT w,
                                                 T* HOSC_RESTRICT eta, T* HOSC_RESTRICT L,
                                                 const int* HOSC_RESTRICT halt, unsigned vbx,
                                                 unsigned nbi) {
  if (*halt) return;
  const int N = P.N;
  sweep_node(N, vbx, nbi, [&](auto wall, int i, int j, int k) {
    constexpr bool WALL = decltype(wall)::value;
    const int t = node32(i, j, k, N);
    if (P.newtonian) {
      eta[t] = T(1);
      L[t] = T(1) / par<T>(P.Pr, P.Prf);
      return;
    }
    if (WALL && on_wall(i, N) + on_wall(j, N) + on_wall(k, N) >= 2) {
      i = inward(i, N);
      j = inward(j, N);
      k = inward(k, N);
    }
    const Grad9T<T> g = velocity_gradients_t<WALL, T>(u, v, w, i, j, k, N, inv2h<T>(P));
    const T a = g.uz + g.wx, b = g.uy + g.vx, c = g.vz + g.wy;
    const T I2 = T(2) * (g.ux * g.ux + g.vy * g.vy + g.wz * g.wz) + a * a + b * b + c * c;
    const T x = I2 + par<T>(P.I2_eps, P.I2_epsf);
    if constexpr (sizeof(T) == sizeof(double)) {
      if (P.eta_root && x >= 1e-30 && x <= 1e30) {
        const double z = inverse_root(x, P.eta_root, P.eta_res);
        const bool thin = P.eta_exp < 0.0;   // the same for every thread
        eta[t] = thin ? z : 1.0 / z;
        L[t] = thin ? 1.0 / (P.Pr * z) : P.iPr * z;
        return;
      }
    }
    const T e = tpow<T>(x, par<T>(P.eta_exp, P.eta_expf));
    eta[t] = e;
    L[t] = T(1) / (par<T>(P.Pr, P.Prf) * e);
  });
}

template <class T>
__global__ void __launch_bounds__(kThreads) k_viscosity(DevParams P, const T* HOSC_RESTRICT u,
                                                        const T* HOSC_RESTRICT v,
                                                        const T* HOSC_RESTRICT w,
                                                        T* HOSC_RESTRICT eta, T* HOSC_RESTRICT L,
                                                        const int* HOSC_RESTRICT halt,
                                                        unsigned nbi) {
  pdl_wait_and_release();
  k_viscosity_body(P, u, v, w, eta, L, halt, blockIdx.x, nbi);
}

// ------------------------------------------------------------------------------------ S2

// E* of the x, y, z momentum equations: the conservative momentum equations divided through by
// Pr eta so that L = 1/(Pr eta):
//   E*_x = -p_x/(Pr eta) + (2/eta)(eps_xx eta_x + eps_yx eta_y + eps_zx eta_z)
//   E*_y = -p_y/(Pr eta) + (2/eta)(eps_xy eta_x + eps_yy eta_y + eps_zy eta_z) + Ra (theta - theta_ref)/eta
//   E*_z = -p_z/(Pr eta) + (2/eta)(eps_xz eta_x + eps_yz eta_y + eps_zz eta_z)
// Gradients are central inside and one-sided at wall nodes.
template <class T>
__device__ __forceinline__ void k_sources_body(const DevParams& P, const T* HOSC_RESTRICT u,
                                               const T* HOSC_RESTRICT v, const T* HOSC_RESTRICT w,
                                               const T* HOSC_RESTRICT th, const T* HOSC_RESTRICT p,
                                               const T* HOSC_RESTRICT eta, T* HOSC_RESTRICT Eu,
                                               T* HOSC_RESTRICT Ev, T* HOSC_RESTRICT Ew,
                                               const int* HOSC_RESTRICT halt, unsigned vbx,
                                               unsigned nbi) {
  if (*halt) return;
  const int N = P.N;
  sweep_node(N, vbx, nbi, [&](auto wall, int i, int j, int k) {
    constexpr bool WALL = decltype(wall)::value;
    const Inv2h<T> i2 = inv2h<T>(P);
    const int sy = N, sz = N * N, t = node32(i, j, k, N);
    const Grad9T<T> g = velocity_gradients_t<WALL, T>(u, v, w, i, j, k, N, i2);
    const T ex = grad_axis_t<WALL>(eta, t, i, N, 1, i2.x);
    const T ey = grad_axis_t<WALL>(eta, t, j, N, sy, i2.y);
    const T ez = grad_axis_t<WALL>(eta, t, k, N, sz, i2.z);
    const T px = grad_axis_t<WALL>(p, t, i, N, 1, i2.x);
    const T py = grad_axis_t<WALL>(p, t, j, N, sy, i2.y);
    const T pz = grad_axis_t<WALL>(p, t, k, N, sz, i2.z);
    const T e = eta[t];
    const T exy = T(0.5) * (g.uy + g.vx), exz = T(0.5) * (g.uz + g.wx),
            eyz = T(0.5) * (g.vz + g.wy);
    const T ie = T(1) / e;
    const T a = ie * par<T>(P.iPr, P.iPrf), b = T(2) * ie;
    const T buoy = par<T>(P.Ra, P.Raf) * (th[t] - par<T>(P.theta_ref, P.theta_reff));
    Eu[t] = -px * a + b * (g.ux * ex + exy * ey + exz * ez);
    // an FP64 division is some 15 instructions of the pipe that bounds the double form
    Ev[t] = -py * a + b * (exy * ex + g.vy * ey + eyz * ez) +
            (sizeof(T) == sizeof(double) ? buoy * ie : buoy / e);
    Ew[t] = -pz * a + b * (exz * ex + eyz * ey + g.wz * ez);
  });
}

template <class T>
__global__ void __launch_bounds__(kThreads) k_sources(DevParams P, const T* HOSC_RESTRICT u,
                                                     const T* HOSC_RESTRICT v,
                                                     const T* HOSC_RESTRICT w,
                                                     const T* HOSC_RESTRICT th,
                                                     const T* HOSC_RESTRICT p,
                                                     const T* HOSC_RESTRICT eta,
                                                     T* HOSC_RESTRICT Eu, T* HOSC_RESTRICT Ev,
                                                     T* HOSC_RESTRICT Ew,
                                                     const int* HOSC_RESTRICT halt, unsigned nbi,
                                                     ulonglong2* exch) {
  pdl_wait_and_release();
  if (exch)   // the exchange buffer of the one-launch solve (in k_rhs this cost the float form 20 %)
    for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < (unsigned)kExchValues;
         e += gridDim.x * blockDim.x)
      exch[e] = make_ulonglong2(0ull, 0ull);
  k_sources_body(P, u, v, w, th, p, eta, Eu, Ev, Ew, halt, blockIdx.x, nbi);
}

// ------------------------------------------------------------------------------------ S3/S4

// 7-point neighbourhood order: centre, x+, x-, y+, y-, z+, z-.
template <class T, class S>
__device__ __forceinline__ void load7(const S* HOSC_RESTRICT a, long c, long sy, long sz, T f[7]) {
  f[0] = (T)a[c];
  f[1] = (T)a[c + 1];
  f[2] = (T)a[c - 1];
  f[3] = (T)a[c + sy];
  f[4] = (T)a[c - sy];
  f[5] = (T)a[c + sz];
  f[6] = (T)a[c - sz];
}

// 19-point neighbourhood: 0 c, 1 x+, 2 x-, 3 y+, 4 y-, 5 z+, 6 z-,
// 7 x+y+, 8 x-y+, 9 x+y-, 10 x-y-, 11 y+z+, 12 y-z+, 13 y+z-, 14 y-z-,
// 15 z+x+, 16 z-x+, 17 z+x-, 18 z-x-.
template <class T>
__device__ __forceinline__ void load19(const T* HOSC_RESTRICT a, long c, long sy, long sz,
                                       T f[19]) {
  load7<T, T>(a, c, sy, sz, f);
  f[7] = (T)a[c + 1 + sy];
  f[8] = (T)a[c - 1 + sy];
  f[9] = (T)a[c + 1 - sy];
  f[10] = (T)a[c - 1 - sy];
  f[11] = (T)a[c + sy + sz];
  f[12] = (T)a[c - sy + sz];
  f[13] = (T)a[c + sy - sz];
  f[14] = (T)a[c - sy - sz];
  f[15] = (T)a[c + sz + 1];
  f[16] = (T)a[c - sz + 1];
  f[17] = (T)a[c + sz - 1];
  f[18] = (T)a[c - sz - 1];
}

// What a 7-point neighbourhood gives to Eq. (5): its centre, the sum of its second differences
// times h_d^2, and f_{+d} - f_{-d} of each direction.
template <class T>
struct Star {
  T c, lap, b[3];
};

template <class T>
__device__ __forceinline__ Star<T> star(const T f[7]) {
  Star<T> s;
  s.c = f[0];
  s.b[0] = f[1] - f[2];
  s.b[1] = f[3] - f[4];
  s.b[2] = f[5] - f[6];
  s.lap = ((f[1] + f[2]) + (f[3] + f[4]) + (f[5] + f[6])) - T(6) * f[0];
  return s;
}

// [(dx^2 - G dx) h^2/12 + (dy^2 - H dy) k^2/12 + (dz^2 - I dz) l^2/12] f, with v24 = (G h, H k,
// I l)/24
template <class T>
__device__ __forceinline__ T compact_terms(const Star<T>& s, const T v24[3]) {
  return T(1.0 / 12.0) * s.lap - v24[0] * s.b[0] - v24[1] * s.b[1] - v24[2] * s.b[2];
}

// The level-n operator of Eq. (5),
//  -al dx^2 - be dy^2 - ga dz^2 + M1 dx + M2 dy + M3 dz
//  - (h^2+k^2)/12 [dx^2 dy^2 - H dx^2 dy - G dx dy^2 - p1 dx dy] - (yz group) - (zx group),
// as weights of the 18 neighbours (the centre's is minus their sum, since no term acts on a
// constant), for the systems with the same G*, H*, I* (K* = 0). One set of weights serves u, v and
// w: 18 differences and 18 fused multiply-adds a system in place of some 110 operations when each
// system evaluates the difference operators. Applied to f_i - f_0 (exact for neighbours within a
// factor of two), so that nothing of the size |f|/h^2 cancels.
template <class T>
struct LevelN {
  T V[3], v24[3];
  T w[18];   // x+, x-, y+, y-, z+, z-, then the edges in load19's order
};

// V: G*, H*, I* at the 7 points (as stars), Vp: at level n-1 (used when hist).
template <class T>
__device__ __forceinline__ LevelN<T> level_n(const Star<T> (&V)[3], const T (&Vp)[3], bool hist,
                                             const RhsC<T>& k) {
  LevelN<T> o;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    o.V[d] = V[d].c;
    o.v24[d] = V[d].c * k.h24[d];
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    // al = 1 + h^2/12 (G^2 - 2 dx G); M1 = [1 + compact terms + (dt/2) dt^-] G
    const T al = T(1) + (k.s12[d] * V[d].c) * V[d].c - k.h12[d] * V[d].b[d];
    T M = V[d].c + compact_terms(V[d], o.v24);
    if (hist) M += T(0.5) * (V[d].c - Vp[d]);
    const T S = k.face[d] - al * k.isq[d];
    const T D = M * k.i2[d] - V[d].c * k.kd[d];
    o.w[2 * d] = S + D;
    o.w[2 * d + 1] = S - D;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {   // the pair (a, b)
    const int a = q, b = (q + 1) % 3;
    // p1 = -G H + 2/(h^2+k^2) (k^2 dy G + h^2 dx H), and cyclically
    const T p1 = k.xa[q] * V[a].b[b] + k.xb[q] * V[b].b[a] - V[a].c * V[b].c;
    const T Ea = k.ea[q] * V[a].c, Eb = k.eb[q] * V[b].c, Ec = k.ec[q] * p1;
    const T hi = Eb - k.e0[q], lo = -k.e0[q] - Eb, up = Ea + Ec, dn = Ea - Ec;
    o.w[6 + 4 * q] = hi + up;       // a+ b+
    o.w[6 + 4 * q + 1] = hi - up;   // a- b+
    o.w[6 + 4 * q + 2] = lo + dn;   // a+ b-
    o.w[6 + 4 * q + 3] = lo - dn;   // a- b-
  }
  return o;
}

template <class T>
__device__ __forceinline__ T apply_level_n(const LevelN<T>& o, const T f[19]) {
  T s = T(0);
#pragma unroll
  for (int q = 0; q < 18; ++q) s += o.w[q] * (f[q + 1] - f[0]);
  return s;
}

// Diagonal pseudo-time mass where the cell Reynolds number is high: the level-n operator carries
// (h_d^2/12)|G*|^2 delta^2 explicitly, and for the grid mode alternating in all three directions
// the level-(n+1) operator is only 2 dt (1/h^2 + 1/k^2 + 1/l^2) = 6 dt s3, so that mode grows once
// |G*|^2 > 24 s3 (and the mode alternating in one direction once dt |G*|^2 > 4 L). Zero in
// resolved flows; it changes the pseudo-time path only, never the steady state.
template <class T>
__device__ __forceinline__ T pseudo_time_mass(T G, T H, T I, T L, T dt, T s3, T kappa) {
  const T g2 = G * G + H * H + I * I;
  const T g6 = g2 * T(1.0 / 6.0);
  const T s = fmax(T(0), fmax(dt * (g6 - s3), dt * g6 - T(2.0 / 3.0) * L));
  return kappa * s;
}

// Right-hand sides of the increment form of Eq. (6),  A (chi^{n+1} - chi^n) = dt (R - B chi^n),
// for u, v, w, theta at interior nodes, and the level-(n+1) operators of the momentum and energy
// systems. Tc: arithmetic and the type of L, E*; Ts: type of the outputs.
//
// Along direction d the +d and -d neighbours of the level-(n+1) operator weigh S_d - B_d and
// S_d + B_d. Of Eq. (6)'s L (M_d/h_d^2 -+ (M_d V_d - M_{14+d})/(2 h_d)) with M_d = -dt/(2L) +
// h_d^2/12 and M_{14+d} = h_d^2/(6L) d_d L, multiplying L through leaves no division:
// S_d = -dt/(2 h_d^2) + L/12, B_d = ((-dt/2 + h_d^2 L/12) V_d - (h_d/12)(L_+ - L_-))/(2 h_d), and
// the diagonal is L/2 + dt (1/h^2 + 1/k^2 + 1/l^2) + M18 + the pseudo-time mass.
//
// The FP64 pipe bounds the double forms (a warp's FP64 instruction takes 16 cycles of its SM): about
// 500 FP64 instructions a node against 1100 when each system evaluated the difference operators:
// 1742 -> 926 us at 101^3, 72 -> 21 us at 21^3 (there with the smaller blocks of kFp64Threads). The
// float form is bound by issue slots: 51.3 -> 39.1 us at 101^3, 823 -> 661 us at 257^3.
template <class Tc, class Ts>
__device__ __forceinline__ void k_rhs_body(const DevParams& P, const Tc* HOSC_RESTRICT u,
                                           const Tc* HOSC_RESTRICT v, const Tc* HOSC_RESTRICT w,
                                           const Tc* HOSC_RESTRICT th, const Tc* HOSC_RESTRICT L,
                                           const Tc* HOSC_RESTRICT Eu, const Tc* HOSC_RESTRICT Ev,
                                           const Tc* HOSC_RESTRICT Ew, const Tc* HOSC_RESTRICT Lp,
                                           const Tc* HOSC_RESTRICT up, const Tc* HOSC_RESTRICT vp,
                                           const Tc* HOSC_RESTRICT wp, const Tc* HOSC_RESTRICT Eup,
                                           const Tc* HOSC_RESTRICT Evp, const Tc* HOSC_RESTRICT Ewp,
                                           const Fields& F, unsigned vbx) {
  const int N = P.N;
  const unsigned ni = N - 2;
  const unsigned t = vbx * blockDim.x + threadIdx.x;
  if (t >= ni * ni * ni || *F.halt) return;
  const unsigned q = t / ni;
  const int i = 1 + (int)(t - q * ni), j = 1 + (int)(q % ni), k = 1 + (int)(q / ni);
  const long sy = N, sz = (long)N * N;
  const long c = node(i, j, k, N);
  const RhsC<Tc>& rc = rhs_constants<Tc>(P);
  if (t < 4) start_system(P, F, (int)t);   // the solve's scalars
  const bool hist = P.have_prev != 0;
  const Tc kap = par<Tc>(P.a_boost, P.a_boostf);
  Tc rv[4], Bm[3], Be[3], Dm, De, Lc;   // right-hand sides and compact operators, stored at the end

  // ---------------- momentum: L = 1/(Pr eta), G* = u L, H* = v L, I* = w L, K* = 0
  {
    Tc L7[7], f7[7];
    load7<Tc, Tc>(L, c, sy, sz, L7);
    Lc = L7[0];
    const Tc Lpc = hist ? Lp[c] : Lc;
    Star<Tc> V[3];
    Tc Vp[3] = {Tc(0), Tc(0), Tc(0)};
    const Tc* const vel[3] = {u, v, w};
    const Tc* const old[3] = {up, vp, wp};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      load7<Tc, Tc>(vel[d], c, sy, sz, f7);
#pragma unroll
      for (int s = 0; s < 7; ++s) f7[s] *= L7[s];
      V[d] = star(f7);
      if (hist) Vp[d] = old[d][c] * Lpc;
    }
    const LevelN<Tc> op = level_n<Tc>(V, Vp, hist, rc);
    // one momentum system: source E (level n, and n-1 when kept) and the field X
    auto system = [&](const Tc* HOSC_RESTRICT E, const Tc* HOSC_RESTRICT Ep,
                      const Tc* HOSC_RESTRICT X) {
      Tc E7[7], f19[19];
      load7<Tc, Tc>(E, c, sy, sz, E7);
      Tc R = E7[0] + compact_terms(star(E7), op.v24);
      if (hist) R += Tc(0.5) * (E7[0] - Ep[c]);
      load19<Tc>(X, c, sy, sz, f19);
      return rc.dt * (R - apply_level_n(op, f19));
    };
    rv[0] = system(Eu, Eup, u);
    rv[1] = system(Ev, Evp, v);
    rv[2] = system(Ew, Ewp, w);
    const Star<Tc> sL = star(L7);
    Tc M18 = compact_terms(sL, op.v24);
    if (hist) M18 += Tc(0.5) * (Lc - Lpc);
    // keep the extrapolated mass positive where L changes fast (the steady state is unaffected)
    const Tc alim = par<Tc>(P.a_limit, P.a_limitf);
    if (alim > Tc(0)) M18 = fmax(M18, -alim * Lc);
#pragma unroll
    for (int d = 0; d < 3; ++d)
      Bm[d] = ((rc.hdt + rc.s12[d] * Lc) * op.V[d] - rc.h12[d] * sL.b[d]) * rc.i2[d];
    Dm = (Tc(0.5) * Lc + rc.dtq) + M18;
    if (kap > Tc(0))
      Dm += pseudo_time_mass<Tc>(op.V[0], op.V[1], op.V[2], Lc, rc.dt, rc.s3, kap);
  }
  // ---------------- energy: L = 1, G* = u, H* = v, I* = w, K* = E* = 0
  {
    Tc f7[7], f19[19];
    Star<Tc> V[3];
    Tc Vp[3] = {Tc(0), Tc(0), Tc(0)};
    const Tc* const vel[3] = {u, v, w};
    const Tc* const old[3] = {up, vp, wp};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      load7<Tc, Tc>(vel[d], c, sy, sz, f7);
      V[d] = star(f7);
      if (hist) Vp[d] = old[d][c];
    }
    const LevelN<Tc> op = level_n<Tc>(V, Vp, hist, rc);
    load19<Tc>(th, c, sy, sz, f19);
    rv[3] = -rc.dt * apply_level_n(op, f19);
#pragma unroll
    for (int d = 0; d < 3; ++d) Be[d] = ((rc.hdt + rc.s12[d]) * rc.i2[d]) * op.V[d];
    De = Tc(0.5) + rc.dtq;
    if (kap > Tc(0))
      De += pseudo_time_mass<Tc>(op.V[0], op.V[1], op.V[2], Tc(1), rc.dt, rc.s3, kap);
  }
  const Tc dm = Dm != Tc(0) ? Dm : Tc(1), de = De != Tc(0) ? De : Tc(1);
  if (P.precond) {   // Jacobi row scaling: each right-hand side over its row's diagonal
#pragma unroll
    for (int s = 0; s < 3; ++s) rv[s] /= dm;
    rv[3] /= de;
  }
  if constexpr (sizeof(Ts) == sizeof(float)) {   // interleaved float storage, compact operators
    F.kr0[c] = make_float4((float)rv[0], (float)rv[1], (float)rv[2], (float)rv[3]);
    F.kwm[c] = make_float4((float)Bm[0], (float)Bm[1], (float)Bm[2], (float)Dm);
    F.kwe[c] = make_float4((float)Be[0], (float)Be[1], (float)Be[2], (float)De);
    F.kL[c] = (float)Lc;
  } else {                                         // planar double storage
#pragma unroll
    for (int s = 0; s < 4; ++s) F.rhs[s][c] = (double)rv[s];
    Tc Am[7], Ae[7];
    Am[0] = Dm;
    Ae[0] = De;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const Tc Sm = rc.cs[d] + Tc(1.0 / 12.0) * Lc, Se = rc.cs[d] + Tc(1.0 / 12.0);
      Am[1 + 2 * d] = Sm - Bm[d];
      Am[2 + 2 * d] = Sm + Bm[d];
      Ae[1 + 2 * d] = Se - Be[d];
      Ae[2 + 2 * d] = Se + Be[d];
    }
    if (P.precond) {   // the weights too (the compact float operators divide by D when applied)
#pragma unroll
      for (int s = 0; s < 7; ++s) {
        Am[s] /= dm;
        Ae[s] /= de;
      }
    }
#pragma unroll
    for (int s = 0; s < 7; ++s) {
      F.Am[s][c] = (double)Am[s];
      F.Ae[s][c] = (double)Ae[s];
    }
  }
}

// The float build is bounded to 80 registers (three 256-thread blocks per SM), the double builds to
// 168 (six blocks of kFp64Threads).
template <class Tc, class Ts>
__global__ void __launch_bounds__(sizeof(Tc) == sizeof(float) ? kThreads : kFp64Threads,
                                  sizeof(Tc) == sizeof(float) ? 3 : 6) k_rhs(
    DevParams P, const Tc* HOSC_RESTRICT u, const Tc* HOSC_RESTRICT v,
    const Tc* HOSC_RESTRICT w, const Tc* HOSC_RESTRICT th, const Tc* HOSC_RESTRICT L,
    const Tc* HOSC_RESTRICT Eu, const Tc* HOSC_RESTRICT Ev, const Tc* HOSC_RESTRICT Ew,
    const Tc* HOSC_RESTRICT Lp, const Tc* HOSC_RESTRICT up, const Tc* HOSC_RESTRICT vp,
    const Tc* HOSC_RESTRICT wp, const Tc* HOSC_RESTRICT Eup, const Tc* HOSC_RESTRICT Evp,
    const Tc* HOSC_RESTRICT Ewp, Fields F) {
  pdl_wait_and_release();
  k_rhs_body<Tc, Ts>(P, u, v, w, th, L, Eu, Ev, Ew, Lp, up, vp, wp, Eup, Evp, Ewp, F,
                     blockIdx.x);
}

// ------------------------------------------------------------------------------------ S6-S8
//
// Four launches: the increments; div V and the adiabatic walls (both need the increments of
// neighbours); the pressure correction (needs max|div V|); the pressure walls (need the corrected
// pressure). In mixed precision each also writes the float copies of what it writes, and the last
// block of the last one appends the step record: seven launches before, whose latencies were most of
// their time below 64^3 (45 -> 29 us a step at 41^3 mixed beside a
// launch for the copies, 91 + 12 -> 81 us at 101^3).

// chi^{n+1} = chi^n + x at interior nodes (u, v, w into the other buffer, theta in place); wall
// velocities are carried over. Max |x| over the four systems goes to the step record.
template <class Ts>
__device__ __forceinline__ void k_increment_body(const DevParams& P, const Fields& F, int cur,
                                                 int nblocks, unsigned vbx) {
  if (*F.halt) return;
  const unsigned N = P.N;
  const unsigned n3 = N * N * N;
  const unsigned t = vbx * blockDim.x + threadIdx.x;
  double m[2] = {0.0, 0.0};   // max |x| of u, v, w and of theta
  if (t < n3) {
    const unsigned q = t / N;
    const unsigned i = t - q * N, j = q % N, k = q / N;
    const bool inner = i > 0 && j > 0 && k > 0 && i < N - 1 && j < N - 1 && k < N - 1;
    double u = F.u[cur][t], v = F.v[cur][t], w = F.w[cur][t];
    if (inner) {
      double xu, xv, xw, xt;
      if constexpr (sizeof(Ts) == sizeof(float)) {   // interleaved float increments
        const float4 x4 = F.kx[t];
        xu = x4.x;
        xv = x4.y;
        xw = x4.z;
        xt = x4.w;
        // magnitudes in float (exact), widened once
        m[0] = fmaxf(fmaxf(absfinf(x4.x), absfinf(x4.y)), absfinf(x4.z));
        m[1] = absfinf(x4.w);
      } else {
        xu = F.x[0][t];
        xv = F.x[1][t];
        xw = F.x[2][t];
        xt = F.x[3][t];
        m[0] = max_nonneg(max_nonneg(absfin(xu), absfin(xv)), absfin(xw));
        m[1] = absfin(xt);
      }
      u += xu;
      v += xv;
      w += xw;
      const double th = F.th[t] + xt;
      F.th[t] = th;
      if constexpr (sizeof(Ts) == sizeof(float)) F.ths[t] = (float)th;
    }
    F.u[1 - cur][t] = u;
    F.v[1 - cur][t] = v;
    F.w[1 - cur][t] = w;
    if constexpr (sizeof(Ts) == sizeof(float)) {
      F.us[1 - cur][t] = (float)u;
      F.vs[1 - cur][t] = (float)v;
      F.ws[1 - cur][t] = (float)w;
    }
  }
  if (const double* tot = grid_total<MaxD, 2>(m, F.rb, vbx, nblocks)) {
    if (threadIdx.x == 0) {
      // an inner pressure pass changes u, v, w only: theta's change stays that of the first pass
      if (!P.inner_pass) F.rec->res_theta = tot[1];
      F.rec->res = fmax(tot[0], F.rec->res_theta);
    }
  }
}

template <class Ts>
__global__ void __launch_bounds__(kThreads) k_increment(DevParams P, Fields F, int cur,
                                                        int nblocks) {
  pdl_wait_and_release();
  k_increment_body<Ts>(P, F, cur, nblocks, blockIdx.x);
}

// Extrapolation weights along one axis for a wall condition of zero normal derivative:
// (4 f_1 - f_2)/3 at the first wall, mirrored at the second; identity inside.
__device__ __forceinline__ int wall_weights(int a, int N, int idx[2], double wt[2]) {
  if (a == 0) {
    idx[0] = 1; idx[1] = 2; wt[0] = 4.0 / 3.0; wt[1] = -1.0 / 3.0;
    return 2;
  }
  if (a == N - 1) {
    idx[0] = N - 2; idx[1] = N - 3; wt[0] = 4.0 / 3.0; wt[1] = -1.0 / 3.0;
    return 2;
  }
  idx[0] = a; wt[0] = 1.0;
  return 1;
}

// Blocks below nbi: central div V^{n+1} at interior nodes and its maximum. The others: adiabatic walls
// y = 0, 1 and z = 0, 1 (x interior), theta_b = (4 theta_1 - theta_2)/3 along each wall normal the
// node lies on (on the y-z edges, the product of the two); the hot and cold walls keep theta = 1
// and theta = 0. Max |change| joins the step record.
__device__ __forceinline__ void k_div_walls_body(const DevParams& P, const Fields& F, int nxt,
                                                 int nbi, int nblocks, unsigned vbx) {
  if (*F.halt) return;
  const int N = P.N, ni = N - 2;
  double m[2] = {0.0, 0.0};   // |div V|, |change of theta|
  if ((int)vbx < nbi) {
    const int t = (int)(vbx * blockDim.x + threadIdx.x);
    if (t < ni * ni * ni) {
      const int q = t / ni, i = 1 + (t - q * ni), j = 1 + q % ni, k = 1 + q / ni;
      const int c = node32(i, j, k, N), sy = N, sz = N * N;
      const double* u = F.u[nxt];
      const double* v = F.v[nxt];
      const double* w = F.w[nxt];
      const double d = (u[c + 1] - u[c - 1]) * P.inv2[0] + (v[c + sy] - v[c - sy]) * P.inv2[1] +
                       (w[c + sz] - w[c - sz]) * P.inv2[2];
      F.div[c] = d;
      m[0] = absfin(d);
    }
  } else {
    const int t = ((int)vbx - nbi) * blockDim.x + threadIdx.x;
    if (t < 2 * ni * N + 2 * ni * ni) {   // the y faces, then the z faces (x interior)
      int i, j, k;
      boundary_yz(t, N, i, j, k);
      int jy[2], kz[2];
      double wy[2], wz[2];
      const int ny = wall_weights(j, N, jy, wy), nz = wall_weights(k, N, kz, wz);
      double s = 0.0;
      for (int b = 0; b < nz; ++b) {
        double sb = 0.0;
        for (int a = 0; a < ny; ++a) sb += wy[a] * F.th[node32(i, jy[a], kz[b], N)];
        s += wz[b] * sb;
      }
      const int c = node32(i, j, k, N);
      m[1] = absfin(s - F.th[c]);
      F.th[c] = s;
      if (P.krylov_fp32) F.ths[c] = (float)s;
    }
  }
  if (const double* tot = grid_total<MaxD, 2>(m, F.rb, vbx, nblocks)) {
    if (threadIdx.x == 0) {
      F.rec->div_max = tot[0];
      F.rec->res = fmax(F.rec->res, tot[1]);
      if (!P.inner_pass) F.rec->res_theta = fmax(F.rec->res_theta, tot[1]);
    }
  }
}

__global__ void __launch_bounds__(kThreads) k_div_walls(DevParams P, Fields F, int nxt, int nbi,
                                                        int nblocks) {
  pdl_wait_and_release();
  k_div_walls_body(P, F, nxt, nbi, nblocks, blockIdx.x);
}

// p <- p - lambda div V at interior nodes when max|div V| > tol_div (Sec. 2.2).
__device__ __forceinline__ void k_pressure_correct_body(const DevParams& P, const Fields& F,
                                                        unsigned vbx) {
  const int N = P.N, ni = N - 2;
  const int cnt = ni * ni * ni;
  const int t = vbx * blockDim.x + threadIdx.x;
  if (t >= cnt || *F.halt) return;
  if (!(F.rec->div_max > P.tol_div)) return;
  const int q = t / ni, i = 1 + (t - q * ni), j = 1 + q % ni, k = 1 + q / ni;
  const int c = node32(i, j, k, N);
  double lam = P.lambda;
  if (P.lambda_mode) {   // viscosity-scaled relaxation: eta of level n (float in FP32 sweeps)
    const double eta =
        P.sweep_fp32 ? (double)reinterpret_cast<const float*>(F.eta)[c] : F.eta[c];
    lam = fmin(P.lambda * eta, P.lambda_cap);
  }
  const double p = F.p[c] - lam * F.div[c];
  F.p[c] = p;
  if (P.krylov_fp32) F.ps[c] = (float)p;
}

__global__ void __launch_bounds__(kThreads) k_pressure_correct(DevParams P, Fields F) {
  pdl_wait_and_release();
  k_pressure_correct_body(P, F, blockIdx.x);
}

// Step record: Krylov outcomes and the overall status; appended to the ring. A failed step (or,
// when asked, a steady one) halts the rest of the enqueued sequence.
__device__ __forceinline__ void k_finish_record_body(const DevParams& P, const Fields& F,
                                                     unsigned vbx) {
  if (threadIdx.x != 0 || vbx != 0) return;
  if (*F.halt) return;
  StepRecord* r = F.rec;
  int st = HOSC_OK;
  double lres = 0.0;
  for (int s = 0; s < 4; ++s) {
    r->iters[s] = F.ks[s].iters;
    r->lin_status[s] = F.ks[s].status;
    const int q_st = system_status(F.ks[s], P.merged);
    if (q_st != HOSC_OK && st != HOSC_ECUDA) st = q_st;
    const double q = F.ks[s].r0norm > 0.0 ? F.ks[s].rnorm / F.ks[s].r0norm : 0.0;
    lres = fmax(lres, isfinite(q) ? q : INFINITY);
  }
  r->lin_res = lres;
  if (!isfinite(r->res) || !isfinite(r->div_max) || !isfinite(lres)) st = HOSC_EDIVERGED;
  r->status = st;
  const unsigned pos = *F.ring_pos;
  F.ring[pos % kRing] = *r;
  *F.ring_pos = pos + 1;
  if (st != HOSC_OK) *F.halt = 1;
  else if (*F.steady_stop && r->res < P.steady_res && r->div_max < P.div_steady) *F.halt = 2;
}

__global__ void k_finish_record(DevParams P, Fields F) {
  k_finish_record_body(P, F, blockIdx.x);
}

// Zero normal pressure gradient on every wall: p_b = (4 p_1 - p_2)/3 along each wall normal the
// node lies on (products on edges and corners); applied after a correction. With record, the last
// of the nblocks blocks (a ticket: every block has read the halt flag by then) ends the step.
__device__ __forceinline__ void k_pressure_walls_body(const DevParams& P, const Fields& F,
                                                      int record, int nblocks, unsigned vbx) {
  if (*F.halt) return;
  const int N = P.N, ni = N - 2;
  const int t = vbx * blockDim.x + threadIdx.x;
  if (t < N * N * N - ni * ni * ni && F.rec->div_max > P.tol_div) {
    int i, j, k;
    boundary_node(t, N, i, j, k);
    int ix[2], jy[2], kz[2];
    double wx[2], wy[2], wz[2];
    const int nx = wall_weights(i, N, ix, wx), ny = wall_weights(j, N, jy, wy),
              nz = wall_weights(k, N, kz, wz);
    double s = 0.0;
    for (int c3 = 0; c3 < nz; ++c3) {
      double s2 = 0.0;
      for (int b = 0; b < ny; ++b) {
        double s1 = 0.0;
        for (int a = 0; a < nx; ++a) s1 += wx[a] * F.p[node32(ix[a], jy[b], kz[c3], N)];
        s2 += wy[b] * s1;
      }
      s += wz[c3] * s2;
    }
    const int c = node32(i, j, k, N);
    F.p[c] = s;
    if (P.krylov_fp32) F.ps[c] = (float)s;
  }
  if (record) {
    __syncthreads();
    if (last_ticket(F.rb.counter, (unsigned)nblocks)) k_finish_record_body(P, F, 0);
  }
}

__global__ void __launch_bounds__(kThreads) k_pressure_walls(DevParams P, Fields F, int record,
                                                             int nblocks) {
  pdl_wait_and_release();
  k_pressure_walls_body(P, F, record, nblocks, blockIdx.x);
}

__global__ void k_arm(int* halt, unsigned int* ring_pos, int* steady_stop, int stop) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    *halt = 0;
    *ring_pos = 0u;
    *steady_stop = stop;
  }
}

}  // namespace

namespace {
// Float copies of the state for the FP32 sweeps (one rounding per node and step).
__device__ __forceinline__ void k_shadow_body(int n3, const double* HOSC_RESTRICT u,
                                              const double* HOSC_RESTRICT v,
                                              const double* HOSC_RESTRICT w,
                                              const double* HOSC_RESTRICT th,
                                              const double* HOSC_RESTRICT p, float* HOSC_RESTRICT us,
                                              float* HOSC_RESTRICT vs, float* HOSC_RESTRICT ws,
                                              float* HOSC_RESTRICT ths, float* HOSC_RESTRICT ps,
                                              const int* HOSC_RESTRICT halt, unsigned vbx) {
  const int t = vbx * blockDim.x + threadIdx.x;
  if (t >= n3 || *halt) return;
  us[t] = (float)u[t];
  vs[t] = (float)v[t];
  ws[t] = (float)w[t];
  if (ths) {
    ths[t] = (float)th[t];
    ps[t] = (float)p[t];
  }
}

__global__ void __launch_bounds__(kThreads) k_shadow(int n3, const double* HOSC_RESTRICT u,
                                                     const double* HOSC_RESTRICT v,
                                                     const double* HOSC_RESTRICT w,
                                                     const double* HOSC_RESTRICT th,
                                                     const double* HOSC_RESTRICT p,
                                                     float* HOSC_RESTRICT us, float* HOSC_RESTRICT vs,
                                                     float* HOSC_RESTRICT ws,
                                                     float* HOSC_RESTRICT ths,
                                                     float* HOSC_RESTRICT ps,
                                                     const int* HOSC_RESTRICT halt) {
  k_shadow_body(n3, u, v, w, th, p, us, vs, ws, ths, ps, halt, blockIdx.x);
}
}  // namespace

}  // namespace hosc
