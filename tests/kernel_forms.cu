// Launches that no public call leads to on this GPU, for tests; linked with the library's objects in
// place of hosc_solve.cu: no shape fits one launch, so that the allocation-free solve runs kernel by
// kernel, and the flat x/r kernel on vectors and scalars of the test's choice.

#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <vector>

#include "hosc.h"
#include "hosc_internal.h"

namespace hosc {
bool solve_shape_planar(int, int, int*, int*) { return false; }
bool solve_shape_mixed(int, int*, int*) { return false; }
void launch_solve(const DevParams&, const Fields&, cudaStream_t) {}
}  // namespace hosc

using namespace hosc;

// One flat x/r launch with the given scalars on an N^3 grid whose vectors are 1 inside and 0 on the
// walls; returns the number of wall values of x and r that are not 0 afterwards, -1 on an error.
extern "C" int flat_xr_walls(int N, double alpha, double omega, int first) {
  const size_t n3 = (size_t)N * N * N;
  std::vector<float4> in(n3), x(n3), r(n3);
  auto wall = [&](size_t c) {
    const int i = (int)(c % N), j = (int)(c / N % N), k = (int)(c / N / N);
    return i == 0 || j == 0 || k == 0 || i == N - 1 || j == N - 1 || k == N - 1;
  };
  for (size_t c = 0; c < n3; ++c) {
    const float v = wall(c) ? 0.f : 1.f;
    in[c] = make_float4(v, v, v, v);
  }
  char* base = nullptr;
  const size_t vec = n3 * sizeof(float4), rows = (size_t)red_rows((long)n3) * kRedSlots * sizeof(double);
  if (cudaMalloc(&base, 8 * vec + 2 * rows + 16384) != cudaSuccess) return -1;
  Fields F;
  memset(&F, 0, sizeof(F));
  float4** to[7] = {&F.kr0, &F.kr, &F.kx, &F.kv[1], &F.kp[1], &F.kt, &F.kv[0]};
  for (int q = 0; q < 7; ++q) {
    *to[q] = (float4*)(base + q * vec);
    cudaMemcpy(*to[q], in.data(), vec, cudaMemcpyHostToDevice);
  }
  char* p = base + 8 * vec;
  F.rb.red = (double*)p;
  F.rb.red2 = (double*)(p + rows);
  p += 2 * rows;
  cudaMemset(p, 0, 16384);
  F.rb.counter = (unsigned*)p;
  F.ks = (KrylovScalars*)(p + 8192);
  F.halt = (int*)(p + 12288);
  F.alg_bytes = (double*)(p + 12544);
  KrylovScalars ks[4];
  memset(ks, 0, sizeof(ks));
  for (auto& k : ks) k.alpha = alpha, k.omega = omega, k.rho = k.r0norm = 1.0;
  cudaMemcpy(F.ks, ks, sizeof(ks), cudaMemcpyHostToDevice);
  DevParams P;
  memset(&P, 0, sizeof(P));
  P.N = N;
  P.krylov_fp32 = P.lean = P.xr_flat = 1;
  P.max_lin_iter = 10;
  launch_bicg_xr(P, F, 0, first != 0, 0);
  int bad = cudaGetLastError() == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess ? 0 : -1;
  if (bad == 0) {
    cudaMemcpy(x.data(), F.kx, vec, cudaMemcpyDeviceToHost);
    cudaMemcpy(r.data(), F.kr, vec, cudaMemcpyDeviceToHost);
    for (size_t c = 0; c < n3; ++c)
      for (const float4& v : {x[c], r[c]})
        if (wall(c) && !(v.x == 0.f && v.y == 0.f && v.z == 0.f && v.w == 0.f)) ++bad;
  }
  cudaFree(base);
  return bad;
}
