// Entry points of the tests around the operator kernels' parts: the sum of four FP32 values in FP64, and the
// kernels whose blocks carry two of the reduction's blocks. Compiled with hz_krylov.cu itself.
#include "hz_krylov.cu"

#include <vector>

namespace hz {
namespace {

__global__ void nb_sum_kernel(const float2* __restrict__ v, double2* __restrict__ sum, double2* __restrict__ exact,
                              int* __restrict__ odd, int count) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= count) return;
  Star<float2> s;
  s.w = v[4 * t];
  s.e = v[4 * t + 1];
  s.s = v[4 * t + 2];
  s.n = v[4 * t + 3];
  unsigned o;
  exact[t] = nb_sum(s.w, s.e, s.s, s.n, o);
  odd[t] = o != 0;
  sum[t] = nb_of<0>(s);
}

// A field and vectors of mixed magnitudes from a counter.
__device__ double mixed(unsigned long long c) {
  const double2 u = shadow_value(0x1234567ull, (long long)c);
  return ldexp(u.x, (int)(24.0 * u.y));
}
__global__ void fill_kernel(float2* y, double2* w, double* d, double* kh, int N) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= N) return;
  y[t] = make_float2((float)mixed(4ull * t), (float)mixed(4ull * t + 1));
  w[t] = make_double2(mixed(4ull * t + 2), mixed(4ull * t + 3));
  kh[t] = 0.3 + 1e-4 * (t % 97);
  d[t] = fma(kh[t], kh[t], -4.0);
}

}  // namespace
}  // namespace hz

using namespace hz;

// sum: the operator's neighbour sums; exact, odd: nb_sum's value and whether it was refused.
extern "C" int probe_nb_sum(const float2* v, double2* sum, double2* exact, int* odd, int count) {
  nb_sum_kernel<<<(count + 127) / 128, 128>>>(v, sum, exact, odd, count);
  return (int)cudaDeviceSynchronize();
}

// Runs the rv (which = 0) or ts (1) operator kernel on an n-grid with a reduction of G blocks, one or (two != 0)
// two per launched block; out: the (n+1)^2 products, then the reduced values.
extern "C" int probe_apply(int n, int G, int which, int two, double2* out) {
  const int N = (n + 1) * (n + 1);
  float2* y = nullptr;
  double2 *w = nullptr, *av = nullptr;
  double *d = nullptr, *kh = nullptr, *partials = nullptr;
  KState* st = nullptr;
  cudaMalloc(&y, sizeof(float2) * N);
  cudaMalloc(&w, sizeof(double2) * N);
  cudaMalloc(&av, sizeof(double2) * N);
  cudaMalloc(&d, sizeof(double) * N);
  cudaMalloc(&kh, sizeof(double) * N);
  cudaMalloc(&partials, sizeof(double) * 4 * G);
  cudaMalloc(&st, sizeof(KState));
  if (cudaGetLastError() != cudaSuccess) return 1;
  cudaMemset(st, 0, sizeof(KState));
  cudaMemset(av, 0xff, sizeof(double2) * N);
  fill_kernel<<<(N + 127) / 128, 128>>>(y, w, d, kh, N);
  KrylovVecs k{};
  k.rhat = k.s = w;
  k.v = k.t = av;
  k.kh = kh;
  k.d = d;
  k.n = n;
  k.N = N;
  k.st = st;
  k.partials = partials;
  k.G = G;
  k.batch = 1;
  const dim3 grid(two ? (G + 1) / 2 : G);
  if (which == 0 && two) k_apply_rv_kernel<float2, 2, 0><<<grid, KB>>>(k, y);
  if (which == 0 && !two) k_apply_rv_kernel<float2, 1, 0><<<grid, KB>>>(k, y);
  if (which == 1 && two) k_apply_ts_kernel<float2, 2, 0><<<grid, KB>>>(k, y);
  if (which == 1 && !two) k_apply_ts_kernel<float2, 1, 0><<<grid, KB>>>(k, y);
  KState hs;
  int e = (int)cudaDeviceSynchronize();
  if (!e) e = (int)cudaMemcpy(&hs, st, sizeof(KState), cudaMemcpyDeviceToHost);
  if (!e) e = (int)cudaMemcpy(out, av, sizeof(double2) * N, cudaMemcpyDeviceToHost);
  out[N] = which == 0 ? hs.rv : hs.ts;
  out[N + 1] = make_double2(which == 0 ? 0.0 : hs.tt, (double)hs.ticket[which == 0 ? KT_RV : KT_TS]);
  for (void* p : {(void*)y, (void*)w, (void*)av, (void*)d, (void*)kh, (void*)partials, (void*)st}) cudaFree(p);
  return e;
}
