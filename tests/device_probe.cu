// The library's own device functions on arrays, for the tests (compiled by test_gpu_device.py):
// device pointers in, device pointers out, one synchronised launch per call.
#include "dd_cell.cu"

namespace {

__global__ void k_unary(int kind, const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  switch (kind) {
    case 0: y[i] = dd_ex2(v); break;
    case 1: y[i] = dd_lg2(v); break;
    case 2: y[i] = dd_rcp(v); break;
    case 3: y[i] = (double)narrow(v); break;
    case 4: y[i] = (double)narrow_any(v); break;
    case 5: y[i] = widen_pos((float)v); break;
  }
}

__global__ void k_binary(int kind, const double* a, const double* b, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = kind == 0 ? dd_log_quotient(a[i], b[i]) : dd_div(a[i], b[i]);
}

__global__ void k_newton(const double* lr, const double* c0, const double* uw, double s, int maxit, double* u, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) u[i] = newton_f64(lr[i], c0[i], uw[i], s, 1.0 / s, 1.0 / (1.0 + s), maxit);
}

// One log-sum-exp of the double cells per group of P lanes: sources f (M), targets j < n.
__global__ void k_lse(const double* f, int M, double q2, const double* prev, int have, int P, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = min(i / P, n - 1);
  const double v = lse_lanes_f64(f, 1, M, j, q2, have ? prev[j] : 0.0, have != 0, i % P, P);
  if (i % P == 0 && i / P < n) out[j] = v;
}

// Block sums of K values of 512 threads, value k of thread t at x[k * 512 + t].
template <int K>
__global__ void __launch_bounds__(512) k_sums(const double* x, double* out) {
  __shared__ double red[33 * K];
  double v[K];
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = x[k * 512 + threadIdx.x];
  cell_sum<float, K>(v, red);
  // every thread holds the result; the last one stores it
  if (threadIdx.x == blockDim.x - 1)
#pragma unroll
    for (int k = 0; k < K; ++k) out[k] = v[k];
}

int done() { return cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess; }

}  // namespace

extern "C" {
int probe_unary(int kind, const double* x, double* y, int n) {
  k_unary<<<(n + 255) / 256, 256>>>(kind, x, y, n);
  return done();
}
int probe_binary(int kind, const double* a, const double* b, double* y, int n) {
  k_binary<<<(n + 255) / 256, 256>>>(kind, a, b, y, n);
  return done();
}
int probe_newton(const double* lr, const double* c0, const double* uw, double s, int maxit, double* u, int n) {
  k_newton<<<(n + 127) / 128, 128>>>(lr, c0, uw, s, maxit, u, n);
  return done();
}
int probe_lse(const double* f, int M, double q2, const double* prev, int have, int P, double* out, int n) {
  k_lse<<<(n * P + 127) / 128, 128>>>(f, M, q2, prev, have, P, out, n);
  return done();
}
int probe_sums(int K, const double* x, double* out) {
  if (K == 2) k_sums<2><<<1, 512>>>(x, out);
  else if (K == 4) k_sums<4><<<1, 512>>>(x, out);
  else if (K == 12) k_sums<12><<<1, 512>>>(x, out);
  else return 1;
  return done();
}
}
