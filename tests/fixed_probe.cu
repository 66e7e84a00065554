// Test probe: fx_apply of csrc/fixed.cuh on lines and operators from the host, and
// the widening of floats.
#include <cuda_runtime.h>

#include "../paper_1406_7416_gb300/csrc/fixed.cuh"

namespace {

using namespace adg;

// out[line][n] = M x[line] for an n x n operator
template <int n>
__global__ void products(const double* M, const double* x, long long lines, double* out) {
  __shared__ FxOp m[n * n];
  __shared__ int g;
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int a = 0; a < n; ++a) {
      double r = 0.0;
      for (int j = 0; j < n; ++j) r += fabs(M[a * n + j]);
      s = r > s ? r : s;
    }
    g = fx_scale(s);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n * n; i += blockDim.x) m[i] = fx_op(M[i], g);
  __syncthreads();
  for (long long l = blockIdx.x * (long long)blockDim.x + threadIdx.x; l < lines;
       l += (long long)gridDim.x * blockDim.x) {
    double v[n];
#pragma unroll
    for (int j = 0; j < n; ++j) v[j] = x[l * n + j];
    fx_apply<n, n, false>(v, m, g, FxRows{M, 1.0}, [&](int a, double y) { out[l * n + a] = y; });
  }
}

// out[line][n] = (row sums of M) x[line][0], the predictor's first time solve
template <int n>
__global__ void sums(const double* M, const double* x, long long lines, double* out) {
  __shared__ FxOp m[n];
  __shared__ int g;
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int a = 0; a < n; ++a) {
      double r = 0.0;
      for (int j = 0; j < n; ++j) r += fabs(M[a * n + j]);
      s = r > s ? r : s;
    }
    g = fx_scale(s);
  }
  __syncthreads();
  for (int a = threadIdx.x; a < n; a += blockDim.x) {
    double r = 0.0;
    for (int j = 0; j < n; ++j) r += M[a * n + j];
    m[a] = fx_op(r, g);
  }
  __syncthreads();
  for (long long l = blockIdx.x * (long long)blockDim.x + threadIdx.x; l < lines;
       l += (long long)gridDim.x * blockDim.x) {
    const double v = x[l * n];
    fx_apply<1, n, true>(&v, m, g, FxSums<n>{M}, [&](int a, double y) { out[l * n + a] = y; });
  }
}

template <int n>
int run(int want, bool sum, const double* M, const double* x, long long lines, double* out) {
  if (want != n) {
    if constexpr (n < 10) return run<n + 1>(want, sum, M, x, lines, out);
    return -1;
  }
  double* d = nullptr;
  if (cudaMalloc(&d, sizeof(double) * (n * n + 2 * lines * n)) != cudaSuccess) return -2;
  double *dx = d + n * n, *dout = dx + lines * n;
  cudaMemcpy(d, M, sizeof(double) * n * n, cudaMemcpyHostToDevice);
  cudaMemcpy(dx, x, sizeof(double) * lines * n, cudaMemcpyHostToDevice);
  if (sum) sums<n><<<64, 128>>>(d, dx, lines, dout);
  else products<n><<<64, 128>>>(d, dx, lines, dout);
  const cudaError_t e = cudaMemcpy(out, dout, sizeof(double) * lines * n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : -3;
}

__global__ void widened(const float* x, int count, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) out[i] = widen_f32_any(x[i]);
}

}  // namespace

extern "C" int widen_floats(const float* x, int count, double* out) {
  double* d = nullptr;
  if (cudaMalloc(&d, (sizeof(double) + sizeof(float)) * count) != cudaSuccess) return -2;
  float* dx = reinterpret_cast<float*>(d + count);
  cudaMemcpy(dx, x, sizeof(float) * count, cudaMemcpyHostToDevice);
  widened<<<(count + 255) / 256, 256>>>(dx, count, d);
  const cudaError_t e = cudaMemcpy(out, d, sizeof(double) * count, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : -3;
}

extern "C" int fixed_products(int n, const double* M, const double* x, long long lines, double* out) {
  return run<1>(n, false, M, x, lines, out);
}

extern "C" int fixed_sums(int n, const double* M, const double* x, long long lines, double* out) {
  return run<1>(n, true, M, x, lines, out);
}
