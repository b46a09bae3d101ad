// Evaluates the FP64 reciprocals, roots and the Jacobi angle of
// csrc/emu_math.cuh beside the plain expressions.
//
// harness host|device IN OUT
// IN:  int64 n, double x[n], int64 k, double p[3 k] (app, aqq, apq)
// OUT: double [6][n] (1/x, 1/sqrt, sqrt of emu_math.cuh, then plain), double t[k]
#include <cstdio>
#include <cstring>
#include <vector>

#include "emu_math.cuh"

__host__ __device__ static void eval(const double* x, long long n, long long i, double* o) {
  const double v = x[i];
  o[i] = emu::inv_n(v);
  o[n + i] = emu::rsqrt_n(v);
  o[2 * n + i] = emu::sqrt_n(v);
  o[3 * n + i] = 1.0 / v;
  o[4 * n + i] = 1.0 / sqrt(v);
  o[5 * n + i] = sqrt(v);
}

__global__ void k_eval(const double* x, long long n, double* o, const double* p, long long k, double* t) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) eval(x, n, i, o);
  if (i < k) t[i] = emu::jacobi_tan(p[3 * i], p[3 * i + 1], p[3 * i + 2]);
}

int main(int argc, char** argv) {
  if (argc != 4) return 2;
  FILE* f = fopen(argv[2], "rb");
  long long n = 0, k = 0;
  if (!f || fread(&n, 8, 1, f) != 1) return 3;
  std::vector<double> x(n);
  if (fread(x.data(), 8, n, f) != (size_t)n || fread(&k, 8, 1, f) != 1) return 4;
  std::vector<double> p(3 * k), o(6 * n), t(k);
  if (fread(p.data(), 8, 3 * k, f) != (size_t)(3 * k)) return 5;
  fclose(f);
  if (!strcmp(argv[1], "host")) {
    for (long long i = 0; i < n; ++i) eval(x.data(), n, i, o.data());
    for (long long i = 0; i < k; ++i) t[i] = emu::jacobi_tan(p[3 * i], p[3 * i + 1], p[3 * i + 2]);
  } else {
    double *dx, *d_o, *dp, *dt;
    if (cudaMalloc(&dx, 8 * n) || cudaMalloc(&d_o, 48 * n) || cudaMalloc(&dp, 24 * k) || cudaMalloc(&dt, 8 * k)) return 6;
    cudaMemcpy(dx, x.data(), 8 * n, cudaMemcpyHostToDevice);
    cudaMemcpy(dp, p.data(), 24 * k, cudaMemcpyHostToDevice);
    k_eval<<<(unsigned)(((n > k ? n : k) + 255) / 256), 256>>>(dx, n, d_o, dp, k, dt);
    if (cudaMemcpy(o.data(), d_o, 48 * n, cudaMemcpyDeviceToHost) || cudaMemcpy(t.data(), dt, 8 * k, cudaMemcpyDeviceToHost))
      return 7;
  }
  f = fopen(argv[3], "wb");
  fwrite(o.data(), 8, o.size(), f);
  fwrite(t.data(), 8, t.size(), f);
  fclose(f);
  return 0;
}
