// linear_probe.cu -- the block fixed-point sums of the float64 step and its
// reciprocal on arrays, on the host and on the device, for
// test_linear_sums.py.
#include <cuda_runtime.h>

#include "lbve_step.cuh"

namespace {

// kind 0: moments of 9 populations (8 results); 1: populations of 8
// coefficients (9 results); third: with the third-order terms
template <bool THIRD>
__host__ __device__ void apply(int kind, const double* in, double* out) {
  if (kind == 0) {
    lbve::Moments<double> m;
    m.nxxy = m.nxyy = 0.0;
    lbve::lattice_moments<THIRD>(in, m);
    const double r[8] = {m.drho, m.jx, m.jy, m.nxx, m.nyy, m.pxy, m.nxxy, m.nxyy};
    for (int i = 0; i < 8; ++i) out[i] = r[i];
  } else {
    double r[9];
    lbve::lattice_populations<THIRD>(in[0], in[1], in[2], in[3], in[4], in[5], in[6], in[7], r);
    for (int i = 0; i < 9; ++i) out[i] = r[i];
  }
}

__host__ __device__ void one(int kind, int third, const double* in, double* out, long long t) {
  const int ni = kind == 0 ? 9 : 8, no = kind == 0 ? 8 : 9;
  if (third) apply<true>(kind, in + t * ni, out + t * no);
  else apply<false>(kind, in + t * ni, out + t * no);
}

__global__ void sums_kernel(int kind, int third, const double* in, double* out, long long n) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t < n) one(kind, third, in, out, t);
}

__global__ void recip_kernel(const double* in, double* out, long long n) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t < n) out[t] = lbve::recip(in[t]);
}

int run(int what, int kind, int third, const double* in, double* out, long long n, int ni, int no) {
  double *di = nullptr, *dv = nullptr;
  cudaError_t e = cudaMalloc(&di, sizeof(double) * ni * n);
  if (e == cudaSuccess) e = cudaMalloc(&dv, sizeof(double) * no * n);
  if (e == cudaSuccess) e = cudaMemcpy(di, in, sizeof(double) * ni * n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    const unsigned grid = (unsigned)((n + 127) / 128);
    if (what == 0) sums_kernel<<<grid, 128>>>(kind, third, di, dv, n);
    else recip_kernel<<<grid, 128>>>(di, dv, n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(out, dv, sizeof(double) * no * n, cudaMemcpyDeviceToHost);
  cudaFree(di);
  cudaFree(dv);
  return (int)e;
}

}  // namespace

extern "C" void probe_sums_host(int kind, int third, const double* in, double* out, long long n) {
  for (long long t = 0; t < n; ++t) one(kind, third, in, out, t);
}
extern "C" int probe_sums_device(int kind, int third, const double* in, double* out, long long n) {
  return run(0, kind, third, in, out, n, kind == 0 ? 9 : 8, kind == 0 ? 8 : 9);
}
extern "C" int probe_recip_device(const double* in, double* out, long long n) {
  return run(1, 0, 0, in, out, n, 1, 1);
}
