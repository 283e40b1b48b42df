// Kernels over the library's device functions, for tests/test_gpu_device_functions.py.
#include "../paper_2008_01990_gb300/csrc/tdc_far.cuh"

using namespace tdc;

// a warp per position x[i]: out[4 i ..] = value, slope, Sf, rd3 of the record
__global__ void k_far(int n, const double* rec, const double* x, double* out) {
  const int i = blockIdx.x;
  if (i >= n) return;
  double p;
  float slope, sf, rd3;
  far_value(rec, x[i], p, slope, sf, rd3);
  if (threadIdx.x == 0) {
    out[4 * i] = p;
    out[4 * i + 1] = slope;
    out[4 * i + 2] = sf;
    out[4 * i + 3] = rd3;
  }
}

extern "C" int run_far(int n, const double* rec, const double* x, double* out) {
  k_far<<<n, 32>>>(n, rec, x, out);
  return cudaDeviceSynchronize();
}

// out[6 i ..] = 1 / sqrt(a) cubic and Newton, then reflector(a, b): tau, beta, sc, and 1 / a
__global__ void k_scalars(int n, const double* a, const double* b, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double* o = out + 6 * i;
  o[0] = rsqrt_cubic(fabs(a[i]));
  o[1] = rsqrt_nr(fabs(a[i]));
  reflector(a[i], b[i], o[2], o[3], o[4]);
  o[5] = rcp_nr(a[i]);
}
// out[3 i ..] = w, c, s of the rotation that takes (a, b)
__global__ void k_rotation(int n, const double* a, const double* b, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) bd_rotation(a[i], b[i], out[3 * i], out[3 * i + 1], out[3 * i + 2]);
}
// a warp per 3 x 32 values: out[(6 i + q) 32 + lane] = warp_sum2 of rows 0, 1, warp_sum3 of 0, 1, 2, warp_sum of 0
__global__ void k_sums(int n, const double* v, double* out) {
  const int i = blockIdx.x, lane = threadIdx.x;
  if (i >= n) return;
  const double x = v[96 * i + lane], y = v[96 * i + 32 + lane], z = v[96 * i + 64 + lane];
  double a = x, b = y, c = x, d = y, e = z;
  warp_sum2(a, b);
  warp_sum3(c, d, e);
  const double r[6] = {a, b, c, d, e, warp_sum(x)};
  for (int q = 0; q < 6; ++q) out[(6 * i + q) * 32 + lane] = r[q];
}

extern "C" int run_scalars(int n, const double* a, const double* b, double* out) {
  k_scalars<<<(n + 127) / 128, 128>>>(n, a, b, out);
  return cudaDeviceSynchronize();
}
extern "C" int run_rotation(int n, const double* a, const double* b, double* out) {
  k_rotation<<<(n + 127) / 128, 128>>>(n, a, b, out);
  return cudaDeviceSynchronize();
}
extern "C" int run_sums(int n, const double* v, double* out) {
  k_sums<<<n, 32>>>(n, v, out);
  return cudaDeviceSynchronize();
}
