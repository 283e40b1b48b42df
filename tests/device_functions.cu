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
