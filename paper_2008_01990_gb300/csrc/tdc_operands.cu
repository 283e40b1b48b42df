// tdc_operands.cu -- products C = A B with a structured B given by generators (the
// further structured operands of Sections 1, 3.1 and 5: matrices of O(n) parameters):
// Toeplitz B(k, j) = t[k - j + n - 1], Hankel t[k + j], Vandermonde x_k^j, and the DFT
// matrix exp(-2 pi i k j / n) as its real and imaginary parts.  B is generated inside the
// product kernels -- the FP64 tiles of k_gemm_dense_seg and the digit images of k_split_b
// (struct_entry) -- so only the generators travel to the GPU (the point made in
// Section 5).  For the split product, column j of B enters scaled by 2^-eb_j with 2^eb_j
// above its largest |entry|: for Toeplitz / Hankel the maximum of |t| over the column's
// window of n consecutive generators, from running maxima outwards from the middle
// generator; for Vandermonde max|x|^j (with a
// margin for the rounding of the powers); for the DFT 0 (|entries| <= 1).  A enters
// scaled by 2^-eA from its largest row norm, and the product's column is scaled back by
// 2^eb_j (cexp) and 2^eA (oexp).
#include "tdc_common.cuh"

namespace tdc {

// Column j's window is t[s .. s + n - 1] with s = n - 1 - j (Toeplitz) or j (Hankel): every
// window holds the middle generator t[n - 1], so its maximum is the larger of a suffix
// maximum of |t[0 .. n-1]| at s and a prefix maximum of |t[n-1 ..]| at s + n - 1.  One block:
// each thread scans a contiguous run outwards from the middle, the runs' maxima are scanned
// over the block, and win[i] becomes the running maximum from the middle to i.  Two passes
// over the generators whatever n is (doubling windows took log2 n: n = 4096, 43 -> 20 us).
__global__ void __launch_bounds__(1024) k_tp_windows(int64_t n, const double* t, int kind, double* win,
                                                     int32_t* eb) {
  __shared__ double s_w[2][32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int side = tid >> 9, q = tid & 511;  // threads 0-511: towards 0; 512-1023: towards 2n - 2
  const int64_t per = (n + 511) / 512, a = min(n, q * per), b = min(n, a + per);
  const int64_t mid = n - 1, dir = side ? 1 : -1;
  double mx = 0.0;
  for (int64_t i = a; i < b; ++i) {
    mx = fmax(mx, fabs(t[mid + dir * i]));
    win[side * n + i] = mx;
  }
  double inc = mx;  // inclusive scan of the runs' maxima over the side's 16 warps
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc = fmax(inc, v);
  }
  if (lane == 31) s_w[side][warp & 15] = inc;
  __syncthreads();
  double before = __shfl_up_sync(0xffffffffu, inc, 1);
  if (lane == 0) before = 0.0;
  for (int w = 0; w < (warp & 15); ++w) before = fmax(before, s_w[side][w]);
  for (int64_t i = a; i < b; ++i) win[side * n + i] = fmax(win[side * n + i], before);
  __syncthreads();
  for (int64_t j = tid; j < n; j += blockDim.x) {
    const int64_t s = kind == 1 ? n - 1 - j : j;  // the window reaches mid - s below the middle, s above it
    eb[j] = exp_above(fmax(win[mid - s], win[n + s]));
  }
}

// Vandermonde: largest |x| (bits of a non-negative double in *mx, zero beforehand).
__global__ void __launch_bounds__(256) k_vd_max(int64_t n, const double* x, unsigned long long* mx) {
  double b = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    b = fmax(b, fabs(x[i]));
  for (int off = 16; off > 0; off >>= 1) b = fmax(b, __shfl_xor_sync(0xffffffffu, b, off));
  if ((threadIdx.x & 31) == 0) atomicMax(mx, (unsigned long long)__double_as_longlong(b));
}

// eb_j from max|x|^j, raised by 2^-40 relative for the rounding of the computed powers
__global__ void __launch_bounds__(256) k_vd_exps(int64_t n, const unsigned long long* mx, int32_t* eb) {
  const double m = __longlong_as_double((long long)*mx);
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
    eb[j] = exp_above(pow(m, (double)j) * (1.0 + 0x1p-40));
}

__global__ void __launch_bounds__(256) k_zero_i32(int64_t n, int32_t* a) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
    a[j] = 0;
}

// cos(2 pi m / n) and -sin(2 pi m / n), m < n: the real and imaginary parts of the DFT
// matrix's entries exp(-2 pi i k j / n) at m = (k j) mod n.
__global__ void __launch_bounds__(256) k_dft_tables(int64_t n, double* cosv, double* msinv) {
  for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < n; m += (int64_t)gridDim.x * blockDim.x) {
    double sv, cv;
    sincospi(2.0 * ((double)m / (double)n), &sv, &cv);
    cosv[m] = cv;
    msinv[m] = -sv;
  }
}

// Largest squared row norm of A (m x n, column-major, lda) as the bits of a non-negative
// double (ordered like the values) in *maxsq (zero beforehand).  A block takes R rows: thread
// (r, g) sums the columns g, g + 1024 / R, ... of row r, then the row's sums are added in
// order.  Bound by the FP64 pipe, one multiply-add an entry at 2 a clock and SM (m = n = 8192:
// 133 us, 4.0 TB/s; one thread a whole row left 32 blocks reading with one load in flight a
// thread: 3343 us.  m = n = 4096: 1669 -> 39 us); R falls with m so that short matrices still
// fill the chip, down to the 64-byte runs of R = 8.
template <int R>
__global__ void __launch_bounds__(1024) k_row_max(int64_t m, int64_t n, const double* A, int64_t lda,
                                                  unsigned long long* maxsq) {
  constexpr int G = 1024 / R;
  __shared__ double part[G][R];
  const int r = threadIdx.x % R, g = threadIdx.x / R;
  const int64_t i = (int64_t)blockIdx.x * R + r;
  double s = 0.0;
  if (i < m) {
#pragma unroll 8
    for (int64_t k = g; k < n; k += G) {
      const double x = A[i + k * lda];
      s = fma(x, x, s);
    }
  }
  part[g][r] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    double best = 0.0;
    if (threadIdx.x < R) {
      double t = 0.0;
#pragma unroll 8
      for (int q = 0; q < G; ++q) t += part[q][threadIdx.x];
      best = fmax(best, t);
    }
    for (int off = 16; off > 0; off >>= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, off));
    if (threadIdx.x == 0) atomicMax(maxsq, (unsigned long long)__double_as_longlong(best));
  }
}

cudaError_t launch_row_max(int64_t m, int64_t n, const double* A, int64_t lda, unsigned long long* maxsq,
                           cudaStream_t s) {
  const cudaError_t e = cudaMemsetAsync(maxsq, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess || m <= 0) return e;
  if (m >= 32 * 152) k_row_max<32><<<(unsigned)((m + 31) / 32), 1024, 0, s>>>(m, n, A, lda, maxsq);
  else if (m >= 16 * 152) k_row_max<16><<<(unsigned)((m + 15) / 16), 1024, 0, s>>>(m, n, A, lda, maxsq);
  else k_row_max<8><<<(unsigned)((m + 7) / 8), 1024, 0, s>>>(m, n, A, lda, maxsq);
  return cudaGetLastError();
}

// eA with (largest row norm of A) 2^-eA < 1, and oexp[j] = eA: the product's columns are
// scaled back by 2^cexp[j] (B's column scale) and then by 2^oexp[j] (A's scale).
__global__ void __launch_bounds__(256) k_tp_exps(int64_t n, const unsigned long long* maxsq, int32_t* oexp,
                                                int32_t* eA) {
  const int e = exp_above(sqrt(__longlong_as_double((long long)*maxsq)));
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
    oexp[j] = e;
  if (blockIdx.x == 0 && threadIdx.x == 0) *eA = e;
}

cudaError_t launch_operand_prep(int64_t m, int64_t n, const double* A, int64_t lda, const double* t, int kind,
                                double* winmax, int32_t* cexp, int32_t* oexp, int32_t* eA,
                                unsigned long long* maxsq, cudaStream_t s) {
  const unsigned g = (unsigned)std::min<int64_t>(1024, (n + 255) / 256);
  cudaError_t e = cudaSuccess;
  if (kind == 1 || kind == 2) {
    k_tp_windows<<<1, 1024, 0, s>>>(n, t, kind, winmax, cexp);
  } else if (kind == 3) {
    e = cudaMemsetAsync(maxsq, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    k_vd_max<<<g, 256, 0, s>>>(n, t, maxsq);
    k_vd_exps<<<g, 256, 0, s>>>(n, maxsq, cexp);
  } else {
    k_zero_i32<<<g, 256, 0, s>>>(n, cexp);
  }
  e = launch_row_max(m, n, A, lda, maxsq, s);
  if (e != cudaSuccess) return e;
  k_tp_exps<<<(unsigned)std::min<int64_t>(1024, (n + 255) / 256), 256, 0, s>>>(n, maxsq, oexp, eA);
  return cudaGetLastError();
}

cudaError_t launch_dft_tables(int64_t n, double* cosv, double* msinv, cudaStream_t s) {
  k_dft_tables<<<(unsigned)std::min<int64_t>(1024, (n + 255) / 256), 256, 0, s>>>(n, cosv, msinv);
  return cudaGetLastError();
}

}  // namespace tdc
