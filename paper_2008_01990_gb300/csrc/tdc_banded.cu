// tdc_banded.cu -- divide and conquer for symmetric band matrices (the band case Section 5
// points to), built from the merge's rank-one machinery.
//
// Tearing.  A node [lo, hi) of bandwidth b splits at m; its coupling block has rows
// r_k = m - b + k (k < b) with B_k(c) = A(m + c, r_k) (zero for c > k: outside the band).
// With s_k = sqrt(||B_k||), x_k = s_k e_{r_k}, y_k = B_k / s_k:
//   A = diag(A11 - sum_k x_k x_k^T, A22 - sum_k y_k y_k^T) + sum_k (x_k; y_k)(x_k; y_k)^T,
// i.e. A(r_k, r_k) -= ||B_k|| and the leading b x b corner of A22 -= sum_k B_k^T B_k / ||B_k||
// (b = 1 is Cuppen's tearing).  Rows with B_k = 0 give no term.
//
// Merge.  With the children's A1 = Q1 L1 Q1^T, A2 = Q2 L2 Q2^T and Q = diag(Q1, Q2), each
// term is one rank-one modification D + z z^T with z = Q^T (x_k; y_k), taken in turn: the
// poles sorted, deflated (type 1: rho |zhat_i| <= tol; type 2: a rotation when
// |t c s| <= tol for neighbouring poles, tol = 8 eps max(|D|max, |zhat|max), the tests of
// Section 3.2), the secular equation and the Cauchy-like update of the non-deflated
// columns (tdc_rank_one's solver and the merge's product), the deflated columns copied.  All
// nodes of a tree level take each term in the same launches, a grid row or a block a node; K
// and the other counts stay on the device, where the products' segment list is built from
// them (n = 2048, b = 8: 120 steps with a host read each -> 32 without, 41.7 -> 16.5 ms).
#include <atomic>

#include "tdc_common.cuh"

namespace tdc {

namespace {
constexpr double kBdEps = 1.1102230246251565e-16;  // 2^-53
}  // namespace

__global__ void __launch_bounds__(32) k_bd_nodes(BdNode* dst, BdNodeTable T, int count) {
  for (int i = threadIdx.x; i < count; i += 32) dst[i] = T.nd[i];
}

// Tearing of every inner node, a block each (they touch disjoint entries: nodes have at
// least 4b rows): the terms (s_k, y_k) into wv[k (b + 1) + 0..b] of the node (s_k = 0: no
// term) and the corner updates of the band copy ABw (lower band storage, ld ldab).
__global__ void __launch_bounds__(256) k_bd_tear(const BdNode* nodes, double* ABw, int64_t ldab, int b, double* wv_all) {
  extern __shared__ double sb[];  // b x b: B_k(c) at sb[k * b + c], then b norms
  const BdNode nd = nodes[blockIdx.x];
  const int64_t m = nd.mid;
  double* wv = wv_all + nd.wi * b * (b + 1);
  double* nrm = sb + b * b;
  for (int t = threadIdx.x; t < b * b; t += blockDim.x) {
    const int k = t / b, c = t % b;
    const int64_t r = m - b + k;
    sb[t] = c <= k ? ABw[(b - k + c) + r * ldab] : 0.0;  // A(m + c, r), m + c - r = b - k + c
  }
  __syncthreads();
  for (int k = threadIdx.x; k < b; k += blockDim.x) {
    double s2 = 0.0;
    for (int c = 0; c < b; ++c) s2 = fma(sb[k * b + c], sb[k * b + c], s2);
    const double nk = sqrt(s2);
    nrm[k] = nk;
    const double sk = sqrt(nk);
    wv[k * (b + 1)] = nk > 0.0 ? sk : 0.0;
    for (int c = 0; c < b; ++c) wv[k * (b + 1) + 1 + c] = nk > 0.0 ? sb[k * b + c] / sk : 0.0;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < b; k += blockDim.x) ABw[(m - b + k) * ldab] -= nrm[k];
  for (int t = threadIdx.x; t < b * b; t += blockDim.x) {
    const int c1 = t / b, c2 = t % b;
    if (c1 < c2) continue;
    double acc = 0.0;
    for (int k = 0; k < b; ++k)
      if (nrm[k] > 0.0) acc = fma(sb[k * b + c1], sb[k * b + c2] / nrm[k], acc);
    ABw[(c1 - c2) + (m + c2) * ldab] -= acc;
  }
}

// Leaves, one block each.  k_bd_leaf_trd: the dense symmetric block of the torn band
// (both triangles) reduced to tridiagonal form by Householder reflectors, column by column
// (the reduction of the dense solver, unblocked: a leaf has at most 8b or 128 rows and the
// block stays in L2): for column k, x = A(k+1:L, k), alpha = x_0, sigma = ||x(1:)||,
// beta = -sign(alpha) hypot(alpha, sigma), tau = (beta - alpha) / beta,
// v = [1, x(1:) / (alpha - beta)] (stored below the subdiagonal), p = tau A22 v,
// w = p - (tau / 2)(p^T v) v, A22 -= v w^T + w v^T (sigma = 0: tau = 0, nothing applied).
// Sum over the block, in every thread: warp sums, then the first warp over them (FP64
// additions by every warp of all partials cost thousands of clocks).
__device__ __forceinline__ double bd_block_sum(double v, double* red) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    const double t = warp_sum(threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0);
    if (threadIdx.x == 0) red[0] = t;
  }
  __syncthreads();
  return red[0];
}
// Largest |v| over the block (not NaN), by the bits of the non-negative doubles.
__device__ __forceinline__ double bd_block_max(double v, double* red) {
  unsigned long long u = (unsigned long long)__double_as_longlong(fabs(v));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, u, o);
    u = w > u ? w : u;
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = __longlong_as_double((long long)u);
  __syncthreads();
  if (threadIdx.x < 32) {
    u = threadIdx.x < (blockDim.x >> 5) ? (unsigned long long)__double_as_longlong(red[threadIdx.x]) : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long w = __shfl_xor_sync(0xffffffffu, u, o);
      u = w > u ? w : u;
    }
    if (threadIdx.x == 0) red[0] = __longlong_as_double((long long)u);
  }
  __syncthreads();
  return red[0];
}

__global__ void __launch_bounds__(kBdLeafThreads) k_bd_leaf_trd(BdLeafArgs P, BdLeafTable T) {
  __shared__ double v[512], pw[512], red[32];
  __shared__ double s_tau, s_scal;
  __shared__ int s_skip;
  const int64_t lo = T.lo[blockIdx.x];
  const int L = T.L[blockIdx.x];
  if (L <= 0 || L > 512) return;
  double* A = P.Ab + lo * P.lmax;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  for (int t = tid; t < L * L; t += blockDim.x) {
    const int i = t % L, j = t / L;
    const int r = i > j ? i - j : j - i, c = i > j ? j : i;
    A[t] = r <= P.b ? P.ABw[r + (lo + c) * P.ldab] : 0.0;
  }
  __syncthreads();
  for (int k = 0; k + 2 < L; ++k) {
    const int m = L - k - 1;
    double* x = A + (k + 1) + (int64_t)k * L;
    double* A22 = A + (k + 1) + (int64_t)(k + 1) * L;
    double ss = 0.0;
    for (int i = tid; i < m; i += blockDim.x) {
      const double xi = x[i];
      v[i] = xi;
      if (i > 0) ss = fma(xi, xi, ss);
    }
    ss = bd_block_sum(ss, red);
    if (tid == 0) {
      const double alpha = v[0];
      P.d[lo + k] = A[k + (int64_t)k * L];
      if (ss == 0.0) {
        s_skip = 1;
        P.e[lo + k] = alpha;
        P.tau[lo + k] = 0.0;
      } else {
        double t, beta, sc;
        reflector(alpha, ss, t, beta, sc);
        s_skip = 0;
        s_tau = t;
        s_scal = sc;
        P.e[lo + k] = beta;
        P.tau[lo + k] = t;
      }
    }
    __syncthreads();
    if (s_skip) continue;
    const double tau = s_tau, scal = s_scal;
    for (int i = tid; i < m; i += blockDim.x) {
      const double vi = i == 0 ? 1.0 : v[i] * scal;
      v[i] = vi;
      if (i > 0) x[i] = vi;
    }
    __syncthreads();
    // p_i = tau (A22 v)_i: column i of the symmetric A22 against v, a warp per column
    for (int i = wid; i < m; i += nw) {
      const double* col = A22 + (int64_t)i * L;
      double acc = 0.0;
      for (int j = lane; j < m; j += 32) acc = fma(col[j], v[j], acc);
      acc = warp_sum(acc);
      if (lane == 0) pw[i] = tau * acc;
    }
    __syncthreads();
    double pv = 0.0;
    for (int i = tid; i < m; i += blockDim.x) pv = fma(pw[i], v[i], pv);
    pv = bd_block_sum(pv, red);
    const double h = 0.5 * tau * pv;
    for (int i = tid; i < m; i += blockDim.x) pw[i] = fma(-h, v[i], pw[i]);
    __syncthreads();
    for (int t = tid; t < m * m; t += blockDim.x) {
      const int i = t % m, j = t / m;
      // the same two products and one addition for (i, j) and (j, i): A22 stays symmetric
      A22[i + (int64_t)j * L] -= __dadd_rn(__dmul_rn(v[i], pw[j]), __dmul_rn(pw[i], v[j]));
    }
    __syncthreads();
  }
  if (tid == 0) {
    if (L == 1) {
      P.d[lo] = A[0];
    } else {
      P.d[lo + L - 2] = A[(L - 2) + (int64_t)(L - 2) * L];
      P.d[lo + L - 1] = A[(L - 1) + (int64_t)(L - 1) * L];
      P.e[lo + L - 2] = A[(L - 1) + (int64_t)(L - 2) * L];
      P.tau[lo + L - 2] = 0.0;
    }
  }
}

// k_bd_leaf_back: Q(lo:lo+L, lo:lo+L) = H_0 ... H_{L-3} Z, Z the leaf tridiagonal's
// eigenvectors (Zb, ld L): the reflectors applied last first to each column of Z, one warp a
// column with its rows in registers (R a lane), so that a leaf spreads over L warps instead
// of one block and nothing waits: bound by 2 R + 5 FP64 instructions a reflector (16 leaves of
// 128 rows: 1.79 -> 0.26 ms).
template <int R>
__global__ void __launch_bounds__(128) k_bd_leaf_back(BdLeafArgs P, BdLeafTable T) {
  const int64_t lo = T.lo[blockIdx.x];
  const int L = T.L[blockIdx.x];
  const int lane = threadIdx.x & 31, j = blockIdx.y * 4 + (threadIdx.x >> 5);
  if (L <= 0 || L > 32 * R || j >= L) return;
  const double* A = P.Ab + lo * P.lmax;
  const double* Z = P.Zb + lo * P.lmax + (int64_t)j * L;
  double q[R];
#pragma unroll
  for (int u = 0; u < R; ++u) q[u] = lane + 32 * u < L ? Z[lane + 32 * u] : 0.0;
  for (int k = L - 3; k >= 0; --k) {
    const double tau = P.tau[lo + k];
    if (tau == 0.0) continue;
    double v[R], acc = 0.0;
#pragma unroll
    for (int u = 0; u < R; ++u) {
      const int r = lane + 32 * u;
      v[u] = r > k + 1 && r < L ? A[r + (int64_t)k * L] : (r == k + 1 ? 1.0 : 0.0);
      if (32 * u + 31 > k) acc = fma(v[u], q[u], acc);
    }
    acc = -tau * warp_sum(acc);
#pragma unroll
    for (int u = 0; u < R; ++u)
      if (32 * u + 31 > k) q[u] = fma(acc, v[u], q[u]);
  }
  double* Qb = P.Q + lo + (lo + j) * P.ldq;
#pragma unroll
  for (int u = 0; u < R; ++u)
    if (lane + 32 * u < L) Qb[lane + 32 * u] = q[u];
}

// Start of a level: the poles are the children's eigenvalues, the first run the left child's.
__global__ void __launch_bounds__(256) k_bd_level_begin(BdLevel L, const double* lam) {
  const BdNode nd = L.nodes[blockIdx.y];
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nd.nn; j += (int64_t)gridDim.x * blockDim.x)
    L.Dcur[nd.lo + j] = lam[nd.lo + j];
  if (blockIdx.x == 0 && threadIdx.x == 0) L.cnt[4 * blockIdx.y + 3] = (int32_t)(nd.mid - nd.lo);
}

// z_j = s Q(ra, j) + sum_c y_c Q(rb + c, j), j < nn, for a node's term k: ra the k-th of the b
// rows above the split, rb the split's first row.
__global__ void __launch_bounds__(256) k_bd_z(BdLevel L, int k) {
  const BdNode nd = L.nodes[blockIdx.y];
  const double* w = L.wv + (nd.wi * L.b + k) * (L.b + 1);
  const double* Q = L.Q + nd.lo + nd.lo * L.ldq;
  const int64_t ra = nd.mid - L.b + k - nd.lo, rb = nd.mid - nd.lo;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nd.nn; j += (int64_t)gridDim.x * blockDim.x) {
    const double* col = Q + j * L.ldq;
    double acc = w[0] * col[ra];
    for (int c = 0; c < L.b; ++c) acc = fma(w[1 + c], col[rb + c], acc);
    L.z[nd.lo + j] = acc;
  }
}

// A double as an integer of the same order (-0 before +0).
__device__ __forceinline__ long long bd_key(double x) {
  const long long u = __double_as_longlong(x);
  return u ^ ((u >> 63) & 0x7fffffffffffffffll);
}

// Sort of a node's poles, as a rule a merge: Dcur is two ascending runs (the children's
// eigenvalues; later the roots in order, then the deflated poles in order of scan), so an
// entry's place is its place in its run plus the count of the other run's entries before it
// (ties: first run first), a binary search on integer keys.  A run that is not ascending (a
// deflating rotation may move a pole past its neighbour) or holds a NaN sets `unsorted` and
// leaves the node to the network below.  One block a node: 4 us where the network and the
// ranks of its chunks took 39.
__global__ void __launch_bounds__(1024) k_bd_merge(BdLevel L, int use_z) {
  const BdNode nd = L.nodes[blockIdx.x];
  const double* D = L.Dcur + nd.lo;
  const int64_t nn = nd.nn, r0 = L.cnt[4 * blockIdx.x + 3];
  bool bad = r0 < 0 || r0 > nn;
  for (int64_t i = threadIdx.x; i < nn; i += blockDim.x) {
    const double d = D[i];
    bad = bad || (__double2hiint(d) & 0x7ff00000) == 0x7ff00000;
    if (i > 0 && i != r0) bad = bad || bd_key(D[i - 1]) > bd_key(d);
  }
  const int any = __syncthreads_or(bad);
  if (threadIdx.x == 0) L.unsorted[blockIdx.x] = any;
  if (any) return;
  for (int64_t i = threadIdx.x; i < nn; i += blockDim.x) {
    const double d = D[i];
    const long long key = bd_key(d);
    const bool first = i < r0;
    int64_t lo = first ? r0 : 0, hi = first ? nn : r0;
    const int64_t base = lo;
    while (lo < hi) {  // entries of the other run before this one
      const int64_t m = (lo + hi) >> 1;
      const long long km = bd_key(D[m]);
      if (first ? km < key : km <= key) lo = m + 1; else hi = m;
    }
    const int64_t rk = (first ? i : i - r0) + (lo - base);
    L.Ds[nd.lo + rk] = d;
    if (use_z) L.zs[nd.lo + rk] = L.z[nd.lo + i];
    L.perm[nd.lo + rk] = (int32_t)i;
  }
}

// (a, ia) before (b, ib) in a strict total order: ascending values, NaNs last, ties by
// index -- so that the ranks below always form a permutation.
__device__ __forceinline__ bool bd_before(double a, int64_t ia, double b, int64_t ib) {
  const bool na = a != a, nb = b != b;
  if (na || nb) return (!na && nb) || (na && nb && ia < ib);
  return a < b || (a == b && ia < ib);
}

// Stable sort by rank in two kernels, of the nodes k_bd_merge left.  k_bd_chunk_sort: one
// block per chunk of ch entries
// (ch = kBdChunk, or the power of two at or above nn when that is smaller) sorts (D[i], i)
// by bd_before with a bitonic network in shared memory (entries past nn pad the chunk and
// sort last), writing the chunk's sorted keys and indices.
// k_bd_rank: entry i at sorted place p of its chunk has rank p + the count of entries before
// it in every other chunk (a binary search each); Ds[rank] = D[i], zs likewise (z may be
// NULL), perm[rank] = i.  The ranks are those of the total order, a permutation.
constexpr int kBdChunk = 2048;

__device__ __forceinline__ bool bd_before_pad(double a, int64_t ia, double b, int64_t ib, int64_t nn) {
  if (ia >= nn || ib >= nn) return ia < nn || (ib >= nn && ia < ib);
  return bd_before(a, ia, b, ib);
}

__global__ void __launch_bounds__(1024) k_bd_chunk_sort(BdLevel L, int ch) {
  __shared__ double key[kBdChunk];
  __shared__ int32_t idx[kBdChunk];
  if (!L.unsorted[blockIdx.y]) return;
  const BdNode nd = L.nodes[blockIdx.y];
  const int64_t nn = nd.nn;
  const double* D = L.Dcur + nd.lo;
  double* sk = L.sk + nd.lo;
  int32_t* si = L.si + nd.lo;
  const int64_t c0 = (int64_t)blockIdx.x * ch;
  if (c0 >= nn) return;
  for (int t = threadIdx.x; t < ch; t += blockDim.x) {
    const int64_t i = c0 + t;
    key[t] = i < nn ? D[i] : 0.0;
    idx[t] = (int32_t)(i < nn ? i : nn + t);
  }
  __syncthreads();
  for (int k = 2; k <= ch; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < ch / 2; t += blockDim.x) {
        const int lo = 2 * j * (t / j) + (t % j), hi = lo + j;
        const bool up = (lo & k) == 0;
        const bool swap = up ? bd_before_pad(key[hi], idx[hi], key[lo], idx[lo], nn)
                             : bd_before_pad(key[lo], idx[lo], key[hi], idx[hi], nn);
        if (swap) {
          const double kv = key[lo];
          key[lo] = key[hi];
          key[hi] = kv;
          const int32_t iv = idx[lo];
          idx[lo] = idx[hi];
          idx[hi] = iv;
        }
      }
      __syncthreads();
    }
  }
  for (int t = threadIdx.x; t < ch && c0 + t < nn; t += blockDim.x) {
    sk[c0 + t] = key[t];
    si[c0 + t] = idx[t];
  }
}

__global__ void __launch_bounds__(256) k_bd_rank(BdLevel L, int ch, int use_z) {
  if (!L.unsorted[blockIdx.y]) return;
  const BdNode nd = L.nodes[blockIdx.y];
  const int64_t nn = nd.nn;
  const double* D = L.Dcur + nd.lo;
  const double* z = use_z ? L.z + nd.lo : nullptr;
  const double* sk = L.sk + nd.lo;
  const int32_t* si = L.si + nd.lo;
  double* Ds = L.Ds + nd.lo;
  double* zs = L.zs + nd.lo;
  int32_t* perm = L.perm + nd.lo;
  const int64_t nch = (nn + ch - 1) / ch;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nn; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = q / ch;  // q: sorted place within chunk c
    const int32_t i = si[q];
    const double v = sk[q];
    int64_t rk = q - c * ch;
    for (int64_t c2 = 0; c2 < nch; ++c2) {
      if (c2 == c) continue;
      const int64_t b0 = c2 * ch, len = nn - b0 < ch ? nn - b0 : ch;
      int64_t lo = 0, hi = len;  // entries of chunk c2 before (v, i)
      while (lo < hi) {
        const int64_t m = (lo + hi) >> 1;
        if (bd_before(sk[b0 + m], si[b0 + m], v, i)) lo = m + 1;
        else hi = m;
      }
      rk += lo;
    }
    if (i < 0 || i >= nn || rk < 0 || rk >= nn) continue;  // cannot happen: a permutation
    Ds[rk] = D[i];
    if (z) zs[rk] = z[i];
    perm[rk] = i;
  }
}

// Deflation of one rank-one step over the sorted poles, by one block.  zs is normalised in
// place (rho = ||z||^2), tol = 8 eps max(|D|max, |z|max); type 1 deflates pole j when
// rho |z_j| <= tol.  Type 2 scans the survivors in order: the candidate p (the previous
// survivor, with its values as left by the scan) and the next survivor j give
// tau = hypot(z_j, z_p), c = z_j / tau, s = -z_p / tau; when |(D_j - D_p) c s| <= tol the
// rotation is recorded, z_j = tau, z_p = 0, both poles rotated, p deflated, else p is kept.
// The pairs are tested in parallel on the original values (valid whenever the previous
// pair did not rotate); one thread then resolves the chain, redoing a test only right after
// a rotation.  The outputs are those of the sequential scan: kept in scan order, rotations
// in order, defl in the order the scan deflates (keyed by the position being scanned),
// cnt = {K, nd, nrot}, *rho_out.  A non-finite pole or weight records TDC_ENONFINITE and
// deflates every pole (no secular solve and no product run on it).
constexpr int kBdDefThreads = 1024;
constexpr int64_t kBdDefMaxN = (int64_t)48 * 1024 * 8;  // two bit arrays in 96 KB of shared memory

// exclusive prefix of f over the block (blockDim.x = kBdDefThreads) and the block's total
__device__ __forceinline__ int block_scan_bd(int f, int* wcnt, int& total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned m = __ballot_sync(0xffffffffu, f);
  __syncthreads();
  if (lane == 0) wcnt[wid] = __popc(m);
  __syncthreads();
  int before = 0;
  total = 0;
  for (int w = 0; w < kBdDefThreads / 32; ++w) {
    if (w < wid) before += wcnt[w];
    total += wcnt[w];
  }
  return before + __popc(m & ((1u << lane) - 1u));
}

__global__ void __launch_bounds__(kBdDefThreads) k_bd_deflate(BdLevel L) {
  extern __shared__ unsigned rotbit[];  // speculative outcome of survivor pair (q - 1, q), then dbit
  __shared__ double red[32];
  __shared__ int wcnt[32];
  const int tid = threadIdx.x;
  const BdNode nd_ = L.nodes[blockIdx.x];
  const int64_t nn = nd_.nn, o = nd_.lo;
  double* Ds = L.Ds + o;
  double* zs = L.zs + o;
  int32_t* kept = L.kept + o;
  int32_t* defl = L.defl + o;
  int32_t* rotp = L.rotp + 2 * o;
  double* rotcs = L.rotcs + 2 * o;
  int32_t* cnt = L.cnt + 4 * blockIdx.x;
  int32_t* surv = L.surv + o;
  int32_t* slot = L.slot + o;
  double* rc = L.rc + o;
  double* rs = L.rs + o;
  double* rw = L.rw + o;
  double* rdp = L.rdp + o;
  double* rdn = L.rdn + o;
  double s2 = 0.0, dmax = 0.0;
  bool fin = true;
  for (int64_t i = tid; i < nn; i += blockDim.x) {
    const double z = zs[i], d = Ds[i];
    s2 = fma(z, z, s2);
    if (bd_key(fabs(d)) > bd_key(dmax)) dmax = fabs(d);
    fin = fin && (__double2hiint(z) & 0x7ff00000) != 0x7ff00000 && (__double2hiint(d) & 0x7ff00000) != 0x7ff00000;
  }
  const int bad = __syncthreads_or(!fin);
  s2 = bd_block_sum(s2, red);
  dmax = bd_block_max(bad ? 0.0 : dmax, red);
  if (bad || !isfinite(s2)) {
    if (tid == 0) set_status(L.status, TDC_ENONFINITE);
    for (int64_t i = tid; i < nn; i += blockDim.x) defl[i] = (int32_t)i;
    if (tid == 0) {
      cnt[0] = 0;
      cnt[1] = (int32_t)nn;
      cnt[2] = 0;
      L.rho[blockIdx.x] = 0.0;
    }
    return;
  }
  const double zn = sqrt(s2), rho = s2;
  double zmax = 0.0;
  for (int64_t i = tid; i < nn; i += blockDim.x) {
    double v = zs[i];
    if (zn > 0.0) v /= zn;
    zs[i] = v;
    if (bd_key(fabs(v)) > bd_key(zmax)) zmax = fabs(v);
  }
  zmax = bd_block_max(zmax, red);
  const double tol = 8.0 * kBdEps * fmax(dmax, zmax);
  // type 1, and the survivors compacted in order
  int64_t M = 0;
  for (int64_t i0 = 0; i0 < nn; i0 += blockDim.x) {
    const int64_t i = i0 + tid;
    const bool t1 = i < nn && (!(zn > 0.0) || rho * fabs(zs[i]) <= tol);
    const bool sv = i < nn && !t1;
    int total = 0;
    const int pos = block_scan_bd(sv ? 1 : 0, wcnt, total);
    if (sv) surv[M + pos] = (int32_t)i;
    if (i < nn) slot[i] = t1 ? (int32_t)i : -1;
    M += total;
  }
  // type 2 on the original values, every consecutive survivor pair at once
  const int64_t nwords = (M + 31) / 32;
  unsigned* dbit = rotbit + (nn + 31) / 32;  // survivor q deflated by a rotation
  for (int64_t w = tid; w < nwords; w += blockDim.x) dbit[w] = 0u;
  __syncthreads();  // the survivors' list is complete: each pair below reads entries of other threads
  for (int64_t q0 = 0; q0 < M; q0 += blockDim.x) {
    const int64_t q = q0 + tid;
    bool rot = false;
    if (q >= 1 && q < M) {
      const int32_t pa = surv[q - 1], pb = surv[q];
      const double zp = zs[pa], zj = zs[pb], dp = Ds[pa], dj = Ds[pb];
      const double t = dj - dp;
      double w, c, s;
      bd_rotation(zj, zp, w, c, s);
      rot = fabs(t * c * s) <= tol;
      if (rot) {
        rc[q] = c;
        rs[q] = s;
        rw[q] = w;
        rdp[q] = dp * c * c + dj * s * s;
        rdn[q] = dp * s * s + dj * c * c;
      }
    }
    const unsigned bits = __ballot_sync(0xffffffffu, rot);
    if ((tid & 31) == 0 && q < M) rotbit[q >> 5] = bits;
  }
  __syncthreads();
  // the chain, in one thread: a pair whose candidate was left unchanged takes its
  // speculative outcome, so the scan jumps from one speculative rotation to the next and
  // evaluates a pair itself only right after a rotation
  if (tid == 0) {
    int32_t nr = 0;
    bool mod = false;  // the candidate's values were changed by the previous rotation
    double zc = 0.0, dc = 0.0;
    int64_t q = 1;
    while (q < M) {
      bool rot;
      double c = 0.0, s = 0.0, w = 0.0, dp = 0.0, dn = 0.0;
      if (!mod) {
        int64_t wd = q >> 5;
        unsigned bits = rotbit[wd] & (0xffffffffu << (q & 31));
        while (bits == 0u && ++wd < nwords) bits = rotbit[wd];
        if (bits == 0u) break;
        q = wd * 32 + (__ffs(bits) - 1);
        if (q >= M) break;
        rot = true;
        c = rc[q];
        s = rs[q];
        w = rw[q];
        dp = rdp[q];
        dn = rdn[q];
      } else {
        const int32_t pb = surv[q];
        const double zj = zs[pb], dj = Ds[pb];
        bd_rotation(zj, zc, w, c, s);
        const double t = dj - dc;
        rot = fabs(t * c * s) <= tol;
        if (rot) {
          dp = dc * c * c + dj * s * s;
          dn = dc * s * s + dj * c * c;
        }
      }
      if (rot) {
        const int32_t pa = surv[q - 1], pb = surv[q];
        zs[pb] = w;
        zs[pa] = 0.0;
        Ds[pa] = dp;
        Ds[pb] = dn;
        rotp[2 * nr] = pa;
        rotp[2 * nr + 1] = pb;
        rotcs[2 * nr] = c;
        rotcs[2 * nr + 1] = s;
        ++nr;
        slot[pb] = pa;
        dbit[(q - 1) >> 5] |= 1u << ((q - 1) & 31);
        mod = true;
        zc = w;
        dc = dn;
      } else {
        mod = false;
      }
      ++q;
    }
    cnt[2] = nr;
    L.rho[blockIdx.x] = rho;
  }
  __syncthreads();
  // kept: the survivors no rotation deflated, in order
  int64_t K = 0;
  for (int64_t q0 = 0; q0 < M; q0 += blockDim.x) {
    const int64_t q = q0 + tid;
    const bool kp = q < M && !((dbit[q >> 5] >> (q & 31)) & 1u);
    int total = 0;
    const int pos = block_scan_bd(kp ? 1 : 0, wcnt, total);
    if (kp) kept[K + pos] = surv[q];
    K += total;
  }
  if (tid == 0) cnt[0] = (int32_t)K;
  // deflated entries in scan order
  int64_t nd = 0;
  for (int64_t i0 = 0; i0 < nn; i0 += blockDim.x) {
    const int64_t i = i0 + tid;
    const int32_t e = i < nn ? slot[i] : -1;
    int total = 0;
    const int pos = block_scan_bd(e >= 0 ? 1 : 0, wcnt, total);
    if (e >= 0) defl[nd + pos] = e;
    nd += total;
  }
  if (tid == 0) cnt[1] = (int32_t)nd;
}

// The deflation rotations on the columns of Q (sorted position p is column perm[p]), in
// order, each row independently.
__global__ void __launch_bounds__(256) k_bd_rotate(BdLevel L) {
  const int nr = L.cnt[4 * blockIdx.y + 2];
  if (nr <= 0) return;
  const BdNode nd = L.nodes[blockIdx.y];
  const int64_t nrows = nd.nn;
  double* Q = L.Q + nd.lo + nd.lo * L.ldq;
  const int32_t* perm = L.perm + nd.lo;
  const int32_t* rotp = L.rotp + 2 * nd.lo;
  const double* rotcs = L.rotcs + 2 * nd.lo;
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < nrows; r += (int64_t)gridDim.x * blockDim.x) {
    for (int t = 0; t < nr; ++t) {
      const int32_t pa = rotp[2 * t], pb = rotp[2 * t + 1];
      if (pa < 0 || pa >= nrows || pb < 0 || pb >= nrows || perm[pa] < 0 || perm[pa] >= nrows || perm[pb] < 0 ||
          perm[pb] >= nrows) {  // cannot happen for a permutation; never touch memory outside Q
        set_status(L.status, TDC_EUNSUPPORTED);
        continue;
      }
      double* a = Q + r + (int64_t)perm[pa] * L.ldq;
      double* bq = Q + r + (int64_t)perm[pb] * L.ldq;
      const double c = rotcs[2 * t], s = rotcs[2 * t + 1];
      const double x = *a, y = *bq;
      *a = c * x + s * y;
      *bq = c * y - s * x;
    }
  }
}

// Qw(:, t) = Q(:, perm[kept[t]]) for t < K, Q(:, perm[defl[t - K]]) after; the kept poles,
// their weights (squared, and the FP32 copies relative to the middle pole for the roots'
// pre-iteration) and the deflated values alongside.
__global__ void __launch_bounds__(256) k_bd_gather(BdLevel L) {
  const BdNode nd = L.nodes[blockIdx.y];
  const int64_t nrows = nd.nn, o = nd.lo;
  const int K = L.cnt[4 * blockIdx.y], ndf = L.cnt[4 * blockIdx.y + 1];
  const double* Q = L.Q + o + o * L.ldq;
  double* Qw = L.Qw + o * L.n;
  for (int64_t t = blockIdx.x; t < (int64_t)K + ndf; t += gridDim.x) {
    const int32_t sp = t < nrows ? (t < K ? L.kept[o + t] : L.defl[o + t - K]) : -1;
    if (sp < 0 || sp >= nrows || L.perm[o + sp] < 0 || L.perm[o + sp] >= nrows) {  // cannot happen; never
      if (threadIdx.x == 0) set_status(L.status, TDC_EUNSUPPORTED);                // read or write outside
      continue;
    }
    const double* src = Q + (int64_t)L.perm[o + sp] * L.ldq;
    double* dst = Qw + t * nrows;
    for (int64_t r = threadIdx.x; r < nrows; r += blockDim.x) dst[r] = src[r];
    if (threadIdx.x == 0) {
      const double d = L.Ds[o + sp];
      if (t < K) {
        const int32_t mid = L.kept[o + (K >> 1)];
        const double zt = L.zs[o + sp], x = d - ((mid >= 0 && mid < nrows) ? L.Ds[o + mid] : 0.0);
        const float xh = (float)x;
        L.DK[o + t] = d;
        L.zK[o + t] = zt;
        L.zz[o + t] = zt * zt;
        L.xz[o + t] = make_float2(xh, (float)(zt * zt));
        L.xlo[o + t] = (float)(x - (double)xh);
      } else {
        L.Dd[o + t - K] = d;
      }
    }
  }
}

// The level's products: split segments for nodes with K >= kBdSplitK (digit images one after
// the other), FP64 tiles for the others.  One warp, 32 nodes at a time.
constexpr int kBdSplitK = 128;
__global__ void __launch_bounds__(32) k_bd_segs(BdLevel L) {
  const int lane = threadIdx.x;
  int64_t base[5] = {0, 0, 0, 0, 0};  // A items, B items, tiles, image elements, segments
  for (int g0 = 0; g0 < L.count; g0 += 32) {
    const int g = g0 + lane;
    GemmSeg sg;
    memset(&sg, 0, sizeof(sg));
    int64_t v[5] = {0, 0, 0, 0, 0}, ael = 0;
    if (g < L.count) {
      const BdNode nd = L.nodes[g];
      const int K = L.cnt[4 * g];
      sg.ars = 1;
      sg.A = L.Qw + nd.lo * L.n;
      sg.lda = nd.nn;
      sg.rows = (int32_t)nd.nn;
      sg.kk = K;
      sg.K = K;
      sg.D = L.DK + nd.lo;
      sg.org = L.org + nd.lo;
      sg.tau = L.tau + nd.lo;
      sg.zhat = L.zhat + nd.lo;
      sg.scol = L.scol + nd.lo;
      sg.C = L.Q + nd.lo + nd.lo * L.ldq;
      sg.ldc = L.ldq;
      GemmSeg ds = sg;
      if (K >= kBdSplitK) {
        const int64_t RT = (nd.nn + kSplitBM - 1) / kSplitBM, KB = (K + kSplitBK - 1) / kSplitBK,
                      CT = (K + kSplitBN - 1) / kSplitBN;
        v[0] = RT * KB;
        v[1] = CT * KB;
        v[2] = RT * CT;
        ael = v[0] * L.S * kSplitBM * kSplitBK;
        v[3] = ael + v[1] * L.S * kSplitBN * kSplitBK;
        v[4] = 1;
        ds.K = 0;
      }
      L.dsegs[g] = ds;
    }
    int64_t at[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      int64_t inc = v[q];
      for (int of = 1; of < 32; of <<= 1) {
        const int64_t u = __shfl_up_sync(0xffffffffu, inc, of);
        if (lane >= of) inc += u;
      }
      at[q] = base[q] + inc - v[q];
      base[q] += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (v[4]) {
      sg.it_a = at[0];
      sg.it_b = at[1];
      sg.it_t = at[2];
      sg.a_img = at[3];
      sg.b_img = at[3] + ael;
      L.segs[at[4]] = sg;
    }
  }
  if (lane == 0) {
    GemmSeg last;
    memset(&last, 0, sizeof(last));
    last.it_a = base[0];
    last.it_b = base[1];
    last.it_t = base[2];
    last.a_img = base[3];
    if (base[3] > L.img_cap) {  // cannot happen with the host's bound; never write past the images
      last.it_a = last.it_b = last.it_t = 0;
      set_status(L.status, TDC_EUNSUPPORTED);
    }
    L.segs[base[4]] = last;
    *L.nsegs = base[4];
  }
}

// Q(:, K + t) = Qw(:, K + t) (deflated columns); D = [roots; deflated values], whose first run
// is the K roots.
__global__ void __launch_bounds__(256) k_bd_finish(BdLevel L) {
  const BdNode nd = L.nodes[blockIdx.y];
  const int64_t nrows = nd.nn, o = nd.lo;
  const int K = L.cnt[4 * blockIdx.y], ndf = L.cnt[4 * blockIdx.y + 1];
  const double* Qw = L.Qw + o * L.n;
  double* Q = L.Q + o + o * L.ldq;
  if (blockIdx.x == 0 && threadIdx.x == 0) L.cnt[4 * blockIdx.y + 3] = K;
  for (int64_t t = blockIdx.x; t < (int64_t)K + ndf && t < nrows; t += gridDim.x) {
    if (t >= K) {
      const double* src = Qw + t * nrows;
      double* dst = Q + t * L.ldq;
      for (int64_t r = threadIdx.x; r < nrows; r += blockDim.x) dst[r] = src[r];
    }
    if (threadIdx.x == 0) {
      const int32_t og = t < K ? L.org[o + t] : 0;
      L.Dcur[o + t] = t >= K ? L.Dd[o + t - K]
                             : (og >= 0 && og < K ? L.DK[o + og] + L.tau[o + t]
                                                  : __longlong_as_double(0x7ff8000000000000ll));
    }
  }
}

// The node's final order: Qw(:, t) = Q(:, perm[t]) (back = 0), Q(:, t) = Qw(:, t) and lam (1).
__global__ void __launch_bounds__(256) k_bd_order(BdLevel L, double* lam, int back) {
  const BdNode nd = L.nodes[blockIdx.y];
  const int64_t nrows = nd.nn, o = nd.lo;
  double* Qw = L.Qw + o * L.n;
  double* Q = L.Q + o + o * L.ldq;
  for (int64_t t = blockIdx.x; t < nrows; t += gridDim.x) {
    const int32_t c = L.perm[o + t];
    if (!back && (c < 0 || c >= nrows)) {  // cannot happen for a permutation
      if (threadIdx.x == 0) set_status(L.status, TDC_EUNSUPPORTED);
      continue;
    }
    const double* src = back ? Qw + t * nrows : Q + (int64_t)c * L.ldq;
    double* dst = back ? Q + t * L.ldq : Qw + t * nrows;
    for (int64_t r = threadIdx.x; r < nrows; r += blockDim.x) dst[r] = src[r];
    if (back && threadIdx.x == 0) lam[o + t] = L.Ds[o + t];
  }
}

__global__ void __launch_bounds__(256) k_bd_zero(int64_t rows, int64_t cols, double* Q, int64_t ldq) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < rows * cols;
       t += (int64_t)gridDim.x * blockDim.x)
    Q[t % rows + (t / rows) * ldq] = 0.0;
}

__global__ void __launch_bounds__(256) k_bd_copy_band(int64_t n, int b, const double* AB, int64_t ldab, double* ABw) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)(b + 1) * n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = t % (b + 1), j = t / (b + 1);
    ABw[r + j * (b + 1)] = (j + r < n) ? AB[r + j * ldab] : 0.0;
  }
}

namespace {
unsigned grid_for(int64_t work, int64_t per = 256, int64_t cap = 4096) {
  const int64_t g = (work + per - 1) / per;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(g, cap));
}
}  // namespace

cudaError_t launch_bd_copy_band(int64_t n, int b, const double* AB, int64_t ldab, double* ABw, cudaStream_t s) {
  k_bd_copy_band<<<grid_for((int64_t)(b + 1) * n), 256, 0, s>>>(n, b, AB, ldab, ABw);
  return cudaGetLastError();
}
cudaError_t launch_bd_nodes(BdNode* dst, const BdNodeTable& T, int count, cudaStream_t s) {
  k_bd_nodes<<<1, 32, 0, s>>>(dst, T, count);
  return cudaGetLastError();
}
cudaError_t launch_bd_tear(const BdNode* nodes, int count, double* ABw, int64_t ldab, int b, double* wv,
                           cudaStream_t s) {
  if (b <= 0 || count <= 0) return cudaSuccess;
  k_bd_tear<<<(unsigned)count, 256, sizeof(double) * (size_t)(b * b + b), s>>>(nodes, ABw, ldab, b, wv);
  return cudaGetLastError();
}
cudaError_t launch_bd_leaf_trd(const BdLeafArgs& A, const BdLeafTable& T, cudaStream_t s) {
  if (A.nleaf <= 0) return cudaSuccess;
  k_bd_leaf_trd<<<(unsigned)A.nleaf, kBdLeafThreads, 0, s>>>(A, T);
  return cudaGetLastError();
}
cudaError_t launch_bd_leaf_back(const BdLeafArgs& A, const BdLeafTable& T, cudaStream_t s) {
  if (A.nleaf <= 0) return cudaSuccess;
  int lmax = 0;
  for (int t = 0; t < A.nleaf; ++t) lmax = std::max(lmax, T.L[t]);
  const dim3 grid((unsigned)A.nleaf, (unsigned)((lmax + 3) / 4));
  if (lmax <= 128) k_bd_leaf_back<4><<<grid, 128, 0, s>>>(A, T);
  else if (lmax <= 256) k_bd_leaf_back<8><<<grid, 128, 0, s>>>(A, T);
  else k_bd_leaf_back<16><<<grid, 128, 0, s>>>(A, T);
  return cudaGetLastError();
}
static dim3 bd_grid(const BdLevel& L, int64_t work, int64_t per, int64_t cap) {
  return dim3(grid_for(work, per, cap), (unsigned)L.count);
}

cudaError_t launch_bd_level_begin(const BdLevel& L, const double* lam, cudaStream_t s) {
  k_bd_level_begin<<<bd_grid(L, L.max_nn, 256, 4096), 256, 0, s>>>(L, lam);
  return cudaGetLastError();
}

static cudaError_t bd_sort(const BdLevel& L, int use_z, cudaStream_t s) {
  int ch = 2;
  while (ch < kBdChunk && ch < L.max_nn) ch <<= 1;
  k_bd_merge<<<(unsigned)L.count, 1024, 0, s>>>(L, use_z);
  k_bd_chunk_sort<<<bd_grid(L, L.max_nn, ch, 1 << 20), std::max(32, std::min(1024, ch / 2)), 0, s>>>(L, ch);
  k_bd_rank<<<bd_grid(L, L.max_nn, 256, 4096), 256, 0, s>>>(L, ch, use_z);
  return cudaGetLastError();
}

cudaError_t launch_bd_term(const BdLevel& L, int term, cudaStream_t s) {
  if (L.max_nn > kBdDefMaxN) return cudaErrorInvalidValue;
  const size_t smem = 2 * sizeof(unsigned) * (size_t)((std::max<int64_t>(L.max_nn, 1) + 31) / 32);
  static std::atomic<bool> attr[64];  // once per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!attr[dev]) {
    e = cudaFuncSetAttribute(k_bd_deflate, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
    if (e != cudaSuccess) return e;
    attr[dev] = true;
  }
  k_bd_z<<<bd_grid(L, L.max_nn, 256, 4096), 256, 0, s>>>(L, term);
  e = bd_sort(L, 1, s);
  if (e != cudaSuccess) return e;
  k_bd_deflate<<<(unsigned)L.count, kBdDefThreads, smem, s>>>(L);
  k_bd_rotate<<<bd_grid(L, L.max_nn, 256, 4096), 256, 0, s>>>(L);
  k_bd_gather<<<bd_grid(L, L.max_nn, 1, 8192), 256, 0, s>>>(L);
  return cudaGetLastError();
}

cudaError_t launch_bd_segs(const BdLevel& L, cudaStream_t s) {
  k_bd_segs<<<1, 32, 0, s>>>(L);
  return cudaGetLastError();
}

cudaError_t launch_bd_finish(const BdLevel& L, cudaStream_t s) {
  k_bd_finish<<<bd_grid(L, L.max_nn, 1, 8192), 256, 0, s>>>(L);
  return cudaGetLastError();
}

cudaError_t launch_bd_order(const BdLevel& L, double* lam, cudaStream_t s) {
  const cudaError_t e = bd_sort(L, 0, s);
  if (e != cudaSuccess) return e;
  k_bd_order<<<bd_grid(L, L.max_nn, 1, 8192), 256, 0, s>>>(L, lam, 0);
  k_bd_order<<<bd_grid(L, L.max_nn, 1, 8192), 256, 0, s>>>(L, lam, 1);
  return cudaGetLastError();
}
cudaError_t launch_bd_zero(int64_t rows, int64_t cols, double* Q, int64_t ldq, cudaStream_t s) {
  k_bd_zero<<<grid_for(rows * cols), 256, 0, s>>>(rows, cols, Q, ldq);
  return cudaGetLastError();
}

}  // namespace tdc
