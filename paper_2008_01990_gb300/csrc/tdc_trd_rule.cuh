// Which blocks take part in the exchanges of the resident reduction (k_trd_resident).  Plain
// integer arithmetic, also compiled for the host, where the counts can be stepped through for
// every order and grid.
//
// Column c of the m x m trailing matrix lies in block c mod G.  Block b (b < m) takes part in
// step k as long as it owns a column past k; then it leaves without arriving any more.  A block
// counts in the arrivals of exactly the steps in which it takes part: with one column a block
// (m <= G) the owner of column 0 takes part in none, not even the first.
#pragma once

#ifdef __CUDACC__
#define TDC_TRD_RULE __host__ __device__ inline
#else
#define TDC_TRD_RULE inline
#endif

namespace tdc {

// the last column of block b
TDC_TRD_RULE int trd_res_last(int b, int m, int G) { return b + (m - 1 - b) / G * G; }
// whether a block whose last column is `last` takes part in step k
TDC_TRD_RULE bool trd_res_takes_part(int last, int k) { return last > k; }
// blocks taking part in step k: the owners of columns k + 1 .. m - 1
TDC_TRD_RULE int trd_res_arrivals(int k, int m, int G) { return m - 1 - k < G ? m - 1 - k : G; }
// the block that writes step k's results (k + 2 < m): one that takes part in step k + 1 too
TDC_TRD_RULE int trd_res_writer(int k, int m, int G) { return (m - 1 - k % trd_res_arrivals(k + 1, m, G)) % G; }

}  // namespace tdc

#undef TDC_TRD_RULE
