// lbm_cols.h -- columns of a row that a lane of the two-node stream-collide
// kernel loads (plain C++, so that the index arithmetic runs on the host too).
#pragma once

#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif

namespace lbm {

// x0: first node of the lane's pair (even, >= nx for lanes past the row); nx
// even, >= 4.  Every column is that of a whole pair inside the row, also for
// the lanes past it (they take the last pair and store nothing).
struct PairCols {
    int own;   // the lane's pair
    int left;  // the pair that holds x0 - 1 as its second node (periodic)
    int right; // the pair that holds x0 + 2 as its first node (periodic)
};

LBM_HD PairCols pair_cols(int x0, int nx) {
    PairCols c;
    c.own = x0 < nx ? x0 : nx - 2;
    c.left = (c.own == 0 ? nx : c.own) - 2;
    c.right = c.own + 2 >= nx ? 0 : c.own + 2;
    return c;
}

} // namespace lbm
