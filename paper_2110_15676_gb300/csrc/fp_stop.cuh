// Stop test of the fixed point in its graph form (Sec. 4), run by every block of a solver launch
// before it solves.
#pragma once

namespace afc {

// fixed-point scalar slots (problem scalars p->scal)
enum : int {
  F_NORMSQ = 0, F_CORR = 1, F_INNER = 2, F_RES0 = 3, F_RESF = 4, F_STATUS = 5, F_THRESH = 6, F_FIXED = 7,
  F_MAXIT = 8, F_REVAL = 10, F_TIMEOUT = 11
};
// F_STATUS: 0 running, 1 converged / fixed count reached, 2 non-finite or a solver that
// could not finish, 3 iteration limit; F_TIMEOUT: 1 after a grid barrier of the
// persistent solve gave up waiting (F_STATUS is then 2)

#ifdef __CUDACC__
// R = ||res|| from the residual pass's block partials (sum(): their total, for every thread of the
// block) and the tests; true: solve.  Block 0 also writes the scalars and, with set(go), the loop's
// condition.  As kernels of their own the sum, the test and the branch over the solve took two graph
// nodes per correction.
//
// Block 0 may store F_STATUS while a later block reads it.  One thread of a block reads the two words
// that change, so that a block decides as one whichever value it meets: blocks that meet the old
// status sum the same partials and decide as block 0 did, blocks that meet the new one return what
// it decided.  (Read by each thread, a store between two warps' reads let one warp leave and the
// other go on into sums and barriers that wait for both.)  F_CORR, and F_STATUS after a decision to
// solve, change only at the end of the solve, after grid sums that every block has joined.
template <class Scalars, class Sum, class Set>
__device__ __forceinline__ bool fp_decide(Scalars sc, Sum&& sum, Set&& set) {
  __shared__ double was, corr;
  __shared__ bool go;
  if (threadIdx.x == 0) {
    was = sc[F_STATUS];
    corr = sc[F_CORR];
  }
  __syncthreads();
  if (was == 1.0 || was == 3.0) return false;   // the loop has stopped earlier in this body
  const double total = sum();
  if (threadIdx.x == 0) {
    const double R = sqrt(total);
    double status = 0.0;
    if (!isfinite(R) || was == 2.0) status = 2.0;
    else if (sc[F_FIXED] > 0.0) status = corr >= sc[F_FIXED] ? 1.0 : 0.0;
    else if (R < sc[F_THRESH]) status = 1.0;
    else if (corr >= sc[F_MAXIT]) status = 3.0;
    go = status == 0.0;
    if (blockIdx.x == 0) {
      sc[F_NORMSQ] = total;
      if (sc[F_REVAL] == 0.0) sc[F_RES0] = R;
      sc[F_RESF] = R;
      sc[F_REVAL] = sc[F_REVAL] + 1.0;
      if (!go) sc[F_STATUS] = status;
      set(go);
    }
  }
  __syncthreads();
  return go;
}
#endif

}  // namespace afc
