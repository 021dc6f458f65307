// Solve-phase launchers and the device-resident CG scalars.
#pragma once

#include <vector>

#include "common.cuh"

namespace sa {

struct CsrView {
  int64_t n = 0, nnz = 0;
  const int64_t* rp = nullptr;
  const int32_t* ci = nullptr;
  const double* v = nullptr;
  int sw = 8;  // lanes per row
};

// right-hand sides one multi-vector solve carries (interleaved storage:
// element (i, c) of an n x k block at i*k + c)
constexpr int KMAX_BLOCK = 8;

struct CgScalars {
  double rz, pq, alpha, beta;
  int breakdown;
  int pad;
};

int pick_sw(int64_t n, int64_t nnz);
struct Fin;  // what the last block of a reduction does (reduce.cuh)
int launch_dots(cudaStream_t st, int64_t n, const double* a0, const double* b0, const double* a1, const double* b1,
                double* part, const Fin& fin);
int launch_fin_wide(cudaStream_t st, const double* part, int np, const Fin& fin);
int launch_cg_update(cudaStream_t st, int64_t n, const CgScalars* s, const double* p, const double* q, double* x,
                     double* r, double* rprev, double* part, const Fin& fin);
int launch_cg_pupdate(cudaStream_t st, int64_t n, const CgScalars* s, const double* z, double* p, int first);

// k-column versions (k <= KMAX_BLOCK), each column summed in the one-vector
// order so that a column of a block solve equals the one-vector solve bitwise
// (bdots: a . b per column, and b . c where c is given)
int launch_bdots(cudaStream_t st, int64_t n, int k, const double* a, const double* b, const double* c, double* part,
                 const Fin& fin);
int launch_bcg_update(cudaStream_t st, int64_t n, int k, const CgScalars* s, const int* active, const double* p,
                      const double* q, double* x, double* r, double* rprev, double* part, const Fin& fin);
int launch_bcg_pupdate(cudaStream_t st, int64_t n, int k, const CgScalars* s, const int* active, const double* z,
                       double* p, int first);
// column-major n x k <-> interleaved n x K (K >= k; columns k..K-1 zero)
int launch_interleave(cudaStream_t st, int64_t n, int k, int K, const double* src, double* dst, int to_interleaved);

// dense coarse level (dense.cu).  The coarse matrix A_c = L L^T (Cholesky)
// is solved by block substitution over diagonal blocks of COARSE_BS rows:
// L (row-major, lower triangle), LT = L^T, W = the inverses of the diagonal
// blocks L_KK (stored at their place in an n x n array; the rest unused) and
// WT = W^T.  Only the diagonal blocks are inverted (n COARSE_BS^2 / 3 flops
// instead of n^3 / 3 for the whole inverse).
constexpr int64_t COARSE_BS = 1024;

// Only the skyline of L is stored (tiles of 32 x 32 from each tile row's
// first nonzero tile column on), the rest of L is unset.

// one step of a coarse solve: rows [rb, re) of the diagonal block [r0, r1)
enum CoarseMode { CS_W = 0, CS_WT = 1, CS_L = 2, CS_LT = 3 };
struct CoarseEnt {
  int blk0;      // first block in a launch of several problems
  int prob;      // and its problem
  int mode;
  int rb, re, r0, r1;
  int split;     // columns below it come from the first operand (dense.cu)
};

struct CoarseFactor {
  Buf<double> L, LT, W, WT;
  // per tile row of 32: the first tile column of its skyline; then per tile
  // column the end of the tile rows that reach it; then the factorisation's
  // own tables
  Buf<int32_t> sky;
  std::vector<CoarseEnt> steps;  // of the solve
  double entries = 0;            // matrix entries that one solve reads
};

struct CoarseView {
  int64_t n = 0;
  const double* L = nullptr;
  const double* LT = nullptr;
  const double* W = nullptr;
  const double* WT = nullptr;
  const int32_t* first = nullptr;  // skyline: first tile column per tile row
  const int32_t* end = nullptr;    // ... and end of the tile rows per tile column
  const std::vector<CoarseEnt>* steps = nullptr;  // host (the factor's)
  double entries = 0;
};

inline CoarseView coarse_view(const CoarseFactor& F, int64_t n) {
  CoarseView v;
  v.n = n; v.L = F.L.p; v.LT = F.LT.p; v.W = F.W.p; v.WT = F.WT.p;
  v.first = F.sky.p; v.end = F.sky.p + (n + 31) / 32;
  v.steps = &F.steps;
  v.entries = F.entries;
  return v;
}

// one coarse solve: x = A_c^-1 bin; t and y: n-vector workspaces (no two of
// bin, t, y, x alias); xo (may be NULL) also receives sq_i x_i in FP32 or FP64
struct CoarseProb {
  int64_t n = 0;
  CoarseView F;
  const double* bin = nullptr;
  double *t = nullptr, *y = nullptr, *x = nullptr;
  void* xo = nullptr;
  const double* sq = nullptr;
  int xo_f32 = 0;
};
inline CoarseProb coarse_prob(const CoarseView& F, const double* b, double* t, double* y, double* x,
                              const double* sq = nullptr, void* xo = nullptr, int xo_f32 = 0) {
  CoarseProb p;
  p.n = F.n; p.F = F; p.bin = b; p.t = t; p.y = y; p.x = x; p.sq = sq; p.xo = xo; p.xo_f32 = xo_f32;
  return p;
}

// dense_start enqueues the whole factorisation on a stream of its own, forked
// from al.stream after the dense copy of A; dense_finish makes al.stream wait
// for it and reports a pivot that was not positive (SA_ERR_NOT_SPD).  Work on
// al.stream in between must not read the factor.
struct DenseJob {
  Buf<double> Dinv;
  Buf<int> err;           // error bits, ticket counter
  Buf<int32_t> flag;      // per tile of L: written
  cudaStream_t main = nullptr, sd = nullptr;
  cudaEvent_t e_fork = nullptr, e_done = nullptr;
  int64_t n = 0;
  int level = 0;         // for the setup-phase profile
  bool pending = false;  // forked and not yet joined
  DenseJob() = default;
  DenseJob(const DenseJob&) = delete;
  DenseJob& operator=(const DenseJob&) = delete;
  ~DenseJob();
};
int dense_start(Alloc& al, int64_t n, const int64_t* rp, const int32_t* ci, const double* v, CoarseFactor& F,
                DenseJob& job);
int dense_finish(DenseJob& job);
// one solve with k in {1, 2, 4, 8} interleaved columns
int launch_coarse_solve(cudaStream_t st, int k, const CoarseProb& P);
// the steps of one solve (first, end: the skyline on the host), and the matrix
// entries they read; one step of several problems in one launch (entries in the
// order of their blocks)
double coarse_steps(int64_t n, const int32_t* first, const int32_t* end, std::vector<CoarseEnt>& out);
int coarse_blocks(const CoarseEnt& E);
int launch_coarse_group(cudaStream_t st, const CoarseEnt* ent, int nent, int blocks, const CoarseProb* probs);

}  // namespace sa
