// Setup kernels whose floating-point results must be bitwise reproducible:
// Dirichlet detection, nodal tensors and their inverses, the two strength
// measures with pointwise dropping, the filtered matrix with lumping and the
// 1-norm diagonal, coarse auxiliary data, and the smoothed prolongator
// values.  This translation unit is compiled with -fmad=false: every
// expression below is evaluated with separately rounded IEEE operations in
// the order written, and every sum runs in ascending column / index order.
#include <math.h>

#include "common.cuh"
#include "kernels.cuh"

namespace sa {

// ---------------------------------------------------------------------------
// a1. Dirichlet detection + diagonal (Sec. 3, Fig. 4 caption: Dirichlet
// nodes are isolated in the filtered graph).  Warp per row.  A row is
// Dirichlet iff every stored off-diagonal value is exactly zero.  err bit 1:
// a row without a stored diagonal.
// ---------------------------------------------------------------------------
__global__ void k_dirichlet_diag(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                 const double* __restrict__ v, uint8_t* __restrict__ dir,
                                 double* __restrict__ diag, int* __restrict__ err) {
  const int lane = lane_id();
  for (int64_t i = global_warp(); i < n; i += warp_stride()) {
    const int64_t b = rp[i], e = rp[i + 1];
    bool offnz = false, has_d = false;
    double d = 0.0;
    for (int64_t p = b + lane; p < e; p += 32) {
      int32_t j = ci[p];
      double a = v[p];
      if (j == (int32_t)i) { d = a; has_d = true; }
      else if (a != 0.0) offnz = true;
    }
    unsigned anyoff = __ballot_sync(FULL, offnz);
    unsigned hd = __ballot_sync(FULL, has_d);
    // exactly one lane holds the diagonal
    double dd = hd ? __shfl_sync(FULL, d, __ffs(hd) - 1) : 0.0;
    if (lane == 0) {
      if (dir) dir[i] = anyoff ? 0 : 1;
      diag[i] = dd;
      if (!hd) atomicOr(err, 1);
    }
  }
}

// input check of the level-0 CSR: row pointers monotone from 0 to nnz,
// columns in [0, n) and strictly ascending in each row.  err bit 32.
__global__ void k_validate_csr(int64_t n, int64_t ncols, int64_t nnz, const int64_t* __restrict__ rp,
                               const int32_t* __restrict__ ci, int* __restrict__ err) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t b = rp[i], e = rp[i + 1];
  if ((i == 0 && b != 0) || (i == n - 1 && e != nnz) || e < b || b < 0 || e > nnz) {
    atomicOr(err, 32);
    return;
  }
  int32_t prev = -1;
  for (int64_t p = b; p < e; ++p) {
    int32_t j = ci[p];
    if (j <= prev || j < 0 || (int64_t)j >= ncols) { atomicOr(err, 32); return; }
    prev = j;
  }
}

// ---------------------------------------------------------------------------
// a2. nodal tensors and inverses (Sec. 3: Clement interpolant of an
// elementwise tensor; inverse by adjugate / determinant)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void invert_packed(int dim, const double* t, double* si) {
  if (dim == 2) {
    double det = t[0] * t[1] - t[2] * t[2];
    si[0] = t[1] / det;
    si[1] = t[0] / det;
    si[2] = -t[2] / det;
  } else {
    double a = t[0], b = t[1], c = t[2], d = t[3], e = t[4], f = t[5];
    double c00 = b * c - f * f;
    double c11 = a * c - e * e;
    double c22 = a * b - d * d;
    double c01 = e * f - d * c;
    double c02 = d * f - b * e;
    double c12 = d * e - a * f;
    double det = a * c00 + d * c01 + e * c02;
    si[0] = c00 / det;
    si[1] = c11 / det;
    si[2] = c22 / det;
    si[3] = c01 / det;
    si[4] = c02 / det;
    si[5] = c12 / det;
  }
}

__global__ void k_node_elem_count(int64_t ne, int npe, const int32_t* __restrict__ en, int64_t n,
                                  int64_t* __restrict__ cnt, int* __restrict__ err) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ne * npe) return;
  int32_t node = en[t];
  if (node < 0 || node >= n) { atomicOr(err, 2); return; }
  atomicAdd((unsigned long long*)&cnt[node + 1], 1ull);
}

__global__ void k_node_elem_fill(int64_t ne, int npe, const int32_t* __restrict__ en, int64_t n,
                                 const int64_t* __restrict__ off, int* __restrict__ cursor,
                                 int32_t* __restrict__ list) {
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ne * npe) return;
  int32_t node = en[t];
  if (node < 0 || node >= n) return;
  int pos = atomicAdd(&cursor[node], 1);
  list[off[node] + pos] = (int32_t)(t / npe);
}

// thread per node: sort incident elements ascending, average, invert
__global__ void k_node_tensor_from_elems(int64_t n, int dim, const int64_t* __restrict__ off,
                                         int32_t* __restrict__ list, const double* __restrict__ meas,
                                         const double* __restrict__ et, double* __restrict__ sigma,
                                         double* __restrict__ sinv, int* __restrict__ err) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int kp = dim == 3 ? 6 : 3;
  const int64_t b = off[i], e = off[i + 1];
  for (int64_t p = b + 1; p < e; ++p) {  // insertion sort of the node's own segment
    int32_t key = list[p];
    int64_t q = p - 1;
    while (q >= b && list[q] > key) { list[q + 1] = list[q]; --q; }
    list[q + 1] = key;
  }
  double num[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  double den = 0.0;
  for (int64_t p = b; p < e; ++p) {
    int64_t el = list[p];
    double m = meas[el];
    for (int c = 0; c < kp; ++c) num[c] += m * et[el * kp + c];
    den += m;
  }
  if (den == 0.0) atomicOr(err, 4);
  double s[6];
  for (int c = 0; c < kp; ++c) {
    s[c] = num[c] / den;
    sigma[i * kp + c] = s[c];
  }
  double si[6];
  invert_packed(dim, s, si);
  for (int c = 0; c < kp; ++c) sinv[i * kp + c] = si[c];
}

// per-node tensors given (copy) or sigma = I (distance Laplacian); invert
__global__ void k_node_tensor_direct(int64_t n, int dim, const double* __restrict__ given,
                                     double* __restrict__ sigma, double* __restrict__ sinv) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int kp = dim == 3 ? 6 : 3;
  double s[6];
  for (int c = 0; c < kp; ++c) {
    s[c] = given ? given[i * kp + c] : (c < dim ? 1.0 : 0.0);
    sigma[i * kp + c] = s[c];
  }
  double si[6];
  invert_packed(dim, s, si);
  for (int c = 0; c < kp; ++c) sinv[i * kp + c] = si[c];
}

// ---------------------------------------------------------------------------
// a4. material-aware distance Laplacian (Sec. 2.1 distance Laplacian,
// Sec. 3 material distance with max symmetrisation):
//   w_ij = 1 / max(d^T sinv_i d, d^T sinv_j d), d = x_i - x_j,
//   D_i = sum_{j != i} w_ij (ascending column order).
// ---------------------------------------------------------------------------
__device__ __forceinline__ double quad_form(int dim, const double* __restrict__ si, const double* d) {
  // t = sigma^-1 d, then d . t, as running sums of fused multiply-adds in
  // index order (explicit __fma_rn: one rounding per term even under
  // -fmad=false); even in d bit for bit
  if (dim == 2) {
    const double t0 = __fma_rn(si[2], d[1], si[0] * d[0]);
    const double t1 = __fma_rn(si[1], d[1], si[2] * d[0]);
    return __fma_rn(d[1], t1, d[0] * t0);
  }
  const double t0 = __fma_rn(si[4], d[2], __fma_rn(si[3], d[1], si[0] * d[0]));
  const double t1 = __fma_rn(si[5], d[2], __fma_rn(si[1], d[1], si[3] * d[0]));
  const double t2 = __fma_rn(si[2], d[2], __fma_rn(si[5], d[1], si[4] * d[0]));
  return __fma_rn(d[2], t2, __fma_rn(d[1], t1, d[0] * t0));
}

// w_ij = 1 / max(q_ij, q_ji) for the entries above the diagonal (j > i);
// the diagonal gets 0 and the lower entries are mirrored afterwards.  For
// (j, i) the difference vector is exactly -(x_i - x_j), and both quadratic
// forms are even in it with sign-symmetric rounding, so w_ji computed from row
// j would be the same bits: computing each pair once halves the FP64 work.
// Bound by FP64 issue (38 FP64 instructions a pair, 16 cycles each per SM), so
// every lane of a warp takes a pair: the pairs of PAIR_ROWS rows are
// numbered through (offsets in shared memory), whatever the rows' lengths -- a
// thread per row left long coarse rows as tails, a warp per row 13 of 32
// lanes.  Where both ends carry the same tensor, bit for bit (the inside of a
// material region), q_ji = q_ij and its twelve instructions are left out.
// 2.1M nodes, 64 Voronoi regions: 1733 us with a thread per row; coarse
// levels of the stretched battery stack: 251 us on average with a warp per row
// Rows of a block: 64, or 8 on small levels of long rows, where blocks of 64 leave
// the chip idle and one long row holds up 63 (both kernels; start: a warp per row):
//   44k rows of 29 entries   137 us, 250 at 64, 99 at 8
//   6.6k rows of 117          71 us, 131 at 64, 59 at 8
//   73k rows of 44           285 us, 226 at 64, 176 at 8
//   131k rows of 26          307 us, 154 at 64, 194 at 8
//   16k rows of 10            30 us,  17 at 64,  21 at 8
constexpr int PAIR_THREADS = 256;

// a level of few rows that are long (coarse 3D levels): a row's work is then spread
// over a warp or a block of few rows
constexpr int64_t FEW_ROWS = 65536, LONG_MEAN = 24;
inline bool few_long_rows(int64_t n, int64_t nnz) { return n < FEW_ROWS && nnz > LONG_MEAN * n; }

// pair numbering of the block's rows r0 .. r0 + ROWS - 1: the entries
// above (UPPER) or below the diagonal of row r0 + r are start[r] + 0, 1, ...
// and pairs off[r] .. off[r + 1] - 1
template <bool UPPER, int ROWS>
__device__ __forceinline__ void pair_offsets(int64_t n, const int64_t* __restrict__ rp,
                                             const int32_t* __restrict__ ci, int64_t r0, int64_t* start, int* off,
                                             double* __restrict__ w) {
  __shared__ int wsum;
  const int t = (int)threadIdx.x, lane = t & 31;
  int cnt = 0;
  if (t < ROWS) {
    const int64_t i = r0 + t;
    int64_t st = 0;
    if (i < n) {
      const int64_t b = rp[i], e = rp[i + 1];
      // first entry with column > i (UPPER) or >= i
      int64_t lo = b, hi = e;
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        const bool left = UPPER ? ci[mid] <= (int32_t)i : ci[mid] < (int32_t)i;
        if (left) lo = mid + 1;
        else hi = mid;
      }
      st = UPPER ? lo : b;
      cnt = (int)(UPPER ? e - lo : lo - b);
      if (UPPER && lo > b && ci[lo - 1] == (int32_t)i) w[lo - 1] = 0.0;
    }
    start[t] = st;
  }
  int inc = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(FULL, inc, o);
    if (lane >= o) inc += u;
  }
  if (t == 31) wsum = inc;
  __syncthreads();
  if (t < ROWS) off[t + 1] = inc + (t >= 32 ? wsum : 0);
  if (t == 0) off[0] = 0;
  __syncthreads();
}

// whether a row of the block is not strictly ascending: a descent between
// neighbouring entries that is not the step from one row to the next
template <int ROWS>
__device__ __forceinline__ bool pair_unsorted(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                              int64_t r0) {
  __shared__ int64_t rs[ROWS + 1];
  const int t = (int)threadIdx.x;
  if (t <= ROWS) rs[t] = rp[r0 + t < n ? r0 + t : n];
  __syncthreads();
  bool bad = false;
  for (int64_t p = rs[0] + t; p + 1 < rs[ROWS]; p += PAIR_THREADS) {
    if (ci[p] < ci[p + 1]) continue;
    int lo = 0, hi = ROWS;  // the last row start <= p + 1
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (rs[mid] <= p + 1) lo = mid;
      else hi = mid - 1;
    }
    bad |= rs[lo] != p + 1;
  }
  return __syncthreads_or(bad) != 0;
}

// the row (of the block) that pair q belongs to
template <int ROWS>
__device__ __forceinline__ int pair_row(const int* off, int q) {
  int lo = 0, hi = ROWS - 1;
#pragma unroll
  for (int s = 1; s < ROWS; s *= 2) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= q) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

template <int DIM>
__device__ __forceinline__ double pair_weight(const double* __restrict__ x, const double* __restrict__ sinv, int64_t i,
                                              int64_t j) {
  constexpr int KP = DIM == 3 ? 6 : 3;
  double d[3], si[KP], sj[KP];
#pragma unroll
  for (int c = 0; c < DIM; ++c) d[c] = x[i * DIM + c] - x[j * DIM + c];
  bool same = true;
#pragma unroll
  for (int c = 0; c < KP; ++c) {
    si[c] = sinv[i * KP + c];
    sj[c] = sinv[j * KP + c];
    same &= __double_as_longlong(si[c]) == __double_as_longlong(sj[c]);
  }
  const double qij = quad_form(DIM, si, d);
  double m = qij;
  if (!same) {
    const double qji = quad_form(DIM, sj, d);
    m = qij > qji ? qij : qji;
  }
  return 1.0 / m;
}

// CHECK: the rows may be in any order (a caller's matrix).  A block that has a
// row out of order takes every entry of its rows by the expression and says so
// in `unsorted`, and the mirror leaves it alone.  The check reads the columns'
// lower half besides (strength filter on 2.1M nodes 2656 -> 2666 us).
template <int DIM, bool CHECK, int ROWS>
__global__ void __launch_bounds__(PAIR_THREADS) k_material_w(int64_t n, const int64_t* __restrict__ rp,
                                                             const int32_t* __restrict__ ci,
                                                             const double* __restrict__ x,
                                                             const double* __restrict__ sinv, double* __restrict__ w,
                                                             uint8_t* __restrict__ unsorted) {
  __shared__ int64_t start[ROWS];
  __shared__ int off[ROWS + 1];
  const int64_t r0 = (int64_t)blockIdx.x * ROWS;
  if constexpr (CHECK) {
    const bool any = pair_unsorted<ROWS>(n, rp, ci, r0);
    if (threadIdx.x == 0) unsorted[blockIdx.x] = any;
    if (any) {
      for (int64_t i = r0 + (threadIdx.x >> 5); i < r0 + ROWS && i < n; i += PAIR_THREADS / 32)
        for (int64_t p = rp[i] + lane_id(); p < rp[i + 1]; p += 32)
          w[p] = ci[p] == (int32_t)i ? 0.0 : pair_weight<DIM>(x, sinv, i, ci[p]);
      return;
    }
  }
  pair_offsets<true, ROWS>(n, rp, ci, r0, start, off, w);
  const int tot = off[ROWS];
  for (int q = (int)threadIdx.x; q < tot; q += PAIR_THREADS) {
    const int r = pair_row<ROWS>(off, q);
    const int64_t p = start[r] + (q - off[r]);
    w[p] = pair_weight<DIM>(x, sinv, r0 + r, ci[p]);
  }
}

// lower entries: w_ij = w_ji.  On a symmetric stencil entry k of row i is
// entry len - 1 - k of row j, which is tried first, then a binary search in
// row j; a pattern without that entry (not structurally symmetric) gets w_ij
// computed here by the same expression.
template <int DIM, int ROWS>
__global__ void __launch_bounds__(PAIR_THREADS) k_material_w_mirror(int64_t n, const int64_t* __restrict__ rp,
                                                                    const int32_t* __restrict__ ci,
                                                                    const double* __restrict__ x,
                                                                    const double* __restrict__ sinv, double* w,
                                                                    const uint8_t* __restrict__ unsorted) {
  if (unsorted && unsorted[blockIdx.x]) return;
  __shared__ int64_t start[ROWS];
  __shared__ int off[ROWS + 1];
  const int64_t r0 = (int64_t)blockIdx.x * ROWS;
  pair_offsets<false, ROWS>(n, rp, ci, r0, start, off, w);
  const int tot = off[ROWS];
  for (int q = (int)threadIdx.x; q < tot; q += PAIR_THREADS) {
    const int r = pair_row<ROWS>(off, q);
    const int k = q - off[r];
    const int64_t p = start[r] + k, i = r0 + r;
    const int32_t j = ci[p];
    int64_t lo = rp[j], hi = rp[j + 1] - 1, f = hi - k;
    if (f < lo || ci[f] != (int32_t)i) {
      f = -1;
      while (lo <= hi) {
        const int64_t mid = (lo + hi) >> 1;
        const int32_t c = ci[mid];
        if (c == (int32_t)i) { f = mid; break; }
        if (c < (int32_t)i) lo = mid + 1; else hi = mid - 1;
      }
    }
    w[p] = f >= 0 ? w[f] : pair_weight<DIM>(x, sinv, i, j);
  }
}

// D_i = sum of the row's w in ascending column order (thread per row, so the
// sequential FP64 additions of 32 rows share one warp instruction).  The
// diagonal's w is +0, and adding +0 to a non-negative sum leaves it unchanged,
// so this equals the sum over the off-diagonal entries only.
__global__ void k_row_sum_ordered(int64_t n, const int64_t* __restrict__ rp, const double* __restrict__ w,
                                  double* __restrict__ D) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double acc = 0.0;
  const int64_t e = rp[i + 1];
  int64_t p = rp[i];
  // eight loads in flight per round (long coarse-level rows are otherwise a
  // chain of dependent load rounds); still added one by one in column order
  for (; p + 8 <= e; p += 8) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = w[p + u];
#pragma unroll
    for (int u = 0; u < 8; ++u) acc += v[u];
  }
  for (; p < e; ++p) acc += w[p];
  D[i] = acc;
}

// keep_ij <=> w_ij*w_ij >= (theta*theta) * (D_i*D_j) (classical measure:
// a_ij*a_ij >= (theta*theta) * |a_ii*a_jj|), the products rounded in FP64.  Four FP64 instructions a pair bound this kernel (2.1M rows 538 us), so
// the comparison is first made on the exponents and on the leading 20 bits of
// the significands in FP32: 1 when w w is larger by more than their error, 0
// when it is smaller, -1 when neither is certain (or an operand's exponent is
// outside +-330, where an FP64 product could overflow or lose bits).
__device__ __forceinline__ int keep_sure(double w, double t2, double Di, double Dj) {
  const int hw = __double2hiint(w), ht = __double2hiint(t2), hi = __double2hiint(Di), hj = __double2hiint(Dj);
  // biased exponents (a set sign bit, zero, infinity and NaN fall outside)
  const unsigned ew = (unsigned)hw >> 20, et = (unsigned)ht >> 20, ei = (unsigned)hi >> 20, ej = (unsigned)hj >> 20;
  const unsigned lim = 660;
  if (ew - 693u > lim || et - 693u > lim || ei - 693u > lim || ej - 693u > lim) return -1;
  const float mw = __int_as_float(0x3f800000 | ((hw & 0xfffff) << 3));
  const float mt = __int_as_float(0x3f800000 | ((ht & 0xfffff) << 3));
  const float mi = __int_as_float(0x3f800000 | ((hi & 0xfffff) << 3));
  const float mj = __int_as_float(0x3f800000 | ((hj & 0xfffff) << 3));
  // w w = L 2^(2 ew - 2046), t2 Di Dj = R 2^(et + ei + ej - 3069); L < 4, R < 8,
  // each low by less than 2^-18 of itself (truncated significands, FP32 rounding)
  const int k = (int)(et + ei + ej) - 2 * (int)ew - 1023;
  if (k > 4) return 0;
  if (k < -4) return 1;
  const float L = mw * mw;
  const float R = mt * mi * mj * __int_as_float((127 + k) << 23);
  if (L > R * 1.00001f) return 1;
  if (R > L * 1.00001f) return 0;
  return -1;
}

template <bool ABS>
__device__ __forceinline__ double keep_arg(double v) {
  // (by its bits: fabs() is an FP64 instruction when its result is taken apart)
  return ABS ? __hiloint2double(__double2hiint(v) & 0x7fffffff, __double2loint(v)) : v;
}
// keep flag of entry p = (i, j), j != i
__device__ __forceinline__ int keep_entry(double wv, double t2, double Di, double Dj, bool dirichlet) {
  if (dirichlet) return 0;
  const int sure = keep_sure(wv, t2, Di, Dj);
  return sure >= 0 ? sure : ((wv * wv >= t2 * (Di * Dj)) ? 1 : 0);
}

// a3 / a4: the pointwise criterion, diagonal kept, Dirichlet nodes excluded;
// kept entries per row (diagonal included) into cnt[i+1].
// A warp takes KEEP_ROWS consecutive rows at a time, their loads together (one
// row after another was a chain of dependent loads), the entries past the 32nd of
// a row after them: four rows (1.06M rows of 26 entries 195 us, 268 a row at a
// time), or one on small levels of long rows, whose further entries then go four
// a lane together (6.6k rows of 117: 18 us a row at a time, 38 by fours, 12 so; in the
// large levels' kernel that form's registers cost 250 against 195 us).  ABS: the
// classical measure, |a_ij| and |a_ii a_jj| in place of w and D (2.1M rows of
// 26 entries: 574 us with fabs(), 487 by its bits).
template <bool ABS, int KEEP_ROWS>
__global__ void __launch_bounds__(256) k_keep(int64_t n, const int64_t* __restrict__ rp,
                                                       const int32_t* __restrict__ ci, const double* __restrict__ w,
                                                       const double* __restrict__ D, const uint8_t* __restrict__ dir,
                                                       double t2, uint8_t* __restrict__ keep,
                                                       int64_t* __restrict__ cnt) {
  const int lane = lane_id();
  for (int64_t i0 = global_warp() * KEEP_ROWS; i0 < n; i0 += warp_stride() * KEEP_ROWS) {
    const int64_t at = i0 + (lane <= KEEP_ROWS ? lane : KEEP_ROWS);
    const int64_t rpl = rp[at < n ? at : n];
    int64_t b[KEEP_ROWS], e[KEEP_ROWS];
    int32_t j[KEEP_ROWS];
    double wv[KEEP_ROWS], Di[KEEP_ROWS], Dj[KEEP_ROWS];
    bool dd[KEEP_ROWS];
    int kept[KEEP_ROWS];
#pragma unroll
    for (int u = 0; u < KEEP_ROWS; ++u) {
      b[u] = __shfl_sync(FULL, rpl, u);
      e[u] = __shfl_sync(FULL, rpl, u + 1);
      const bool in = b[u] + lane < e[u];
      j[u] = in ? ci[b[u] + lane] : -1;
      wv[u] = in ? keep_arg<ABS>(w[b[u] + lane]) : 0.0;
      const int64_t i = i0 + u < n ? i0 + u : n - 1;
      Di[u] = keep_arg<ABS>(D[i]);
      dd[u] = dir && dir[i];
    }
#pragma unroll
    for (int u = 0; u < KEEP_ROWS; ++u) {
      Dj[u] = j[u] >= 0 ? keep_arg<ABS>(D[j[u]]) : 0.0;
      if (dir && j[u] >= 0) dd[u] |= dir[j[u]] != 0;
    }
#pragma unroll
    for (int u = 0; u < KEEP_ROWS; ++u) {
      int k = 0;
      if (j[u] >= 0) {
        k = j[u] == (int32_t)(i0 + u) ? 1 : keep_entry(wv[u], t2, Di[u], Dj[u], dd[u]);
        keep[b[u] + lane] = (uint8_t)k;
      }
      kept[u] = __popc(__ballot_sync(FULL, k != 0));
    }
#pragma unroll
    for (int u = 0; u < KEEP_ROWS; ++u) {
      if (e[u] - b[u] > 32) {  // warp-uniform
        const int64_t i = i0 + u;
        const bool diri = dir && dir[i];
        int c = 0;
        if constexpr (KEEP_ROWS == 1) {
          // four entries a lane, their loads together
          for (int64_t p = b[u] + 32 + lane; p < e[u]; p += 128) {
            int32_t jj[4];
            double wt[4], Dt[4];
            bool dt[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const bool in = p + 32 * v < e[u];
              jj[v] = in ? ci[p + 32 * v] : -1;
              wt[v] = in ? keep_arg<ABS>(w[p + 32 * v]) : 0.0;
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              Dt[v] = jj[v] >= 0 ? keep_arg<ABS>(D[jj[v]]) : 0.0;
              dt[v] = diri || (dir && jj[v] >= 0 && dir[jj[v]]);
            }
#pragma unroll
            for (int v = 0; v < 4; ++v)
              if (jj[v] >= 0) {
                const int k = jj[v] == (int32_t)i ? 1 : keep_entry(wt[v], t2, Di[u], Dt[v], dt[v]);
                keep[p + 32 * v] = (uint8_t)k;
                c += k;
              }
          }
        } else {
          for (int64_t p = b[u] + 32 + lane; p < e[u]; p += 32) {
            const int32_t jj = ci[p];
            const int k = jj == (int32_t)i ? 1 : keep_entry(keep_arg<ABS>(w[p]), t2, Di[u], keep_arg<ABS>(D[jj]),
                                                             diri || (dir && dir[jj]));
            keep[p] = (uint8_t)k;
            c += k;
          }
        }
        kept[u] += __reduce_add_sync(FULL, c);
      }
      if (lane == 0 && cnt && i0 + u < n) cnt[i0 + u + 1] = kept[u];
    }
  }
}

// ---------------------------------------------------------------------------
// Cut-drop criterion (Sec. 2.1, Eq. C^cut-drop) on squared strengths:
// classical s2 = a_ij^2 / |a_ii a_jj|, material s2 = w_ij^2 / (D_i D_j).
// Per row the off-diagonal strengths are ordered descending; the first k with
// theta^2 s2_k >= s2_{k+1} gives the threshold s2_k (no such k: keep all);
// an edge survives when both of its rows keep it.
// ---------------------------------------------------------------------------
__global__ void k_s2_classical(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                               const double* __restrict__ v, const double* __restrict__ diag,
                               double* __restrict__ s2) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double di = diag[i];
  for (int64_t p = rp[i]; p < rp[i + 1]; ++p) {
    int32_t j = ci[p];
    s2[p] = (j == (int32_t)i) ? 0.0 : (v[p] * v[p]) / fabs(di * diag[j]);
  }
}

__global__ void k_s2_material(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                              const double* __restrict__ w, const double* __restrict__ D, double* __restrict__ s2) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double Di = D[i];
  for (int64_t p = rp[i]; p < rp[i + 1]; ++p) {
    int32_t j = ci[p];
    s2[p] = (j == (int32_t)i) ? 0.0 : (w[p] * w[p]) / (Di * D[j]);
  }
}

constexpr int CUT_CAP = 256;   // row entries sorted in shared memory
constexpr int CUT_WARPS = 4;

// serial threshold for rows longer than CUT_CAP: walk the distinct values in
// descending order (ties form pairs of equal neighbours in the ordering)
__device__ double cut_threshold_serial(const int64_t b, const int64_t e, const int32_t* __restrict__ ci, int64_t i,
                                       const uint8_t* __restrict__ dir, const double* __restrict__ s2, double t2) {
  const bool diri = dir && dir[i];
  double cur = INFINITY, last = 0.0;
  bool any = false;
  for (;;) {
    double nxt = -1.0;
    int mult = 0;
    for (int64_t p = b; p < e; ++p) {
      int32_t j = ci[p];
      if (j == (int32_t)i || diri || (dir && dir[j])) continue;
      double x = s2[p];
      if (x < cur) {
        if (x > nxt) { nxt = x; mult = 1; }
        else if (x == nxt) ++mult;
      }
    }
    if (nxt < 0.0) return any ? last : 0.0;  // values exhausted: no gap, keep all
    if (any && t2 * last >= nxt) return last;
    if (mult >= 2 && t2 * nxt >= nxt) return nxt;
    any = true;
    last = nxt;
    cur = nxt;
  }
}

__global__ void __launch_bounds__(CUT_WARPS * 32)
k_cut_rows(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
           const uint8_t* __restrict__ dir, const double* __restrict__ s2, double t2,
           uint8_t* __restrict__ rowkeep) {
  __shared__ double vals_all[CUT_WARPS][CUT_CAP];
  __shared__ double srt_all[CUT_WARPS][CUT_CAP];
  const int w = threadIdx.x >> 5, lane = lane_id();
  const unsigned lt = (1u << lane) - 1u;
  double* vals = vals_all[w];
  double* srt = srt_all[w];
  for (int64_t i = global_warp(); i < n; i += warp_stride()) {
    const int64_t b = rp[i], e = rp[i + 1];
    const bool diri = dir && dir[i];
    // collect the row's valid strengths in column order
    int m = 0;
    for (int64_t p0 = b; p0 < e; p0 += 32) {
      int64_t p = p0 + lane;
      bool ok = false;
      double x = 0.0;
      if (p < e) {
        int32_t j = ci[p];
        ok = j != (int32_t)i && !diri && !(dir && dir[j]);
        x = s2[p];
      }
      unsigned bm = __ballot_sync(FULL, ok);
      if (ok && m + __popc(bm & lt) < CUT_CAP) vals[m + __popc(bm & lt)] = x;
      m += __popc(bm);
    }
    __syncwarp();
    double thr = 0.0;
    if (m > CUT_CAP) {
      if (lane == 0) thr = cut_threshold_serial(b, e, ci, i, dir, s2, t2);
      thr = __shfl_sync(FULL, thr, 0);
    } else if (m > 0) {
      // rank sort, descending (ties by position)
      for (int t = lane; t < m; t += 32) {
        const double x = vals[t];
        int r = 0;
        for (int u = 0; u < m; ++u) r += (vals[u] > x) || (vals[u] == x && u < t);
        srt[r] = x;
      }
      __syncwarp();
      thr = srt[m - 1];
      for (int k0 = 0; k0 < m - 1; k0 += 32) {
        const int k = k0 + lane;
        const bool gap = k < m - 1 && t2 * srt[k] >= srt[k + 1];
        const unsigned gm = __ballot_sync(FULL, gap);
        if (gm) {
          thr = srt[k0 + __ffs(gm) - 1];
          break;
        }
      }
    }
    for (int64_t p = b + lane; p < e; p += 32) {
      int32_t j = ci[p];
      bool ok = j != (int32_t)i && !diri && !(dir && dir[j]);
      rowkeep[p] = (ok && m > 0 && s2[p] >= thr) ? 1 : 0;
    }
    __syncwarp();
  }
}

// keep = diagonal, or kept by both rows; counts kept entries into cnt[i+1]
__global__ void k_cut_symmetrize(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                 const uint8_t* __restrict__ rowkeep, uint8_t* __restrict__ keep,
                                 int64_t* __restrict__ cnt) {
  const int lane = lane_id();
  for (int64_t i = global_warp(); i < n; i += warp_stride()) {
    int kept = 0;
    for (int64_t p = rp[i] + lane; p < rp[i + 1]; p += 32) {
      int32_t j = ci[p];
      uint8_t k;
      if (j == (int32_t)i) k = 1;
      else if (!rowkeep[p]) k = 0;
      else {
        int64_t lo = rp[j], hi = rp[j + 1] - 1, f = -1;
        while (lo <= hi) {
          int64_t mid = (lo + hi) >> 1;
          int32_t c = ci[mid];
          if (c == (int32_t)i) { f = mid; break; }
          if (c < (int32_t)i) lo = mid + 1; else hi = mid - 1;
        }
        k = (f >= 0 && rowkeep[f]) ? 1 : 0;
      }
      keep[p] = k;
      kept += k;
    }
    for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(FULL, kept, o);
    if (lane == 0) cnt[i + 1] = kept;
  }
}

// ---------------------------------------------------------------------------
// a10. filtered matrix A_F and 1-norm diagonal (Sec. 2.2, Eqs.
// filtered_matrix and 1_norm_diagonal).  rpF is the scan of
// the kept counts.  A row whose filtered 1-norm is <= 1e-12 times the 1-norm
// of its row of A (every off-diagonal dropped, lumped row sum ~ 0) gets
// Dt = +inf: it is not smoothed.
// ---------------------------------------------------------------------------
// Thread per row: the three ordered sums are sequential FP64 chains, so one
// warp instruction advances 32 rows.  The block's rows are one segment of the
// CSR arrays, copied to shared memory first: three passes over rows 216 bytes
// apart cost each warp load 32 lines of a cache that 64 warps shared (2.1M rows of
// 27 entries: 785 us, 480 us staged).  Levels of longer rows, and short ones of
// coarse 3D rows, read in place (109k rows of 59 entries: 117 us; staged, with
// most blocks above the buffer, 377).  Rows of up to 12 entries on average take a
// third of the buffer, for residency (160k rows of 9: 22.9 us in the larger one, 18.8).  A block above
// its buffer reads in place too, by a copy of the row loop whose pointers stay
// global and read-only.
constexpr int FILT_ROWS = 64;
constexpr int FILT_CAP = 2048, FILT_CAP_SHORT = 768;
constexpr int64_t FILT_MEAN = 27, FILT_SMALL = 4096;

// row i, entries [b, e) of V, C, K
template <typename I>
__device__ __forceinline__ void filter_row(int64_t i, I b, I e, const double* __restrict__ V,
                                           const int32_t* __restrict__ C, const uint8_t* __restrict__ K,
                                           const int64_t* __restrict__ rpF, int32_t* __restrict__ ciF,
                                           double* __restrict__ vF, double* __restrict__ Dt) {
  // lumped diagonal: a_ii, then the dropped entries in ascending order
  double dg = 0.0;
  for (I p = b; p < e; ++p)
    if (C[p] == (int32_t)i) dg = V[p];
  for (I p = b; p < e; ++p)
    if (C[p] != (int32_t)i && !K[p]) dg += V[p];
  // the filtered row and both 1-norms in ascending order
  int64_t out = rpF[i];
  double s = 0.0, a1 = 0.0;
  for (I p = b; p < e; ++p) {
    const int32_t j = C[p];
    const double a = V[p];
    a1 += fabs(a);
    if (j == (int32_t)i || K[p]) {
      const double fv = (j == (int32_t)i) ? dg : a;
      ciF[out] = j;
      vF[out] = fv;
      ++out;
      s += fabs(fv);
    }
  }
  Dt[i] = (s <= 1e-12 * a1) ? INFINITY : s;
}

template <int CAP>
__global__ void __launch_bounds__(FILT_ROWS) k_filter(int64_t n, const int64_t* __restrict__ rp,
                                                      const int32_t* __restrict__ ci, const double* __restrict__ v,
                                                      const uint8_t* __restrict__ keep,
                                                      const int64_t* __restrict__ rpF, int32_t* __restrict__ ciF,
                                                      double* __restrict__ vF, double* __restrict__ Dt) {
  const int64_t i0 = (int64_t)blockIdx.x * FILT_ROWS, i1 = i0 + FILT_ROWS < n ? i0 + FILT_ROWS : n;
  const int64_t i = i0 + threadIdx.x;
  if constexpr (CAP > 0) {
    __shared__ double s_v[CAP];
    __shared__ int32_t s_c[CAP];
    __shared__ uint8_t s_k[CAP];
    const int64_t b0 = rp[i0], tot = rp[i1] - b0;
    if (tot <= CAP) {
      for (int p = (int)threadIdx.x; p < (int)tot; p += FILT_ROWS) {
        s_v[p] = v[b0 + p];
        s_c[p] = ci[b0 + p];
        s_k[p] = keep[b0 + p];
      }
      __syncthreads();
      if (i < n) filter_row<int>(i, (int)(rp[i] - b0), (int)(rp[i + 1] - b0), s_v, s_c, s_k, rpF, ciF, vF, Dt);
      return;
    }
  }
  if (i < n) filter_row<int64_t>(i, rp[i], rp[i + 1], v, ci, keep, rpF, ciF, vF, Dt);
}

// ---------------------------------------------------------------------------
// a9. coarse coordinates and tensors (Sec. 3, Eq. auxiliary_transfer):
// means over the aggregate members, summed in ascending fine index (mlist is
// sorted per aggregate); the coarse inverse tensors follow by inversion.
// ---------------------------------------------------------------------------
__global__ void k_coarse_aux(int64_t nc, int dim, const int64_t* __restrict__ mrp, const int32_t* __restrict__ mlist,
                             const double* __restrict__ x, const double* __restrict__ sigma,
                             double* __restrict__ xc, double* __restrict__ sc, double* __restrict__ sic) {
  int64_t a = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= nc) return;
  const int kp = dim == 3 ? 6 : 3;
  double sx[3] = {0.0, 0.0, 0.0}, ss[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  double cnt = 0.0;
  for (int64_t p = mrp[a]; p < mrp[a + 1]; ++p) {
    int64_t i = mlist[p];
    for (int c = 0; c < dim; ++c) sx[c] += x[i * dim + c];
    for (int c = 0; c < kp; ++c) ss[c] += sigma[i * kp + c];
    cnt += 1.0;
  }
  for (int c = 0; c < dim; ++c) xc[a * dim + c] = sx[c] / cnt;
  double s[6];
  for (int c = 0; c < kp; ++c) {
    s[c] = ss[c] / cnt;
    sc[a * kp + c] = s[c];
  }
  double si[6];
  invert_packed(dim, s, si);
  for (int c = 0; c < kp; ++c) sic[a * kp + c] = si[c];
}

// ---------------------------------------------------------------------------
// a12. smoothed prolongator values from T = A_F P^ (Sec. 2.2):
//   c_i = omega / Dt_i,  P_ij = [j == agg(i)] - c_i * T_ij
// P shares the pattern of T.  omega is read from device memory.
// ---------------------------------------------------------------------------
__global__ void k_smooth_p_values(int64_t n, const int64_t* __restrict__ rpT, const int32_t* __restrict__ ciT,
                                  const double* __restrict__ vT, const int32_t* __restrict__ agg,
                                  const double* __restrict__ Dt, const double* __restrict__ omega_p,
                                  double* __restrict__ vP) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double omega = *omega_p;
  const double c = omega / Dt[i];
  const int32_t ai = agg[i];
  for (int64_t p = rpT[i]; p < rpT[i + 1]; ++p) {
    double t = vT[p];
    vP[p] = (ciT[p] == ai) ? 1.0 - c * t : -(c * t);
  }
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
int launch_dirichlet_diag(cudaStream_t s, int64_t n, const int64_t* rp, const int32_t* ci, const double* v,
                          uint8_t* dir, double* diag, int* err) {
  if (n <= 0) return SA_OK;
  k_dirichlet_diag<<<warp_rows_grid(n), 256, 0, s>>>(n, rp, ci, v, dir, diag, err);
  SA_LAUNCHED();
  return SA_OK;
}

int64_t strength_blocks(int64_t n, int64_t nnz) { return (int64_t)blocks_for(n, few_long_rows(n, nnz) ? 8 : 64); }

int launch_validate_csr(cudaStream_t s, int64_t n, int64_t ncols, int64_t nnz, const int64_t* rp, const int32_t* ci,
                        int* err) {
  if (n <= 0) return SA_OK;
  k_validate_csr<<<blocks_for(n, 256), 256, 0, s>>>(n, ncols, nnz, rp, ci, err);
  SA_LAUNCHED();
  return SA_OK;
}

int launch_nodal_tensors(Alloc& al, int dim, int64_t n, int tloc, const double* tensors, int64_t ne, int npe,
                         const int32_t* en, const double* meas, double* sigma, double* sinv, int* err) {
  cudaStream_t s = al.stream;
  if (tloc == 1) {
    Buf<int64_t> off;
    Buf<int> cursor;
    Buf<int32_t> list;
    SA_TRY(off.alloc(&al, n + 1));
    SA_TRY(cursor.alloc(&al, n));
    SA_TRY(list.alloc(&al, ne * npe));
    SA_TRY(memset_d(off.p, 0, off.bytes(), s));
    SA_TRY(memset_d(cursor.p, 0, cursor.bytes(), s));
    k_node_elem_count<<<blocks_for(ne * npe, 256), 256, 0, s>>>(ne, npe, en, n, off.p, err);
    SA_LAUNCHED();
    SA_TRY(scan_inplace(al, off.p + 1, n));
    k_node_elem_fill<<<blocks_for(ne * npe, 256), 256, 0, s>>>(ne, npe, en, n, off.p, cursor.p, list.p);
    SA_LAUNCHED();
    k_node_tensor_from_elems<<<blocks_for(n, 128), 128, 0, s>>>(n, dim, off.p, list.p, meas, tensors, sigma, sinv,
                                                               err);
    SA_LAUNCHED();
  } else {
    k_node_tensor_direct<<<blocks_for(n, 256), 256, 0, s>>>(n, dim, tensors, sigma, sinv);
    SA_LAUNCHED();
  }
  return SA_OK;
}

template <bool ABS>
static int launch_keep(cudaStream_t s, int64_t n, int64_t nnz, const int64_t* rp, const int32_t* ci, const double* w,
                       const double* D, const uint8_t* dir, double t2, uint8_t* keep, int64_t* cnt) {
  if (few_long_rows(n, nnz)) k_keep<ABS, 1><<<warp_rows_grid(n), 256, 0, s>>>(n, rp, ci, w, D, dir, t2, keep, cnt);
  else k_keep<ABS, 4><<<warp_rows_grid((n + 3) / 4), 256, 0, s>>>(n, rp, ci, w, D, dir, t2, keep, cnt);
  SA_LAUNCHED();
  return SA_OK;
}

int launch_strength_classical(cudaStream_t s, int64_t n, int64_t nnz, const int64_t* rp, const int32_t* ci, const double* v,
                              const double* diag, const uint8_t* dir, double theta, uint8_t* keep,
                              int64_t* cnt) {
  if (n <= 0) return SA_OK;
  const double t2 = theta * theta;
  return launch_keep<true>(s, n, nnz, rp, ci, v, diag, dir, t2, keep, cnt);
}

template <int DIM, int ROWS>
static int launch_pairs_rows(cudaStream_t s, int64_t n, const int64_t* rp, const int32_t* ci, const double* x,
                             const double* sinv, double* w, uint8_t* unsorted) {
  const unsigned g = blocks_for(n, ROWS);
  if (unsorted) k_material_w<DIM, true, ROWS><<<g, PAIR_THREADS, 0, s>>>(n, rp, ci, x, sinv, w, unsorted);
  else k_material_w<DIM, false, ROWS><<<g, PAIR_THREADS, 0, s>>>(n, rp, ci, x, sinv, w, nullptr);
  SA_LAUNCHED();
  k_material_w_mirror<DIM, ROWS><<<g, PAIR_THREADS, 0, s>>>(n, rp, ci, x, sinv, w, unsorted);
  SA_LAUNCHED();
  return SA_OK;
}
template <int DIM>
static int launch_pairs(cudaStream_t s, int64_t n, int64_t nnz, const int64_t* rp, const int32_t* ci, const double* x,
                        const double* sinv, double* w, uint8_t* unsorted) {
  return few_long_rows(n, nnz) ? launch_pairs_rows<DIM, 8>(s, n, rp, ci, x, sinv, w, unsorted)
                               : launch_pairs_rows<DIM, 64>(s, n, rp, ci, x, sinv, w, unsorted);
}

int launch_strength_material(cudaStream_t s, int dim, int64_t n, int64_t nnz, const int64_t* rp, const int32_t* ci,
                             const double* x, const double* sinv, const uint8_t* dir, double theta,
                             double* w, double* D, uint8_t* keep, int64_t* cnt, uint8_t* unsorted) {
  if (n <= 0) return SA_OK;
  const double t2 = theta * theta;
  if (dim == 3) SA_TRY(launch_pairs<3>(s, n, nnz, rp, ci, x, sinv, w, unsorted));
  else SA_TRY(launch_pairs<2>(s, n, nnz, rp, ci, x, sinv, w, unsorted));
  k_row_sum_ordered<<<blocks_for(n, 128), 128, 0, s>>>(n, rp, w, D);
  SA_LAUNCHED();
  return launch_keep<false>(s, n, nnz, rp, ci, w, D, dir, t2, keep, cnt);
}

int launch_cut_drop(Alloc& al, int measure_classical, int64_t n, int64_t nnz, const int64_t* rp, const int32_t* ci,
                    const double* v, const double* diag, const double* w, const double* D, const uint8_t* dir,
                    double theta, uint8_t* keep, int64_t* cnt) {
  cudaStream_t s = al.stream;
  if (n <= 0) return SA_OK;
  Buf<double> s2;
  Buf<uint8_t> rowkeep;
  SA_TRY(s2.alloc(&al, nnz));
  SA_TRY(rowkeep.alloc(&al, nnz));
  if (measure_classical) k_s2_classical<<<blocks_for(n, 128), 128, 0, s>>>(n, rp, ci, v, diag, s2.p);
  else k_s2_material<<<blocks_for(n, 128), 128, 0, s>>>(n, rp, ci, w, D, s2.p);
  SA_LAUNCHED();
  const double t2 = theta * theta;
  k_cut_rows<<<warp_rows_grid(n, CUT_WARPS * 32), CUT_WARPS * 32, 0, s>>>(n, rp, ci, dir, s2.p, t2, rowkeep.p);
  SA_LAUNCHED();
  k_cut_symmetrize<<<warp_rows_grid(n), 256, 0, s>>>(n, rp, ci, rowkeep.p, keep, cnt);
  SA_LAUNCHED();
  return SA_OK;
}

int launch_filter(cudaStream_t s, int64_t n, int64_t nnz, const int64_t* rp, const int32_t* ci, const double* v,
                  const uint8_t* keep, const int64_t* rpF, int32_t* ciF, double* vF, double* Dt) {
  if (n <= 0) return SA_OK;
  const unsigned g = blocks_for(n, FILT_ROWS);
  if (nnz <= n * (FILT_CAP_SHORT / FILT_ROWS))
    k_filter<FILT_CAP_SHORT><<<g, FILT_ROWS, 0, s>>>(n, rp, ci, v, keep, rpF, ciF, vF, Dt);
  else if (nnz <= n * FILT_MEAN && n >= FILT_SMALL)
    k_filter<FILT_CAP><<<g, FILT_ROWS, 0, s>>>(n, rp, ci, v, keep, rpF, ciF, vF, Dt);
  else
    k_filter<0><<<g, FILT_ROWS, 0, s>>>(n, rp, ci, v, keep, rpF, ciF, vF, Dt);
  SA_LAUNCHED();
  return SA_OK;
}

int launch_coarse_aux(cudaStream_t s, int64_t nc, int dim, const int64_t* mrp, const int32_t* mlist,
                      const double* x, const double* sigma, double* xc, double* sc, double* sic) {
  if (nc <= 0) return SA_OK;
  k_coarse_aux<<<blocks_for(nc, 128), 128, 0, s>>>(nc, dim, mrp, mlist, x, sigma, xc, sc, sic);
  SA_LAUNCHED();
  return SA_OK;
}

int launch_smooth_p_values(cudaStream_t s, int64_t n, const int64_t* rpT, const int32_t* ciT, const double* vT,
                           const int32_t* agg, const double* Dt, const double* omega_dev, double* vP) {
  if (n <= 0) return SA_OK;
  k_smooth_p_values<<<blocks_for(n, 256), 256, 0, s>>>(n, rpT, ciT, vT, agg, Dt, omega_dev, vP);
  SA_LAUNCHED();
  return SA_OK;
}

}  // namespace sa
