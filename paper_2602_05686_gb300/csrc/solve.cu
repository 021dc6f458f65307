// Iteration kernels: the power method on CSR matrices (sub-warp per row),
// fixed-order dot products, and the CG vector updates with device-resident
// scalars.  The V-cycle itself lives in vcycle.cu.
#include <math.h>

#include <functional>

#include "common.cuh"
#include "kernels.cuh"
#include "reduce.cuh"
#include "solve.cuh"

namespace sa {

// ---------------------------------------------------------------------------
// CSR row products with SW lanes per row (power method on the setup's CSR
// matrices); the result is valid in every lane of the group
// ---------------------------------------------------------------------------
#define ROW_SETUP(SW)                                                   \
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   \
  const int64_t i = gt / SW;                                            \
  const int sl = (int)(gt % SW);                                        \
  const bool valid = i < n;

// power method: y_j = s_j v_j with v_j = X_j * sc[4] (the previous product
// times the reciprocal of its norm; 1 for the start vector), formed once per
// step so that the product below costs one FP64 FMA per stored entry
__global__ void k_power_prep(int64_t n, const double* X, const double* __restrict__ s,
                             const double* sc, double* __restrict__ y) {
  pdl_sync();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = s ? s[i] * (X[i] * sc[4]) : X[i] * sc[4];  // s NULL: a pre-scaled operator
}

// w_i = s_i * sum_p a_p y_j
template <int SW>
__global__ void k_power_spmv(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                             const double* __restrict__ v, const double* __restrict__ s, const double* y,
                             double* __restrict__ w) {
  pdl_sync();
  ROW_SETUP(SW)
  double acc = 0.0;
  if (valid) {
    const int64_t e = rp[i + 1];
    for (int64_t p = rp[i] + sl; p < e; p += SW) acc += v[p] * y[ci[p]];
  }
#pragma unroll
  for (int o = SW / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o, SW);
  if (valid && sl == 0) w[i] = s[i] * acc;
}

// ---------------------------------------------------------------------------
// fixed-order block reductions
// ---------------------------------------------------------------------------
template <int NV>
__device__ __forceinline__ void block_sum_to(double (&val)[NV], double* __restrict__ out, int stride) {
  __shared__ double sh[NV][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    double t = warp_sum(val[k]);
    if (lane == 0) sh[k][w] = t;
  }
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double t = lane < nw ? sh[k][lane] : 0.0;
      t = warp_sum(t);
      if (lane == 0) out[(int64_t)k * stride + blockIdx.x] = t;
    }
  }
}

// one or two dot products over a fixed grid, finished by the last block
template <int NV>
__global__ void __launch_bounds__(RED_THREADS) k_dots(int64_t n, const double* a0,
                                                      const double* b0, const double* a1,
                                                      const double* b1, double* __restrict__ part,
                                                      Fin fin) {
  pdl_sync();
  double acc[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) acc[v] = 0.0;
  // two grid-stride elements per trip, their loads issued together and
  // added in the grid-stride order (the sums do not depend on the unroll)
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 2 * st) {
    const int64_t j = i + st;
    const bool two = j < n;
    const double u0 = a0[i], v0 = b0[i], u1 = two ? a0[j] : 0.0, v1 = two ? b0[j] : 0.0;
    acc[0] = fma(u0, v0, acc[0]);
    if (two) acc[0] = fma(u1, v1, acc[0]);
    if constexpr (NV > 1) {
      const double e0 = a1[i], f0 = b1[i], e1 = two ? a1[j] : 0.0, f1 = two ? b1[j] : 0.0;
      acc[1] = fma(e0, f0, acc[1]);
      if (two) acc[1] = fma(e1, f1, acc[1]);
    }
  }
  block_sum_to<NV>(acc, part, RED_BLOCKS);
  fin_inline<NV, RED_THREADS, NV - 1>(fin, part, (int)gridDim.x, RED_BLOCKS);
}

// ---------------------------------------------------------------------------
// power method (Sec. 2.2): spectral-radius estimate of diag(s) A diag(s)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t fmix32_s(uint32_t h) {
  // MurmurHash3 32-bit finaliser (Appleby, public domain)
  h ^= h >> 16;
  h *= 0x85ebca6bu;
  h ^= h >> 13;
  h *= 0xc2b2ae35u;
  h ^= h >> 16;
  return h;
}

__global__ void k_start_vector(int64_t n, uint32_t tag, uint32_t seed, double* __restrict__ v) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    uint32_t h = fmix32_s((uint32_t)i ^ (0x7F4A7C15u * tag) ^ (seed * 0x2545F491u));
    double u = (double)h * (1.0 / 4294967296.0);
    v[i] = 2.0 * u - 1.0;
  }
}

// w.w and v.v with v_j = X_j * sc[4]; the last block takes the estimate and
// the next scale from them (FIN_POWER)
__global__ void __launch_bounds__(RED_THREADS) k_power_dots(int64_t n, const double* w,
                                                            const double* X, const double* sc,
                                                            double* __restrict__ part, Fin fin) {
  pdl_sync();
  const double inv = sc[4];
  double acc[2] = {0.0, 0.0};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double vi = X[i] * inv;
    acc[0] += w[i] * w[i];
    acc[1] += vi * vi;
  }
  block_sum_to<2>(acc, part, RED_BLOCKS);
  fin_inline<2, RED_THREADS, 1>(fin, part, (int)gridDim.x, RED_BLOCKS);
}

__global__ void k_rsqrt_scale(int64_t n, const double* __restrict__ d, double* __restrict__ out) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = 1.0 / sqrt(d[i]);  // +inf -> 0
}

__global__ void k_reciprocal(int64_t n, const double* __restrict__ d, double* __restrict__ out) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = 1.0 / d[i];
}

__global__ void k_omega(const double* __restrict__ lam, double omega_sym, double* __restrict__ omega) {
  *omega = *lam > 0.0 ? omega_sym / *lam : 0.0;
}

int pick_sw(int64_t n, int64_t nnz) {
  double avg = n > 0 ? (double)nnz / (double)n : 1.0;
  if (avg <= 6) return 4;
  if (avg <= 40) return 8;
  if (avg <= 96) return 16;
  return 32;
}

#define DISPATCH_SW(sw, KERNEL, GRIDN, ...)                                                 \
  do {                                                                                       \
    const int _sw = (sw);                                                                    \
    const unsigned _g = blocks_for((GRIDN) * (int64_t)_sw, 256);                             \
    switch (_sw) {                                                                           \
      case 4: launch_pdl(KERNEL<4>, _g, 256, 0, st, __VA_ARGS__); break;                             \
      case 8: launch_pdl(KERNEL<8>, _g, 256, 0, st, __VA_ARGS__); break;                             \
      case 16: launch_pdl(KERNEL<16>, _g, 256, 0, st, __VA_ARGS__); break;                           \
      default: launch_pdl(KERNEL<32>, _g, 256, 0, st, __VA_ARGS__); break;                           \
    }                                                                                        \
  } while (0)

int launch_dots(cudaStream_t st, int64_t n, const double* a0, const double* b0, const double* a1,
                const double* b1, double* part, const Fin& fin) {
  if (fin.op == FIN_BETA && fin.flexible > 0 && !a1) return SA_ERR_INVALID_ARG;  // needs the second dot
  const unsigned g = red_blocks(n);
  if (a1) launch_pdl(k_dots<2>, g, RED_THREADS, 0, st, n, a0, b0, a1, b1, part, fin);
  else launch_pdl(k_dots<1>, g, RED_THREADS, 0, st, n, a0, b0, nullptr, nullptr, part, fin);
  SA_LAUNCHED();
  return SA_OK;
}

int run_power(Alloc& al, int64_t n, int64_t nnz, const int64_t* rp, const int32_t* ci, const double* v, const double* s,
              int steps, uint32_t tag, uint32_t seed, double* lam_dev) {
  cudaStream_t st = al.stream;
  if (n <= 0) return SA_OK;
  Buf<double> x, w, y, part, sc;
  SA_TRY(x.alloc(&al, n));
  SA_TRY(w.alloc(&al, n));
  SA_TRY(y.alloc(&al, n));
  SA_TRY(part.alloc(&al, 2 * RED_BLOCKS));
  SA_TRY(sc.alloc(&al, 6));  // scalars, ticket of the finishing block
  const double init[6] = {0.0, 0.0, 1.0, 0.0, 1.0, 0.0};
  SA_CUDA(cudaMemcpyAsync(sc.p, init, sizeof(init), cudaMemcpyHostToDevice, st));
  Fin fin;
  fin.op = FIN_POWER;
  fin.tick = reinterpret_cast<unsigned*>(sc.p + 5);
  fin.sc = sc.p;
  fin.lam = lam_dev;
  const double avg = (double)nnz / (double)n;
  const int sw = avg <= 40.0 ? 4 : (avg <= 96.0 ? 8 : 16);
  k_start_vector<<<blocks_for(n, 256), 256, 0, st>>>(n, tag, seed, x.p);
  SA_LAUNCHED();
  double* X = x.p;  // previous product (the start vector at first)
  double* W = w.p;
  for (int it = 0; it < steps; ++it) {
    launch_pdl(k_power_prep, blocks_for(n, 256), 256, 0, st, n, X, s, sc.p, y.p);
    SA_LAUNCHED();
    DISPATCH_SW(sw, k_power_spmv, n, n, rp, ci, v, s, y.p, W);
    SA_LAUNCHED();
    launch_pdl(k_power_dots, red_blocks(n), RED_THREADS, 0, st, n, W, X, sc.p, part.p, fin);
    SA_LAUNCHED();
    double* t = X; X = W; W = t;
  }
  return SA_OK;
}

int run_power_op(Alloc& al, int64_t n, int steps, uint32_t tag, uint32_t seed, double* lam_dev,
                 const std::function<int(const double*, double*)>& apply) {
  cudaStream_t st = al.stream;
  if (n <= 0) return SA_OK;
  Buf<double> x, w, y, part, sc;
  SA_TRY(x.alloc(&al, n));
  SA_TRY(w.alloc(&al, n));
  SA_TRY(y.alloc(&al, n));
  SA_TRY(part.alloc(&al, 2 * RED_BLOCKS));
  SA_TRY(sc.alloc(&al, 6));  // scalars, ticket of the finishing block
  const double init[6] = {0.0, 0.0, 1.0, 0.0, 1.0, 0.0};
  SA_CUDA(cudaMemcpyAsync(sc.p, init, sizeof(init), cudaMemcpyHostToDevice, st));
  Fin fin;
  fin.op = FIN_POWER;
  fin.tick = reinterpret_cast<unsigned*>(sc.p + 5);
  fin.sc = sc.p;
  fin.lam = lam_dev;
  // (these two launches also stand between the kernels that built the operator
  // and its first product, which reads it before its wait)
  k_start_vector<<<blocks_for(n, 256), 256, 0, st>>>(n, tag, seed, x.p);
  SA_LAUNCHED();
  double* X = x.p;
  double* W = w.p;
  for (int it = 0; it < steps; ++it) {
    launch_pdl(k_power_prep, blocks_for(n, 256), 256, 0, st, n, X, nullptr, sc.p, y.p);
    SA_LAUNCHED();
    SA_TRY(apply(y.p, W));
    launch_pdl(k_power_dots, red_blocks(n), RED_THREADS, 0, st, n, W, X, sc.p, part.p, fin);
    SA_LAUNCHED();
    double* t = X; X = W; W = t;
  }
  return SA_OK;
}

int launch_rsqrt_scale(cudaStream_t s, int64_t n, const double* d, double* out) {
  if (n <= 0) return SA_OK;
  k_rsqrt_scale<<<blocks_for(n, 256), 256, 0, s>>>(n, d, out);
  SA_LAUNCHED();
  return SA_OK;
}

int launch_reciprocal(cudaStream_t s, int64_t n, const double* d, double* out) {
  if (n <= 0) return SA_OK;
  k_reciprocal<<<blocks_for(n, 256), 256, 0, s>>>(n, d, out);
  SA_LAUNCHED();
  return SA_OK;
}

int launch_omega(cudaStream_t s, const double* lam_dev, double omega_sym, double* omega_dev) {
  k_omega<<<1, 1, 0, s>>>(lam_dev, omega_sym, omega_dev);
  SA_LAUNCHED();
  return SA_OK;
}

// ---------------------------------------------------------------------------
// CG with device-resident scalars (Sec. 4)
// ---------------------------------------------------------------------------
// x += alpha p; r -= alpha q; (r_prev = r before the update, if given); r.r,
// finished by the last block
__global__ void __launch_bounds__(RED_THREADS) k_cg_update(int64_t n, const CgScalars* s, const double* p,
                                                           const double* q, double* __restrict__ x,
                                                           double* __restrict__ r, double* __restrict__ rprev,
                                                           double* __restrict__ part, Fin fin) {
  pdl_sync();
  const double alpha = s->alpha;
  double acc[1] = {0.0};
  // two grid-stride elements per trip (loads together; r.r added in the
  // grid-stride order)
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 2 * st) {
    const int64_t j = i + st;
    const bool two = j < n;
    double r0 = r[i];
    const double p0 = p[i], q0 = q[i], x0 = x[i];
    double r1 = 0.0, p1 = 0.0, q1 = 0.0, x1 = 0.0;
    if (two) {
      r1 = r[j];
      p1 = p[j];
      q1 = q[j];
      x1 = x[j];
    }
    if (rprev) {
      rprev[i] = r0;
      if (two) rprev[j] = r1;
    }
    x[i] = fma(alpha, p0, x0);
    r0 = fma(-alpha, q0, r0);
    r[i] = r0;
    acc[0] = fma(r0, r0, acc[0]);
    if (two) {
      x[j] = fma(alpha, p1, x1);
      r1 = fma(-alpha, q1, r1);
      r[j] = r1;
      acc[0] = fma(r1, r1, acc[0]);
    }
  }
  block_sum_to<1>(acc, part, 0);
  fin_inline<1, RED_THREADS, 0>(fin, part, (int)gridDim.x, 0);
}

__global__ void k_cg_pupdate(int64_t n, const CgScalars* s, const double* z,
                             double* __restrict__ p, int first) {
  pdl_sync();
  const double beta = s->beta;
  const int64_t st = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += 2 * st) {
    const int64_t j = i + st;
    const bool two = j < n;
    const double z0 = z[i], p0 = first ? 0.0 : p[i];
    const double z1 = two ? z[j] : 0.0, p1 = (two && !first) ? p[j] : 0.0;
    p[i] = first ? z0 : fma(beta, p0, z0);
    if (two) p[j] = first ? z1 : fma(beta, p1, z1);
  }
}

// the sums of np partials (k columns, or one vector with k = 0) that the
// producing launch did not finish itself
int launch_fin_wide(cudaStream_t st, const double* part, int np, const Fin& fin) {
  // as many values as the producing launch has columns
  switch (fin.k) {
    case 0: launch_pdl(k_fin_wide<1>, 32, 32, 0, st, part, np, 0, fin); break;
    case 2: launch_pdl(k_fin_wide<2>, 32, 64, 0, st, part, np, np, fin); break;
    case 4: launch_pdl(k_fin_wide<4>, 32, 128, 0, st, part, np, np, fin); break;
    case 8: launch_pdl(k_fin_wide<8>, 32, 256, 0, st, part, np, np, fin); break;
    default: return SA_ERR_INVALID_ARG;
  }
  SA_LAUNCHED();
  return SA_OK;
}

int launch_cg_update(cudaStream_t st, int64_t n, const CgScalars* s, const double* p, const double* q, double* x,
                     double* r, double* rprev, double* part, const Fin& fin) {
  launch_pdl(k_cg_update, red_blocks(n), RED_THREADS, 0, st, n, s, p, q, x, r, rprev, part, fin);
  SA_LAUNCHED();
  return SA_OK;
}

int launch_cg_pupdate(cudaStream_t st, int64_t n, const CgScalars* s, const double* z, double* p, int first) {
  launch_pdl(k_cg_pupdate, red_blocks(n), RED_THREADS, 0, st, n, s, z, p, first);
  SA_LAUNCHED();
  return SA_OK;
}


// ---------------------------------------------------------------------------
// k-column CG (k independent solves in lockstep, interleaved n x k storage).
// Every column goes through the one-vector kernels' arithmetic in the same
// order (same grid, same per-thread stride, same reduction trees), so column
// c of a block solve equals the one-vector solve of that right-hand side.
// Columns that are done (converged, broken down) are frozen by `active`.
// ---------------------------------------------------------------------------
constexpr int KB = KMAX_BLOCK;

// Rows of an interleaved n x KK block move as vectors of G = 4 columns (one
// 256-bit access; rows on 32-byte boundaries) or G = 2 (KK = 2).  A row of
// eight columns takes two lanes: a warp's access is then 1 KB of whole lines
// (a lane that took both halves of its row left every access a line of half
// used sectors, and its second half's loads behind the first half's store).
// The kernels keep the one-vector kernels' grid, per-thread stride and
// reduction trees: a warp holds the 32 rows of the one-vector kernel's 32
// threads, slot u of lane l row l / LPR + u * (32 / LPR), so that the first
// stage of the butterfly (rows 16 apart) is an addition in the lane and the
// others are shuffles.  Bound by memory; the three kernels of an iteration
// average 194 us (before: 236 us) on 160^3 rows, eight columns, FP32 form, 89 us
// (97 us) on 128^3 rows, FP64 form.  Two 512-thread blocks per SM (64 registers).
template <int KK>
struct BRow {
  static constexpr int G = KK >= 4 ? 4 : 2;
  static constexpr int LPR = KK / G;      // lanes per row
  static constexpr int RPL = 32 / LPR;    // rows of one access
};

// sums of D values per column (val[d][u][h]: slot u, column h of the lane's
// group) into out[(d * KB + c) * stride + block]; columns KK .. KB - 1 get 0
template <int KK, int D>
__device__ __forceinline__ void bblock_sum_to(double (&val)[D][BRow<KK>::LPR][BRow<KK>::G], double* __restrict__ out,
                                              int stride) {
  using B = BRow<KK>;
  __shared__ double sh[D * KMAX_BLOCK][RED_THREADS / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int d = 0; d < D; ++d)
#pragma unroll
    for (int h = 0; h < B::G; ++h) {
      double t = val[d][0][h];
      if constexpr (B::LPR == 2) t += val[d][1][h];
#pragma unroll
      for (int o = 16; o >= B::LPR; o >>= 1) t += __shfl_xor_sync(FULL, t, o);
      if (lane < B::LPR) sh[d * KMAX_BLOCK + lane * B::G + h][w] = t;
    }
  if constexpr (KK < KMAX_BLOCK) {
#pragma unroll
    for (int d = 0; d < D; ++d)
      if (lane >= KK && lane < KMAX_BLOCK) sh[d * KMAX_BLOCK + lane][w] = 0.0;
  }
  __syncthreads();
  for (int k = w; k < D * KMAX_BLOCK; k += RED_THREADS / 32) {
    const double t = warp_sum(lane < RED_THREADS / 32 ? sh[k][lane] : 0.0);
    if (lane == 0) out[(int64_t)k * stride + blockIdx.x] = t;
  }
}

template <int G>
__device__ __forceinline__ void ldgrp(const double* p, double (&v)[G]) {
  if constexpr (G == 4) {
    asm volatile("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p) : "memory");
  } else {
    const double2 t = *reinterpret_cast<const double2*>(p);
    v[0] = t.x;
    v[1] = t.y;
  }
}
template <int G>
__device__ __forceinline__ void stgrp(double* p, const double (&v)[G]) {
  if constexpr (G == 4) {
    asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3]) : "memory");
  } else {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  }
}

// D = 1: a . b per column; D = 2: and b . c
template <int KK, int D>
__global__ void __launch_bounds__(RED_THREADS, 2) k_bdots(int64_t n, const double* a,
                                                          const double* b, const double* c,
                                                          double* __restrict__ part, Fin fin) {
  pdl_sync();
  using B = BRow<KK>;
  constexpr int G = B::G, L = B::LPR;
  const int lane = threadIdx.x & 31;
  double acc[D][L][G];
#pragma unroll
  for (int d = 0; d < D; ++d)
#pragma unroll
    for (int u = 0; u < L; ++u)
#pragma unroll
      for (int h = 0; h < G; ++h) acc[d][u][h] = 0.0;
  for (int64_t i0 = (int64_t)blockIdx.x * RED_THREADS + (threadIdx.x & ~31u); i0 < n;
       i0 += (int64_t)gridDim.x * RED_THREADS) {
    const int64_t i = i0 + lane / L;
    const int64_t o = i * KK + lane % L * G;
    if (D == 1 && i + (L - 1) * B::RPL < n) {  // all slots' loads together
      double av[L][G], bv[L][G];
#pragma unroll
      for (int u = 0; u < L; ++u) {
        ldgrp<G>(a + o + u * B::RPL * KK, av[u]);
        ldgrp<G>(b + o + u * B::RPL * KK, bv[u]);
      }
#pragma unroll
      for (int u = 0; u < L; ++u)
#pragma unroll
        for (int h = 0; h < G; ++h) acc[0][u][h] = fma(av[u][h], bv[u][h], acc[0][u][h]);
    } else {
#pragma unroll
      for (int u = 0; u < L; ++u) {
        if (i + u * B::RPL >= n) continue;
        double av[G], bv[G], cv[G];
        ldgrp<G>(a + o + u * B::RPL * KK, av);
        ldgrp<G>(b + o + u * B::RPL * KK, bv);
        if constexpr (D == 2) ldgrp<G>(c + o + u * B::RPL * KK, cv);
#pragma unroll
        for (int h = 0; h < G; ++h) {
          acc[0][u][h] = fma(av[h], bv[h], acc[0][u][h]);
          if constexpr (D == 2) acc[1][u][h] = fma(bv[h], cv[h], acc[1][u][h]);
        }
      }
    }
  }
  bblock_sum_to<KK, D>(acc, part, RED_BLOCKS);
  fin_inline<D * KB, RED_THREADS, (D - 1) * KB>(fin, part, (int)gridDim.x, RED_BLOCKS);
}

template <int KK>
__global__ void __launch_bounds__(RED_THREADS, 2)
    k_bcg_update(const int64_t n, const CgScalars* s, const int* active,
                 const double* p, const double* q, double* __restrict__ x,
                 double* __restrict__ r, double* __restrict__ rprev, double* __restrict__ part, Fin fin) {
  pdl_sync();
  using B = BRow<KK>;
  constexpr int G = B::G, L = B::LPR;
  __shared__ double alpha[KB];
  __shared__ int on[KB];
  if (threadIdx.x < KB) {
    const int c = threadIdx.x;
    on[c] = c < KK && active[c];
    alpha[c] = c < KK ? s[c].alpha : 0.0;
  }
  __syncthreads();
  bool any = false;
#pragma unroll
  for (int c = 0; c < KK; ++c) any |= on[c] != 0;
  const int lane = threadIdx.x & 31, g = lane % L * G;
  double acc[1][L][G];
#pragma unroll
  for (int u = 0; u < L; ++u)
#pragma unroll
    for (int h = 0; h < G; ++h) acc[0][u][h] = 0.0;
  // each column updated and summed exactly as in the one-vector kernel; a
  // frozen column's values are written back unchanged
  for (int64_t i0 = (int64_t)blockIdx.x * RED_THREADS + (threadIdx.x & ~31u); i0 < n;
       i0 += (int64_t)gridDim.x * RED_THREADS) {
#pragma unroll
    for (int u = 0; u < L; ++u) {
      const int64_t i = i0 + lane / L + u * B::RPL;
      if (i >= n) continue;
      const int64_t o = i * KK + g;
      double rv[G];
      ldgrp<G>(r + o, rv);
      if (any) {
        double qv[G], xv[G], pv[G];
        ldgrp<G>(q + o, qv);
        ldgrp<G>(x + o, xv);
        ldgrp<G>(p + o, pv);
        if (rprev) stgrp<G>(rprev + o, rv);
#pragma unroll
        for (int h = 0; h < G; ++h)
          if (on[g + h]) rv[h] = fma(-alpha[g + h], qv[h], rv[h]);
        stgrp<G>(r + o, rv);
#pragma unroll
        for (int h = 0; h < G; ++h)
          if (on[g + h]) xv[h] = fma(alpha[g + h], pv[h], xv[h]);
        stgrp<G>(x + o, xv);
      }
#pragma unroll
      for (int h = 0; h < G; ++h) acc[0][u][h] = fma(rv[h], rv[h], acc[0][u][h]);
    }
  }
  bblock_sum_to<KK, 1>(acc, part, RED_BLOCKS);
  fin_inline<KB, RED_THREADS, 0>(fin, part, (int)gridDim.x, RED_BLOCKS);
}

template <int KK>
__global__ void __launch_bounds__(RED_THREADS, 2)
    k_bcg_pupdate(int64_t n, const CgScalars* s, const int* active,
                  const double* z, double* __restrict__ p, int first) {
  pdl_sync();
  using B = BRow<KK>;
  constexpr int G = B::G, L = B::LPR;
  __shared__ double beta[KB];
  __shared__ int on[KB];
  if (threadIdx.x < KB) {
    const int c = threadIdx.x;
    on[c] = c < KK && active[c];
    beta[c] = c < KK ? s[c].beta : 0.0;
  }
  __syncthreads();
  bool any = false;
#pragma unroll
  for (int c = 0; c < KK; ++c) any |= on[c] != 0;
  if (!any) return;
  const int lane = threadIdx.x & 31, g = lane % L * G;
  for (int64_t i0 = (int64_t)blockIdx.x * RED_THREADS + (threadIdx.x & ~31u); i0 < n;
       i0 += (int64_t)gridDim.x * RED_THREADS) {
    const int64_t i = i0 + lane / L;
    const int64_t o = i * KK + g;
    double zv[L][G], pv[L][G];
#pragma unroll
    for (int u = 0; u < L; ++u) {
      if (i + u * B::RPL < n) {
        ldgrp<G>(z + o + u * B::RPL * KK, zv[u]);
        ldgrp<G>(p + o + u * B::RPL * KK, pv[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < L; ++u) {
      if (i + u * B::RPL < n) {
#pragma unroll
        for (int h = 0; h < G; ++h)
          if (on[g + h]) pv[u][h] = first ? zv[u][h] : fma(beta[g + h], pv[u][h], zv[u][h]);
        stgrp<G>(p + o + u * B::RPL * KK, pv[u]);
      }
    }
  }
}

// column-major n x k <-> interleaved n x K (columns k..K-1 of the block are zero)
__global__ void k_interleave(int64_t n, int k, int K, const double* __restrict__ src, double* __restrict__ dst,
                             int to_interleaved) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * K) return;
  const int64_t i = e / K;
  const int c = (int)(e % K);
  if (to_interleaved) dst[e] = c < k ? src[(int64_t)c * n + i] : 0.0;
  else if (c < k) dst[(int64_t)c * n + i] = src[e];
}

int launch_bdots(cudaStream_t st, int64_t n, int k, const double* a, const double* b, const double* c, double* part,
                 const Fin& fin) {
  if (k != 2 && k != 4 && k != 8) return SA_ERR_INVALID_ARG;  // whole-row vectors
  if (fin.op == FIN_BETA && fin.flexible > 0 && !c) return SA_ERR_INVALID_ARG;  // needs the second dot
  const unsigned g = red_blocks(n);
  // one dot per column (a . b), or two (b . c into out[KB + column])
  if (c) {
    if (k == 2) launch_pdl(k_bdots<2, 2>, g, RED_THREADS, 0, st, n, a, b, c, part, fin);
    else if (k == 4) launch_pdl(k_bdots<4, 2>, g, RED_THREADS, 0, st, n, a, b, c, part, fin);
    else launch_pdl(k_bdots<8, 2>, g, RED_THREADS, 0, st, n, a, b, c, part, fin);
  } else {
    if (k == 2) launch_pdl(k_bdots<2, 1>, g, RED_THREADS, 0, st, n, a, b, c, part, fin);
    else if (k == 4) launch_pdl(k_bdots<4, 1>, g, RED_THREADS, 0, st, n, a, b, c, part, fin);
    else launch_pdl(k_bdots<8, 1>, g, RED_THREADS, 0, st, n, a, b, c, part, fin);
  }
  SA_LAUNCHED();
  return SA_OK;
}

int launch_bcg_update(cudaStream_t st, int64_t n, int k, const CgScalars* s, const int* active, const double* p,
                      const double* q, double* x, double* r, double* rprev, double* part, const Fin& fin) {
  if (k != 2 && k != 4 && k != 8) return SA_ERR_INVALID_ARG;  // whole-row vectors
  const unsigned g = red_blocks(n);
  if (k == 2) launch_pdl(k_bcg_update<2>, g, RED_THREADS, 0, st, n, s, active, p, q, x, r, rprev, part, fin);
  else if (k == 4) launch_pdl(k_bcg_update<4>, g, RED_THREADS, 0, st, n, s, active, p, q, x, r, rprev, part, fin);
  else launch_pdl(k_bcg_update<8>, g, RED_THREADS, 0, st, n, s, active, p, q, x, r, rprev, part, fin);
  SA_LAUNCHED();
  return SA_OK;
}

int launch_bcg_pupdate(cudaStream_t st, int64_t n, int k, const CgScalars* s, const int* active, const double* z,
                       double* p, int first) {
  if (k != 2 && k != 4 && k != 8) return SA_ERR_INVALID_ARG;  // whole-row vectors
  if (k == 2) launch_pdl(k_bcg_pupdate<2>, red_blocks(n), RED_THREADS, 0, st, n, s, active, z, p, first);
  else if (k == 4) launch_pdl(k_bcg_pupdate<4>, red_blocks(n), RED_THREADS, 0, st, n, s, active, z, p, first);
  else launch_pdl(k_bcg_pupdate<8>, red_blocks(n), RED_THREADS, 0, st, n, s, active, z, p, first);
  SA_LAUNCHED();
  return SA_OK;
}

int launch_interleave(cudaStream_t st, int64_t n, int k, int K, const double* src, double* dst, int to_interleaved) {
  if (n * K <= 0) return SA_OK;
  k_interleave<<<blocks_for(n * K, 256), 256, 0, st>>>(n, k, K, src, dst, to_interleaved);
  SA_LAUNCHED();
  return SA_OK;
}

}  // namespace sa
