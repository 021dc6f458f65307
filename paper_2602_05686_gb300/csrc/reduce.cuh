// Fixed-order sums of per-block partials, finished inside the launch that
// wrote them.
//
// A dot product of the outer CG is per-block partial sums over a fixed grid,
// summed in a fixed order: FIN_T virtual threads, thread v adding partials v,
// v + FIN_T, ... in that order; a butterfly over each group of 32; the groups
// in index order.  The block that finishes last does this and the scalar step
// that follows (alpha, beta, loop control): a launch of its own for the sum
// held one SM for 9.5 us at 304 partials (three values in 1024 threads, the 32
// group sums added one by one at 65 cycles a DADD) and another launch the
// scalar.  Groups without partials add zeros and are skipped, as are blocks
// without elements (red_blocks), so the bits do not depend on them.
#pragma once

#include "common.cuh"
#include "solve.cuh"

namespace sa {

constexpr int FIN_T = 1024;
// above this many partials (times columns) the finishing block's loads would
// be the longer part: a launch of 32 blocks then takes one group each (7.2M
// rows, 28k partials: 33 us in one block of 1024)
constexpr int FIN_INLINE = 4096;

enum FinOp {
  FIN_STORE = 0,  // out[v] = the sums
  FIN_ALPHA = 1,  // ... and alpha = rz / pq
  FIN_BETA = 2,   // ... and beta (flexible: -1 initialises rz)
  FIN_LOOP = 3,   // ... and the captured CG loop's control (out[0] = r.r)
  FIN_POWER = 4   // power step: w.w and v.v -> estimate and next scale
};

struct Fin {
  int op = FIN_STORE;
  double* out = nullptr;
  unsigned* tick = nullptr;   // zero before and after every launch
  double* wsum = nullptr;     // KMAX_BLOCK x 32 doubles (the wide form's group sums)
  CgScalars* cg = nullptr;    // one problem, or k columns
  int k = 0;                  // columns (0: one vector)
  const int* active = nullptr;
  int flexible = 0;
  unsigned long long loop = 0;  // conditional handle
  int* it = nullptr;
  const double* ctl = nullptr;
  int maxit = 0;
  double* sc = nullptr;       // power method scalars
  double* lam = nullptr;
};

// blocks of a reduction over n elements: those of the fixed grid that have any
inline unsigned red_blocks(int64_t n) {
  const int64_t b = (n + RED_THREADS - 1) / RED_THREADS;
  return (unsigned)(b < 1 ? 1 : (b < RED_BLOCKS ? b : RED_BLOCKS));
}

__host__ __device__ __forceinline__ void cg_alpha_step(CgScalars* s, double pq) {
  s->pq = pq;
  if (!(pq > 0.0)) { s->breakdown = 1; s->alpha = 0.0; return; }
  s->alpha = s->rz / pq;
}

// beta from the new r.z (and z.r_prev for flexible CG)
__host__ __device__ __forceinline__ void cg_beta_step(CgScalars* s, double rz_new, double zr, int flexible) {
  if (flexible < 0) {
    s->rz = rz_new;
    s->beta = 0.0;
    s->breakdown = 0;
    return;
  }
  const double num = flexible ? rz_new - zr : rz_new;
  s->beta = num / s->rz;
  s->rz = rz_new;
}

// the block that calls this last among `blocks` (its writes and those of all
// others are visible to it)
__device__ __forceinline__ bool last_block(unsigned* tick, unsigned blocks) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicInc(tick, blocks - 1) == blocks - 1;
    __threadfence();
  }
  __syncthreads();
  return s_last != 0;
}

// sums of NV values over np partials (value v at part[v * stride + t]) into
// res (shared), by a block of NT threads
template <int NV, int NT>
__device__ __forceinline__ void fin_sums(const double* part, int np, int64_t stride, double* res) {
  __shared__ double sh[NV][33];
  const int lane = (int)(threadIdx.x & 31), w = (int)(threadIdx.x >> 5);
  const int groups = np < FIN_T ? (np + 31) >> 5 : 32;
  for (int q = w; q < groups; q += NT / 32) {
    double acc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[v] = 0.0;
    for (int t = q * 32 + lane; t < np; t += FIN_T)
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] += __ldcg(part + v * stride + t);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double s = warp_sum(acc[v]);
      if (lane == 0) sh[v][q] = s;
    }
  }
  __syncthreads();
  if (threadIdx.x < NV) {
    double s = 0.0;
    for (int q = 0; q < groups; ++q) s += sh[threadIdx.x][q];
    res[threadIdx.x] = s;
  }
  __syncthreads();
}

// the step that follows the sums res[0 .. NV), by thread c; the second values
// (flexible beta) are res[OFF2 ...], OFF2 = 0 where the reduction has none: the
// k-column forms hold OFF2 columns of first values before as many second ones.
// (Arithmetic only, so that it runs on the host too.)
template <int NV, int OFF2>
__host__ __device__ __forceinline__ void fin_step(const Fin& f, const double* res, int c) {
  static_assert(OFF2 == 0 || 2 * OFF2 == NV, "a second value for every first one");
  if (f.op != FIN_POWER && c < NV) f.out[c] = res[c];
  if (f.k > 0) {
    if (c >= f.k) return;
    if (f.op == FIN_ALPHA) {
      if (f.active[c]) cg_alpha_step(f.cg + c, res[c]);
      else f.cg[c].alpha = 0.0;
    } else if (f.op == FIN_BETA) {
      if (f.active[c]) {
        double zr = 0.0;
        if constexpr (OFF2 > 0) zr = res[OFF2 + c];  // c < k <= OFF2
        cg_beta_step(f.cg + c, res[c], zr, f.flexible);
      }
    }
    return;
  }
  if (c != 0) return;
  switch (f.op) {
    case FIN_ALPHA: cg_alpha_step(f.cg, res[0]); break;
    case FIN_BETA: cg_beta_step(f.cg, res[0], NV > 1 ? res[NV - 1] : 0.0, f.flexible); break;
    case FIN_LOOP: {
      // count the iteration and decide whether the WHILE node runs the body again
      const int k = *f.it + 1;
      *f.it = k;
      const int cont = !f.cg->breakdown && !(sqrt(res[0]) <= f.ctl[0]) && k < f.maxit;
#ifdef __CUDA_ARCH__
      cudaGraphSetConditional((cudaGraphConditionalHandle)f.loop, cont ? 1u : 0u);
#else
      (void)cont;
#endif
      break;
    }
    case FIN_POWER: {
      // lam = ||w|| / ||v||, sc[2] = ||w||, sc[4] = 1 / ||w|| (the scale of
      // the next iterate).  A zero product (every row unscaled) gives lam = 0
      // and stops the iteration (sc[3] = 1).
      const double nw2 = sqrt(res[0]);
      if (nw2 == 0.0 || f.sc[3] != 0.0) {
        f.sc[3] = 1.0;
        *f.lam = 0.0;
        break;
      }
      *f.lam = nw2 / sqrt(NV > 1 ? res[1] : 0.0);
      f.sc[2] = nw2;
      f.sc[4] = 1.0 / nw2;
      break;
    }
    default: break;
  }
}

// end of a reduction kernel whose blocks have written their partials (thread
// 0 of each wrote or waited for them): the last block sums and steps
template <int NV, int NT, int OFF2>
__device__ __forceinline__ void fin_inline(const Fin& f, const double* part, int np, int64_t stride) {
  __shared__ double res[NV];
  if (!last_block(f.tick, gridDim.x)) return;
  fin_sums<NV, NT>(part, np, stride, res);
  fin_step<NV, OFF2>(f, res, (int)threadIdx.x);
}

// the wide form: block q takes group q, a warp per value
template <int NV>
__global__ void __launch_bounds__(32 * NV) k_fin_wide(const double* part, int np, int64_t stride,
                                                      Fin f) {
  pdl_sync();
  __shared__ double res[NV];
  const int lane = (int)(threadIdx.x & 31), v = (int)(threadIdx.x >> 5);
  const int q = (int)blockIdx.x;
  double acc = 0.0;
  const double* p = part + v * stride;
  int t = q * 32 + lane;
  for (; t + 7 * FIN_T < np; t += 8 * FIN_T) {
    double u[8];
#pragma unroll
    for (int h = 0; h < 8; ++h) u[h] = p[t + h * FIN_T];
#pragma unroll
    for (int h = 0; h < 8; ++h) acc += u[h];
  }
  for (; t < np; t += FIN_T) acc += p[t];
  acc = warp_sum(acc);
  if (lane == 0) f.wsum[v * 32 + q] = acc;
  if (!last_block(f.tick, gridDim.x)) return;
  if (threadIdx.x < NV) {
    double s = 0.0;
    double u[32];
#pragma unroll
    for (int h = 0; h < 32; ++h) u[h] = __ldcg(f.wsum + threadIdx.x * 32 + h);
#pragma unroll
    for (int h = 0; h < 32; ++h) s += u[h];
    res[threadIdx.x] = s;
  }
  __syncthreads();
  fin_step<NV, 0>(f, res, (int)threadIdx.x);
}

}  // namespace sa
