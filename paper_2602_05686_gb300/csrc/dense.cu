// Coarsest level (Sec. 4: the coarsest level is solved directly).  A_L
// (n_L <= a few thousand) is factored A_L = L L^T by a tiled Cholesky in FP64
// (32 x 32 tiles) inside its skyline; then the inverses of the diagonal
// blocks of COARSE_BS rows, W_KK = L_KK^-1, are formed by blocked forward
// substitution on the identity.  Every coarse solve is block substitution:
// per diagonal block a row-parallel product with the blocks already solved
// and one with W_KK (forward with L, backward with L^T and W_KK^T), so it uses
// every SM instead of running row-by-row sweeps.  L^T and W^T are stored
// explicitly so all products read contiguous rows.
//
// Skyline: Cholesky without pivoting creates no entry left of a row's first
// nonzero, so with f_i the first nonzero tile column of tile row i, L_ij = 0
// for j < f_i, and a product of a zero tile changes nothing.  Factor, inverses
// and solve skip those tiles.  The coarse operators are numbered along the
// mesh (aggregates by ascending root index), so their skylines hold 0.06
// (4225-row square) to 0.45 (3989-row 3D level) of the lower triangle and
// 0.002 to 0.16 of the dense factor's tile products.
#include <math.h>

#include <vector>

#include "common.cuh"
#include "profile.cuh"
#include "group.cuh"
#include "solve.cuh"
#include "sqrt_rcp.cuh"

namespace sa {

constexpr int NB = 32;
constexpr int CH_THREADS = 256;
constexpr int CH_STRIP = 16;             // columns of one inverse task
constexpr int CH_BT = (int)(COARSE_BS / NB);  // tiles per diagonal block
constexpr uint32_t CH_INV = 0x80000000u;      // task word of an inverse strip
constexpr int CH_POLLS = 1 << 24;             // about ten seconds; the longest wait is some tasks of 8 us a product

// f[i]: first nonzero tile column of tile row i (at most the diagonal tile):
// a warp over the tile row's entries, whatever their order
__global__ void k_sky_first(int64_t n, int nb, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                            int32_t* __restrict__ f) {
  const int i = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
  if (i >= nb) return;
  const int64_t o = (int64_t)i * NB, r1 = o + NB < n ? o + NB : n;
  int c = i;
  for (int64_t p = rp[o] + lane_id(); p < rp[r1]; p += 32) {
    const int t = ci[p] / NB;
    c = t < c ? t : c;
  }
  c = __reduce_min_sync(FULL, c);
  if (lane_id() == 0) f[i] = c;
}

// the skyline of tile row blockIdx.x as dense rows: zeros, then the entries of
// the lower triangle (and of the diagonal tile)
__global__ void k_densify_sky(int64_t n, const int32_t* __restrict__ f, const int64_t* __restrict__ rp,
                              const int32_t* __restrict__ ci, const double* __restrict__ v, double* __restrict__ M) {
  const int64_t o = (int64_t)blockIdx.x * NB;
  const int64_t c0 = (int64_t)f[blockIdx.x] * NB, c1 = o + NB < n ? o + NB : n;
  const int64_t r1 = o + NB < n ? o + NB : n;
  for (int64_t r = o; r < r1; ++r)
    for (int64_t c = c0 + threadIdx.x; c < c1; c += blockDim.x) M[r * n + c] = 0.0;
  __syncthreads();
  const int w = (int)(threadIdx.x >> 5), nw = (int)(blockDim.x >> 5), lane = lane_id();
  for (int64_t r = o + w; r < r1; r += nw)
    for (int64_t p = rp[r] + lane; p < rp[r + 1]; p += 32) {
      const int32_t c = ci[p];
      if (c < c1) M[r * n + c] = v[p];
    }
}

struct CholView {
  int64_t n;
  int nb;
  const int32_t* f;      // first tile column of each tile row
  const int32_t* off;    // flag index of tile (i, f_i); tile (i, j) at off[i] + j - f[i]
  const uint32_t* task;
  int ntask;
  double *M, *LT, *W, *WT, *Dinv;
  int* flag;             // 1: the tile of L is written; on the diagonal: chunks of its inverse written
  int* ticket;
  int* err;              // 1: pivot not positive; 2: a wait ran out
  int limit;             // polls of a wait
};

// bounded wait of one thread for *p >= want: false when it ran out or another
// wait did
__device__ bool ch_poll(const int* p, int want, int limit, int* err) {
  for (int it = 0; it < limit; ++it) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    if (v >= want) return true;
    if (it > 64) {
      __nanosleep(64);
      if ((it & 1023) == 0 && (*(volatile int*)err & 2)) return false;
    }
  }
  atomicOr(err, 2);
  return false;
}

__device__ __forceinline__ void ch_publish(int* p, int v) {
  // the writers' stores are ordered before the flag: barrier (by the caller),
  // then this thread's fence and release
  __threadfence();
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// handoff between warps of a block without a barrier: the writer's warps meet at
// a barrier, one thread then releases the count, each reader acquires it
__device__ __forceinline__ void cta_release(int* p, int v) {
  asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int cta_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.cta.shared.s32 %0, [%1];" : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
  return v;
}

// factor the tile in T (rows and columns < bs) in place and form its inverse
// in Y (lower triangular, zero elsewhere), published to D in CH_CHUNKS chunks
// of rows.  The chain is sqrt -> 1/x -> scale -> update of the next pivot; FP64
// issue (64 cycles an instruction on each of the four schedulers) is the next
// bound.  Warp 0 runs the chain alone (a row per lane); warps 1-3 apply the
// previous column to the columns right of the next one, one barrier of these
// four per column; warps 4-7 form the inverse's rows behind them at their own
// pace (a column of the inverse needs no other column).
// 32 columns with the inverse: 45 us as one block's loop over columns, 31 us
// with the inverse inside the per-column barrier, 27 us now (22 us for the
// columns; 14 us is the FP64 issue of both on one SM).
constexpr int CH_CHUNKS = 4;
__device__ __forceinline__ void potrf_inv(int bs, double (*T)[NB + 1], double (*Y)[NB + 1], double* rinv, int* ready,
                                          double* __restrict__ D, int* dflag, int* err) {
  const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
  if (warp < 4) {
    double l = 0.0;  // warp 0: row `lane` of the previous column of L
    for (int j = 0; j < bs; ++j) {
      if (warp == 0) {
        double t = T[lane][j];
        if (j > 0) {
          const double lj = __shfl_sync(FULL, l, j);
          if (lane >= j) t = fma(-l, lj, t);
        }
        double d = __shfl_sync(FULL, t, j);
        // !(d > 0), as integers (an FP64 comparison is 65 cycles of the chain)
        const long long db = __double_as_longlong(d);
        if (db <= 0 || db > 0x7ff0000000000000ll) {
          if (lane == 0) atomicOr(err, 1);
          d = 1.0;
        }
        double dr, ri;
        sqrt_rcp(d, dr, ri);
        l = lane == j ? dr : (lane > j ? t * ri : 0.0);
        if (lane >= j) T[lane][j] = l;
        if (lane == 0) rinv[j] = ri;
      } else if (j > 0) {
        const int m = j - 1;
        const double lm = T[lane][m];
        for (int q0 = j + warp; q0 < bs; q0 += 15) {
          double a[5], b[5];
#pragma unroll
          for (int u = 0; u < 5; ++u) {
            const int q = q0 + 3 * u;
            const bool in = q < bs && lane >= q && lane < bs;
            a[u] = in ? T[lane][q] : 0.0;
            b[u] = in ? T[q][m] : 0.0;
          }
#pragma unroll
          for (int u = 0; u < 5; ++u) {
            const int q = q0 + 3 * u;
            if (q < bs && lane >= q && lane < bs) T[lane][q] = fma(-lm, b[u], a[u]);
          }
        }
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
      // column j is written (the barrier): tell the inverse's warps
      if (threadIdx.x == 32) cta_release(ready, j + 1);
    }
  } else {
    // eight lanes per column split each row's dot product; two columns a lane
    const int c0 = (warp - 4) * 4 + (lane >> 3), c1 = c0 + 16, g = lane & 7;
    for (int m = 0; m < NB; ++m) {
      if (m < bs) {
        // (the column warps end without waiting for these; bounded all the same)
        int it = 0;
        while (cta_acquire(ready) <= m && ++it < (1 << 22)) __nanosleep(20);
        if (it >= (1 << 22)) atomicOr(err, 2);
        double p0 = 0.0, p1 = 0.0;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int q0 = c0 + g + 8 * t, q1 = c1 + g + 8 * t;
          if (q0 < m) p0 = fma(T[m][q0], Y[q0][c0], p0);
          if (q1 < m) p1 = fma(T[m][q1], Y[q1][c1], p1);
        }
        // the butterfly over the eight lanes (4, 2, 1), lanes 0-3 keeping
        // column c0 after the first exchange and lanes 4-7 column c1
        const bool up = (lane & 4) != 0;
        double part = (up ? p1 : p0) + __shfl_xor_sync(FULL, up ? p0 : p1, 4, 8);
        part += __shfl_xor_sync(FULL, part, 2, 8);
        part += __shfl_xor_sync(FULL, part, 1, 8);
        const int c = up ? c1 : c0;
        const double y = ((m == c ? 1.0 : 0.0) - part) * rinv[m];
        if ((g & 3) == 0 && c <= m) Y[m][c] = y;
        __syncwarp();
      }
      if ((m + 1) % (NB / CH_CHUNKS) == 0) {
        const int r0 = m + 1 - NB / CH_CHUNKS, t = (int)threadIdx.x - 128;
        asm volatile("bar.sync 2, 128;" ::: "memory");
        for (int e = t; e < NB * NB / CH_CHUNKS; e += 128) D[r0 * NB + e] = Y[r0 + e / NB][e % NB];
        asm volatile("bar.sync 2, 128;" ::: "memory");
        if (t == 0) ch_publish(dflag, (m + 1) / (NB / CH_CHUNKS));
      }
    }
  }
  __syncthreads();
}

// One launch factors the matrix and inverts its diagonal blocks.  A task is
// one tile of L (left-looking: all its products, then its solve or its own
// factor) or a strip of CH_STRIP columns of one W_KK; the tile left of a
// diagonal tile is part of the diagonal tile's task (the factor's chain is
// L_jj -> L_(j+1)j -> L_(j+1)(j+1), one hop between CTAs per tile column).
// Tasks are numbered so that a task reads only tiles of lower-numbered tasks,
// CTAs draw tickets in that order and wait (bounded) on the tiles' flags.  The lowest unfinished
// task never waits for one that no CTA has drawn, so the launch makes
// progress with any number of resident CTAs.
// Every tile sees the products of the blocked right-looking form in the same
// order (per product a sum over the tile's 32 columns, subtracted from the
// tile; tile columns ascending), so the factor is bitwise that form's.
// Bound by the chain of diagonal tiles (32 us a tile column) on narrow
// skylines, by FP64 issue (8 us a tile product and SM) on wide ones.  4225-row
// square 34.4 ms as launches per panel over the whole triangle, 4.1 ms now;
// 2210-row 3D level (skyline 0.26) 10.7 ms, 3.3 ms.
__global__ void __launch_bounds__(CH_THREADS) k_chol(CholView C) {
  __shared__ double As[2][NB][NB + 1];
  __shared__ double Bs[2][NB][NB + 1];
  __shared__ double rinv[NB];
  __shared__ int s_task, s_ready;
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t n = C.n;
  for (;;) {
    __syncthreads();  // the previous task's reads of shared memory
    if (tid == 0) s_task = atomicAdd(C.ticket, 1);
    __syncthreads();
    const int tk = s_task;
    if (tk >= C.ntask) return;
    const uint32_t tw = C.task[tk];
    if (tw & CH_INV) {
      // columns c0 .. c0 + CH_STRIP - 1 of W_KK: for tile rows i downwards
      // X = (I)_i - sum_m L_im W_m,  W_i = L_ii^-1 X
      const int q = (int)((tw >> 16) & 0x7fff), s = (int)(tw & 0xffff);
      const int64_t c0 = (int64_t)q * COARSE_BS + (int64_t)s * CH_STRIP;
      const int jt = (int)(c0 / NB);
      const int e = (q + 1) * CH_BT < C.nb ? (q + 1) * CH_BT : C.nb;
      const int cw = (int)(n - c0 < CH_STRIP ? n - c0 : CH_STRIP);
      const int r = tid >> 4, c = tid & 15;  // outputs (r, c) and (r + 16, c)
      int buf = 0;
      for (int i = jt; i < e; ++i) {
        const int64_t oi = (int64_t)i * NB;
        const int bi = (int)(n - oi < NB ? n - oi : NB);
        const int fi = C.f[i];
        double x0 = c0 + c == oi + r ? 1.0 : 0.0, x1 = c0 + c == oi + r + 16 ? 1.0 : 0.0;
        for (int m = fi > jt ? fi : jt; m < i; ++m) {
          const bool ok = tid != 0 || ch_poll(&C.flag[C.off[i] + m - fi], 1, C.limit, C.err);
          if (!__syncthreads_and(ok)) return;
          const int64_t om = (int64_t)m * NB;
          for (int t = tid; t < NB * NB; t += CH_THREADS) {
            const int a = t / NB, b = t % NB;
            As[buf][a][b] = a < bi ? __ldcg(&C.M[(oi + a) * n + om + b]) : 0.0;
          }
          for (int t = tid; t < NB * CH_STRIP; t += CH_THREADS) {
            const int a = t / CH_STRIP, b = t % CH_STRIP;
            Bs[buf][a][b] = b < cw ? __ldcg(&C.W[(om + a) * n + c0 + b]) : 0.0;
          }
          __syncthreads();
          double s0 = 0.0, s1 = 0.0;
#pragma unroll 8
          for (int u = 0; u < NB; ++u) {
            const double b = Bs[buf][u][c];
            s0 = fma(As[buf][r][u], b, s0);
            s1 = fma(As[buf][r + 16][u], b, s1);
          }
          x0 -= s0;
          x1 -= s1;
          buf ^= 1;
        }
        const bool ok = tid != 0 || ch_poll(&C.flag[C.off[i] + i - fi], CH_CHUNKS, C.limit, C.err);
        if (!__syncthreads_and(ok)) return;
        const double* D = C.Dinv + (int64_t)i * NB * NB;
        for (int t = tid; t < NB * NB; t += CH_THREADS) As[buf][t / NB][t % NB] = __ldcg(&D[t]);
        Bs[buf][r][c] = x0;
        Bs[buf][r + 16][c] = x1;
        __syncthreads();
        double w0 = 0.0, w1 = 0.0;
        for (int u = 0; u <= r; ++u) w0 = fma(As[buf][r][u], Bs[buf][u][c], w0);
        for (int u = 0; u <= r + 16; ++u) w1 = fma(As[buf][r + 16][u], Bs[buf][u][c], w1);
        if (c < cw) {
          if (r < bi) {
            C.W[(oi + r) * n + c0 + c] = w0;
            C.WT[(c0 + c) * n + oi + r] = w0;
          }
          if (r + 16 < bi) {
            C.W[(oi + r + 16) * n + c0 + c] = w1;
            C.WT[(c0 + c) * n + oi + r + 16] = w1;
          }
        }
        buf ^= 1;
        __syncthreads();  // this strip's rows of W before they are read back
      }
      continue;
    }
    const int i = (int)(tw >> 15), j = (int)(tw & 0x7fff);
    const bool diag = i == j;
    const int fi = C.f[i];
    // the off-diagonal tile of this task: (i, j), or (i, i - 1) on the diagonal
    const int jo = diag ? i - 1 : j;
    const bool off = !diag || fi < i;
    const int fo = off ? C.f[jo] : 0;
    const int64_t oi = (int64_t)i * NB, oj = (int64_t)jo * NB;
    const int bi = (int)(n - oi < NB ? n - oi : NB);  // column tiles left of the diagonal are full
    // this thread's elements: rows warp + 8u of column `lane`; of the diagonal
    // tile the lower triangle's 528 elements in order
    double acc[4] = {0.0, 0.0, 0.0, 0.0}, dac[3] = {0.0, 0.0, 0.0};
    int er[3], ec[3];
    if (off) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int a = warp + 8 * u;
        acc[u] = a < bi ? __ldcg(&C.M[(oi + a) * n + oj + lane]) : 0.0;
      }
    }
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      const int t = tid + CH_THREADS * u;
      int a = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
      while ((a + 1) * (a + 2) / 2 <= t) ++a;
      while (a * (a + 1) / 2 > t) --a;
      er[u] = a;
      ec[u] = t - a * (a + 1) / 2;
      if (diag && a < bi) dac[u] = __ldcg(&C.M[(oi + a) * n + oi + ec[u]]);
    }
    int buf = 0;
    for (int k = diag || fi > fo ? fi : fo; k < jo; ++k) {
      const bool prod = k >= fo;  // (diagonal tasks: the off-diagonal tile's skyline may start later)
      bool ok = true;
      if (tid == 0) ok = ch_poll(&C.flag[C.off[i] + k - fi], 1, C.limit, C.err);
      if (tid == 32 && prod) ok = ch_poll(&C.flag[C.off[jo] + k - fo], 1, C.limit, C.err);
      if (!__syncthreads_and(ok)) return;
      const int64_t kc = (int64_t)k * NB;
      for (int t = tid; t < NB * NB; t += CH_THREADS) {
        const int a = t / NB, b = t % NB;
        As[buf][a][b] = a < bi ? __ldcg(&C.M[(oi + a) * n + kc + b]) : 0.0;
        if (prod) Bs[buf][a][b] = __ldcg(&C.M[(oj + a) * n + kc + b]);
      }
      __syncthreads();
      if (prod) {
        double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 8
        for (int m = 0; m < NB; ++m) {
          const double b = Bs[buf][lane][m];
#pragma unroll
          for (int u = 0; u < 4; ++u) s[u] = fma(As[buf][warp + 8 * u][m], b, s[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] -= s[u];
      }
      if (diag) {
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          if (er[u] < NB) {
            double s = 0.0;
#pragma unroll 8
            for (int m = 0; m < NB; ++m) s = fma(As[buf][er[u]][m], As[buf][ec[u]][m], s);
            dac[u] -= s;
          }
        }
      }
      buf ^= 1;
    }
    double(*T)[NB + 1] = As[buf];
    double(*Y)[NB + 1] = Bs[buf];
    if (off) {
      // L_ij = X L_jj^-T, (L^-T)_qc = (L^-1)_cq, nonzero for q <= c: columns by
      // chunks as the inverse's rows arrive, row `lane`, column c0 + warp; on
      // the diagonal each chunk's part of the tile's last product follows
      double(*Lb)[NB + 1] = As[buf ^ 1];
      double s[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int u = 0; u < 4; ++u) T[warp + 8 * u][lane] = acc[u];
      const double* D = C.Dinv + (int64_t)jo * NB * NB;
      for (int ch = 0; ch < CH_CHUNKS; ++ch) {
        const int r0 = ch * (NB / CH_CHUNKS);
        const bool ok = tid != 0 || ch_poll(&C.flag[C.off[jo] + jo - fo], ch + 1, C.limit, C.err);
        if (!__syncthreads_and(ok)) return;
        Y[r0 + warp][lane] = __ldcg(&D[(r0 + warp) * NB + lane]);
        __syncthreads();
        const int c = r0 + warp;
        double o = 0.0;
        for (int q = 0; q <= c; ++q) o = fma(T[lane][q], Y[c][q], o);
        Lb[lane][c] = o;
        if (diag) {
          __syncthreads();
#pragma unroll
          for (int u = 0; u < 3; ++u)
            if (er[u] < NB)
#pragma unroll
              for (int m = 0; m < NB / CH_CHUNKS; ++m) s[u] = fma(Lb[er[u]][r0 + m], Lb[ec[u]][r0 + m], s[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < 3; ++u) dac[u] -= s[u];
      __syncthreads();
      for (int t = tid; t < NB * NB; t += CH_THREADS) {
        const int a = t / NB, b = t % NB;
        if (a < bi) C.M[(oi + a) * n + oj + b] = Lb[a][b];
        if (b < bi) C.LT[(oj + a) * n + oi + b] = Lb[b][a];
      }
    }
    if (diag) {
      for (int t = tid; t < NB * NB; t += CH_THREADS) {
        T[t / NB][t % NB] = 0.0;
        Y[t / NB][t % NB] = 0.0;
      }
      if (tid == 0) s_ready = 0;
    }
    __syncthreads();
    if (off && tid == 128) ch_publish(&C.flag[C.off[i] + jo - fi], 1);
    if (diag) {
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (er[u] < NB) T[er[u]][ec[u]] = dac[u];
      __syncthreads();
      potrf_inv(bi, T, Y, rinv, &s_ready, C.Dinv + (int64_t)i * NB * NB, &C.flag[C.off[i] + i - fi], C.err);
      for (int t = tid; t < NB * NB; t += CH_THREADS) {
        const int a = t / NB, b = t % NB;
        if (a < bi && b < bi) {
          C.M[(oi + a) * n + oi + b] = b <= a ? T[a][b] : 0.0;
          C.LT[(oi + a) * n + oi + b] = a <= b ? T[b][a] : 0.0;
        }
      }
    }
  }
}

DenseJob::~DenseJob() {
  // left without dense_finish (an error in between): the temporaries are
  // released on the caller's stream after this returns, so the dense
  // launches must have ended first
  if (pending && sd) cudaStreamSynchronize(sd);
  if (e_fork) cudaEventDestroy(e_fork);
  if (e_done) cudaEventDestroy(e_done);
  if (sd) cudaStreamDestroy(sd);
}

int dense_start(Alloc& al, int64_t n, const int64_t* rp, const int32_t* ci, const double* v, CoarseFactor& F,
                DenseJob& job) {
  cudaStream_t s = al.stream;
  job.main = s;
  job.n = n;
  if (n <= 0) return SA_OK;
  const int nb = (int)((n + NB - 1) / NB);
  SA_TRY(F.L.alloc(&al, n * n));
  SA_TRY(F.LT.alloc(&al, n * n));
  SA_TRY(F.W.alloc(&al, n * n));
  SA_TRY(F.WT.alloc(&al, n * n));
  SA_TRY(job.err.alloc(&al, 2));  // error bits, ticket counter
  SA_TRY(memset_d(job.err.p, 0, 2 * sizeof(int), s));
  // host tables, uploaded as one block: first tile column of each tile row,
  // end of the tile rows that reach each tile column (both kept for the
  // solve), flag offsets, tasks
  std::vector<int32_t> tab(3 * (size_t)nb + 1);
  {
    Buf<int32_t> f_dev;
    SA_TRY(f_dev.alloc(&al, nb));
    k_sky_first<<<blocks_for((int64_t)nb * 32, 256), 256, 0, s>>>(n, nb, rp, ci, f_dev.p);
    SA_LAUNCHED();
    SA_TRY(copy_d2h(tab.data(), f_dev.p, sizeof(int32_t) * nb, s));
  }
  int32_t ntile = 0;
  {
    const int32_t* f = tab.data();
    int32_t *env = tab.data() + nb, *off = tab.data() + 2 * nb;
    for (int j = 0; j < nb; ++j) env[j] = j + 1;
    off[0] = 0;
    for (int i = 0; i < nb; ++i) {
      off[i + 1] = off[i] + (i - f[i] + 1);
      if (env[f[i]] < i + 1) env[f[i]] = i + 1;
    }
    for (int j = 1; j < nb; ++j)
      if (env[j] < env[j - 1]) env[j] = env[j - 1];
    ntile = off[nb];
  }
  // tasks: tiles by columns, a diagonal tile (with the tile left of it) where
  // the tile left of it stands; a diagonal block's inverse strips once its
  // last column is numbered
  int64_t nprod = 0;  // tile products of the factor
  tab.reserve(tab.size() + (size_t)ntile + (size_t)(n / CH_STRIP) + 1);
  for (int j = 0; j < nb; ++j) {
    const int e = tab[nb + j];
    if (tab[j] == j) tab.push_back((j << 15) | j);  // no tile left of it
    if (j + 1 < nb && tab[j + 1] <= j) tab.push_back(((j + 1) << 15) | (j + 1));
    for (int i = j + 2; i < e; ++i)
      if (tab[i] <= j) {
        tab.push_back((i << 15) | j);
        nprod += j - (tab[i] > tab[j] ? tab[i] : tab[j]);
      }
    if ((j + 1) % CH_BT == 0 || j + 1 == nb) {
      const int q = j / CH_BT;
      const int64_t r0 = (int64_t)q * COARSE_BS, r1 = (int64_t)(j + 1) * NB < n ? (int64_t)(j + 1) * NB : n;
      for (int64_t c = r0; c < r1; c += CH_STRIP)
        tab.push_back((int32_t)(CH_INV | ((uint32_t)q << 16) | (uint32_t)((c - r0) / CH_STRIP)));
    }
  }
  const int64_t nt = (int64_t)tab.size() - (3 * (int64_t)nb + 1);
  SA_TRY(F.sky.alloc(&al, (int64_t)tab.size()));
  SA_TRY(job.flag.alloc(&al, ntile));
  SA_TRY(job.Dinv.alloc(&al, (int64_t)nb * NB * NB));
  // (pageable source: the copy has left it when the call returns)
  SA_TRY(copy_h2d(F.sky.p, tab.data(), sizeof(int32_t) * tab.size(), s));
  F.steps.clear();  // the solve's steps
  F.entries = coarse_steps(n, tab.data(), tab.data() + nb, F.steps);
  SA_TRY(memset_d(job.flag.p, 0, job.flag.bytes(), s));
  // L^T rows are read up to the last tile row that reaches them; tiles of
  // that range outside another row's skyline stay zero
  SA_TRY(memset_d(F.LT.p, 0, F.LT.bytes(), s));
  k_densify_sky<<<(unsigned)nb, 256, 0, s>>>(n, F.sky.p, rp, ci, v, F.L.p);
  SA_LAUNCHED();
  // The factor runs on its own stream `sd`, forked from the caller's stream
  // after the dense copy; the caller goes on with work that does not read
  // the factor (Chebyshev bounds, SELL packing) and joins in dense_finish.
  // It gets the highest priority: the factor is the setup's critical path,
  // the work it overlaps has slack.  Without the extra stream it runs on the
  // caller's.
  int prio_lo = 0, prio_hi = 0;
  if (cudaDeviceGetStreamPriorityRange(&prio_lo, &prio_hi) != cudaSuccess) {
    cudaGetLastError();
    prio_hi = 0;
  }
  const bool own = cudaStreamCreateWithPriority(&job.sd, cudaStreamNonBlocking, prio_hi) == cudaSuccess &&
                   cudaEventCreateWithFlags(&job.e_fork, cudaEventDisableTiming) == cudaSuccess &&
                   cudaEventCreateWithFlags(&job.e_done, cudaEventDisableTiming) == cudaSuccess;
  if (!own) cudaGetLastError();
  cudaStream_t m = s;
  if (own) {
    SA_CUDA(cudaEventRecord(job.e_fork, s));
    SA_CUDA(cudaStreamWaitEvent(job.sd, job.e_fork, 0));
    m = job.sd;
  }
  job.pending = own;
  const int ph = prof_begin(m, PK_S_DENSE, job.level, 0.0);
  CholView C;
  C.n = n; C.nb = nb; C.f = F.sky.p; C.off = F.sky.p + 2 * nb;
  C.task = reinterpret_cast<const uint32_t*>(F.sky.p + 3 * nb + 1); C.ntask = (int)nt;
  C.M = F.L.p; C.LT = F.LT.p; C.W = F.W.p; C.WT = F.WT.p; C.Dinv = job.Dinv.p;
  C.flag = job.flag.p; C.ticket = job.err.p + 1; C.err = job.err.p; C.limit = CH_POLLS;
  // one block per SM where the chain of diagonal tiles is the time (a second
  // block takes FP64 issue from it), two from 200 tile products per SM on.  Bands
  // and dense skylines of 512 to 5000 rows and 18 coarse levels, one against two:
  //   2744 rows,  8 products per SM     2.9, 3.5 ms
  //   2900 rows, 32                     4.6, 5.9
  //   3002 rows, 80                     6.6, 7.2
  //   1883 rows, 151                    5.5, 6.1
  //   3000 rows, 203                    8.4, 7.7
  //   4017 rows, 292                   21.6, 14.4
  //   5000 rows, 510                   16.7, 14.3
  // (Against it: 3 % of 3.7 ms at 1022 rows and 6 products, 3 to 9 % at 2000 and
  // 2500 dense rows, 249 and 500.)
  const int64_t g = (nprod < 200 * (int64_t)num_sms() ? 1 : 2) * (int64_t)num_sms();
  k_chol<<<(unsigned)(nt < g ? nt : g), CH_THREADS, 0, m>>>(C);
  SA_LAUNCHED();
  prof_end(m, ph);
  if (own) SA_CUDA(cudaEventRecord(job.e_done, m));
  return SA_OK;
}

int dense_finish(DenseJob& job) {
  if (job.n <= 0) return SA_OK;
  if (job.pending) {
    SA_CUDA(cudaStreamWaitEvent(job.main, job.e_done, 0));
    job.pending = false;
  }
  int h_err = 0;
  SA_TRY(copy_d2h(&h_err, job.err.p, sizeof(int), job.main));
  if (h_err & 2) {
    set_error_text("coarse factor: a wait for a tile ran out");
    return SA_ERR_CUDA;
  }
  return h_err ? SA_ERR_NOT_SPD : SA_OK;
}

// ---------------------------------------------------------------------------
// Coarse solve x = A_c^-1 b = L^-T (L^-1 b) by substitution over the diagonal
// blocks K (rows [r0, r1) of COARSE_BS):
//   forward   t_K = b_K - L_{K,<K} y_{<K};  y_K = W_KK t_K   (W_KK = L_KK^-1)
//   backward  t_K = y_K - (L^T)_{K,>K} x_{>K};  x_K = W_KK^T t_K
// Each step is a row-parallel product over one row range: TRI_WARPS warps per
// row, warp q taking the q-th of TRI_WARPS consecutive column segments of the
// row's range (segments of a multiple of 32 columns; lanes stride the segment,
// each lane summing in column order; a shuffle tree adds the lanes), the
// warps' sums added in warp order.  CS_W sums over [r0, i] (lower triangle of a
// diagonal block), CS_WT over [i, r1) (upper), CS_L rhs_i minus the sum over
// [0, r0), CS_LT rhs_i minus the sum over [r1, n); the last two leave out the
// columns outside the skyline (a lane starts at the first of its own columns
// inside it, so the sums are those over the whole range) and are taken for
// the rows whose skyline leaves the block only -- the others' t is the right-
// hand side itself.  The K-column forms run the same sums for every column as
// the one-column form (bitwise equal columns).
//
// One launch per step, for one problem or for all of a group that have it; a
// warp takes a row with its four segment sums side by side, all its loads in
// flight, and the exchanging butterfly over them (6 FP64 additions a row; a
// warp per segment took 20, and FP64 issue was half of a step's time).  Bound by
// the chain of steps, up to 4 per diagonal block: 3989 rows, 14 steps: 124 us
// with a block per row and a warp per segment, 97 us of kernels now (8 columns
// of 2062 rows, 10 steps: 165 -> 143 us).  (All steps in one launch, tasks on
// tickets and step counters, took 105 to 147 us: release, acquire and the
// uneven spread of the tasks cost more than the launches.)
// ---------------------------------------------------------------------------
constexpr int CS_SEG = 4;       // column segments of a row
constexpr int CS_ROWS = 4;      // rows of a block, a warp each
constexpr int CS_THREADS = CS_ROWS * 32;

// entries per segment loaded together; four columns take two on levels of up to
// CS_SHORT rows (175 rows 14.7 us a solve, 17.0 with four) and four above (39.9 us,
// 31.7 with four, 35.3 as a block per row)
constexpr int coarse_pf(int K) { return K == 1 ? 8 : (K == 2 ? 4 : 2); }
constexpr int64_t CS_SHORT = 512;

template <int K, int PF = coarse_pf(K)>
__device__ __forceinline__ void coarse_rows(const CoarseEnt& E, const CoarseProb& P, unsigned blk) {
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = (int)P.n;
  const int i = E.rb + (int)blk * CS_ROWS + warp;
  if (i >= E.re) {  // warp-uniform
    pdl_sync();
    return;
  }
  const int lo = E.mode == CS_W ? E.r0 : (E.mode == CS_WT ? i : (E.mode == CS_L ? 0 : E.r1));
  const int hi = E.mode == CS_W ? i + 1 : (E.mode == CS_WT ? E.r1 : (E.mode == CS_L ? E.r0 : n));
  const int seg = (((hi - lo) + CS_SEG - 1) / CS_SEG + 31) & ~31;
  int js[CS_SEG], je[CS_SEG];
  int top = hi, bot = 0;
  if (E.mode == CS_L) bot = P.F.first[i / NB] * NB;
  if (E.mode == CS_LT) top = min(hi, P.F.end[i / NB] * NB);
#pragma unroll
  for (int q = 0; q < CS_SEG; ++q) {
    const int b = lo + q * seg;
    je[q] = min(b + seg, top);
    js[q] = b + lane;
    if (js[q] < bot) js[q] += (bot - js[q] + 31) & ~31;
  }
  const double* M = E.mode == CS_W ? P.F.W : (E.mode == CS_WT ? P.F.WT : (E.mode == CS_L ? P.F.L : P.F.LT));
  const double* __restrict__ Mi = M + (int64_t)i * n;
  // columns below `split` come from va, the others from vb
  const double* va = E.mode == CS_W ? P.t : (E.mode == CS_LT ? P.x : P.y);
  const double* vb = E.mode == CS_W ? P.bin : P.t;
  double sum[CS_SEG * K];
#pragma unroll
  for (int c = 0; c < CS_SEG * K; ++c) sum[c] = 0.0;
  {
    double w[CS_SEG][PF];
#pragma unroll
    for (int q = 0; q < CS_SEG; ++q)
#pragma unroll
      for (int u = 0; u < PF; ++u) w[q][u] = js[q] + 32 * u < je[q] ? __ldcs(&Mi[js[q] + 32 * u]) : 0.0;
    pdl_sync();  // the matrix is not written by this stream's solves
    if constexpr (K == 1) {
      double v[CS_SEG][PF];
#pragma unroll
      for (int q = 0; q < CS_SEG; ++q)
#pragma unroll
        for (int u = 0; u < PF; ++u) {
          const int p = js[q] + 32 * u;
          v[q][u] = p < je[q] ? (p < E.split ? va : vb)[p] : 0.0;
        }
#pragma unroll
      for (int u = 0; u < PF; ++u)
#pragma unroll
        for (int q = 0; q < CS_SEG; ++q)
          if (js[q] + 32 * u < je[q]) sum[q] = fma(w[q][u], v[q][u], sum[q]);
    } else {
#pragma unroll
      for (int u = 0; u < PF; ++u)
#pragma unroll
        for (int q = 0; q < CS_SEG; ++q) {
          const int p = js[q] + 32 * u;
          if (p < je[q]) {
            const double* v = (p < E.split ? va : vb) + (int64_t)p * K;
#pragma unroll
            for (int c = 0; c < K; ++c) sum[q * K + c] = fma(w[q][u], v[c], sum[q * K + c]);
          }
        }
    }
  }
  // the rest of the segments, four entries of one segment at a time
#pragma unroll
  for (int q = 0; q < CS_SEG; ++q)
    for (int p = js[q] + 32 * PF; p < je[q]; p += 128) {
      double a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = p + 32 * u < je[q] ? __ldcs(&Mi[p + 32 * u]) : 0.0;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (p + 32 * u < je[q]) {
          const double* v = (p + 32 * u < E.split ? va : vb) + (int64_t)(p + 32 * u) * K;
#pragma unroll
          for (int c = 0; c < K; ++c) sum[q * K + c] = fma(a[u], v[c], sum[q * K + c]);
        }
    }
  // value q K + c ends in lane 8 q + (8 / K) c; the segments in order
  int c0;
  lane_reduce<double, CS_SEG * K, 32>(sum, lane, c0);
  double s = sum[0];
#pragma unroll
  for (int q = 1; q < CS_SEG; ++q) s += __shfl_down_sync(FULL, sum[0], 8 * q);
  if (lane < 8 && lane % (8 / K) == 0) {
    const int64_t o = (int64_t)i * K + lane / (8 / K);
    if (E.mode == CS_L) s = P.bin[o] - s;
    if (E.mode == CS_LT) s = P.y[o] - s;
    (E.mode == CS_W ? P.y : (E.mode == CS_WT ? P.x : P.t))[o] = s;
    if (E.mode == CS_WT && P.xo) {
      if (P.xo_f32) static_cast<float*>(P.xo)[o] = (float)(P.sq[i] * s);
      else static_cast<double*>(P.xo)[o] = P.sq[i] * s;
    }
  }
}

template <int K, int PF = coarse_pf(K)>
__global__ void __launch_bounds__(CS_THREADS) k_coarse(CoarseEnt E, CoarseProb P) {
  coarse_rows<K, PF>(E, P, blockIdx.x);
}

// the same step of several problems (group solve): blocks blk0 ... of entry k
__global__ void __launch_bounds__(CS_THREADS) k_g_coarse(const CoarseEnt* __restrict__ ent, int nent,
                                                         const CoarseProb* __restrict__ probs) {
  int lo = 0, hi = nent - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (ent[mid].blk0 <= (int)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const CoarseEnt E = ent[lo];
  coarse_rows<1>(E, probs[E.prob], blockIdx.x - E.blk0);
}

// the steps of one problem's solve, in order
double coarse_steps(int64_t n, const int32_t* first, const int32_t* end, std::vector<CoarseEnt>& out) {
  const int nbk = (int)((n + COARSE_BS - 1) / COARSE_BS);
  auto push = [&](int mode, int64_t rb, int64_t re, int64_t r0, int64_t r1, int64_t split) {
    if (re <= rb) return;
    CoarseEnt E = {};
    E.mode = mode;
    E.rb = (int)rb; E.re = (int)re; E.r0 = (int)r0; E.r1 = (int)r1; E.split = (int)split;
    out.push_back(E);
  };
  for (int q = 0; q < nbk; ++q) {
    const int64_t r0 = q * COARSE_BS, r1 = r0 + COARSE_BS < n ? r0 + COARSE_BS : n;
    int64_t ek = r0;  // rows [r0, ek) reach left of the block
    for (int64_t i = r0 / NB; i * NB < r1; ++i)
      if ((int64_t)first[i] * NB < r0) ek = (i + 1) * NB < r1 ? (i + 1) * NB : r1;
    push(CS_L, r0, ek, r0, r1, n);
    push(CS_W, r0, r1, r0, r1, ek);
  }
  for (int q = nbk - 1; q >= 0; --q) {
    const int64_t r0 = q * COARSE_BS, r1 = r0 + COARSE_BS < n ? r0 + COARSE_BS : n;
    int64_t sk = r1;  // rows [sk, r1) are reached from below the block
    if (r1 < n)
      for (int64_t i = (r1 - 1) / NB; i * NB >= r0 && i >= 0; --i)
        if ((int64_t)end[i] * NB > r1) sk = i * NB;
    push(CS_LT, sk, r1, r0, r1, n);
    push(CS_WT, r0, r1, r0, r1, sk);
  }
  double read = 0.0;
  for (const CoarseEnt& E : out) {
    const int64_t rows = E.re - E.rb;
    if (E.mode == CS_W || E.mode == CS_WT) {
      read += 0.5 * (double)rows * (double)(rows + 1);
      continue;
    }
    for (int64_t i = E.rb; i < E.re; ++i) {
      const int64_t in = E.mode == CS_L ? E.r0 - (int64_t)first[i / NB] * NB
                                        : ((int64_t)end[i / NB] * NB < n ? (int64_t)end[i / NB] * NB : n) - E.r1;
      read += in > 0 ? (double)in : 0.0;
    }
  }
  return read;
}

int coarse_blocks(const CoarseEnt& E) { return (E.re - E.rb + CS_ROWS - 1) / CS_ROWS; }

int launch_coarse_group(cudaStream_t st, const CoarseEnt* ent, int nent, int blocks, const CoarseProb* probs) {
  if (blocks <= 0) return SA_OK;
  launch_pdl(k_g_coarse, (unsigned)blocks, CS_THREADS, 0, st, ent, nent, probs);
  SA_LAUNCHED();
  return SA_OK;
}

int launch_coarse_solve(cudaStream_t st, int k, const CoarseProb& P) {
  if (P.n <= 0) return SA_OK;
  for (const CoarseEnt& E : *P.F.steps) {
    const unsigned g = (unsigned)coarse_blocks(E);
    switch (k) {
      case 1: launch_pdl(k_coarse<1>, g, CS_THREADS, 0, st, E, P); break;
      case 2: launch_pdl(k_coarse<2>, g, CS_THREADS, 0, st, E, P); break;
      case 4:
        if (P.n > CS_SHORT) launch_pdl(k_coarse<4, 4>, g, CS_THREADS, 0, st, E, P);
        else launch_pdl(k_coarse<4>, g, CS_THREADS, 0, st, E, P);
        break;
      case 8: launch_pdl(k_coarse<8>, g, CS_THREADS, 0, st, E, P); break;
      default: return SA_ERR_INVALID_ARG;
    }
    SA_LAUNCHED();
  }
  return SA_OK;
}

}  // namespace sa
