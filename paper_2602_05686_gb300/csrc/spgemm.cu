// Sparse matrix product C = A B used for the smoothed prolongator (A_F P^,
// Sec. 2.2) and the Galerkin product (R (A P), Sec. 2), in two phases (count,
// then fill) or in one pass into slots sized by the rows' product counts, packed
// afterwards.  Three tiers by the row's distinct column count: one thread per
// row (narrow products, e.g. the aggregation prolongators with one to a few
// entries per row) with a sorted column list in shared memory (two phases) or a
// hash table of its own (one pass: rows of up to TCAP columns leave in table
// order and the packing ranks them); then one warp per row with a hash table of
// column indices in shared memory, whose fill sorts the row's columns.  Every
// entry's products are accumulated in ascending order of the A column
// (the order of Gustavson's row algorithm), with separately rounded multiply
// and add, so the values do not depend on scheduling or form.  Rows whose distinct
// column count exceeds the table go to a block-per-row path with a dense
// accumulator in global scratch memory.
#include <stdlib.h>

#include "common.cuh"
#include "kernels.cuh"

namespace sa {

// table sizes: hash slots per warp and the distinct columns the warp tier
// holds (the Galerkin rows hold about 60; rows above go to the block tier),
// and (below) TCAP for the thread tier -- sized so that more warps stay
// resident (shared memory per warp is what limits the tiers)
constexpr int HB = 256;             // hash slots per warp
constexpr int HCAP = 192;           // max distinct columns on the warp path
static_assert(HB <= 256, "hslot gives 8 bits; slots and ranks are stored in bytes");
static_assert(HCAP + 32 < HB, "a round of 32 insertions is made before the count is checked");
constexpr int SG_WARPS = 4;         // warps per CTA
constexpr int BIG_THREADS = 512;

__device__ __forceinline__ int hslot(int32_t j) { return (int)(((uint32_t)j * 0x9E3779B1u) >> 24); }  // 8 bits

// insert j; returns 1 if newly inserted, 0 if present, -1 if the table is full
__device__ __forceinline__ int hinsert(int32_t* keys, int32_t j) {
  int h = hslot(j);
  for (int probe = 0; probe < HB; ++probe) {
    int32_t old = atomicCAS(&keys[h], -1, j);
    if (old == -1) return 1;
    if (old == j) return 0;
    h = (h + 1) & (HB - 1);
  }
  return -1;
}

__device__ __forceinline__ int hfind(const int32_t* keys, int32_t j) {
  int h = hslot(j);
  for (int probe = 0; probe < HB; ++probe) {
    int32_t k = keys[h];
    if (k == j) return h;
    if (k == -1) return -1;
    h = (h + 1) & (HB - 1);
  }
  return -1;
}

// The products of a row of A B, flattened: 32 entries of A at a time (a lane
// each: column, value, bounds of its B row), their B rows numbered through,
// lane t of a round taking product t.  One gather of row bounds per 32 entries
// and full lanes, where an entry at a time was a chain of three dependent loads
// with half the lanes idle (B rows of about 15 entries).
struct ProdChunk {
  int32_t k = 0;          // this lane's A column
  double a = 0.0;
  int64_t qb = 0;         // start of its B row
  int off = 0, tot = 0;   // first product of this lane's B row in the chunk; products of the chunk
};

__device__ __forceinline__ ProdChunk chunk_load(int64_t p0, int64_t e, const int32_t* __restrict__ Aci,
                                                const double* __restrict__ Av, const int64_t* __restrict__ Brp) {
  const int lane = lane_id();
  ProdChunk c;
  int len = 0;
  if (p0 + lane < e) {
    c.k = Aci[p0 + lane];
    if (Av) c.a = Av[p0 + lane];
    c.qb = Brp[c.k];
    len = (int)(Brp[c.k + 1] - c.qb);
  }
  int inc = len;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(FULL, inc, o);
    if (lane >= o) inc += u;
  }
  c.off = inc - len;
  c.tot = __shfl_sync(FULL, inc, 31);
  return c;
}

// the lane whose B row holds product t (< tot): the last with off <= t (of
// equal offsets the last one: empty rows share their successor's)
__device__ __forceinline__ int chunk_owner(const ProdChunk& c, int t) {
  int lo = 0;
#pragma unroll
  for (int st = 16; st > 0; st >>= 1) {
    const int o = __shfl_sync(FULL, c.off, lo + st);
    if (o <= t) lo += st;
  }
  return lo;
}

// inserts every column of row i of A*B; returns the distinct count, or -1 on
// overflow (more than HCAP distinct columns)
__device__ int warp_build_row(int64_t i, const int64_t* __restrict__ Arp, const int32_t* __restrict__ Aci,
                              const int64_t* __restrict__ Brp, const int32_t* __restrict__ Bci, int32_t* keys) {
  const int lane = lane_id();
  for (int t = lane; t < HB; t += 32) keys[t] = -1;
  __syncwarp();
  const int64_t b = Arp[i], e = Arp[i + 1];
  int total = 0;
  for (int64_t p0 = b; p0 < e && total <= HCAP; p0 += 32) {
    const ProdChunk c = chunk_load(p0, e, Aci, nullptr, Brp);
    for (int t0 = 0; t0 < c.tot && total <= HCAP; t0 += 64) {
      // two rounds' loads together
      int32_t j[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int t = t0 + 32 * u + lane;
        const int o = chunk_owner(c, t < c.tot ? t : c.tot - 1);
        const int64_t q = __shfl_sync(FULL, c.qb, o) + (t - __shfl_sync(FULL, c.off, o));
        j[u] = t < c.tot ? Bci[q] : -1;
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        // at most HCAP + 32 columns before the check: the table holds them
        int r = 0;
        if (total <= HCAP && j[u] >= 0) r = hinsert(keys, j[u]);
        total += __popc(__ballot_sync(FULL, r == 1)) + (__any_sync(FULL, r < 0) ? HCAP + 1 : 0);
      }
    }
  }
  __syncwarp();
  return total > HCAP ? -1 : total;
}

__global__ void __launch_bounds__(SG_WARPS * 32)
k_spgemm_count(int64_t n, const unsigned long long* __restrict__ nrows, const int32_t* __restrict__ rows,
               const int64_t* __restrict__ Arp,
               const int32_t* __restrict__ Aci, const int64_t* __restrict__ Brp, const int32_t* __restrict__ Bci,
               int64_t* __restrict__ cnt, int32_t* __restrict__ big, unsigned long long* __restrict__ nbig) {
  __shared__ int32_t keys_all[SG_WARPS][HB];
  const int w = threadIdx.x >> 5;
  int32_t* keys = keys_all[w];
  if (nrows) n = (int64_t)*nrows;
  for (int64_t t = global_warp(); t < n; t += warp_stride()) {
    const int64_t i = rows ? rows[t] : t;  // rows: the rows the thread tier could not hold
    int c = warp_build_row(i, Arp, Aci, Brp, Bci, keys);
    if (lane_id() == 0) {
      if (c < 0) {
        unsigned long long slot = atomicAdd(nbig, 1ull);
        big[slot] = (int32_t)i;
        cnt[i + 1] = 0;  // set by the big-row pass
      } else {
        cnt[i + 1] = c;
      }
    }
    __syncwarp();
  }
}

__global__ void __launch_bounds__(SG_WARPS * 32)
k_spgemm_fill(int64_t n, const unsigned long long* __restrict__ nrows, const int32_t* __restrict__ rows,
              const int64_t* __restrict__ Arp,
              const int32_t* __restrict__ Aci, const double* __restrict__ Av, const int64_t* __restrict__ Brp,
              const int32_t* __restrict__ Bci, const double* __restrict__ Bv, const int64_t* __restrict__ Crp,
              int32_t* __restrict__ Cci, double* __restrict__ Cv, const uint8_t* __restrict__ isbig, int upper_only,
              int32_t* __restrict__ defer, unsigned long long* __restrict__ ndefer, int64_t* __restrict__ cnt) {
  // one-pass mode (isbig NULL): Crp holds each row's upper-bound offset, a
  // row wider than the table goes to `defer` (the big tier), the distinct
  // count of every other row to cnt[i + 1]
  __shared__ int32_t keys_all[SG_WARPS][HB];
  __shared__ uint8_t rank_all[SG_WARPS][HB];
  __shared__ int32_t cols_all[SG_WARPS][HCAP];
  __shared__ uint8_t slot_all[SG_WARPS][HCAP];
  __shared__ double acc_all[SG_WARPS][HCAP];
  const int w = threadIdx.x >> 5, lane = lane_id();
  int32_t* keys = keys_all[w];
  uint8_t* rank_of = rank_all[w];
  int32_t* cols = cols_all[w];
  uint8_t* slot_of = slot_all[w];
  double* acc = acc_all[w];
  if (nrows) n = (int64_t)*nrows;
  for (int64_t t = global_warp(); t < n; t += warp_stride()) {
    const int64_t i = rows ? rows[t] : t;
    if (isbig && isbig[i]) continue;  // warp-uniform
    const int c = warp_build_row(i, Arp, Aci, Brp, Bci, keys);
    if (!isbig && lane == 0) {
      if (c < 0) defer[atomicAdd(ndefer, 1ull)] = (int32_t)i;
      else cnt[i + 1] = c;
    }
    if (c <= 0) continue;
    // compact the keys (slot order), remember each key's slot
    int out = 0;
    for (int t0 = 0; t0 < HB; t0 += 32) {
      const int32_t k = keys[t0 + lane];
      const bool has = k != -1;
      const unsigned m = __ballot_sync(FULL, has);
      if (has) {
        const int pos = out + __popc(m & ((1u << lane) - 1u));
        cols[pos] = k;
        slot_of[pos] = (uint8_t)(t0 + lane);
      }
      out += __popc(m);
    }
    __syncwarp();
    // rank sort (keys are distinct): slot -> rank in ascending column order
    const int64_t cb = Crp[i];
    for (int u = lane; u < c; u += 32) {
      const int32_t k = cols[u];
      int r = 0;
      for (int v = 0; v < c; ++v) r += cols[v] < k;
      rank_of[slot_of[u]] = (uint8_t)r;
      Cci[cb + r] = k;
      acc[u] = 0.0;
    }
    __syncwarp();
    // ordered accumulation: the products in A-column order, a round of 32 at
    // a time; lanes of one round that share an accumulator (products of
    // successive A entries) add one after the other in lane order.
    // upper_only: entries left of the diagonal stay 0 (the caller mirrors
    // the upper triangle into them)
    const int64_t b = Arp[i], e = Arp[i + 1];
    const int32_t jmin = upper_only ? (int32_t)i : 0;
    for (int64_t p0 = b; p0 < e; p0 += 32) {
      const ProdChunk pc = chunk_load(p0, e, Aci, Av, Brp);
      int32_t jn = -1;
      double vn = 0.0, an = 0.0;
      auto fetch = [&](int t0) {
        const int tt = t0 + lane;
        const int o = chunk_owner(pc, tt < pc.tot ? tt : pc.tot - 1);
        const int64_t q = __shfl_sync(FULL, pc.qb, o) + (tt - __shfl_sync(FULL, pc.off, o));
        an = __shfl_sync(FULL, pc.a, o);
        const bool in = tt < pc.tot;
        jn = in ? Bci[q] : -1;
        vn = in ? Bv[q] : 0.0;
      };
      if (pc.tot > 0) fetch(0);
      for (int t0 = 0; t0 < pc.tot; t0 += 32) {
        const int32_t j = jn;
        const double prod = __dmul_rn(an, vn);
        if (t0 + 32 < pc.tot) fetch(t0 + 32);  // the next round's loads
        int r = -1;
        if (j >= jmin) {
          const int h = hfind(keys, j);
          if (h >= 0) r = rank_of[h];  // always found: the keys were inserted from the same rows
        }
        const unsigned same = __match_any_sync(FULL, r);
        const int turn = r >= 0 ? __popc(same & ((1u << lane) - 1u)) : 0;
        const int turns = __reduce_max_sync(FULL, r >= 0 ? turn + 1 : 0);
        for (int u = 0; u < turns; ++u) {
          if (r >= 0 && turn == u) acc[r] = __dadd_rn(acc[r], prod);
          __syncwarp();
        }
      }
    }
    for (int u = lane; u < c; u += 32) Cv[cb + u] = acc[u];
    __syncwarp();
  }
}


// ---------------------------------------------------------------------------
// thread tier: one thread per row, its distinct columns kept sorted in a
// private column of shared memory (element k of thread t at [k * TB + t]);
// rows with more than TCAP distinct columns go to the warp tier
// ---------------------------------------------------------------------------
constexpr int TB = 128;
constexpr int TCAP = 24;
constexpr int TG = 4;  // A entries whose B rows are looked up together

__device__ __forceinline__ int tlower(const int32_t* cols, int c, int32_t j) {
  int lo = 0, hi = c;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (cols[mid * TB] < j) lo = mid + 1; else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(TB)
k_spgemm_tcount(int64_t n, const int64_t* __restrict__ Arp, const int32_t* __restrict__ Aci,
                const int64_t* __restrict__ Brp, const int32_t* __restrict__ Bci, int64_t* __restrict__ cnt,
                int32_t* __restrict__ mid, unsigned long long* __restrict__ nmid) {
  __shared__ int32_t cols_all[TCAP * TB];
  int32_t* cols = cols_all + threadIdx.x;
  const int64_t i = (int64_t)blockIdx.x * TB + threadIdx.x;
  if (i >= n) return;
  int c = 0;
  bool over = false;
  const int64_t e = Arp[i + 1];
  // A entries in groups of TG: their columns and B row bounds are fetched
  // together (one dependent load chain per group instead of per entry); the
  // B rows are then inserted in ascending A order
  for (int64_t p0 = Arp[i]; p0 < e && !over; p0 += TG) {
    int64_t qb[TG], qe[TG];
#pragma unroll
    for (int u = 0; u < TG; ++u) {
      qb[u] = 0;
      qe[u] = 0;
      if (p0 + u < e) {
        const int32_t k = Aci[p0 + u];
        qb[u] = Brp[k];
        qe[u] = Brp[k + 1];
      }
    }
    for (int u = 0; u < TG && !over; ++u) {
      for (int64_t q = qb[u]; q < qe[u]; ++q) {
        const int32_t j = Bci[q];
        const int pos = tlower(cols, c, j);
        if (pos < c && cols[pos * TB] == j) continue;
        if (c == TCAP) { over = true; break; }
        for (int t = c; t > pos; --t) cols[t * TB] = cols[(t - 1) * TB];
        cols[pos * TB] = j;
        ++c;
      }
    }
  }
  if (over) {
    const unsigned long long slot = atomicAdd(nmid, 1ull);
    mid[slot] = (int32_t)i;
    cnt[i + 1] = 0;  // set by the warp tier
  } else {
    cnt[i + 1] = c;
  }
}

// same insertion order as the count; each entry starts at 0 and adds its
// products in ascending A-column order (Gustavson order), like the warp tier
__global__ void __launch_bounds__(TB)
k_spgemm_tfill(int64_t n, const int64_t* __restrict__ Arp, const int32_t* __restrict__ Aci,
               const double* __restrict__ Av, const int64_t* __restrict__ Brp, const int32_t* __restrict__ Bci,
               const double* __restrict__ Bv, const int64_t* __restrict__ Crp, int32_t* __restrict__ Cci,
               double* __restrict__ Cv, const uint8_t* __restrict__ ismid, int upper_only) {
  __shared__ int32_t cols_all[TCAP * TB];
  __shared__ double vals_all[TCAP * TB];
  int32_t* cols = cols_all + threadIdx.x;
  double* vals = vals_all + threadIdx.x;
  const int64_t i = (int64_t)blockIdx.x * TB + threadIdx.x;
  if (i >= n || ismid[i]) return;
  const int32_t jmin = upper_only ? (int32_t)i : INT32_MIN;
  int c = 0;
  const int64_t e = Arp[i + 1];
  for (int64_t p0 = Arp[i]; p0 < e; p0 += TG) {
    int64_t qb[TG], qe[TG];
    double av[TG];
#pragma unroll
    for (int u = 0; u < TG; ++u) {
      qb[u] = 0;
      qe[u] = 0;
      av[u] = 0.0;
      if (p0 + u < e) {
        const int32_t k = Aci[p0 + u];
        av[u] = Av[p0 + u];
        qb[u] = Brp[k];
        qe[u] = Brp[k + 1];
      }
    }
    for (int u = 0; u < TG; ++u) {
      const double a = av[u];
      for (int64_t q = qb[u]; q < qe[u]; ++q) {
        const int32_t j = Bci[q];
        const int pos = tlower(cols, c, j);
        if (!(pos < c && cols[pos * TB] == j)) {
          if (c == TCAP) return;  // cannot happen (the count held this row)
          for (int t = c; t > pos; --t) {
            cols[t * TB] = cols[(t - 1) * TB];
            vals[t * TB] = vals[(t - 1) * TB];
          }
          cols[pos * TB] = j;
          vals[pos * TB] = 0.0;
          ++c;
        }
        if (j >= jmin) vals[pos * TB] = __dadd_rn(vals[pos * TB], __dmul_rn(a, Bv[q]));
      }
    }
  }
  const int64_t cb = Crp[i];
  for (int t = 0; t < c; ++t) {
    Cci[cb + t] = cols[t * TB];
    Cv[cb + t] = vals[t * TB];
  }
}

// the thread tier of the one-pass form: the same sums on an open-addressing
// table of TCAP slots per thread (its own column of shared memory) instead of
// the sorted list -- inserting into that list shifted up to TCAP columns and
// values, and with 32 rows a warp nearly every product met a lane that did.
// The row is written in table order; the packing pass sorts it.
__global__ void __launch_bounds__(TB)
k_spgemm_thash(int64_t n, const int64_t* __restrict__ Arp, const int32_t* __restrict__ Aci,
               const double* __restrict__ Av, const int64_t* __restrict__ Brp, const int32_t* __restrict__ Bci,
               const double* __restrict__ Bv, const int64_t* __restrict__ ub, int32_t* __restrict__ Cci,
               double* __restrict__ Cv, int upper_only, int32_t* __restrict__ defer,
               unsigned long long* __restrict__ ndefer, int64_t* __restrict__ cnt) {
  __shared__ int32_t cols_all[TCAP * TB];
  __shared__ double vals_all[TCAP * TB];
  int32_t* cols = cols_all + threadIdx.x;
  double* vals = vals_all + threadIdx.x;
  const int64_t i = (int64_t)blockIdx.x * TB + threadIdx.x;
  if (i >= n) return;
#pragma unroll
  for (int t = 0; t < TCAP; ++t) cols[t * TB] = -1;
  const int32_t jmin = upper_only ? (int32_t)i : 0;
  int c = 0;
  const int64_t e = Arp[i + 1];
  for (int64_t p0 = Arp[i]; p0 < e; p0 += TG) {
    int64_t qb[TG], qe[TG];
    double av[TG];
#pragma unroll
    for (int u = 0; u < TG; ++u) {
      qb[u] = 0;
      qe[u] = 0;
      av[u] = 0.0;
      if (p0 + u < e) {
        const int32_t k = Aci[p0 + u];
        av[u] = Av[p0 + u];
        qb[u] = Brp[k];
        qe[u] = Brp[k + 1];
      }
    }
#pragma unroll
    for (int u = 0; u < TG; ++u) {
      const double a = av[u];
      for (int64_t q0 = qb[u]; q0 < qe[u]; q0 += TG) {
        // B entries of one row in groups, loaded together
        int32_t jj[TG];
        double bv[TG];
#pragma unroll
        for (int v = 0; v < TG; ++v) {
          const bool in = q0 + v < qe[u];
          jj[v] = in ? Bci[q0 + v] : -1;
          bv[v] = in ? Bv[q0 + v] : 0.0;
        }
#pragma unroll
        for (int v = 0; v < TG; ++v) {
          const int32_t j = jj[v];
          if (j >= 0) {
            int h = (int)__umulhi((uint32_t)j * 0x9E3779B1u, (uint32_t)TCAP);
            int32_t k = cols[h * TB];
            while (k != j && k != -1) {
              h = h + 1 < TCAP ? h + 1 : 0;
              k = cols[h * TB];
              // (a full table without j: every slot holds another column)
              if (c == TCAP && h == (int)__umulhi((uint32_t)j * 0x9E3779B1u, (uint32_t)TCAP)) break;
            }
            if (k != j) {
              if (c == TCAP) {
                defer[atomicAdd(ndefer, 1ull)] = (int32_t)i;
                return;
              }
              cols[h * TB] = j;
              vals[h * TB] = 0.0;
              ++c;
            }
            if (j >= jmin) vals[h * TB] = __dadd_rn(vals[h * TB], __dmul_rn(a, bv[v]));
          }
        }
      }
    }
  }
  int64_t o = ub[i];
#pragma unroll
  for (int t = 0; t < TCAP; ++t) {
    const int32_t j = cols[t * TB];
    if (j >= 0) {
      Cci[o] = j;
      Cv[o] = vals[t * TB];
      ++o;
    }
  }
  cnt[i + 1] = c;
}

// ---------------------------------------------------------------------------
// big rows: one CTA per row with a dense accumulator of width m in global
// scratch (stamp[m] holds the row currently using a column)
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t block_excl_scan_count(int flag, int* sh, int* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned m = __ballot_sync(FULL, flag);
  int before = __popc(m & ((1u << lane) - 1u));
  if (lane == 0) sh[w] = __popc(m);
  __syncthreads();
  if (threadIdx.x == 0) {
    int run = 0;
    for (int k = 0; k < nw; ++k) { int t = sh[k]; sh[k] = run; run += t; }
    sh[nw] = run;
  }
  __syncthreads();
  int r = sh[w] + before;
  *total = sh[nw];
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(BIG_THREADS)
k_spgemm_big(int phase, int64_t nbig, const int32_t* __restrict__ big, int64_t m,
             const int64_t* __restrict__ Arp, const int32_t* __restrict__ Aci, const double* __restrict__ Av,
             const int64_t* __restrict__ Brp, const int32_t* __restrict__ Bci, const double* __restrict__ Bv,
             int64_t* __restrict__ cnt, const int64_t* __restrict__ Crp, int32_t* __restrict__ Cci,
             double* __restrict__ Cv, int32_t* __restrict__ stamp_all, double* __restrict__ acc_all) {
  __shared__ int sh[BIG_THREADS / 32 + 1];
  int32_t* stamp = stamp_all + (int64_t)blockIdx.x * m;
  double* acc = acc_all + (int64_t)blockIdx.x * m;
  for (int64_t t = blockIdx.x; t < nbig; t += gridDim.x) {
    const int32_t i = big[t];
    const int64_t b = Arp[i], e = Arp[i + 1];
    for (int64_t p = b; p < e; ++p) {
      const int32_t k = Aci[p];
      const double a = phase ? Av[p] : 0.0;
      for (int64_t q = Brp[k] + threadIdx.x; q < Brp[k + 1]; q += blockDim.x) {
        const int32_t j = Bci[q];
        if (stamp[j] != i) {
          stamp[j] = i;
          acc[j] = 0.0;
        }
        if (phase) acc[j] = __dadd_rn(acc[j], __dmul_rn(a, Bv[q]));
      }
      __syncthreads();
    }
    // compact in ascending column order
    int64_t run = 0;
    for (int64_t j0 = 0; j0 < m; j0 += blockDim.x) {
      int64_t j = j0 + threadIdx.x;
      int f = (j < m && stamp[j] == i) ? 1 : 0;
      int tot;
      int r = (int)block_excl_scan_count(f, sh, &tot);
      if (phase && f) {
        Cci[Crp[i] + run + r] = (int32_t)j;
        Cv[Crp[i] + run + r] = acc[j];
      }
      run += tot;
    }
    if (cnt && threadIdx.x == 0) cnt[i + 1] = run;  // count pass, or the one-pass fill
    // release the stamps of this row
    for (int64_t j = threadIdx.x; j < m; j += blockDim.x)
      if (stamp[j] == i) stamp[j] = -1;
    __syncthreads();
  }
}

__global__ void k_mark_big(const unsigned long long* __restrict__ nbig, const int32_t* __restrict__ big,
                           uint8_t* __restrict__ isbig) {
  const int64_t n = (int64_t)*nbig;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    isbig[big[t]] = 1;
}

// products of each row of A B (an upper bound of its distinct columns)
__global__ void k_spgemm_pcount(int64_t n, const int64_t* __restrict__ Arp, const int32_t* __restrict__ Aci,
                                const int64_t* __restrict__ Brp, int64_t* __restrict__ ub) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int64_t t = 0;
  for (int64_t p = Arp[i]; p < Arp[i + 1]; ++p) {
    const int32_t k = Aci[p];
    t += Brp[k + 1] - Brp[k];
  }
  ub[i + 1] = t;
}

// rows from their upper-bound slots to the packed CSR (a warp per row); rows of
// up to 32 columns are ranked on the way (the thread tier leaves them in table
// order), longer ones come sorted
static_assert(TCAP <= 32, "the packing ranks the thread tier's rows by one warp");
__global__ void k_spgemm_compact(int64_t n, const int64_t* __restrict__ ub, const int32_t* __restrict__ uci,
                                 const double* __restrict__ uv, const int64_t* __restrict__ Crp,
                                 int32_t* __restrict__ Cci, double* __restrict__ Cv) {
  const int lane = lane_id();
  for (int64_t i = global_warp(); i < n; i += warp_stride()) {
    const int64_t src = ub[i], dst = Crp[i], c = Crp[i + 1] - dst;
    if (c <= 32) {
      const int32_t k = lane < c ? uci[src + lane] : INT32_MAX;
      int r = 0;
      for (int t = 0; t < (int)c; ++t) r += __shfl_sync(FULL, k, t) < k;
      if (lane < c) {
        Cci[dst + r] = k;
        Cv[dst + r] = uv[src + lane];
      }
      continue;
    }
    for (int64_t t = lane; t < c; t += 32) {
      Cci[dst + t] = uci[src + t];
      Cv[dst + t] = uv[src + t];
    }
  }
}

// blocks of a warp-tier launch: every row, or (row count on the device) as many
// as stay resident
static unsigned warp_tier_grid(int64_t n, bool listed) {
  const unsigned g = warp_rows_grid(n, SG_WARPS * 32), r = 16u * (unsigned)num_sms();
  return listed && g > r ? r : g;
}

static int spgemm_two_phase(Alloc& al, int64_t n, int64_t m, const int64_t* Arp, const int32_t* Aci,
                            const double* Av, const int64_t* Brp, const int32_t* Bci, const double* Bv,
                            Buf<int64_t>& Crp, Buf<int32_t>& Cci, Buf<double>& Cv, int64_t* nnzC, int upper_only,
                            bool thread_tier) {
  cudaStream_t s = al.stream;
  Buf<int32_t> big, midl;
  Buf<unsigned long long> nbig_d, nmid_d;
  Buf<uint8_t> isbig, ismid;
  SA_TRY(big.alloc(&al, n));
  SA_TRY(nbig_d.alloc(&al, 1));
  SA_TRY(isbig.alloc(&al, n));
  SA_TRY(memset_d(nbig_d.p, 0, sizeof(unsigned long long), s));
  SA_TRY(memset_d(isbig.p, 0, isbig.bytes(), s));
  // the rows the thread tier could not hold are counted on the device: the
  // warp tier's launches read the count instead of the host
  const int32_t* wrows = nullptr;  // NULL: every row
  const unsigned long long* nwrows = nullptr;
  const unsigned wgrid = warp_tier_grid(n, thread_tier);
  if (thread_tier) {
    SA_TRY(midl.alloc(&al, n));
    SA_TRY(nmid_d.alloc(&al, 1));
    SA_TRY(ismid.alloc(&al, n));
    SA_TRY(memset_d(nmid_d.p, 0, sizeof(unsigned long long), s));
    SA_TRY(memset_d(ismid.p, 0, ismid.bytes(), s));
    k_spgemm_tcount<<<blocks_for(n, TB), TB, 0, s>>>(n, Arp, Aci, Brp, Bci, Crp.p, midl.p, nmid_d.p);
    SA_LAUNCHED();
    wrows = midl.p;
    nwrows = nmid_d.p;
    k_mark_big<<<(unsigned)num_sms(), 256, 0, s>>>(nmid_d.p, midl.p, ismid.p);
    SA_LAUNCHED();
  }
  k_spgemm_count<<<wgrid, SG_WARPS * 32, 0, s>>>(n, nwrows, wrows, Arp, Aci, Brp, Bci, Crp.p, big.p, nbig_d.p);
  SA_LAUNCHED();
  unsigned long long nbig = 0;
  SA_TRY(copy_d2h(&nbig, nbig_d.p, sizeof(nbig), s));
  Buf<int32_t> stamp;
  Buf<double> dacc;
  unsigned gbig = 0;
  if (nbig > 0) {
    gbig = (unsigned)(nbig < 64 ? nbig : 64);
    SA_TRY(stamp.alloc(&al, (int64_t)gbig * m));
    SA_TRY(dacc.alloc(&al, (int64_t)gbig * m));
    SA_TRY(memset_d(stamp.p, 0xff, stamp.bytes(), s));
    k_mark_big<<<(unsigned)num_sms(), 256, 0, s>>>(nbig_d.p, big.p, isbig.p);
    SA_LAUNCHED();
    k_spgemm_big<<<gbig, BIG_THREADS, 0, s>>>(0, (int64_t)nbig, big.p, m, Arp, Aci, Av, Brp, Bci, Bv, Crp.p,
                                                nullptr, nullptr, nullptr, stamp.p, dacc.p);
    SA_LAUNCHED();
  }
  SA_TRY(scan_inplace(al, Crp.p + 1, n));
  SA_TRY(copy_d2h(nnzC, Crp.p + n, sizeof(int64_t), s));
  SA_TRY(Cci.alloc(&al, *nnzC));
  SA_TRY(Cv.alloc(&al, *nnzC));
  if (thread_tier) {
    k_spgemm_tfill<<<blocks_for(n, TB), TB, 0, s>>>(n, Arp, Aci, Av, Brp, Bci, Bv, Crp.p, Cci.p, Cv.p, ismid.p,
                                                    upper_only);
    SA_LAUNCHED();
  }
  k_spgemm_fill<<<wgrid, SG_WARPS * 32, 0, s>>>(n, nwrows, wrows, Arp, Aci, Av, Brp, Bci, Bv, Crp.p, Cci.p, Cv.p,
                                                isbig.p, upper_only, nullptr, nullptr, nullptr);
  SA_LAUNCHED();
  if (nbig > 0) {
    k_spgemm_big<<<gbig, BIG_THREADS, 0, s>>>(1, (int64_t)nbig, big.p, m, Arp, Aci, Av, Brp, Bci, Bv, nullptr,
                                                Crp.p, Cci.p, Cv.p, stamp.p, dacc.p);
    SA_LAUNCHED();
  }
  return SA_OK;
}

// One pass: every row is filled once into slots sized by its product count
// (ub, exclusive offsets), its distinct count recorded, and the rows are then
// packed.  Same tiers, same per-entry arithmetic and column order as the
// two-phase form (bitwise the same C); the count pass over every product is
// saved for 12 bytes of scratch per product.
static int spgemm_one_pass(Alloc& al, int64_t n, int64_t m, const int64_t* Arp, const int32_t* Aci,
                           const double* Av, const int64_t* Brp, const int32_t* Bci, const double* Bv,
                           const int64_t* ub, int64_t ubtot, Buf<int64_t>& Crp, Buf<int32_t>& Cci, Buf<double>& Cv,
                           int64_t* nnzC, int upper_only, bool thread_tier) {
  cudaStream_t s = al.stream;
  Buf<int32_t> uci, defw, defb;
  Buf<double> uv;
  Buf<unsigned long long> nd;
  SA_TRY(uci.alloc(&al, ubtot));
  SA_TRY(uv.alloc(&al, ubtot));
  SA_TRY(defw.alloc(&al, n));
  SA_TRY(defb.alloc(&al, n));
  SA_TRY(nd.alloc(&al, 2));
  SA_TRY(memset_d(nd.p, 0, nd.bytes(), s));
  const int32_t* wrows = nullptr;
  const unsigned long long* nwrows = nullptr;  // counted on the device (as above)
  if (thread_tier) {
    k_spgemm_thash<<<blocks_for(n, TB), TB, 0, s>>>(n, Arp, Aci, Av, Brp, Bci, Bv, ub, uci.p, uv.p, upper_only,
                                                    defw.p, nd.p, Crp.p);
    SA_LAUNCHED();
    wrows = defw.p;
    nwrows = nd.p;
  }
  unsigned long long nbig = 0;
  k_spgemm_fill<<<warp_tier_grid(n, thread_tier), SG_WARPS * 32, 0, s>>>(n, nwrows, wrows, Arp, Aci, Av, Brp, Bci, Bv,
                                                                        ub, uci.p, uv.p, nullptr, upper_only, defb.p,
                                                                        nd.p + 1, Crp.p);
  SA_LAUNCHED();
  SA_TRY(copy_d2h(&nbig, nd.p + 1, sizeof(nbig), s));
  if (nbig > 0) {
    const unsigned gbig = (unsigned)(nbig < 64 ? nbig : 64);
    Buf<int32_t> stamp;
    Buf<double> dacc;
    SA_TRY(stamp.alloc(&al, (int64_t)gbig * m));
    SA_TRY(dacc.alloc(&al, (int64_t)gbig * m));
    SA_TRY(memset_d(stamp.p, 0xff, stamp.bytes(), s));
    k_spgemm_big<<<gbig, BIG_THREADS, 0, s>>>(1, (int64_t)nbig, defb.p, m, Arp, Aci, Av, Brp, Bci, Bv, Crp.p, ub,
                                                uci.p, uv.p, stamp.p, dacc.p);
    SA_LAUNCHED();
  }
  SA_TRY(scan_inplace(al, Crp.p + 1, n));
  SA_TRY(copy_d2h(nnzC, Crp.p + n, sizeof(int64_t), s));
  SA_TRY(Cci.alloc(&al, *nnzC));
  SA_TRY(Cv.alloc(&al, *nnzC));
  k_spgemm_compact<<<warp_rows_grid(n), 256, 0, s>>>(n, ub, uci.p, uv.p, Crp.p, Cci.p, Cv.p);
  SA_LAUNCHED();
  return SA_OK;
}

int run_spgemm(Alloc& al, int64_t n, int64_t m, int64_t kdim, int64_t nnzA, int64_t nnzB, const int64_t* Arp, const int32_t* Aci,
               const double* Av, const int64_t* Brp, const int32_t* Bci, const double* Bv, Buf<int64_t>& Crp,
               Buf<int32_t>& Cci, Buf<double>& Cv, int64_t* nnzC, int upper_only) {
  cudaStream_t s = al.stream;
  SA_TRY(Crp.alloc(&al, n + 1));
  SA_TRY(memset_d(Crp.p, 0, Crp.bytes(), s));
  *nnzC = 0;
  if (n <= 0) {
    SA_TRY(Cci.alloc(&al, 0));
    SA_TRY(Cv.alloc(&al, 0));
    return SA_OK;
  }
  // tier choice by the expected products per row, (nnz(A)/n) (nnz(B)/kdim),
  // an upper bound of the distinct columns (FE products repeat columns
  // about 8 times: 90 products per row give about 11 distinct columns in the
  // aggregation prolongators); wide products go straight to the warp tier
  const double per_row = kdim > 0 ? ((double)nnzA / (double)n) * ((double)nnzB / (double)kdim) : 0.0;
  const bool thread_tier = kdim > 0 && per_row <= 256.0;
  // one pass for wide products (48 or more per row expected: the Galerkin
  // products; measured slower than count-then-fill at 27 per row, the
  // smoothed prolongator, where the count pass is cheap) when the
  // upper-bound slots (12 bytes per product) fit in half of the device's free
  // memory and can be had; else count then fill (SA_SPGEMM_PASSES=2 in the
  // environment forces that, for its tests)
  const char* passes = getenv("SA_SPGEMM_PASSES");
  if ((passes && passes[0] == '2') || per_row < 48.0)
    return spgemm_two_phase(al, n, m, Arp, Aci, Av, Brp, Bci, Bv, Crp, Cci, Cv, nnzC, upper_only, thread_tier);
  Buf<int64_t> ub;
  SA_TRY(ub.alloc(&al, n + 1));
  SA_TRY(memset_d(ub.p, 0, sizeof(int64_t), s));
  k_spgemm_pcount<<<blocks_for(n, 256), 256, 0, s>>>(n, Arp, Aci, Brp, ub.p);
  SA_LAUNCHED();
  SA_TRY(scan_inplace(al, ub.p + 1, n));
  int64_t ubtot = 0;
  SA_TRY(copy_d2h(&ubtot, ub.p + n, sizeof(int64_t), s));
  // (the query takes 20 us; 16 MB are taken without it)
  size_t fr = 0, tot = 0;
  const bool little = (double)ubtot * 12.0 <= 16e6;
  if (!little && cudaMemGetInfo(&fr, &tot) != cudaSuccess) {
    cudaGetLastError();
    fr = 0;
  }
  if (little || (double)ubtot * 12.0 <= 0.5 * (double)fr) {
    const int st = spgemm_one_pass(al, n, m, Arp, Aci, Av, Brp, Bci, Bv, ub.p, ubtot, Crp, Cci, Cv, nnzC, upper_only,
                                   thread_tier);
    if (st != SA_ERR_OOM) return st;
    // the scratch was not to be had (a nearly full device, an allocator's
    // limit): count then fill does without it
    SA_TRY(memset_d(Crp.p, 0, Crp.bytes(), s));
  }
  ub.release();
  return spgemm_two_phase(al, n, m, Arp, Aci, Av, Brp, Bci, Bv, Crp, Cci, Cv, nnzC, upper_only, thread_tier);
}

// ---------------------------------------------------------------------------
// exact symmetry of the coarse operator: lower-triangle entries take the
// value of the mirrored upper-triangle entry (found by binary search).
// err bit 16: the pattern is not structurally symmetric.
// ---------------------------------------------------------------------------
__global__ void k_symmetrize(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                             double* __restrict__ v, int* __restrict__ err) {
  const int lane = lane_id();
  for (int64_t i = global_warp(); i < n; i += warp_stride()) {
    for (int64_t p = rp[i] + lane; p < rp[i + 1]; p += 32) {
      int32_t j = ci[p];
      if (j >= (int32_t)i) continue;
      int64_t lo = rp[j], hi = rp[j + 1] - 1, f = -1;
      while (lo <= hi) {
        int64_t mid = (lo + hi) >> 1;
        int32_t c = ci[mid];
        if (c == (int32_t)i) { f = mid; break; }
        if (c < (int32_t)i) lo = mid + 1; else hi = mid - 1;
      }
      if (f < 0) atomicOr(err, 16);
      else v[p] = v[f];
    }
  }
}

int launch_symmetrize(cudaStream_t s, int64_t n, const int64_t* rp, const int32_t* ci, double* v, int* err) {
  if (n <= 0) return SA_OK;
  k_symmetrize<<<warp_rows_grid(n), 256, 0, s>>>(n, rp, ci, v, err);
  SA_LAUNCHED();
  return SA_OK;
}

}  // namespace sa
