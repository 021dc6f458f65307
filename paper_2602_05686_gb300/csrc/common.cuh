// Internal helpers shared by the CUDA translation units of the library:
// status handling, the device allocator, launch geometry and warp utilities.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

#include "sa.h"

namespace sa {

// ---------------------------------------------------------------------------
// status handling
// ---------------------------------------------------------------------------
void set_cuda_error(cudaError_t e, const char* what);
void set_error_text(const char* text);

#define SA_CUDA(call)                                   \
  do {                                                  \
    cudaError_t _e = (call);                            \
    if (_e != cudaSuccess) {                            \
      ::sa::set_cuda_error(_e, #call);                  \
      return SA_ERR_CUDA;                               \
    }                                                   \
  } while (0)

#define SA_TRY(call)              \
  do {                            \
    int _s = (call);              \
    if (_s != SA_OK) return _s;   \
  } while (0)

// after every kernel launch: error check + launch count
void count_launch();
void count_launches(long long k);  // k may be negative (kernels captured into a graph, not run)
long long launch_counter();
#define SA_LAUNCHED()        \
  do {                       \
    ::sa::count_launch();    \
    SA_CUDA(cudaGetLastError()); \
  } while (0)

// ---------------------------------------------------------------------------
// device memory: stream-ordered, optionally through a caller allocator
// ---------------------------------------------------------------------------
struct Alloc {
  cudaStream_t stream = nullptr;
  void* (*fn_alloc)(size_t, void*) = nullptr;
  void (*fn_free)(void*, void*) = nullptr;
  void* ctx = nullptr;
  int64_t live_bytes = 0;
  int64_t peak_bytes = 0;

  int get(void** p, size_t bytes);
  void put(void* p, size_t bytes);
};

// typed buffer owned by an Alloc
template <typename T>
struct Buf {
  T* p = nullptr;
  int64_t n = 0;
  Alloc* a = nullptr;
  Buf() = default;
  Buf(const Buf&) = delete;
  Buf& operator=(const Buf&) = delete;
  Buf(Buf&& o) noexcept { p = o.p; n = o.n; a = o.a; o.p = nullptr; o.n = 0; }
  Buf& operator=(Buf&& o) noexcept {
    if (this != &o) { release(); p = o.p; n = o.n; a = o.a; o.p = nullptr; o.n = 0; }
    return *this;
  }
  ~Buf() { release(); }
  int alloc(Alloc* al, int64_t count) {
    release();
    a = al;
    n = count;
    void* q = nullptr;
    int st = al->get(&q, sizeof(T) * (size_t)(count > 0 ? count : 1));
    p = static_cast<T*>(q);
    return st;
  }
  void release() {
    if (p && a) a->put(p, sizeof(T) * (size_t)(n > 0 ? n : 1));
    p = nullptr;
    n = 0;
  }
  size_t bytes() const { return sizeof(T) * (size_t)(n > 0 ? n : 1); }
};

// ---------------------------------------------------------------------------
// launch geometry
// ---------------------------------------------------------------------------
int num_sms();
inline unsigned blocks_for(int64_t threads, int block) {
  int64_t b = (threads + block - 1) / block;
  if (b < 1) b = 1;
  if (b > 0x7fffffffLL) b = 0x7fffffffLL;
  return (unsigned)b;
}
// grid of `block`-thread CTAs that gives one warp per row (grid-stride inside)
inline unsigned warp_rows_grid(int64_t rows, int block = 256) {
  int64_t warps = rows;
  int64_t cap = (int64_t)num_sms() * 32 * (2048 / block);  // a few waves
  if (warps > cap * (block / 32)) warps = cap * (block / 32);
  return blocks_for(warps * 32, block);
}

// Programmatic dependent launch: a kernel launched by launch_pdl may start while
// its predecessor in the stream drains, and waits in pdl_sync() for that
// predecessor's completion.  The trigger follows the wait, so no kernel starts
// before the one before its predecessor has ended.  What a kernel launched this
// way has to keep to:
// - Before its wait a thread reads only what was complete two launches (or a
//   copy) earlier: matrices, row pointers, factors and launch descriptors, read
//   ahead by the row kernels.  A kernel that builds such data is therefore
//   followed by another launch before the first that reads it early.
// - Whatever the stream's solves write -- vectors, CG scalars, partial sums -- is
//   touched after the wait only.  The predecessor may still write it while this
//   kernel is alive, so it is not read-only data: such pointers carry no
//   __restrict__ and are read with plain loads; __ldg, ld.global.nc and const
//   __restrict__ are for matrices, scalings and descriptors.
// - At least one thread of the grid waits (threads and blocks without a row of
//   their own may leave at once): the grid's end then still follows its
//   predecessor's, which the kernel after it relies on.
// The launches of one V-cycle on small levels are 2 to 4 us of work with 1.3 us
// between them.
template <typename... P, typename... A>
inline void launch_pdl(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}
__device__ __forceinline__ void pdl_sync() {
  asm volatile("griddepcontrol.wait;\ngriddepcontrol.launch_dependents;" ::: "memory");
}

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }
__device__ __forceinline__ int64_t global_warp() {
  return ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
}
__device__ __forceinline__ int64_t warp_stride() { return ((int64_t)gridDim.x * blockDim.x) >> 5; }

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}

// Reduction of the K per-lane partial sums over the W lanes of one row.  The
// one-vector kernels add a row's lane sums by the butterfly xor W/2, ..., 1;
// here every exchange also halves the columns a lane carries (a lane keeps
// the lower or upper half and receives its partner's values of that half),
// so each column is added in exactly the butterfly's tree -- bitwise the
// one-vector sum -- with K/2 + K/4 + ... additions per lane instead of
// K log2(W).  On return the lane holds the sums of columns c0 .. c0+V-1 in
// acc[0 .. V); V = K/W when K >= W, else 1 (then lanes whose low bits
// (lane mod W/K) are not zero hold copies).
template <typename T, int K, int W>
__device__ __forceinline__ int lane_reduce(T (&acc)[K], int lane, int& c0) {
  int V = K;
  c0 = 0;
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) {
    if (V > 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int j = 0; j < K / 2; ++j) {
        if (j < V / 2) {
          const T send = up ? acc[j] : acc[j + V / 2];
          const T keep = up ? acc[j + V / 2] : acc[j];
          acc[j] = keep + __shfl_xor_sync(FULL, send, o, W);
        }
      }
      if (up) c0 += V / 2;
      V /= 2;
    } else {
      acc[0] += __shfl_xor_sync(FULL, acc[0], o, W);
    }
  }
  return V;
}

// ---------------------------------------------------------------------------
// primitives (prim.cu)
// ---------------------------------------------------------------------------
// in-place inclusive prefix sum of a[0..n) (int64)
int scan_inplace(Alloc& al, int64_t* a, int64_t n);
// fixed-order reductions: partial sums per CTA of a fixed grid, then one CTA
// sums the partials in index order; deterministic for a given n.
constexpr int RED_BLOCKS = 304;   // 2 x 152 SMs
constexpr int RED_THREADS = 512;
// device values to the host, waited for; several with one wait
struct ReadBack {
  void* dst;
  const void* src;
  size_t bytes;
};
int read_back(const ReadBack* r, int count, cudaStream_t s);
int copy_d2h(void* dst, const void* src, size_t bytes, cudaStream_t s);
int copy_h2d(void* dst, const void* src, size_t bytes, cudaStream_t s);
int memset_d(void* dst, int v, size_t bytes, cudaStream_t s);

}  // namespace sa
