// sqrt_rcp.cuh against sqrt() and a division, bit for bit.
//   pivot host: the settled result on the host, from a starting value up to four
//               units off;
//   pivot gpu:  sqrt_rcp itself on the GPU, fallback operands included.
// Prints the first operands that differ; exits 0 when none does.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include "sqrt_rcp.cuh"

using namespace sa;

__host__ __device__ inline uint64_t mix(uint64_t x) {  // splitmix64 (Vigna, public domain)
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}

// operand t: random significands at every exponent; neighbours of powers of two;
// neighbours of exact squares; neighbours of reciprocals of such
__host__ __device__ inline uint64_t operand(uint64_t t) {
  const uint64_t h = mix(t), ex = 1 + (t / 4) % 2046;
  const uint64_t near = h % 9;  // 0 .. 8: four below to four above
  switch (t % 4) {
    case 0: return (ex << 52) | (h >> 12);
    case 1: {
      const uint64_t b = (ex << 52) + near;
      return b > (1ull << 52) + 4 ? b - 4 : b;
    }
    case 2: {
      const double q = (double)(1 + (h >> 38));  // 26 bits: the square is exact
      return f64_bits(q * q) + near - 4;
    }
    default: return f64_bits(1.0 + (double)(h >> 38) * 0x1p-26) + ((uint64_t)(ex % 1000) << 52) - (500ull << 52);
  }
}

static int host() {
  int bad = 0;
  for (uint64_t t = 0; t < 8000000; ++t) {
    const uint64_t db = operand(t);
    const double d = f64_of(db);
    uint32_t fb = rsqrt_arg(db);
    float f;
    memcpy(&f, &fb, 4);
    const float y = (float)(1.0 / sqrt((double)f));
    uint32_t yb;
    memcpy(&yb, &y, 4);
    yb += (uint32_t)(mix(~t) % 9) - 4;
    double s, r;
    sqrt_rcp_from(db, yb, s, r);
    const double s0 = sqrt(d), r0 = 1.0 / s0;
    if (f64_bits(s) != f64_bits(s0) || f64_bits(r) != f64_bits(r0))
      if (++bad < 10) printf("%a from %a: %a %a, not %a %a\n", d, y, s, r, s0, r0);
  }
  return bad != 0;
}

__global__ void k_check(uint64_t t0, uint64_t n, unsigned long long* bad, double* first) {
  for (uint64_t t = t0 + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < t0 + n;
       t += (uint64_t)gridDim.x * blockDim.x) {
    uint64_t db = operand(t);
    if (t % 1024 == 0) db = mix(t) >> 12;           // subnormal (or zero)
    if (t % 1024 == 1) db = 0x7ff0000000000000ull;  // infinity
    const double d = f64_of(db);
    double s, r;
    sqrt_rcp(d, s, r);
    const double s0 = sqrt(d), r0 = 1.0 / s0;
    if ((f64_bits(s) != f64_bits(s0) || f64_bits(r) != f64_bits(r0)) && atomicAdd(bad, 1ull) == 0) *first = d;
  }
}

static int gpu() {
  unsigned long long* bad;
  double* first;
  unsigned long long h = 1;
  double d = 0.0;
  if (cudaMalloc(&bad, 8) != cudaSuccess || cudaMalloc(&first, 8) != cudaSuccess) return 2;
  if (cudaMemset(bad, 0, 8) != cudaSuccess) return 2;
  k_check<<<608, 256>>>(0, 200000000ull, bad, first);
  if (cudaMemcpy(&h, bad, 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  if (h && cudaMemcpy(&d, first, 8, cudaMemcpyDeviceToHost) == cudaSuccess) printf("%llu differ, one is %a\n", h, d);
  return h != 0;
}

int main(int argc, char** argv) { return argc > 1 && !strcmp(argv[1], "gpu") ? gpu() : host(); }
