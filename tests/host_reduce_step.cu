// Runs the scalar step after a reduction (reduce.cuh, fin_step) on the host, its
// sums against an unreadable page: a read past them ends the program.  Prints
// nothing and exits 0 when every value is right.
#include <math.h>
#include <stdio.h>
#include <string.h>
#include <sys/mman.h>
#include <unistd.h>

#include "reduce.cuh"

using namespace sa;

static double* guarded(int n) {
  const size_t pg = (size_t)sysconf(_SC_PAGESIZE);
  char* p = (char*)mmap(nullptr, 2 * pg, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
  if (p == MAP_FAILED || mprotect(p + pg, pg, PROT_NONE) != 0) _exit(3);
  return (double*)(p + pg) - n;
}

#define CHECK(c)                                  \
  do {                                            \
    if (!(c)) {                                   \
      fprintf(stderr, "line %d: %s\n", __LINE__, #c); \
      return 1;                                   \
    }                                             \
  } while (0)

// a block of k columns (0: one vector), all values distinct
template <int NV, int OFF2>
static int beta(int k, int flexible) {
  double* res = guarded(NV);
  for (int c = 0; c < NV; ++c) res[c] = 3.0 + c;
  double out[16];
  CgScalars cg[KMAX_BLOCK];
  int active[KMAX_BLOCK];
  for (int c = 0; c < KMAX_BLOCK; ++c) {
    cg[c] = CgScalars();
    cg[c].rz = 2.0 + c;
    cg[c].beta = -1.0;
    active[c] = c != 1;
  }
  Fin f;
  f.op = FIN_BETA;
  f.out = out;
  f.cg = cg;
  f.k = k;
  f.active = active;
  f.flexible = flexible;
  for (int t = 511; t >= 0; --t) fin_step<NV, OFF2>(f, res, t);
  for (int c = 0; c < NV; ++c) CHECK(out[c] == res[c]);
  for (int c = 0; c < KMAX_BLOCK; ++c) {
    const bool on = k > 0 ? c < k && active[c] : c == 0;
    const double zr = OFF2 > 0 && flexible > 0 ? res[OFF2 + c < NV ? OFF2 + c : NV - 1] : 0.0;
    const double b = !on ? -1.0 : flexible < 0 ? 0.0 : (res[c] - zr) / (2.0 + c);
    CHECK(cg[c].beta == b && cg[c].rz == (on ? res[c] : 2.0 + c));
  }
  return 0;
}

int main() {
  for (int flexible = -1; flexible <= 0; ++flexible) {
    if (beta<1, 0>(0, flexible)) return 1;
    for (int k = 2; k <= KMAX_BLOCK; k *= 2)
      if (beta<KMAX_BLOCK, 0>(k, flexible)) return 1;
  }
  for (int flexible = -1; flexible <= 1; ++flexible) {
    if (beta<2, 1>(0, flexible)) return 1;
    for (int k = 2; k <= KMAX_BLOCK; k *= 2)
      if (beta<2 * KMAX_BLOCK, KMAX_BLOCK>(k, flexible)) return 1;
  }
  return 0;
}
