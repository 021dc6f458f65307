// The coarse factor's launch (dense.cu) on a 96 x 96 matrix: as it is; then with
// a first task that no block takes, so that every wait for its tile runs out;
// then as it is again.  Exits 0 when the second launch ends by itself with the
// error bit of a wait and the others with the factor.
#include <stdio.h>

#include "dense.cu"

using namespace sa;

#define CK(c)                                        \
  do {                                               \
    if (!(c)) {                                      \
      fprintf(stderr, "line %d: %s\n", __LINE__, #c); \
      return 1;                                      \
    }                                                \
  } while (0)

int main() {
  constexpr int N = 96, T = N / NB;
  std::vector<double> A(N * N), L(N * N);
  for (int i = 0; i < N; ++i)
    for (int j = 0; j < N; ++j) A[i * N + j] = i == j ? 4.0 : 1.0 / (1.0 + (i > j ? i - j : j - i) * 3.0);
  // full skyline: f, flag offsets, tasks in the order of dense_start
  std::vector<int32_t> f(T, 0), off(T + 1);
  for (int i = 0; i < T; ++i) off[i + 1] = off[i] + i + 1;
  std::vector<uint32_t> task;
  for (int j = 0; j < T; ++j) {
    if (f[j] == j) task.push_back((uint32_t)(j << 15 | j));
    if (j + 1 < T) task.push_back((uint32_t)((j + 1) << 15 | (j + 1)));
    for (int i = j + 2; i < T; ++i) task.push_back((uint32_t)(i << 15 | j));
  }
  for (int s = 0; s < N / CH_STRIP; ++s) task.push_back(CH_INV | (uint32_t)s);
  int32_t *df, *doff;
  uint32_t* dtask;
  double* d[5];
  int* di;  // flags, then the ticket and the error bits
  const int nflag = off[T];
  CK(cudaMalloc(&df, 4 * T) == cudaSuccess && cudaMalloc(&doff, 4 * (T + 1)) == cudaSuccess);
  CK(cudaMalloc(&dtask, 4 * task.size()) == cudaSuccess && cudaMalloc(&di, 4 * (nflag + 2)) == cudaSuccess);
  for (double*& p : d) CK(cudaMalloc(&p, 8 * N * N) == cudaSuccess);
  CK(cudaMemcpy(df, f.data(), 4 * T, cudaMemcpyHostToDevice) == cudaSuccess);
  CK(cudaMemcpy(doff, off.data(), 4 * (T + 1), cudaMemcpyHostToDevice) == cudaSuccess);
  CK(cudaMemcpy(dtask, task.data(), 4 * task.size(), cudaMemcpyHostToDevice) == cudaSuccess);
  for (int pass = 0; pass < 3; ++pass) {
    CholView C;
    C.n = N; C.nb = T; C.f = df; C.off = doff; C.task = dtask; C.ntask = (int)task.size();
    C.M = d[0]; C.LT = d[1]; C.W = d[2]; C.WT = d[3]; C.Dinv = d[4];
    C.flag = di; C.ticket = di + nflag; C.err = di + nflag + 1; C.limit = pass == 1 ? 2000 : CH_POLLS;
    const int start = pass == 1;  // the first task is passed over
    CK(cudaMemcpy(d[0], A.data(), 8 * N * N, cudaMemcpyHostToDevice) == cudaSuccess);
    CK(cudaMemset(di, 0, 4 * (nflag + 2)) == cudaSuccess);
    CK(cudaMemcpy(C.ticket, &start, 4, cudaMemcpyHostToDevice) == cudaSuccess);
    k_chol<<<(unsigned)task.size(), CH_THREADS>>>(C);
    int err = -1;
    CK(cudaDeviceSynchronize() == cudaSuccess);
    CK(cudaMemcpy(&err, C.err, 4, cudaMemcpyDeviceToHost) == cudaSuccess);
    CK(err == (pass == 1 ? 2 : 0));
    if (pass == 1) continue;
    CK(cudaMemcpy(L.data(), d[0], 8 * N * N, cudaMemcpyDeviceToHost) == cudaSuccess);
    for (int i = 0; i < N; ++i)
      for (int j = 0; j <= i; ++j) {
        double s = 0.0;
        for (int k = 0; k <= j; ++k) s += L[i * N + k] * L[j * N + k];
        CK(fabs(s - A[i * N + j]) <= 4.0 * N * 1.2e-16 * 4.0);
      }
  }
  return 0;
}
