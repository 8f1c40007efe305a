// The block tridiagonal eigensolver (csrc/tridiag.cuh) beside the plain form of the same algorithm, which
// counts at every point of every round and divides in every sweep.  Built and driven by
// test_ranges_gpu.py.
#include <cmath>
#include <cstdint>

#include "tridiag.cuh"

namespace {

__global__ void k_fast(const double* a, const double* b, int n, double* eval, double* vec) {
  ed::tridiag_lowest_block(a, b, n, eval, vec);
  __syncthreads();
  ed::tridiag_second_block(a, b, n, eval, vec + n);
}

__device__ int count_below(const double* a, const double* b, int n, double x) {
  double q = a[0] - x;
  int cnt = q < 0.0;
  for (int i = 1; i < n; ++i) {
    if (q == 0.0) q = 1e-300;
    q = a[i] - x - b[i] * b[i] / q;
    cnt += q < 0.0;
  }
  return cnt;
}

__global__ void k_plain(const double* a, const double* b, int n, double* eval, double* y, double* cp) {
  __shared__ int first;
  const int nt = blockDim.x, tid = threadIdx.x;
  double glo = 1e300, ghi = -1e300;
  for (int i = 0; i < n; ++i) {
    const double r = (i > 0 ? fabs(b[i]) : 0.0) + (i + 1 < n ? fabs(b[i + 1]) : 0.0);
    glo = fmin(glo, a[i] - r);
    ghi = fmax(ghi, a[i] + r);
  }
  const double pad = 1e-12 * fmax(1.0, fmax(fabs(glo), fabs(ghi))) + 1e-300;
  glo -= pad;
  ghi += pad;
  double lam[2] = {0.0, INFINITY};
  for (int k = 0; k < (n < 2 ? 1 : 2); ++k) {
    double lo = glo, hi = ghi;
    for (int round = 0; round < 16; ++round) {
      if (tid == 0) first = nt;
      __syncthreads();
      const double x = lo + (hi - lo) * (double)(tid + 1) / (double)(nt + 1);
      if (count_below(a, b, n, x) >= k + 1) atomicMin(&first, tid);
      __syncthreads();
      const int j = first;
      const double nlo = j == 0 ? lo : lo + (hi - lo) * (double)j / (double)(nt + 1);
      const double nhi = j == nt ? hi : lo + (hi - lo) * (double)(j + 1) / (double)(nt + 1);
      lo = nlo;
      hi = nhi;
      __syncthreads();
      if (hi - lo <= 4e-16 * fmax(fabs(lo), fabs(hi))) break;
    }
    lam[k] = 0.5 * (lo + hi);
  }
  if (tid) return;
  const double sigma = lam[0] - 1e-10 * fmax(1.0, fmax(fabs(glo), fabs(ghi)));
  for (int i = 0; i < n; ++i) y[i] = 1.0 + 0.1 * sin((double)i);
  for (int it = 0; it < 3; ++it) {
    double m = a[0] - sigma;
    cp[0] = (n > 1 ? b[1] : 0.0) / m;
    y[0] = y[0] / m;
    for (int i = 1; i < n; ++i) {
      m = (a[i] - sigma) - b[i] * cp[i - 1];
      cp[i] = (i + 1 < n ? b[i + 1] : 0.0) / m;
      y[i] = (y[i] - b[i] * y[i - 1]) / m;
    }
    for (int i = n - 2; i >= 0; --i) y[i] -= cp[i] * y[i + 1];
    double nr = 0.0;
    for (int i = 0; i < n; ++i) nr += y[i] * y[i];
    nr = 1.0 / sqrt(nr);
    for (int i = 0; i < n; ++i) y[i] *= nr;
  }
  if (y[0] < 0.0)
    for (int i = 0; i < n; ++i) y[i] = -y[i];
  eval[0] = lam[0];
  eval[1] = lam[1];
  eval[2] = fabs(b[n]) * fabs(y[n - 1]);
}

}  // namespace

// a: n diagonal entries, b: n + 1 (b[0] unused, b[n] the next norm); eval: 4, vec: 2 n doubles each.
extern "C" int tridiag_both(const double* a, const double* b, int n, int threads, double* eval_fast, double* vec_fast,
                            double* eval_plain, double* vec_plain) {
  k_fast<<<1, threads>>>(a, b, n, eval_fast, vec_fast);
  k_plain<<<1, threads>>>(a, b, n, eval_plain, vec_plain, vec_plain + n);
  return (int)cudaDeviceSynchronize();
}
