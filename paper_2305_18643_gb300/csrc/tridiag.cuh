// Lowest eigenpair of the Lanczos tridiagonal matrix (Eq. tridiag), computed by one thread block:
// multisection on the Sturm count for the two lowest eigenvalues, then inverse iteration with a
// shift just below the lowest one (T - sigma I is positive definite, so elimination without
// pivoting is stable).  Used by the single-cluster driver and by the batched per-block solver.
//
// A thread block runs one matrix, so the kernel is bound by the dependent chain of the recurrences
// and by the FP64 pipe of one SM (two lanes per clock on this GPU).  The count of record is the
// quotient form q_k = a_k - x - b_k^2 / q_{k-1}, whose division alone is a dozen FP64 operations, so it
// runs only where it decides something: both eigenvalues are first located to a few ulps of the
// matrix norm with the division-free recurrence p_k = (a_k - x) p_{k-1} - b_k^2 p_{k-2} on entries scaled
// by a power of two (three rounds in FP32 on every thread, then FP64 on 16 lanes per eigenvalue);
// the multisection then counts only at points inside that uncertainty, and its result is bit for bit that
// of counting at every point.
//
// One call, over the checks of a 100-level run: 927 us with the quotient form at every point and a
// division per pivot and sweep, 254 us now; over those of a 160-level run 1,418 and 380 us.  The ground
// states of 64 clusters of at most 7 orbitals, where every block runs its own (csrc/batch.cu): 225.4 ms
// before, 78.2 ms now.
#pragma once

#include <cuda_runtime.h>

namespace ed {

// Number of negative p_k / p_{k-1} over the n levels of the scaled matrix (ab[k] = {a_k, b_k^2}, b_0
// = 0), i.e. of eigenvalues below x, in FP32.
static __device__ inline int sturm_count32(const float2* __restrict__ ab, int n, float x) {
  int cnt = 0;
  float pp = 0.f, p = 1.f;
  for (int k = 0; k < n; ++k) {
    const float2 v = ab[k];
    float q = fmaf(v.x - x, p, -v.y * pp);
    if (q == 0.f) q = p * 1e-10f;  // as a tiny positive pivot
    cnt += (__float_as_int(q) ^ __float_as_int(p)) < 0;
    pp = p;
    p = q;
    if ((k & 3) == 3) {  // |q| <= 2 max(|p|, |pp|) per level: four levels stay in range
      const int e = max(__float_as_int(p) & 0x7f800000, __float_as_int(pp) & 0x7f800000);
      const float f = __int_as_float(min(max((254 << 23) - e, 1 << 23), 253 << 23));
      p *= f;
      pp *= f;
    }
  }
  return cnt;
}

// The same in FP64: a[k], b2[k] the scaled entries.
static __device__ inline int sturm_count64(const double* a, const double* b2, int n, double x) {
  int cnt = 0;
  double pp = 0.0, p = 1.0;
  for (int k = 0; k < n; ++k) {
    double q = fma(a[k] - x, p, -b2[k] * pp);
    if ((__double2hiint(q) & 0x7fffffff) < 0x00100000) q = p * 1e-30;
    cnt += (__double2hiint(q) ^ __double2hiint(p)) < 0;
    pp = p;
    p = q;
    if ((k & 7) == 7) {
      const int e = max(__double2hiint(p) & 0x7ff00000, __double2hiint(pp) & 0x7ff00000);
      const double f = __hiloint2double(min(max((2046 << 20) - e, 1 << 20), 2045 << 20), 0);
      p *= f;
      pp *= f;
    }
  }
  return cnt;
}

// Number of eigenvalues below x in the quotient form: diagonal a[0..n-1], off-diagonal b[1..n-1].
static __device__ inline int sturm_count(const double* __restrict__ a, const double* __restrict__ b, int n, double x) {
  int cnt = 0;
  double q = a[0] - x;
  if (q < 0.0) ++cnt;
  for (int i = 1; i < n; ++i) {
    if (q == 0.0) q = 1e-300;
    q = a[i] - x - b[i] * b[i] / q;
    if (q < 0.0) ++cnt;
  }
  return cnt;
}

// Gershgorin interval [lo, hi] of the matrix, padded.  All threads of the block must call it.
static __device__ __forceinline__ void tridiag_interval(const double* __restrict__ a, const double* __restrict__ b, int n, double* out_lo,
                                               double* out_hi) {
  __shared__ double s_lo, s_hi;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {
    double lo = 1e300, hi = -1e300;
    for (int i = lane; i < n; i += 32) {
      const double r = (i > 0 ? fabs(b[i]) : 0.0) + (i + 1 < n ? fabs(b[i + 1]) : 0.0);
      lo = fmin(lo, a[i] - r);
      hi = fmax(hi, a[i] + r);
    }
    for (int o = 16; o > 0; o >>= 1) {
      lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) {
      const double pad = 1e-12 * fmax(1.0, fmax(fabs(lo), fabs(hi))) + 1e-300;
      s_lo = lo - pad;
      s_hi = hi + pad;
    }
  }
  __syncthreads();
  *out_lo = s_lo;
  *out_hi = s_hi;
}

// Multisection of [lo, hi] for the k-th lowest eigenvalue (from 1) with blockDim.x points a round, given
// that it lies within `slack` of `near` for any matrix within rounding of this one: points further away
// need no count, and points that round to the same number need one.  cand: room for ncand ints.  All
// threads of the block must call it; the midpoint of the last interval is returned to each.
static __device__ __forceinline__ double tridiag_multisect(const double* __restrict__ a, const double* __restrict__ b, int n, int k, double lo,
                                                  double hi, double near, double slack, int* cand, int ncand) {
  __shared__ int s_first, s_cand;
  const int tid = threadIdx.x, nt = blockDim.x;
  auto point = [&](int j) { return lo + (hi - lo) * (double)(j + 1) / (double)(nt + 1); };
  for (int round = 0; round < 16; ++round) {
    if (tid == 0) {
      s_first = nt;
      s_cand = 0;
    }
    __syncthreads();
    const double x = point(tid);
    if (x > near + slack) {
      atomicMin(&s_first, tid);
    } else if (x >= near - slack && (tid == 0 || point(tid - 1) != x)) {
      const int c = atomicAdd(&s_cand, 1);
      if (c < ncand) cand[c] = tid;
    }
    __syncthreads();
    const int nc = s_cand;
    if (nc <= ncand) {
      for (int c = tid; c < nc; c += nt) {
        const int j = cand[c];
        if (sturm_count(a, b, n, point(j)) >= k) atomicMin(&s_first, j);
      }
    } else if (x >= near - slack && x <= near + slack) {
      if (sturm_count(a, b, n, x) >= k) atomicMin(&s_first, tid);
    }
    __syncthreads();
    const int j = s_first;
    const double nlo = j == 0 ? lo : lo + (hi - lo) * (double)j / (double)(nt + 1);
    const double nhi = j == nt ? hi : lo + (hi - lo) * (double)(j + 1) / (double)(nt + 1);
    lo = nlo;
    hi = nhi;
    __syncthreads();
    if (hi - lo <= 4e-16 * fmax(fabs(lo), fabs(hi))) break;
  }
  return 0.5 * (lo + hi);
}

// How far the brackets of the division-free counts may be off: their width and 100 ulps of the norm (both
// counts are exact for matrices within ~10 ulps of this one).
static __device__ __forceinline__ double tridiag_slack(double width, double sc) { return 0.5 * width + 100.0 * 2.3e-16 * sc; }

// out_eval: [0] lowest eigenvalue, [1] about the second eigenvalue (inf if n < 2; tridiag_second_block
// settles it), [2] Ritz estimate b_n |s_{n-1}|, [3] how far [1] may be off.  vec: [0, n) unit eigenvector of the lowest eigenvalue (s_0 >= 0), [n, 2n) scratch.
// The block has a multiple of 32 threads, at least 64.
static __device__ void tridiag_lowest_block(const double* __restrict__ a, const double* __restrict__ b, int n,
                                            double* out_eval, double* vec) {
  __shared__ int s_first[2];
  __shared__ double s_near[2], s_width[2];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  double glo, ghi;
  tridiag_interval(a, b, n, &glo, &ghi);
  // scale by a power of two (exact), so that |entries|, |x| <= 1/2 and |a - x| <= 1
  int ex;
  frexp(fmax(fabs(glo), fabs(ghi)), &ex);
  const double is = ldexp(1.0, -(ex + 1)), sc = ldexp(1.0, ex + 1);
  float2* ab = reinterpret_cast<float2*>(vec + n);
  for (int i = tid; i < n; i += nt) {
    const double as = a[i] * is, bs = i > 0 ? b[i] * is : 0.0;
    vec[i] = as;
    ab[i] = make_float2((float)as, (float)(bs * bs));
  }
  // FP32 rounds: the first on the whole interval for both eigenvalues, then half the threads each
  const int half = nt / 2, k = tid >= half ? 1 : 0;
  float lo[2], hi[2];
  lo[0] = lo[1] = (float)(glo * is);
  hi[0] = hi[1] = (float)(ghi * is);
  for (int round = 0; round < 3; ++round) {
    const int m = round == 0 ? nt : half, j = round == 0 ? tid : tid - k * half;
    if (tid < 2) s_first[tid] = m;
    __syncthreads();
    const float x = lo[k] + (hi[k] - lo[k]) * ((float)(j + 1) / (float)(m + 1));
    const int cnt = sturm_count32(ab, n, x);
    if ((round == 0 || k == 0) && cnt >= 1) atomicMin(&s_first[0], j);
    if ((round == 0 || k == 1) && cnt >= 2) atomicMin(&s_first[1], j);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int f = s_first[q];
      const float l = lo[q], w = hi[q] - lo[q];
      if (f > 0) lo[q] = l + w * ((float)f / (float)(m + 1));
      if (f < m) hi[q] = l + w * ((float)(f + 1) / (float)(m + 1));
    }
    __syncthreads();
  }
  for (int i = tid; i < n; i += nt) {
    const double bs = i > 0 ? b[i] * is : 0.0;
    vec[n + i] = bs * bs;  // over the FP32 entries
  }
  __syncthreads();
  // FP64 rounds by warp 0: lanes 0..15 bracket the lowest, 16..31 the second eigenvalue, end points
  // included.  The FP32 counts are those of a matrix within a few 2^-24 of this one; a bracket that
  // the FP64 counts of the first round refute is widened to the whole interval.
  if (tid < 32) {
    const int e = lane >> 4, pt = lane & 15;
    double dlo = (double)lo[e] - 2e-6, dhi = (double)hi[e] + 2e-6;
    bool first = true, done = e == 1 && n < 2;
    for (int round = 0; round < 24; ++round) {
      const double x = dlo + (dhi - dlo) * ((double)pt * (1.0 / 15.0));
      const bool above = sturm_count64(vec, vec + n, n, x) >= e + 1;
      const unsigned bal = (__ballot_sync(0xffffffffu, above) >> (16 * e)) & 0xffffu;
      if (!done) {
        const int f = bal ? __ffs(bal) - 1 : 16;
        if (f == 0 || f == 16) {
          if (first) {
            dlo = glo * is;
            dhi = ghi * is;
          } else {
            done = true;  // the bracket is down to rounding
          }
        } else {
          const double w = dhi - dlo;
          const double nlo = dlo + w * ((double)(f - 1) * (1.0 / 15.0));
          const double nhi = f == 15 ? dhi : dlo + w * ((double)f * (1.0 / 15.0));
          dlo = nlo;
          dhi = nhi;
        }
        first = false;
        if (dhi - dlo <= 2e-15) done = true;
      }
      if (__all_sync(0xffffffffu, done)) break;
    }
    if (pt == 0) {
      s_near[e] = 0.5 * (dlo + dhi) * sc;
      s_width[e] = (dhi - dlo) * sc;
    }
  }
  __syncthreads();
  const double lam = tridiag_multisect(a, b, n, 1, glo, ghi, s_near[0], tridiag_slack(s_width[0], sc), reinterpret_cast<int*>(vec),
                                       4 * n);  // vec holds 2 n doubles
  if (tid >= 32) return;
  // inverse iteration with shift just below lam: T - sigma I is positive definite, so the
  // Thomas elimination without pivoting is stable.  The pivots m_i are those of every iteration, so
  // they are found once (lane 0; cp_i = b_{i+1} / m_i is kept); the quotients by m_i in the sweeps
  // come from the rounded reciprocals r_i (Markstein, "Computation of elementary functions on the
  // IBM RISC System/6000 processor", 1990: q = y r, q + r (y - q m) is the rounded quotient).
  const double scale = fmax(1.0, fmax(fabs(glo), fabs(ghi)));
  const double sigma = lam - 1e-10 * scale;
  double* y = vec;
  double* cp = vec + n;
  if (lane == 0) {
    double m = a[0] - sigma;
    cp[0] = (n > 1 ? b[1] : 0.0) / m;
    for (int i = 1; i < n; ++i) {
      m = (a[i] - sigma) - b[i] * cp[i - 1];
      cp[i] = (i + 1 < n ? b[i + 1] : 0.0) / m;
    }
  }
  __syncwarp();
  for (int i = lane; i < n; i += 32) y[i] = 1.0 + 0.1 * sin((double)i);
  __syncwarp();
  for (int it = 0; it < 3; ++it) {
    double t = 0.0;
    for (int i0 = 0; i0 < n; i0 += 32) {  // forward sweep: pivots and reciprocals by 32 lanes, then lane by lane
      const int i = i0 + lane;
      const double bi = i > 0 && i < n ? b[i] : 0.0;
      const double m = i == 0 ? a[0] - sigma : i < n ? (a[i] - sigma) - bi * cp[i - 1] : 1.0;
      const double r = 1.0 / m;
      double yi = i < n ? y[i] : 0.0;
      for (int l = 0; l < 32; ++l) {
        // every lane runs the quotient on its own entry; lane l's is the one that is final
        const double num = i == 0 ? yi : yi - bi * t;
        const double q = num * r;
        const double v = fma(fma(-q, m, num), r, q);
        if (lane == l) yi = v;
        t = __shfl_sync(0xffffffffu, v, l);
      }
      if (i < n) y[i] = yi;
      t = __shfl_sync(0xffffffffu, yi, 31);
    }
    __syncwarp();
    double nr = 0.0;
    if (lane == 0) {
      for (int i = n - 2; i >= 0; --i) y[i] -= cp[i] * y[i + 1];
      for (int i = 0; i < n; ++i) nr += y[i] * y[i];
      nr = 1.0 / sqrt(nr);
    }
    nr = __shfl_sync(0xffffffffu, nr, 0);
    for (int i = lane; i < n; i += 32) y[i] *= nr;
    __syncwarp();
  }
  if (y[0] < 0.0) {
    __syncwarp();
    for (int i = lane; i < n; i += 32) y[i] = -y[i];
  }
  __syncwarp();
  if (lane == 0) {
    out_eval[0] = lam;
    out_eval[1] = n < 2 ? INFINITY : s_near[1];
    out_eval[2] = fabs(b[n]) * fabs(y[n - 1]);
    out_eval[3] = tridiag_slack(s_width[1], sc);
  }
}

// The second eigenvalue by counts of record, bit for bit that of counting at every point, from what
// tridiag_lowest_block left in out_eval for the same matrix.  Callers compare gaps with thresholds, and need it
// only where a threshold lies within out_eval[3] of theirs: in every check it made the ground states of 64
// clusters of at most 6 orbitals 13 % slower, after every run those of a 2x4 cluster 5 %.  scratch: n doubles.
static __device__ void tridiag_second_block(const double* __restrict__ a, const double* __restrict__ b, int n, double* out_eval,
                                            double* scratch) {
  if (n < 2) return;
  double glo, ghi;
  tridiag_interval(a, b, n, &glo, &ghi);
  const double lam = tridiag_multisect(a, b, n, 2, glo, ghi, out_eval[1], out_eval[3], reinterpret_cast<int*>(scratch), 2 * n);
  if (threadIdx.x == 0) out_eval[1] = lam;
}

}  // namespace ed
