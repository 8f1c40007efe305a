// Lowest eigenpair of the Lanczos tridiagonal matrix (Eq. tridiag), computed by one thread block:
// multisection on the Sturm count for the two lowest eigenvalues, then inverse iteration with a
// shift just below the lowest one (T - sigma I is positive definite, so elimination without
// pivoting is stable).  Used by the single-cluster driver and by the batched per-block solver.
//
// A thread block runs one matrix, so the kernel is bound by the dependent chain of the recurrences
// and by the FP64 pipe of one SM (two lanes per clock on this GPU).  Hence:
//  - the count uses the division-free recurrence p_k = (a_k - x) p_{k-1} - b_k^2 p_{k-2} (three FP64
//    operations per level; the quotient form's division is a dozen) on entries scaled by a power
//    of two, rescaled every few levels;
//  - the first three rounds run in FP32 on every thread, and only the last bits, inside a bracket
//    that the FP64 counts verify, on 16 lanes per eigenvalue;
//  - the sweeps of the inverse iteration are first-order linear recurrences, done by one warp as
//    a scan over 32 chunks.
// One call, over the checks of a 120-level run: 1,020 us in the quotient form on 256 threads with a
// serial inverse iteration, 155 us now.  The ground states of 64 clusters of at most 7 orbitals,
// where every block runs its own (csrc/batch.cu): 225.4 ms before, 42.4 ms now.
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

// One sweep y_i <- im_i (y_i - b_i y_{i-1}) (forward) or y_i <- y_i - b_{i+1} im_i y_{i+1} (backward)
// by one warp: lane l owns the chunk of c indices from l c; the chunks' affine maps are composed by
// a scan over the lanes, then every lane runs its chunk from the right start.
template <bool FWD>
static __device__ inline void tridiag_sweep(const double* __restrict__ b, const double* im, double* y, int n, int c) {
  const int lane = threadIdx.x & 31;
  const int i0 = lane * c, i1 = min(n, i0 + c);
  double A = 1.0, B = 0.0;
  if (FWD) {
    for (int i = i0; i < i1; ++i) {
      const double l = i > 0 ? b[i] * im[i] : 0.0;
      B = fma(-l, B, y[i] * im[i]);
      A *= -l;
    }
  } else {
    for (int i = i1 - 1; i >= i0; --i) {
      const double u = i + 1 < n ? b[i + 1] * im[i] : 0.0;
      B = fma(-u, B, y[i]);
      A *= -u;
    }
  }
  // in: value entering this lane's chunk = composition of the maps of all chunks before it
  for (int o = 1; o < 32; o <<= 1) {
    const double Ao = FWD ? __shfl_up_sync(0xffffffffu, A, o) : __shfl_down_sync(0xffffffffu, A, o);
    const double Bo = FWD ? __shfl_up_sync(0xffffffffu, B, o) : __shfl_down_sync(0xffffffffu, B, o);
    if (FWD ? lane >= o : lane + o < 32) {
      B = fma(A, Bo, B);
      A *= Ao;
    }
  }
  double t = FWD ? __shfl_up_sync(0xffffffffu, B, 1) : __shfl_down_sync(0xffffffffu, B, 1);
  if (FWD ? lane == 0 : lane == 31) t = 0.0;
  if (FWD) {
    for (int i = i0; i < i1; ++i) {
      const double l = i > 0 ? b[i] * im[i] : 0.0;
      y[i] = t = fma(-l, t, y[i] * im[i]);
    }
  } else {
    for (int i = i1 - 1; i >= i0; --i) {
      const double u = i + 1 < n ? b[i + 1] * im[i] : 0.0;
      y[i] = t = fma(-u, t, y[i]);
    }
  }
  __syncwarp();
}

// out_eval: [0] lowest eigenvalue, [1] second eigenvalue (inf if n < 2), [2] Ritz estimate
// b_n |s_{n-1}|.  vec: [0, n) unit eigenvector of the lowest eigenvalue (s_0 >= 0), [n, 2n) scratch.
// The block has a multiple of 32 threads, at least 64.
static __device__ void tridiag_lowest_block(const double* __restrict__ a, const double* __restrict__ b, int n,
                                            double* out_eval, double* vec) {
  __shared__ double s_lo, s_hi;
  __shared__ int s_first[2];
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  // Gershgorin interval
  if (tid < 32) {
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
  const double glo = s_lo, ghi = s_hi;
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
  if (tid >= 32) return;
  // FP64 rounds: lanes 0..15 bracket the lowest, 16..31 the second eigenvalue, end points included.
  // The FP32 counts are those of a matrix within a few 2^-24 of this one; a bracket that the
  // FP64 counts of the first round refute is widened to the whole interval.
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
      if (dhi - dlo <= 4e-16 * fmax(fabs(dlo), fabs(dhi))) done = true;
    }
    if (__all_sync(0xffffffffu, done)) break;
  }
  const double mid = 0.5 * (dlo + dhi) * sc;
  const double lam = __shfl_sync(0xffffffffu, mid, 0);
  const double lam1 = __shfl_sync(0xffffffffu, mid, 16);
  // inverse iteration with a shift just below lam: pivots m_i = p_i / p_{i-1} of T - sigma from the
  // same recurrence (lane 0; every p_i > 0), then three solves
  const double scale = fmax(1.0, fmax(fabs(glo), fabs(ghi)));
  const double sigma = (lam - 1e-10 * scale) * is;
  if (lane == 0) {
    double pp = 0.0, p = 1.0;
    for (int i = 0; i < n; ++i) {
      const double q = fma(vec[i] - sigma, p, -vec[n + i] * pp);
      vec[i] = q;
      vec[n + i] = p;
      pp = p;
      p = q;
      if ((i & 7) == 7) {
        const int ee = max(__double2hiint(p) & 0x7ff00000, __double2hiint(pp) & 0x7ff00000);
        const double f = __hiloint2double(min(max((2046 << 20) - ee, 1 << 20), 2045 << 20), 0);
        p *= f;
        pp *= f;
      }
    }
  }
  __syncwarp();
  double* y = vec;
  double* im = vec + n;
  for (int i = lane; i < n; i += 32) {
    im[i] = vec[n + i] / (vec[i] * sc);
    y[i] = 1.0 + 0.1 * (double)sinf((float)i);
  }
  __syncwarp();
  const int c = (n + 31) / 32;
  for (int it = 0; it < 3; ++it) {
    tridiag_sweep<true>(b, im, y, n, c);
    tridiag_sweep<false>(b, im, y, n, c);
    double nr = 0.0;
    for (int i = lane; i < n; i += 32) nr = fma(y[i], y[i], nr);
    for (int o = 16; o > 0; o >>= 1) nr += __shfl_xor_sync(0xffffffffu, nr, o);
    nr = 1.0 / sqrt(nr);
    if (it == 2 && y[0] < 0.0) nr = -nr;
    __syncwarp();
    for (int i = lane; i < n; i += 32) y[i] *= nr;
    __syncwarp();
  }
  if (lane == 0) {
    out_eval[0] = lam;
    out_eval[1] = n < 2 ? INFINITY : lam1;
    out_eval[2] = fabs(b[n]) * fabs(y[n - 1]);
  }
}

}  // namespace ed
