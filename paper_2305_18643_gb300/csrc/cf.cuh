// Continued fractions of Eq. jacobi shifted by E0 (s = -1 electron part, +1 hole part),
//
//   G(z) = b_0^2 / (D_0 - b_1^2 / (D_1 - b_2^2 / (D_2 - ...))),   D_n = z + s (a_n - E0),
//
// without a division per level: FP64 runs two lanes per clock and SM on this GPU and a division is
// a chain of a dozen FP64 operations, so both directions use the linear recurrences of the
// numerators and denominators (rescaled by powers of two every eight levels) and divide once.
//
//  - Backward, P_n = D_n P_{n+1} - b_{n+1}^2 P_{n+2} from the last level up, G = b_0^2 P_1 / P_0: the
//    value of record (each quotient P_n / P_{n+1} is the den_n of the quotient form, with the same
//    contraction of errors).
//  - Forward (Wallis), A_k = D_{k-1} A_{k-1} - b_{k-1}^2 A_{k-2} and B_k likewise, G = A_k / B_k: the state
//    of a frequency is four numbers, so a convergence check pays for the levels since the last
//    check only.
#pragma once

#include "ed_common.cuh"

namespace ed {

// 2^-e for the largest exponent e of the four values (clamped to the normal range).
__device__ __forceinline__ double cf_down_scale(double a, double b, double c, double d) {
  const int m = max(max(__double2hiint(a) & 0x7ff00000, __double2hiint(b) & 0x7ff00000),
                    max(__double2hiint(c) & 0x7ff00000, __double2hiint(d) & 0x7ff00000));
  return __hiloint2double(min(max((2046 << 20) - m, 1 << 20), 2045 << 20), 0);
}

// The rescaling after level n runs where (n & mask) is the mask's first or last value: every eight levels,
// and after each level for |z| beyond 1e30, where eight levels may leave the range of FP64.  A level whose own
// coefficients are that large (cf_wide) is rescaled before and after.
__device__ __forceinline__ int cf_scale_mask(double2 z) { return fabs(z.x) + fabs(z.y) > 1e30 ? 0 : 7; }

// |x| of a level beyond 2^100 or its y beyond 2^200 (by the exponents: no FP64 comparison).
__device__ __forceinline__ bool cf_wide(double2 e) {
  return (__double2hiint(e.x) & 0x7fffffff) > ((1023 + 100) << 20) || __double2hiint(e.y) > ((1023 + 200) << 20);
}

// A level as the recurrences read it: x = s (a_n - E0), y = b_{n+1}^2 (backward; 0 behind the last
// level) or b_n^2 (forward; -1 for level 0, so that A_1 = 1).
struct CfBackward {
  double pr = 1.0, pi = 0.0, qr = 0.0, qi = 0.0;  // P_{n+1}, P_{n+2}
  __device__ __forceinline__ void level(double2 e, double2 z) {
    const double dr = z.x + e.x;
    const double nr = fma(dr, pr, fma(-z.y, pi, -e.y * qr)), ni = fma(dr, pi, fma(z.y, pr, -e.y * qi));
    qr = pr;
    qi = pi;
    pr = nr;
    pi = ni;
  }
  __device__ __forceinline__ void rescale() {
    const double f = cf_down_scale(pr, pi, qr, qi);
    pr *= f;
    pi *= f;
    qr *= f;
    qi *= f;
  }
  __device__ __forceinline__ double2 value(double b0sq) const {  // b_0^2 P_1 / P_0
    const double f = b0sq / (pr * pr + pi * pi);
    return make_double2(f * (qr * pr + qi * pi), f * (qi * pr - qr * pi));
  }
};

struct CfForward {
  double2 a1{0.0, 0.0}, a0{1.0, 0.0}, b1{1.0, 0.0}, b0{0.0, 0.0};  // A_k, A_{k-1}, B_k, B_{k-1}
  __device__ __forceinline__ void level(double2 e, double2 z) {
    const double dr = z.x + e.x;
    const double2 a = make_double2(fma(dr, a1.x, fma(-z.y, a1.y, -e.y * a0.x)), fma(dr, a1.y, fma(z.y, a1.x, -e.y * a0.y)));
    const double2 b = make_double2(fma(dr, b1.x, fma(-z.y, b1.y, -e.y * b0.x)), fma(dr, b1.y, fma(z.y, b1.x, -e.y * b0.y)));
    a0 = a1;
    b0 = b1;
    a1 = a;
    b1 = b;
  }
  __device__ __forceinline__ void rescale() {
    const double f = cf_down_scale(b1.x, b1.y, b0.x, b0.y);
    a1.x *= f;
    a1.y *= f;
    a0.x *= f;
    a0.y *= f;
    b1.x *= f;
    b1.y *= f;
    b0.x *= f;
    b0.y *= f;
  }
  __device__ __forceinline__ double2 value(double b0sq) const {  // b_0^2 A_k / B_k
    const double f = b0sq / (b1.x * b1.x + b1.y * b1.y);
    return make_double2(f * (a1.x * b1.x + a1.y * b1.y), f * (a1.y * b1.x - a1.x * b1.y));
  }
};

constexpr int kCfChunk = 128;  // levels staged in shared memory at a time

// The fraction of m levels at z by the threads of a block (each its own z; `use` false for threads
// without one), levels staged through sm[kCfChunk].  All threads of the block must call it.
__device__ __forceinline__ double2 cf_eval_block(const double* __restrict__ a, const double* __restrict__ b, int m,
                                                 double b0sq, double2 z, double E0, double s, double2* sm, bool use) {
  CfBackward st;
  const int mask = cf_scale_mask(z);
  for (int hi = m; hi > 0; hi -= kCfChunk) {
    const int lo = hi > kCfChunk ? hi - kCfChunk : 0;
    __syncthreads();
    for (int n = lo + threadIdx.x; n < hi; n += blockDim.x) {
      const double bn = n + 1 < m ? b[n + 1] : 0.0;
      sm[n - lo] = make_double2(s * (a[n] - E0), bn * bn);
    }
    __syncthreads();
    if (use)
      for (int n = hi - 1; n >= lo; --n) {
        const double2 e = sm[n - lo];
        const bool wide = cf_wide(e);
        if (wide) st.rescale();
        st.level(e, z);
        if (wide || (n & mask) == 0) st.rescale();
      }
  }
  return m > 0 ? st.value(b0sq) : make_double2(0.0, 0.0);
}

// Advances the forward state of z over levels [m0, m).  Same calling rule.
__device__ __forceinline__ void cf_advance_block(CfForward& st, const double* __restrict__ a, const double* __restrict__ b,
                                                 int m0, int m, double2 z, double E0, double s, double2* sm, bool use) {
  const int mask = cf_scale_mask(z);
  for (int lo = m0; lo < m; lo += kCfChunk) {
    const int hi = min(m, lo + kCfChunk);
    __syncthreads();
    for (int n = lo + threadIdx.x; n < hi; n += blockDim.x)
      sm[n - lo] = make_double2(s * (a[n] - E0), n == 0 ? -1.0 : b[n] * b[n]);
    __syncthreads();
    if (use)
      for (int n = lo; n < hi; ++n) {
        const double2 e = sm[n - lo];
        const bool wide = cf_wide(e);
        if (wide) st.rescale();
        st.level(e, z);
        if (wide || (n & mask) == mask) st.rescale();
      }
  }
  st.rescale();
}

}  // namespace ed
