// One element of the factorized product y = H x (Eq. factorized, Sec. 4.1), shared by every
// kernel that computes H.psi element by element (the one-pass kernels of hpsi.cu and the
// allocation-free entry point of noalloc.cu), so that the diagonal and the sign handling exist
// once:
//
//   y[u][d] = D(u, d) x[u][d] + sum_{d'} K_dn[d][d'] x[u][d'] + sum_{u'} K_up[u][u'] x[u'][d]
//   D(u, d) = e_up[u] + e_dn[d] + sum_{i in cluster} U_i n_{i up} n_{i dn}
#pragma once

#include "ed_common.cuh"

namespace ed {

// Per-precision views of the diagonal tables and hopping values.
template <typename T>
struct Prec;
template <>
struct Prec<double> {
  __device__ static const double* e_up(const SectorArgs& s) { return s.e_up; }
  __device__ static const double* e_dn(const SectorArgs& s) { return s.e_dn; }
  __device__ static double val(const HopParams& h, int i) { return h.val[i]; }
  __device__ static double U(const HopParams& h, int i) { return h.U[i]; }
  __device__ static double u0(const HopParams& h) { return h.u0; }
};
template <>
struct Prec<float> {
  __device__ static const float* e_up(const SectorArgs& s) { return s.e_up32; }
  __device__ static const float* e_dn(const SectorArgs& s) { return s.e_dn32; }
  __device__ static float val(const HopParams& h, int i) { return h.valf[i]; }
  __device__ static float U(const HopParams& h, int i) { return h.Uf[i]; }
  __device__ static float u0(const HopParams& h) { return h.u0f; }
};

// Deterministic block reduction of three FP64 sums over NT threads (fixed shuffle tree, fixed
// warp order); the totals end in warp 0's lane 0.
template <int NT>
__device__ __forceinline__ void block_sum3(double& a, double& b, double& c) {
  __shared__ double sm[3][NT / 32];
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
    c += __shfl_down_sync(0xffffffffu, c, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    sm[0][w] = a;
    sm[1][w] = b;
    sm[2][w] = c;
  }
  __syncthreads();
  if (w == 0) {
    a = l < NT / 32 ? sm[0][l] : 0.0;
    b = l < NT / 32 ? sm[1][l] : 0.0;
    c = l < NT / 32 ? sm[2][l] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_down_sync(0xffffffffu, a, o);
      b += __shfl_down_sync(0xffffffffu, b, o);
      c += __shfl_down_sync(0xffffffffu, c, o);
    }
  }
  __syncthreads();
}

// The same for any block of whole warps, at most 32 of them.
__device__ __forceinline__ void block_sum3_any(double& a, double& b, double& c) {
  __shared__ double sm[3][32];
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
    c += __shfl_down_sync(0xffffffffu, c, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (l == 0) {
    sm[0][w] = a;
    sm[1][w] = b;
    sm[2][w] = c;
  }
  __syncthreads();
  if (w == 0) {
    a = l < nw ? sm[0][l] : 0.0;
    b = l < nw ? sm[1][l] : 0.0;
    c = l < nw ? sm[2][l] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_down_sync(0xffffffffu, a, o);
      b += __shfl_down_sync(0xffffffffu, b, o);
      c += __shfl_down_sync(0xffffffffu, c, o);
    }
  }
  __syncthreads();
}

// Hopping values and per-orbital U staged in shared memory (sval[kMaxVals], sU[kMaxOrb]).
template <typename T>
__device__ __forceinline__ void load_params(const HopParams& hp, T* sval, T* sU) {
  for (int i = threadIdx.x; i < kMaxVals; i += blockDim.x) sval[i] = Prec<T>::val(hp, i);
  for (int i = threadIdx.x; i < kMaxOrb; i += blockDim.x) sU[i] = Prec<T>::U(hp, i);
  __syncthreads();
}

// v with its sign bit flipped when neg is 1 (an integer operation: FP64 ones are scarce here).
__device__ __forceinline__ double flip_sign(double v, uint32_t neg) {
  return __hiloint2double(__double2hiint(v) ^ (int)(neg << 31), __double2loint(v));
}
__device__ __forceinline__ float flip_sign(float v, uint32_t neg) { return __int_as_float(__float_as_int(v) ^ (int)(neg << 31)); }

// acc + sum over the entries ent[p0, p1) of +-val X[col * stride], in their order; the entries, values
// and operands of four hops are loaded before their multiply-adds.  The last hops, fewer than four: in FP64
// predicated in the same loop (20 orbitals, (10, 1) particles: 124 us a product, 136 us one at a time), in
// FP32, where the issue of the predicates costs more, one at a time (70 and 60 us).
template <typename T>
__device__ __forceinline__ T add_entries(T acc, const uint32_t* __restrict__ ent, int32_t p0, int32_t p1,
                                         const T* __restrict__ sval, const T* __restrict__ X, int64_t stride) {
  constexpr bool TAIL = sizeof(T) == 4;
  int32_t k = p0;
  for (; TAIL ? k + 4 <= p1 : k < p1; k += 4) {
    uint32_t e[4];
    T x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) e[i] = __ldg(ent + (TAIL || k + i < p1 ? k + i : k));
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = __ldg(X + (int64_t)ent_col(e[i]) * stride);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (TAIL || k + i < p1) acc = fma(flip_sign(sval[ent_vidx(e[i])], ent_neg(e[i])), x[i], acc);
  }
  if (TAIL)
    for (; k < p1; ++k) {
      const uint32_t e = __ldg(ent + k);
      acc = fma(flip_sign(sval[ent_vidx(e)], ent_neg(e)), __ldg(X + (int64_t)ent_col(e) * stride), acc);
    }
  return acc;
}

// Diagonal D(u, d) from the spins' one-body parts and the doubly occupied interacting orbitals.
template <typename T>
__device__ __forceinline__ T hpsi_diag(T e, uint32_t dbl, const T* __restrict__ sU, bool uni, T u0) {
  if (uni) return fma(u0, (T)__popc(dbl), e);
  while (dbl) {
    e += sU[__ffs(dbl) - 1];
    dbl &= dbl - 1u;
  }
  return e;
}

// y[u][d] of a vector X with leading dimension sv.ld: the diagonal by masked popcount of the
// doubly occupied interacting orbitals, then the down-spin hops (inside row u) and the up-spin
// hops (down column d), each entry (-1)^{M_ab} h_ab x[source].
template <typename T>
__device__ __forceinline__ T hpsi_element(const SectorView& sv, const T* __restrict__ sval, const T* __restrict__ sU,
                                          const HopParams& hp, const T* __restrict__ X, int64_t u, int64_t d) {
  const T* xr = X + u * sv.ld;
  const T diag = hpsi_diag<T>(Prec<T>::e_up(sv)[u] + Prec<T>::e_dn(sv)[d], sv.B_up[u] & sv.B_dn[d] & hp.umask, sU,
                              hp.uniform_u != 0, Prec<T>::u0(hp));
  T acc = diag * xr[d];
  acc = add_entries<T>(acc, sv.ent_dn, sv.ptr_dn[d], sv.ptr_dn[d + 1], sval, xr, 1);
  return add_entries<T>(acc, sv.ent_up, sv.ptr_up[u], sv.ptr_up[u + 1], sval, X + d, sv.ld);
}

}  // namespace ed
