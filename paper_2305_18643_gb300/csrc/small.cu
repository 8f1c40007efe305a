// Lanczos levels of small sectors without a launch per level (Eq. LanczosRecursion, Secs. 4.2, 4.3).
//
// A sector of a few thousand states spends its time in launches and in kernels too short to fill the
// GPU.  Here a thread-block cluster runs many levels of one run in one launch: every block keeps the
// whole vector v_n in shared memory and owns a slice of the elements.  A level is
//
//   w = H v_n - b_n v_{n-1} on the slice, partial sums of <v,w>, <w,w>, <v,v>  -> every block's shared memory
//   cluster barrier; a_n and b_{n+1} in every block from the same partials in the same order
//   v_{n+1} = (w - a_n v_n) / b_{n+1} on the slice                              -> every block's shared memory
//   cluster barrier.
//
// Bound by the FP64 pipe for FP64 vectors (a warp instruction holds its SM sub-partition for 64
// cycles: 16 + 2 operations per element at 11 hops) and by the latency of the scalars, so the sums
// over a warp take six additions instead of fifteen and the scalars no division.
// 36 runs of 3,920 states (the fractions of the 2x4 cluster), FP64, per level: 22 + 5 us in two
// launches, 10.8 us here in clusters of four blocks.
#include <cooperative_groups.h>

#include <algorithm>

#include "ed_common.cuh"
#include "hpsi_element.cuh"

namespace ed {

namespace cg = cooperative_groups;

constexpr int kSmallThreads = 256;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kSmallMaxCluster = 8;

// Sums of a, b, c over the warp: lane 0 ends with a's, lane 8 with b's, lane 16 with c's.
__device__ __forceinline__ double warp_sum3(double a, double b, double c) {
  const int lane = threadIdx.x & 31;
  const bool h = lane & 16, q = lane & 8;
  const double a1 = (h ? c : a) + __shfl_xor_sync(0xffffffffu, h ? a : c, 16);
  const double b1 = (h ? 0.0 : b) + __shfl_xor_sync(0xffffffffu, h ? b : 0.0, 16);
  double v = (q ? b1 : a1) + __shfl_xor_sync(0xffffffffu, q ? a1 : b1, 8);
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v;
}

// Shared memory of one block: v (all), then w, v_{n-1} and the diagonal of its slice, then the
// (u, d) pairs of the slice.
__host__ __device__ inline size_t small_smem(int64_t dim, int slice, size_t es) {
  return (size_t)(dim + 3 * (int64_t)slice) * es + (size_t)slice * sizeof(uint32_t);
}

template <typename T>
__global__ void __launch_bounds__(kSmallThreads) k_small_levels(SectorView sv, HopParams hp, T* __restrict__ V, T* __restrict__ VP,
                                                                int64_t vstride, int slice, int n0, int n1, LanczosScalars ls) {
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), nb = (int)cluster.num_blocks();
  const int run = blockIdx.x / nb;
  extern __shared__ __align__(16) unsigned char sl_smem[];
  __shared__ double red[kSmallMaxCluster * kSmallWarps][3];
  __shared__ T sval[2 * kMaxVals];  // signed: (vidx << 1) | neg
  __shared__ T sU[kMaxOrb];
  if (!ls.active[run]) return;
  const int dim = (int)(sv.d_up * sv.d_dn), dd = (int)sv.d_dn;
  T* X = reinterpret_cast<T*>(sl_smem);
  T* W = X + dim;
  T* P = W + slice;
  T* D = P + slice;
  uint32_t* ud = reinterpret_cast<uint32_t*>(D + slice);
  const int s0 = min(dim, rank * slice), ns = min(dim, s0 + slice) - s0;
  V += run * vstride;
  VP += run * vstride;
  for (int i = threadIdx.x; i < 2 * kMaxVals; i += blockDim.x) sval[i] = flip_sign(Prec<T>::val(hp, i >> 1), i & 1);
  for (int i = threadIdx.x; i < kMaxOrb; i += blockDim.x) sU[i] = Prec<T>::U(hp, i);
  __syncthreads();
  for (int i = threadIdx.x; i < dim; i += blockDim.x) X[i] = V[(int64_t)(i / dd) * sv.ld + i % dd];
  for (int i = threadIdx.x; i < ns; i += blockDim.x) {
    const int u = (s0 + i) / dd, d = (s0 + i) - u * dd;
    ud[i] = ((uint32_t)u << 16) | (uint32_t)d;
    P[i] = VP[(int64_t)u * sv.ld + d];
    D[i] = hpsi_diag<T>(Prec<T>::e_up(sv)[u] + Prec<T>::e_dn(sv)[d], sv.B_up[u] & sv.B_dn[d] & hp.umask, sU,
                        hp.uniform_u != 0, Prec<T>::u0(hp));
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t cb = (int64_t)run * ls.mstride;
  double b = ls.beta[(int64_t)run * (ls.mstride + 1) + n0];
  const double stop = ls.btol * ls.beta0[run];
  cluster.sync();  // every block has its vector
  auto hops = [&](T acc, const uint32_t* __restrict__ ent, int p0, int p1, const T* x, int stride) {
    for (int k = p0; k < p1; k += 4) {
      uint32_t e[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) e[i] = __ldg(ent + (k + i < p1 ? k + i : k));
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (k + i < p1) acc = fma(sval[((e[i] & 127u) << 1) | ent_neg(e[i])], x[(int)ent_col(e[i]) * stride], acc);
    }
    return acc;
  };
  for (int n = n0; n < n1; ++n) {
    const T bT = (T)b;
    double sxw = 0.0, sww = 0.0, sxx = 0.0;
    for (int i = threadIdx.x; i < ns; i += blockDim.x) {
      const int u = (int)(ud[i] >> 16), d = (int)(ud[i] & 0xffffu);
      const T x = X[s0 + i];
      T acc = D[i] * x;
      acc = hops(acc, sv.ent_dn, sv.ptr_dn[d], sv.ptr_dn[d + 1], X + u * dd, 1);
      acc = hops(acc, sv.ent_up, sv.ptr_up[u], sv.ptr_up[u + 1], X + d, dd);
      const T w = fma(-bT, P[i], acc);
      W[i] = w;
      const double xd = (double)x, wd = (double)w;
      sxw = fma(xd, wd, sxw);
      sww = fma(wd, wd, sww);
      sxx = fma(xd, xd, sxx);
    }
    const double part = warp_sum3(sxw, sww, sxx);
    if ((lane & 7) == 0 && lane < 24)
      for (int r = 0; r < nb; ++r) cluster.map_shared_rank(&red[0][0], r)[(rank * kSmallWarps + warp) * 3 + (lane >> 3)] = part;
    cluster.sync();
    sxw = sww = sxx = 0.0;
    for (int i = lane; i < nb * kSmallWarps; i += 32) {
      sxw += red[i][0];
      sww += red[i][1];
      sxx += red[i][2];
    }
    const double tot = warp_sum3(sxw, sww, sxx);
    sxw = __shfl_sync(0xffffffffu, tot, 0);
    sww = __shfl_sync(0xffffffffu, tot, 8);
    sxx = __shfl_sync(0xffffffffu, tot, 16);
    // 1 / <v,v> of a vector normalized to rounding: 1 + e + e^2 with e = 1 - <v,v>
    const double e = 1.0 - sxx;
    const double rxx = fabs(e) < 1e-6 ? fma(e, fma(e, e, e), e) + 1.0 : sxx > 0.0 ? 1.0 / sxx : 0.0;
    const double alpha = sxw * rxx;
    const double b2 = fma(-sxw, alpha, sxx > 0.0 ? sww : 0.0);
    const double ib = b2 > 0.0 ? rsqrt(b2) : 0.0;
    b = b2 * ib;
    const bool last = !(b > stop) || n + 1 >= ls.mstride;
    if (rank == 0 && threadIdx.x == 0) {
      ls.alpha[cb + n] = alpha;
      ls.beta[(int64_t)run * (ls.mstride + 1) + n + 1] = b2 > 0.0 ? b : 0.0;
      if (ls.nsteps) ls.nsteps[run] = n + 1;
      if (last) ls.active[run] = 0;
    }
    if (last) break;  // the same in every block
    const T aT = (T)alpha, ibT = (T)ib;
    for (int i = threadIdx.x; i < ns; i += blockDim.x) {
      const T x = X[s0 + i];
      const T v = fma(-aT, x, W[i]) * ibT;
      P[i] = x;
      for (int r = 0; r < nb; ++r) cluster.map_shared_rank(X, r)[s0 + i] = v;
    }
    cluster.sync();
  }
  for (int i = threadIdx.x; i < ns; i += blockDim.x) {
    const int64_t o = (int64_t)(ud[i] >> 16) * sv.ld + (ud[i] & 0xffffu);
    V[o] = X[s0 + i];
    VP[o] = P[i];
  }
}

// Blocks per run for `runs` runs of a sector, 0 when the launches of the one-pass kernels are the
// better choice.  Model of both, in clocks per level (FP64 operations per element: hops + 7; an SM does
// two a clock): a cluster pays for the rounds of its slice over the SMs and ~4,000 clocks of barriers
// and scalars, the launches for all elements over all SMs (at ~75 % of the pipe) and ~14,000 clocks of
// launches and tails (7 us, as measured on 36 runs of 3,920 states).
int small_cluster_size(const SectorView& sv, int dtype, int runs, double hops) {
  const int64_t dim = sv.d_up * sv.d_dn;
  if (dim > 24576 || sv.d_up > 65535 || sv.d_dn > 65535 || runs < 1 || runs > 4096) return 0;
  const size_t es = dtype == ED_FP64 ? 8 : 4;
  const double per = (dtype == ED_FP64 ? hops + 7.0 : 6.0) / 2.0;
  double best = runs * (double)dim * per / 152.0 / 0.75 + 14000.0;
  int pick = 0;
  for (int nb = 1; nb <= kSmallMaxCluster; nb *= 2) {
    const int slice = (int)((dim + nb - 1) / nb);
    if (small_smem(dim, slice, es) > 200 * 1024) continue;
    const double rounds = std::max(1.0, runs * nb / 152.0);
    const double whole = rounds > 1.0 ? std::ceil(rounds) : 1.0;
    const double t = whole * slice * per + 4000.0;
    if (t < best) {
      best = t;
      pick = nb;
    }
  }
  return pick;
}

// Levels [n0, n1) of `runs` runs (V = v_{n0}, VP = v_{n0 - 1}; on return the last two vectors), nb blocks
// per run.  A run stops early as in launch_lanczos_step.
void launch_small_levels(const SectorView& sv, const HopParams& hp, int dtype, void* V, void* VP, int64_t vstride, int runs,
                         int n0, int n1, const LanczosScalars& ls, int nb, cudaStream_t s) {
  const int64_t dim = sv.d_up * sv.d_dn;
  const int slice = (int)((dim + nb - 1) / nb);
  const size_t es = dtype == ED_FP64 ? 8 : 4;
  ProfScope ps_(K_LANCZOS_STEP, s, 3.0 * es * (double)dim * runs * (n1 - n0));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(runs * nb));
  cfg.blockDim = dim3(kSmallThreads);
  cfg.dynamicSmemBytes = small_smem(dim, slice, es);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)nb;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (dtype == ED_FP64) {
    allow_max_dynamic_smem(k_small_levels<double>);
    ED_CUDA(cudaLaunchKernelEx(&cfg, k_small_levels<double>, sv, hp, (double*)V, (double*)VP, vstride, slice, n0, n1, ls));
  } else {
    allow_max_dynamic_smem(k_small_levels<float>);
    ED_CUDA(cudaLaunchKernelEx(&cfg, k_small_levels<float>, sv, hp, (float*)V, (float*)VP, vstride, slice, n0, n1, ls));
  }
}

}  // namespace ed
