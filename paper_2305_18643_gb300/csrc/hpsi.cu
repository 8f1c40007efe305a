// K3: matrix-free factorized H.psi (Eq. factorized, Sec. 4.1) and the fused Lanczos step
// (Eq. LanczosRecursion, Sec. 4.2).
//
//   y[u][d] = D(u, d) x[u][d] + sum_{u'} K_up[u][u'] x[u'][d] + sum_{d'} K_dn[d][d'] x[u][d']
//   D(u, d) = e_up[u] + e_dn[d] + sum_{i in cluster} U_i n_{i up} n_{i dn}
//
// e_s[r] = sum_a h_aa n_a is the one-body diagonal of each spin state; the interaction is a
// popcount-style loop over the set bits of b_up & b_dn & (orbitals with U != 0).  The
// off-diagonal K_s come from the packed tables of sector.cu.  Vectors are psi[u][d] with leading
// dimension ld; the up-spin hop reads whole rows, the down-spin hop gathers inside a row.
//
// The fused step computes w = H x - b_n x_prev, overwrites x_prev with w and reduces
// <x, w>, <w, w>, <x, x> in FP64 with a fixed-order block tree; the last block of each run
// (ticket counter) adds the block partials in a fixed order and finishes
// alpha_n = <x,w>/<x,x> and b_{n+1}^2 = <w,w> - <x,w>^2/<x,x>, so the recursion never leaves
// the device and repeated runs are bitwise identical.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "ed_common.cuh"
#include "hpsi_element.cuh"

namespace ed {

constexpr int kThreads = 256;

// ---- one-pass forms ---------------------------------------------------------------------
// With FP64 vectors they are bound by the FP64 pipe (two lanes per clock and SM): one multiply-add per
// hop and as little else in FP64 as possible (signs by integer operations, U sum n n by one
// multiply-add on the popcount), all lanes of a warp on elements.
//  - k_hpsi_flat: a thread per element of the flat index, for sectors of short rows (d_dn < 192),
//    where rows dealt to blocks would leave most of their threads idle; with ROWS, rows over blocks, for
//    rows too long for shared memory or (FP32) that fill an SM's by themselves.  Rows are cut into chunks of columns
//    until every block has four: 20 rows of 184,756 (20 orbitals, (1, 10) particles) took 1,560 us FP32 and
//    1,814 us FP64 whole, 62 and 144 us in chunks.  8,568 rows of 48,620 (18 orbitals, (5, 9)) stay whole, so that
//    a row's operands stay in its SM's L1: 8.0 ms FP32, 9.3 ms in chunks of 512, 11.1 ms staged one row a tile.
//  - k_hpsi_tile: TU rows at a time staged in shared memory as [d][TU], a thread per column: every
//    down-spin entry serves TU rows, the up-spin entries of the rows are staged once per tile.
// The fused forms compute w = H x - b_n x_prev over x_prev and reduce <x, w>, <w, w>, <x, x>; the last block
// of a run (ticket) finishes alpha_n and b_{n+1}.
// 12-orbital impurity, 853,776 states, FP64: 94 us with rows dealt to blocks of 256 and a
// product, its negative and a sum per hop; 42 us in tiles.  36 runs of 3,920 states, fused: 32 us
// before, 22 us flat.

// Block sums, the ticket and the scalars of a fused step; part3 in FP64.  part holds 3 gridDim.x slots.
__device__ __forceinline__ void finish_step(double sxw, double sww, double sxx, int run, int n, const LanczosScalars& ls) {
  __shared__ bool s_last;
  block_sum3_any(sxw, sww, sxx);
  double* part = ls.partial + ((int64_t)run * gridDim.x) * 3;
  if (threadIdx.x == 0) {
    part[blockIdx.x * 3 + 0] = sxw;
    part[blockIdx.x * 3 + 1] = sww;
    part[blockIdx.x * 3 + 2] = sxx;
    __threadfence();
    unsigned t = atomicAdd(ls.counter + run, 1u);
    s_last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double a = 0.0, b = 0.0, c = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
    a += __ldcg(part + i * 3 + 0);
    b += __ldcg(part + i * 3 + 1);
    c += __ldcg(part + i * 3 + 2);
  }
  block_sum3_any(a, b, c);
  if (threadIdx.x == 0) {
    double alpha = c > 0.0 ? a / c : 0.0;
    double b2 = c > 0.0 ? b - a * a / c : 0.0;
    double bnext = b2 > 0.0 ? sqrt(b2) : 0.0;
    int64_t base = (int64_t)run * ls.mstride;
    ls.alpha[base + n] = alpha;
    ls.beta[(int64_t)run * (ls.mstride + 1) + n + 1] = bnext;
    if (ls.nsteps) ls.nsteps[run] = n + 1;
    if (!(bnext > ls.btol * ls.beta0[run]) || n + 1 >= ls.mstride) ls.active[run] = 0;
    ls.counter[run] = 0u;
  }
}

template <typename T, bool FUSED, bool ROWS>
__global__ void __launch_bounds__(kThreads) k_hpsi_flat(SectorView sv, HopParams hp, const T* __restrict__ X0,
                                                        T* __restrict__ O0, int64_t vstride, int n, LanczosScalars ls) {
  __shared__ T sval[kMaxVals];
  __shared__ T sU[kMaxOrb];
  const int run = blockIdx.y;
  if (FUSED && !ls.active[run]) return;
  load_params<T>(hp, sval, sU);
  const T* X = X0 + run * vstride;
  T* O = O0 + run * vstride;
  const T* P = FUSED && ls.prev ? (const T*)ls.prev : O;
  const T bn = FUSED ? (T)ls.beta[(int64_t)run * (ls.mstride + 1) + n] : T(0);
  double sxw = 0.0, sww = 0.0, sxx = 0.0;
  auto element = [&](int64_t u, int64_t d) {
    const int64_t o = u * sv.ld + d;
    T w = hpsi_element<T>(sv, sval, sU, hp, X, u, d);
    if (FUSED) {
      w = fma(-bn, P[o], w);
      const double x = (double)X[o], wd = (double)w;
      sxw = fma(x, wd, sxw);
      sww = fma(wd, wd, sww);
      sxx = fma(x, x, sxx);
    }
    O[o] = w;
  };
  if constexpr (ROWS) {
    const int64_t per = (4 * (int64_t)gridDim.x + sv.d_up - 1) / sv.d_up;  // chunks of a row
    const int64_t chunk = ((sv.d_dn + per - 1) / per + 31) / 32 * 32;
    const int64_t nchunk = (sv.d_dn + chunk - 1) / chunk, units = sv.d_up * nchunk;
    for (int64_t unit = blockIdx.x; unit < units; unit += gridDim.x) {
      const int64_t u = unit / nchunk, c0 = (unit - u * nchunk) * chunk;
      const int64_t c1 = c0 + chunk < sv.d_dn ? c0 + chunk : sv.d_dn;
      for (int64_t d = c0 + threadIdx.x; d < c1; d += blockDim.x) element(u, d);
    }
  } else {
    const uint32_t dim = (uint32_t)(sv.d_up * sv.d_dn), dd = (uint32_t)sv.d_dn;  // d_dn < 192 keeps it below 2^32
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < dim; i += gridDim.x * blockDim.x) {
      const uint32_t u = i / dd;
      element(u, i - u * dd);
    }
  }
  if (FUSED) finish_step(sxw, sww, sxx, run, n, ls);
}

// Threads of a tiled block, at most.  FP32 products wait for their loads, so a tile that leaves no room for a second
// block on its SM takes 1,024: 16 orbitals, (5, 8) particles, rows of 12,870, 1,308 us with 512, 762 us with 1,024
// (992 us with rows dealt to blocks, 1,039 us in two blocks with tiles of half the rows).  FP64 is bound by its pipe.
constexpr int kTileThreads = 512;
constexpr int kTileThreadsAlone = 1024;
constexpr int kFlatMaxRow = 192;   // shorter rows take the flat form

// The staged tile: TU values of one column side by side.
template <typename T, int TU>
struct alignas(TU * sizeof(T) < 16 ? TU * sizeof(T) : 16) TileCol {
  T v[TU];
};
// An up-spin entry of a row: element offset of the operand row and signed value.
template <typename T>
struct alignas(16) UpHop {
  int64_t off;
  T v;
};

template <typename T, int TU, bool FUSED>
__global__ void __launch_bounds__(sizeof(T) == 4 ? kTileThreadsAlone : kTileThreads) k_hpsi_tile(SectorView sv, HopParams hp, const T* __restrict__ X0,
                                                            T* __restrict__ O0, int64_t vstride, int nchunk, int chunk,
                                                            int zup, int n, LanczosScalars ls) {
  using Col = TileCol<T, TU>;
  extern __shared__ __align__(16) unsigned char tile_smem[];
  Col* sx = reinterpret_cast<Col*>(tile_smem);                                          // [d_dn]
  UpHop<T>* sup = reinterpret_cast<UpHop<T>*>(tile_smem + (sv.d_dn * sizeof(Col) + 15) / 16 * 16);  // [TU][zup]
  __shared__ T sval[2 * kMaxVals];  // signed: (vidx << 1) | neg
  __shared__ T sU[kMaxOrb];
  const int run = blockIdx.y;
  if (FUSED && !ls.active[run]) return;
  for (int i = threadIdx.x; i < 2 * kMaxVals; i += blockDim.x) sval[i] = flip_sign(Prec<T>::val(hp, i >> 1), i & 1);
  for (int i = threadIdx.x; i < kMaxOrb; i += blockDim.x) sU[i] = Prec<T>::U(hp, i);
  const T* X = X0 + run * vstride;
  T* O = O0 + run * vstride;
  const T* P = FUSED && ls.prev ? (const T*)ls.prev : O;
  const T bn = FUSED ? (T)ls.beta[(int64_t)run * (ls.mstride + 1) + n] : T(0);
  const bool uni = hp.uniform_u != 0;
  const T u0 = Prec<T>::u0(hp);
  const int dd = (int)sv.d_dn;
  const T* eup = Prec<T>::e_up(sv);
  const T* edn = Prec<T>::e_dn(sv);
  double sxw = 0.0, sww = 0.0, sxx = 0.0;
  const int64_t units = (sv.d_up + TU - 1) / TU * nchunk;
  for (int64_t unit = blockIdx.x; unit < units; unit += gridDim.x) {
    const int64_t ub = unit / nchunk * TU;
    const int c0 = (int)(unit % nchunk) * chunk, c1 = min(dd, c0 + chunk);
    __syncthreads();
    for (int d = threadIdx.x; d < dd; d += blockDim.x) {
      Col c;
#pragma unroll
      for (int r = 0; r < TU; ++r) c.v[r] = ub + r < sv.d_up ? __ldg(X + (ub + r) * sv.ld + d) : T(0);
      sx[d] = c;
    }
    int nup[TU];
    uint32_t bu[TU];
    T eu[TU];
#pragma unroll
    for (int r = 0; r < TU; ++r) {
      const bool ok = ub + r < sv.d_up;
      const int32_t p0 = ok ? sv.ptr_up[ub + r] : 0;
      nup[r] = ok ? sv.ptr_up[ub + r + 1] - p0 : 0;
      bu[r] = ok ? sv.B_up[ub + r] & hp.umask : 0u;
      eu[r] = ok ? eup[ub + r] : T(0);
      for (int k = threadIdx.x; k < nup[r]; k += blockDim.x) {
        const uint32_t e = __ldg(sv.ent_up + p0 + k);
        sup[r * zup + k] = UpHop<T>{(int64_t)ent_col(e) * sv.ld, flip_sign(Prec<T>::val(hp, ent_vidx(e)), ent_neg(e))};
      }
    }
    __syncthreads();
    for (int d = c0 + threadIdx.x; d < c1; d += blockDim.x) {
      const Col x = sx[d];
      const uint32_t bd = sv.B_dn[d];
      const T ed = edn[d];
      T acc[TU];
#pragma unroll
      for (int r = 0; r < TU; ++r) acc[r] = hpsi_diag<T>(eu[r] + ed, bu[r] & bd, sU, uni, u0) * x.v[r];
      const int32_t p1 = sv.ptr_dn[d + 1];
      for (int32_t k = sv.ptr_dn[d]; k < p1; k += 4) {
        uint32_t e[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) e[i] = __ldg(sv.ent_dn + (k + i < p1 ? k + i : k));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (k + i >= p1) break;
          const T v = sval[((e[i] & 127u) << 1) | ent_neg(e[i])];
          const Col g = sx[ent_col(e[i])];
#pragma unroll
          for (int r = 0; r < TU; ++r) acc[r] = fma(v, g.v[r], acc[r]);
        }
      }
      const T* Xd = X + d;
#pragma unroll
      for (int r = 0; r < TU; ++r) {
        const UpHop<T>* h = sup + r * zup;
        int k = 0;
        for (; k + 4 <= nup[r]; k += 4) {
          T xv[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) xv[i] = __ldg(Xd + h[k + i].off);
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[r] = fma(h[k + i].v, xv[i], acc[r]);
        }
        for (; k < nup[r]; ++k) acc[r] = fma(h[k].v, __ldg(Xd + h[k].off), acc[r]);
      }
#pragma unroll
      for (int r = 0; r < TU; ++r) {
        if (ub + r >= sv.d_up) break;
        const int64_t o = (ub + r) * sv.ld + d;
        T w = acc[r];
        if (FUSED) {
          w = fma(-bn, P[o], w);
          const double xd = (double)x.v[r], wd = (double)w;
          sxw = fma(xd, wd, sxw);
          sww = fma(wd, wd, sww);
          sxx = fma(xd, xd, sxx);
        }
        O[o] = w;
      }
    }
  }
  if (FUSED) finish_step(sxw, sww, sxx, run, n, ls);
}

// ---- two-pass form for vectors larger than L2 ------------------------------------------
// Row pass: R rows are staged in shared memory interleaved as [d][R] (one 16-byte vector per
// column), so every down-spin gather serves R rows; the diagonal and -b_n x_prev are applied
// in the same pass, in place on the output.  Column pass: the grid walks column chunks of
// 32 * NV columns (slow index) over row blocks (fast index), so the chunk of x that the up-spin
// hops read, d_up x 32 NV elements, stays in L2 while every row block reads it; each warp owns
// one row at a time and gathers whole 16-byte-per-lane row segments; the Lanczos reductions are
// fused.  Requires ld >= round_up(d_dn, 128), ld % NV == 0, 16-byte aligned vectors and zero
// padding columns (kept zero by every kernel).
template <typename T>
struct Vec;
template <>
struct Vec<float> {
  using t = float4;
  static constexpr int n = 4;
  __device__ static float get(const float4& v, int j) { return j == 0 ? v.x : j == 1 ? v.y : j == 2 ? v.z : v.w; }
  __device__ static float4 make(const float* a) { return make_float4(a[0], a[1], a[2], a[3]); }
  __device__ static void fma(float4& acc, float s, const float4& x) {
    acc.x = fmaf(s, x.x, acc.x);
    acc.y = fmaf(s, x.y, acc.y);
    acc.z = fmaf(s, x.z, acc.z);
    acc.w = fmaf(s, x.w, acc.w);
  }
};
template <>
struct Vec<double> {
  using t = double2;
  static constexpr int n = 2;
  __device__ static double get(const double2& v, int j) { return j == 0 ? v.x : v.y; }
  __device__ static double2 make(const double* a) { return make_double2(a[0], a[1]); }
  __device__ static void fma(double2& acc, double s, const double2& x) {
    acc.x = ::fma(s, x.x, acc.x);
    acc.y = ::fma(s, x.y, acc.y);
  }
};

constexpr int kRowThreads = 1024;

// Per-thread partial sums of <x,w>, <w,w>, <x,x>: FP64 for FP64 vectors; compensated (Kahan)
// FP32 for FP32 vectors, so that no per-element FP64 arithmetic is needed (FP64 runs at a
// small fraction of the FP32 rate on this GPU).
template <typename T>
struct Partial3;
template <>
struct Partial3<double> {
  double s[3] = {0.0, 0.0, 0.0};
  __device__ void add(double x, double w) {
    s[0] += x * w;
    s[1] += w * w;
    s[2] += x * x;
  }
  __device__ void get(double& a, double& b, double& c) const {
    a = s[0];
    b = s[1];
    c = s[2];
  }
};
template <>
struct Partial3<float> {
  float s[3] = {0.f, 0.f, 0.f}, k[3] = {0.f, 0.f, 0.f};
  __device__ void add1(int i, float v) {
    const float y = v - k[i];
    const float t = s[i] + y;
    k[i] = (t - s[i]) - y;
    s[i] = t;
  }
  __device__ void add(float x, float w) {
    add1(0, x * w);
    add1(1, w * w);
    add1(2, x * x);
  }
  __device__ void get(double& a, double& b, double& c) const {
    a = (double)s[0] - (double)k[0];
    b = (double)s[1] - (double)k[1];
    c = (double)s[2] - (double)k[2];
  }
};

// ---- accumulators of 16-byte groups: four FP32 rows (packed FMAs, fma.rn.f32x2, on the row
// pairs (0,1) and (2,3)) or two FP64 rows.
__device__ __forceinline__ unsigned long long f2_pack(float x, float y) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 f2_unpack(unsigned long long r) {
  float2 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(r));
  return v;
}
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

template <typename T>
struct Acc16;
template <>
struct Acc16<float> {
  unsigned long long a, b;  // rows (0,1), rows (2,3)
  __device__ void set(const float* v) {
    a = f2_pack(v[0], v[1]);
    b = f2_pack(v[2], v[3]);
  }
  // acc += s * (16-byte group x)
  __device__ void fma(float s, const ulonglong2& x) {
    const unsigned long long ss = f2_pack(s, s);
    a = f2_fma(ss, x.x, a);
    b = f2_fma(ss, x.y, b);
  }
  // the same with s given as the pair (s, s)
  __device__ void fma_pair(unsigned long long ss, const ulonglong2& x) {
    a = f2_fma(ss, x.x, a);
    b = f2_fma(ss, x.y, b);
  }
  __device__ float get(int r) const {
    const float2 p = f2_unpack(r < 2 ? a : b);
    return (r & 1) ? p.y : p.x;
  }
  __device__ void set_vec(const float4& v) {
    a = f2_pack(v.x, v.y);
    b = f2_pack(v.z, v.w);
  }
  __device__ float4 vec() const {
    const float2 p = f2_unpack(a), q = f2_unpack(b);
    return make_float4(p.x, p.y, q.x, q.y);
  }
};
template <>
struct Acc16<double> {
  double a, b;
  __device__ void set(const double* v) {
    a = v[0];
    b = v[1];
  }
  __device__ void fma(double s, const ulonglong2& x) {
    a = ::fma(s, __longlong_as_double((long long)x.x), a);
    b = ::fma(s, __longlong_as_double((long long)x.y), b);
  }
  __device__ void fma_pair(unsigned long long s, const ulonglong2& x) { fma(__longlong_as_double((long long)s), x); }
  __device__ double get(int r) const { return r == 0 ? a : b; }
  __device__ void set_vec(const double2& v) {
    a = v.x;
    b = v.y;
  }
  __device__ double2 vec() const { return make_double2(a, b); }
};

// Row pass: O[u][:] = (D + K_dn) X[u][:] - b O[u][:] for R interleaved rows per step.  The rows
// are staged in shared memory as 16-byte groups (one per column); each thread owns columns d and
// gathers the groups sx[col] of its hops.  The slot-major entries (row_ell_pack) carry the byte
// offsets of the group and of the signed hop value, so a hop costs one table load, two shared
// loads and the FMAs (one shared load when the cluster has at most four distinct hop values,
// REG: the value is then selected in registers).  Table loads run one chunk of kPre slots ahead
// of their use (the table has kEllPad zero slots at its end, so the look-ahead needs no bounds
// check).
// PREV: the vector of the -b term (beta) is P0's, else it is the output's old content.
template <typename T, bool REG, bool PREV>
__global__ void __launch_bounds__(kRowThreads) k_down_rows(SectorArgs sv, HopParams hp, const T* __restrict__ X0,
                                                   T* __restrict__ O0, const T* P0, int64_t vstride,
                                                   const double* __restrict__ beta, int beta_stride, int n_step,
                                                   const int* __restrict__ active) {
  constexpr int R = Vec<T>::n;
  constexpr int kPre = kEllPad;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* sxb = smem_raw;                                  // [d_dn] 16-byte groups
  T* ssv = reinterpret_cast<T*>(smem_raw + sv.d_dn * 16);         // [256] signed values, (vidx << 1) | neg
  T* sU = ssv + 256;
  const int run = blockIdx.y;
  if (active && !active[run]) return;
  for (int i = threadIdx.x; i < 256; i += blockDim.x) {
    const T v = Prec<T>::val(hp, i >> 1);
    ssv[i] = (i & 1) ? -v : v;
  }
  for (int i = threadIdx.x; i < kMaxOrb; i += blockDim.x) sU[i] = Prec<T>::U(hp, i);
  const T u0 = sizeof(T) == 8 ? (T)hp.u0 : (T)hp.u0f;
  const bool uni = hp.uniform_u != 0;
  const T* X = X0 + run * vstride;
  T* O = O0 + run * vstride;
  const T b = beta ? (T)beta[(int64_t)run * beta_stride + n_step] : T(0);
  const int64_t du = sv.d_up, dd = sv.d_dn, ld = sv.ld;
  const T* eup = Prec<T>::e_up(sv);
  const T* edn = Prec<T>::e_dn(sv);
  const unsigned char* ssvb = reinterpret_cast<const unsigned char*>(ssv);
  const T v0 = Prec<T>::val(hp, 0), v1 = Prec<T>::val(hp, 1), v2 = Prec<T>::val(hp, 2), v3 = Prec<T>::val(hp, 3);
  auto hop = [&](Acc16<T>& acc, uint32_t e) {
    T v;
    if constexpr (REG) {  // at most four distinct values: select in registers, sign bit from the entry
      const uint32_t i = (e >> 3) & 3u;
      v = (i & 2u) ? ((i & 1u) ? v3 : v2) : ((i & 1u) ? v1 : v0);
      if constexpr (sizeof(T) == 4)
        v = __int_as_float(__float_as_int(v) ^ (int)((e & 4u) << 29));
      else
        v = __longlong_as_double(__double_as_longlong(v) ^ ((long long)(e & 4u) << 61));
    } else {
      v = *reinterpret_cast<const T*>(ssvb + (e & 0x3FCu) * (sizeof(T) / 4));
    }
    acc.fma(v, *reinterpret_cast<const ulonglong2*>(sxb + (e >> 10)));
  };
  for (int64_t u0r = (int64_t)blockIdx.x * R; u0r < du; u0r += (int64_t)gridDim.x * R) {
    __syncthreads();
    for (int64_t d = threadIdx.x; d < dd; d += blockDim.x) {
      T v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = (u0r + r < du) ? X[(u0r + r) * ld + d] : T(0);
      *reinterpret_cast<typename Vec<T>::t*>(sxb + d * 16) = Vec<T>::make(v);
    }
    __syncthreads();
    uint32_t bu[R];
    T eu[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      bool ok = u0r + r < du;
      bu[r] = ok ? sv.B_up[u0r + r] : 0u;
      eu[r] = ok ? eup[u0r + r] : T(0);
    }
    for (int64_t d = threadIdx.x; d < dd; d += blockDim.x) {
      const int32_t nz = sv.ptr_dn[d + 1] - sv.ptr_dn[d];
      const uint32_t* p = sv.ell_dn + d;
      uint32_t e[kPre];
#pragma unroll
      for (int i = 0; i < kPre; ++i) e[i] = __ldg(p + i * dd);
      p += kPre * dd;
      const uint32_t bd = sv.B_dn[d];
      const T ed = edn[d];
      [[maybe_unused]] T pv[R];  // v_{n-1}, requested before the hops
      if constexpr (PREV) {
#pragma unroll
        for (int r = 0; r < R; ++r) pv[r] = u0r + r < du ? P0[run * vstride + (u0r + r) * ld + d] : T(0);
      }
      Acc16<T> acc;
      {
        const typename Vec<T>::t xv = *reinterpret_cast<const typename Vec<T>::t*>(sxb + d * 16);
        T a[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          T diag = eu[r] + ed;
          uint32_t dbl = bu[r] & bd & hp.umask;
          if (uni) {
            diag += u0 * (T)__popc(dbl);
          } else {
            while (dbl) {
              diag += sU[__ffs(dbl) - 1];
              dbl &= dbl - 1u;
            }
          }
          a[r] = diag * Vec<T>::get(xv, r);
        }
        acc.set(a);
      }
      int32_t k = 0;
      for (; k + kPre <= nz; k += kPre) {
        uint32_t f[kPre];
#pragma unroll
        for (int i = 0; i < kPre; ++i) {
          f[i] = e[i];
          e[i] = __ldg(p + i * dd);  // slots k + kPre + i <= zmax + kEllPad - 1
        }
        p += kPre * dd;
#pragma unroll
        for (int i = 0; i < kPre; ++i) hop(acc, f[i]);
      }
#pragma unroll
      for (int i = 0; i < kPre; ++i)
        if (k + i < nz) hop(acc, e[i]);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (u0r + r >= du) continue;
        const int64_t o = (u0r + r) * ld + d;
        T out = acc.get(r);
        if (PREV)
          out -= b * pv[r];
        else if (beta)
          out -= b * O[o];
        O[o] = out;
      }
    }
  }
}

template <typename T, bool FUSED>
__global__ void __launch_bounds__(kThreads, 4) k_up_cols(SectorArgs sv, HopParams hp, const T* __restrict__ X0,
                                                      T* __restrict__ O0, int64_t vstride, int rows_per_cta, int n,
                                                      LanczosScalars ls) {
  using RV = typename Vec<T>::t;
  constexpr int NV = Vec<T>::n;
  __shared__ T sval[kMaxVals];
  __shared__ bool s_last;
  const int run = blockIdx.z;
  if (FUSED && !ls.active[run]) return;
  for (int i = threadIdx.x; i < kMaxVals; i += blockDim.x) sval[i] = Prec<T>::val(hp, i);
  __syncthreads();
  const T* X = X0 + run * vstride;
  T* O = O0 + run * vstride;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const int64_t ld = sv.ld;
  const int64_t c0 = (int64_t)blockIdx.y * (32 * NV) + lane * NV;
  const T* Xc = X + c0;
  const int64_t ub = (int64_t)blockIdx.x * rows_per_cta;
  const int64_t ue = ub + rows_per_cta < sv.d_up ? ub + rows_per_cta : sv.d_up;
  Partial3<T> part3;
  for (int64_t u = ub + warp; u < ue; u += nwarp) {
    RV* op = reinterpret_cast<RV*>(O + u * ld + c0);
    RV acc = *op;
    const int32_t p0 = sv.ptr_up[u], p1 = sv.ptr_up[u + 1];
    Acc16<T> a16;
    a16.set_vec(acc);
    for (int32_t base = p0; base < p1; base += 32) {
      // the warp's next 32 entries: lane j holds entry base + j (column and signed value)
      const int cnt = p1 - base < 32 ? p1 - base : 32;
      const uint32_t me = lane < cnt ? __ldg(sv.ent_up + base + lane) : 0u;
      const uint32_t mcol = ent_col(me);
      T mv = sval[ent_vidx(me)];
      mv = ent_neg(me) ? -mv : mv;
      int j = 0;
      for (; j + 4 <= cnt; j += 4) {
        ulonglong2 xv[4];
        T v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t col = __shfl_sync(0xffffffffu, mcol, j + i);
          v[i] = __shfl_sync(0xffffffffu, mv, j + i);
          xv[i] = __ldg(reinterpret_cast<const ulonglong2*>(Xc + (int64_t)col * ld));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) a16.fma(v[i], xv[i]);
      }
      for (; j < cnt; ++j) {
        const uint32_t col = __shfl_sync(0xffffffffu, mcol, j);
        const T v = __shfl_sync(0xffffffffu, mv, j);
        a16.fma(v, __ldg(reinterpret_cast<const ulonglong2*>(Xc + (int64_t)col * ld)));
      }
    }
    acc = a16.vec();
    *op = acc;
    if (FUSED) {
      const RV xs = __ldg(reinterpret_cast<const RV*>(X + u * ld + c0));
#pragma unroll
      for (int j = 0; j < NV; ++j)
        if (c0 + j < sv.d_dn) part3.add(Vec<T>::get(xs, j), Vec<T>::get(acc, j));
    }
  }
  if (!FUSED) return;
  double sxw, sww, sxx;
  part3.get(sxw, sww, sxx);
  block_sum3<kThreads>(sxw, sww, sxx);
  const unsigned nblk = gridDim.x * gridDim.y;
  const unsigned bid = blockIdx.y * gridDim.x + blockIdx.x;
  double* part = ls.partial + ((int64_t)run * nblk) * 3;
  if (threadIdx.x == 0) {
    part[bid * 3 + 0] = sxw;
    part[bid * 3 + 1] = sww;
    part[bid * 3 + 2] = sxx;
    __threadfence();
    unsigned t = atomicAdd(ls.counter + run, 1u);
    s_last = (t == nblk - 1);
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double a = 0.0, b = 0.0, c = 0.0;
  for (unsigned i = threadIdx.x; i < nblk; i += blockDim.x) {
    a += __ldcg(part + i * 3 + 0);
    b += __ldcg(part + i * 3 + 1);
    c += __ldcg(part + i * 3 + 2);
  }
  block_sum3<kThreads>(a, b, c);
  if (threadIdx.x == 0) {
    double alpha = c > 0.0 ? a / c : 0.0;
    double b2 = c > 0.0 ? b - a * a / c : 0.0;
    double bnext = b2 > 0.0 ? sqrt(b2) : 0.0;
    ls.alpha[(int64_t)run * ls.mstride + n] = alpha;
    ls.beta[(int64_t)run * (ls.mstride + 1) + n + 1] = bnext;
    if (ls.nsteps) ls.nsteps[run] = n + 1;
    if (!(bnext > ls.btol * ls.beta0[run]) || n + 1 >= ls.mstride) ls.active[run] = 0;
    ls.counter[run] = 0u;
  }
}

constexpr int kRowsPerCta = 64;
static std::atomic<int> g_smem_optin{-1};  // opt-in shared memory per block (read by concurrent lanes)

static int smem_optin() {
  int lim = g_smem_optin.load(std::memory_order_relaxed);
  if (lim < 0) {
    int dev = 0;
    ED_CUDA(cudaGetDevice(&dev));
    ED_CUDA(cudaDeviceGetAttribute(&lim, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    g_smem_optin.store(lim, std::memory_order_relaxed);
  }
  return lim;
}

static size_t down_rows_smem(const SectorView& sv, int dtype) {
  const size_t es = dtype == ED_FP64 ? 8 : 4;
  return (size_t)sv.d_dn * 16 + (256 + kMaxOrb) * es;
}

// The two-pass form applies when the vector has at least sv.two_pass_min_bytes (32 MiB unless the
// cluster's ED_OPT_TWO_PASS_MIN_BYTES says otherwise: beyond that it no longer fits L2
// comfortably) and the layout allows 16-byte vector access.
bool use_two_pass(const SectorView& sv, int dtype, const void* X, const void* O, int64_t vstride) {
  const int64_t es = dtype == ED_FP64 ? 8 : 4, NV = dtype == ED_FP64 ? 2 : 4;
  if (sv.d_up * sv.d_dn * es < sv.two_pass_min_bytes) return false;
  const int64_t need = (sv.d_dn + 32 * NV - 1) / (32 * NV) * (32 * NV);
  if (sv.ld < need || sv.ld % NV != 0) return false;
  if (((uintptr_t)X | (uintptr_t)O) % 16 != 0 || (vstride * es) % 16 != 0) return false;
  return down_rows_smem(sv, dtype) <= (size_t)smem_optin();
}

template <typename T>
static void launch_two_pass(const SectorView& sv, const HopParams& hp, const T* X, T* O, int64_t vstride, int runs,
                            const double* beta, int beta_stride, int n, const LanczosScalars* ls, cudaStream_t s) {
  const double es = sizeof(T);
  const double dim = (double)sv.d_up * sv.d_dn;
  const size_t smem = down_rows_smem(sv, sizeof(T) == 8 ? ED_FP64 : ED_FP32);
  const bool reg = hp.nvals <= 4;
  const int64_t groups = (sv.d_up + Vec<T>::n - 1) / Vec<T>::n;
  dim3 g1((unsigned)std::min<int64_t>(groups, 152), runs);
  dim3 g2((unsigned)((sv.d_up + kRowsPerCta - 1) / kRowsPerCta), (unsigned)((sv.d_dn + 32 * Vec<T>::n - 1) / (32 * Vec<T>::n)),
          runs);
  // one timed unit per step: both passes (the second launch is counted separately)
  ProfScope ps_(ls ? K_LANCZOS_STEP : K_HPSI, s, (beta ? 3.0 : 2.0) * es * dim * runs);
  auto rows = [&](auto r, auto prev) {
    constexpr bool REG = decltype(r)::value, PREV = decltype(prev)::value;
    allow_max_dynamic_smem(k_down_rows<T, REG, PREV>);
    k_down_rows<T, REG, PREV><<<g1, kRowThreads, smem, s>>>(sv, hp, X, O, ls ? (const T*)ls->prev : nullptr, vstride, beta,
                                                            beta_stride, n, ls ? ls->active : nullptr);
  };
  const bool prev = ls && ls->prev;
  if (reg && prev)
    rows(std::true_type(), std::true_type());
  else if (reg)
    rows(std::true_type(), std::false_type());
  else if (prev)
    rows(std::false_type(), std::true_type());
  else
    rows(std::false_type(), std::false_type());
  ED_CHECK_LAUNCH();
  note_launch();
  if (ls)
    k_up_cols<T, true><<<g2, kThreads, 0, s>>>(sv, hp, X, O, vstride, kRowsPerCta, n, *ls);
  else
    k_up_cols<T, false><<<g2, kThreads, 0, s>>>(sv, hp, X, O, vstride, kRowsPerCta, n, LanczosScalars{});
  ED_CHECK_LAUNCH();
}

int two_pass_blocks(const SectorView& sv, int dtype) {
  const int NV = dtype == ED_FP64 ? 2 : 4;
  return (int)(((sv.d_up + kRowsPerCta - 1) / kRowsPerCta) * ((sv.d_dn + 32 * NV - 1) / (32 * NV)));
}

// Rows, chunks and shared memory of the tiled one-pass form for one vector (tu = 0: it does not
// apply and the flat form runs).  Rows below 192 columns cannot fill their warps; four rows per
// tile unless that leaves fewer than four tiles per SM (then the rows are split into chunks of columns,
// each staging the tile again) or the tile exceeds shared memory.  One FP32 row by itself, without a second block beside
// it, is not worth its staging.
struct TilePlan {
  int tu = 0, nchunk = 1, chunk = 0, threads = 0, zup = 0;
  size_t smem = 0;
  int64_t units = 0;
};

static TilePlan tile_plan(const SectorView& sv, int dtype) {
  TilePlan p;
  if (sv.d_dn < kFlatMaxRow) return p;
  const size_t es = dtype == ED_FP64 ? 8 : 4;
  p.zup = std::max(sv.zmax_up, 1);
  const size_t limit = (size_t)smem_optin() - 8 * 1024;  // less the static shared memory
  for (int tu : {4, 2, 1}) {
    const size_t smem = ((size_t)sv.d_dn * tu * es + 15) / 16 * 16 + (size_t)tu * p.zup * 16;
    if (smem > limit || (dtype == ED_FP32 && tu == 1 && smem > limit / 2)) continue;
    // small sectors: fewer rows per tile rather than idle SMs
    if (tu > 1 && (sv.d_up + tu - 1) / tu * ((sv.d_dn + 255) / 256) < 2 * 152) continue;
    p.tu = tu;
    p.smem = smem;
    break;
  }
  if (!p.tu) return p;
  const int64_t tiles = (sv.d_up + p.tu - 1) / p.tu;
  const int64_t want = std::max<int64_t>(1, (4 * 152 + tiles - 1) / tiles);
  p.nchunk = (int)std::min<int64_t>(want, (sv.d_dn + 255) / 256);
  p.chunk = (int)(((sv.d_dn + p.nchunk - 1) / p.nchunk + 31) / 32 * 32);
  p.nchunk = (int)((sv.d_dn + p.chunk - 1) / p.chunk);
  p.threads = std::min(dtype == ED_FP32 && p.smem > limit / 2 ? kTileThreadsAlone : kTileThreads, p.chunk);
  p.units = tiles * p.nchunk;
  return p;
}

constexpr int kOnePassBlocks = 152 * 8;  // blocks per vector of the one-pass forms

static int flat_grid(const SectorView& sv) {
  const int64_t b = (sv.d_up * sv.d_dn + kThreads - 1) / kThreads;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, kOnePassBlocks));
}

template <typename T, int TU>
static void launch_tile(const TilePlan& p, const SectorView& sv, const HopParams& hp, const T* X, T* O, int64_t vstride,
                        int runs, int n, const LanczosScalars* ls, cudaStream_t s) {
  const dim3 g((unsigned)std::min<int64_t>(p.units, kOnePassBlocks), runs);
  if (ls) {
    allow_max_dynamic_smem(k_hpsi_tile<T, TU, true>, p.smem);
    k_hpsi_tile<T, TU, true><<<g, p.threads, p.smem, s>>>(sv, hp, X, O, vstride, p.nchunk, p.chunk, p.zup, n, *ls);
  } else {
    allow_max_dynamic_smem(k_hpsi_tile<T, TU, false>, p.smem);
    k_hpsi_tile<T, TU, false><<<g, p.threads, p.smem, s>>>(sv, hp, X, O, vstride, p.nchunk, p.chunk, p.zup, n,
                                                          LanczosScalars{});
  }
}

// y_r = H x_r (ls == nullptr) or the fused Lanczos step, `runs` vectors vstride apart in one launch.
template <typename T>
static void launch_one_pass(const SectorView& sv, const HopParams& hp, const T* X, T* O, int64_t vstride, int runs, int n,
                            const LanczosScalars* ls, cudaStream_t s) {
  ProfScope ps_(ls ? K_LANCZOS_STEP : K_HPSI, s, (ls ? 3.0 : 2.0) * sizeof(T) * (double)(sv.d_up * sv.d_dn) * runs);
  const TilePlan p = tile_plan(sv, sizeof(T) == 8 ? ED_FP64 : ED_FP32);
  if (p.tu == 4)
    launch_tile<T, 4>(p, sv, hp, X, O, vstride, runs, n, ls, s);
  else if (p.tu == 2)
    launch_tile<T, 2>(p, sv, hp, X, O, vstride, runs, n, ls, s);
  else if (p.tu == 1)
    launch_tile<T, 1>(p, sv, hp, X, O, vstride, runs, n, ls, s);
  else {
    const dim3 g(flat_grid(sv), runs);
    const bool rows = sv.d_dn >= kFlatMaxRow;
    if (ls && rows)
      k_hpsi_flat<T, true, true><<<g, kThreads, 0, s>>>(sv, hp, X, O, vstride, n, *ls);
    else if (ls)
      k_hpsi_flat<T, true, false><<<g, kThreads, 0, s>>>(sv, hp, X, O, vstride, n, *ls);
    else if (rows)
      k_hpsi_flat<T, false, true><<<g, kThreads, 0, s>>>(sv, hp, X, O, vstride, n, LanczosScalars{});
    else
      k_hpsi_flat<T, false, false><<<g, kThreads, 0, s>>>(sv, hp, X, O, vstride, n, LanczosScalars{});
  }
  ED_CHECK_LAUNCH();
}

static int one_pass_blocks(const SectorView& sv, int dtype) {
  const TilePlan p = tile_plan(sv, dtype);
  return p.tu ? (int)std::min<int64_t>(p.units, kOnePassBlocks) : flat_grid(sv);
}

int lanczos_blocks(const SectorView& sv) {
  // capacity for every form (the two-pass column kernel has the most blocks on large sectors)
  return std::max({one_pass_blocks(sv, ED_FP64), one_pass_blocks(sv, ED_FP32), two_pass_blocks(sv, ED_FP64)});
}

void launch_hpsi(const SectorView& sv, const HopParams& hp, int dtype, const void* x, void* y, cudaStream_t s) {
  launch_hpsi_block(sv, hp, dtype, x, y, 0, 1, s);
}

void launch_hpsi_block(const SectorView& sv, const HopParams& hp, int dtype, const void* X, void* Y, int64_t vstride,
                       int runs, cudaStream_t s) {
  const bool two = use_two_pass(sv, dtype, X, Y, vstride);
  if (dtype == ED_FP64) {
    if (two)
      launch_two_pass<double>(sv, hp, (const double*)X, (double*)Y, vstride, runs, nullptr, 0, 0, nullptr, s);
    else
      launch_one_pass<double>(sv, hp, (const double*)X, (double*)Y, vstride, runs, 0, nullptr, s);
  } else {
    if (two)
      launch_two_pass<float>(sv, hp, (const float*)X, (float*)Y, vstride, runs, nullptr, 0, 0, nullptr, s);
    else
      launch_one_pass<float>(sv, hp, (const float*)X, (float*)Y, vstride, runs, 0, nullptr, s);
  }
}

void launch_lanczos_step(const SectorView& sv, const HopParams& hp, int dtype, const void* X, void* XP,
                         int64_t vstride, int runs, int n, const LanczosScalars& ls, int nblk_cap, cudaStream_t s) {
  const bool two = use_two_pass(sv, dtype, X, XP, vstride);
  if ((two ? two_pass_blocks(sv, dtype) : one_pass_blocks(sv, dtype)) > nblk_cap) throw Error(ED_ERR_INVALID, "partial buffer too small");
  if (dtype == ED_FP64) {
    if (two)
      launch_two_pass<double>(sv, hp, (const double*)X, (double*)XP, vstride, runs, ls.beta, ls.mstride + 1, n, &ls, s);
    else
      launch_one_pass<double>(sv, hp, (const double*)X, (double*)XP, vstride, runs, n, &ls, s);
  } else {
    if (two)
      launch_two_pass<float>(sv, hp, (const float*)X, (float*)XP, vstride, runs, ls.beta, ls.mstride + 1, n, &ls, s);
    else
      launch_one_pass<float>(sv, hp, (const float*)X, (float*)XP, vstride, runs, n, &ls, s);
  }
}

}  // namespace ed
