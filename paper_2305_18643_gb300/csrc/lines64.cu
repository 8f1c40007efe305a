// H.psi on FP64 vectors with the hop sums in 64-bit integers (Eq. factorized, Sec. 4.1).
//
// FP64 runs at two lanes per clock and SM on this GPU, a thirtieth of the integer rate, so a product of
// 34 hops per spin and element is bound by its FP64 multiply-adds.  Most clusters have few distinct hop
// magnitudes |t|, and a sum of +-x over the hops of one magnitude needs no FP64: a line of the vector (a
// row for the down-spin hops, a column for the up-spin hops) is staged in shared memory as fixed-point
// numbers of 56 bits below the line's largest exponent, the sums are exact 64-bit integer sums (at most 64
// terms), and each magnitude costs one conversion and one multiply-add per element.
//
// Error: rounding x to the fixed point, at most 2^-57 of the line's maximum, in place of a rounding at
// 2^-53 of the partial sum per hop.  That is the smaller error where the operands are of one order
// (Lanczos vectors: 1 % of a normal distribution lies below 2^-8 of the maximum of 10^4 draws), and the
// larger one for sums of operands far below the line's maximum.  So a line of which more than 1/16 is
// neither zero nor within 2^8 of its maximum, or which is not finite, or below 2^-958, takes the FP64 sums
// of the same kernel.
//
// Two passes, two lines at a time per block interleaved as 16-byte groups [position][2]: rows (down-spin
// hops, diagonal, -b_n x_prev), then columns (up-spin hops; with FUSED the Lanczos sums).  No alignment is
// asked of the vectors or the leading dimension.
// 4x4 periodic cluster (166 M states, 34 hops per spin, 2 magnitudes): rows 13.0, columns 9.8 ms in FP64
// arithmetic; 5.3 and 6.3 ms here, bound by the integer pipes and the shared-memory gathers.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

#include "bank_order.cuh"
#include "ed_common.cuh"
#include "hpsi_element.cuh"

namespace ed {

constexpr int kLineMaxClasses = 4;
constexpr int kLineMaxSlots = 62;  // hops per state: sums of 25-bit upper limbs stay below 2^31
constexpr int kLinePad = 8;        // slots behind a table, for the look-ahead
constexpr int kLineBits = 56;

// Hops of one spin, slot-major [slot][dim]: (source << 4) | (magnitude << 1) | sign, so that an entry less
// its low bits is the byte offset of the source's group.  One list for all magnitudes: the loops of
// lists by magnitude and sign end at different slots in every lane, which leaves gathers half empty.
struct LineTables {
  int classes = 0;  // magnitudes; 0: the spin has too many of them or too many hops
  double mag[kLineMaxClasses] = {};
  DevBuf<uint32_t> ell;  // slots past a state's hops hold (dim << 4): a group of zeros behind the line
  DevBuf<uint8_t> cnt;   // [dim]
  double hops = 0.0;    // mean hops per state
};

struct LineView {
  double mag[kLineMaxClasses];
  const uint32_t* ell;
  const uint8_t* cnt;
};

struct ClassMap {
  uint8_t of[kMaxVals];  // (magnitude << 1) | (the value is negative)
};
// Fills the table for 8 consecutive states per thread, ordered against bank conflicts.
__global__ void k_line_fill(int64_t dim, const int32_t* __restrict__ ptr, const uint32_t* __restrict__ ent, ClassMap cm,
                            int slots, uint32_t* __restrict__ ell, uint8_t* __restrict__ cnt) {
  const int64_t r0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * 8;
  if (r0 >= dim) return;
  const int nr = (int)(dim - r0 < 8 ? dim - r0 : 8);
  for (int i = 0; i < nr; ++i) {
    const int n = ptr[r0 + i + 1] - ptr[r0 + i];
    cnt[r0 + i] = (uint8_t)n;
    for (int k = n; k < slots; ++k) ell[(int64_t)k * dim + r0 + i] = (uint32_t)dim << 4;
  }
  bank_order_group(ptr, ent, r0, nr, [&](int slot, int i, uint32_t e) {
    ell[(int64_t)slot * dim + r0 + i] = (ent_col(e) << 4) | (cm.of[ent_vidx(e)] ^ ent_neg(e));
  });
}

// Builds the table of one spin.
static std::unique_ptr<LineTables> build_lines(const SpinTables& t, const ModelHost& m, cudaStream_t s) {
  PlainAllocScope plain;  // the table is read on any stream
  auto lt = std::make_unique<LineTables>();
  if (t.dim < 2 || t.nnz == 0 || t.zmax > kLineMaxSlots) return lt;
  ClassMap cm = {};
  int classes = 0;
  for (size_t k = 0; k < m.vals.size(); ++k) {
    const double a = std::fabs(m.vals[k]);
    int c = 0;
    while (c < classes && lt->mag[c] != a) ++c;
    if (c == classes) {
      if (classes == kLineMaxClasses) return lt;
      lt->mag[classes++] = a;
    }
    cm.of[k] = (uint8_t)(2 * c + (m.vals[k] < 0.0));
  }
  const size_t n = (size_t)(t.zmax + kLinePad) * t.dim;
  lt->ell.alloc(n);
  lt->cnt.alloc(t.dim);
  {
    ProfScope ps_(K_TABLES, s, 0.0);
    k_line_fill<<<(unsigned)((t.dim + 8 * 32 - 1) / (8 * 32)), 32, 0, s>>>(t.dim, t.ptr.p, t.ent.p, cm, t.zmax + kLinePad,
                                                                               lt->ell.p, lt->cnt.p);
    ED_CHECK_LAUNCH();
  }
  lt->hops = (double)t.nnz / t.dim;
  ED_CUDA(cudaStreamSynchronize(s));  // ready for every stream
  lt->classes = classes;
  return lt;
}

// x as a fixed-point number of kLineBits bits below exponent field emax, rounded to nearest.
__device__ __forceinline__ long long to_fixed(double x, int emax) {
  const int hi = __double2hiint(x);
  const int e = (hi >> 20) & 0x7ff, sh = emax - e;
  if (e == 0 || sh > kLineBits + 1) return 0;
  unsigned long long q = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)__double2loint(x)) << (kLineBits - 53);
  if (sh > 0) q = (q + (1ull << (sh - 1))) >> sh;
  const long long sg = hi >> 31;
  return ((long long)q ^ sg) - sg;
}

__device__ __forceinline__ int block_max(int v, int* sm) {
  v = __reduce_max_sync(0xffffffffu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  v = sm[0];
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = max(v, sm[w]);
  return v;
}
__device__ __forceinline__ int block_add(int v, int* sm) {
  v = __reduce_add_sync(0xffffffffu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  v = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += sm[w];
  return v;
}
// 1 if x is not zero and below 2^-8 of the line's maximum (its exponent field emax).
__device__ __forceinline__ int is_small(double x, int emax) {
  const int hi = __double2hiint(x) & 0x7fffffff;
  return (hi | __double2loint(x)) != 0 && (hi >> 20) < emax - 8;
}

template <bool COLS, bool FUSED, int C>
__global__ void __launch_bounds__(1024, 1) k_lines64(SectorView sv, HopParams hp, LineView lv, const double* __restrict__ X0,
                                                  double* __restrict__ O0, const double* P0, int64_t vstride,
                                                  const double* __restrict__ beta,
                                                  int beta_stride, int n_step, const int* __restrict__ active,
                                                  LanczosScalars ls) {
  extern __shared__ __align__(16) unsigned char ln_smem[];
  __shared__ int smi[32];
  __shared__ double sU[kMaxOrb];
  __shared__ double2 sUn[kMaxOrb + 1], st[kLineMaxClasses];
  __shared__ bool s_last;
  const int run = blockIdx.y;
  if (active && !active[run]) return;
  const double* X = X0 + run * vstride;
  double* O = O0 + run * vstride;
  const int64_t ld = sv.ld;
  const int N = (int)(COLS ? sv.d_up : sv.d_dn), NL = (int)(COLS ? sv.d_dn : sv.d_up);
  int4* sx = reinterpret_cast<int4*>(ln_smem);  // [N + 1]: (low, high) limbs of both lines
  double2* sd = reinterpret_cast<double2*>(ln_smem);
  const bool uni = hp.uniform_u != 0;
  const bool wide = ld % 2 == 0 && (((uintptr_t)X | (uintptr_t)O) & 15) == 0;
  for (int i = threadIdx.x; i < kMaxOrb; i += blockDim.x) sU[i] = hp.U[i];
  if (threadIdx.x == 0) sx[N] = make_int4(0, 0, 0, 0);
  const double b = !COLS && beta ? beta[(int64_t)run * beta_stride + n_step] : 0.0;
  double sxw = 0.0, sww = 0.0, sxx = 0.0;
  for (int l0 = blockIdx.x * 2; l0 < NL; l0 += gridDim.x * 2) {
    const bool two = l0 + 1 < NL;
    const double* Xl = COLS ? X + l0 : X + (int64_t)l0 * ld;
    double* Ol = COLS ? O + l0 : O + (int64_t)l0 * ld;
    const double* Pl = P0 ? P0 + run * vstride + (int64_t)l0 * ld : Ol;  // v_{n-1} (rows)
    const int64_t pstep = COLS ? ld : 1, lstep = COLS ? 1 : ld;
    const bool pair = COLS && two && wide;  // both columns of a position in one 16-byte access
    __syncthreads();
    auto stage = [&](int& m0, int& m1) {
#pragma unroll 4
      for (int i = threadIdx.x; i < N; i += blockDim.x) {
        double2 v;
        if (pair) {
          v = __ldg(reinterpret_cast<const double2*>(Xl + i * pstep));
        } else {
          v.x = __ldg(Xl + i * pstep);
          v.y = two ? __ldg(Xl + i * pstep + lstep) : 0.0;
        }
        sd[i] = v;
        m0 = max(m0, __double2hiint(v.x) & 0x7fffffff);
        m1 = max(m1, __double2hiint(v.y) & 0x7fffffff);
      }
    };
    int m0 = 0, m1 = 0;
    stage(m0, m1);
    const int e0 = block_max(m0, smi) >> 20;
    int e1 = block_max(m1, smi) >> 20;
    if (!two) e1 = e0;
    bool fixed = e0 > 64 && e0 < 0x7ff && e1 > 64 && e1 < 0x7ff;
    if (fixed) {
      int small0 = 0, small1 = 0;
      for (int i = threadIdx.x; i < N; i += blockDim.x) {  // every thread converts what it staged
        const double2 v = sd[i];
        const long long q0 = to_fixed(v.x, e0), q1 = to_fixed(v.y, e1);
        sx[i] = make_int4((int)(q0 & 0x7fffffff), (int)(q0 >> 31), (int)(q1 & 0x7fffffff), (int)(q1 >> 31));
        small0 += is_small(v.x, e0);
        small1 += is_small(v.y, e1);
      }
      small0 = block_add(small0, smi);
      small1 = block_add(small1, smi);
      fixed = small0 <= N / 16 && small1 <= N / 16;
      if (!fixed) stage(m0, m1);
    }
    __syncthreads();
    // 2^(emax - 1022 - kLineBits), the unit of the fixed-point numbers
    const double unit0 = fixed ? __hiloint2double((e0 + 1 - kLineBits) << 20, 0) : 1.0;
    const double unit1 = fixed ? __hiloint2double((e1 + 1 - kLineBits) << 20, 0) : 1.0;
    if (threadIdx.x < C) st[threadIdx.x] = make_double2(lv.mag[threadIdx.x] * unit0, lv.mag[threadIdx.x] * unit1);
    uint32_t bl0 = 0u, bl1 = 0u;
    double el0 = 0.0, el1 = 0.0;
    if (!COLS) {
      bl0 = sv.B_up[l0] & hp.umask;
      el0 = sv.e_up[l0];
      bl1 = two ? sv.B_up[l0 + 1] & hp.umask : 0u;
      el1 = two ? sv.e_up[l0 + 1] : 0.0;
      // the lines' part of a uniform diagonal by the number of doubly occupied sites
      for (int i = threadIdx.x; i <= kMaxOrb; i += blockDim.x)
        sUn[i] = make_double2(fma(hp.u0, (double)i, el0), fma(hp.u0, (double)i, el1));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
      double y0 = 0.0, y1 = 0.0;
      double* o = Ol + i * pstep;
      const double* xg = Xl + i * pstep;
      double2 w;  // what the hop sums are added to, requested before them
      if (pair) w = *reinterpret_cast<const double2*>(o);
      const uint32_t* p = lv.ell + i;
      const int n = lv.cnt[i];
      if (fixed) {
        // per magnitude: low limbs (31 bits) into 64 bits, high limbs (25 bits and sign) into 32, times the
        // sign or 0: multiply-adds of the FMA pipe, so that the ALU pipe is left with the decoding
        long long l0[C], l1[C];
        int h0[C], h1[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
          l0[c] = l1[c] = 0;
          h0[c] = h1[c] = 0;
        }
        uint32_t e[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) e[q] = __ldg(p + q * N);
        for (int k = 0; k < n; k += 4) {
          uint32_t f[4];
          p += 4 * N;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            f[q] = e[q];
            e[q] = __ldg(p + q * N);  // slots up to zmax + kLinePad - 1
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int4 x = *reinterpret_cast<const int4*>(ln_smem + (f[q] & ~15u));
            const int sg = 1 - 2 * (int)(f[q] & 1u);
            int sc[C];
            if constexpr (C == 1) {
              sc[0] = sg;
            } else if constexpr (C == 2) {
              sc[1] = sg & -(int)((f[q] >> 1) & 1u);
              sc[0] = sg - sc[1];
            } else {
#pragma unroll
              for (int c = 0; c < C; ++c) sc[c] = (f[q] & 6u) == 2u * c ? sg : 0;
            }
#pragma unroll
            for (int c = 0; c < C; ++c) {
              asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(l0[c]) : "r"(x.x), "r"(sc[c]));
              asm("mad.lo.s32 %0, %1, %2, %0;" : "+r"(h0[c]) : "r"(x.y), "r"(sc[c]));
              asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(l1[c]) : "r"(x.z), "r"(sc[c]));
              asm("mad.lo.s32 %0, %1, %2, %0;" : "+r"(h1[c]) : "r"(x.w), "r"(sc[c]));
            }
          }
        }
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const double2 t = st[c];
          y0 = fma(t.x, (double)(((long long)h0[c] << 31) + l0[c]), y0);
          y1 = fma(t.y, (double)(((long long)h1[c] << 31) + l1[c]), y1);
        }
      } else {
        for (int k = 0; k < n; ++k) {
          const uint32_t f = __ldg(p + k * N);
          const double2 x = *reinterpret_cast<const double2*>(ln_smem + (f & ~15u));
          const double v = flip_sign(st[(f >> 1) & 3u].x, f & 1u);
          y0 = fma(v, x.x, y0);
          y1 = fma(v, x.y, y1);
        }
      }
      if (!COLS) {
        const uint32_t bi = sv.B_dn[i];
        const double ei = sv.e_dn[i];
        const uint32_t d0 = bl0 & bi, d1 = bl1 & bi;
        double g0, g1;
        if (uni) {
          g0 = ei + sUn[__popc(d0)].x;
          g1 = ei + sUn[__popc(d1)].y;
        } else {
          g0 = hpsi_diag<double>(el0 + ei, d0, sU, false, 0.0);
          g1 = hpsi_diag<double>(el1 + ei, d1, sU, false, 0.0);
        }
        y0 = fma(g0, __ldg(xg), y0);
        const double* pv = Pl + i;
        if (beta) y0 = fma(-b, pv[0], y0);
        o[0] = y0;
        if (two) {
          y1 = fma(g1, __ldg(xg + lstep), y1);
          if (beta) y1 = fma(-b, pv[lstep], y1);
          o[lstep] = y1;
        }
      } else if (pair) {
        w.x += y0;
        w.y += y1;
        *reinterpret_cast<double2*>(o) = w;
        if (FUSED) {
          const double2 x = __ldg(reinterpret_cast<const double2*>(xg));
          sxw = fma(x.x, w.x, fma(x.y, w.y, sxw));
          sww = fma(w.x, w.x, fma(w.y, w.y, sww));
          sxx = fma(x.x, x.x, fma(x.y, x.y, sxx));
        }
      } else {
        y0 += o[0];
        o[0] = y0;
        if (two) {
          y1 += o[1];
          o[1] = y1;
        }
        if (FUSED) {
          const double x0 = __ldg(xg), x1 = two ? __ldg(xg + 1) : 0.0;
          if (!two) y1 = 0.0;
          sxw = fma(x0, y0, fma(x1, y1, sxw));
          sww = fma(y0, y0, fma(y1, y1, sww));
          sxx = fma(x0, x0, fma(x1, x1, sxx));
        }
      }
    }
  }
  if (!FUSED) return;
  block_sum3_any(sxw, sww, sxx);
  double* part = ls.partial + ((int64_t)run * gridDim.x) * 3;
  if (threadIdx.x == 0) {
    part[blockIdx.x * 3 + 0] = sxw;
    part[blockIdx.x * 3 + 1] = sww;
    part[blockIdx.x * 3 + 2] = sxx;
    __threadfence();
    s_last = atomicAdd(ls.counter + run, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double a = 0.0, bb = 0.0, c = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) {
    a += __ldcg(part + i * 3 + 0);
    bb += __ldcg(part + i * 3 + 1);
    c += __ldcg(part + i * 3 + 2);
  }
  block_sum3_any(a, bb, c);
  if (threadIdx.x == 0) {
    const double alpha = c > 0.0 ? a / c : 0.0;
    const double b2 = c > 0.0 ? bb - a * a / c : 0.0;
    const double bnext = b2 > 0.0 ? sqrt(b2) : 0.0;
    ls.alpha[(int64_t)run * ls.mstride + n_step] = alpha;
    ls.beta[(int64_t)run * (ls.mstride + 1) + n_step + 1] = bnext;
    if (ls.nsteps) ls.nsteps[run] = n_step + 1;
    if (!(bnext > ls.btol * ls.beta0[run]) || n_step + 1 >= ls.mstride) ls.active[run] = 0;
    ls.counter[run] = 0u;
  }
}

static size_t lines_smem(int64_t n) { return (size_t)(n + 1) * 16; }  // a line pair and a group of zeros

static int lines_threads(int64_t n) { return n >= 4096 ? 1024 : n >= 1024 ? 512 : 256; }

static unsigned lines_grid(int64_t n, int64_t lines) {
  const int threads = lines_threads(n);
  const int per_sm = (int)std::max<int64_t>(1, std::min<int64_t>(1024 / threads, (220 * 1024) / (int64_t)(lines_smem(n) + 2048)));
  return (unsigned)std::min<int64_t>((lines + 1) / 2, 152 * per_sm);
}

int lines64_blocks(const SectorView& sv) { return (int)lines_grid(sv.d_up, sv.d_dn); }

// Whether FP64 products of this sector take the integer sums.  They cost a conversion and a multiply-add
// per magnitude in each pass, and the columns a second pass over the vector: worth it from 2 x magnitudes + 4
// hops per spin on, for vectors of at least kLinesMinDim elements (below, the second launch and the staging
// of short lines eat the gain: 2x6 ladder, 853,776 states, 57 us against 68 us in tiles with FP64 sums; 12-site
// chain 40 and 41 us; 2x5 ladder, 63,504 states, 23 and 19 us).  The tables are built on the first call that wants them, not
// during a stream capture.
constexpr int64_t kLinesMinDim = int64_t(1) << 19;
static std::mutex g_lines_mu;

bool lines64_usable(const SectorView& sv, cudaStream_t s) {
  if (!sv.tab_up || sv.d_up * sv.d_dn < kLinesMinDim) return false;
  if (std::max(lines_smem(sv.d_up), lines_smem(sv.d_dn)) > (size_t)216 * 1024) return false;
  const ModelHost& m = *sv.model;
  if (m.vals.size() > 2 * kLineMaxClasses) return false;
  std::lock_guard<std::mutex> lk(g_lines_mu);
  for (SpinTables* t : {sv.tab_up, sv.tab_dn}) {
    if (t->lines) continue;
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    ED_CUDA(cudaStreamIsCapturing(s, &st));
    if (st != cudaStreamCaptureStatusNone) return false;
    t->lines = std::shared_ptr<LineTables>(build_lines(*t, m, sv.tab_stream));
  }
  for (SpinTables* t : {sv.tab_up, sv.tab_dn})
    if (t->lines->classes == 0 || t->lines->hops < 2.0 * t->lines->classes + 4.0) return false;
  return true;
}

static LineView line_view(const LineTables& t) {
  LineView v = {};
  for (int c = 0; c < t.classes; ++c) v.mag[c] = t.mag[c];
  v.ell = t.ell.p;
  v.cnt = t.cnt.p;
  return v;
}

// y_r = H x_r (ls == nullptr) or the fused Lanczos step, as launch_two_pass of hpsi.cu.
void launch_lines64(const SectorView& sv, const HopParams& hp, const double* X, double* O, int64_t vstride, int runs,
                    const double* beta, int beta_stride, int n, const LanczosScalars* ls, cudaStream_t s) {
  const int cu = sv.tab_up->lines->classes, cd = sv.tab_dn->lines->classes;
  const int* active = ls ? ls->active : nullptr;
  // one timed unit per step: both passes (the second launch is counted separately)
  ProfScope ps_(ls ? K_LANCZOS_STEP : K_HPSI, s, (beta ? 3.0 : 2.0) * 8.0 * (double)(sv.d_up * sv.d_dn) * runs);
  auto with = [](int c, auto&& f) {
    if (c == 1) f(std::integral_constant<int, 1>());
    else if (c == 2) f(std::integral_constant<int, 2>());
    else if (c == 3) f(std::integral_constant<int, 3>());
    else f(std::integral_constant<int, 4>());
  };
  with(cd, [&](auto c) {
    constexpr int C = decltype(c)::value;
    allow_max_dynamic_smem(k_lines64<false, false, C>);
    k_lines64<false, false, C><<<dim3(lines_grid(sv.d_dn, sv.d_up), runs), lines_threads(sv.d_dn), lines_smem(sv.d_dn), s>>>(
        sv, hp, line_view(*sv.tab_dn->lines), X, O, ls ? (const double*)ls->prev : nullptr, vstride, beta, beta_stride, n, active, LanczosScalars{});
  });
  ED_CHECK_LAUNCH();
  note_launch();
  const dim3 g(lines_grid(sv.d_up, sv.d_dn), runs);
  const int threads = lines_threads(sv.d_up);
  with(cu, [&](auto c) {
    constexpr int C = decltype(c)::value;
    const LineView up = line_view(*sv.tab_up->lines);
    if (ls) {
      allow_max_dynamic_smem(k_lines64<true, true, C>);
      k_lines64<true, true, C><<<g, threads, lines_smem(sv.d_up), s>>>(sv, hp, up, X, O, nullptr, vstride, nullptr, 0, n, active, *ls);
    } else {
      allow_max_dynamic_smem(k_lines64<true, false, C>);
      k_lines64<true, false, C><<<g, threads, lines_smem(sv.d_up), s>>>(sv, hp, up, X, O, nullptr, vstride, nullptr, 0, n, nullptr,
                                                                         LanczosScalars{});
    }
  });
  ED_CHECK_LAUNCH();
}

}  // namespace ed
