// Device building blocks of the matrix-free operators: launch shapes, shared-memory sum
// factorisation passes and the neo-Hookean point code.
//
// Sum factorisation (Section 2.4): values of a Q_p field at the (p+1)^3 Gauss points of an
// element are three 1D passes with B[q][i] = l_i(x_q), one per direction; reference-cell
// gradients at the points are then one collocation pass Dc per direction.  The transposed
// contraction with the test-function gradients is one combined Dc^T pass followed by three
// B^T passes.  Every pass maps an [n][n][n] block (x fastest) to another, with n = p + 1.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "df64.cuh"
#include "internal.h"
#include "pdl.cuh"

namespace nhmf {

// Elements per thread block and threads per block for each degree and precision.  Chosen so
// that NE * (p+1)^3 work items fill whole warps and the shared-memory footprint allows
// several blocks per SM.
template <int P, typename T> struct Cfg;
template <> struct Cfg<1, double> { static constexpr int NE = 32, THREADS = 256; };
#ifndef NHMF_Q2D_NE
#define NHMF_Q2D_NE 27
#define NHMF_Q2D_THREADS 256
#endif
#ifndef NHMF_Q4D_NE
#define NHMF_Q4D_NE 3
#define NHMF_Q4D_THREADS 192
#endif
template <> struct Cfg<2, double> { static constexpr int NE = NHMF_Q2D_NE, THREADS = NHMF_Q2D_THREADS; };
template <> struct Cfg<3, double> { static constexpr int NE = 8, THREADS = 256; };
template <> struct Cfg<4, double> { static constexpr int NE = NHMF_Q4D_NE, THREADS = NHMF_Q4D_THREADS; };
template <int P> struct Cfg<P, df64> : Cfg<P, double> {};
template <> struct Cfg<4, df64> { static constexpr int NE = 4, THREADS = 256; };
// Launch shape per strategy: Algorithm 2's point code (120 registers) keeps 256 threads at Q4
// so that two blocks fit an SM.
template <int P, typename T, int STRAT> struct LaunchCfg : Cfg<P, T> {};
template <> struct LaunchCfg<4, double, NHMF_SPATIAL> { static constexpr int NE = 4, THREADS = 256; };
#ifndef NHMF_Q2D_OTF_NE
#define NHMF_Q2D_OTF_NE NHMF_Q2D_NE
#define NHMF_Q2D_OTF_THREADS NHMF_Q2D_THREADS
#endif
template <> struct LaunchCfg<2, double, NHMF_ON_THE_FLY> {
  static constexpr int NE = NHMF_Q2D_OTF_NE, THREADS = NHMF_Q2D_OTF_THREADS;
};

// Block shapes: the launch shape above, and for the FP64 and double-float kernels (issue bound
// within an SM) small blocks of one to four elements for meshes whose normal blocks would not give
// every SM `per_sm` of them: a block of 27 Q2 elements keeps one SM's FP64 pipe busy for 34 us
// while the others idle.  The line, small / normal blocks in us just below it and just above (Q1
// 24^3, 34^3; Q2 20^3, 28^3; Q3 14^3, 18^3; Q4 10^3, 14^3):
//   cached       43/44 88/93    81/107 206/203   78/100 148/177   70/96 167/187
//   on the fly   58/60 138/146  125/140 319/316  114/142 229/238  100/131 247/281
//   Algorithm 2  53/54 129/134  112/124 287/298  100/119 195/219  93/107 207/215
//   residual     63/69 112/114  102/126 225/213  99/127 172/176   90/114 186/191
//   point cache  50/51 87/88    88/79 176/167    77/89 124/126    72/80 131/145
// and far below it Q2 8^3 takes 0.35 to 0.66 of the normal blocks' time.  The diagonal, whose normal
// blocks hold half the elements, has its line there too (Q2 16^3 54/77, 20^3 87/90; Q3 8^3 0.97) and
// loses up to 17 % to it at Q1 and Q3 (24^3 44/38, 14^3 87/78).  Double-float blocks take less time
// each: Q2 16^3 44/69, 20^3 56/75, 28^3 122/112; Q3 14^3 48/58, 18^3 88/74; Q4 12^3 66/72, 14^3 94/86;
// at Q1 the normal blocks are 5 to 20 % faster at every size.
template <typename T> struct SmallRule { static constexpr int per_sm = 4; };
template <> struct SmallRule<df64> { static constexpr int per_sm = 2; };
template <int P> struct SmallCfg;
template <> struct SmallCfg<1> { static constexpr int NE = 4, THREADS = 32; };
template <> struct SmallCfg<2> { static constexpr int NE = 3, THREADS = 96; };
template <> struct SmallCfg<3> { static constexpr int NE = 1, THREADS = 64; };
template <> struct SmallCfg<4> { static constexpr int NE = 1, THREADS = 128; };
template <int P, typename T, int STRAT, bool SMALL> struct Shape : LaunchCfg<P, T, STRAT> {};
template <int P, typename T, int STRAT> struct Shape<P, T, STRAT, true> : SmallCfg<P> {};

// Coefficients of one n x n operator in even-odd form (odd n <= 5): S, A ((h+1) x h each) and C
// (h+1), h = n / 2.
constexpr int kEoSlots = 16;

// One n x n line operator of the FP32 column kernel in even-odd form, M[n-1-r][n-1-m] = +-M[r][m], h =
// n / 2: S = (M_rm + M_r,n-1-m) / 2 and A = (M_rm - M_r,n-1-m) / 2 for r, m < h, C = M_rh, and the
// centre row of odd n: mid_m = M_hm (its even or odd half) and ch = M_hh.
struct EoTab {
  float S[2][2], A[2][2], C[2], mid[2], ch;
};

// Kernel arguments (by value; lives in the constant bank).
struct OpArgs {
  int N, M, bc, model;
  long long M3, nq;
  double h, mu, lam;
  Colour col;
  double B[kMaxN * kMaxN], Dc[kMaxN * kMaxN], D[kMaxN * kMaxN], w[kMaxN];
  // Tables of the tangent apply, which carry the quadrature weight, mu and h so that its
  // point code returns dP / mu unweighted:
  //   BW[q][i] = B[q][i] w_q,  DcW[m][r] = Dc[m][r] w_m / w_r mu h,  Dch = Dc / h,
  //   eo[0..2], eoh: even-odd coefficients of B, Dc, BW^T and Dch (odd n, see eo_line),
  //   r2mu = 2 lambda / mu.
  double BW[kMaxN * kMaxN], DcW[kMaxN * kMaxN], Dch[kMaxN * kMaxN];
  double eo[3][kEoSlots];
  double eoh[kEoSlots];  // of Dch
  double r2mu;
  int reg32;  // FP32 point cache in the register kernel's tiles [E/32][10][n^3][32] (see kRegMaxP)
  float BWf[kMaxN * kMaxN], DcWf[kMaxN * kMaxN], Dchf[kMaxN * kMaxN], eof[3][kEoSlots];  // FP32 copies
  float Bf[kMaxN * kMaxN], Dcf[kMaxN * kMaxN];  // FP32 copies (register kernels)
  EoTab cB, cD, cBT, cDT, cBTz, cDTz;  // B, D and the weighted transposes; z: times mu h
  float invhf, r2muf;                  // 1 / h, r2mu
  const double* u64;
  const float* u32;
  const void* du;
  void* v;
  const void* cache;
  double* cache64_out;
  float* cache32_out;
  float2* cachedf_out;
  double* cachesp_out;
  const double* cachesp_in;
  const double* factor;  // per-element material factor (natural element order) or null
  unsigned* status;
  float* vloc;           // element-local FP32 results [3][n^3][E] (element-local apply) or null
};

// ------------------------------------------------------------------ memory helpers (PTX)
// L2 eviction-priority policies (createpolicy) and loads/stores that carry them: the applies
// stream their point caches with evict_first, so that the vectors they reuse stay in L2 (the
// FP64 colour launches re-read du and v eight times), and the FP32 apply writes its
// element-local results with evict_last, so that they are still in L2 when the gather reads them.
#ifndef NHMF_L2HINT
#define NHMF_L2HINT 1
#endif
__device__ __forceinline__ unsigned long long l2_evict_first() {
  unsigned long long p;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ unsigned long long l2_evict_last() {
  unsigned long long p;
  asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ float ld_policy(const float* a, unsigned long long pol) {
#if NHMF_L2HINT
  float v;
  asm("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(a), "l"(pol));
  return v;
#else
  return __ldg(a);
#endif
}
// The same, kept in program order (a prefetch that must not sink to its use).
__device__ __forceinline__ float ld_policy_ordered(const float* a, unsigned long long pol) {
  float v;
  asm volatile("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(a), "l"(pol));
  return v;
}
// A value that the launch before this one writes, for after pdl_wait(): that launch may still run when
// this grid starts, so the load must not be .nc (data constant while the grid lives), and the
// compiler has to keep it behind the wait.
__device__ __forceinline__ float ld_produced(const float* a, unsigned long long pol) {
  float v;
#if NHMF_L2HINT
  asm volatile("ld.global.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(a), "l"(pol) : "memory");
#else
  v = *static_cast<const volatile float*>(a);
#endif
  return v;
}
__device__ __forceinline__ double ld_policy(const double* a, unsigned long long pol) {
#if NHMF_L2HINT
  double v;
  asm("ld.global.nc.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(a), "l"(pol));
  return v;
#else
  return __ldg(a);
#endif
}
__device__ __forceinline__ void st_policy(float* a, float v, unsigned long long pol) {
#if NHMF_L2HINT
  asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(a), "f"(v), "l"(pol) : "memory");
#else
  *a = v;
#endif
}
__device__ __forceinline__ bool is_constrained(int bc, int c, int gi, int gk, int M) {
  if (bc == NHMF_BC_CLAMP_X0) return gi == 0;
  if (bc == NHMF_BC_COMPRESSION) return gk == 0 || (c == 2 && gk == M - 1);
  return false;
}

// A block's colour class and first element in it, for a launch whose blocks (NE elements each) cover all
// eight classes.  The classes are laid out as build_geometry (api.cu) does: class cx + 2 cy + 4 cz
// holds the elements of these parities, slots in class order.
template <int NE>
__device__ __forceinline__ Colour block_colour(int N, long long& e0) {
  Colour c;
  c.stride = 2;
  c.slot0 = 0;
  long long first = 0;
  for (int k = 0;; ++k) {
    c.cx = k & 1, c.cy = (k >> 1) & 1, c.cz = k >> 2;
    c.nx = (N + 1 - c.cx) / 2, c.ny = (N + 1 - c.cy) / 2, c.nz = (N + 1 - c.cz) / 2;
    c.count = c.nx * c.ny * c.nz;
    const long long blocks = (c.count + NE - 1) / NE;
    if (k == 7 || blockIdx.x < first + blocks) break;
    first += blocks;
    c.slot0 += c.count;
  }
  e0 = ((long long)blockIdx.x - first) * NE;
  return c;
}

// Global node of work item t (element t / n^3 of this block, local point/node t % n^3).
template <int P>
__device__ __forceinline__ void item_node(const Colour& c, long long e_in_colour, int q, int& gi, int& gj, int& gk) {
  constexpr int n = P + 1;
  const int ix = int(e_in_colour % c.nx);
  const int iy = int((e_in_colour / c.nx) % c.ny);
  const int iz = int(e_in_colour / ((long long)c.nx * c.ny));
  gi = P * (c.cx + c.stride * ix) + q % n;
  gj = P * (c.cy + c.stride * iy) + (q / n) % n;
  gk = P * (c.cz + c.stride * iz) + q / (n * n);
}

// Natural index ex + N (ey + N ez) of element e_in_colour of the class.
__device__ __forceinline__ long long elem_natural(const OpArgs& a, const Colour& c, long long e_in_colour) {
  const long long ix = e_in_colour % c.nx, iy = (e_in_colour / c.nx) % c.ny, iz = e_in_colour / ((long long)c.nx * c.ny);
  const long long ex = c.cx + c.stride * ix, ey = c.cy + c.stride * iy, ez = c.cz + c.stride * iz;
  return ex + (long long)a.N * (ey + (long long)a.N * ez);
}

// Material factor of element e_in_colour of the class (1 if homogeneous).
__device__ __forceinline__ double elem_factor(const OpArgs& a, const Colour& c, long long e_in_colour) {
  return a.factor ? a.factor[elem_natural(a, c, e_in_colour)] : 1.0;
}

// One 1D pass along direction DIR over NC arrays of NI items:
//   out[c][t] = sum_m Mat(r, m) in[c][t with coordinate r along DIR replaced by m]
// with Mat(r, m) = mat[r][m] (TR = false) or mat[m][r] (TR = true).
// Items t >= nitems (those of absent elements, which come last) are skipped.
template <int n, int NI, int NC, int DIR, bool TR, typename T>
__device__ __forceinline__ void sf_pass(const T* __restrict__ mat, const T* in, T* out, int nitems = NI) {
  constexpr int s = DIR == 0 ? 1 : (DIR == 1 ? n : n * n);
  for (int t = threadIdx.x; t < nitems; t += blockDim.x) {
    const int r = (t / s) % n;
    const int base = t - r * s;
    Acc<T> acc[NC];
    {
      const T c0 = TR ? mat[r] : mat[r * n];
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c].mul(c0, in[c * NI + base]);
    }
#pragma unroll
    for (int m = 1; m < n; ++m) {
      const T cm = TR ? mat[m * n + r] : mat[r * n + m];
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c].fma(cm, in[c * NI + base + m * s]);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) out[c * NI + t] = acc[c].get();
  }
}

// One line x[0..n-1] through a centro-symmetric operator (ANTI = false: M[n-1-r][n-1-m] =
// M[r][m], as B and B^T w have) or an anti-centro-symmetric one (ANTI = true: = -M[r][m], as the
// collocation derivative has), odd n, in even-odd form (h = n / 2, m < h, r < h):
//   e_m = x_m + x_{n-1-m},  o_m = x_m - x_{n-1-m},
//   E_r = C_r x_h + sum_m S_rm e_m,  O_r = sum_m A_rm o_m,
//   y_r = E_r + O_r,  y_{n-1-r} = +-(E_r - O_r),  y_h = E_h (symmetric) or O_h (anti),
// with S_rm = (M_rm + M_r,n-1-m) / 2, A_rm = (M_rm - M_r,n-1-m) / 2, C_r = M_rh.  n = 3 takes 8
// (symmetric) or 7 (anti) operations per line instead of 9; n = 5 takes 21 or 20 instead of 25.
// FORM uses that the middle Gauss point is the middle GLL node (x = 1/2) for odd n:
//   kEoCentreRow:  the centre row of M is e_h (M = B): y_h = x_h, 2 (n = 3) or 3 (n = 5) fewer;
//   kEoCentreCol:  the centre column of M vanishes off the centre (M = B^T w): C_r = 0 for r < h.
enum { kEoGeneral = 0, kEoCentreRow = 1, kEoCentreCol = 2 };
template <int n, bool ANTI, int FORM, typename T>
__device__ __forceinline__ void eo_line(const T (&k)[kEoSlots], const T (&x)[n], T (&y)[n]) {
  constexpr int h = n / 2, A0 = (h + 1) * h, C0 = 2 * (h + 1) * h;
  T e[h], o[h];
#pragma unroll
  for (int m = 0; m < h; ++m) {
    e[m] = x[m] + x[n - 1 - m];
    o[m] = x[m] - x[n - 1 - m];
  }
#pragma unroll
  for (int r = 0; r < h; ++r) {
    Acc<T> E;
    if constexpr (FORM == kEoCentreCol) {
      E.mul(k[r * h], e[0]);
#pragma unroll
      for (int m = 1; m < h; ++m) E.fma(k[r * h + m], e[m]);
    } else {
      E.mul(k[C0 + r], x[h]);
#pragma unroll
      for (int m = 0; m < h; ++m) E.fma(k[r * h + m], e[m]);
    }
    Acc<T> yp = E, ym = E;
    if (ANTI) ym.neg();
#pragma unroll
    for (int m = 0; m < h; ++m) {
      yp.fma(k[A0 + r * h + m], o[m]);
      ym.fma(ANTI ? k[A0 + r * h + m] : -k[A0 + r * h + m], o[m]);
    }
    y[r] = yp.get();
    y[n - 1 - r] = ym.get();
  }
  if constexpr (ANTI) {
    Acc<T> c;
    c.mul(k[A0 + h * h], o[0]);
#pragma unroll
    for (int m = 1; m < h; ++m) c.fma(k[A0 + h * h + m], o[m]);
    y[h] = c.get();
  } else if constexpr (FORM == kEoCentreRow) {
    y[h] = x[h];
  } else {
    Acc<T> c;
    c.mul(k[C0 + h], x[h]);
#pragma unroll
    for (int m = 0; m < h; ++m) c.fma(k[h * h + m], e[m]);
    y[h] = c.get();
  }
}

// One 1D pass along DIR over NC fields with one thread per (field, line of n items), odd n:
//   out[(c OS + OO)][line] = M in[c][line]
// where M is given by its even-odd coefficients `coef` (see eo_line).
// TH is the block size; the task loop is unrolled so that independent lines interleave (not for
// double-float, whose unrolled lines would cost an SM its second block).
// Lines of absent elements (line index >= nlines; they come last) are skipped.
template <int n, int NI, int NC, int DIR, bool ANTI, int FORM, int TH, int OS = 1, int OO = 0, typename T>
__device__ __forceinline__ void eo_pass(const T* __restrict__ coef, const T* __restrict__ in,
                                        T* __restrict__ out, int nlines = NI / n) {
  constexpr int s = DIR == 0 ? 1 : (DIR == 1 ? n : n * n), NL = NI / n, ITER = (NC * NL + TH - 1) / TH;
  constexpr int UNROLL = std::is_same<T, df64>::value ? 1 : ITER;
  T k[kEoSlots];
#pragma unroll
  for (int i = 0; i < kEoSlots; ++i) k[i] = coef[i];
#pragma unroll UNROLL
  for (int it = 0; it < ITER; ++it) {
    const int task = threadIdx.x + it * TH;
    if (ITER * TH != NC * NL && task >= NC * NL) break;
    const int c = task / NL, L = task - c * NL;
    const int base = DIR == 0 ? L * n
                              : (DIR == 1 ? (L % n) + (L / n) * n * n : (L % (n * n)) + (L / (n * n)) * n * n * n);
    if (L >= nlines) continue;
    T x[n], y[n];
#pragma unroll
    for (int m = 0; m < n; ++m) x[m] = in[c * NI + base + m * s];
    eo_line<n, ANTI, FORM>(k, x, y);
#pragma unroll
    for (int m = 0; m < n; ++m) out[(c * OS + OO) * NI + base + m * s] = y[m];
  }
}

// Reference-cell gradient of NC fields at item t from their point values (collocation).
//   g[c][d] = sum_m Dc[r_d][m] val[c][t with coordinate d replaced by m]
template <int n, int NI, typename T>
__device__ __forceinline__ void colloc_grad(const T* __restrict__ Dc, const T* val, int t, T g[9]) {
  const int rx = t % n, ry = (t / n) % n, rz = (t / (n * n)) % n;
  const int bx = t - rx, by = t - ry * n, bz = t - rz * n * n;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const T* vc = val + c * NI;
    Acc<T> gx, gy, gz;
    gx.mul(Dc[rx * n], vc[bx]);
    gy.mul(Dc[ry * n], vc[by]);
    gz.mul(Dc[rz * n], vc[bz]);
#pragma unroll
    for (int m = 1; m < n; ++m) {
      gx.fma(Dc[rx * n + m], vc[bx + m]);
      gy.fma(Dc[ry * n + m], vc[by + m * n]);
      gz.fma(Dc[rz * n + m], vc[bz + m * n * n]);
    }
    g[c * 3 + 0] = gx.get();
    g[c * 3 + 1] = gy.get();
    g[c * 3 + 2] = gz.get();
  }
}

// Combined transposed collocation pass: y[c][t] = sum_d sum_m Dc[m][r_d] G[3c+d][t_d(m)].
template <int n, int NI, typename T>
__device__ __forceinline__ void colloc_grad_T(const T* __restrict__ Dc, const T* G, T* y, int nitems = NI) {
  for (int t = threadIdx.x; t < nitems; t += blockDim.x) {
    const int rx = t % n, ry = (t / n) % n, rz = (t / (n * n)) % n;
    const int bx = t - rx, by = t - ry * n, bz = t - rz * n * n;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const T* gx = G + (3 * c + 0) * NI;
      const T* gy = G + (3 * c + 1) * NI;
      const T* gz = G + (3 * c + 2) * NI;
      Acc<T> acc;
      acc.mul(Dc[rx], gx[bx]);
      acc.fma(Dc[ry], gy[by]);
      acc.fma(Dc[rz], gz[bz]);
#pragma unroll
      for (int m = 1; m < n; ++m) {
        acc.fma(Dc[m * n + rx], gx[bx + m]);
        acc.fma(Dc[m * n + ry], gy[by + m * n]);
        acc.fma(Dc[m * n + rz], gz[bz + m * n * n]);
      }
      y[c * NI + t] = acc.get();
    }
  }
}

// ------------------------------------------------------------------ point code
// The FP64 pipe (2 DFMA per clock and SM) bounds every FP64 kernel, so its point code counts FP64
// instructions.  CUDA's 1 / x and log1p took about 70 of them at a point; the two below take 16.

// 1 / x by Newton's iteration, third order: y0 = rcp.approx(x) (relative error below 2^-20), e = 1 -
// x y0, y = y0 (1 + e + e^2) with error e^3 < 2^-60 before rounding.  x and its reciprocal are
// normal numbers.
__device__ __forceinline__ double fast_rcp(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// log1p(x) given J = 1 + x, table driven (P. T. P. Tang, "Table-driven implementation of the
// logarithm function in IEEE floating-point arithmetic", ACM TOMS 16, 1990): J = 2^k m with m in
// [0.75, 1.5), c from the table near 1 / m, r = c 2^-k (1 + x) - 1 from x itself (one rounding, so
// small x keep their relative accuracy; c = 1 next to J = 1), |r| <= 2^-7, and log1p(x) = k ln 2 -
// ln c + log1p(r) with the series to r^8 (next term below 2^-66).  J in [2^-1000, 2^1000].
#include "log_table.h"
__device__ __forceinline__ double fast_log1p(double x, double J) {
  const int t = __double2hiint(J) - 0x3fe80000, k = t >> 20, i = (t >> 13) & 127;  // m >= 0.75: exponent field of 0.75
  double c = __ldg(&kLogTable[i][0]), l = __ldg(&kLogTable[i][1]);
  if (k != 0) {
    c *= __hiloint2double((1023 - k) << 20, 0);
    l = fma((double)k, 0.69314718055994530942, l);
  }
  const double r = fma(c, x, c - 1.0);
  double p = fma(r, -1.0 / 8.0, 1.0 / 7.0);
  p = fma(r, p, -1.0 / 6.0);
  p = fma(r, p, 1.0 / 5.0);
  p = fma(r, p, -1.0 / 4.0);
  p = fma(r, p, 1.0 / 3.0);
  p = fma(r, p, -1.0 / 2.0);
  return l + fma(r * r, p, r);
}

// J in [2^-500, 2^500): positive, and 1 / J^2 is a normal number too.
__device__ __forceinline__ bool ordinary(double J) { return (unsigned)(__double2hiint(J) - (523 << 20)) < 1000u << 20; }

// Kinematics at a point from the physical displacement gradient H (row-major H[3c+d]), F = I + H:
// the adjugate A = J F^-1, 1 / J, ln J and J - 1.  With C00 - 1 = H4 + H8 + H4 H8 - H5 H7,
//   J - 1 = H0 + F0 (C00 - 1) + H1 C01 + H2 C02
// has no cancellation near F = I (25 operations for A and J - 1).  F^-1 = A invJ always.  In FP64, where
// J is not ordinary (not positive, not finite, or so large that the point code's 1 / J^2 would
// underflow while F^-1 is still an ordinary number), A is F^-1 itself and invJ is 1.
template <typename T>
struct Kinematics {
  T A[9], invJ, lnJ, Jm1;
  __device__ __forceinline__ Kinematics() {}
  __device__ __forceinline__ explicit Kinematics(const T H[9]) {
    const T F0 = T(1) + H[0], F4 = T(1) + H[4], F8 = T(1) + H[8];
    const T C = fma(-H[5], H[7], fma(H[4], F8, H[8]));  // C00 - 1
    A[0] = T(1) + C;
    A[1] = fma(H[2], H[7], -(H[1] * F8));
    A[2] = fma(H[1], H[5], -(H[2] * F4));
    A[3] = fma(H[5], H[6], -(H[3] * F8));
    A[4] = fma(F0, F8, -(H[2] * H[6]));
    A[5] = fma(H[2], H[3], -(F0 * H[5]));
    A[6] = fma(H[3], H[7], -(F4 * H[6]));
    A[7] = fma(H[1], H[6], -(F0 * H[7]));
    A[8] = fma(F0, F4, -(H[1] * H[3]));
    Jm1 = fma(F0, C, fma(H[1], A[3], fma(H[2], A[6], H[0])));
    const T J = T(1) + Jm1;
    if constexpr (sizeof(T) == 8) {
      if (ordinary(J)) {
        invJ = fast_rcp(J);
        lnJ = fast_log1p(Jm1, J);
      } else {
        const T inv = 1.0 / J;
#pragma unroll
        for (int k = 0; k < 9; ++k) A[k] *= inv;
        invJ = 1.0;
        lnJ = log1p(Jm1);
      }
    } else {
      invJ = T(1) / J;
      lnJ = log1pf(Jm1);
    }
  }
};

// The same as F^-1 = A / J and ln J; returns J - 1.
template <typename T>
__device__ __forceinline__ T kinematics(const T H[9], T Fi[9], T& lnJ) {
  const Kinematics<T> k(H);
#pragma unroll
  for (int i = 0; i < 9; ++i) Fi[i] = k.A[i] * k.invJ;
  lnJ = k.lnJ;
  return k.Jm1;
}

// Linearised first Piola stress at a point, scaled by s (Eq. LG: G = L : Grad du):
//   dP = mu dH + (mu - 2 lambda ln J) F^-T dH^T F^-T + 2 lambda tr(F^-1 dH) F^-T
// with K = F^-1 dH and Q = K F^-1 (so F^-T dH^T F^-T = Q^T).  Written into g[3i+J].
template <typename T>
__device__ __forceinline__ void linearised_stress(const T Fi[9], T lnJ, const T dH[9], T mu,
                                                  T lam, T s, T g[9]) {
  T K[9];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      K[3 * i + j] = fma(Fi[3 * i + 0], dH[j], fma(Fi[3 * i + 1], dH[3 + j], Fi[3 * i + 2] * dH[6 + j]));
  const T trK = K[0] + K[4] + K[8];
  const T smu = s * mu;
  const T sc1 = s * (mu - T(2) * lam * lnJ);
  const T sc2 = s * (T(2) * lam * trK);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      // Q[j][i] = sum_c K[j][c] Fi[c][i]
      const T Qji = fma(K[3 * j + 0], Fi[i], fma(K[3 * j + 1], Fi[3 + i], K[3 * j + 2] * Fi[6 + i]));
      g[3 * i + j] = fma(smu, dH[3 * i + j], fma(sc1, Qji, sc2 * Fi[3 * j + i]));
    }
}

// The same linearised stress divided by mu and without the point weight (the tangent apply
// carries w_q, mu and h on its transposed tables), r = 2 lambda / mu:
//   g = dH + (1 - r ln J) (K F^-1)^T + r tr(K) F^-T = dH + ((c1 K + c2 I) F^-1)^T:
// 67 operations instead of 76 with the two terms added separately.
template <typename T>
__device__ __forceinline__ void linearised_stress_unit(const T Fi[9], T c1, T rs, const T dH[9], T g[9]) {
  T K[9];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      Acc<T> k;
      k.mul(Fi[3 * i + 2], dH[6 + j]);
      k.fma(Fi[3 * i + 1], dH[3 + j]);
      k.fma(Fi[3 * i + 0], dH[j]);
      K[3 * i + j] = k.get();
    }
  const T c2 = rs * (K[0] + K[4] + K[8]);
#pragma unroll
  for (int k = 0; k < 9; ++k) K[k] = k % 4 == 0 ? fma(c1, K[k], c2) : c1 * K[k];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      Acc<T> q;
      q.set(dH[3 * i + j]);
      q.fma(K[3 * j + 2], Fi[6 + i]);
      q.fma(K[3 * j + 1], Fi[3 + i]);
      q.fma(K[3 * j + 0], Fi[i]);
      g[3 * i + j] = q.get();
    }
}
// The two terms added separately: nine more operations, but none waits for the trace before the second
// product starts.  The FP32 register kernel at two warps a scheduler is faster this way (Q2 64^3
// cached: 97 us against 109).
template <typename T>
__device__ __forceinline__ void linearised_stress_terms(const T Fi[9], T c1, T rs, const T dH[9], T g[9]) {
  T K[9];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      K[3 * i + j] = fma(Fi[3 * i + 0], dH[j], fma(Fi[3 * i + 1], dH[3 + j], Fi[3 * i + 2] * dH[6 + j]));
  const T c2 = rs * (K[0] + K[4] + K[8]);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const T Qji = fma(K[3 * j + 0], Fi[i], fma(K[3 * j + 1], Fi[3 + i], K[3 * j + 2] * Fi[6 + i]));
      g[3 * i + j] = fma(c1, Qji, fma(c2, Fi[3 * j + i], dH[3 * i + j]));
    }
}
// from F^-1 and ln J
template <typename T>
__device__ __forceinline__ void linearised_stress_unit(const T Fi[9], T lnJ, const T dH[9], T r, T g[9]) {
  linearised_stress_unit(Fi, fma(-r, lnJ, T(1)), r, dH, g);
}
// from the adjugate: F^-1 = A / J enters twice, so both coefficients carry 1 / J^2
template <typename T>
__device__ __forceinline__ void linearised_stress_unit(const Kinematics<T>& k, const T dH[9], T r, T g[9]) {
  const T s = k.invJ * k.invJ;
  linearised_stress_unit(k.A, fma(-r, k.lnJ, T(1)) * s, r * s, dH, g);
}

// Split neo-Hookean model (Eq. hypcomplex), with a = J^(-2/3), I1 = F : F:
//   P  = mu a (F - I1/3 F^-T) + kappa/2 (J^2 - 1) F^-T
//   dP = mu a dH - 2/3 mu a tr(F^-1 dH) F
//        + (2/9 mu a I1 tr(F^-1 dH) - 2/3 mu a F:dH + kappa J^2 tr(F^-1 dH)) F^-T
//        + (mu a I1/3 - kappa/2 (J^2 - 1)) F^-T dH^T F^-T
template <typename T>
__device__ __forceinline__ void split_stress_dP(const T F[9], const T Fi[9], T lnJ, T Jm1, const T dH[9], T mu,
                                                T kappa, T s, T g[9]) {
  const T a = exp(T(-2) / T(3) * lnJ);
  const T J = T(1) + Jm1;
  const T J2 = J * J;
  T I1 = T(0), FdH = T(0);
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    I1 = fma(F[k], F[k], I1);
    FdH = fma(F[k], dH[k], FdH);
  }
  T K[9];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      K[3 * i + j] = fma(Fi[3 * i + 0], dH[j], fma(Fi[3 * i + 1], dH[3 + j], Fi[3 * i + 2] * dH[6 + j]));
  const T trK = K[0] + K[4] + K[8];
  const T mua = mu * a;
  const T c1 = s * mua;
  const T cF = -s * T(2) / T(3) * mua * trK;
  const T c3 = s * (T(2) / T(9) * mua * I1 * trK - T(2) / T(3) * mua * FdH + kappa * J2 * trK);
  const T c4 = s * (mua * I1 / T(3) - kappa / T(2) * (J2 - T(1)));
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const T Qji = fma(K[3 * j + 0], Fi[i], fma(K[3 * j + 1], Fi[3 + i], K[3 * j + 2] * Fi[6 + i]));
      g[3 * i + j] = fma(c1, dH[3 * i + j], fma(cF, F[3 * i + j], fma(c3, Fi[3 * j + i], c4 * Qji)));
    }
}

// P of the selected model
template <typename T>
__device__ __forceinline__ void model_piola(int model, const T F[9], const T Fi[9], T lnJ, T Jm1, T mu, T lam, T P[9]) {
  if (model == NHMF_MODEL_SPLIT) {
    const T a = exp(T(-2) / T(3) * lnJ);
    const T J = T(1) + Jm1;
    T I1 = T(0);
#pragma unroll
    for (int k = 0; k < 9; ++k) I1 = fma(F[k], F[k], I1);
    const T cT = -mu * a * I1 / T(3) + lam / T(2) * (J * J - T(1));
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) P[3 * i + j] = fma(mu * a, F[3 * i + j], cT * Fi[3 * j + i]);
  } else {
    const T c2 = T(2) * lam * lnJ - mu;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) P[3 * i + j] = fma(mu, F[3 * i + j], c2 * Fi[3 * j + i]);
  }
}

// dP[dH] of the selected model, scaled by s (F = I + H needed by the split model only)
template <typename T>
__device__ __forceinline__ void model_dP(int model, const T F[9], const T Fi[9], T lnJ, T Jm1, const T dH[9], T mu,
                                         T lam, T s, T g[9]) {
  if (model == NHMF_MODEL_SPLIT)
    split_stress_dP(F, Fi, lnJ, Jm1, dH, mu, lam, s, g);
  else
    linearised_stress(Fi, lnJ, dH, mu, lam, s, g);
}

// Voigt index of the pair (i, j): 11, 22, 33, 23, 13, 12 -> 0..5.
__host__ __device__ constexpr int voigt(int i, int j) {
  return i == j ? i : (i + j == 3 ? 3 : (i + j == 2 ? 4 : 5));
}
// Index of (I, K), I <= K, in the row-major upper triangle of a 6x6 matrix.
__host__ __device__ constexpr int tri6(int I, int K) { return I * 6 - I * (I - 1) / 2 + (K - I); }

// Algorithm 2 point code (current configuration, Eq. DF:cur), scaled by s:
//   g = dH F^-1 (spatial gradient), e_hat = (g00, g11, g22, g12+g21, g02+g20, g01+g10),
//   sig_I = sum_K Jc[I][K] e_hat_K (J c : sym(g)), X = sig + g tau, G = s X F^-T.
template <typename T>
__device__ __forceinline__ void spatial_stress(const T Jc[21], const T tau[6], const T Fi[9], const T dH[9], T s,
                                               T out[9]) {
  T gs[9];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int l = 0; l < 3; ++l)
      gs[3 * k + l] = fma(dH[3 * k + 0], Fi[l], fma(dH[3 * k + 1], Fi[3 + l], dH[3 * k + 2] * Fi[6 + l]));
  const T eh[6] = {gs[0], gs[4], gs[8], gs[5] + gs[7], gs[2] + gs[6], gs[1] + gs[3]};
  T sv[6];
#pragma unroll
  for (int I = 0; I < 6; ++I) {
    T acc = T(0);
#pragma unroll
    for (int K = 0; K < 6; ++K) acc = fma(Jc[I <= K ? tri6(I, K) : tri6(K, I)], eh[K], acc);
    sv[I] = acc;
  }
  T X[9];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      X[3 * i + j] = fma(gs[3 * i + 0], tau[voigt(0, j)],
                         fma(gs[3 * i + 1], tau[voigt(1, j)], fma(gs[3 * i + 2], tau[voigt(2, j)], sv[voigt(i, j)])));
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int J = 0; J < 3; ++J)
      out[3 * i + J] = s * fma(X[3 * i + 0], Fi[3 * J + 0], fma(X[3 * i + 1], Fi[3 * J + 1], X[3 * i + 2] * Fi[3 * J + 2]));
}

}  // namespace nhmf
