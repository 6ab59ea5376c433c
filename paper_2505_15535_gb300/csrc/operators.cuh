// Matrix-free operators of compressible neo-Hookean elasticity on the GPU:
//   k_apply         FP64 and double-float tangent application, on the fly (Algorithm 1) or from the point cache
//   k_apply_reg     FP32 tangent application, one element per thread in registers (p <= 2)
//   k_apply_col     FP32 tangent application, one column of points per thread (p >= 2; apply32.cuh)
//   k_gather_local  FP32: sums the element-local results of the apply at the nodes
//   k_cache         point cache {F^-1, ln J} at the linearisation point (partial assembly, Section 3.2)
//   k_residual      residual R(u) (Eq. F)
//   k_diagonal      operator diagonal (Section 2.3)
// FP64 and double-float: each block processes NE elements of one colour class; elements of a
// class share no node, so the read-modify-write scatter of a launch is race-free and
// deterministic, and the eight classes run as eight launches in a fixed order, chained by
// programmatic dependent launch (see run_colours): a class computes while the classes before it
// still run and waits for them only before its scatter.  FP32: one
// launch over all elements writes element-local results, and the gather adds each node's
// contributions in a fixed order (also deterministic, no atomics).
#pragma once
#include <algorithm>
#include <type_traits>

#include "apply32.cuh"
#include "df64.cuh"
#include "sumfact.cuh"

namespace nhmf {
namespace {

// Table slots ahead of the per-item arrays, the most of any kernel: B, Dc, BW, DcW, Dch, 3 even-odd sets
// and NE factors in the apply, 7 tables, an even-odd set and NE factors in the diagonal.
constexpr int kTabSlots = 3 * kMaxN * kMaxN + 128 + 32;
static_assert(5 * kMaxN * kMaxN + 3 * kEoSlots + 32 <= kTabSlots, "apply tables exceed the table slots");

// The apply's tables: B and Dc (forward), BW and DcW (transposed, carrying w, mu, h), Dch and
// the even-odd coefficient sets, laid out as in k_apply.
// `deriv`: the even-odd set in the place of Dc's (the residual takes physical gradients), or null.
template <int P, typename T>
__device__ __forceinline__ void load_apply_tables(const OpArgs& a, T* tab, const double* deriv = nullptr) {
  constexpr int n = P + 1, S = kMaxN * kMaxN;
  for (int i = threadIdx.x; i < n * n; i += blockDim.x) {
    tab[i] = T(a.B[i]);
    tab[S + i] = T(a.Dc[i]);
    tab[2 * S + i] = T(a.BW[i]);
    tab[3 * S + i] = T(a.DcW[i]);
    tab[4 * S + i] = T(a.Dch[i]);
  }
  for (int i = threadIdx.x; i < 3 * kEoSlots; i += blockDim.x)
    tab[5 * S + i] = T(deriv && i / kEoSlots == 1 ? deriv[i % kEoSlots] : a.eo[i / kEoSlots][i % kEoSlots]);
}

// Gather three components of a global vector into dst[c][t] for the block's elements,
// optionally zeroing constrained DoFs and scaling by a per-element factor fac[e]; items of
// absent elements are zero.
template <int P, int NI, typename TS, typename T>
__device__ __forceinline__ void gather(const OpArgs& a, const Colour& col, const TS* __restrict__ src, long long e0,
                                       int nvalid, bool mask, T* dst, const T* fac = nullptr) {
  constexpr int n3 = (P + 1) * (P + 1) * (P + 1);
  for (int t = threadIdx.x; t < NI; t += blockDim.x) {
    const int e = t / n3;
    if (e < nvalid) {
      int gi, gj, gk;
      item_node<P>(col, e0 + e, t % n3, gi, gj, gk);
      const long long node = gi + (long long)a.M * (gj + (long long)a.M * gk);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        T val = T(src[c * a.M3 + node]);
        if (mask && is_constrained(a.bc, c, gi, gk, a.M)) val = T(0);
        dst[c * NI + t] = fac ? val * fac[e] : val;
      }
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c) dst[c * NI + t] = T(0);
    }
  }
}

template <typename T> struct Store { using type = T; };
template <> struct Store<df64> { using type = double; };
__device__ __forceinline__ double to_store(double x) { return x; }
__device__ __forceinline__ float to_store(float x) { return x; }
__device__ __forceinline__ double to_store(df64 x) { return to_double(x); }

// Adds the block's element results to `out` once the launches before this one are complete
// (rows of constrained DoFs keep what k_init_rows wrote), scaled by a per-element factor fac[e].
template <int P, int NI, typename T>
__device__ __forceinline__ void scatter_add(const OpArgs& a, const T* src, long long e0, int nvalid,
                                            typename Store<T>::type* out, const T* fac = nullptr) {
  constexpr int n3 = (P + 1) * (P + 1) * (P + 1);
  pdl_wait();
  for (int t = threadIdx.x; t < NI; t += blockDim.x) {
    const int e = t / n3;
    if (e >= nvalid) continue;
    int gi, gj, gk;
    item_node<P>(a.col, e0 + e, t % n3, gi, gj, gk);
    const long long node = gi + (long long)a.M * (gj + (long long)a.M * gk);
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (!is_constrained(a.bc, c, gi, gk, a.M))
        out[c * a.M3 + node] += to_store(fac ? src[c * NI + t] * fac[e] : src[c * NI + t]);
  }
}

// Forward interpolation of three components to the points: in -> out (tmp is clobbered).
template <int n, int NI, typename T>
__device__ __forceinline__ void to_points(const T* sB, T* in, T* tmp, T* out, int nitems) {
  sf_pass<n, NI, 3, 0, false>(sB, in, tmp, nitems);
  __syncthreads();
  sf_pass<n, NI, 3, 1, false>(sB, tmp, in, nitems);
  __syncthreads();
  sf_pass<n, NI, 3, 2, false>(sB, in, out, nitems);
  __syncthreads();
}

// Transposed integration of the nine point fluxes G[3c+d] to nodal values in `out`
// (`tmp` clobbered; G's first three slots are reused).
template <int n, int NI, typename T>
__device__ __forceinline__ void from_points(const T* sB, const T* sDc, T* G, T* tmp, T* out, int nitems) {
  colloc_grad_T<n, NI>(sDc, G, tmp, nitems);
  __syncthreads();
  sf_pass<n, NI, 3, 0, true>(sB, tmp, G, nitems);
  __syncthreads();
  sf_pass<n, NI, 3, 1, true>(sB, G, tmp, nitems);
  __syncthreads();
  sf_pass<n, NI, 3, 2, true>(sB, tmp, out, nitems);
  __syncthreads();
}

// The transposed passes of the apply and the residual: fluxes G[3c+d] with the weighted tables BW,
// DcW (kBW: even-odd coefficients of BW^T) to nodal values in G[3..5].
template <int n, int NI, int TH, bool EO, typename T>
__device__ __forceinline__ void transposed(const T* sBW, const T* sDcW, const T* kBW, T* G, T* Vq, int nitems,
                                           int nlines) {
  if constexpr (EO) {
    colloc_grad_T<n, NI>(sDcW, G, Vq, nitems);
    __syncthreads();
    eo_pass<n, NI, 3, 0, false, kEoCentreCol, TH>(kBW, Vq, G, nlines);
    __syncthreads();
    eo_pass<n, NI, 3, 1, false, kEoCentreCol, TH>(kBW, G, Vq, nlines);
    __syncthreads();
    eo_pass<n, NI, 3, 2, false, kEoCentreCol, TH>(kBW, Vq, G + 3 * NI, nlines);
    __syncthreads();
  } else {
    from_points<n, NI>(sBW, sDcW, G, Vq, G + 3 * NI, nitems);
  }
}

// ------------------------------------------------------------------ tangent application
// The quadrature weight, mu and h ride on the transposed tables (BW, DcW) and the element's
// material factor on the gathered du (the operator is linear in du), so the point code returns
// dP / mu without any scaling.  For odd n (Q2, Q4) every non-accumulating pass (forward B,
// forward collocation derivative, transposed B) runs one thread per line in even-odd form, and
// the gradient of du reaches the point code through shared memory.
template <int P, typename T, int STRAT, int MODEL, bool SMALL>
__global__ void __launch_bounds__(Shape<P, T, STRAT, SMALL>::THREADS) k_apply(const OpArgs a) {
  constexpr int n = P + 1, n3 = n * n * n, NE = Shape<P, T, STRAT, SMALL>::NE, NI = NE * n3;
  constexpr int S = kMaxN * kMaxN, TH = Shape<P, T, STRAT, SMALL>::THREADS;
  constexpr bool EO = n % 2 == 1;
  static_assert(5 * S + 3 * kEoSlots + NE <= kTabSlots, "the factor table exceeds the table slots");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tab = reinterpret_cast<T*>(smem_raw);
  const T* sB = tab;
  const T* sDc = tab + S;
  const T* sBW = tab + 2 * S;
  const T* sDcW = tab + 3 * S;
  const T* sDch = tab + 4 * S;
  const T* kB = tab + 5 * S;                    // even-odd coefficients of B, Dc, BW^T
  const T* kDc = kB + kEoSlots;
  const T* kBW = kDc + kEoSlots;
  T* sF = tab + 5 * S + 3 * kEoSlots;          // [NE] material factors of the block's elements
  T* U = tab + kTabSlots;                       // [3][NI] ubar at the points (on the fly)
  T* Vq = U + (STRAT == NHMF_ON_THE_FLY ? 3 * NI : 0);  // [3][NI] du at the points
  T* G = Vq + 3 * NI;                           // [9][NI] gradients, then fluxes; G[0..2] gathers

  pdl_launch_next();
  load_apply_tables<P>(a, tab);
  const Colour& col = a.col;
  const long long e0 = (long long)blockIdx.x * NE;
  const int nvalid = (int)min((long long)NE, (long long)col.count - e0);
  const int nitems = nvalid * n3, nlines = nvalid * n * n;  // items / lines of present elements
  for (int e = threadIdx.x; e < NE; e += blockDim.x) sF[e] = T(elem_factor(a, col, e0 + min(e, nvalid - 1)));
  __syncthreads();

  if constexpr (STRAT == NHMF_ON_THE_FLY) {
    gather<P, NI>(a, col, a.u64, e0, nvalid, false, G);
    __syncthreads();
    if constexpr (EO) {
      eo_pass<n, NI, 3, 0, false, kEoCentreRow, TH>(kB, G, Vq, nlines);
      __syncthreads();
      eo_pass<n, NI, 3, 1, false, kEoCentreRow, TH>(kB, Vq, G, nlines);
      __syncthreads();
      eo_pass<n, NI, 3, 2, false, kEoCentreRow, TH>(kB, G, U, nlines);
      __syncthreads();
    } else {
      to_points<n, NI>(sB, G, Vq, U, nitems);
    }
  }
  gather<P, NI>(a, col, static_cast<const typename Store<T>::type*>(a.du), e0, nvalid, true, G,
                a.factor ? (const T*)sF : nullptr);
  __syncthreads();
  if constexpr (EO) {
    eo_pass<n, NI, 3, 0, false, kEoCentreRow, TH>(kB, G, Vq, nlines);
    __syncthreads();
    eo_pass<n, NI, 3, 1, false, kEoCentreRow, TH>(kB, Vq, G, nlines);
    __syncthreads();
    eo_pass<n, NI, 3, 2, false, kEoCentreRow, TH>(kB, G, Vq, nlines);
    __syncthreads();
    // reference gradient of du: G[3c+d] = Dc along d of du[c]
    eo_pass<n, NI, 3, 0, true, kEoGeneral, TH, 3, 0>(kDc, Vq, G, nlines);
    eo_pass<n, NI, 3, 1, true, kEoGeneral, TH, 3, 1>(kDc, Vq, G, nlines);
    eo_pass<n, NI, 3, 2, true, kEoGeneral, TH, 3, 2>(kDc, Vq, G, nlines);
    __syncthreads();
  } else {
    to_points<n, NI>(sB, G, Vq + 0, Vq, nitems);  // passes ping-pong via G: x G->Vq, y Vq->G, z G->Vq
  }

  const T inv_mu = T(1.0 / a.mu), r2 = T(a.r2mu);
  const typename Store<T>::type* cache = static_cast<const typename Store<T>::type*>(a.cache);
  const long long cbase = (col.slot0 + e0) * n3;
  bool bad = false;
  for (int t = threadIdx.x; t < nitems; t += blockDim.x) {
    T dH[9], g[9];
    if constexpr (EO) {
#pragma unroll
      for (int k = 0; k < 9; ++k) dH[k] = G[k * NI + t];
    } else {
      colloc_grad<n, NI>(sDc, Vq, t, dH);
    }
    if constexpr (STRAT == NHMF_SPATIAL) {
      // Algorithm 2: J c, tau and F^-1 from the 36-value cache
      T Jc[21], tau[6], Fs[9];
      if (t / n3 < nvalid) {
        const double* sp = a.cachesp_in;
#pragma unroll
        for (int k = 0; k < 21; ++k) Jc[k] = T(sp[k * a.nq + cbase + t]);
#pragma unroll
        for (int k = 0; k < 6; ++k) tau[k] = T(sp[(21 + k) * a.nq + cbase + t]);
#pragma unroll
        for (int k = 0; k < 9; ++k) Fs[k] = T(sp[(27 + k) * a.nq + cbase + t]);
      } else {
#pragma unroll
        for (int k = 0; k < 21; ++k) Jc[k] = T(0);
#pragma unroll
        for (int k = 0; k < 6; ++k) tau[k] = T(0);
#pragma unroll
        for (int k = 0; k < 9; ++k) Fs[k] = (k % 4 == 0) ? T(1) : T(0);
      }
      spatial_stress(Jc, tau, Fs, dH, inv_mu, g);
#pragma unroll
      for (int k = 0; k < 9; ++k) G[k * NI + t] = g[k];
      continue;
    }
    if constexpr (STRAT == NHMF_ON_THE_FLY) {
      T H[9];
      colloc_grad<n, NI>(sDch, U, t, H);  // physical gradient: Dch = Dc / h
      const Kinematics<T> kin(H);
      bad |= !(kin.Jm1 > T(-1));
      if constexpr (MODEL == NHMF_MODEL_SPLIT) {
        T F[9], Fi[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          F[k] = (k % 4 == 0 ? T(1) : T(0)) + H[k];
          Fi[k] = kin.A[k] * kin.invJ;
        }
        split_stress_dP(F, Fi, kin.lnJ, kin.Jm1, dH, T(a.mu), T(a.lam), inv_mu, g);
      } else {
        linearised_stress_unit(kin, dH, r2, g);
      }
    } else {
      T Fi[9], lnJ;
      if (t / n3 < nvalid) {
        if constexpr (std::is_same<T, df64>::value) {
          const float2* cdf = static_cast<const float2*>(a.cache);
#pragma unroll
          for (int k = 0; k < 9; ++k) {
            const float2 z = cdf[k * a.nq + cbase + t];
            Fi[k] = T(z.x, z.y);
          }
          const float2 z = cdf[9 * a.nq + cbase + t];
          lnJ = T(z.x, z.y);
        } else {
          // the cache is read once per apply: evict it first, keep du and v in L2
          const unsigned long long pol = l2_evict_first();
#pragma unroll
          for (int k = 0; k < 9; ++k) Fi[k] = T(ld_policy(cache + k * a.nq + cbase + t, pol));
          lnJ = T(ld_policy(cache + 9 * a.nq + cbase + t, pol));
        }
      } else {
#pragma unroll
        for (int k = 0; k < 9; ++k) Fi[k] = (k % 4 == 0) ? T(1) : T(0);
        lnJ = T(0);
      }
      linearised_stress_unit(Fi, lnJ, dH, r2, g);
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) G[k * NI + t] = g[k];
  }
  if (bad) atomicOr(a.status, kStatusNonPosJ);
  __syncthreads();
  transposed<n, NI, TH, EO>(sBW, sDcW, kBW, G, Vq, nitems, nlines);
  scatter_add<P, NI>(a, G + 3 * NI, e0, nvalid, static_cast<typename Store<T>::type*>(a.v));
}

// ------------------------------------------------------------------ FP32 register kernel
// One thread per element: the element's three components (3 (p+1)^3 values), their values at
// the Gauss points and the transposed-derivative accumulators stay in registers; every 1D pass
// is fully unrolled, so its coefficients are compile-time-indexed kernel parameters (constant
// bank operands of the FMAs) and no shared memory is touched.  For p <= 2.  As in k_apply, w_q,
// mu and h ride on the transposed tables and the material factor on du.  The on-the-fly kernel
// runs its B and B^T passes in even-odd form at odd n; the cached kernel keeps the matrix form.
// Launched once over the class of all elements; each thread writes its element's results to
// its column of the element tile of vloc (a warp writes whole 128-byte rows) for
// k_gather_local, and reads the point cache from the same tiling.
#ifndef NHMF_REG_THREADS
#define NHMF_REG_THREADS 128
#endif
#ifndef NHMF_REG_MINB
#define NHMF_REG_MINB 1
#endif
constexpr int kRegThreads = NHMF_REG_THREADS;  // threads (= elements) per block

template <int P, int STRAT, int MODEL>
__global__ void __launch_bounds__(kRegThreads, NHMF_REG_MINB) k_apply_reg(const OpArgs a) {
  constexpr int n = P + 1, n3 = n * n * n;
  pdl_launch_next();
  pdl_wait();
  const long long ec = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (ec >= a.col.count) return;
  const Colour& col = a.col;
  const int ix = int(ec % col.nx), iy = int((ec / col.nx) % col.ny), iz = int(ec / ((long long)col.nx * col.ny));
  const int gi0 = P * (col.cx + col.stride * ix), gj0 = P * (col.cy + col.stride * iy),
            gk0 = P * (col.cz + col.stride * iz);
  const long long M = a.M;
  const long long slot = col.slot0 + ec;
  const float* du = static_cast<const float*>(a.du);
  // this element's column of its tile in the point cache and in vloc
  float* __restrict__ vloc = a.vloc + (slot / kTile) * (3 * n3 * kTile) + slot % kTile;
  const float* __restrict__ cache =
      static_cast<const float*>(a.cache) + (slot / kTile) * (10 * n3 * kTile) + slot % kTile;
  const unsigned long long stream_pol = l2_evict_first();  // the point cache is read once
  auto node = [&](int i, int j, int k) { return (gi0 + i) + M * ((gj0 + j) + M * (long long)(gk0 + k)); };
  auto idx = [](int i, int j, int k) { return i + n * (j + n * k); };

  // one 1D pass over the n^2 lines of direction DIR of f[c]: even-odd coefficients `eo` (odd
  // n) or the matrix Mat(r, m) = mat[r n + m] (TR = false) / mat[m n + r] (TR = true)
  auto pass = [&](float (&f)[n3], int dir, const float (&eo)[kEoSlots], const float* mat, bool tr) {
    // tr = false: the forward B (centre row e_h); tr = true: the transposed B^T w (centre
    // column zero off the centre) -- see eo_line
    const int st = dir == 0 ? 1 : (dir == 1 ? n : n * n);
#pragma unroll
    for (int b = 0; b < n * n; ++b) {
      const int base = dir == 0 ? b * n : (dir == 1 ? (b % n) + (b / n) * n * n : b);
      float x[n], y[n];
#pragma unroll
      for (int m = 0; m < n; ++m) x[m] = f[base + m * st];
      if constexpr (n % 2 == 1 && STRAT == NHMF_ON_THE_FLY) {
        if (tr)
          eo_line<n, false, kEoCentreCol>(eo, x, y);
        else
          eo_line<n, false, kEoCentreRow>(eo, x, y);
      } else {
#pragma unroll
        for (int r = 0; r < n; ++r) {
          float s = (tr ? mat[r] : mat[r * n]) * x[0];
#pragma unroll
          for (int m = 1; m < n; ++m) s = fmaf(tr ? mat[m * n + r] : mat[r * n + m], x[m], s);
          y[r] = s;
        }
      }
#pragma unroll
      for (int m = 0; m < n; ++m) f[base + m * st] = y[m];
    }
  };
  auto to_points = [&](float (&f)[3][n3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      pass(f[c], 0, a.eof[0], a.Bf, false);
      pass(f[c], 1, a.eof[0], a.Bf, false);
      pass(f[c], 2, a.eof[0], a.Bf, false);
    }
  };
  auto grad_at = [&](const float* Dc, const float (&f)[3][n3], int qx, int qy, int qz, float g[9]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float gx = Dc[qx * n] * f[c][idx(0, qy, qz)];
      float gy = Dc[qy * n] * f[c][idx(qx, 0, qz)];
      float gz = Dc[qz * n] * f[c][idx(qx, qy, 0)];
#pragma unroll
      for (int m = 1; m < n; ++m) {
        gx = fmaf(Dc[qx * n + m], f[c][idx(m, qy, qz)], gx);
        gy = fmaf(Dc[qy * n + m], f[c][idx(qx, m, qz)], gy);
        gz = fmaf(Dc[qz * n + m], f[c][idx(qx, qy, m)], gz);
      }
      g[3 * c + 0] = gx;
      g[3 * c + 1] = gy;
      g[3 * c + 2] = gz;
    }
  };

  float qv[3][n3];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int k = 0; k < n; ++k)
#pragma unroll
      for (int j = 0; j < n; ++j)
#pragma unroll
        for (int i = 0; i < n; ++i) {
          const bool fixed = is_constrained(a.bc, c, gi0 + i, gk0 + k, a.M);
          qv[c][idx(i, j, k)] = fixed ? 0.f : du[c * a.M3 + node(i, j, k)];
        }
  if (a.factor) {
    const float fac = float(elem_factor(a, col, ec));
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int q = 0; q < n3; ++q) qv[c][q] *= fac;
  }
  to_points(qv);
  float ub[STRAT == NHMF_ON_THE_FLY ? 3 : 1][STRAT == NHMF_ON_THE_FLY ? n3 : 1];
  if constexpr (STRAT == NHMF_ON_THE_FLY) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int k = 0; k < n; ++k)
#pragma unroll
        for (int j = 0; j < n; ++j)
#pragma unroll
          for (int i = 0; i < n; ++i) ub[c][idx(i, j, k)] = a.u32[c * a.M3 + node(i, j, k)];
    to_points(ub);
  }
  // Compressible model on the fly: the values of ubar at the points go to shared memory
  // ([3 n^3][T], one column per thread), and the kinematics (F^-1, J - 1, ln J) of each
  // qz-slice are computed in a rolled loop into a slice buffer ([10][n^2][T]) that the unrolled
  // point code then reads: the kinematics code exists once instead of n^3 times, which keeps
  // the unrolled kernel within the instruction cache, and ubar holds no registers there.
  constexpr bool KIN = STRAT == NHMF_ON_THE_FLY && MODEL == NHMF_MODEL_COMPRESSIBLE;
  constexpr int n2 = n * n;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* ubs = reinterpret_cast<float*>(smem_raw);
  float* kin = ubs + 3 * n3 * blockDim.x;
  const int T = blockDim.x;
  if constexpr (KIN) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int q = 0; q < n3; ++q) ubs[(c * n3 + q) * T + threadIdx.x] = ub[c][q];
  }

  float acc[3][n3];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int q = 0; q < n3; ++q) acc[c][q] = 0.f;
  const float r2 = float(a.r2mu), inv_mu = float(1.0 / a.mu);
  bool bad = false;
#pragma unroll
  for (int qz = 0; qz < n; ++qz) {
    if constexpr (KIN) {
#pragma unroll 1
      for (int pt = 0; pt < n2; ++pt) {
        const int qx = pt % n, qy = pt / n;
        const float* u0 = ubs + threadIdx.x;
        float H[9], Fi[9], lnJ;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
          for (int m = 0; m < n; ++m) {
            gx = fmaf(a.Dchf[qx * n + m], u0[(c * n3 + idx(m, qy, qz)) * T], gx);
            gy = fmaf(a.Dchf[qy * n + m], u0[(c * n3 + idx(qx, m, qz)) * T], gy);
            gz = fmaf(a.Dchf[qz * n + m], u0[(c * n3 + idx(qx, qy, m)) * T], gz);
          }
          H[3 * c + 0] = gx;
          H[3 * c + 1] = gy;
          H[3 * c + 2] = gz;
        }
        const float Jm1 = kinematics(H, Fi, lnJ);
        bad |= !(Jm1 > -1.f);
        float* k0 = kin + pt * T + threadIdx.x;
#pragma unroll
        for (int k = 0; k < 9; ++k) k0[k * n2 * T] = Fi[k];
        k0[9 * n2 * T] = lnJ;
      }
    }
#pragma unroll
    for (int qy = 0; qy < n; ++qy)
#pragma unroll
      for (int qx = 0; qx < n; ++qx) {
        const int q = idx(qx, qy, qz);
        float Fi[9], lnJ, Jm1 = 0.f, F[9];
        if constexpr (KIN) {
          const float* k0 = kin + (qx + n * qy) * T + threadIdx.x;
#pragma unroll
          for (int k = 0; k < 9; ++k) Fi[k] = k0[k * n2 * T];
          lnJ = k0[9 * n2 * T];
        } else if constexpr (STRAT == NHMF_ON_THE_FLY) {
          float H[9];
          grad_at(a.Dchf, ub, qx, qy, qz, H);  // physical gradient: Dch = Dc / h
          Jm1 = kinematics(H, Fi, lnJ);
          bad |= !(Jm1 > -1.f);
#pragma unroll
          for (int k = 0; k < 9; ++k) F[k] = (k % 4 == 0 ? 1.f : 0.f) + H[k];
        } else {
#pragma unroll
          for (int k = 0; k < 9; ++k) Fi[k] = ld_policy(cache + (k * n3 + q) * kTile, stream_pol);
          lnJ = ld_policy(cache + (9 * n3 + q) * kTile, stream_pol);
        }
        float dH[9], g[9];
        grad_at(a.Dcf, qv, qx, qy, qz, dH);
        if constexpr (STRAT == NHMF_ON_THE_FLY && MODEL == NHMF_MODEL_SPLIT)
          split_stress_dP(F, Fi, lnJ, Jm1, dH, float(a.mu), float(a.lam), inv_mu, g);
        else
          linearised_stress_terms(Fi, fmaf(-r2, lnJ, 1.f), r2, dH, g);
        // transposed collocation derivative with the weights, mu and h:
        //   acc[c][point on the line through q] += DcW[q][m] g
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int m = 0; m < n; ++m) {
            acc[c][idx(m, qy, qz)] = fmaf(a.DcWf[qx * n + m], g[3 * c + 0], acc[c][idx(m, qy, qz)]);
            acc[c][idx(qx, m, qz)] = fmaf(a.DcWf[qy * n + m], g[3 * c + 1], acc[c][idx(qx, m, qz)]);
            acc[c][idx(qx, qy, m)] = fmaf(a.DcWf[qz * n + m], g[3 * c + 2], acc[c][idx(qx, qy, m)]);
          }
      }
  }
  if (bad) atomicOr(a.status, kStatusNonPosJ);
  // transposed weighted interpolation back to the nodes: out[i] = sum_q B[q][i] w_q acc[q]
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    pass(acc[c], 0, a.eof[2], a.BWf, true);
    pass(acc[c], 1, a.eof[2], a.BWf, true);
    pass(acc[c], 2, a.eof[2], a.BWf, true);
  }
  const unsigned long long keep_pol = l2_evict_last();  // read back by the gather that follows
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int q = 0; q < n3; ++q) st_policy(vloc + (c * n3 + q) * kTile, acc[c][q], keep_pol);
}

// ------------------------------------------------------------------ element-local gather
// v[c][node] = sum of vloc(e; c, q) over the elements e whose closure holds the node (1, 2, 4
// or 8 of them; q the node's local index in e), always in increasing (ez, ey, ex) order, so
// the result is bitwise deterministic without atomics.  Dirichlet rows (unless raw):
// v = du there.  One thread per node.  The multigrid's vector updates ride on the gather (see
// Gather32): a node's result is final here, so b - A x, a Chebyshev step or a power-iteration
// step costs no further pass over A x and no launch.  v may be du in those forms: every thread
// reads and writes its own node only.
template <int P, int MODE>
__global__ void __launch_bounds__(256) k_gather_local(const float* vloc, const float* du, float* v, int N,
                                                     int M, int bc, const Gather32 g32) {
  constexpr int n = P + 1, n3 = n * n * n;
  static_assert(kTile == 32, "tile index by shift and mask");
  pdl_launch_next();
  // grid: x covers the M^2 nodes of one z-plane, y the plane (32-bit index arithmetic; the
  // launcher keeps the element count below 2^31)
  const int ij = blockIdx.x * blockDim.x + threadIdx.x;
  if (ij >= M * M) return;
  const int gj = ij / M;
  const int g[3] = {ij - gj * M, gj, (int)blockIdx.y};
  const long long node = ij + (long long)M * M * blockIdx.y, M3 = (long long)M * M * M;
  const unsigned long long done_pol = l2_evict_first();  // each element-local value is read once
  pdl_wait();
  // per direction: the element below the node (local index P), if any, then the element at or
  // above it (local index g % P); an absent element in x gets a clamped (valid) index and is
  // masked after the load
  int el[3][2], lo[3][2];
  bool has[3][2];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int gp = g[d] / P, gr = g[d] - gp * P;
    const bool shared = gr == 0;
    has[d][0] = shared && g[d] > 0;
    el[d][0] = max(gp - 1, 0);
    lo[d][0] = P;
    has[d][1] = !shared || g[d] < M - 1;
    el[d][1] = min(gp, N - 1);
    lo[d][1] = gr;
  }
  // the (z, y) element pairs are the same for every node of a grid row, so a warp skips the
  // absent ones as a whole (a branch, not 6 issued loads); the loads of the present ones are
  // issued before any of them is used
  float val[3][8];
#pragma unroll
  for (int z = 0; z < 2; ++z)
#pragma unroll
    for (int y = 0; y < 2; ++y) {
#pragma unroll
      for (int c = 0; c < 3; ++c) val[c][4 * z + 2 * y] = val[c][4 * z + 2 * y + 1] = 0.f;
      if (!(has[2][z] && has[1][y])) continue;
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const unsigned e = (unsigned)el[0][x] + (unsigned)N * ((unsigned)el[1][y] + (unsigned)N * (unsigned)el[2][z]);
        const int q = lo[0][x] + n * (lo[1][y] + n * lo[2][z]);
        const float* src = vloc + (size_t)(e >> 5) * (3 * n3 * kTile) + q * kTile + (e & 31u);
#pragma unroll
        for (int c = 0; c < 3; ++c) val[c][4 * z + 2 * y + x] = ld_produced(src + c * n3 * kTile, done_pol);
      }
    }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float s = 0.f;
#pragma unroll
    for (int z = 0; z < 2; ++z)
#pragma unroll
      for (int y = 0; y < 2; ++y)
#pragma unroll
        for (int x = 0; x < 2; ++x)
          if (has[2][z] && has[1][y] && has[0][x]) s += val[c][4 * z + 2 * y + x];
    const long long i = c * M3 + node;
    if (is_constrained(bc, c, g[0], g[2], M)) s = du[i];
    if constexpr (MODE == Gather32::kApply) {
      v[i] = s;
    } else if constexpr (MODE == Gather32::kResidual) {
      v[i] = g32.b[i] - s;
    } else if constexpr (MODE == Gather32::kChebyshev) {
      const float t = g32.c_new * g32.dinv[i] * (g32.b[i] - s);
      const float di = g32.c_old == 0.f ? t : fmaf(g32.c_old, g32.d[i], t);
      g32.d[i] = di;
      v[i] = du[i] + di;
    } else {
      v[i] = 0.25f * g32.dinv[i] * s;
    }
  }
}

// ------------------------------------------------------------------ point cache
// SPATIAL: Algorithm 2's 36 values as well (compiled apart: its code takes the registers that let
// a second and third block hide the plain cache's latencies).
template <int P, bool SMALL, bool SPATIAL>
__global__ void __launch_bounds__(Shape<P, double, NHMF_CACHED, SMALL>::THREADS) k_cache(const OpArgs a) {
  using T = double;
  constexpr int n = P + 1, n3 = n * n * n, NE = Shape<P, T, NHMF_CACHED, SMALL>::NE, NI = NE * n3;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sB = reinterpret_cast<T*>(smem_raw);
  T* sDch = sB + kMaxN * kMaxN;
  T* A = sB + kTabSlots;  // [3][NI]
  T* Vq = A + 3 * NI;     // [3][NI]
  for (int i = threadIdx.x; i < n * n; i += blockDim.x) {
    sB[i] = a.B[i];
    sDch[i] = a.Dch[i];  // physical gradients
  }
  long long e0;
  const Colour col = block_colour<NE>(a.N, e0);  // one launch: the classes are independent here
  const int nvalid = (int)min((long long)NE, (long long)col.count - e0);
  gather<P, NI>(a, col, a.u64, e0, nvalid, false, A);
  __syncthreads();
  to_points<n, NI>(sB, A, Vq, Vq, nvalid * n3);
  const long long cbase = (col.slot0 + e0) * n3;
  bool bad = false;
  for (int t = threadIdx.x; t < nvalid * n3; t += blockDim.x) {
    double H[9], Fi[9], lnJ;
    colloc_grad<n, NI>(sDch, Vq, t, H);
    const double Jm1 = kinematics(H, Fi, lnJ);
    bad |= !(Jm1 > -1.0);
    if (a.cache64_out) {
#pragma unroll
      for (int k = 0; k < 9; ++k) a.cache64_out[k * a.nq + cbase + t] = Fi[k];
      a.cache64_out[9 * a.nq + cbase + t] = lnJ;
    }
    if constexpr (SPATIAL) {
      // Algorithm 2 cache from the model's P and dP only: tau = P F^T;
      // J a_ijkl = (dP[e_k (x) F_l.] F^T)_ij, J c_ijkl = J a_ijkl - delta_ik tau_jl
      double F[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) F[k] = (k % 4 == 0 ? 1.0 : 0.0) + H[k];
      double P[9], tau[9];
      model_piola(a.model, F, Fi, lnJ, Jm1, a.mu, a.lam, P);
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
          tau[3 * i + j] = fma(P[3 * i], F[3 * j], fma(P[3 * i + 1], F[3 * j + 1], P[3 * i + 2] * F[3 * j + 2]));
      double* out = a.cachesp_out;
      const int pk[6] = {0, 1, 2, 1, 0, 0}, pl[6] = {0, 1, 2, 2, 2, 1};
#pragma unroll
      for (int K = 0; K < 6; ++K) {
        const int k = pk[K], l = pl[K];
        double X[9], dP[9];
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
          for (int L = 0; L < 3; ++L) X[3 * m + L] = (m == k) ? F[3 * l + L] : 0.0;
        model_dP(a.model, F, Fi, lnJ, Jm1, X, a.mu, a.lam, 1.0, dP);
#pragma unroll
        for (int I = 0; I <= K; ++I) {
          const int i = pk[I], j = pl[I];
          const double Ja = fma(dP[3 * i], F[3 * j], fma(dP[3 * i + 1], F[3 * j + 1], dP[3 * i + 2] * F[3 * j + 2]));
          out[tri6(I, K) * a.nq + cbase + t] = Ja - (i == k ? tau[3 * j + l] : 0.0);
        }
      }
      const int vi[6] = {0, 4, 8, 5, 2, 1};  // tau in Voigt order 11, 22, 33, 23, 13, 12
#pragma unroll
      for (int V = 0; V < 6; ++V) out[(21 + V) * a.nq + cbase + t] = tau[vi[V]];
#pragma unroll
      for (int k = 0; k < 9; ++k) out[(27 + k) * a.nq + cbase + t] = Fi[k];
    }
    if (a.cachedf_out) {
      auto split = [](double d) {
        const float hi = __double2float_rn(d);
        return make_float2(hi, __double2float_rn(d - (double)hi));
      };
#pragma unroll
      for (int k = 0; k < 9; ++k) a.cachedf_out[k * a.nq + cbase + t] = split(Fi[k]);
      a.cachedf_out[9 * a.nq + cbase + t] = split(lnJ);
    }
    if (a.cache32_out) {
      // the FP32 applies run over all elements in natural order (element-local results)
      const long long en = elem_natural(a, col, e0 + t / n3), q = t % n3;
      if (P <= kRegMaxP && a.reg32) {
        // element tiles [E/32][10][n^3][32] for the register kernel (one thread per element)
        float* tile = a.cache32_out + (en / kTile) * (10 * n3 * kTile) + en % kTile;
#pragma unroll
        for (int k = 0; k < 9; ++k) tile[(k * n3 + q) * kTile] = float(Fi[k]);
        tile[(9 * n3 + q) * kTile] = float(lnJ);
      } else {
        // layout [10][E n^3] for the column kernel
#pragma unroll
        for (int k = 0; k < 9; ++k) a.cache32_out[k * a.nq + en * n3 + q] = float(Fi[k]);
        a.cache32_out[9 * a.nq + en * n3 + q] = float(lnJ);
      }
    }
  }
  if (bad) atomicOr(a.status, kStatusNonPosJ);
}

// ------------------------------------------------------------------ residual
// The passes of the on-the-fly apply with P(F) / mu in place of dP / mu: the weights, mu and h ride
// on the transposed tables, the other h of the integral and the material factor on the scatter.  FP64 operations per point
// bound it: with the kinematics above, P from the adjugate (P / mu = F + c A^T) and the even-odd
// passes of odd n, Q3 48^3 takes 320 -> 165 of them.
template <int P, bool SMALL>
__global__ void __launch_bounds__(Shape<P, double, 0, SMALL>::THREADS) k_residual(const OpArgs a) {
  using T = double;
  constexpr int n = P + 1, n3 = n * n * n, NE = Shape<P, T, 0, SMALL>::NE, NI = NE * n3;
  constexpr int S = kMaxN * kMaxN, TH = Shape<P, T, 0, SMALL>::THREADS;
  constexpr bool EO = n % 2 == 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tab = reinterpret_cast<T*>(smem_raw);
  const T *kB = tab + 5 * S, *kDch = kB + kEoSlots, *kBW = kDch + kEoSlots;
  T* sF = tab + 5 * S + 3 * kEoSlots;  // [NE] h times the material factors
  T* Vq = tab + kTabSlots;             // [3][NI] u at the points
  T* G = Vq + 3 * NI;                  // [9][NI] gradients, then fluxes
  pdl_launch_next();
  load_apply_tables<P>(a, tab, a.eoh);
  const Colour& col = a.col;
  const long long e0 = (long long)blockIdx.x * NE;
  const int nvalid = (int)min((long long)NE, (long long)col.count - e0);
  const int nitems = nvalid * n3, nlines = nvalid * n * n;
  for (int e = threadIdx.x; e < NE; e += blockDim.x) sF[e] = a.h * elem_factor(a, col, e0 + min(e, nvalid - 1));
  gather<P, NI>(a, col, a.u64, e0, nvalid, false, G);
  __syncthreads();
  if constexpr (EO) {
    eo_pass<n, NI, 3, 0, false, kEoCentreRow, TH>(kB, G, Vq, nlines);
    __syncthreads();
    eo_pass<n, NI, 3, 1, false, kEoCentreRow, TH>(kB, Vq, G, nlines);
    __syncthreads();
    eo_pass<n, NI, 3, 2, false, kEoCentreRow, TH>(kB, G, Vq, nlines);
    __syncthreads();
    eo_pass<n, NI, 3, 0, true, kEoGeneral, TH, 3, 0>(kDch, Vq, G, nlines);
    eo_pass<n, NI, 3, 1, true, kEoGeneral, TH, 3, 1>(kDch, Vq, G, nlines);
    eo_pass<n, NI, 3, 2, true, kEoGeneral, TH, 3, 2>(kDch, Vq, G, nlines);
    __syncthreads();
  } else {
    to_points<n, NI>(tab, G, Vq, Vq, nitems);
  }
  const T r2 = a.r2mu, inv_mu = 1.0 / a.mu;
  unsigned flags = 0;
  for (int t = threadIdx.x; t < nitems; t += blockDim.x) {
    T H[9], g[9];
    if constexpr (EO) {
#pragma unroll
      for (int k = 0; k < 9; ++k) H[k] = G[k * NI + t];
    } else {
      colloc_grad<n, NI>(tab + 4 * S, Vq, t, H);
    }
    const Kinematics<T> kin(H);
    // a NaN deformation gradient is a non-finite input; det F <= 0 makes P non-finite too,
    // but is reported as what it is (the Newton backtracking acts on it)
    const bool inverted = kin.Jm1 <= -1.0;
    if (inverted) flags |= kStatusNonPosJ;
    if (a.model == NHMF_MODEL_SPLIT) {
      T F[9], Fi[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        F[k] = (k % 4 == 0 ? 1.0 : 0.0) + H[k];
        Fi[k] = kin.A[k] * kin.invJ;
      }
      model_piola(a.model, F, Fi, kin.lnJ, kin.Jm1, a.mu, a.lam, g);
#pragma unroll
      for (int k = 0; k < 9; ++k) g[k] *= inv_mu;
    } else {
      const T c = fma(r2, kin.lnJ, -1.0) * kin.invJ;
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
          g[3 * i + j] = fma(c, kin.A[3 * j + i], i == j ? 1.0 + H[3 * i + j] : H[3 * i + j]);
    }
    bool finite = true;  // by the exponent bits: the FP64 pipe is the busy unit
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      finite &= (__double2hiint(g[k]) & 0x7ff00000) != 0x7ff00000;
      G[k * NI + t] = g[k];
    }
    if (!inverted && !finite) flags |= kStatusNonFinite;
  }
  if (flags) atomicOr(a.status, flags);
  __syncthreads();
  transposed<n, NI, TH, EO>(tab + 2 * S, tab + 3 * S, kBW, G, Vq, nitems, nlines);
  scatter_add<P, NI>(a, G + 3 * NI, e0, nvalid, static_cast<double*>(a.v), (const T*)sF);
}

// ------------------------------------------------------------------ diagonal
// diag(K)_{c,I} = sum_q sum_{d,l} L_{cdcl} dphi_I/dX_d dphi_I/dX_l w_q h^3 with
// L_{cdcl} = mu delta_dl + (mu + 2 lambda (1 - ln J)) Finv[d][c] Finv[l][c].  The products of 1D
// factors are separable: with T0 = B.B, T1 = B.D, T2 = D.D (times w), pair (d, l) contracts
// direction e with T_m, m the number of d, l equal to e.  x: six pairs, in place; y: the pairs of one
// z-factor are added as they are contracted (00, 01, 11 | 02, 12 | 22); z: the three sums
// at once.  15 line passes per component instead of 18 and the additions; the symmetric pairs'
// factor 2 rides on the x tables, h and the material factor on the scatter.  FP64 operations per
// point bound it.
template <int P, bool SMALL> struct DiagCfg {
  using S = Shape<P, double, NHMF_CACHED, SMALL>;
  static constexpr int NE = SMALL ? S::NE : (S::NE / 2 > 0 ? S::NE / 2 : 1), THREADS = S::THREADS;
};
constexpr int kDiagFields = 21;  // 18 pair fields and u at the points

// One line of NIN fields contracted and summed into `out`: y_k = sum_f sum_q tab[f][q][k] x_f[q].
template <int n, int NIN>
__device__ __forceinline__ void diag_line(const double* const (&tab)[NIN], const double* const (&in)[NIN], double* out,
                                          int s) {
  double y[n];
#pragma unroll
  for (int f = 0; f < NIN; ++f) {
    double x[n];
#pragma unroll
    for (int q = 0; q < n; ++q) x[q] = in[f][q * s];
#pragma unroll
    for (int k = 0; k < n; ++k) {
#pragma unroll
      for (int q = 0; q < n; ++q) y[k] = f == 0 && q == 0 ? tab[f][k] * x[0] : fma(tab[f][q * n + k], x[q], y[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < n; ++k) out[k * s] = y[k];
}

// CACHED: F^-1 and ln J come from the FP64 point cache of the linearisation point (compressible
// model), which saves a third of the operations (u's values, gradient and kinematics).
template <int P, bool SMALL, bool CACHED>
__global__ void __launch_bounds__(DiagCfg<P, SMALL>::THREADS) k_diagonal(const OpArgs a) {
  using T = double;
  constexpr int n = P + 1, n3 = n * n * n, NE = DiagCfg<P, SMALL>::NE, NI = NE * n3, NL = NE * n * n;
  constexpr int S = kMaxN * kMaxN, TH = DiagCfg<P, SMALL>::THREADS;
  constexpr bool EO = n % 2 == 1;
  static_assert(7 * S + kEoSlots + NE <= kTabSlots, "the diagonal's tables exceed the table slots");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* sB = reinterpret_cast<T*>(smem_raw);
  T *sDch = sB + S, *tBB = sDch + S, *tBD = tBB + S, *tDD = tBD + S, *t2BB = tDD + S, *t2BD = t2BB + S;
  T *kB = t2BD + S, *sF = kB + kEoSlots;
  T* X = sB + kTabSlots;  // [18][NI]: field 3 pair + c, pairs 00, 01, 02, 11, 12, 22
  T* Vq = X + 18 * NI;    // [3][NI]
  pdl_launch_next();
  for (int i = threadIdx.x; i < n * n; i += blockDim.x) {
    const T b = a.B[i], d = a.D[i], wq = a.w[i / n];
    sB[i] = b;
    sDch[i] = a.Dch[i];
    tBB[i] = wq * b * b;
    tBD[i] = wq * b * d;
    tDD[i] = wq * d * d;
    t2BB[i] = 2.0 * (wq * b * b);
    t2BD[i] = 2.0 * (wq * b * d);
  }
  for (int i = threadIdx.x; i < kEoSlots; i += blockDim.x) kB[i] = a.eo[0][i];
  const Colour& col = a.col;
  const long long e0 = (long long)blockIdx.x * NE;
  const int nvalid = (int)min((long long)NE, (long long)col.count - e0);
  const int nitems = nvalid * n3, nlines = nvalid * n * n;
  for (int e = threadIdx.x; e < NE; e += blockDim.x) sF[e] = a.h * elem_factor(a, col, e0 + min(e, nvalid - 1));
  if constexpr (!CACHED) {
    gather<P, NI>(a, col, a.u64, e0, nvalid, false, X);
    __syncthreads();
    if constexpr (EO) {
      eo_pass<n, NI, 3, 0, false, kEoCentreRow, TH>(kB, X, Vq, nlines);
      __syncthreads();
      eo_pass<n, NI, 3, 1, false, kEoCentreRow, TH>(kB, Vq, X, nlines);
      __syncthreads();
      eo_pass<n, NI, 3, 2, false, kEoCentreRow, TH>(kB, X, Vq, nlines);
      __syncthreads();
    } else {
      to_points<n, NI>(sB, X, Vq, Vq, nitems);
    }
  }
  const double* cache = static_cast<const double*>(a.cache) + (col.slot0 + e0) * n3;
  const unsigned long long pol = l2_evict_first();
  for (int t = threadIdx.x; t < nitems; t += blockDim.x) {
    T H[9];
    // the matrix f whose entries enter L twice, and the factor that makes f f the product of F^-1's
    T f9[9], kap;
    Kinematics<T> kin;
    if constexpr (CACHED) {
#pragma unroll
      for (int k = 0; k < 9; ++k) f9[k] = ld_policy(cache + k * a.nq + t, pol);
      kap = fma(2.0 * a.lam, 1.0 - ld_policy(cache + 9 * a.nq + t, pol), a.mu);
    } else {
      colloc_grad<n, NI>(sDch, Vq, t, H);
      kin = Kinematics<T>(H);
#pragma unroll
      for (int k = 0; k < 9; ++k) f9[k] = kin.A[k];
      kap = fma(2.0 * a.lam, 1.0 - kin.lnJ, a.mu) * (kin.invJ * kin.invJ);
    }
    const int pd[6] = {0, 0, 0, 1, 1, 2}, pl[6] = {0, 1, 2, 1, 2, 2};
    if (!CACHED && a.model == NHMF_MODEL_SPLIT) {
      // L_cdcl = mu a d_dl - 2/3 mu a (F_cd Fi_lc + Fi_dc F_cl) + (2/9 mu a I1 + kappa J^2
      //          + mu a I1/3 - kappa/2 (J^2 - 1)) Fi_dc Fi_lc
      const T J = 1.0 + kin.Jm1, J2 = J * J, mua = a.mu * exp(-2.0 / 3.0 * kin.lnJ);
      T I1 = 0.0, F[9], Fi[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        F[k] = (k % 4 == 0 ? 1.0 : 0.0) + H[k];
        Fi[k] = kin.A[k] * kin.invJ;
        I1 += F[k] * F[k];
      }
      const T cff = 2.0 / 9.0 * mua * I1 + a.lam * J2 + mua * I1 / 3.0 - 0.5 * a.lam * (J2 - 1.0);
#pragma unroll
      for (int pr = 0; pr < 6; ++pr)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int d = pd[pr], l = pl[pr];
          const T Fidc = Fi[3 * d + c], Filc = Fi[3 * l + c];
          X[(3 * pr + c) * NI + t] = (d == l ? mua : 0.0) - 2.0 / 3.0 * mua * (F[3 * c + d] * Filc + Fidc * F[3 * c + l]) +
                                     cff * Fidc * Filc;
        }
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        T f[3], kf[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          f[d] = f9[3 * d + c];
          kf[d] = kap * f[d];
        }
#pragma unroll
        for (int pr = 0; pr < 6; ++pr)
          X[(3 * pr + c) * NI + t] = pd[pr] == pl[pr] ? fma(kf[pd[pr]], f[pl[pr]], a.mu) : kf[pd[pr]] * f[pl[pr]];
      }
    }
  }
  __syncthreads();
  for (int task = threadIdx.x; task < 18 * NL; task += TH) {
    const int f = task / NL, L = task - f * NL;
    if (L >= nlines) continue;
    const int pr = f / 3;
    T* x = X + f * NI + L * n;
    const T* const tab[1] = {pr == 0 ? tDD : pr < 3 ? t2BD : pr == 4 ? t2BB : tBB};
    const T* const in[1] = {x};
    diag_line<n, 1>(tab, in, x, 1);
  }
  __syncthreads();
  for (int task = threadIdx.x; task < 9 * NL; task += TH) {
    const int g = task / (3 * NL), rest = task - g * 3 * NL, c = rest / NL, L = rest - c * NL;
    if (L >= nlines) continue;
    T* x = X + c * NI + (L % n) + (L / n) * n * n;
    if (g == 0) {
      const T* const tab[3] = {tBB, tBD, tDD};
      const T* const in[3] = {x, x + 3 * NI, x + 9 * NI};
      diag_line<n, 3>(tab, in, x, n);
    } else if (g == 1) {
      const T* const tab[2] = {tBB, tBD};
      const T* const in[2] = {x + 6 * NI, x + 12 * NI};
      diag_line<n, 2>(tab, in, x + 6 * NI, n);
    } else {
      const T* const tab[1] = {tBB};
      const T* const in[1] = {x + 15 * NI};
      diag_line<n, 1>(tab, in, x + 15 * NI, n);
    }
  }
  __syncthreads();
  for (int task = threadIdx.x; task < 3 * NL; task += TH) {
    const int c = task / NL, L = task - c * NL;
    if (L >= nlines) continue;
    T* x = X + c * NI + (L % (n * n)) + (L / (n * n)) * n * n * n;
    const T* const tab[3] = {tBB, tBD, tDD};
    const T* const in[3] = {x, x + 6 * NI, x + 15 * NI};
    diag_line<n, 3>(tab, in, x, n * n);
  }
  __syncthreads();
  scatter_add<P, NI>(a, X, e0, nvalid, static_cast<double*>(a.v), (const T*)sF);
}

// ------------------------------------------------------------------ result vector
// What the colour classes add to: zero, and on every constrained DoF src[d], or `value` where
// src is null.  Grid: x covers the M^2 nodes of a z-plane, y the 3 M planes of the three
// components.
constexpr int kInitPer = 4;  // entries per thread
template <typename T>
__global__ void __launch_bounds__(256) k_init_rows(int bc, int M, const T* src, T* out, T value) {
  pdl_wait();
  pdl_launch_next();  // after the wait: the first class reads du, which earlier launches write, before its own
  const int c = (int)blockIdx.y / M, k = (int)blockIdx.y - c * M, M2 = M * M;
  const long long base = (long long)M2 * blockIdx.y;
#pragma unroll
  for (int j = 0; j < kInitPer; ++j) {
    const int ij = (blockIdx.x * kInitPer + j) * 256 + threadIdx.x;
    if (ij < M2) out[base + ij] = !is_constrained(bc, c, ij % M, k, M) ? T(0) : src ? src[base + ij] : value;
  }
}

// ------------------------------------------------------------------ host side
// Even-odd coefficients (see eo_line) of the n x n row-major operator M, odd n.
void eo_pack(const double* M, int n, double* k) {
  const int h = n / 2, A0 = (h + 1) * h, C0 = 2 * (h + 1) * h;
  for (int i = 0; i < kEoSlots; ++i) k[i] = 0.0;
  for (int r = 0; r <= h; ++r) {
    for (int m = 0; m < h; ++m) {
      k[r * h + m] = 0.5 * (M[r * n + m] + M[r * n + n - 1 - m]);
      k[A0 + r * h + m] = 0.5 * (M[r * n + m] - M[r * n + n - 1 - m]);
    }
    k[C0 + r] = M[r * n + h];
  }
}

// The even-odd form of an n x n line operator M (row-major) for the FP32 column kernel.
EoTab eo_tab(const double* M, int n) {
  EoTab t{};
  const int h = n / 2;
  for (int r = 0; r < h; ++r) {
    for (int m = 0; m < h; ++m) {
      t.S[r][m] = float(0.5 * (M[r * n + m] + M[r * n + n - 1 - m]));
      t.A[r][m] = float(0.5 * (M[r * n + m] - M[r * n + n - 1 - m]));
    }
    t.C[r] = n % 2 == 1 ? float(M[r * n + h]) : 0.f;
    t.mid[r] = n % 2 == 1 ? float(M[h * n + r]) : 0.f;
  }
  t.ch = n % 2 == 1 ? float(M[h * n + h]) : 0.f;
  return t;
}

OpArgs base_args(nhmf_ctx* c) {
  OpArgs a{};
  a.N = c->g.N;
  a.M = c->g.M;
  a.bc = c->prm.bc;
  a.model = c->prm.model;
  a.M3 = c->g.M3;
  a.nq = c->g.nq;
  a.h = c->g.h;
  a.mu = c->prm.mu;
  a.lam = c->prm.lambda;
  const int n = c->g.n;
  for (int q = 0; q < n; ++q) {
    a.w[q] = c->tab.w[q];
    for (int i = 0; i < n; ++i) {
      a.B[q * n + i] = c->tab.B[q][i];
      a.Dc[q * n + i] = c->tab.Dc[q][i];
      a.D[q * n + i] = c->tab.D[q][i];
      a.Bf[q * n + i] = float(c->tab.B[q][i]);
      a.Dcf[q * n + i] = float(c->tab.Dc[q][i]);
    }
  }
  // tables of the tangent apply (see OpArgs)
  double BWt[kMaxN * kMaxN];
  for (int q = 0; q < n; ++q)
    for (int i = 0; i < n; ++i) {
      const double wq = c->tab.w[q];
      a.BW[q * n + i] = c->tab.B[q][i] * wq;
      BWt[i * n + q] = a.BW[q * n + i];
      a.DcW[q * n + i] = c->tab.Dc[q][i] * wq / c->tab.w[i] * c->prm.mu * c->g.h;
      a.Dch[q * n + i] = c->tab.Dc[q][i] / c->g.h;
    }
  if (n % 2 == 1) {
    eo_pack(a.B, n, a.eo[0]);
    eo_pack(a.Dc, n, a.eo[1]);
    eo_pack(BWt, n, a.eo[2]);
    eo_pack(a.Dch, n, a.eoh);
  }
  if (n >= 3) {
    double DWt[kMaxN * kMaxN], BWz[kMaxN * kMaxN], DWz[kMaxN * kMaxN];
    for (int q = 0; q < n; ++q)
      for (int i = 0; i < n; ++i) {
        DWt[i * n + q] = c->tab.D[q][i] * c->tab.w[q];
        BWz[i * n + q] = BWt[i * n + q] * c->prm.mu * c->g.h;
        DWz[i * n + q] = DWt[i * n + q] * c->prm.mu * c->g.h;
      }
    a.cB = eo_tab(a.B, n);
    a.cD = eo_tab(a.D, n);
    a.cBT = eo_tab(BWt, n);
    a.cDT = eo_tab(DWt, n);
    a.cBTz = eo_tab(BWz, n);
    a.cDTz = eo_tab(DWz, n);
  }
  a.invhf = float(1.0 / c->g.h);
  a.r2mu = 2.0 * c->prm.lambda / c->prm.mu;
  a.r2muf = float(a.r2mu);
  a.reg32 = c->reg32 ? 1 : 0;
  for (int i = 0; i < kMaxN * kMaxN; ++i) {
    a.BWf[i] = float(a.BW[i]);
    a.DcWf[i] = float(a.DcW[i]);
    a.Dchf[i] = float(a.Dch[i]);
  }
  for (int k = 0; k < 3; ++k)
    for (int i = 0; i < kEoSlots; ++i) a.eof[k][i] = float(a.eo[k][i]);
  a.status = c->status;
  a.factor = c->factor;
  return a;
}

template <typename KernelT>
cudaError_t prepare(KernelT kernel, size_t smem) {
  if (smem > 48 * 1024)
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  return cudaSuccess;
}

// Runs `kernel` once per colour class with NE elements per block, after k_init_rows on `out`.  The
// classes are chained by programmatic dependent launch: everything before a class's scatter depends
// on no other class, so its blocks fill the SMs that the classes before it leave idle, and it waits
// for those classes only before it adds to `out`.  FP64 cached apply against plain launches: Q1 8^3
// 140 -> 30 us and Q2 16^3 368 -> 57 us (with the small blocks), Q2 64^3 2174 -> 2072 us (the
// classes' last waves).  The first launch of the chain waits for all earlier work of the stream as
// usual; each class waits for the one before it, so the last one ends after all.
template <typename T, typename KernelT>
nhmf_status run_colours(nhmf_ctx* c, KernelT kernel, OpArgs a, int NE, int threads, size_t smem, const T* src, T* out,
                        T value, cudaStream_t s, const char* what, int kind) {
  if (cudaError_t e = prepare(kernel, smem); e != cudaSuccess) return cuda_check(c, e, what);
  const long long M2 = (long long)c->g.M * c->g.M;
  const dim3 init_grid((unsigned)((M2 + 256 * kInitPer - 1) / (256 * kInitPer)), (unsigned)(3 * c->g.M));
  if (cudaError_t e = launch(k_init_rows<T>, init_grid, 256, 0, s, true, a.bc, c->g.M, src, out, value); e != cudaSuccess)
    return cuda_check(c, e, what);
  bool pdl = !c->profiling;  // the event below lies between the two launches
  nhmf_ctx::Rec rec{kind, 0, nullptr, nullptr};
  if (c->profiling) {
    cudaEventCreate(&rec.a);
    cudaEventCreate(&rec.b);
    cudaEventRecord(rec.a, s);
  }
  for (int k = 0; k < 8; ++k) {
    const Colour& col = c->g.colour[k];
    if (col.count == 0) continue;
    a.col = col;
    const int blocks = (col.count + NE - 1) / NE;
    if (cudaError_t e = launch(kernel, dim3((unsigned)blocks), threads, smem, s, pdl, a); e != cudaSuccess)
      return cuda_check(c, e, what);
    pdl = true;
    ++rec.launches;
  }
  if (c->profiling) {
    cudaEventRecord(rec.b, s);
    c->prof.push_back(rec);
  }
  return cuda_check(c, cudaGetLastError(), what);
}

// The element-local FP32 apply: `kernel` once over the class of all elements (NE per block),
// writing c->vloc, then k_gather_local<P> onto v with the Dirichlet rows (bc of `a`) and the
// update `g32`.
template <int P, typename KernelT>
nhmf_status run_local(nhmf_ctx* c, KernelT kernel, OpArgs a, int NE, int threads, size_t smem, const float* du,
                      float* v, const Gather32& g32, cudaStream_t s) {
  if (cudaError_t e = prepare(kernel, smem); e != cudaSuccess) return cuda_check(c, e, "apply");
  if (!c->vloc) return fail(c, NHMF_ERR_STATE, "apply: no element-local buffer (set_linearization first)");
  if (c->g.E > 0x7fffffffLL || (long long)c->g.M * c->g.M > 0x7fffffffLL)
    return fail(c, NHMF_ERR_ARG, "apply: the FP32 element-local path needs fewer than 2^31 elements");
  nhmf_ctx::Rec rec{NHMF_KIND_APPLY, 2, nullptr, nullptr};
  if (c->profiling) {
    cudaEventCreate(&rec.a);
    cudaEventCreate(&rec.b);
    cudaEventRecord(rec.a, s);
  }
  a.col = c->g.all;
  a.vloc = c->vloc;
  // both launches may start while the one before them drains (they wait for it before they read)
  cudaError_t e = launch(kernel, dim3((unsigned)((c->g.E + NE - 1) / NE)), threads, smem, s, true, a);
  if (e != cudaSuccess) return cuda_check(c, e, "apply");
  const dim3 gather_grid((unsigned)(((long long)c->g.M * c->g.M + 255) / 256), (unsigned)c->g.M);
  auto* gather = g32.mode == Gather32::kApply       ? k_gather_local<P, Gather32::kApply>
                 : g32.mode == Gather32::kResidual  ? k_gather_local<P, Gather32::kResidual>
                 : g32.mode == Gather32::kChebyshev ? k_gather_local<P, Gather32::kChebyshev>
                                                    : k_gather_local<P, Gather32::kPower>;
  e = launch(gather, gather_grid, 256, 0, s, true, (const float*)c->vloc, du, v, c->g.N, c->g.M, a.bc, g32);
  if (e != cudaSuccess) return cuda_check(c, e, "apply");
  if (c->profiling) {
    cudaEventRecord(rec.b, s);
    c->prof.push_back(rec);
  }
  return cuda_check(c, cudaGetLastError(), "apply");
}

// Small blocks where the normal ones would leave SMs idle (see Shape).
template <typename T, int NE>
bool small_blocks(const nhmf_ctx* c) {
  return c->g.E < (long long)NE * SmallRule<T>::per_sm * c->sms;
}

// The k_apply instance of one block shape, on all colour classes.
template <int P, typename T, int STRAT, int MODEL, bool SMALL>
nhmf_status apply_colours(nhmf_ctx* c, const OpArgs& a, size_t slots_per_item, cudaStream_t s) {
  using St = typename Store<T>::type;
  using Sh = Shape<P, T, STRAT, SMALL>;
  constexpr int n3 = (P + 1) * (P + 1) * (P + 1);
  const size_t smem = (kTabSlots + slots_per_item * Sh::NE * n3) * sizeof(T);
  return run_colours<St>(c, k_apply<P, T, STRAT, MODEL, SMALL>, a, Sh::NE, Sh::THREADS, smem,
                         static_cast<const St*>(a.du), static_cast<St*>(a.v), St(0), s, "apply", NHMF_KIND_APPLY);
}

template <int P, typename T, int STRAT>
nhmf_status apply_p(nhmf_ctx* c, const void* du, void* v, bool raw, const Gather32& g32, cudaStream_t s) {
  OpArgs a = base_args(c);
  if (raw) a.bc = NHMF_BC_NONE;  // unconstrained operator K: no masking, no identity rows
  a.u64 = c->u_at ? c->u_at : c->ubar;
  a.u32 = c->ubar32;
  a.du = du;
  a.v = v;
  a.cache = std::is_same<T, df64>::value ? (const void*)c->cachedf
            : (sizeof(T) == 8 ? (const void*)c->cache64 : (const void*)c->cache32);
  a.cachesp_in = c->cachesp;
  constexpr size_t per_item = STRAT == NHMF_ON_THE_FLY ? 15 : 12;  // spatial: as cached
  // the energy model is a compile-time parameter of the on-the-fly point code (a runtime
  // branch would charge the split model's registers to every model)
  constexpr int SPLIT = STRAT == NHMF_ON_THE_FLY ? NHMF_MODEL_SPLIT : NHMF_MODEL_COMPRESSIBLE;
  const bool split = STRAT == NHMF_ON_THE_FLY && c->prm.model == NHMF_MODEL_SPLIT;
  if constexpr (std::is_same<T, float>::value) {
    // FP32: one launch over all elements with element-local results, then the node gather
    // (which also writes the Dirichlet rows): no memset, no colour classes
    const float* du32 = static_cast<const float*>(du);
    float* v32 = static_cast<float*>(v);
    if constexpr (P <= kRegMaxP) {
      if (c->reg32) {
        // the compressible on-the-fly kernel's point values and slice kinematics (see k_apply_reg)
        constexpr size_t n3 = (P + 1) * (P + 1) * (P + 1), n2 = (P + 1) * (P + 1);
        const size_t kin_smem = (3 * n3 + 10 * n2) * kRegThreads * sizeof(float);
        if (split)
          return run_local<P>(c, k_apply_reg<P, STRAT, SPLIT>, a, kRegThreads, kRegThreads, 0, du32, v32, g32, s);
        return run_local<P>(c, k_apply_reg<P, STRAT, NHMF_MODEL_COMPRESSIBLE>, a, kRegThreads, kRegThreads,
                            STRAT == NHMF_ON_THE_FLY ? kin_smem : 0, du32, v32, g32, s);
      }
    }
    if constexpr (P >= 2) {
      using Sh = ColShape<P + 1>;
      constexpr size_t field = (size_t)Sh::NE * (P + 1) * (P + 1) * (P + 1) * sizeof(float);
      if (split)
        return run_local<P>(c, k_apply_col<P, STRAT, SPLIT>, a, Sh::NE, Sh::THREADS,
                            col_fields<P + 1, STRAT, SPLIT>() * field, du32, v32, g32, s);
      return run_local<P>(c, k_apply_col<P, STRAT, NHMF_MODEL_COMPRESSIBLE>, a, Sh::NE, Sh::THREADS,
                          col_fields<P + 1, STRAT, NHMF_MODEL_COMPRESSIBLE>() * field, du32, v32, g32, s);
    } else {
      return fail(c, NHMF_ERR_STATE, "apply: p = 1 without the register kernel");  // reg32 is always set there
    }
  } else {
    if (small_blocks<T, Shape<P, T, STRAT, false>::NE>(c))
      return split ? apply_colours<P, T, STRAT, SPLIT, true>(c, a, per_item, s)
                   : apply_colours<P, T, STRAT, NHMF_MODEL_COMPRESSIBLE, true>(c, a, per_item, s);
    return split ? apply_colours<P, T, STRAT, SPLIT, false>(c, a, per_item, s)
                 : apply_colours<P, T, STRAT, NHMF_MODEL_COMPRESSIBLE, false>(c, a, per_item, s);
  }
}

template <int P>
nhmf_status apply_dispatch_p(nhmf_ctx* c, int prec, int strat, const void* du, void* v, bool raw,
                             const Gather32& g32, cudaStream_t s) {
  if (prec == NHMF_DF64) {
    if (strat != NHMF_CACHED) return fail(c, NHMF_ERR_ARG, "df64 apply: cached strategy only");
    return apply_p<P, df64, NHMF_CACHED>(c, du, v, raw, g32, s);
  }
  if (prec == NHMF_FP64) {
    if (strat == NHMF_SPATIAL) return apply_p<P, double, NHMF_SPATIAL>(c, du, v, raw, g32, s);
    return strat == NHMF_CACHED ? apply_p<P, double, NHMF_CACHED>(c, du, v, raw, g32, s)
                                : apply_p<P, double, NHMF_ON_THE_FLY>(c, du, v, raw, g32, s);
  }
  return strat == NHMF_CACHED ? apply_p<P, float, NHMF_CACHED>(c, du, v, raw, g32, s)
                              : apply_p<P, float, NHMF_ON_THE_FLY>(c, du, v, raw, g32, s);
}

template <int P, bool SMALL, bool SPATIAL>
nhmf_status cache_shape(nhmf_ctx* c, const OpArgs& a, cudaStream_t s) {
  using Sh = Shape<P, double, NHMF_CACHED, SMALL>;
  constexpr int n3 = (P + 1) * (P + 1) * (P + 1);
  const size_t smem = (kTabSlots + 6 * (size_t)Sh::NE * n3) * sizeof(double);
  auto* kernel = k_cache<P, SMALL, SPATIAL>;
  if (cudaError_t e = prepare(kernel, smem); e != cudaSuccess) return cuda_check(c, e, "cache build");
  nhmf_ctx::Rec rec{NHMF_KIND_CACHE, 1, nullptr, nullptr};
  if (c->profiling) {
    cudaEventCreate(&rec.a);
    cudaEventCreate(&rec.b);
    cudaEventRecord(rec.a, s);
  }
  long long blocks = 0;
  for (int k = 0; k < 8; ++k) blocks += (c->g.colour[k].count + Sh::NE - 1) / Sh::NE;
  const cudaError_t e = launch(kernel, dim3((unsigned)blocks), Sh::THREADS, smem, s, false, a);
  if (c->profiling) {
    cudaEventRecord(rec.b, s);
    c->prof.push_back(rec);
  }
  return cuda_check(c, e, "cache build");
}

template <int P>
nhmf_status cache_p(nhmf_ctx* c, cudaStream_t s) {
  OpArgs a = base_args(c);
  a.u64 = c->ubar;
  a.cache64_out = c->cache64;
  a.cache32_out = c->cache32;
  a.cachedf_out = c->cachedf;
  a.cachesp_out = c->cachesp;
  const bool small = small_blocks<double, Shape<P, double, NHMF_CACHED, false>::NE>(c);
  if (c->cachesp) return small ? cache_shape<P, true, true>(c, a, s) : cache_shape<P, false, true>(c, a, s);
  return small ? cache_shape<P, true, false>(c, a, s) : cache_shape<P, false, false>(c, a, s);
}

template <int P, bool SMALL>
nhmf_status residual_shape(nhmf_ctx* c, const OpArgs& a, double* r, cudaStream_t s) {
  using Sh = Shape<P, double, 0, SMALL>;
  constexpr int n3 = (P + 1) * (P + 1) * (P + 1);
  const size_t smem = (kTabSlots + 12 * (size_t)Sh::NE * n3) * sizeof(double);
  return run_colours<double>(c, k_residual<P, SMALL>, a, Sh::NE, Sh::THREADS, smem, nullptr, r, 0.0, s, "residual",
                             NHMF_KIND_RESIDUAL);
}

template <int P>
nhmf_status residual_p(nhmf_ctx* c, const double* u, double* r, cudaStream_t s) {
  OpArgs a = base_args(c);
  a.u64 = u;
  a.v = r;
  return small_blocks<double, Shape<P, double, 0, false>::NE>(c) ? residual_shape<P, true>(c, a, r, s)
                                                         : residual_shape<P, false>(c, a, r, s);
}

template <int P, bool SMALL, bool CACHED>
nhmf_status diagonal_shape(nhmf_ctx* c, const OpArgs& a, double* d, cudaStream_t s) {
  using Sh = DiagCfg<P, SMALL>;
  constexpr int n3 = (P + 1) * (P + 1) * (P + 1);
  const size_t smem = (kTabSlots + kDiagFields * (size_t)Sh::NE * n3) * sizeof(double);
  return run_colours<double>(c, k_diagonal<P, SMALL, CACHED>, a, Sh::NE, Sh::THREADS, smem, nullptr, d, 1.0, s, "diagonal",
                             NHMF_KIND_DIAGONAL);
}

template <int P>
nhmf_status diagonal_p(nhmf_ctx* c, double* d, cudaStream_t s) {
  OpArgs a = base_args(c);
  a.u64 = c->ubar;
  a.v = d;
  // the FP64 cache, where it exists, holds the current linearisation point (set_linearization)
  a.cache = c->cache64;
  const bool small = small_blocks<double, DiagCfg<P, false>::NE>(c);
  if (c->cache64 && c->prm.model == NHMF_MODEL_COMPRESSIBLE)
    return small ? diagonal_shape<P, true, true>(c, a, d, s) : diagonal_shape<P, false, true>(c, a, d, s);
  return small ? diagonal_shape<P, true, false>(c, a, d, s) : diagonal_shape<P, false, false>(c, a, d, s);
}

}  // namespace

template <int P>
nhmf_status Operators<P>::apply(nhmf_ctx* c, int prec, int strat, const void* du, void* v, bool raw,
                                const Gather32& g32, cudaStream_t s) {
  return apply_dispatch_p<P>(c, prec, strat, du, v, raw, g32, s);
}
template <int P>
nhmf_status Operators<P>::cache(nhmf_ctx* c, cudaStream_t s) {
  return cache_p<P>(c, s);
}
template <int P>
nhmf_status Operators<P>::residual(nhmf_ctx* c, const double* u, double* r, cudaStream_t s) {
  return residual_p<P>(c, u, r, s);
}
template <int P>
nhmf_status Operators<P>::diagonal(nhmf_ctx* c, double* d, cudaStream_t s) {
  return diagonal_p<P>(c, d, s);
}

}  // namespace nhmf
