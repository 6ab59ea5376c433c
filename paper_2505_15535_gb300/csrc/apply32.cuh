// FP32 tangent apply for p >= 2 with planes and columns of an element in registers.
//
// A block takes NE consecutive elements.  Field f of the block lives in shared memory as [z][e][y][x].
//   gather   thread (e, x, y) copies its z column of du;
//   planes   thread (c, z, e) takes a nodal z-plane into registers and contracts x and y there:
//            t = Bx By u, tx = Dx By u, ty = Bx Dy u (B: values, D: derivatives of the nodal basis at
//            the Gauss points of a line) - three fields out of one;
//   columns  thread (e, x, y) takes the z columns of the nine fields, forms Grad du = (Bz tx, Bz
//            ty, Dz t) at the Gauss points of its column two at a time (points z and n - 1 - z
//            share their even and odd halves), runs the point code and adds the nine fluxes into
//            the nine transposed columns, all in registers;
//   planes   thread (c, z, e) contracts the three transposed fields with Bx^T, Dx^T, By^T, Dy^T and
//            writes the element's nodal plane to vloc (eight elements: whole 32-byte sectors).
// What bounded the line-pass form (one thread per line and pass, every value through shared memory
// between passes) was the shared-memory pipe, 102 words per point; this form moves 42, and pays for
// it with 63 instead of 43 operations per point and field set in z.  Every contraction is in
// even-odd form (the rules of M[n-1-r][n-1-m] = +-M[r][m]), coefficients are constant-bank operands.
#pragma once
#include "sumfact.cuh"

namespace nhmf {
namespace {

// Elements and threads of a block, and blocks an SM.  Five at Q3 for both models: four, with which the
// split model's on-the-fly instance does not spill (88 bytes at five), measure the same (on the fly,
// five / four: 47^3 172.1 / 171.4 us, split 189.8 / 189.4; 36^3 74.9 / 74.6, split 86.0 / 84.4).
template <int n> struct ColShape;
template <> struct ColShape<3> { static constexpr int NE = 16, THREADS = 160, BLOCKS = 4; };
template <> struct ColShape<4> { static constexpr int NE = 8, THREADS = 128, BLOCKS = 5; };
template <> struct ColShape<5> { static constexpr int NE = 8, THREADS = 224, BLOCKS = 2; };

template <int n>
__device__ __forceinline__ void eo_split(const float (&x)[n], float (&e)[n / 2], float (&o)[n / 2]) {
#pragma unroll
  for (int m = 0; m < n / 2; ++m) {
    e[m] = x[m] + x[n - 1 - m];
    o[m] = x[m] - x[n - 1 - m];
  }
}

// Rows r and n-1-r of a matrix at once from the halves e, o and the centre value xh of a line.
//   symmetric: y_r = E + O, y_r' = E - O, E = S e (+ C xh), O = A o
//   anti-symmetric: y_r = O + E, y_r' = O - E
// kCentre says whether the centre column enters rows off the centre (it does not for B^T).
template <int n, bool ANTI, bool kCentre>
__device__ __forceinline__ void eo_pair(const EoTab& T, int r, const float (&e)[n / 2], const float (&o)[n / 2],
                                        float xh, float& yr, float& ys) {
  constexpr int h = n / 2;
  float E = T.S[r][0] * e[0];
#pragma unroll
  for (int m = 1; m < h; ++m) E = fmaf(T.S[r][m], e[m], E);
  if (n % 2 == 1 && kCentre) E = fmaf(T.C[r], xh, E);
  float p = E, q = ANTI ? -E : E;
#pragma unroll
  for (int m = 0; m < h; ++m) {
    p = fmaf(T.A[r][m], o[m], p);
    q = fmaf(ANTI ? T.A[r][m] : -T.A[r][m], o[m], q);
  }
  yr = p;
  ys = q;
}

// The centre row (odd n): B's is the centre value itself, an anti-symmetric matrix's A o, and
// B^T's mid . e + ch xh.
template <int n>
__device__ __forceinline__ float eo_mid(const EoTab& T, const float (&v)[n / 2]) {
  float s = T.mid[0] * v[0];
#pragma unroll
  for (int m = 1; m < n / 2; ++m) s = fmaf(T.mid[m], v[m], s);
  return s;
}

// Whole lines: y = B x, y = D x (also D^T), y = B^T x.
template <int n>
__device__ __forceinline__ void line_B(const EoTab& T, const float (&e)[n / 2], const float (&o)[n / 2], float xh,
                                       float (&y)[n]) {
#pragma unroll
  for (int r = 0; r < n / 2; ++r) eo_pair<n, false, true>(T, r, e, o, xh, y[r], y[n - 1 - r]);
  if constexpr (n % 2 == 1) y[n / 2] = xh;
}
template <int n>
__device__ __forceinline__ void line_D(const EoTab& T, const float (&e)[n / 2], const float (&o)[n / 2], float xh,
                                       float (&y)[n]) {
#pragma unroll
  for (int r = 0; r < n / 2; ++r) eo_pair<n, true, true>(T, r, e, o, xh, y[r], y[n - 1 - r]);
  if constexpr (n % 2 == 1) y[n / 2] = eo_mid<n>(T, o);
}
template <int n>
__device__ __forceinline__ void line_BT(const EoTab& T, const float (&e)[n / 2], const float (&o)[n / 2], float xh,
                                        float (&y)[n]) {
#pragma unroll
  for (int r = 0; r < n / 2; ++r) eo_pair<n, false, false>(T, r, e, o, xh, y[r], y[n - 1 - r]);
  if constexpr (n % 2 == 1) y[n / 2] = fmaf(T.ch, xh, eo_mid<n>(T, e));
}

// Offset of (e, y, x) in a z-plane of a field.  n = 4: rows of four floats move as one 16-byte access,
// and the rows of element e are permuted by e so that eight elements' rows cover all banks.
template <int n>
__device__ __forceinline__ int plane_pos(int e, int y) {
  return n == 4 ? e * 16 + ((y ^ ((e >> 1) & 3)) << 2) : e * n * n + y * n;
}
template <int n>
__device__ __forceinline__ void load_row(const float* p, float (&x)[n]) {
  if constexpr (n == 4) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    x[0] = v.x, x[1] = v.y, x[2] = v.z, x[3] = v.w;
  } else {
#pragma unroll
    for (int i = 0; i < n; ++i) x[i] = p[i];
  }
}
template <int n>
__device__ __forceinline__ void store_row(float* p, const float (&x)[n]) {
  if constexpr (n == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
  } else {
#pragma unroll
    for (int i = 0; i < n; ++i) p[i] = x[i];
  }
}

// Forward plane phase in place: field c's nodal plane z of element e becomes t in field c, tx in
// field 3 + c and ty in field 6 + c.
template <int n, int NE>
__device__ __forceinline__ void plane_forward(const OpArgs& a, float* F, int tid) {
  constexpr int n2 = n * n, FS = NE * n2 * n, h = n / 2;
  if (tid >= 3 * n * NE) return;
  const int e = tid % NE, cz = tid / NE, c = cz / n, z = cz - c * n;
  float* f = F + c * FS + z * NE * n2;
  float by[n][n], dy[n][n];  // [y][x]
#pragma unroll
  for (int y = 0; y < n; ++y) load_row<n>(f + plane_pos<n>(e, y), by[y]);
#pragma unroll
  for (int x = 0; x < n; ++x) {
    float u[n], b[n], d[n], eh[h], oh[h];
#pragma unroll
    for (int y = 0; y < n; ++y) u[y] = by[y][x];
    eo_split<n>(u, eh, oh);
    line_B<n>(a.cB, eh, oh, u[h], b);
    line_D<n>(a.cD, eh, oh, u[h], d);
#pragma unroll
    for (int y = 0; y < n; ++y) by[y][x] = b[y], dy[y][x] = d[y];
  }
#pragma unroll
  for (int y = 0; y < n; ++y) {
    float v[n], eh[h], oh[h];
    float* row = f + plane_pos<n>(e, y);
    eo_split<n>(by[y], eh, oh);
    line_B<n>(a.cB, eh, oh, by[y][h], v);
    store_row<n>(row, v);
    line_D<n>(a.cD, eh, oh, by[y][h], v);
    store_row<n>(row + 3 * FS, v);
    eo_split<n>(dy[y], eh, oh);
    line_B<n>(a.cB, eh, oh, dy[y][h], v);
    store_row<n>(row + 6 * FS, v);
  }
}

// The column's nine fields at points r and n-1-r (pair r < n/2), or at the centre (r = n/2, odd n;
// gs is not written): g[3c] = Bz tx, g[3c+1] = Bz ty, g[3c+2] = Dz t, from the columns in halves.
template <int n>
struct Columns {
  static constexpr int h = n / 2;
  float e[9][h], o[9][h], xh[9];  // field 3 k + c: k = 0 t, 1 tx, 2 ty
  __device__ __forceinline__ void load(const float* col, int fs, int zs) {
#pragma unroll
    for (int f = 0; f < 9; ++f) {
#pragma unroll
      for (int m = 0; m < h; ++m) {
        const float lo = col[f * fs + m * zs], hi = col[f * fs + (n - 1 - m) * zs];
        e[f][m] = lo + hi;
        o[f][m] = lo - hi;
      }
      xh[f] = n % 2 == 1 ? col[f * fs + h * zs] : 0.f;
    }
  }
  __device__ __forceinline__ void gradient(const OpArgs& a, int r, float (&g)[9], float (&gs)[9]) const {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (n % 2 == 1 && r == h) {
        g[3 * c] = xh[3 + c];
        g[3 * c + 1] = xh[6 + c];
        g[3 * c + 2] = eo_mid<n>(a.cD, o[c]);
      } else {
        eo_pair<n, false, true>(a.cB, r, e[3 + c], o[3 + c], xh[3 + c], g[3 * c], gs[3 * c]);
        eo_pair<n, false, true>(a.cB, r, e[6 + c], o[6 + c], xh[6 + c], g[3 * c + 1], gs[3 * c + 1]);
        eo_pair<n, true, true>(a.cD, r, e[c], o[c], xh[c], g[3 * c + 2], gs[3 * c + 2]);
      }
    }
  }
  // The transposed columns, kept as even and odd parts: zero; add the fluxes of a pair or of the
  // centre; write the columns back.
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int f = 0; f < 9; ++f) {
#pragma unroll
      for (int m = 0; m < h; ++m) e[f][m] = o[f][m] = 0.f;
      xh[f] = 0.f;
    }
  }
  __device__ __forceinline__ void add(const OpArgs& a, int r, const float (&g)[9], const float (&gs)[9]) {
#pragma unroll
    for (int f = 0; f < 9; ++f) {
      const int c = f % 3, k = f / 3;                // g index of field f: t takes gz, tx gx, ty gy
      const int gi = 3 * c + (k == 0 ? 2 : k - 1);
      const EoTab& T = k == 0 ? a.cDTz : a.cBTz;
      if (n % 2 == 1 && r == h) {
        if (k == 0) {
#pragma unroll
          for (int m = 0; m < h; ++m) e[f][m] = fmaf(T.C[m], g[gi], e[f][m]);
        } else {
          xh[f] = fmaf(T.ch, g[gi], xh[f]);
        }
      } else {
        const float ge = g[gi] + gs[gi], go = g[gi] - gs[gi];
#pragma unroll
        for (int m = 0; m < h; ++m) {
          e[f][m] = fmaf(T.S[m][r], ge, e[f][m]);
          o[f][m] = fmaf(T.A[m][r], go, o[f][m]);
        }
        if (n % 2 == 1) xh[f] = fmaf(T.mid[r], k == 0 ? go : ge, xh[f]);
      }
    }
  }
  __device__ __forceinline__ void store(float* col, int fs, int zs) const {
#pragma unroll
    for (int f = 0; f < 9; ++f) {
#pragma unroll
      for (int m = 0; m < h; ++m) {
        col[f * fs + m * zs] = e[f][m] + o[f][m];
        col[f * fs + (n - 1 - m) * zs] = f < 3 ? o[f][m] - e[f][m] : e[f][m] - o[f][m];
      }
      if (n % 2 == 1) col[f * fs + h * zs] = xh[f];
    }
  }
};

// From this J on 1 / J^2 leaves FP32's range before F^-1 does.
constexpr float kLargeJ32 = 1.152921504606847e18f;  // 2^60

// On the fly, per point: A = J F^-1 and the two coefficients of linearised_stress_unit (compressible),
// or Grad u (split model).
template <int MODEL> struct PointState { static constexpr int K = MODEL == NHMF_MODEL_SPLIT ? 9 : 11; };

template <int n, int STRAT, int MODEL>
constexpr int col_fields() {
  return 9 + (STRAT == NHMF_ON_THE_FLY ? PointState<MODEL>::K : 0);
}

template <int P, int STRAT, int MODEL>
__global__ void __launch_bounds__(ColShape<P + 1>::THREADS, ColShape<P + 1>::BLOCKS) k_apply_col(const OpArgs a) {
  constexpr int n = P + 1, n2 = n * n, n3 = n2 * n, h = n / 2, NE = ColShape<n>::NE, ZS = NE * n2, FS = ZS * n;
  static_assert(kTile % NE == 0, "a block's elements lie in one tile of vloc");
  extern __shared__ __align__(16) float F[];  // [9][n][NE][n][n], then the point state
  const int tid = threadIdx.x;
  pdl_launch_next();
  const long long e0 = (long long)blockIdx.x * NE;
  const int nvalid = (int)min((long long)NE, a.col.count - e0);

  // this thread's column: element ce, (x, y) of the column's nodes and of its Gauss points
  // (an absent element computes the block's first one again, and stores nothing)
  const bool column = tid < ZS;
  const int ce = tid / n2, cxy = tid - ce * n2, cy = cxy / n, cx = cxy - cy * n;
  float* col = F + plane_pos<n>(ce, cy) + cx;
  const long long el = e0 + (ce < nvalid ? ce : 0), M2 = (long long)a.M * a.M;  // natural order
  const unsigned N = (unsigned)a.N, eu = (unsigned)el;                          // fewer than 2^31 elements
  const unsigned ex = eu % N, eyz = eu / N, ey = eyz % N, ez = eyz / N;
  const int gi = P * ex + cx, gk = P * ez;
  const long long node = gi + (long long)a.M * (P * ey + cy + (long long)a.M * gk);
  const float fac = a.factor ? float(a.factor[el]) : 1.f;
  bool bad = false;
  pdl_wait();

  if constexpr (STRAT == NHMF_ON_THE_FLY) {
    if (column) {
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int z = 0; z < n; ++z) col[c * FS + z * ZS] = a.u32[c * a.M3 + node + z * M2];
    }
    __syncthreads();
    plane_forward<n, NE>(a, F, tid);
    __syncthreads();
    if (column) {
      Columns<n> u;
      u.load(col, FS, ZS);
      float* st = F + 9 * FS + tid;
      float largest = 0.f;  // J of the column
#pragma unroll
      for (int r = 0; r <= (n - 1) / 2; ++r) {
        float H[2][9];
        u.gradient(a, r, H[0], H[1]);
#pragma unroll
        for (int s = 0; s < ((n % 2 == 1 && r == h) ? 1 : 2); ++s) {
          const int z = s == 0 ? r : n - 1 - r;
#pragma unroll
          for (int k = 0; k < 9; ++k) H[s][k] *= a.invhf;
          if constexpr (MODEL == NHMF_MODEL_SPLIT) {
#pragma unroll
            for (int k = 0; k < 9; ++k) st[k * FS + z * ZS] = H[s][k];
          } else {
            const Kinematics<float> kin(H[s]);
            bad |= !(kin.Jm1 > -1.f);
            largest = fmaxf(largest, kin.Jm1);
            const float i2 = kin.invJ * kin.invJ;
#pragma unroll
            for (int k = 0; k < 9; ++k) st[k * FS + z * ZS] = kin.A[k];
            st[9 * FS + z * ZS] = fmaf(-a.r2muf, kin.lnJ, 1.f) * i2;
            st[10 * FS + z * ZS] = a.r2muf * i2;
          }
        }
      }
      // the column's points again, with F^-1 itself in the place of A (kept out of the loop above,
      // where a test per point cost 1.5 %: Q3 47^3 171 -> 173 us)
      if (MODEL == NHMF_MODEL_COMPRESSIBLE && largest >= kLargeJ32) {
#pragma unroll 1
        for (int z = 0; z < n; ++z) {
          float H[9] = {};
#pragma unroll 1
          for (int m = 0; m < n; ++m) {
            const float b = a.Bf[z * n + m], d = float(a.D[z * n + m]);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              H[3 * c] = fmaf(b, col[(3 + c) * FS + m * ZS], H[3 * c]);
              H[3 * c + 1] = fmaf(b, col[(6 + c) * FS + m * ZS], H[3 * c + 1]);
              H[3 * c + 2] = fmaf(d, col[c * FS + m * ZS], H[3 * c + 2]);
            }
          }
#pragma unroll
          for (int k = 0; k < 9; ++k) H[k] *= a.invhf;
          const Kinematics<float> kin(H);
#pragma unroll
          for (int k = 0; k < 9; ++k) st[k * FS + z * ZS] = kin.A[k] * kin.invJ;
          st[9 * FS + z * ZS] = fmaf(-a.r2muf, kin.lnJ, 1.f);
          st[10 * FS + z * ZS] = a.r2muf;
        }
      }
    }
    __syncthreads();
  }

  // The point data of a pair of points, loaded ahead of its use: the first pair's before the plane
  // phase, the next one's while the fluxes of the pair before it are added.
  constexpr int NK = STRAT == NHMF_CACHED ? 10 : PointState<MODEL>::K;
  float K[2][NK];
  const float* st = STRAT == NHMF_CACHED ? static_cast<const float*>(a.cache) + el * n3 + cxy  // [10][E n^3]
                                         : F + 9 * FS + tid;
  const unsigned long long pol = l2_evict_first();
  auto load_points = [&](int r) {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if (s == 1 && n % 2 == 1 && r == h) continue;
      const int z = s == 0 ? r : n - 1 - r;
#pragma unroll
      for (int k = 0; k < NK; ++k) {
        if constexpr (STRAT == NHMF_CACHED)
          K[s][k] = ld_policy_ordered(st + k * a.nq + z * n2, pol);
        else
          K[s][k] = st[k * FS + z * ZS];
      }
    }
  };
  if (column) {
    // only the first and the last node of a column can be constrained on their own (compression)
    const bool on = a.bc != NHMF_BC_CLAMP_X0 || gi != 0, bottom = a.bc == NHMF_BC_COMPRESSION && gk == 0,
               top = a.bc == NHMF_BC_COMPRESSION && gk + P == a.M - 1;
    const float* du = static_cast<const float*>(a.du) + node;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int z = 0; z < n; ++z) {
        float val = fac * du[c * a.M3 + z * M2];
        if (z == 0) val = on && !bottom ? val : 0.f;
        else if (z == n - 1 && c == 2) val = on && !top ? val : 0.f;
        else val = on ? val : 0.f;
        col[c * FS + z * ZS] = val;
      }
    if constexpr (STRAT == NHMF_CACHED) load_points(0);
  }
  __syncthreads();
  plane_forward<n, NE>(a, F, tid);
  __syncthreads();

  if (column) {
    Columns<n> d, v;
    d.load(col, FS, ZS);
    v.zero();
    if constexpr (STRAT != NHMF_CACHED) load_points(0);
#pragma unroll
    for (int r = 0; r <= (n - 1) / 2; ++r) {
      float g[2][9];
      d.gradient(a, r, g[0], g[1]);
#pragma unroll
      for (int s = 0; s < ((n % 2 == 1 && r == h) ? 1 : 2); ++s) {
        float dH[9], A[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          dH[k] = g[s][k];
          A[k] = K[s][k];
        }
        if constexpr (STRAT == NHMF_CACHED) {
          linearised_stress_unit(A, K[s][9], dH, a.r2muf, g[s]);
        } else if constexpr (MODEL == NHMF_MODEL_SPLIT) {
          const Kinematics<float> kin(A);  // A holds Grad u
          bad |= !(kin.Jm1 > -1.f);
          float Fd[9], Fi[9];
#pragma unroll
          for (int k = 0; k < 9; ++k) {
            Fd[k] = (k % 4 == 0 ? 1.f : 0.f) + A[k];
            Fi[k] = kin.A[k] * kin.invJ;
          }
          split_stress_dP(Fd, Fi, kin.lnJ, kin.Jm1, dH, float(a.mu), float(a.lam), float(1.0 / a.mu), g[s]);
        } else {
          linearised_stress_unit(A, K[s][9], K[s][10], dH, g[s]);
        }
      }
      if (r < (n - 1) / 2) load_points(r + 1);
      v.add(a, r, g[0], g[1]);
    }
    v.store(col, FS, ZS);
  }
  if (bad) atomicOr(a.status, kStatusNonPosJ);
  __syncthreads();

  // transposed planes: a1 = Bx^T t + Dx^T tx, a2 = Bx^T ty per row, then By^T a1 + Dy^T a2 per column
  if (tid < 3 * n * NE) {
    const int e = tid % NE, cz = tid / NE, c = cz / n, z = cz - c * n;
    const float* f = F + c * FS + z * ZS;
    float a1[n][n], a2[n][n];
#pragma unroll
    for (int y = 0; y < n; ++y) {
      float x[n], y1[n], eh[h], oh[h];
      const float* row = f + plane_pos<n>(e, y);
      load_row<n>(row, x);
      eo_split<n>(x, eh, oh);
      line_BT<n>(a.cBT, eh, oh, x[h], a1[y]);
      load_row<n>(row + 3 * FS, x);
      eo_split<n>(x, eh, oh);
      line_D<n>(a.cDT, eh, oh, x[h], y1);
#pragma unroll
      for (int i = 0; i < n; ++i) a1[y][i] += y1[i];
      load_row<n>(row + 6 * FS, x);
      eo_split<n>(x, eh, oh);
      line_BT<n>(a.cBT, eh, oh, x[h], a2[y]);
    }
    if (e < nvalid) {
      const long long slot = e0 + e;
      float* out = a.vloc + ((slot / kTile) * 3 * n3 + c * n3 + z * n2) * kTile + slot % kTile;
      const unsigned long long keep_pol = l2_evict_last();  // read back by the gather that follows
#pragma unroll
      for (int x = 0; x < n; ++x) {
        float u[n], y1[n], y2[n], eh[h], oh[h];
#pragma unroll
        for (int y = 0; y < n; ++y) u[y] = a1[y][x];
        eo_split<n>(u, eh, oh);
        line_BT<n>(a.cBT, eh, oh, u[h], y1);
#pragma unroll
        for (int y = 0; y < n; ++y) u[y] = a2[y][x];
        eo_split<n>(u, eh, oh);
        line_D<n>(a.cDT, eh, oh, u[h], y2);
#pragma unroll
        for (int y = 0; y < n; ++y) st_policy(out + (y * n + x) * kTile, y1[y] + y2[y], keep_pol);
      }
    }
  }
}

}  // namespace
}  // namespace nhmf
