// The coarsest multigrid level as an explicit matrix and its Jacobi-CG solve in one launch.
//
// The coarsest level is a Q1 mesh of 2^3 elements (81 DoFs) for every mesh that halves down to
// it, of an odd N0^3 otherwise.  Up to kCoarseMaxN the operator is assembled once per
// linearisation as rows of 27 neighbour nodes x 3 components, and one thread-block cluster runs
// the whole conjugate-gradient solve on it: the vectors stay in shared memory, the scalars in
// registers, a matrix row is read by four lanes, and the blocks of the cluster exchange the search
// direction and the partial sums through distributed shared memory.  The host neither launches
// nor reads anything per iteration.
//
// What bounds it: latency.  An iteration is an 81-term row product, two FP64 reductions and two
// divisions in one warp (about 45 dependent FP64 operations; rows are spread over blocks at about 200
// per block) and two barriers of the block or three of the cluster: 3.5 us on 81 DoFs in FP32, against
// 70 us for the same iteration as six launches.  The sums are FP64 also in the FP32 solve: as pairs of FP32 numbers they
// took 1.4 us less an iteration (linear solve Q4 16^3 77.3 ms against 85.4), but had four bits fewer
// and FP32's exponent range, which the squares of a stiff material's system leave.
#include <algorithm>
#include <cooperative_groups.h>

#include "gmg.h"
#include "sumfact.cuh"

namespace nhmf {
namespace {

namespace cg = cooperative_groups;

constexpr int kRow = 81;             // entries of a matrix row: 27 neighbours x 3 components
constexpr int kCgThreads = 512;
constexpr int kLanes = 4;            // lanes per row
constexpr size_t kCgSmemMax = 220 * 1024;  // most dynamic shared memory of a block

struct ElemArgs {
  int N, model;
  double h, mu, lam;
  double B[4], D[4], w[2];           // Q1 tables, D per unit reference length
  const double* u;                   // [3][(N+1)^3]
  const double* factor;              // [N^3] or null
  double* Ke;                        // [N^3][24][24], index 3 a + c
};

// Element matrices of the Q1 tangent at u: K[3a+c][3b+k] = sum_q w_q h^3 f_e
//   (alpha delta_ck ga.gb + beta (sa_c tb_k + ta_c sb_k) + gamma ta_c tb_k + delta tb_c ta_k),
// g the basis gradients, t = F^-T g, s = F g: the linearised stress of either model
// (linearised_stress, split_stress_dP) contracted with the two basis gradients.  One block per
// element: 64 threads are (node, point) pairs, then (a, b) node pairs.
__global__ void __launch_bounds__(64) k_coarse_elements(const ElemArgs a) {
  __shared__ double g[8][8][3], t[8][8][3], s[8][8][3], F[8][9], Fi[8][9], co[8][4];  // [point][node]
  const int e = blockIdx.x, N = a.N, M = N + 1;
  const int ex = e % N, ey = (e / N) % N, ez = e / (N * N);
  const int q = threadIdx.x >> 3, nd = threadIdx.x & 7;
  const int qx = q & 1, qy = (q >> 1) & 1, qz = q >> 2, ax = nd & 1, ay = (nd >> 1) & 1, az = nd >> 2;
  g[q][nd][0] = a.D[qx * 2 + ax] * a.B[qy * 2 + ay] * a.B[qz * 2 + az] / a.h;
  g[q][nd][1] = a.B[qx * 2 + ax] * a.D[qy * 2 + ay] * a.B[qz * 2 + az] / a.h;
  g[q][nd][2] = a.B[qx * 2 + ax] * a.B[qy * 2 + ay] * a.D[qz * 2 + az] / a.h;
  __syncthreads();
  if (threadIdx.x < 8) {
    const int p = threadIdx.x;
    double H[9] = {};
    for (int b = 0; b < 8; ++b) {
      const long long node = (ex + (b & 1)) + (long long)M * ((ey + ((b >> 1) & 1)) + (long long)M * (ez + (b >> 2)));
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double ub = a.u[c * (long long)M * M * M + node];
#pragma unroll
        for (int d = 0; d < 3; ++d) H[3 * c + d] = fma(ub, g[p][b][d], H[3 * c + d]);
      }
    }
    double Fv[9], Fiv[9], lnJ;
    const double Jm1 = kinematics(H, Fiv, lnJ);
    double I1 = 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      Fv[k] = (k % 4 == 0 ? 1.0 : 0.0) + H[k];
      I1 = fma(Fv[k], Fv[k], I1);
      F[p][k] = Fv[k];
      Fi[p][k] = Fiv[k];
    }
    const double wt = a.w[p & 1] * a.w[(p >> 1) & 1] * a.w[p >> 2] * a.h * a.h * a.h * (a.factor ? a.factor[e] : 1.0);
    if (a.model == NHMF_MODEL_SPLIT) {
      const double mua = a.mu * exp(-2.0 / 3.0 * lnJ), J = 1.0 + Jm1;
      co[p][0] = wt * mua;
      co[p][1] = -2.0 / 3.0 * wt * mua;
      co[p][2] = wt * (2.0 / 9.0 * mua * I1 + a.lam * J * J);
      co[p][3] = wt * (mua * I1 / 3.0 - 0.5 * a.lam * (J * J - 1.0));
    } else {
      co[p][0] = wt * a.mu;
      co[p][1] = 0.0;
      co[p][2] = wt * 2.0 * a.lam;
      co[p][3] = wt * (a.mu - 2.0 * a.lam * lnJ);
    }
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    double tv = 0.0, sv = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      tv = fma(Fi[q][3 * d + c], g[q][nd][d], tv);
      sv = fma(F[q][3 * c + d], g[q][nd][d], sv);
    }
    t[q][nd][c] = tv;
    s[q][nd][c] = sv;
  }
  __syncthreads();
  const int A = threadIdx.x >> 3, b = threadIdx.x & 7;
  double K[9] = {};
  for (int p = 0; p < 8; ++p) {
    double gg = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) gg = fma(g[p][A][d], g[p][b][d], gg);
    const double c0 = co[p][0] * gg, c1 = co[p][1], c2 = co[p][2], c3 = co[p][3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double ta = t[p][A][c], tb = t[p][b][k];
        double v = fma(c2 * ta, tb, K[3 * c + k]);
        v = fma(c3 * t[p][b][c], t[p][A][k], v);
        if (a.model == NHMF_MODEL_SPLIT) v = fma(c1, fma(s[p][A][c], tb, ta * s[p][b][k]), v);
        K[3 * c + k] = c == k ? v + c0 : v;
      }
  }
  double* out = a.Ke + (long long)e * 576;
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int k = 0; k < 3; ++k) out[(3 * A + c) * 24 + 3 * b + k] = K[3 * c + k];
}

// Rows of the constrained operator P_f K P_f + P_D from the element matrices, in the solve's layout
// [block][81 entries][Rpad rows]: entry 3 nb + k of row (c, node) is the coupling to component
// k of neighbour nb = (dx + 1) + 3 (dy + 1) + 9 (dz + 1); 0 outside the mesh.  An entry sums its
// elements in increasing order.
__global__ void k_coarse_rows(const double* __restrict__ Ke, int N, int bc, int R, int Rpad, int blocks,
                              double* __restrict__ A64, float* __restrict__ A32) {
  const int M = N + 1, M3 = M * M * M, n = 3 * M3;
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= blocks * kRow * Rpad) return;
  const int lr = id % Rpad, j = (id / Rpad) % kRow, r = (id / (Rpad * kRow)) * R + lr;
  double v = 0.0;
  if (lr < R && r < n) {
    const int c = r / M3, node = r % M3, x = node % M, y = (node / M) % M, z = node / (M * M);
    const int nb = j / 3, k = j % 3, dx = nb % 3 - 1, dy = (nb / 3) % 3 - 1, dz = nb / 9 - 1;
    const int X = x + dx, Y = y + dy, Z = z + dz;
    if (is_constrained(bc, c, x, z, M)) {
      v = (nb == 13 && k == c) ? 1.0 : 0.0;
    } else if (X >= 0 && X < M && Y >= 0 && Y < M && Z >= 0 && Z < M && !is_constrained(bc, k, X, Z, M)) {
      for (int ez = max(max(z, Z) - 1, 0); ez <= min(min(z, Z), N - 1); ++ez)
        for (int ey = max(max(y, Y) - 1, 0); ey <= min(min(y, Y), N - 1); ++ey)
          for (int ex = max(max(x, X) - 1, 0); ex <= min(min(x, X), N - 1); ++ex) {
            const int a = (x - ex) + 2 * ((y - ey) + 2 * (z - ez)), b = (X - ex) + 2 * ((Y - ey) + 2 * (Z - ez));
            v += Ke[(long long)(ex + N * (ey + N * ez)) * 576 + (3 * a + c) * 24 + 3 * b + k];
          }
    }
  }
  A64[id] = v;
  A32[id] = float(v);
}

template <typename T>
struct CgArgs {
  const T *A, *b, *dinv;
  T* x;
  int n, M, R, Rpad, in_smem;        // DoFs, nodes per direction, rows per block and their padding
  double rtol;
  int maxit, check;
  unsigned long long* words;         // [0] += iterations, [1] |= status flags
};

// x / y rounded to T, the step lengths from the FP64 sums.  In FP32 by the reciprocal (two units in the
// last of 53 bits before the rounding to 24) where it is in range: half the latency of a division.
template <typename T>
__device__ __forceinline__ T quotient(double x, double y) {
  if constexpr (sizeof(T) == 4) {
    const double m = fabs(y);
    if (m > 0x1p-1000 && m < 0x1p1000) return T(x * fast_rcp(y));
  }
  return T(x / y);
}

// Jacobi-CG from x = 0 to ||r|| <= rtol ||b||, tested every `check` iterations as pcg() does;
// p.q <= 0 or a non-finite residual is recorded in the status word and ends the solve.  One
// cluster; block `rank` owns rows [rank R, rank R + R).  All warps of a block form q = A p; warp 0
// alone does the vector updates, the sums and the scalars, so that a reduction is five shuffles
// and the divisions are issued once.
template <typename T>
__global__ void __launch_bounds__(kCgThreads) k_coarse_cg(const CgArgs<T> a) {
  extern __shared__ __align__(16) unsigned char sm[];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), nblk = (int)cl.num_blocks(), tid = threadIdx.x, nthr = blockDim.x;
  const int M = a.M, M3 = M * M * M, pad = M * M + M + 1, R = a.R, Rpad = a.Rpad;
  const int row0 = rank * R, rows = max(0, min(R, a.n - row0));
  double* part = reinterpret_cast<double*>(sm);      // [2][16][2] sums of the cluster's blocks, double buffered
  int* stop = reinterpret_cast<int*>(part + 64);     // [1] (+ 1)
  int* off = stop + 2;                               // [81] (+ 1)
  T* p = reinterpret_cast<T*>(off + 82) + pad;       // [n], `pad` zeros on either side
  T* q = p + a.n + pad;                              // this block's rows
  T *r = q + R, *x = r + R, *di = x + R;
  T* As = di + R;                                    // [81][Rpad] if it fits
  const T* Ag = a.A + (size_t)rank * kRow * Rpad;
  const T* A = a.in_smem ? As : Ag;
  for (int j = tid; j < kRow; j += nthr) {
    const int nb = j / 3;
    off[j] = (j % 3) * M3 + (nb % 3 - 1) + M * ((nb / 3) % 3 - 1 + M * (nb / 9 - 1));
  }
  for (int i = tid; i < pad; i += nthr) p[i - pad] = p[a.n + i] = T(0);
  if (a.in_smem)
    for (int i = tid; i < kRow * Rpad; i += nthr) As[i] = Ag[i];
  if (tid == 0) *stop = 0;

  auto barrier = [&]() {  // the cluster's blocks have met, and see one another's shared-memory writes
    if (nblk == 1)
      __syncthreads();
    else
      cl.sync();
  };
  int buf = 0;
  // Sums of warp 0's two values over the cluster, in a fixed order, in warp 0 of every block; with
  // more than one block every thread has to call it.
  auto sum2 = [&](double& v0, double& v1) {
    if (tid < 32) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, o);
        v1 += __shfl_xor_sync(0xffffffffu, v1, o);
      }
      if (nblk > 1 && tid < nblk) {
        double* dst = cl.map_shared_rank(part, tid) + 32 * buf + 2 * rank;
        dst[0] = v0;
        dst[1] = v1;
      }
    }
    if (nblk == 1) return;
    cl.sync();
    if (tid < 32) {
      v0 = tid < nblk ? part[32 * buf + 2 * tid] : 0.0;
      v1 = tid < nblk ? part[32 * buf + 2 * tid + 1] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, o);
        v1 += __shfl_xor_sync(0xffffffffu, v1, o);
      }
    }
    buf ^= 1;
  };
  auto sum1 = [&](double& v) {
    if (nblk > 1) {
      double unused = 0.0;
      sum2(v, unused);
    } else if (tid < 32) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    }
  };
  // p over the whole cluster: own row i gets v
  auto set_p = [&](int i, T v) {
    for (int k = 0; k < nblk; ++k) (nblk == 1 ? p : cl.map_shared_rank(p, k))[row0 + i] = v;
  };
  barrier();  // every block's arrays exist and are initialised
  double v0 = 0.0, v1 = 0.0;
  if (tid < 32)
    for (int i = tid; i < rows; i += 32) {
      const T bi = a.b[row0 + i], d = a.dinv[row0 + i], zi = d * bi;
      x[i] = T(0);
      r[i] = bi;
      di[i] = d;
      v0 = fma(double(bi), double(zi), v0);
      v1 = fma(double(bi), double(bi), v1);
      set_p(i, zi);
    }
  sum2(v0, v1);
  double rz = v0;
  const double bn = sqrt(v1);
  unsigned flag = isfinite(v1) ? 0u : kStatusNonFinite;
  if (tid == 0 && (!(bn > 0.0) || flag)) *stop = 1;  // the same in every block
  barrier();                                         // also orders the writes of p before the reads below
  int k = 0;
  const int vrows = (rows * kLanes + 31) / 32 * 32;
  // The loop's exit is block-uniform (`stop`) and the same in every block (it depends on the
  // cluster's sums alone).
  // A block whose rows all have their own lanes keeps them, and their column offsets, in registers.
  constexpr int kPart = (kRow + kLanes - 1) / kLanes;
  const bool own = vrows <= nthr;
  T ar[kPart];
  int ao[kPart];
  if (own && rows > 0) {
    const int row = min(tid / kLanes, rows - 1), node = (row0 + row) % M3;
#pragma unroll
    for (int u = 0; u < kPart; ++u) {
      const int j = tid % kLanes + u * kLanes;
      ar[u] = j < kRow ? A[j * Rpad + row] : T(0);
      ao[u] = node + off[min(j, kRow - 1)];
    }
  }
  while (k < a.maxit && !*stop) {
    if (own) {
      if (tid < vrows) {
        T s = T(0), s1 = T(0);
#pragma unroll
        for (int u = 0; u < kPart; u += 2) {
          s = fma(ar[u], p[ao[u]], s);
          if (u + 1 < kPart) s1 = fma(ar[u + 1], p[ao[u + 1]], s1);
        }
        s += s1;
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (tid % kLanes == 0 && tid / kLanes < rows) q[tid / kLanes] = s;
      }
    } else {
      for (int i = tid; i < vrows; i += nthr) {
        const int row = min(i / kLanes, rows - 1), node = (row0 + row) % M3;
        T s = T(0);
#pragma unroll 7
        for (int j = i % kLanes; j < kRow; j += kLanes) s = fma(A[j * Rpad + row], p[node + off[j]], s);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (i % kLanes == 0 && i / kLanes < rows) q[row] = s;
      }
    }
    ++k;
    __syncthreads();
    v0 = v1 = 0.0;
    if (tid < 32)
      for (int i = tid; i < rows; i += 32) v0 = fma(double(p[row0 + i]), double(q[i]), v0);
    sum1(v0);
    const bool ok = v0 > 0.0 && isfinite(v0);  // warp 0
    if (tid < 32) {
      const T alpha = ok ? quotient<T>(rz, v0) : T(0);
      v0 = 0.0;
      for (int i = tid; i < rows; i += 32) {
        x[i] = fma(alpha, p[row0 + i], x[i]);
        const T ri = fma(-alpha, q[i], r[i]), zi = di[i] * ri;
        r[i] = ri;
        q[i] = zi;
        v0 = fma(double(ri), double(zi), v0);
        v1 = fma(double(ri), double(ri), v1);
      }
    }
    sum2(v0, v1);
    if (tid < 32) {
      bool end = !ok;
      if (!ok) {
        flag = kStatusBreakdown;
      } else if (k % a.check == 0 || k == a.maxit) {
        if (!isfinite(v1)) flag = kStatusNonFinite;
        end = flag || sqrt(v1) <= a.rtol * bn;
      }
      if (end) {
        if (tid == 0) *stop = 1;
      } else {
        const T beta = quotient<T>(v0, rz);
        rz = v0;
        for (int i = tid; i < rows; i += 32) set_p(i, fma(beta, p[row0 + i], q[i]));
      }
    }
    barrier();
  }
  for (int i = tid; i < rows; i += nthr) a.x[row0 + i] = x[i];
  if (rank == 0 && tid == 0) {
    a.words[0] += (unsigned long long)k;
    a.words[1] |= flag;
  }
  barrier();  // no block leaves while another may still write to its shared memory
}

// Shared memory of a solve without and with the matrix rows.
template <typename T>
size_t cg_smem(int n, int M, int R, int Rpad, bool rows) {
  const size_t pad = (size_t)M * M + M + 1;
  return 64 * sizeof(double) + 84 * sizeof(int) +
         (n + 2 * pad + 4 * (size_t)R + (rows ? (size_t)kRow * Rpad : 0)) * sizeof(T);
}

// The kernel's limits belong to the device, not to one hierarchy: every set-up sets the same ones, so
// that none lowers what another one, alive beside it, launches with.
template <typename T>
cudaError_t allow() {
  cudaError_t e = cudaFuncSetAttribute(k_coarse_cg<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCgSmemMax);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_coarse_cg<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

template <typename T>
cudaLaunchConfig_t cg_config(const CoarseSolve& C, int n, int M, cudaLaunchAttribute* attr, bool* in_smem,
                             cudaStream_t s) {
  const size_t with = cg_smem<T>(n, M, C.R, C.Rpad, true);
  *in_smem = with <= kCgSmemMax;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)C.blocks;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)C.blocks);
  cfg.blockDim = dim3((unsigned)std::min(kCgThreads, (C.R * kLanes + 31) / 32 * 32));
  cfg.dynamicSmemBytes = *in_smem ? with : cg_smem<T>(n, M, C.R, C.Rpad, false);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

template <typename T>
bool cluster_fits(const CoarseSolve& C, int n, int M) {
  cudaLaunchAttribute attr;
  bool in_smem;
  const cudaLaunchConfig_t cfg = cg_config<T>(C, n, M, &attr, &in_smem, nullptr);
  int clusters = 0;
  const bool ok = allow<T>() == cudaSuccess &&
                  cudaOccupancyMaxActiveClusters(&clusters, k_coarse_cg<T>, &cfg) == cudaSuccess && clusters > 0;
  if (!ok) cudaGetLastError();
  return ok;
}

}  // namespace

void coarse_setup(Gmg& G) {
  GmgLevel& L = G.L[0];
  CoarseSolve& C = G.coarse;
  if (L.ctx->g.p != 1 || L.ctx->g.N > kCoarseMaxN) return;
  const int n = (int)L.n, M = L.M;
  // about 200 rows per block (the FP64 reductions), at most one cluster of 16
  C.blocks = 1;
  while (C.blocks < 16 && (n + C.blocks - 1) / C.blocks > 200) C.blocks *= 2;
  C.R = (n + C.blocks - 1) / C.blocks;
  C.Rpad = (C.R + 31 - 8) / 32 * 32 + 8;  // = 8 mod 32: the four lanes of a row read distinct banks
  const size_t entries = (size_t)C.blocks * kRow * C.Rpad;
  if (cluster_fits<double>(C, n, M) && cluster_fits<float>(C, n, M) &&
      cudaMalloc(&C.words, 2 * sizeof(unsigned long long)) == cudaSuccess &&
      cudaMalloc(&C.Ke, (size_t)L.ctx->g.E * 576 * sizeof(double)) == cudaSuccess &&
      cudaMalloc(&C.A64, entries * sizeof(double)) == cudaSuccess &&
      cudaMalloc(&C.A32, entries * sizeof(float)) == cudaSuccess)
    return;
  // no room on the chip or in memory (18 MB at 13^3): pcg() solves the level on its operator
  cudaGetLastError();
  coarse_free(G);
}

void coarse_free(Gmg& G) {
  cudaFree(G.coarse.words);
  cudaFree(G.coarse.Ke);
  cudaFree(G.coarse.A64);
  cudaFree(G.coarse.A32);
  G.coarse = CoarseSolve{};
}

nhmf_status coarse_assemble(Gmg& G, cudaStream_t s) {
  GmgLevel& L = G.L[0];
  const CoarseSolve& C = G.coarse;
  const nhmf_ctx* c = L.ctx;
  ElemArgs a{};
  a.N = c->g.N;
  a.model = c->prm.model;
  a.h = c->g.h;
  a.mu = c->prm.mu;
  a.lam = c->prm.lambda;
  for (int q = 0; q < 2; ++q) {
    a.w[q] = c->tab.w[q];
    for (int i = 0; i < 2; ++i) {
      a.B[2 * q + i] = c->tab.B[q][i];
      a.D[2 * q + i] = c->tab.D[q][i];
    }
  }
  a.u = c->ubar;
  a.factor = c->factor;
  a.Ke = C.Ke;
  k_coarse_elements<<<(unsigned)c->g.E, 64, 0, s>>>(a);
  const int entries = C.blocks * kRow * C.Rpad;
  k_coarse_rows<<<(entries + 255) / 256, 256, 0, s>>>(C.Ke, a.N, c->prm.bc, C.R, C.Rpad, C.blocks, C.A64, C.A32);
  return cuda_check(L.ctx, cudaGetLastError(), "coarse matrix");
}

template <typename T>
nhmf_status coarse_cg(Gmg& G, const T* b, T* x, double rtol, int maxit, int check, cudaStream_t s) {
  GmgLevel& L = G.L[0];
  const CoarseSolve& C = G.coarse;
  CgArgs<T> a{};
  a.A = reinterpret_cast<const T*>(sizeof(T) == 4 ? (const void*)C.A32 : (const void*)C.A64);
  a.b = b;
  a.dinv = Buf<T>::dinv(L);
  a.x = x;
  a.n = (int)L.n;
  a.M = L.M;
  a.R = C.R;
  a.Rpad = C.Rpad;
  a.rtol = rtol;
  a.maxit = maxit;
  a.check = check;
  a.words = C.words;
  cudaLaunchAttribute attr;
  bool in_smem;
  const cudaLaunchConfig_t cfg = cg_config<T>(C, a.n, a.M, &attr, &in_smem, s);
  a.in_smem = in_smem;
  return cuda_check(L.ctx, cudaLaunchKernelEx(&cfg, k_coarse_cg<T>, a), "coarse solve");
}

template nhmf_status coarse_cg<float>(Gmg&, const float*, float*, double, int, int, cudaStream_t);
template nhmf_status coarse_cg<double>(Gmg&, const double*, double*, double, int, int, cudaStream_t);

}  // namespace nhmf
