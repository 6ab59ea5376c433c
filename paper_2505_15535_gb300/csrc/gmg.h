// Geometric multigrid on the nested structured meshes (see gmg.cu).
#pragma once
#include <vector>

#include "internal.h"

namespace nhmf {

// A 1D linear map between node lines, as CSR rows: out[i] = sum_k w[k] in[col[k]], k in [ptr[i], ptr[i+1]).
struct Map1D {
  int rows = 0, cols = 0;
  int *ptr = nullptr, *col = nullptr;  // device
  double* w64 = nullptr;
  float* w32 = nullptr;
};

struct GmgLevel {
  nhmf_ctx* ctx = nullptr;  // level context (owned; index 0 = coarsest)
  long long n = 0;          // DoFs
  int M = 0;
  double lmax = 0.0;        // estimate of the largest eigenvalue of D^-1 A
  double *diag = nullptr, *dinv = nullptr;
  float* dinv32 = nullptr;
  double *x = nullptr, *b = nullptr, *r = nullptr, *d = nullptr, *q = nullptr, *t1 = nullptr, *t2 = nullptr;
  float *x32 = nullptr, *b32 = nullptr, *r32 = nullptr, *d32 = nullptr, *q32 = nullptr, *t132 = nullptr, *t232 = nullptr;
  Map1D P;   // prolongation from the next coarser level to this one (rows: this level's M)
  Map1D R;   // its transpose (rows: the coarser level's M)
  Map1D I;   // interpolation of the linearisation point from this level to the coarser one
};

// The coarsest level's matrix and solve (coarse.cu).
// Elements per direction up to which the level is a matrix; above it the rows no longer stay in shared
// memory and pcg() on the operator is as fast or faster.  Solves of a one-level hierarchy, matrix /
// operator, in ms: FP64 7^3 2.8 / 7.6, 9^3 3.5 / 10.5, 11^3 6.4 / 11.9, 13^3 10.5 / 14.6, 15^3 17.3 / 17.6;
// FP32 7^3 1.6 / 3.3, 9^3 1.9 / 4.4, 11^3 3.3 / 5.2, 13^3 4.6 / 5.6, 15^3 8.4 / 6.8.
constexpr int kCoarseMaxN = 13;
struct CoarseSolve {
  int blocks = 0;            // blocks of the solve's cluster; 0: the level is solved by pcg() on its operator
  int R = 0, Rpad = 0;       // rows per block, padded
  double *Ke = nullptr, *A64 = nullptr;
  float* A32 = nullptr;
  unsigned long long* words = nullptr;  // device: iterations since zeroed, status flags met
};

constexpr int kMaxLevels = 13;     // twelve meshes and the p-coarsened one

struct Gmg {
  CoarseSolve coarse;
  std::vector<GmgLevel> L;  // L.back() mirrors the fine context (its ctx pointer is not owned)
};

void gmg_free(nhmf_ctx* c);
nhmf_status gmg_build(nhmf_ctx* c);
// Level linearisation points (interpolated from the fine one, or zero on the coarse levels),
// diagonals and eigenvalue estimates.
// fine_diag: the fine operator's diagonal if the caller has it (else it is computed).
nhmf_status gmg_prepare(nhmf_ctx* c, int strategy, bool fp32, cudaStream_t s, bool coarse_at_zero,
                        const double* fine_diag = nullptr);
// per-level buffers by precision
template <typename T> struct Buf;
template <> struct Buf<double> {
  static double* x(GmgLevel& l) { return l.x; }
  static double* b(GmgLevel& l) { return l.b; }
  static double* r(GmgLevel& l) { return l.r; }
  static double* d(GmgLevel& l) { return l.d; }
  static double* q(GmgLevel& l) { return l.q; }
  static double* t1(GmgLevel& l) { return l.t1; }
  static double* t2(GmgLevel& l) { return l.t2; }
  static const double* dinv(GmgLevel& l) { return l.dinv; }
  static constexpr int prec = NHMF_FP64;
};
template <> struct Buf<float> {
  static float* x(GmgLevel& l) { return l.x32; }
  static float* b(GmgLevel& l) { return l.b32; }
  static float* r(GmgLevel& l) { return l.r32; }
  static float* d(GmgLevel& l) { return l.d32; }
  static float* q(GmgLevel& l) { return l.q32; }
  static float* t1(GmgLevel& l) { return l.t132; }
  static float* t2(GmgLevel& l) { return l.t232; }
  static const float* dinv(GmgLevel& l) { return l.dinv32; }
  static constexpr int prec = NHMF_FP32;
};

template <typename T>
nhmf_status chebyshev(GmgLevel& L, int strat, const T* b, T* x, int degree, double range, bool zero_start,
                      cudaStream_t s);
template <typename T>
nhmf_status gmg_residual(GmgLevel& L, int strat, const T* b, const T* x, T* r, cudaStream_t s);
template <typename T>
void gmg_restrict(GmgLevel& F, GmgLevel& C, const T* r_fine, T* r_coarse, cudaStream_t s);
template <typename T>
void gmg_prolong_add(GmgLevel& F, GmgLevel& C, const T* e_coarse, T* x_fine, cudaStream_t s);
// Memory and cluster shape of the coarsest level's solve; where they cannot be had, blocks stays 0.
void coarse_setup(Gmg& G);
void coarse_free(Gmg& G);
// The coarsest operator's matrix at its level's linearisation point.
nhmf_status coarse_assemble(Gmg& G, cudaStream_t s);
// Jacobi-CG on it from x = 0, as pcg() does it; asynchronous, see CoarseSolve::words.
template <typename T>
nhmf_status coarse_cg(Gmg& G, const T* b, T* x, double rtol, int maxit, int check, cudaStream_t s);
void gmg_start_vector(long long n, double* v, cudaStream_t s);

}  // namespace nhmf
