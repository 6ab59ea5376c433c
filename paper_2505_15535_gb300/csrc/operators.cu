// Entry points of the matrix-free operators: the degree of the context selects the kernels, which
// operators_p1.cu ... operators_p4.cu instantiate (one translation unit per degree, so that they
// compile in parallel).
#include "sumfact.cuh"

namespace nhmf {
namespace {

// ------------------------------------------------------------------ Dirichlet rows
// out[d] = src[d] on every constrained DoF.
__global__ void k_fix_constrained(int bc, int M, long long M3, const double* src, double* out) {
  const long long f = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long M2 = (long long)M * M;
  if (f >= M2) return;
  const int x = int(f % M), y = int(f / M);
  auto fix = [&](int c, long long node) { out[c * M3 + node] = src[c * M3 + node]; };
  if (bc == NHMF_BC_CLAMP_X0) {
    const long long node = (long long)M * (x + (long long)M * y);  // (0, x, y)
    for (int c = 0; c < 3; ++c) fix(c, node);
  } else if (bc == NHMF_BC_COMPRESSION) {
    const long long bottom = x + (long long)M * y;
    const long long top = bottom + M2 * (M - 1);
    for (int c = 0; c < 3; ++c) fix(c, bottom);
    fix(2, top);
  }
}

__global__ void k_to_fp32(const double* x, float* y, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    y[i] = float(x[i]);
}

nhmf_status apply(nhmf_ctx* c, int prec, int strat, const void* du, void* v, bool raw, const Gather32& g32,
                  cudaStream_t s) {
  switch (c->g.p) {
    case 1: return Operators<1>::apply(c, prec, strat, du, v, raw, g32, s);
    case 2: return Operators<2>::apply(c, prec, strat, du, v, raw, g32, s);
    case 3: return Operators<3>::apply(c, prec, strat, du, v, raw, g32, s);
    case 4: return Operators<4>::apply(c, prec, strat, du, v, raw, g32, s);
  }
  return fail(c, NHMF_ERR_ARG, "degree out of range");
}
}  // namespace

nhmf_status launch_apply(nhmf_ctx* c, int prec, int strat, const void* du, void* v, cudaStream_t s, bool raw) {
  return apply(c, prec, strat, du, v, raw, Gather32{}, s);
}

nhmf_status launch_apply32(nhmf_ctx* c, int strat, const float* du, float* v, const Gather32& g32, cudaStream_t s) {
  return apply(c, NHMF_FP32, strat, du, v, false, g32, s);
}

nhmf_status launch_cache_build(nhmf_ctx* c, cudaStream_t s) {
  switch (c->g.p) {
    case 1: return Operators<1>::cache(c, s);
    case 2: return Operators<2>::cache(c, s);
    case 3: return Operators<3>::cache(c, s);
    case 4: return Operators<4>::cache(c, s);
  }
  return fail(c, NHMF_ERR_ARG, "degree out of range");
}

nhmf_status launch_residual(nhmf_ctx* c, const double* u, double* r, cudaStream_t s) {
  switch (c->g.p) {
    case 1: return Operators<1>::residual(c, u, r, s);
    case 2: return Operators<2>::residual(c, u, r, s);
    case 3: return Operators<3>::residual(c, u, r, s);
    case 4: return Operators<4>::residual(c, u, r, s);
  }
  return fail(c, NHMF_ERR_ARG, "degree out of range");
}

nhmf_status launch_diagonal(nhmf_ctx* c, double* d, cudaStream_t s) {
  switch (c->g.p) {
    case 1: return Operators<1>::diagonal(c, d, s);
    case 2: return Operators<2>::diagonal(c, d, s);
    case 3: return Operators<3>::diagonal(c, d, s);
    case 4: return Operators<4>::diagonal(c, d, s);
  }
  return fail(c, NHMF_ERR_ARG, "degree out of range");
}

nhmf_status fix_rows64(nhmf_ctx* c, const double* src, double* out, cudaStream_t s) {
  if (c->prm.bc == NHMF_BC_NONE) return NHMF_OK;
  const long long M2 = (long long)c->g.M * c->g.M;
  k_fix_constrained<<<(unsigned)((M2 + 255) / 256), 256, 0, s>>>(c->prm.bc, c->g.M, c->g.M3, src, out);
  return cuda_check(c, cudaGetLastError(), "dirichlet rows");
}

nhmf_status launch_to_fp32(const double* x, float* y, long long n, cudaStream_t s) {
  k_to_fp32<<<1216, 256, 0, s>>>(x, y, n);
  return cudaGetLastError() == cudaSuccess ? NHMF_OK : NHMF_ERR_CUDA;
}

}  // namespace nhmf
