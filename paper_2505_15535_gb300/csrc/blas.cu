// Vector kernels of the Krylov solvers (Section 2.3: CG on the matrix-free operator).
// Reductions are deterministic: a grid that depends on the length alone accumulates FP64 partial
// sums with a fixed grid-stride order and a fixed shuffle tree; the last block to finish reduces
// the partials in a fixed order.  Results stay on the device.  The kernels start while the launch
// before them drains and wait for it before they read (pdl.cuh).
#include "blas.h"
#include "pdl.cuh"

namespace nhmf {
namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Sums of NS values per thread over the grid: every block writes its partial sums, and the block
// that comes last (a counter behind the partials, back at zero afterwards) adds them in block
// order, so the sums do not depend on timing.  True, with the sums in `tot`, in that block's thread
// 0 alone.  (A second launch for the final sum cost 3-4 us on every dot product.)
template <int NS>
__device__ __forceinline__ bool grid_sum(double (&acc)[NS], double* partials, double (&tot)[NS]) {
  __shared__ double sh[NS][kRedThreads / 32];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  auto block_sum = [&](double (&v)[NS]) {  // in warp 0's lane 0
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      v[s] = warp_sum(v[s]);
      if (lane == 0) sh[s][wid] = v[s];
    }
    __syncthreads();
    if (wid == 0) {
#pragma unroll
      for (int s = 0; s < NS; ++s) v[s] = warp_sum(lane < kRedThreads / 32 ? sh[s][lane] : 0.0);
    }
  };
  block_sum(acc);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int s = 0; s < NS; ++s) partials[s * kRedBlocks + blockIdx.x] = acc[s];
    __threadfence();
    last = atomicInc(reinterpret_cast<unsigned*>(partials + kRedBlocks * 3), gridDim.x - 1) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    tot[s] = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += kRedThreads) tot[s] += __ldcg(partials + s * kRedBlocks + i);
  }
  block_sum(tot);
  return threadIdx.x == 0;
}

// Blocks of a reduction over n values: at least four values a thread, at most kRedBlocks.
unsigned red_blocks(long long n) {
  const long long b = (n + 4 * kRedThreads - 1) / (4 * kRedThreads);
  return (unsigned)(b < 1 ? 1 : (b > kRedBlocks ? kRedBlocks : b));
}

// *out = x . y, its square root if `root`; with `den`, also *quot = sign * *out / *den.
template <typename TX, typename TY>
__global__ void __launch_bounds__(kRedThreads) k_dot(long long n, const TX* x, const TY* y, double* partials, double* out,
                                                     bool root, const double* den, double sign, double* quot) {
  pdl_launch_next();
  pdl_wait();
  double acc[1] = {0.0}, tot[1];
  for (long long i = blockIdx.x * (long long)kRedThreads + threadIdx.x; i < n; i += (long long)gridDim.x * kRedThreads)
    acc[0] = fma(double(x[i]), double(y[i]), acc[0]);
  if (!grid_sum<1>(acc, partials, tot)) return;
  const double v = root ? sqrt(tot[0]) : tot[0];
  *out = v;
  if (den) *quot = sign * (v / *den);
}

// PCG update (Jacobi): alpha = rz/pq; x += alpha p; r -= alpha q; z = dinv r;
// r.z and r.r.  A non-positive p.q is a breakdown: alpha = 0 and flag.
template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_pcg_update(long long n, const double* rz, const double* pq, T* x, T* r,
                                                            const T* p, const T* q, const T* dinv, T* z, double* partials,
                                                            double* rz_new, double* rr, unsigned* flag) {
  pdl_launch_next();
  pdl_wait();
  const double pqv = *pq;
  const bool ok = pqv > 0.0 && isfinite(pqv);
  const T alpha = ok ? T(*rz / pqv) : T(0);
  if (!ok && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(flag, 4u);
  double acc[2] = {0.0, 0.0}, tot[2];
  for (long long i = blockIdx.x * (long long)kRedThreads + threadIdx.x; i < n; i += (long long)gridDim.x * kRedThreads) {
    x[i] = fma(alpha, p[i], x[i]);
    const T ri = fma(-alpha, q[i], r[i]);
    r[i] = ri;
    const T zi = dinv[i] * ri;
    z[i] = zi;
    acc[0] = fma(double(ri), double(zi), acc[0]);
    acc[1] = fma(double(ri), double(ri), acc[1]);
  }
  if (!grid_sum<2>(acc, partials, tot)) return;
  *rz_new = tot[0];
  *rr = tot[1];
}

// Flexible CG: *pq = p.q, *alpha = p.r / p.q.
__global__ void __launch_bounds__(kRedThreads) k_fcg_alpha(long long n, const double* p, const double* q, const double* r,
                                                           double* partials, double* pq, double* alpha) {
  pdl_launch_next();
  pdl_wait();
  double acc[2] = {0.0, 0.0}, tot[2];
  for (long long i = blockIdx.x * (long long)kRedThreads + threadIdx.x; i < n; i += (long long)gridDim.x * kRedThreads) {
    acc[0] = fma(p[i], q[i], acc[0]);
    acc[1] = fma(p[i], r[i], acc[1]);
  }
  if (!grid_sum<2>(acc, partials, tot)) return;
  *pq = tot[0];
  *alpha = tot[1] / tot[0];
}

// x += alpha p, r -= alpha q, *rnorm = ||r||.
__global__ void __launch_bounds__(kRedThreads) k_fcg_update(long long n, const double* alpha, const double* p,
                                                            const double* q, double* x, double* r, double* partials,
                                                            double* rnorm) {
  pdl_launch_next();
  pdl_wait();
  const double al = *alpha;
  double acc[1] = {0.0}, tot[1];
  for (long long i = blockIdx.x * (long long)kRedThreads + threadIdx.x; i < n; i += (long long)gridDim.x * kRedThreads) {
    x[i] = fma(al, p[i], x[i]);
    const double ri = fma(-al, q[i], r[i]);
    r[i] = ri;
    acc[0] = fma(ri, ri, acc[0]);
  }
  if (grid_sum<1>(acc, partials, tot)) *rnorm = sqrt(tot[0]);
}

// p = z + beta p with beta = rz_new / rz_old (beta = 0 when rz_old is null).
template <typename T>
__global__ void k_pcg_direction(long long n, const double* rz_new, const double* rz_old, const T* z, T* p) {
  pdl_launch_next();
  pdl_wait();
  const T beta = rz_old ? T(*rz_new / *rz_old) : T(0);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    p[i] = rz_old ? fma(beta, p[i], z[i]) : z[i];
}

// z = dinv r, r.z and r.r (start of PCG).
template <typename T>
__global__ void __launch_bounds__(kRedThreads) k_jacobi(long long n, const T* r, const T* dinv, T* z, double* partials,
                                                        double* rz, double* rr) {
  pdl_launch_next();
  pdl_wait();
  double acc[2] = {0.0, 0.0}, tot[2];
  for (long long i = blockIdx.x * (long long)kRedThreads + threadIdx.x; i < n; i += (long long)gridDim.x * kRedThreads) {
    const T zi = dinv[i] * r[i];
    z[i] = zi;
    acc[0] = fma(double(r[i]), double(zi), acc[0]);
    acc[1] = fma(double(r[i]), double(r[i]), acc[1]);
  }
  if (!grid_sum<2>(acc, partials, tot)) return;
  *rz = tot[0];
  *rr = tot[1];
}

// y = a x + b y with scalars a = sa * (*pa) (pa may be null -> sa), same for b.
__global__ void k_axpby(long long n, double sa, const double* pa, const double* x, double sb, const double* pb, double* y) {
  pdl_launch_next();
  pdl_wait();
  const double a = pa ? sa * *pa : sa;
  const double b = pb ? sb * *pb : sb;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = b == 0.0 ? a * x[i] : fma(a, x[i], b * y[i]);
}

// z = noise in [-1, 1) from a hash of the index and the seed.
__global__ void k_noise(long long n, double* z, unsigned long long seed) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    unsigned long long v = (unsigned long long)i + seed * 0x9E3779B97F4A7C15ull;
    v = (v ^ (v >> 30)) * 0xBF58476D1CE4E5B9ull;
    v = (v ^ (v >> 27)) * 0x94D049BB133111EBull;
    v ^= v >> 31;
    z[i] = double(v >> 11) * 0x1.0p-52 - 1.0;
  }
}

__global__ void k_ratio_or_zero(const double* num, const double* den, double* out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    const double r = *num / *den;
    *out = (*den > 0.0 && isfinite(r)) ? r : 0.0;
  }
}

template <typename TI, typename TO>
__global__ void k_scale_convert(long long n, const TI* x, const double* scale, bool invert, TO* y) {
  pdl_launch_next();
  pdl_wait();
  double s = scale ? *scale : 1.0;
  if (invert) s = s > 0.0 ? 1.0 / s : 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    y[i] = TO(double(x[i]) * s);
}

__global__ void k_reciprocal(long long n, const double* d, double* dinv64, float* dinv32) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double v = 1.0 / d[i];
    if (dinv64) dinv64[i] = v;
    if (dinv32) dinv32[i] = float(v);
  }
}

constexpr int kEwBlocks = 1216;  // 8 blocks per SM for element-wise kernels
constexpr int kEwThreads = 256;
unsigned ew_blocks(long long n) {
  const long long b = (n + kEwThreads - 1) / kEwThreads;
  return (unsigned)(b < 1 ? 1 : (b > kEwBlocks ? kEwBlocks : b));
}

template <typename TX, typename TY>
void launch_dot(long long n, const TX* x, const TY* y, double* partials, double* out, bool root, const double* den,
                double sign, double* quot, cudaStream_t s) {
  launch(k_dot<TX, TY>, dim3(red_blocks(n)), kRedThreads, 0, s, true, n, x, y, partials, out, root, den, sign, quot);
}

}  // namespace

void dot(long long n, const double* x, const double* y, double* out, double* partials, cudaStream_t s) {
  launch_dot(n, x, y, partials, out, false, nullptr, 0.0, nullptr, s);
}
void dot(long long n, const float* x, const float* y, double* out, double* partials, cudaStream_t s) {
  launch_dot(n, x, y, partials, out, false, nullptr, 0.0, nullptr, s);
}
void dot_ratio(long long n, const double* x, const double* y, double* out, const double* den, double sign, double* quot,
               double* partials, cudaStream_t s) {
  launch_dot(n, x, y, partials, out, false, den, sign, quot, s);
}
void norm2(long long n, const double* x, double* out, double* partials, cudaStream_t s) {
  launch_dot(n, x, x, partials, out, true, nullptr, 0.0, nullptr, s);
}
void norm2(long long n, const float* x, double* out, double* partials, cudaStream_t s) {
  launch_dot(n, x, x, partials, out, true, nullptr, 0.0, nullptr, s);
}
void fcg_alpha(long long n, const double* p, const double* q, const double* r, double* pq, double* alpha,
               double* partials, cudaStream_t s) {
  launch(k_fcg_alpha, dim3(red_blocks(n)), kRedThreads, 0, s, true, n, p, q, r, partials, pq, alpha);
}
void fcg_update(long long n, const double* alpha, const double* p, const double* q, double* x, double* r, double* rnorm,
                double* partials, cudaStream_t s) {
  launch(k_fcg_update, dim3(red_blocks(n)), kRedThreads, 0, s, true, n, alpha, p, q, x, r, partials, rnorm);
}

template <typename T>
void pcg_update(long long n, const double* rz, const double* pq, T* x, T* r, const T* p, const T* q, const T* dinv, T* z,
                double* rz_new, double* rr, double* partials, unsigned* flag, cudaStream_t s) {
  launch(k_pcg_update<T>, dim3(red_blocks(n)), kRedThreads, 0, s, true, n, rz, pq, x, r, p, q, dinv, z, partials, rz_new, rr, flag);
}
template <typename T>
void pcg_direction(long long n, const double* rz_new, const double* rz_old, const T* z, T* p, cudaStream_t s) {
  launch(k_pcg_direction<T>, dim3(ew_blocks(n)), kEwThreads, 0, s, true, n, rz_new, rz_old, z, p);
}
template <typename T>
void jacobi(long long n, const T* r, const T* dinv, T* z, double* rz, double* rr, double* partials, cudaStream_t s) {
  launch(k_jacobi<T>, dim3(red_blocks(n)), kRedThreads, 0, s, true, n, r, dinv, z, partials, rz, rr);
}
template void pcg_update<double>(long long, const double*, const double*, double*, double*, const double*, const double*,
                                 const double*, double*, double*, double*, double*, unsigned*, cudaStream_t);
template void pcg_update<float>(long long, const double*, const double*, float*, float*, const float*, const float*,
                                const float*, float*, double*, double*, double*, unsigned*, cudaStream_t);
template void pcg_direction<double>(long long, const double*, const double*, const double*, double*, cudaStream_t);
template void pcg_direction<float>(long long, const double*, const double*, const float*, float*, cudaStream_t);
template void jacobi<double>(long long, const double*, const double*, double*, double*, double*, double*, cudaStream_t);
template void jacobi<float>(long long, const float*, const float*, float*, double*, double*, double*, cudaStream_t);

void axpby(long long n, double a, const double* pa, const double* x, double b, const double* pb, double* y, cudaStream_t s) {
  launch(k_axpby, dim3(ew_blocks(n)), kEwThreads, 0, s, true, n, a, pa, x, b, pb, y);
}
void fill_noise(long long n, double* z, unsigned long long seed, cudaStream_t s) {
  k_noise<<<kRedBlocks, kRedThreads, 0, s>>>(n, z, seed);
}
void ratio_or_zero(const double* num, const double* den, double* out, cudaStream_t s) {
  k_ratio_or_zero<<<1, 32, 0, s>>>(num, den, out);
}
void to_fp32_scaled(long long n, const double* x, const double* scale, bool invert, float* y, cudaStream_t s) {
  launch(k_scale_convert<double, float>, dim3(ew_blocks(n)), kEwThreads, 0, s, true, n, x, scale, invert, y);
}
void to_fp64_scaled(long long n, const float* x, const double* scale, double* y, cudaStream_t s) {
  launch(k_scale_convert<float, double>, dim3(ew_blocks(n)), kEwThreads, 0, s, true, n, x, scale, false, y);
}
void reciprocal(long long n, const double* d, double* dinv64, float* dinv32, cudaStream_t s) {
  k_reciprocal<<<kEwBlocks, kEwThreads, 0, s>>>(n, d, dinv64, dinv32);
}

}  // namespace nhmf
