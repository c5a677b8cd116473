// Vector kernels of the Lanczos method on the SQH matvec (lowest eigenvalues of H(t) and the
// gap above the ground state along the path, Sec. IV.B): block inner products with FP64
// accumulation in a fixed order, block updates w -= sum_i c_i v_i, and scaling by a device
// scalar.  Basis vectors are rows of one array with leading dimension `ld` elements.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "aqc_internal.h"

namespace aqc {

namespace {

template <typename R>
struct C2of;
template <>
struct C2of<float> {
  using T = float2;
};
template <>
struct C2of<double> {
  using T = double2;
};

constexpr int kLzThreads = 256;

// double of a float, exactly, in integer instructions for normal numbers (a conversion instruction
// runs at the FP64 rate, a tenth of what these sums can spare)
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f), e = (u >> 23) & 0xffu;
  if (e - 1u < 254u)
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
  return (double)f;
}
__device__ __forceinline__ double widen(double d) { return d; }

// Sums over the CTA of K doubles per thread in a fixed order, in thread 0.  A tree through shared
// memory: an FP64 instruction of a warp holds its multiprocessor's pipe for about 19 cycles, and the
// tree issues a third of a shuffle reduction's.
template <int K>
__device__ __forceinline__ void cta_tree(double (&v)[K], double (*s)[kLzThreads]) {
  const int t = threadIdx.x;
#pragma unroll
  for (int k = 0; k < K; k++) s[k][t] = v[k];
  for (int o = kLzThreads / 2; o > 0; o >>= 1) {
    __syncthreads();
    if (t < o)
#pragma unroll
      for (int k = 0; k < K; k++) s[k][t] += s[k][t + o];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; k++) v[k] = s[k][0];
}

// True in every thread of the launch's last CTA to come here (their partials are then visible).
__device__ __forceinline__ bool last_cta(unsigned* counter) {
  __shared__ int s_last;
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(counter, 1u) == gridDim.x * gridDim.y - 1u ? 1 : 0;
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  if (threadIdx.x == 0) *counter = 0u;
  return true;
}

// out[2i], out[2i+1] = <v_i, w>; acc (nullable) is set to Re <v_last, w> (mode 1) or raised by it (2).
// Bound by the FP64 pipe (4 multiply-adds per element and vector): blocks of few elements, so that one
// vector alone spreads over the GPU too, each row's blocks summed in order by the last CTA of the
// launch.  64 Lanczos steps at n = 16 (complex128): 13.5 -> 8.6 ms with one launch per reduction, the norm summed in
// the update and coefficients read eight steps at a time (the FP64 floor is 4.1 ms).
template <typename R>
__global__ void __launch_bounds__(kLzThreads) k_dotc_multi(const typename C2of<R>::T* __restrict__ V, uint64_t ld,
                                                           const typename C2of<R>::T* __restrict__ w, uint64_t N,
                                                           double* partials, double* out, double* acc, int mode,
                                                           unsigned* counter) {
  using C2 = typename C2of<R>::T;
  __shared__ double s_sum[2][kLzThreads];
  const uint32_t i = blockIdx.y, G = gridDim.x, m = gridDim.y;
  const C2* v = V + (uint64_t)i * ld;
  double s[2] = {0.0, 0.0};
#pragma unroll 4
  for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < N; e += (uint64_t)G * blockDim.x) {
    const C2 a = v[e], b = w[e];
    const double ax = widen(a.x), ay = widen(a.y), bx = widen(b.x), by = widen(b.y);
    s[0] = fma(ax, bx, fma(ay, by, s[0]));
    s[1] = fma(ax, by, fma(-ay, bx, s[1]));
  }
  cta_tree<2>(s, s_sum);
  if (threadIdx.x == 0) {
    partials[((uint64_t)i * G + blockIdx.x) * 2] = s[0];
    partials[((uint64_t)i * G + blockIdx.x) * 2 + 1] = s[1];
  }
  if (!last_cta(counter)) return;
  for (uint32_t k = threadIdx.x; k < 2 * m; k += blockDim.x) {
    double a = 0.0;
#pragma unroll 8
    for (uint32_t g = 0; g < G; g++) a += __ldcg(&partials[((uint64_t)(k >> 1) * G + g) * 2 + (k & 1u)]);
    out[k] = a;
    if (acc && k == 2 * (m - 1)) *acc = mode == 2 ? *acc + a : a;
  }
}

// w -= sum_i c_i v_i  (c complex, FP64, on the device); norm (nullable): norm[0] = ||w||^2 after it
template <typename R>
__global__ void __launch_bounds__(kLzThreads) k_sub_multi(typename C2of<R>::T* __restrict__ w,
                                                          const typename C2of<R>::T* __restrict__ V, uint64_t ld,
                                                          uint32_t m, const double* __restrict__ c, uint64_t N,
                                                          double* norm, double* partials, unsigned* counter) {
  using C2 = typename C2of<R>::T;
  __shared__ double s_sum[1][kLzThreads];
  double n2[1] = {0.0};
  for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < N; e += (uint64_t)gridDim.x * blockDim.x) {
    double re = (double)w[e].x, im = (double)w[e].y;
#pragma unroll 4
    for (uint32_t i = 0; i < m; i++) {
      const C2 v = V[(uint64_t)i * ld + e];
      const double cr = c[2 * i], ci = c[2 * i + 1], vx = widen(v.x), vy = widen(v.y);
      re = fma(-cr, vx, fma(ci, vy, re));
      im = fma(-cr, vy, fma(-ci, vx, im));
    }
    const C2 r = C2{(R)re, (R)im};
    w[e] = r;
    if (norm) {
      const double x = widen(r.x), y = widen(r.y);
      n2[0] = fma(x, x, fma(y, y, n2[0]));
    }
  }
  if (!norm) return;
  cta_tree<1>(n2, s_sum);
  if (threadIdx.x == 0) partials[blockIdx.x] = n2[0];
  if (!last_cta(counter)) return;
  n2[0] = 0.0;
  for (uint32_t g = threadIdx.x; g < gridDim.x; g += blockDim.x) n2[0] += __ldcg(&partials[g]);
  cta_tree<1>(n2, s_sum);
  if (threadIdx.x == 0) norm[0] = n2[0];
}

// v = w / sqrt(nrm2[0])
template <typename R>
__global__ void __launch_bounds__(kLzThreads) k_scale_to(typename C2of<R>::T* __restrict__ v,
                                                         const typename C2of<R>::T* __restrict__ w, uint64_t N,
                                                         const double* __restrict__ nrm2) {
  using C2 = typename C2of<R>::T;
  const double s = 1.0 / sqrt(nrm2[0]);
  for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < N; e += (uint64_t)gridDim.x * blockDim.x) {
    const C2 a = w[e];
    v[e] = C2{(R)((double)a.x * s), (R)((double)a.y * s)};
  }
}

int lz_grid(uint64_t N) {
  uint64_t g = (N + 4095) / 4096;
  if (g > 256) g = 256;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

uint32_t lanczos_dot_blocks(uint64_t N) { return (uint32_t)lz_grid(N); }

cudaError_t launch_dotc_multi(int prec, const void* V, uint64_t ld, uint32_t m, const void* w, uint64_t N,
                              const LzScratch& sc, double* out, double* acc, int mode, cudaStream_t s) {
  if (m == 0) return cudaSuccess;
  // four elements per thread where the scratch holds that many partials
  uint64_t g = (N + 4 * kLzThreads - 1) / (4 * kLzThreads);
  if (g > sc.doubles / (2 * (uint64_t)m)) g = sc.doubles / (2 * (uint64_t)m);
  if (g > 256) g = 256;
  if (g < 1) g = 1;
  const dim3 grid((unsigned)g, m);
  if (prec == 0)
    k_dotc_multi<double><<<grid, kLzThreads, 0, s>>>((const double2*)V, ld, (const double2*)w, N, sc.partials, out, acc,
                                                     mode, sc.counter);
  else
    k_dotc_multi<float><<<grid, kLzThreads, 0, s>>>((const float2*)V, ld, (const float2*)w, N, sc.partials, out, acc, mode,
                                                    sc.counter);
  return cudaGetLastError();
}

cudaError_t launch_sub_multi(int prec, void* w, const void* V, uint64_t ld, uint32_t m, const double* c, uint64_t N,
                             const LzScratch& sc, double* norm, cudaStream_t s) {
  if (m == 0) return cudaSuccess;
  uint64_t g = (N + kLzThreads - 1) / kLzThreads;
  if (g > 4096) g = 4096;
  if (norm && g > sc.doubles) g = sc.doubles;
  if (prec == 0)
    k_sub_multi<double><<<(int)g, kLzThreads, 0, s>>>((double2*)w, (const double2*)V, ld, m, c, N, norm, sc.partials,
                                                      sc.counter);
  else
    k_sub_multi<float><<<(int)g, kLzThreads, 0, s>>>((float2*)w, (const float2*)V, ld, m, c, N, norm, sc.partials,
                                                     sc.counter);
  return cudaGetLastError();
}

cudaError_t launch_scale_to(int prec, void* v, const void* w, uint64_t N, const double* nrm2, cudaStream_t s) {
  const int grid = (int)((N + kLzThreads - 1) / kLzThreads < 4096 ? (N + kLzThreads - 1) / kLzThreads : 4096);
  if (prec == 0)
    k_scale_to<double><<<grid, kLzThreads, 0, s>>>((double2*)v, (const double2*)w, N, nrm2);
  else
    k_scale_to<float><<<grid, kLzThreads, 0, s>>>((float2*)v, (const float2*)w, N, nrm2);
  return cudaGetLastError();
}

}  // namespace aqc
