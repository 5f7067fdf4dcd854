// Macroscopic kernels that close one IUGKP iteration: the macro update (arXiv
// 2506.09465 Sec. 3.1 step (3), Sec. 3.2 step (2)), the residual, and the element-wise steps of
// the adjoint iteration and the averaging (the correction solve is in mgpcg.cu). All FP64.
#include <cuda_runtime.h>

#include "internal.h"

namespace iugkp {

__device__ __forceinline__ int find_inst(const InstDesc* inst, int n_inst, long long g) {
  int lo = 0, hi = n_inst - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (inst[mid].cell_off <= g) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// T_half = sum_b R_b / (V m); T_E = sum_b W_b / (V sum_b C_b).
__global__ void macro_kernel(const InstDesc* inst, int n_inst, int nb, long long total, const double* R,
                             const double* W, const double* Vm, const double* VC, double* T_half, double* T_E) {
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < total; g += (long long)gridDim.x * blockDim.x) {
    const int k = find_inst(inst, n_inst, g);
    const InstDesc& in = inst[k];
    const long long i = g - in.cell_off;
    const long long base = in.bc_off + i;
    double r = 0.0, w = 0.0;
    for (int b = 0; b < nb; ++b) r += R[base + (long long)b * in.ncells];
    if (T_half) T_half[g] = r / Vm[g];
    if (T_E && W) {
      for (int b = 0; b < nb; ++b) w += W[base + (long long)b * in.ncells];
      T_E[g] = w / VC[g];
    }
  }
}

__global__ void add_kernel(long long total, const double* a, const double* b, double* out) {
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < total; g += (long long)gridDim.x * blockDim.x)
    out[g] = a[g] + b[g];
}

__global__ void div_kernel(long long total, const double* a, const double* b, double* out) {
  for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < total; g += (long long)gridDim.x * blockDim.x)
    out[g] = a[g] / b[g];
}

// Block-wide sum in a fixed order (deterministic). All threads get the result.
template <int NT>
__device__ __forceinline__ double block_sum(double x, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sh[warp] = x;
  __syncthreads();
  if (warp == 0) {
    double y = lane < NT / 32 ? sh[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) y += __shfl_down_sync(0xffffffffu, y, o);
    if (lane == 0) sh[32] = y;
  }
  __syncthreads();
  return sh[32];
}

// Deterministic two-stage sums of (T1 - T0)^2 and T1^2 over all cells.
constexpr int RES_BLOCKS = 256;
__global__ void __launch_bounds__(256) residual_stage1(long long total, const double* T0, const double* T1,
                                                       double* partial) {
  __shared__ double sh[33];
  double a = 0.0, c = 0.0;
  for (long long g = (long long)blockIdx.x * 256 + threadIdx.x; g < total; g += (long long)RES_BLOCKS * 256) {
    const double d = T1[g] - T0[g];
    a += d * d;
    c += T1[g] * T1[g];
  }
  a = block_sum<256>(a, sh);
  c = block_sum<256>(c, sh);
  if (threadIdx.x == 0) {
    partial[2 * blockIdx.x] = a;
    partial[2 * blockIdx.x + 1] = c;
  }
}
__global__ void __launch_bounds__(256) residual_stage2(const double* partial, double* out) {
  __shared__ double sh[33];
  double a = partial[2 * threadIdx.x], c = partial[2 * threadIdx.x + 1];
  a = block_sum<256>(a, sh);
  c = block_sum<256>(c, sh);
  if (threadIdx.x == 0) {
    out[0] = a;
    out[1] = c;
  }
}

// Largest |x| (NaN left out) as the bit pattern of a non-negative double, max-reduced into *out.
__global__ void __launch_bounds__(256) absmax_kernel(long long total, const double* x, unsigned long long* out) {
  unsigned long long m = 0;
  for (long long i = blockIdx.x * 256ll + threadIdx.x; i < total; i += (long long)gridDim.x * 256) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x[i]) & 0x7fffffffffffffffull;
    if (b <= 0x7ff0000000000000ull && b > m) m = b;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_down_sync(0xffffffffu, m, o);
    m = t > m ? t : m;
  }
  if ((threadIdx.x & 31) == 0 && m) atomicMax(out, m);
}

static unsigned grid_for(const Ctx* c, long long n) {
  long long b = (n + 255) / 256;
  long long cap = (long long)c->sm_count * 8;
  if (b > cap) b = cap;
  return (unsigned)(b < 1 ? 1 : b);
}

cudaError_t launch_macro(const Ctx* c, const double* R, const double* W, double* T_half, double* T_E, cudaStream_t s) {
  macro_kernel<<<grid_for(c, c->total_cells), 256, 0, s>>>(c->d_inst, c->n_inst, c->nb, c->total_cells, R, W, c->d_Vm,
                                                          c->d_VC, T_half, T_E);
  return cudaGetLastError();
}

cudaError_t launch_residual(const Ctx* c, const double* T0, const double* T1, double, double* out_dev, cudaStream_t s) {
  residual_stage1<<<RES_BLOCKS, 256, 0, s>>>(c->total_cells, T0, T1, c->d_red);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  residual_stage2<<<1, 256, 0, s>>>(c->d_red, out_dev);
  return cudaGetLastError();
}

// Sets ERR_PCG in the device error word when any instance's CG hit its iteration cap
// (lets an iteration run without a host round trip for the CG status).
__global__ void pcg_check_kernel(const int* iters, int n_inst, int* err) {
  for (int k = threadIdx.x; k < n_inst; k += blockDim.x)
    if (iters[k] < 0) atomicOr(err, ERR_PCG);
}

cudaError_t launch_pcg_check(const Ctx* c, cudaStream_t s) {
  pcg_check_kernel<<<1, 128, 0, s>>>(c->d_pcg_iters, c->n_inst, c->d_err);
  return cudaGetLastError();
}

// Statistical averaging (Sec. 4.4-4.5): the k-th sample x updates the running mean and the
// sum of squared deviations M2 (Welford's one-pass update; FP64).
__global__ void welford_kernel(long long total, const double* x, double* mean, double* m2, double inv_k) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const double d = x[i] - mean[i];
    const double mu = mean[i] + d * inv_k;
    mean[i] = mu;
    if (m2) m2[i] += d * (x[i] - mu);
  }
}

__global__ void scale_kernel(long long total, double* x, double a) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x)
    x[i] *= a;
}

cudaError_t launch_welford(const Ctx* c, const double* x, double* mean, double* m2, long long n, int k,
                           cudaStream_t s) {
  welford_kernel<<<grid_for(c, n), 256, 0, s>>>(n, x, mean, m2, 1.0 / (double)k);
  return cudaGetLastError();
}

cudaError_t launch_scale(const Ctx* c, double* x, long long n, double a, cudaStream_t s) {
  scale_kernel<<<grid_for(c, n), 256, 0, s>>>(n, x, a);
  return cudaGetLastError();
}

cudaError_t launch_absmax(const Ctx* c, const double* x, long long n, double* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double), s);
  if (e != cudaSuccess) return e;
  absmax_kernel<<<grid_for(c, n), 256, 0, s>>>(n, x, reinterpret_cast<unsigned long long*>(out));
  return cudaGetLastError();
}

cudaError_t launch_axpy_grad(const Ctx* c, const double* at, const double* g, double* lam_half, cudaStream_t s) {
  add_kernel<<<grid_for(c, c->total_cells), 256, 0, s>>>(c->total_cells, at, g, lam_half);
  return cudaGetLastError();
}

cudaError_t launch_grad_source(const Ctx* c, const double* at, double* grad, cudaStream_t s) {
  div_kernel<<<grid_for(c, c->total_cells), 256, 0, s>>>(c->total_cells, at, c->d_m, grad);
  return cudaGetLastError();
}

}  // namespace iugkp
