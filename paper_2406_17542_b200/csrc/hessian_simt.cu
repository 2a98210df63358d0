// H = X^T X on the CUDA cores (paper: Section 3 "Notation"; Algorithm 1).
//  - verify kernels: every entry is the ascending-k fp64 sum without fused
//    multiply-add, rounded once to fp32 (bit-reproducible on a CPU);
//  - SIMT kernel: tiled, fp64 accumulation, any shape and input type; used for
//    fp32 inputs and for shapes the tensor-core kernel does not take.
#include "common.cuh"

namespace cdq {

template <typename T> __device__ __forceinline__ double ld_as_double(const T* p, long long i);
template <> __device__ __forceinline__ double ld_as_double<float>(const float* p, long long i) { return (double)p[i]; }
template <> __device__ __forceinline__ double ld_as_double<__nv_bfloat16>(const __nv_bfloat16* p, long long i) {
  return (double)__bfloat162float(p[i]);
}

template <typename T>
__global__ void hessian_verify_kernel(const T* __restrict__ X, long long n, long long d_in, long long ldx,
                                      double* __restrict__ H64) {
  const long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long p = blockIdx.y;
  if (r >= d_in) return;
  double acc = 0.0;
  for (long long k = 0; k < n; ++k) {
    const double xp = ld_as_double(X, k * ldx + p);
    const double xr = ld_as_double(X, k * ldx + r);
    acc = __dadd_rn(acc, __dmul_rn(xp, xr));
  }
  H64[p * d_in + r] = acc;
}

// One thread: trace in ascending order, then the regulariser on the diagonal.
__global__ void lambda_verify_kernel(double* H64, long long d_in, double lambda_rel) {
  if (blockIdx.x || threadIdx.x) return;
  double tr = 0.0;
  for (long long p = 0; p < d_in; ++p) tr = __dadd_rn(tr, H64[p * d_in + p]);
  const double add = __dmul_rn(lambda_rel, __ddiv_rn(tr, (double)d_in));
  for (long long p = 0; p < d_in; ++p) H64[p * d_in + p] = __dadd_rn(H64[p * d_in + p], add);
}

__global__ void round_to_f32_kernel(const double* __restrict__ src, float* __restrict__ dst, long long count) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < count) dst[i] = (float)src[i];
}

cudaError_t launch_hessian_verify(const void* X, cdq_dtype xt, long long n, long long d_in, long long ldx,
                                  double lambda_rel, float* H, double* H64, cudaStream_t st) {
  dim3 block(128), grid((unsigned)((d_in + 127) / 128), (unsigned)d_in);
  if (xt == CDQ_BF16)
    { hessian_verify_kernel<__nv_bfloat16><<<grid, block, 0, st>>>((const __nv_bfloat16*)X, n, d_in, ldx, H64); count_launch(); }
  else
    { hessian_verify_kernel<float><<<grid, block, 0, st>>>((const float*)X, n, d_in, ldx, H64); count_launch(); }
  if (lambda_rel > 0.0) { lambda_verify_kernel<<<1, 32, 0, st>>>(H64, d_in, lambda_rel); count_launch(); }
  const long long count = d_in * d_in;
  { round_to_f32_kernel<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(H64, H, count); count_launch(); }
  return cudaGetLastError();
}

// ---- tiled SIMT kernel -----------------------------------------------------
// T x T tiles of the lower triangle, (T / M)^2 threads with M x M entries each, fp64 fused multiply-adds in ascending
// order of the rows, whatever the tile.  Bound by the fp64 pipe (64 per clock and SM): the operands are widened once,
// when a stage is stored to shared memory (widening them at every use kept the conversion pipe busy twice as long as the
// fp64 pipe: 1.2 ms at 4099 rows by 1350 features), and the next stage's loads are issued before the present stage is used.
// T = 64 for layers whose tiles fill the SMs; smaller tiles for narrow ones, where a 64-tile list leaves most SMs idle
// (256 features: 10 tiles, 140 us at 1024 rows).
constexpr int HK = 16;   // rows of X per stage

template <typename TX, int T, int M>
__global__ void __launch_bounds__((T / M) * (T / M)) hessian_simt_kernel(const TX* __restrict__ X, long long n, long long d_in,
                                                                         long long ldx, int accumulate, float* __restrict__ H) {
  // Only tiles on or below the diagonal are computed; the mirror image is written too.
  const int tp = blockIdx.y, tr = blockIdx.x;
  if (tr > tp) return;
  constexpr int TT = T / M, NTH = TT * TT, LD = HK * T / NTH;
  __shared__ __align__(16) double sa[HK][T + 2];
  __shared__ __align__(16) double sb[HK][T + 2];
  const int tx = threadIdx.x % TT, ty = threadIdx.x / TT;
  const long long p0 = (long long)tp * T, r0 = (long long)tr * T;
  double acc[M][M];
#pragma unroll
  for (int a = 0; a < M; ++a)
#pragma unroll
    for (int b = 0; b < M; ++b) acc[a][b] = 0.0;
  TX xa[LD], xb[LD];
  auto fetch = [&](long long k0) {
#pragma unroll
    for (int e = 0; e < LD; ++e) {
      const int idx = threadIdx.x + e * NTH, kk = idx / T, cc = idx % T;
      const long long k = k0 + kk;
      xa[e] = (k < n && p0 + cc < d_in) ? X[k * ldx + p0 + cc] : TX(0.f);
      xb[e] = (k < n && r0 + cc < d_in) ? X[k * ldx + r0 + cc] : TX(0.f);
    }
  };
  fetch(0);
  for (long long k0 = 0; k0 < n; k0 += HK) {
#pragma unroll
    for (int e = 0; e < LD; ++e) {
      const int idx = threadIdx.x + e * NTH, kk = idx / T, cc = idx % T;
      sa[kk][cc] = (double)(float)xa[e];
      sb[kk][cc] = (double)(float)xb[e];
    }
    __syncthreads();
    if (k0 + HK < n) fetch(k0 + HK);
#pragma unroll
    for (int kk = 0; kk < HK; ++kk) {
      double a[M], b[M];
#pragma unroll
      for (int u = 0; u < M; u += 2) {
        // (a thread's entries are pairs of neighbours, so that the 16-byte loads of neighbouring threads are contiguous)
        const double2 va = *reinterpret_cast<const double2*>(&sa[kk][u * TT + 2 * ty]);
        const double2 vb = *reinterpret_cast<const double2*>(&sb[kk][u * TT + 2 * tx]);
        a[u] = va.x; a[u + 1] = va.y; b[u] = vb.x; b[u + 1] = vb.y;
      }
#pragma unroll
      for (int u = 0; u < M; ++u)
#pragma unroll
        for (int v = 0; v < M; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < M; ++u)
#pragma unroll
    for (int v = 0; v < M; ++v) {
      const long long p = p0 + (u & ~1) * TT + 2 * ty + (u & 1), r = r0 + (v & ~1) * TT + 2 * tx + (v & 1);
      if (p < d_in && r < d_in) {
        const float prev = accumulate ? H[p * d_in + r] : 0.f;
        const float val = (float)((double)prev + acc[u][v]);
        H[p * d_in + r] = val;
        if (tp != tr) H[r * d_in + p] = val;   // (a diagonal tile computes every entry directly)
      }
    }
}

template <int T, int M>
static void run_hessian_simt(const void* X, cdq_dtype xt, long long n, long long d_in, long long ldx, int accumulate,
                             float* H, cudaStream_t st) {
  const unsigned t = (unsigned)((d_in + T - 1) / T);
  dim3 grid(t, t), block((T / M) * (T / M));
  if (xt == CDQ_BF16)
    { hessian_simt_kernel<__nv_bfloat16, T, M><<<grid, block, 0, st>>>((const __nv_bfloat16*)X, n, d_in, ldx, accumulate, H); count_launch(); }
  else
    { hessian_simt_kernel<float, T, M><<<grid, block, 0, st>>>((const float*)X, n, d_in, ldx, accumulate, H); count_launch(); }
}

cudaError_t launch_hessian_simt(const void* X, cdq_dtype xt, long long n, long long d_in, long long ldx,
                                int accumulate, float* H, cudaStream_t st) {
  if (d_in <= 512) run_hessian_simt<16, 2>(X, xt, n, d_in, ldx, accumulate, H, st);
  else if (d_in <= 1024) run_hessian_simt<32, 2>(X, xt, n, d_in, ldx, accumulate, H, st);
  else run_hessian_simt<64, 4>(X, xt, n, d_in, ldx, accumulate, H, st);
  return cudaGetLastError();
}

// H_ii += lambda_rel * mean(diag H), trace reduced in fp64 by one block.
__global__ void lambda_kernel(float* H, long long d_in, double lambda_rel) {
  __shared__ double red[256];
  double s = 0.0;
  for (long long p = threadIdx.x; p < d_in; p += blockDim.x) s += (double)H[p * d_in + p];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  const double add = lambda_rel * (red[0] / (double)d_in);
  for (long long p = threadIdx.x; p < d_in; p += blockDim.x) H[p * d_in + p] = (float)((double)H[p * d_in + p] + add);
}

cudaError_t launch_hessian_lambda(float* H, long long d_in, double lambda_rel, double*, cudaStream_t st) {
  { lambda_kernel<<<1, 256, 0, st>>>(H, d_in, lambda_rel); count_launch(); }
  return cudaGetLastError();
}

}  // namespace cdq
