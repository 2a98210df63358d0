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
// TP x TR tiles that reach the lower triangle, MP x MR entries per thread, fp64 fused multiply-adds.  The operands are
// widened once, when a stage is stored to shared memory (widening them at every use kept the conversion pipe busy twice as
// long as the fp64 pipe), and the next stage's loads are issued before the present stage is used.  What bounds it is shared
// memory (MP / 2 + MR / 2 loads of 16 bytes per MP MR multiply-adds) and idle SMs: 1350 features by 4099 rows took 1.2 ms with
// floats in shared memory, 0.9 in 128 x 64 tiles with 8 x 4, 0.8 in 64 x 64 with 4 x 4, 0.7 in 64 x 32 tiles with two groups of
// threads that take every other row of a stage (KS groups, their sums added in a fixed order).  Narrow layers are bound by the
// chain of multiply-adds behind an entry: 16 x 16 tiles and four groups (256 features by 1024 rows: 140 us with 64 x 64 tiles,
// 33 with 16 x 16 and one group, 21 with four).
template <typename TX, int TP, int TR, int MP, int MR, int HK, int KS>
__global__ void __launch_bounds__((TP / MP) * (TR / MR) * KS) hessian_simt_kernel(const TX* __restrict__ X, long long n,
                                                                                  long long d_in, long long ldx, int accumulate,
                                                                                  float* __restrict__ H) {
  const long long p0 = (long long)blockIdx.y * TP, r0 = (long long)blockIdx.x * TR;
  if (r0 > p0 + TP - 1) return;   // above the diagonal: the mirror image is written from below it
  constexpr int NP = TP / MP, NR = TR / MR, NTH = NP * NR * KS, LP = HK * TP / NTH, LR = HK * TR / NTH;
  static_assert(HK * TP % NTH == 0 && HK * TR % NTH == 0 && HK % KS == 0 && MP % 2 == 0 && MR % 2 == 0, "whole loads");
  __shared__ __align__(16) double sa[HK][TP + 2];
  __shared__ __align__(16) double sb[HK][TR + 2];
  __shared__ double red[KS > 1 ? (KS - 1) * TP * TR : 1];
  const int ks = threadIdx.x / (NP * NR), tx = threadIdx.x % NR, ty = threadIdx.x / NR % NP;
  double acc[MP][MR];
#pragma unroll
  for (int a = 0; a < MP; ++a)
#pragma unroll
    for (int b = 0; b < MR; ++b) acc[a][b] = 0.0;
  TX xa[LP], xb[LR];
  auto fetch = [&](long long k0) {
#pragma unroll
    for (int e = 0; e < LP; ++e) {
      const int idx = threadIdx.x + e * NTH, kk = idx / TP, cc = idx % TP;
      xa[e] = (k0 + kk < n && p0 + cc < d_in) ? X[(k0 + kk) * ldx + p0 + cc] : TX(0.f);
    }
#pragma unroll
    for (int e = 0; e < LR; ++e) {
      const int idx = threadIdx.x + e * NTH, kk = idx / TR, cc = idx % TR;
      xb[e] = (k0 + kk < n && r0 + cc < d_in) ? X[(k0 + kk) * ldx + r0 + cc] : TX(0.f);
    }
  };
  fetch(0);
  for (long long k0 = 0; k0 < n; k0 += HK) {
#pragma unroll
    for (int e = 0; e < LP; ++e) {
      const int idx = threadIdx.x + e * NTH;
      sa[idx / TP][idx % TP] = (double)(float)xa[e];
    }
#pragma unroll
    for (int e = 0; e < LR; ++e) {
      const int idx = threadIdx.x + e * NTH;
      sb[idx / TR][idx % TR] = (double)(float)xb[e];
    }
    __syncthreads();
    if (k0 + HK < n) fetch(k0 + HK);
#pragma unroll
    for (int k = 0; k < HK / KS; ++k) {
      const int kk = k * KS + ks;
      double a[MP], b[MR];
      // (a thread's entries are pairs of neighbours, so that the 16-byte loads of neighbouring threads are contiguous)
#pragma unroll
      for (int u = 0; u < MP; u += 2) {
        const double2 va = *reinterpret_cast<const double2*>(&sa[kk][u * NP + 2 * ty]);
        a[u] = va.x; a[u + 1] = va.y;
      }
#pragma unroll
      for (int u = 0; u < MR; u += 2) {
        const double2 vb = *reinterpret_cast<const double2*>(&sb[kk][u * NR + 2 * tx]);
        b[u] = vb.x; b[u + 1] = vb.y;
      }
#pragma unroll
      for (int u = 0; u < MP; ++u)
#pragma unroll
        for (int v = 0; v < MR; ++v) acc[u][v] = fma(a[u], b[v], acc[u][v]);
    }
    __syncthreads();
  }
  if constexpr (KS > 1) {
    const int t = threadIdx.x % (NP * NR);
#pragma unroll
    for (int u = 0; u < MP; ++u)
#pragma unroll
      for (int v = 0; v < MR; ++v)
        if (ks > 0) red[((ks - 1) * MP * MR + u * MR + v) * NP * NR + t] = acc[u][v];
    __syncthreads();
    if (ks > 0) return;
    for (int s = 0; s < KS - 1; ++s)
#pragma unroll
      for (int u = 0; u < MP; ++u)
#pragma unroll
        for (int v = 0; v < MR; ++v) acc[u][v] += red[(s * MP * MR + u * MR + v) * NP * NR + t];
  }
#pragma unroll
  for (int u = 0; u < MP; ++u)
#pragma unroll
    for (int v = 0; v < MR; ++v) {
      const long long p = p0 + (u & ~1) * NP + 2 * ty + (u & 1), r = r0 + (v & ~1) * NR + 2 * tx + (v & 1);
      if (p < d_in && r <= p) {
        const float prev = accumulate ? H[p * d_in + r] : 0.f;
        const float val = (float)((double)prev + acc[u][v]);
        H[p * d_in + r] = val;
        if (r < p) H[r * d_in + p] = val;
      }
    }
}

template <int TP, int TR, int MP, int MR, int HK, int KS>
static void run_hessian_simt(const void* X, cdq_dtype xt, long long n, long long d_in, long long ldx, int accumulate,
                             float* H, cudaStream_t st) {
  const dim3 grid((unsigned)((d_in + TR - 1) / TR), (unsigned)((d_in + TP - 1) / TP)), block((TP / MP) * (TR / MR) * KS);
  if (xt == CDQ_BF16)
    { hessian_simt_kernel<__nv_bfloat16, TP, TR, MP, MR, HK, KS><<<grid, block, 0, st>>>((const __nv_bfloat16*)X, n, d_in, ldx, accumulate, H); count_launch(); }
  else
    { hessian_simt_kernel<float, TP, TR, MP, MR, HK, KS><<<grid, block, 0, st>>>((const float*)X, n, d_in, ldx, accumulate, H); count_launch(); }
}

cudaError_t launch_hessian_simt(const void* X, cdq_dtype xt, long long n, long long d_in, long long ldx,
                                int accumulate, float* H, cudaStream_t st) {
  if (d_in <= 512) run_hessian_simt<16, 16, 2, 2, 64, 4>(X, xt, n, d_in, ldx, accumulate, H, st);
  else run_hessian_simt<64, 32, 4, 4, 32, 2>(X, xt, n, d_in, ldx, accumulate, H, st);
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
