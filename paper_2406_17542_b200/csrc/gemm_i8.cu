// C = E^T H on the integer tensor cores, exact to a chosen number of bits: the contraction
// behind the gradient G = 2 H (W_hat - W) (paper: Algorithm 1, the gradient step), the column losses
// e_j^T H e_j (paper: Eq. 1 with H = X^T X) and the loss per clipping strength of the OWC
// search (the minimisation stated after Eq. 2).
//
// Why integers.  The descent compares scores whose gradient term must be right to ~1e-9 of
// a_j H_pp, while a row of H mixes entries that differ by many powers of two (feature scales),
// so the products need about 40 bits.  The fp64 pipe of B200 gives ~15 TFLOP/s to a SIMT GEMM;
// the int8 tensor cores give two orders of magnitude more, and integer accumulation is exact.
// So both operands are cut into 7-bit signed slices (error-free splitting):
//     H[p,k]   = 2^hexp[p] * sum_i hs_i[p,k] 128^-i,     i = 1..NH   (row p scaled by its max)
//     E[k,j]   = 2^eexp[j] * sum_i es_i[j,k] 128^-i,     i = 1..NE   (column j scaled by its max)
// with hs_i, es_i in [-127, 127].  Every slice pair is an int8 x int8 -> int32 GEMM without
// rounding; pairs with the same i + j = s share one accumulator (up to 5 pairs x K x 127^2 fits
// in 31 bits for K <= 26 000) and the result is sum_s 128^-s acc_s, summed in fp64 from the
// smallest term up.  Pairs beyond i + j = smax are dropped: that is the only approximation, and
// it is bounded by K * (#dropped) * 128^-(smax+1) relative to (row max) x (column max).
//
// Kernel: M = 128 columns j of the layer (rows of E^T), N = 256 coordinates p (rows of H),
// K-major operands in 128-byte swizzled tiles loaded by TMA, tcgen05.mma kind::i8 with the
// int32 accumulators in TMEM (two of them, so the epilogue of one group overlaps the MMAs of
// the next), the same warp roles as the Hessian kernel.  Every mbarrier wait is bounded.
//
// Losses alone take half of the product.  e^T H e is that of H's symmetric part S = (H + H^T) / 2, and with the rows and columns of S
// in blocks of 256, a column's loss is
//     e^T S e = 2 sum_P e_P^T (T_P e_P + sum_{K in half(P)} S_PK e_K),
// where half(P) holds one of the blocks (P, K), (K, P) of every pair: the nb / 2 blocks that follow P, in a circle, so that every tile
// has the same work.  (S is formed where the slices are, so that an H which is symmetric only up to rounding, or not at all, has the loss
// that the whole product gives it.)  T_P is the lower triangle of the diagonal block with half of its diagonal.
// The two halves of the whole product average an entry's slicing error with that of its mirror image; here it counts twice.  Two things
// make up for that.  The digits are balanced (balanced_bits below).  And the clipping search, whose screen has two or three digits of
// either operand, takes the product of H D^-1 and D E, D_kk = 2^s_k near sqrt(H_kk): |H_pk| <= sqrt(H_pp H_kk) (or D = 1, see
// feature_check_kernel), so the rows no longer mix entries of many sizes, and what an entry of E weighs in the loss is its size.  The
// residuals of given codes are a few dozen bits on one grid, which five digits hold exactly, and D would take them off it: cdq_layer_loss
// goes without (column losses of 8192 x 300 codes against 64 bits, rms: with D 3.9e-13, without 1.1e-13; whole product 1.0e-13).  Errors against 64 bits, whole -> half:
//   thirteen pairs (largest of five layers of 2 to 8 bits, heavy weights among them) 2.4e-7 -> 1e-8
//   27 pairs, rms over columns and eight layers each, given codes: 3072 x 512 9.5e-14 -> 9.6e-14, 4096 x 4096 in groups 3.1e-12 -> 3.2e-12,
//   6144 x 256 in groups 9.3e-13 -> 9.4e-13; solved codes 1.5e-12 -> 1.4e-12, 5.8e-10 -> 4.5e-11, 6.0e-11 -> 1.5e-11
#include <cuda.h>

#include "async_copy.cuh"
#include "common.cuh"

namespace cdq {
namespace i8 {

constexpr int BM = 128, BN = 256, BKB = 128;       // tile; BKB = bytes (= int8 elements) of K per stage
constexpr int STAGES = 4;
constexpr int A_BYTES = BM * BKB, B_BYTES = BN * BKB, STAGE_BYTES = A_BYTES + B_BYTES;  // 16 + 32 KB
constexpr int NUM_THREADS = 320;     // producer, MMA issuer, 8 epilogue warps (two per TMEM lane quarter)
constexpr int EPI_WARPS = 8;
constexpr int TMEM_COLS = 512;
constexpr uint32_t SPIN_LIMIT = 1u << 24;
constexpr size_t SMEM_BYTES = 1024 + (size_t)STAGES * STAGE_BYTES + 256;
constexpr int MAX_SLICES = 6;
constexpr int MAX_GROUPS = 12;

// ---------------------------------------------------------------------------------------------
// Slicing.  exps[r] = e with max_k |x[r,k]| 2^-e in [0.5, 1) (0 for an all-zero row).

// BALANCED: for balanced digits (below), whose top one is at most 127: max_k |x[r,k]| 2^-e at most 127.49 / 128.
template <bool BALANCED>
__device__ __forceinline__ int slice_exponent(double m) {
  // (a normal number, as products of fp32 data are: its exponent field)
  return m > 0.0 ? (__double2hiint(BALANCED ? 1.004 * m : m) >> 20) - 1022 : 0;
}

// 2^e for the exponents of normal numbers (those of products of fp32 data are).
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// Row maxima of a row-major fp32 matrix [rows, cols] -> exponent per row.
__global__ void row_exp_f32_kernel(const float* __restrict__ x, long long rows, long long cols, int* __restrict__ exps) {
  const long long r = blockIdx.x;
  float m = 0.f;
  for (long long k = threadIdx.x; k < cols; k += blockDim.x) m = fmaxf(m, fabsf(x[r * cols + k]));
  __shared__ float red[32];
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    if (threadIdx.x == 0) exps[r] = m < __int_as_float(0x7f800000) ? slice_exponent<false>((double)m) : 0;
  }
}

// Column maxima (ordered bit patterns) -> exponent per column.
template <bool BALANCED>
__global__ void col_exp_kernel(const unsigned long long* __restrict__ colmax_bits, long long cols, int* __restrict__ exps) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c >= cols) return;
  exps[c] = slice_exponent<BALANCED>(__longlong_as_double((long long)colmax_bits[c]));
}

// |x| 2^-e 128^ns, truncated, as an integer (x 2^-e in (-1, 1), ns <= 6): slice i of x is its 7-bit digit number ns - i from
// below with the sign of x, which is what truncating, subtracting and scaling up digit by digit gives.  The addition of
// 2^52 towards zero leaves the integer in the mantissa; scale = 2^(7 ns - e), a normal number for every exponent of H and E.
// A NaN counts as zero, whatever its payload (that of CUDA's float NaN would pass for digits): a product leaves out the
// entry and keeps the rest of its row.
__device__ __forceinline__ unsigned long long slice_bits(double x, double scale) {
  const double s = __dadd_rz(fabs(x) * scale, 4503599627370496.0);
  return s != s ? 0ull : (unsigned long long)__double_as_longlong(s) & 0xFFFFFFFFFFFFFull;
}
// Digit i (from 1) of four neighbours, negated where `neg` has the byte's bits set, as four bytes.
__device__ __forceinline__ unsigned slice_bytes(const unsigned long long (&v)[4], int shift, unsigned neg) {
  unsigned d = 0u;
#pragma unroll
  for (int k = 0; k < 4; ++k) d |= ((unsigned)(v[k] >> shift) & 127u) << (8 * k);
  return __vsub4(d ^ neg, neg);
}
// Balanced digits, for half products: x 2^-e 128^ns rounded to the nearest integer, digits from -64 to 63 (the top one from -127 to 127),
// so that every prefix of the digits is x to the nearest multiple of its last one.  A truncated prefix is off by up to a whole
// unit, always towards zero: half of a product does not average that over an entry and its mirror image, and the two-digit screen of
// the clipping search came out with 1.4 times the error of the whole product (see kScreenBand).
// balanced_magic: 1.5 2^52, which leaves the integer in the mantissa, and 64 in each of the lower digits, which makes them non-negative
// there.  What is no number or beyond the digits counts as zero.
__device__ __forceinline__ double balanced_magic(int ns) {
  return 6755399441055744.0 + (double)(64ll * (((1ll << (7 * (ns - 1))) - 1) / 127));
}
__device__ __forceinline__ unsigned long long balanced_bits(double x, double scale, double magic) {
  const double s = x * scale + magic;
  return (unsigned long long)__double_as_longlong(__double2hiint(s) >> 20 == 0x433 ? s : magic);   // (2^52 to 2^53)
}
__device__ __forceinline__ unsigned balanced_bytes(const unsigned long long (&v)[4], int shift, bool top) {
  const unsigned d = __byte_perm(__byte_perm((unsigned)(v[0] >> shift), (unsigned)(v[1] >> shift), 0x0040),
                                 __byte_perm((unsigned)(v[2] >> shift), (unsigned)(v[3] >> shift), 0x0040), 0x5410);
  return top ? d : ((d | 0x80808080u) - 0x40404040u) ^ 0x80808080u;   // the lower seven bits, less 64, in every byte
}
// The ns slices of four neighbours x, the first at `out`, the next `step` bytes on.
template <bool BALANCED>
__device__ __forceinline__ void write_slices(const double (&x)[4], int ns, int e, signed char* out, size_t step) {
  const double scale = pow2(7 * ns - e);
  unsigned long long b[4];
  if constexpr (BALANCED) {
    const double magic = balanced_magic(ns);
#pragma unroll
    for (int v = 0; v < 4; ++v) b[v] = balanced_bits(x[v], scale, magic);
    for (int i = 0; i < ns; ++i) *reinterpret_cast<unsigned*>(out + i * step) = balanced_bytes(b, 7 * (ns - 1 - i), i == 0);
  } else {
    unsigned neg = 0u;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      b[v] = slice_bits(x[v], scale);
      if (x[v] < 0.0) neg |= 0xFFu << (8 * v);
    }
    for (int i = 0; i < ns; ++i) *reinterpret_cast<unsigned*>(out + i * step) = slice_bytes(b, 7 * (ns - 1 - i), neg);
  }
}

// H [d, d] fp32 -> slices [ns][d][kp] int8 (row p scaled by 2^-exps[p]; columns >= d zero), four columns per thread.
// 4 bytes read and ns written per entry; what bounds it is the integer operations of the digits (4096^2, six slices: 45 us, the ALU pipe
// 63 % busy, 2.5 TB/s).  (One column per thread, with the digits taken off one after
// the other in fp64: 1.46 ms for 14336^2 and six slices.)
__global__ void slice_h_kernel(const float* __restrict__ H, long long d, long long kp, const int* __restrict__ exps,
                               int ns, signed char* __restrict__ out) {
  const long long p = blockIdx.y;
  const long long k = 4 * (blockIdx.x * (long long)blockDim.x + threadIdx.x);
  if (k >= kp) return;
  double x[4] = {0.0, 0.0, 0.0, 0.0};
  if ((d & 3) == 0) {
    if (k < d) {
      const float4 f = *reinterpret_cast<const float4*>(H + p * d + k);
      x[0] = (double)f.x; x[1] = (double)f.y; x[2] = (double)f.z; x[3] = (double)f.w;
    }
  } else {
#pragma unroll
    for (int v = 0; v < 4; ++v)
      if (k + v < d) x[v] = (double)H[p * d + k + v];
  }
  write_slices<false>(x, ns, exps[p], out + (size_t)p * kp + k, (size_t)d * kp);
}

// ---- half products ----
// Half of the product: how many blocks of 256 columns of H follow the diagonal one in tile column tn.
__device__ __forceinline__ int blocks_after(int tn, int nb) { return (nb - 1) / 2 + ((nb & 1) == 0 && tn < nb / 2 ? 1 : 0); }

// feat[k] = s_k with 2^s_k near sqrt(H_kk); 0 for a diagonal entry that is no positive number.
__global__ void feature_exp_kernel(const float* __restrict__ H, long long d, int* __restrict__ feat) {
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (k >= d) return;
  const float h = H[k * d + k];
  int e = 0;
  if (h > 0.f && h < __int_as_float(0x7f800000)) frexpf(h, &e);
  feat[k] = e >> 1;
}
// Four neighbours of a row of H from column k on (zero from d on).  VEC: rows start on 16-byte boundaries.
template <bool VEC>
__device__ __forceinline__ float4 four_of_row(const float* __restrict__ H, long long d, long long row, long long k) {
  const float* p = H + row * d + k;
  if (VEC) return k < d ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
  return make_float4(k < d ? p[0] : 0.f, k + 1 < d ? p[1] : 0.f, k + 2 < d ? p[2] : 0.f, k + 3 < d ? p[3] : 0.f);
}
// An entry that is no finite number counts as zero.
__device__ __forceinline__ float finite(float x) { return fabsf(x) <= 3.402823466e38f ? x : 0.f; }
// rowmax[p]: the largest |H_pk| and |H_kp| (SCALED: times 2^-feat[k], rounded up), as a bit pattern; no entry of row p of S (of S D^-1) is above it.
// `rows` rows x 1024 columns per block, four columns per thread: one pass over H from memory (24 us at 4096^2, 56 at 8192^2, 4.8 TB/s).  only_if (may be NULL): nothing is
// done where it is zero.
template <bool VEC, bool SCALED>
__global__ void __launch_bounds__(256) half_max_kernel(const float* __restrict__ H, long long d, const int* __restrict__ feat,
                                                       const int* __restrict__ only_if, int rows, unsigned* __restrict__ rowmax) {
  __shared__ unsigned s_row[64];
  if (only_if && *only_if == 0) return;
  const long long c = 4 * (blockIdx.x * 256ll + threadIdx.x), r0 = (long long)blockIdx.y * rows;
  if (threadIdx.x < rows) s_row[threadIdx.x] = 0u;
  __syncthreads();
  auto weight = [&](long long k) { return SCALED && k < d ? __int_as_float((127 - feat[k]) << 23) : 1.f; };   // (feat: -75 to 64)
  float wc[4], col[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int v = 0; v < 4; ++v) wc[v] = weight(c + v);
#pragma unroll 8
  for (int r = 0; r < rows; ++r) {
    if (r0 + r >= d) break;
    const float4 h4 = four_of_row<VEC>(H, d, r0 + r, c);
    const float h[4] = {fabsf(finite(h4.x)), fabsf(finite(h4.y)), fabsf(finite(h4.z)), fabsf(finite(h4.w))}, wr = weight(r0 + r);
    float row = 0.f;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      row = fmaxf(row, SCALED ? __fmul_ru(h[v], wc[v]) : h[v]);
      col[v] = fmaxf(col[v], SCALED ? __fmul_ru(h[v], wr) : h[v]);
    }
    const unsigned most = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(row));
    if ((threadIdx.x & 31) == 0) atomicMax(&s_row[r], most);
  }
#pragma unroll
  for (int v = 0; v < 4; ++v)
    if (c + v < d) atomicMax(&rowmax[c + v], __float_as_uint(col[v]));
  __syncthreads();
  if (threadIdx.x < rows && r0 + threadIdx.x < d) atomicMax(&rowmax[r0 + threadIdx.x], s_row[threadIdx.x]);
}
// D only where H is positive, as far as its pairs of entries show: then |H_pk| <= sqrt(H_pp H_kk), and rowmax[k] is at most 2^(feat[k] + 1) and
// a rounding.  Where a row is above twice that, the diagonal says nothing about the size of the entries (some random symmetric
// matrices lost strengths with D): D is 1, and without[0] says that the row maxima are to be taken again.  One block.
__global__ void __launch_bounds__(1024) feature_check_kernel(long long d, int* __restrict__ feat, unsigned* __restrict__ rowmax,
                                                             int* __restrict__ without) {
  int above = 0;
  for (long long k = threadIdx.x; k < d; k += blockDim.x) above |= rowmax[k] > (unsigned)(127 + feat[k] + 2) << 23;
  above = __syncthreads_or(above);
  if (threadIdx.x == 0) *without = above;
  if (!above) return;
  for (long long k = threadIdx.x; k < d; k += blockDim.x) { feat[k] = 0; rowmax[k] = 0u; }
}
// Slices of S D^-1 (rows scaled by 2^-exps) into `out`, [ns][d][kp]: the blocks (P, K) of 256 with K in half(P) and, in the place of the
// diagonal blocks, the triangles T_P; nothing reads the other blocks.  64 rows x 128 columns per block; the mirror image of the tile is turned round in
// shared memory, so that both are read along their rows, once.  An entry that is no finite number is left out, its mirror image is not.
// 4 bytes read and ns / 2 written per entry (4096^2, six slices: 39 us; all blocks of H, without its mirror image, and the triangles 53 us).
template <bool VEC>
__global__ void __launch_bounds__(256) half_slice_kernel(const float* __restrict__ H, long long d, long long kp, const int* __restrict__ feat,
                                                         const unsigned* __restrict__ rowmax, int ns, int* __restrict__ exps,
                                                         signed char* __restrict__ out) {
  constexpr int TP = 64, TK = 128;
  __shared__ __align__(16) float mirror[TP][TK];   // H[k][p] at [p][k ^ 4 (p / 4 % 8)]
  const int nb = (int)((d + BN - 1) / BN), P = (int)blockIdx.z, m = (int)blockIdx.y;
  if (m > blocks_after(P, nb)) return;
  const int K = P + m < nb ? P + m : P + m - nb;
  const long long p0 = (long long)P * BN + (blockIdx.x >> 1) * TP, k0 = (long long)K * BN + (blockIdx.x & 1) * TK;
  if (p0 >= d || k0 >= kp) return;
  const int kk = 4 * (threadIdx.x & 31);
  float4 h[TP / 8];   // rows p0 + warp, 8 further on, ...: on their way beside the mirror image
#pragma unroll
  for (int i = 0; i < TP / 8; ++i) {
    const long long p = p0 + 8 * i + (threadIdx.x >> 5);
    h[i] = p < d ? four_of_row<VEC>(H, d, p, k0 + kk) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  {
    const int t = 4 * (threadIdx.x & 15);
#pragma unroll
    for (int i = 0; i < TK / 16; ++i) {
      const int k = 16 * i + (threadIdx.x >> 4);
      const float4 g = k0 + k < d ? four_of_row<VEC>(H, d, k0 + k, p0 + t) : make_float4(0.f, 0.f, 0.f, 0.f);
      const int at = k ^ (t & 28);
      mirror[t][at] = g.x; mirror[t + 1][at] = g.y; mirror[t + 2][at] = g.z; mirror[t + 3][at] = g.w;
    }
  }
  __syncthreads();
  double w[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) w[v] = feat && k0 + kk + v < d ? 0.5 * pow2(-feat[k0 + kk + v]) : 0.5;
#pragma unroll
  for (int i = 0; i < TP / 8; ++i) {
    const int pp = 8 * i + (threadIdx.x >> 5);
    const long long p = p0 + pp;
    if (p >= d) break;
    const float4 g = *reinterpret_cast<const float4*>(&mirror[pp][kk ^ (pp & 28)]);
    const unsigned top = rowmax[p];
    const int e = slice_exponent<true>((double)__uint_as_float(top));
    const float a[4] = {h[i].x, h[i].y, h[i].z, h[i].w}, b[4] = {g.x, g.y, g.z, g.w};
    double x[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) x[v] = w[v] * ((double)finite(a[v]) + (double)finite(b[v]));
    if (m == 0) {
#pragma unroll
      for (int v = 0; v < 4; ++v) x[v] = k0 + kk + v > p ? 0.0 : k0 + kk + v == p ? 0.5 * x[v] : x[v];
      if ((blockIdx.x & 1) == 0 && (threadIdx.x & 31) == 0) exps[p] = e;
    }
    write_slices<true>(x, ns, e, out + (size_t)p * kp + k0 + kk, (size_t)d * kp);
  }
}

// E [d_in, d_out] fp64 -> slices of E^T [ns][d_out][kp] int8 (column j scaled by 2^-exps[j], BALANCED: row k by 2^feat[k]), 128 x 32 tiles turned round
// in shared memory so that reads and writes are contiguous, four rows of E per thread.  8 bytes read and ns
// written per entry; bound as slice_h_kernel (4096^2, five slices: 52 us, ALU pipe 63 %, 3.5 TB/s).  (32 x 32 tiles, single bytes, digits one after the other in fp64: 0.74 ms for 4096 x 32768 and
// two slices.)
constexpr int SK = 128, SJ = 32;
template <bool BALANCED>
__global__ void __launch_bounds__(256) slice_et_kernel(const double* __restrict__ E, long long d_in, long long d_out, long long kp,
                                                       const int* __restrict__ exps, const int* __restrict__ feat, int ns,
                                                       signed char* __restrict__ out) {
  // entry (k, j) at [j][k ^ 2 (j & 15)]: the stores down a column spread over the banks, pairs of k stay together
  __shared__ __align__(16) double tile[SJ][SK];
  const long long k0 = (long long)blockIdx.x * SK, j0 = (long long)blockIdx.y * SJ;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
  for (int r = ty; r < SK; r += 8) {
    const long long k = k0 + r, j = j0 + tx;
    double x = (k < d_in && j < d_out) ? E[k * d_out + j] : 0.0;
    if (BALANCED && feat && k < d_in) x *= pow2(feat[k]);
    tile[tx][r ^ (2 * (tx & 15))] = x;
  }
  __syncthreads();
#pragma unroll
  for (int jj = ty; jj < SJ; jj += 8) {
    const long long j = j0 + jj, k = k0 + 4 * tx;
    if (j >= d_out) continue;   // (k < kp: kp is a multiple of SK)
    const double2 x01 = *reinterpret_cast<const double2*>(&tile[jj][(4 * tx) ^ (2 * (jj & 15))]);
    const double2 x23 = *reinterpret_cast<const double2*>(&tile[jj][(4 * tx + 2) ^ (2 * (jj & 15))]);
    const double x[4] = {x01.x, x01.y, x23.x, x23.y};
    write_slices<BALANCED>(x, ns, exps[j], out + (size_t)j * kp + k, (size_t)d_out * kp);
  }
}

// ---------------------------------------------------------------------------------------------
// The int8 GEMM.

struct Params {
  int M, N;                 // rows of E^T (layer columns j), rows of H (coordinates p)
  int kblocks;              // K blocks of BKB bytes
  int tiles_m, tiles_n;
  int ngroups;              // groups in the order they are processed: descending i + j
  int group_first[MAX_GROUPS + 1];    // pairs [first, next first) of each group
  int group_s[MAX_GROUPS];            // i + j of the group (slices numbered from 1)
  signed char pair_e[MAX_SLICES * MAX_SLICES], pair_h[MAX_SLICES * MAX_SLICES];  // slice indices (from 0)
  double* C;                // [M, ldc] fp64
  int keep_c;               // C is wanted, else only the column dots are
  int half;                 // half of the product, the losses twice the dots
  long long ldc;
  const int* eexp;          // [M]
  const int* hexp;          // [N]
  double final_scale;       // applied with the exponents after the last group
  const double* E;          // optional, [N, lde]: with dot_part, the epilogue also sums E[p, j] C[j, p] over its columns
  long long lde;
  double* dot_part;         // [2 * tiles_n, M] partial column dots, one row per (tile column, epilogue half)
  int* status;
};

// Bounded wait of this pipeline's roles (see async_copy.cuh).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_wait_or_abort(bar, parity, abort_flag, SPIN_LIMIT);
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
// Shared-memory matrix descriptor, K-major, 128-byte swizzle: rows of 128 bytes, groups of 8
// rows 1024 bytes apart (SBO); the leading-dimension offset is not used by swizzled K-major
// layouts.  Bits [0,14) start >> 4, [16,30) LBO >> 4, [32,46) SBO >> 4, [46,48) version 1,
// [61,64) layout 2 (128-byte swizzle).
__device__ __forceinline__ uint64_t make_desc(uint32_t smem_addr) {
  return (uint64_t)((smem_addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// Instruction descriptor: int32 accumulate, signed 8-bit A and B, both K-major, N = 256, M = 128.
constexpr uint32_t IDESC = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);

__device__ __forceinline__ void mma_i8(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(IDESC), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

// Exact, and on the fp64 pipe instead of the conversion pipe.
__device__ __forceinline__ double int_to_double(uint32_t r) {
  return __hiloint2double(0x43300000, (int)(r ^ 0x80000000u)) - 4503601774854144.0;   // 2^52 + 2^31
}
// Tiles are handed out in bands of 8 tile rows, column by column inside a band, so that the
// tiles in flight at one time share their operand panels in L2.
__device__ __forceinline__ void tile_coords(int t, int tiles_m, int tiles_n, int& tm, int& tn) {
  const int band = t / (8 * tiles_n);
  const int rows = min(8, tiles_m - band * 8);
  const int tl = t - band * 8 * tiles_n;
  tn = tl / rows;
  tm = band * 8 + tl - tn * rows;
}

__global__ void __launch_bounds__(NUM_THREADS, 1)
gemm_i8_kernel(const __grid_constant__ CUtensorMap map_e, const __grid_constant__ CUtensorMap map_h, const Params p) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles = (raw + 1023u) & ~1023u;           // stage buffers, 1 KB aligned
  unsigned char* ctrl = smem_raw + (tiles - raw) + (size_t)STAGES * STAGE_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(ctrl);      // full[4] empty[4] tfull[2] tempty[2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(ctrl + 128);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(ctrl + 136);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (STAGES + s); };
  auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + b); };
  auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * STAGES + 2 + b); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar(b), 1); mbar_init(tempty_bar(b), EPI_WARPS); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;

  const int ntiles = p.tiles_m * p.tiles_n;

  if (warp == 0) {
    // ---------------- TMA producer: one stage per (pair, K block) ----------------
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int issued = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        int tm, tn;
        tile_coords(t, p.tiles_m, p.tiles_n, tm, tn);
        for (int g = 0; g < p.ngroups && ok; ++g) {
          for (int pr = p.group_first[g]; pr < p.group_first[g + 1] && ok; ++pr) {
            const int se = p.pair_e[pr], sh = p.pair_h[pr];
            const int steps = !p.half ? p.kblocks : 2 + 2 * blocks_after(tn, p.tiles_n);
            for (int it = 0; it < steps; ++it) {
              // K block of this step (half of the product: those of the diagonal block first; past the last column, zeros)
              int kb = it;
              if (p.half) {
                const int block = tn + (it >> 1);
                kb = 2 * (block < p.tiles_n ? block : block - p.tiles_n) + (it & 1);
              }
              if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag)) { ok = false; break; }
              mbar_expect_tx(full_bar(stage), STAGE_BYTES);
              const uint32_t a_dst = tiles + (uint32_t)stage * STAGE_BYTES;
              tma_load_3d(a_dst, &map_e, kb * BKB, tm * BM, se, full_bar(stage));
              tma_load_3d(a_dst + A_BYTES, &map_h, kb * BKB, tn * BN, sh, full_bar(stage));
              ++issued;
              if (++stage == STAGES) { stage = 0; phase ^= 1u; }
            }
          }
        }
      }
      if (!ok) {
        // let copies already in flight land before the CTA goes away (bounded)
        const int pending = issued < STAGES ? issued : STAGES;
        for (int q = 0; q < pending; ++q) {
          int s2 = stage - 1 - q;
          uint32_t ph2 = phase;
          if (s2 < 0) { s2 += STAGES; ph2 ^= 1u; }
          for (uint32_t it = 0; it < SPIN_LIMIT; ++it)
            if (mbar_try_wait(full_bar(s2), ph2)) break;
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: one accumulator per (tile, group) ----------------
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      int buf = 0;
      uint32_t tphase = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        int tm, tn;
        tile_coords(t, p.tiles_m, p.tiles_n, tm, tn);
        const int steps = !p.half ? p.kblocks : 2 + 2 * blocks_after(tn, p.tiles_n);
        for (int g = 0; g < p.ngroups && ok; ++g) {
          if (!mbar_wait(tempty_bar(buf), tphase ^ 1u, abort_flag)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t tmem_d = tmem_base + (uint32_t)buf * BN;
          const int nsteps = (p.group_first[g + 1] - p.group_first[g]) * steps;
          for (int it = 0; it < nsteps; ++it) {
            if (!mbar_wait(full_bar(stage), phase, abort_flag)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a_src = tiles + (uint32_t)stage * STAGE_BYTES;
            const uint32_t b_src = a_src + A_BYTES;
#pragma unroll
            for (int kk = 0; kk < BKB / 32; ++kk)   // 32 bytes of K per MMA, inside the 128-byte swizzled row
              mma_i8(tmem_d, make_desc(a_src + kk * 32), make_desc(b_src + kk * 32), (it > 0 || kk > 0) ? 1u : 0u);
            mma_commit(empty_bar(stage));   // frees the stage once these MMAs have read it
            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
          }
          if (!ok) break;
          mma_commit(tfull_bar(buf));       // accumulator complete
          if (++buf == 2) { buf = 0; tphase ^= 1u; }
        }
      }
    }
  } else {
    // ---------------- epilogue: TMEM -> fp64 running sum in C, or column dots alone ----------------
    // Two warps per TMEM lane quarter; they take the 16-column chunks of the tile in turn.  Where only the dots are wanted, every group
    // gives its own, 128^-s E . acc, and there is no running sum
    // (16 bytes per entry and group; loss of 4096 x 4096 codes 1290 -> 1001 us, 1350 x 677 291 -> 202, clipping search 4.3 -> 4.1 ms).
    const int q = warp & 3;                 // TMEM lane quarter this warp may read
    const int half = (warp - 2) >> 2;       // which of the two warps of the quarter
    const int row = q * 32 + lane;          // row of the tile
    int buf = 0;
    uint32_t tphase = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      int tm, tn;
      tile_coords(t, p.tiles_m, p.tiles_n, tm, tn);
      const long long j = (long long)tm * BM + row;
      const long long p0 = (long long)tn * BN;
      const bool row_ok = j < p.M;
      double* crow = p.C + (row_ok ? j : 0) * p.ldc;   // (read and written with keep_c only)
      const int ej = row_ok ? p.eexp[j] : 0;
      double dot = 0.0;
      for (int g = 0; g < p.ngroups && ok; ++g) {
        if (!mbar_wait(tfull_bar(buf), tphase, abort_flag)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const double w = pow2(-7 * p.group_s[g]);
        const bool first = g == 0, last = g == p.ngroups - 1;
        double part = 0.0;
#pragma unroll 1
        for (int c = half; c < BN / 16; c += 2) {
          uint32_t r[16];
          tmem_ld16(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * BN + c * 16), r);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (!row_ok) continue;
          const long long pc0 = p0 + c * 16;
          if (!p.keep_c) {
            const double* e = p.E + pc0 * p.lde + j;
            if (pc0 + 16 <= p.N) {
#pragma unroll
              for (int v = 0; v < 16; ++v) part = fma(e[v * p.lde], int_to_double(r[v]) * pow2(p.hexp[pc0 + v]), part);
            } else {
#pragma unroll
              for (int v = 0; v < 16; ++v)
                if (pc0 + v < p.N) part = fma(e[v * p.lde], int_to_double(r[v]) * pow2(p.hexp[pc0 + v]), part);
            }
          } else if (pc0 + 16 <= p.N) {
            // whole chunk inside the matrix: 16-byte accesses (ldc is a multiple of 4, pc0 of 16)
            double2* cp = reinterpret_cast<double2*>(crow + pc0);
            double x[16];
#pragma unroll
            for (int v = 0; v < 16; ++v) x[v] = w * int_to_double(r[v]);
            if (!first) {
              double2 old[8];
#pragma unroll
              for (int v = 0; v < 8; ++v) old[v] = cp[v];
#pragma unroll
              for (int v = 0; v < 8; ++v) { x[2 * v] += old[v].x; x[2 * v + 1] += old[v].y; }
            }
            if (last) {
#pragma unroll
              for (int v = 0; v < 16; ++v) x[v] = x[v] * p.final_scale * pow2(ej + p.hexp[pc0 + v]);
              if (p.dot_part) {
#pragma unroll
                for (int v = 0; v < 16; ++v) dot = fma(p.E[(pc0 + v) * p.lde + j], x[v], dot);
              }
            }
#pragma unroll
            for (int v = 0; v < 8; ++v) cp[v] = make_double2(x[2 * v], x[2 * v + 1]);
          } else {
#pragma unroll
            for (int v = 0; v < 16; ++v) {
              const long long pc = pc0 + v;
              if (pc < p.N) {
                double x = w * int_to_double(r[v]);
                if (!first) x += crow[pc];
                if (last) {
                  x = x * p.final_scale * pow2(ej + p.hexp[pc]);
                  if (p.dot_part) dot = fma(p.E[pc * p.lde + j], x, dot);
                }
                crow[pc] = x;
              }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty_bar(buf));
        dot = fma(w, part, dot);   // (the smallest group comes first)
        if (++buf == 2) { buf = 0; tphase ^= 1u; }
      }
      if (p.dot_part && row_ok && ok) p.dot_part[(size_t)(2 * tn + half) * p.M + j] = p.keep_c ? dot : dot * p.final_scale * pow2(ej);
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) atomicExch(p.status, (int)kFlagWaitTimeout);
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS)
                 : "memory");
  }
}

// col_loss[j] = inv_scale * sum_b part[b, j], b ascending: the partial column dots
// sum_p E[p, j] C[j, p] that the GEMM's epilogue leaves per (tile column, epilogue half).  The
// order of the sum is fixed, so the result does not depend on the schedule.
__global__ void __launch_bounds__(256) dot_reduce_kernel(const double* __restrict__ part, int nparts, long long m,
                                                         double inv_scale, double* __restrict__ col_loss) {
  const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= m) return;
  double v = 0.0;
  for (int b = 0; b < nparts; ++b) v += part[(size_t)b * m + j];
  col_loss[j] = v * inv_scale;
}

}  // namespace i8

// ---------------------------------------------------------------------------------------------
// Host side.

static long long tc_kpad(long long d_in) { return (d_in + 127) / 128 * 128; }

bool gemm_tc_supported(long long d_in, long long d_out) {
  // 5 slice pairs of one accumulator must stay below 2^31: 5 * K * 127^2
  return d_in >= 256 && d_out >= 128 && d_in <= 26000 && d_out < (1ll << 30);
}

// Losses by half of the product.  Short sums are bound by the slices and the epilogue: loss of given codes, whole / half (us): 257 x 16384
// 219 / 248, 512 x 8192 156 / 174, 1024 x 1024 167 / 167, 1350 x 677 195 / 189, 2048 x 2048 263 / 228, 2560 x 1024 297 / 239, 3072 x 130 314 /
// 247, 3072 x 2048 585 / 416, 4096 x 4096 1477 / 965, 5376 x 300 573 / 393, 8192 x 1024 1541 / 965.  It would be the faster one from some 1350
// rows on, but with fewer blocks the errors of given codes are up to 17 % larger (rms: 1024 x 1024 in groups 8.9e-13 -> 1.04e-12, 2048 x 512 in
// groups 1.02e-12 -> 1.06e-12; from 2560 x 512 on no larger, 4.5e-13 -> 4.2e-13).
static bool half_product(long long d_in) { return d_in >= 3072; }

size_t gemm_tc_h_bytes(long long d_in, int nh, TcUse use) {
  const size_t row_words = align_up(sizeof(int) * (size_t)d_in);
  size_t bytes = align_up((size_t)nh * d_in * tc_kpad(d_in)) + row_words;   // slices, row exponents
  if (use != kTcProduct && half_product(d_in)) bytes += row_words;                                       // row maxima
  if (use == kTcSearch && half_product(d_in)) bytes += row_words + align_up(sizeof(int));                // D, whether it was given up
  return bytes;
}
size_t gemm_tc_e_bytes(long long d_in, long long d_out, int ne) {
  return align_up(sizeof(double) * 2 * (size_t)((d_in + i8::BN - 1) / i8::BN) * (size_t)d_out) +   // partial column dots
         align_up((size_t)ne * d_out * tc_kpad(d_in)) + align_up(sizeof(int) * (size_t)d_out) +
         align_up(sizeof(unsigned long long) * (size_t)d_out);
}

// Slices of H (done once per call of the library; the OWC search reuses them for every gamma).
cudaError_t gemm_tc_prepare_h(const float* H, long long d_in, int nh, TcUse use, void* hbuf, cudaStream_t st) {
  const long long kp = tc_kpad(d_in);
  const bool half = use != kTcProduct && half_product(d_in);
  signed char* slices = (signed char*)hbuf;
  int* hexp = (int*)((char*)hbuf + align_up((size_t)nh * d_in * kp));
  if (half) {
    unsigned* rowmax = (unsigned*)((char*)hexp + align_up(sizeof(int) * (size_t)d_in));
    int* feat = use == kTcSearch ? (int*)((char*)rowmax + align_up(sizeof(int) * (size_t)d_in)) : nullptr;
    int* without = feat ? (int*)((char*)feat + align_up(sizeof(int) * (size_t)d_in)) : nullptr;
    const int nb = (int)((d_in + i8::BN - 1) / i8::BN);
    const int rows = d_in < 6144 ? 16 : 64;   // few fill the SMs, many spare atomics (8192^2 with 16 rows 95 us, with 64 56)
    const dim3 grid_m((unsigned)((d_in + 1023) / 1024), (unsigned)((d_in + rows - 1) / rows)), grid_s(8, 1 + nb / 2, (unsigned)nb);
    cudaError_t e = cudaMemsetAsync(rowmax, 0, sizeof(int) * (size_t)d_in, st);
    if (e != cudaSuccess) return e;
    if (feat) { i8::feature_exp_kernel<<<(unsigned)((d_in + 255) / 256), 256, 0, st>>>(H, d_in, feat); count_launch(); }
    auto run = [&](auto scaled_kern, auto max_kern, auto slice_kern) {
      if (feat) {
        { scaled_kern<<<grid_m, 256, 0, st>>>(H, d_in, feat, nullptr, rows, rowmax); count_launch(); }
        { i8::feature_check_kernel<<<1, 1024, 0, st>>>(d_in, feat, rowmax, without); count_launch(); }
      }
      { max_kern<<<grid_m, 256, 0, st>>>(H, d_in, nullptr, without, rows, rowmax); count_launch(); }
      { slice_kern<<<grid_s, 256, 0, st>>>(H, d_in, kp, feat, rowmax, nh, hexp, slices); count_launch(); }
    };
    if (d_in % 4 == 0) run(i8::half_max_kernel<true, true>, i8::half_max_kernel<true, false>, i8::half_slice_kernel<true>);
    else run(i8::half_max_kernel<false, true>, i8::half_max_kernel<false, false>, i8::half_slice_kernel<false>);
  } else {
    const dim3 grid((unsigned)((kp / 4 + 127) / 128), (unsigned)d_in);
    { i8::row_exp_f32_kernel<<<(unsigned)d_in, 256, 0, st>>>(H, d_in, d_in, hexp); count_launch(); }
    { i8::slice_h_kernel<<<grid, 128, 0, st>>>(H, d_in, kp, hexp, nh, slices); count_launch(); }
  }
  return cudaGetLastError();
}

static cudaError_t encode_map3(CUtensorMap* map, const void* base, long long kp, long long rows, int ns, int box_rows) {
  typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                               const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                               CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static EncodeFn encode = nullptr;
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    cudaError_t ge = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
    if (ge != cudaSuccess) return ge;
    if (qres != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    encode = (EncodeFn)fn;
  }
  const cuuint64_t gdim[3] = {(cuuint64_t)kp, (cuuint64_t)rows, (cuuint64_t)ns};
  const cuuint64_t gstride[2] = {(cuuint64_t)kp, (cuuint64_t)kp * (cuuint64_t)rows};
  const cuuint32_t box[3] = {(cuuint32_t)i8::BKB, (cuuint32_t)box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult cr = encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<void*>(base), gdim, gstride, box, estr,
                             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return cr == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// E = the residual of `src`, then C[j, p] = scale * sum_k E[k, j] H[p, k]  for j < d_out, p < d_in, to the precision of
// (ne, nh, smax); optionally col_loss[j] = sum_p E[p, j] C[j, p] / scale.
// hbuf: from gemm_tc_prepare_h with the same nh and use.  ebuf: gemm_tc_e_bytes of scratch.
cudaError_t gemm_tc_run(const void* hbuf, int nh, TcUse use, const ResidualSrc& src, double* E, long long d_in, long long d_out, int ne, int smax,
                        double scale, double* C, long long ldc, double* col_loss, void* ebuf, cudaStream_t st) {
  using namespace i8;
  if (nh < 1 || nh > MAX_SLICES || ne < 1 || ne > MAX_SLICES || smax < 2) return cudaErrorInvalidValue;
  const long long kp = tc_kpad(d_in);
  const bool keep_c = use == kTcProduct, half = !keep_c && half_product(d_in);
  const signed char* hsl = (const signed char*)hbuf;
  const int* hexp = (const int*)((const char*)hbuf + align_up((size_t)nh * d_in * kp));
  const int* feat = half && use == kTcSearch ? (const int*)((const char*)hexp + 2 * align_up(sizeof(int) * (size_t)d_in)) : nullptr;
  signed char* esl = (signed char*)ebuf;
  int* eexp = (int*)((char*)ebuf + align_up((size_t)ne * d_out * kp));
  unsigned long long* colmax = (unsigned long long*)((char*)eexp + align_up(sizeof(int) * (size_t)d_out));
  double* dot_part = (double*)((char*)colmax + align_up(sizeof(unsigned long long) * (size_t)d_out));

  cudaError_t e = cudaMemsetAsync(colmax, 0, sizeof(unsigned long long) * (size_t)d_out, st);
  if (e != cudaSuccess) return e;
  e = launch_residual_f64(src, d_in, E, st, colmax, feat);
  if (e != cudaSuccess) return e;
  const unsigned cols = (unsigned)((d_out + 255) / 256);
  if (half) col_exp_kernel<true><<<cols, 256, 0, st>>>(colmax, d_out, eexp);
  else col_exp_kernel<false><<<cols, 256, 0, st>>>(colmax, d_out, eexp);
  count_launch();
  const dim3 slices((unsigned)(kp / SK), (unsigned)((d_out + SJ - 1) / SJ));
  if (half) slice_et_kernel<true><<<slices, 256, 0, st>>>(E, d_in, d_out, kp, eexp, feat, ne, esl);
  else slice_et_kernel<false><<<slices, 256, 0, st>>>(E, d_in, d_out, kp, eexp, nullptr, ne, esl);
  count_launch();
  Params p{};
  p.M = (int)d_out; p.N = (int)d_in; p.kblocks = (int)(kp / BKB);
  p.tiles_m = (int)((d_out + BM - 1) / BM); p.tiles_n = (int)((d_in + BN - 1) / BN);
  int npairs = 0, ng = 0;
  for (int s = smax; s >= 2; --s) {
    const int first = npairs;
    for (int i = 1; i <= ne; ++i) {
      const int j = s - i;
      if (j >= 1 && j <= nh) { p.pair_e[npairs] = (signed char)(i - 1); p.pair_h[npairs] = (signed char)(j - 1); ++npairs; }
    }
    if (npairs > first) {
      if (ng >= MAX_GROUPS) return cudaErrorInvalidValue;
      if ((long long)(npairs - first) * kp * 16129ll >= (1ll << 31)) return cudaErrorInvalidValue;
      p.group_first[ng] = first; p.group_s[ng] = s; ++ng;
    }
  }
  if (ng == 0) return cudaErrorInvalidValue;
  p.group_first[ng] = npairs;
  p.ngroups = ng;
  p.C = C; p.keep_c = keep_c ? 1 : 0; p.half = half ? 1 : 0; p.ldc = ldc; p.eexp = eexp; p.hexp = hexp; p.final_scale = scale;
  p.E = E; p.lde = d_out; p.dot_part = col_loss ? dot_part : nullptr;
  p.status = device_status_word();
  if (!p.status) return cudaErrorInvalidSymbol;

  CUtensorMap map_e, map_h;
  e = encode_map3(&map_e, esl, kp, d_out, ne, BM);
  if (e != cudaSuccess) return e;
  e = encode_map3(&map_h, hsl, kp, d_in, nh, BN);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  e = cudaFuncSetAttribute(gemm_i8_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int ntiles = p.tiles_m * p.tiles_n;
  { gemm_i8_kernel<<<ntiles < sms ? ntiles : sms, NUM_THREADS, SMEM_BYTES, st>>>(map_e, map_h, p); count_launch(); }
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (col_loss) {
    { dot_reduce_kernel<<<(unsigned)((d_out + 255) / 256), 256, 0, st>>>(dot_part, 2 * p.tiles_n, d_out, (half ? 2.0 : 1.0) / scale, col_loss); count_launch(); }
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace cdq
