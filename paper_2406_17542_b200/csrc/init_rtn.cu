// Grid and round-to-nearest codes (paper: Eq. 2), with the OWC grid search over the
// clipping strength gamma (the minimisation stated after Eq. 2).
//
//   min/max per (group, column)  ->  b = min, a = fp32(gamma (max-min) / L)
//   q = clamp(round_half_even((w - b) / a), 0, L)      (decided in fp64)
//   OWC: loss_k[j] = e_k^T H e_k for every gamma_k, argmin over k per column.
#include <type_traits>

#include "common.cuh"
#include "rtn_code.cuh"

namespace cdq {

constexpr int kChunkRows = 128;  // rows of one min/max partial

// V neighbouring weights of one row as floats (V = 4: one 8- or 16-byte load).
template <int V, bool BF16>
__device__ __forceinline__ void load_weights(const void* __restrict__ W, long long idx, float (&w)[V]) {
  if constexpr (V == 4 && BF16) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>((const __nv_bfloat16*)W + idx));
    w[0] = __uint_as_float(u.x << 16); w[1] = __uint_as_float(u.x & 0xFFFF0000u);
    w[2] = __uint_as_float(u.y << 16); w[3] = __uint_as_float(u.y & 0xFFFF0000u);
  } else if constexpr (V == 4) {
    const float4 f = __ldg(reinterpret_cast<const float4*>((const float*)W + idx));
    w[0] = f.x; w[1] = f.y; w[2] = f.z; w[3] = f.w;
  } else if constexpr (BF16) {
    w[0] = __bfloat162float(((const __nv_bfloat16*)W)[idx]);
  } else {
    w[0] = ((const float*)W)[idx];
  }
}
// Four columns per thread: rows of W, and of what is d_out wide, have to start on the vector's boundaries.
static bool four_columns(const Layer& ly) {
  const size_t esz = ly.wt == CDQ_BF16 ? 2 : 4;
  return ly.d_out % 4 == 0 && ly.ldw % 4 == 0 && reinterpret_cast<uintptr_t>(ly.W) % (4 * esz) == 0;
}

template <int V, bool BF16>
__global__ void minmax_partial_kernel(const void* __restrict__ W, long long d_out,
                                      long long ldw, long long g, long long cpg, float* __restrict__ pmn,
                                      float* __restrict__ pmx) {
  const long long j = V * (blockIdx.x * (long long)blockDim.x + threadIdx.x);
  const long long chunk = blockIdx.y;  // global chunk id = t * cpg + c
  if (j >= d_out) return;
  const long long t = chunk / cpg, c = chunk % cpg;
  const long long i0 = t * g + c * kChunkRows;
  long long i1 = i0 + kChunkRows;
  if (i1 > (t + 1) * g) i1 = (t + 1) * g;
  float mn[V], mx[V];
  load_weights<V, BF16>(W, i0 * ldw + j, mn);
#pragma unroll
  for (int v = 0; v < V; ++v) mx[v] = mn[v];
#pragma unroll 16
  for (long long i = i0 + 1; i < i1; ++i) {
    float w[V];
    load_weights<V, BF16>(W, i * ldw + j, w);
#pragma unroll
    for (int v = 0; v < V; ++v) { mn[v] = fminf(mn[v], w[v]); mx[v] = fmaxf(mx[v], w[v]); }
  }
#pragma unroll
  for (int v = 0; v < V; ++v) { pmn[chunk * d_out + j + v] = mn[v]; pmx[chunk * d_out + j + v] = mx[v]; }
}
static void run_minmax_partial(const Layer& ly, long long cpg, float* pmn, float* pmx, cudaStream_t st) {
  // (narrow layers: a column per thread, or there are too few threads to hide the latency of the loads: 4096 x 2048 weights in groups of 64,
  // 2^17 columns and chunks, 14.5 us against 16.9 with four columns, 4096 x 4096 20.6 / 26.4; 4096 x 4096 in groups of 16, 2^20, 35 / 14)
  const int v = four_columns(ly) && ly.d_out * ly.ng * cpg >= (1 << 18) ? 4 : 1;
  const dim3 grid((unsigned)((ly.d_out + 128 * v - 1) / (128 * v)), (unsigned)(ly.ng * cpg));
  auto run = [&](auto kern) { kern<<<grid, 128, 0, st>>>(ly.W, ly.d_out, ly.ldw, ly.g, cpg, pmn, pmx); };
  if (ly.wt == CDQ_BF16) run(v == 4 ? minmax_partial_kernel<4, true> : minmax_partial_kernel<1, true>);
  else run(v == 4 ? minmax_partial_kernel<4, false> : minmax_partial_kernel<1, false>);
  count_launch();
}

__global__ void minmax_final_kernel(const float* __restrict__ pmn, const float* __restrict__ pmx, long long ng,
                                    long long d_out, long long cpg, float* __restrict__ mn_out,
                                    float* __restrict__ mx_out) {
  const long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long t = blockIdx.y;
  if (j >= d_out) return;
  float mn = pmn[(t * cpg) * d_out + j], mx = pmx[(t * cpg) * d_out + j];
  for (long long c = 1; c < cpg; ++c) {
    mn = fminf(mn, pmn[(t * cpg + c) * d_out + j]);
    mx = fmaxf(mx, pmx[(t * cpg + c) * d_out + j]);
  }
  mn_out[t * d_out + j] = mn;
  mx_out[t * d_out + j] = mx;
}

// a = fp32((gamma * (max - min)) / L) in fp64, b = min.  gamma per column (gam != NULL) or 1.
__global__ void scale_zero_kernel(const float* __restrict__ mn, const float* __restrict__ mx, long long ng,
                                  long long d_out, int L, const double* __restrict__ gam,
                                  float* __restrict__ scale, float* __restrict__ zero) {
  const long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long t = blockIdx.y;
  if (j >= d_out) return;
  const double lo = (double)mn[t * d_out + j], hi = (double)mx[t * d_out + j];
  const double gamma = gam ? gam[j] : 1.0;
  const double a = __ddiv_rn(__dmul_rn(gamma, __dadd_rn(hi, -lo)), (double)L);
  scale[t * d_out + j] = (float)a;
  zero[t * d_out + j] = (float)lo;
}

// Codes of kCodeRows rows of one group by V columns per thread (see rtn_code).  Bound by instructions (14336 x 16384 bf16 weights in
// groups of 256: 208 us, 22 instructions per weight, issue slots 70 % busy, 3.3 TB/s): as many weights
// took 1180 us with an fp64 division and one byte per thread.
constexpr int kCodeRows = 16;
template <int V, bool BF16>
__global__ void __launch_bounds__(128) rtn_codes_kernel(const void* __restrict__ W, long long d_out,
                                                        long long ldw, long long g, int blocks_per_group, int L,
                                                        const float* __restrict__ scale, const float* __restrict__ zero,
                                                        unsigned char* __restrict__ Q) {
  const long long j = V * (blockIdx.x * (long long)blockDim.x + threadIdx.x);
  if (j >= d_out) return;
  const long long t = blockIdx.y / blocks_per_group, i0 = t * g + (blockIdx.y % blocks_per_group) * (long long)kCodeRows;
  const long long i1 = min(i0 + kCodeRows, (t + 1) * g);
  float a[V], b[V], inv[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    a[v] = scale[t * d_out + j + v];
    b[v] = zero[t * d_out + j + v];
    inv[v] = rtn_inverse_or_zero(a[v]);
  }
  constexpr int R = 8;   // rows whose loads are in flight together (the compiler moves no load past the branch of rtn_code)
  for (long long i = i0; i < i1; i += R) {
    float w[R][V];
#pragma unroll
    for (int r = 0; r < R; ++r) load_weights<V, BF16>(W, min(i + r, i1 - 1) * ldw + j, w[r]);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (i + r >= i1) break;
      if constexpr (V == 4) *reinterpret_cast<unsigned*>(Q + (i + r) * d_out + j) = rtn_code4(w[r], a, inv, b, (float)L);
      else Q[(i + r) * d_out + j] = (unsigned char)(a[0] > 0.f ? rtn_code(w[r][0], a[0], inv[0], b[0], (float)L) : 0u);
    }
  }
}

// Grid and codes of one group of at most 8 WARPS rows for 128 columns, without a clipping search: the weights are read once and stay in
// registers, eight rows of four columns per thread, while the block's warps put their minima and maxima together.  14336 x 16384
// weights in groups of 128, against three passes: bf16 336 -> 265 us (2.7 TB/s), fp32 399 -> 271 (4.3).  Bound by instructions and by what a
// block's warps wait for together (bf16: 27 instructions per weight, issue slots 67 % busy, 26 warps per SM; the first loads and the barrier around
// the divisions are the first stalls).  At 64 registers fp32 weights spill 124 bytes per thread, bf16 20 to 24.
template <int WARPS, bool BF16>
__global__ void __launch_bounds__(32 * WARPS, 1024 / (32 * WARPS)) group_codes_kernel(const void* __restrict__ W, long long d_out, long long ldw, long long g, int L,
                                                          float* __restrict__ scale, float* __restrict__ zero,
                                                          unsigned char* __restrict__ Q) {
  constexpr int ROWS = 8;
  __shared__ __align__(16) float s_mn[WARPS][128], s_mx[WARPS][128], s_a[128], s_b[128], s_inv[128];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long j0 = blockIdx.x * 128ll, j = j0 + 4 * lane, t = blockIdx.y, i1 = (t + 1) * g, i0 = t * g + warp * ROWS;
  const bool inside = j < d_out;   // (d_out is a multiple of four)
  using Four = std::conditional_t<BF16, uint2, float4>;   // four weights as they lie in memory
  Four w[ROWS];
#pragma unroll
  for (int r = 0; r < ROWS; ++r)
    w[r] = __ldg(reinterpret_cast<const Four*>((const char*)W + (min(i0 + r, i1 - 1) * ldw + (inside ? j : 0)) * (BF16 ? 2 : 4)));
  auto widen = [](const Four& f, float (&x)[4]) {
    if constexpr (BF16) {
      x[0] = __uint_as_float(f.x << 16); x[1] = __uint_as_float(f.x & 0xFFFF0000u);
      x[2] = __uint_as_float(f.y << 16); x[3] = __uint_as_float(f.y & 0xFFFF0000u);
    } else {
      x[0] = f.x; x[1] = f.y; x[2] = f.z; x[3] = f.w;
    }
  };
  float4 mn, mx;
  if constexpr (BF16) {   // two at a time
    uint2 lo = w[0], hi = w[0];
#pragma unroll
    for (int r = 1; r < ROWS; ++r) {
      asm("min.bf16x2 %0, %0, %1;" : "+r"(lo.x) : "r"(w[r].x)); asm("min.bf16x2 %0, %0, %1;" : "+r"(lo.y) : "r"(w[r].y));
      asm("max.bf16x2 %0, %0, %1;" : "+r"(hi.x) : "r"(w[r].x)); asm("max.bf16x2 %0, %0, %1;" : "+r"(hi.y) : "r"(w[r].y));
    }
    float x[4];
    widen(lo, x); mn = make_float4(x[0], x[1], x[2], x[3]);
    widen(hi, x); mx = make_float4(x[0], x[1], x[2], x[3]);
  } else {
    mn = mx = w[0];
#pragma unroll
    for (int r = 1; r < ROWS; ++r) {
      mn.x = fminf(mn.x, w[r].x); mn.y = fminf(mn.y, w[r].y); mn.z = fminf(mn.z, w[r].z); mn.w = fminf(mn.w, w[r].w);
      mx.x = fmaxf(mx.x, w[r].x); mx.y = fmaxf(mx.y, w[r].y); mx.z = fmaxf(mx.z, w[r].z); mx.w = fmaxf(mx.w, w[r].w);
    }
  }
  *reinterpret_cast<float4*>(&s_mn[warp][4 * lane]) = mn;
  *reinterpret_cast<float4*>(&s_mx[warp][4 * lane]) = mx;
  __syncthreads();
  if (threadIdx.x < 128) {
    const int c = threadIdx.x;
    float lo = s_mn[0][c], hi = s_mx[0][c];
#pragma unroll
    for (int k = 1; k < WARPS; ++k) { lo = fminf(lo, s_mn[k][c]); hi = fmaxf(hi, s_mx[k][c]); }
    // as scale_zero_kernel with a clipping strength of one
    const float a = (float)__ddiv_rn(__dadd_rn((double)hi, -(double)lo), (double)L);
    s_a[c] = a; s_b[c] = lo; s_inv[c] = rtn_inverse_or_zero(a);
    if (j0 + c < d_out) { scale[t * d_out + j0 + c] = a; zero[t * d_out + j0 + c] = lo; }
  }
  __syncthreads();
  if (!inside) return;
  const float4 a4 = *reinterpret_cast<const float4*>(&s_a[4 * lane]), b4 = *reinterpret_cast<const float4*>(&s_b[4 * lane]);
  const float4 v4 = *reinterpret_cast<const float4*>(&s_inv[4 * lane]);
  const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w}, inv[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    float x[4];
    widen(w[r], x);
    if (i0 + r < i1) *reinterpret_cast<unsigned*>(Q + (i0 + r) * d_out + j) = rtn_code4(x, a, inv, b, (float)L);
  }
}

// Residual E[i][c] = (a q + b) - w in fp64, either from stored codes or, for the OWC search, from min/max and a clipping
// strength (codes formed on the fly, never stored).  With colmax it also leaves the largest |E| 2^row_exp of every column there (as
// ordered bit patterns, zeroed by the caller), which the slicing of the int8 product needs.  8 bytes written
// per entry; bound by the latency of its loads (4096 x 4096 bf16 weights in groups: 43 us, 13 warps per SM at 97 registers, 3.0 TB/s).
// (One entry per thread with an fp64 division, and the maxima by a pass of their own over E: 1.0 ms for eight
// strengths of a 4096 x 4096 layer, 0.16 ms of them the maxima.)
template <int V, bool BF16>
__global__ void __launch_bounds__(128) residual_kernel(ResidualSrc s, int rows_per_block, int blocks_per_group, double* __restrict__ E,
                                                       unsigned long long* __restrict__ colmax, const int* __restrict__ row_exp) {
  const long long c = V * (blockIdx.x * (long long)blockDim.x + threadIdx.x);   // column of E
  const long long width = s.n_cols ? s.n_cols : s.d_out;
  if (c >= width) return;
  const long long j = s.col_idx ? (long long)s.col_idx[c] : c % s.d_out;        // column of the layer
  const long long t = blockIdx.y / blocks_per_group, i0 = t * s.g + (blockIdx.y % blocks_per_group) * (long long)rows_per_block;
  const long long i1 = min(i0 + rows_per_block, (t + 1) * s.g);
  float a[V], b[V], inv[V];
  double m[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    m[v] = 0.0;
    if (s.use_gamma) {
      const double lo = (double)s.mn[t * s.d_out + j + v], hi = (double)s.mx[t * s.d_out + j + v];
      const double gamma = s.col_gamma ? s.gammas[s.col_gamma[c + v]] : s.n_cols ? s.gammas[s.k0 + c / s.d_out] : s.gamma;
      a[v] = (float)__ddiv_rn(__dmul_rn(gamma, __dadd_rn(hi, -lo)), (double)s.L);
      b[v] = (float)lo;
      inv[v] = rtn_inverse_or_zero(a[v]);
    } else {
      a[v] = s.scale[t * s.d_out + j + v];
      b[v] = s.zero[t * s.d_out + j + v];
    }
  }
  constexpr int R = 4;   // rows whose loads are in flight together (the compiler moves no load past the branch of rtn_code)
  for (long long i = i0; i < i1; i += R) {
    float w[R][V];
    unsigned q4[R];
    int weight[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const long long row = min(i + r, i1 - 1);
      weight[r] = row_exp ? row_exp[row] : 0;
      load_weights<V, BF16>(s.W, row * s.ldw + j, w[r]);
      q4[r] = 0u;
      if (!s.use_gamma) {
        if constexpr (V == 4) q4[r] = *reinterpret_cast<const unsigned*>(s.Q + row * s.d_out + j);
        else q4[r] = s.Q[row * s.d_out + j];
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (i + r >= i1) break;
      double e[V];
      if (s.use_gamma) {
        if constexpr (V == 4) q4[r] = rtn_code4(w[r], a, inv, b, (float)s.L);
        else q4[r] = a[0] > 0.f ? rtn_code(w[r][0], a[0], inv[0], b[0], (float)s.L) : 0u;
      }
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const unsigned q = (q4[r] >> (8 * v)) & 255u;
        // 2^52 + q: its lower word is q
        const double qd = __hiloint2double(0x43300000, (int)q) - 4503599627370496.0;
        e[v] = __dadd_rn(__dadd_rn(__dmul_rn((double)a[v], qd), (double)b[v]), -(double)w[r][v]);
        m[v] = fmax(m[v], fabs(e[v]) * __hiloint2double((1023 + weight[r]) << 20, 0));
      }
      double* dst = E + (i + r) * width + c;
      if constexpr (V == 4) {
        *reinterpret_cast<double2*>(dst) = make_double2(e[0], e[1]);
        *reinterpret_cast<double2*>(dst + 2) = make_double2(e[2], e[3]);
      } else {
        dst[0] = e[0];
      }
    }
  }
  if (colmax) {
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (isfinite(m[v])) atomicMax(&colmax[c + v], (unsigned long long)__double_as_longlong(m[v]));   // >= 0: bits order like values
  }
}

cudaError_t launch_residual_f64(const ResidualSrc& src, long long d_in, double* E, cudaStream_t st, unsigned long long* colmax,
                                const int* row_exp) {
  const long long width = src.n_cols ? src.n_cols : src.d_out;
  // rows per block, all of one group: few on small layers, which have no more blocks to offer (1024 x 1024 entries with 32 rows 17 us)
  const int rows = width * d_in >= (1ll << 22) ? 32 : 4, bpg = (int)((src.g + rows - 1) / rows);
  const size_t esz = src.wt == CDQ_BF16 ? 2 : 4;
  // four columns per thread: rows of W, Q and E on the vectors' boundaries, four neighbouring columns of one strength, and 32 rows per
  // block (residual of codes with column maxima, one column against four, us: 1024 x 1024 entries with four rows per block 8.0 / 14.1, 2048 x
  // 1024 11.6 / 25.5, 4096 x 256 14.0 / 43.2; 2048 x 2048 with 32 rows 21.0 / 15.8, 2048 x 4096 37.9 / 22.9, 4096 x 4096 60.5 / 49.7)
  const bool four = rows == 32 && !src.col_idx && src.d_out % 4 == 0 && src.ldw % 4 == 0 && reinterpret_cast<uintptr_t>(src.W) % (4 * esz) == 0 &&
                    reinterpret_cast<uintptr_t>(src.Q) % 4 == 0;
  const dim3 grid((unsigned)((width + (four ? 511 : 127)) / (four ? 512 : 128)), (unsigned)(d_in / src.g * bpg));
  auto run = [&](auto kern) { kern<<<grid, 128, 0, st>>>(src, rows, bpg, E, colmax, row_exp); count_launch(); };
  if (src.wt == CDQ_BF16) run(four ? residual_kernel<4, true> : residual_kernel<1, true>);
  else run(four ? residual_kernel<4, false> : residual_kernel<1, false>);
  return cudaGetLastError();
}

// Per column: index of the smallest loss (lowest index on ties) and its gamma.
__global__ void owc_argmin_kernel(const double* __restrict__ table, int n_clip, long long d_out,
                                  const double* __restrict__ gammas, double* __restrict__ gam_col,
                                  float* __restrict__ gamma_out) {
  const long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (j >= d_out) return;
  double best = table[j];
  int bk = 0;
  for (int k = 1; k < n_clip; ++k) {
    const double v = table[(long long)k * d_out + j];
    if (v < best) { best = v; bk = k; }
  }
  gam_col[j] = gammas[bk];
  if (gamma_out) gamma_out[j] = (float)gammas[bk];
}

// ---- screening of the clipping search (production mode, tensor-core losses) ----
// The losses of all clipping strengths are first formed cheaply (three slice-pair products instead of thirteen);
// a strength stays a candidate of a column if its screened loss is within kScreenBand of the column's smallest.
// Only candidates get the thirteen-pair loss, and the argmin is taken over those: the same result as the full
// table as long as the screening errors of a column's strengths differ by less than the band.  The loss as a function of the strength is
// smooth with one minimum, and the second-best strength of a column is typically percents away (median 2.5 % on 2-bit,
// 5 % on 3-bit grouped layers), so a band of 1 % keeps 1.1 to 1.3 candidates per column.  The screen keeps two
// 7-bit slices of the residual and of H on grids of up to 4 bits: it cuts off 2^-14 of the column's largest residual, and a clipped
// weight leaves a residual up to (1 - gamma) L times the typical rounding error (7.5 times at 4 bits).  Against 64 bits, on layers of 3072 and
// 4096 rows with 2 to 4 bits, heavy weights among them, a screened loss is off by up to 4.2e-3 (3.4e-4 to 4.7e-4 rms), and the errors of a
// column's strengths differ by up to 5.4e-3: half of the band.  (Below 3072 rows, by the whole product of truncated slices, up to 6.7e-3, 6e-4
// to 9e-4 rms, and they differ by up to 7.9e-3.  By half of the product with truncated slices it was 1.0e-2, 1.3e-3 and 1.2e-2; rows of H that one
// feature dominates lost strengths.)  Finer grids (L up to 255) keep three slices and six products: up to 3e-5.
constexpr double kScreenBand = 1e-2;
__host__ __device__ constexpr int screen_slices(int bits) { return bits <= 4 ? 2 : 3; }   // pairs up to i + j = slices + 1

// mask[k][j] = 1 for candidates; the table starts at +inf everywhere.
__global__ void owc_candidates_kernel(const double* __restrict__ screen, int n_clip, long long d_out,
                                      unsigned char* __restrict__ mask, double* __restrict__ table) {
  const long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (j >= d_out) return;
  double best = screen[j];
  for (int k = 1; k < n_clip; ++k) best = fmin(best, screen[(long long)k * d_out + j]);
  const double lim = best + kScreenBand * fabs(best);
  for (int k = 0; k < n_clip; ++k) {
    mask[(long long)k * d_out + j] = screen[(long long)k * d_out + j] <= lim ? 1 : 0;
    table[(long long)k * d_out + j] = __longlong_as_double(0x7FF0000000000000ll);
  }
}

// One CTA per clipping strength: its candidate columns in ascending order; cnt[k] = their number.
__global__ void __launch_bounds__(1024) owc_compact_kernel(const unsigned char* __restrict__ mask, long long d_out,
                                                           int* __restrict__ idx, int* __restrict__ cnt) {
  __shared__ int s_scan[1024];
  __shared__ int s_base;
  const int k = blockIdx.x, tid = threadIdx.x;
  const unsigned char* m = mask + (long long)k * d_out;
  int* out = idx + (long long)k * (d_out + 128);
  if (tid == 0) s_base = 0;
  __syncthreads();
  for (long long j0 = 0; j0 < d_out; j0 += 1024) {
    const long long j = j0 + tid;
    const int f = (j < d_out && m[j]) ? 1 : 0;
    s_scan[tid] = f;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
      const int v = tid >= o ? s_scan[tid - o] : 0;
      __syncthreads();
      s_scan[tid] += v;
      __syncthreads();
    }
    if (f) out[s_base + s_scan[tid] - 1] = (int)j;
    __syncthreads();
    if (tid == 0) s_base += s_scan[1023];
    __syncthreads();
  }
  if (tid == 0) cnt[k] = s_base;
}

// The candidates of all strengths as one list of (column, strength) in the order of the strengths, so that the
// exact losses take a few wide products instead of one narrow product per strength.  off[k]: where strength k's
// candidates start (off[n_clip] = their total); entries from the total up to `padded` (a multiple of 128, the
// granularity of the tensor-core product) repeat the last candidate.
struct OwcOffsets { int off[257]; };
__global__ void owc_concat_kernel(const int* __restrict__ idx, long long d_out, OwcOffsets offs, int n_clip, int padded,
                                  int* __restrict__ cj, int* __restrict__ ck) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= padded) return;
  const int total = offs.off[n_clip];
  const int cc = c < total ? c : total - 1;
  int k = 0;
  while (k + 1 < n_clip && offs.off[k + 1] <= cc) ++k;
  cj[c] = idx[(long long)k * (d_out + 128) + (cc - offs.off[k])];
  ck[c] = k;
}

__global__ void owc_scatter_kernel(const double* __restrict__ loss_c, const int* __restrict__ cj, const int* __restrict__ ck,
                                   int n, long long d_out, double* __restrict__ table) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < n) table[(long long)ck[c] * d_out + cj[c]] = loss_c[c];   // padding repeats a candidate with its own value
}

__global__ void fill_gamma_kernel(float* gamma_out, long long d_out) {
  const long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (j < d_out) gamma_out[j] = 1.0f;
}

long long minmax_chunks(long long g) { return (g + kChunkRows - 1) / kChunkRows; }

// Group minima and maxima of every column: mn, mx [ng, d_out]; pmn, pmx [ng * minmax_chunks(g), d_out] scratch.
cudaError_t launch_group_minmax(const Layer& ly, float* pmn, float* pmx, float* mn, float* mx, cudaStream_t st) {
  const long long cpg = minmax_chunks(ly.g);
  const unsigned bx = (unsigned)((ly.d_out + 127) / 128);
  run_minmax_partial(ly, cpg, pmn, pmx, st);
  { minmax_final_kernel<<<dim3(bx, (unsigned)ly.ng), 128, 0, st>>>(pmn, pmx, ly.ng, ly.d_out, cpg, mn, mx); count_launch(); }
  return cudaGetLastError();
}

// Workspace layout (all blocks 256-byte aligned):
//   pmn, pmx : [ng*cpg, d_out] f32     mn, mx : [ng, d_out] f32
//   OWC only : gammas [n_clip] f64, gam_col [d_out] f64, table [n_clip, d_out] f64,
//              E [d_in, d_out] f64, loss partials (FAST) or the product H E (VERIFY)
struct InitWs {
  size_t pmn, pmx, mn, mx, gammas, gam_col, table, E, part, hbuf, ebuf, screen, mask, idx, cnt, loss_c, cj, ck, total;
  bool screened;    // cheap losses first, exact ones for the near-tied strengths only
  int sbatch;       // strengths per screening product (several on small layers, where a product per strength is launch-bound)
  long long wcap;   // columns that E and the slice buffers hold
  bool tc;          // losses on the int8 tensor cores
};
static InitWs init_ws_layout(long long d_in, long long d_out, long long g, int n_clip, cdq_mode mode) {
  InitWs w{};
  const long long ng = d_in / g;
  const long long cpg = minmax_chunks(g);
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += align_up(bytes); return o; };
  w.pmn = take(sizeof(float) * ng * cpg * d_out);
  w.pmx = take(sizeof(float) * ng * cpg * d_out);
  w.mn = take(sizeof(float) * ng * d_out);
  w.mx = take(sizeof(float) * ng * d_out);
  if (n_clip > 1) {
    w.gammas = take(sizeof(double) * n_clip);
    w.gam_col = take(sizeof(double) * d_out);
    w.table = take(sizeof(double) * n_clip * d_out);
    w.tc = mode == CDQ_MODE_FAST && gemm_tc_supported(d_in, d_out);
    w.screened = w.tc && n_clip >= 4;
    w.sbatch = 1;
    if (w.screened) {   // up to 1 GiB of residuals per product
      const long long fit = (1ll << 30) / (8 * d_in * d_out);
      w.sbatch = (int)(fit < 1 ? 1 : (fit > n_clip ? n_clip : fit));
    }
    w.wcap = d_out + 128 > (long long)w.sbatch * d_out ? d_out + 128 : (long long)w.sbatch * d_out;
    w.E = take(sizeof(double) * d_in * w.wcap);
    w.part = take(sizeof(double) * (mode == CDQ_MODE_FAST ? gemm_partials_elems(d_in, d_out) : (size_t)d_in * d_out));
    if (w.tc) {
      w.hbuf = take(gemm_tc_h_bytes(d_in, kTcLossNH, kTcSearch));
      w.ebuf = take(gemm_tc_e_bytes(d_in, w.wcap, kTcLossNE));
      if (w.screened) {
        w.screen = take(sizeof(double) * n_clip * d_out);
        w.mask = take((size_t)n_clip * d_out);
        w.idx = take(sizeof(int) * (size_t)n_clip * (d_out + 128));
        w.cnt = take(sizeof(int) * n_clip);
        w.loss_c = take(sizeof(double) * w.wcap);
        w.cj = take(sizeof(int) * ((size_t)n_clip * d_out + 128));
        w.ck = take(sizeof(int) * ((size_t)n_clip * d_out + 128));
      }
    }
  }
  w.total = off;
  return w;
}

size_t init_rtn_workspace(long long d_in, long long d_out, long long g, int n_clip, cdq_mode mode) {
  return init_ws_layout(d_in, d_out, g, n_clip, mode).total;
}

cudaError_t launch_init_rtn(const Layer& ly, const cdq_grid_desc& grid, float* scale, float* zero,
                            unsigned char* Q, float* gamma_out, cdq_mode mode, void* ws, cudaStream_t st) {
  const long long d_in = ly.d_in, d_out = ly.d_out, g = ly.g, ng = ly.ng;
  const long long cpg = minmax_chunks(g);
  const int n_clip = grid.n_clip > 1 ? grid.n_clip : 1;
  const InitWs L = init_ws_layout(d_in, d_out, g, n_clip, mode);
  char* base = (char*)ws;
  float* pmn = (float*)(base + L.pmn);
  float* pmx = (float*)(base + L.pmx);
  float* mn = (float*)(base + L.mn);
  float* mx = (float*)(base + L.mx);
  const unsigned bx = (unsigned)((d_out + 127) / 128);

  const bool fours = four_columns(ly) && reinterpret_cast<uintptr_t>(Q) % 4 == 0;
  const dim3 grid_g(bx, (unsigned)ng);
  // Groups that a block holds at once, and blocks enough to fill the SMs twice (three passes / this, us: 4096 x 4096 bf16 in groups
  // of 128 50 / 37, 1536 x 4100 in groups of 4 46 / 30; with fewer blocks the two are equal, both launches: 512 x 700 38 / 38).
  if (n_clip == 1 && fours && g <= 128 && (long long)bx * ng >= 592) {
    if (gamma_out) { fill_gamma_kernel<<<bx, 128, 0, st>>>(gamma_out, d_out); count_launch(); }
    const int warps = g <= 32 ? 4 : g <= 64 ? 8 : 16;
    auto run = [&](auto kern) { kern<<<grid_g, 32 * warps, 0, st>>>(ly.W, d_out, ly.ldw, g, ly.L, scale, zero, Q); count_launch(); };
    if (ly.wt == CDQ_BF16) run(warps == 4 ? group_codes_kernel<4, true> : warps == 8 ? group_codes_kernel<8, true> : group_codes_kernel<16, true>);
    else run(warps == 4 ? group_codes_kernel<4, false> : warps == 8 ? group_codes_kernel<8, false> : group_codes_kernel<16, false>);
    return cudaGetLastError();
  }
  run_minmax_partial(ly, cpg, pmn, pmx, st);
  { minmax_final_kernel<<<dim3(bx, (unsigned)ng), 128, 0, st>>>(pmn, pmx, ng, d_out, cpg, mn, mx); count_launch(); }

  const double* gam_col = nullptr;
  if (n_clip > 1) {
    double* gammas = (double*)(base + L.gammas);
    double* gcol = (double*)(base + L.gam_col);
    double* table = (double*)(base + L.table);
    double* E = (double*)(base + L.E);
    double* part = (double*)(base + L.part);
    double hg[256];
    const double lo = (double)grid.clip_lo, hi = (double)grid.clip_hi;
    for (int k = 0; k < n_clip; ++k) hg[k] = lo + ((hi - lo) * (double)k) / (double)(n_clip - 1);
    cudaError_t e = cudaMemcpyAsync(gammas, hg, sizeof(double) * n_clip, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    // the host array must outlive the copy: pageable memcpy is staged before return
    if (L.tc) {   // the slices of H serve every clipping strength
      e = gemm_tc_prepare_h(ly.H, d_in, kTcLossNH, kTcSearch, base + L.hbuf, st);
      if (e != cudaSuccess) return e;
    }
    if (L.screened) {
      double* screen = (double*)(base + L.screen);
      unsigned char* mask = (unsigned char*)(base + L.mask);
      int* idx = (int*)(base + L.idx);
      int* cnt = (int*)(base + L.cnt);
      double* loss_c = (double*)(base + L.loss_c);
      int* cj = (int*)(base + L.cj);
      int* ck = (int*)(base + L.ck);
      for (int k0 = 0; k0 < n_clip; k0 += L.sbatch) {   // screening, L.sbatch strengths per product
        const int gb = n_clip - k0 < L.sbatch ? n_clip - k0 : L.sbatch;
        const long long width = (long long)gb * d_out;
        ResidualSrc src{};
        src.W = ly.W; src.wt = ly.wt; src.ldw = ly.ldw;
        src.mn = mn; src.mx = mx; src.gamma = hg[k0]; src.L = ly.L; src.use_gamma = 1;
        src.g = g; src.d_out = d_out;
        if (gb > 1) { src.n_cols = width; src.k0 = k0; src.gammas = gammas; }   // column c: layer column c % d_out
        e = gemm_tc_run(base + L.hbuf, kTcLossNH, kTcSearch, src, E, d_in, width, screen_slices(ly.bits), screen_slices(ly.bits) + 1, 1.0,
                        nullptr, 0, screen + (long long)k0 * d_out, base + L.ebuf, st);
        if (e != cudaSuccess) return e;
      }
      { owc_candidates_kernel<<<bx, 128, 0, st>>>(screen, n_clip, d_out, mask, table); count_launch(); }
      { owc_compact_kernel<<<(unsigned)n_clip, 1024, 0, st>>>(mask, d_out, idx, cnt); count_launch(); }
      int hcnt[256];
      e = cudaMemcpyAsync(hcnt, cnt, sizeof(int) * n_clip, cudaMemcpyDeviceToHost, st);
      if (e != cudaSuccess) return e;
      e = cudaStreamSynchronize(st);   // the sizes of the exact products are decided on the host
      if (e != cudaSuccess) return e;
      OwcOffsets offs{};
      for (int k = 0; k < n_clip; ++k) offs.off[k + 1] = offs.off[k] + hcnt[k];
      const int total = offs.off[n_clip], padded = (total + 127) / 128 * 128;
      if (total <= 0) return cudaErrorUnknown;   // every column has at least its best strength as a candidate
      { owc_concat_kernel<<<(unsigned)((padded + 255) / 256), 256, 0, st>>>(idx, d_out, offs, n_clip, padded, cj, ck); count_launch(); }
      const int cap = (int)(L.wcap / 128 * 128);   // columns per product: what E and the slice buffers hold
      for (int b0 = 0; b0 < padded; b0 += cap) {
        const int width = padded - b0 < cap ? padded - b0 : cap;
        ResidualSrc src{};
        src.W = ly.W; src.wt = ly.wt; src.ldw = ly.ldw;
        src.mn = mn; src.mx = mx; src.L = ly.L; src.use_gamma = 1;
        src.g = g; src.d_out = d_out; src.col_idx = cj + b0; src.n_cols = width;
        src.col_gamma = ck + b0; src.gammas = gammas;
        e = gemm_tc_run(base + L.hbuf, kTcLossNH, kTcSearch, src, E, d_in, width, kTcLossNE, kTcLossSmax, 1.0, nullptr, 0,
                        loss_c, base + L.ebuf, st);
        if (e != cudaSuccess) return e;
        { owc_scatter_kernel<<<(unsigned)((width + 255) / 256), 256, 0, st>>>(loss_c, cj + b0, ck + b0, width, d_out, table); count_launch(); }
      }
    } else
    for (int k = 0; k < n_clip; ++k) {
      ResidualSrc src{};
      src.W = ly.W; src.wt = ly.wt; src.ldw = ly.ldw;
      src.mn = mn; src.mx = mx; src.gamma = hg[k]; src.L = ly.L; src.use_gamma = 1;
      src.g = g; src.d_out = d_out;
      if (L.tc) {
        e = gemm_tc_run(base + L.hbuf, kTcLossNH, kTcSearch, src, E, d_in, d_out, kTcLossNE, kTcLossSmax, 1.0, nullptr, 0,
                        table + (long long)k * d_out, base + L.ebuf, st);
      } else {
        e = launch_residual_f64(src, d_in, E, st);
        if (e != cudaSuccess) return e;
        if (mode == CDQ_MODE_FAST)
          e = launch_gemm_he(ly.H, d_in, d_out, E, nullptr, 0, table + (long long)k * d_out, part, false, st);
        else
          e = launch_gemm_he_verify(ly.H, d_in, d_out, E, part, nullptr, 0, table + (long long)k * d_out, st);
      }
      if (e != cudaSuccess) return e;
    }
    { owc_argmin_kernel<<<bx, 128, 0, st>>>(table, n_clip, d_out, gammas, gcol, gamma_out); count_launch(); }
    gam_col = gcol;
  } else if (gamma_out) {
    { fill_gamma_kernel<<<bx, 128, 0, st>>>(gamma_out, d_out); count_launch(); }
  }
  { scale_zero_kernel<<<dim3(bx, (unsigned)ng), 128, 0, st>>>(mn, mx, ng, d_out, ly.L, gam_col, scale, zero); count_launch(); }
  const int bpg = (int)((g + kCodeRows - 1) / kCodeRows);
  // (as for the minima; bf16 weights, one column against four, us: 1024 x 2048, 2^17 columns and row blocks, 5.7 / 7.2, 2048 x 2048 9.5 / 7.6,
  // 4096 x 4096 27 / 19)
  const bool four = fours && d_out * ng * bpg >= (1 << 18);
  const dim3 grid_q((unsigned)(four ? (d_out + 511) / 512 : bx), (unsigned)(ng * bpg));
  auto run = [&](auto kern) { kern<<<grid_q, 128, 0, st>>>(ly.W, d_out, ly.ldw, g, bpg, ly.L, scale, zero, Q); count_launch(); };
  if (ly.wt == CDQ_BF16) run(four ? rtn_codes_kernel<4, true> : rtn_codes_kernel<1, true>);
  else run(four ? rtn_codes_kernel<4, false> : rtn_codes_kernel<1, false>);
  return cudaGetLastError();
}

}  // namespace cdq
