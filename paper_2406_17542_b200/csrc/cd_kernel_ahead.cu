// Greedy coordinate descent (paper: the loop of Algorithm 1; Algorithm 4 for sub-channel grids) for rows of H of more
// than 8192 entries, which come from HBM: the next row travels while the present one is applied.
//
// As in cd_kernel_tma.cu a team owns one column at a time, with its gradient (fp64) and codes in registers, and a row
// of H arrives by one bulk copy.  There the row of move t + 1 can only be asked for when the sweep of move t has scored
// every coordinate, so that copy and sweep take turns.  Here the next move is known before the sweep:
//   * A full pass over the scores finds the best move and a level theta somewhat below its decrease.  Every coordinate
//     gets an interval for its gradient inside which it cannot lower the loss by more than theta (`reach`).
//   * The few coordinates outside their interval are *watched*: a lane of the warp keeps a copy of the gradient (the
//     same fused multiply-adds in the same order, so the same bits) with what its score needs.
//   * When a row has landed, the lanes update and score the watched coordinates alone -- one entry of the row each --
//     and the best of them, if it is above theta, is taken as the next move: its row is asked for at once, into the
//     other buffer.  Only then does the team sweep the whole row, and the sweep does not score: it tests intervals.
//   * A coordinate that the sweep finds outside its interval is watched from then on.  If it beats the move in flight
//     (one move in twenty), that move is dropped before it has touched anything but the watched copies.
//   * When all watched coordinates are down to theta, theta is lowered and the intervals are drawn anew (every 50 to
//     100 moves).
// What bounds it: with one team of 12 or 16 warps per SM, latency -- a scheduler has three or four warps; the copy, which the
// sweep used to wait 1700 cycles for, is all but hidden (180 cycles).  Descent, before (copy and sweep in turn, every
// coordinate scored) -> after: 14336 entries x 1184 columns 277 -> 218 ms, 18432 in groups of 128 x 592 241 -> 193,
// 16384 x 296 88 -> 72, 11008 x 296 51 -> 43.  Rows of up to 8192 entries, of which two or more teams share an SM, hide the
// copies behind one another's sweeps and do not gain: 8192 entries 27.6 -> 28.9 ms, 5120 23.8 -> 27.8, 3072 12.3 -> 15.9.
// Every move is the one that scoring all coordinates in fp32 would name: the intervals are drawn with a margin that
// covers the roundings of the score, and every coordinate outside its interval is scored as the full pass scores it.
//
// Waits on the copy barriers are bounded by a cycle count.  A thread whose wait runs out enters the argmin with a key
// that no move can have; the whole team sees it, starts no further step or column, waits (bounded) for the copy in
// flight, records kFlagWaitTimeout in the device status word and returns.
#include "async_copy.cuh"
#include "cd_params.cuh"
#include "cd_sweep.cuh"

namespace cdq {
namespace {

constexpr unsigned kWaitCycles = 400u * 1000u * 1000u;   // about 0.2 s
// Keys of the argmin below those of all real moves (a move's key is at least 0x007FFFFF and at most 0x7FFFFFFE).
constexpr unsigned kAbortKey = 0u;    // a copy did not land
constexpr unsigned kFullKey = 1u;     // drop the move in flight and score everything (a warp has no idle lane left)
constexpr unsigned kCrowdKey = 2u;    // the move in flight stands, but score everything after it (same reason)
constexpr unsigned kNever = 0x7F000000u;   // a threshold that no gradient reaches
// Coordinates a warp hands over to its idle lanes at a time.  (16: no faster on any row, 16384 x 296 columns 17.7 ms against 17.5, the others
// within 0.5 %; and with 8 the table of H_ii fits beside 8 x 448 chunk slots.)
constexpr int kHand = 8;
constexpr float kGap0 = 0.3f, kGapMin = 1.f / 256, kGapMax = 0.5f, kGapGrow = 1.25f;

// A coordinate that a lane is to watch, handed over by the thread that owns its chunk.
struct __align__(16) Handover {
  double g;
  unsigned id;     // chunk slot << 21 | thread << 11 | position << 9: the order of the coordinate index
  unsigned q;
};

// Largest |g| (upper word of a double, less one unit) up to which a coordinate with `room` levels on the side it would
// move to cannot lower the loss by more than theta.  A move of k levels lowers it by k a |g| - k^2 a^2 H, so the bound
// is the minimum over 1 <= k <= room of theta / (k a) + k a H; over real k that minimum is a lower bound, and it is
// lowered by another 2^-18 of itself, which covers every rounding of the fp32 score (a few 2^-24 of |g|).
// x = sqrt(theta / H) / a: the real minimiser; ta = theta / a; ah = a H.
__device__ __forceinline__ unsigned reach(float x, float ta, float ah, float room) {
  const float k = fminf(fmaxf(x, 1.f), room);
  const float t = fmaf(k, ah, __fdividef(ta, k)) * (1.f - 3.8e-6f);
  unsigned u = (__float_as_uint(t) >> 3) + 0x38000000u - 1u;
  if (!(t > 1e-37f)) u = 0u;            // also a NaN: never leave the coordinate out
  return u < kNever ? u : kNever;
}
// Gradient and codes of chunk slot k (the same k in every lane) out of the register arrays.  The passes that are made
// once in many moves loop over k with it: unrolled, their code (some 50 KB) came from L2 every time they ran.
template <int NCH>
__device__ __forceinline__ void pick_chunk(int k, const double (&g)[4 * NCH], const unsigned (&qp)[NCH], double (&x)[4],
                                           unsigned& q4) {
#define CDQ_PICK(K)                                                                                  \
  case K:                                                                                            \
    if constexpr (K < NCH) {                                                                         \
      x[0] = g[4 * K]; x[1] = g[4 * K + 1]; x[2] = g[4 * K + 2]; x[3] = g[4 * K + 3]; q4 = qp[K];    \
    }                                                                                                \
    break;
  switch (k) {
    CDQ_PICK(0) CDQ_PICK(1) CDQ_PICK(2) CDQ_PICK(3) CDQ_PICK(4) CDQ_PICK(5) CDQ_PICK(6) CDQ_PICK(7)
    CDQ_PICK(8) CDQ_PICK(9) CDQ_PICK(10) CDQ_PICK(11) CDQ_PICK(12) CDQ_PICK(13) CDQ_PICK(14) CDQ_PICK(15)
    default: break;
  }
#undef CDQ_PICK
}

// Whether the table of H_ii fits beside the rows, the thresholds and the handovers of so many chunk slots is known when the kernel is compiled,
// but to say it there changes what the compiler spills, for better or worse.  A quarter of a pass, said at run time / here (ms): 18432 x 296 per
// channel 22.2 / 21.95, bf16 12288 x 296 in groups of 128 12.1 / 11.85, 14336 16.65 / 16.45; 14336 x 592 per channel 26.2 / 26.5, 17408 x 296 in
// groups of 128 21.0 / 22.0, bf16 11264 x 296 9.96 / 10.1, 15360 x 296 per channel 14.5 / 14.6.  Bf16 rows of 15361 to 16384 entries in groups
// are better off without either table (16384 x 296 in groups of 128 22.2 / 21.9).
enum Table { kTableNever, kTableAlways, kTableIfFits };
__host__ __device__ constexpr Table hd_table(int slots, bool grouped, bool row16) {
  if (row16 && grouped) return slots <= 3840 ? kTableAlways : slots <= 4096 ? kTableNever : kTableIfFits;
  return !row16 && !grouped && slots > 4224 ? kTableNever : kTableIfFits;
}

// NCH chunk slots per thread; the team covers ceil(d_in / 4) <= NT * NCH chunks.
// ROW16: the rows come from a bf16 copy of H (half the bytes per move); the row's own diagonal element is
// replaced by the exact H_ii, so the iteration is the descent on H with its off-diagonal entries rounded to bf16.
template <int NCH, int MAXNT, int MINB, bool GROUPED, bool ROW16>
__global__ void __launch_bounds__(MAXNT, MINB) cd_ahead_kernel(CdParams p) {
  extern __shared__ __align__(128) unsigned char dyn_smem[];
  __shared__ __align__(8) unsigned long long s_bar[2];   // completion of the rows' copies
  __shared__ __align__(16) uint4 s_exch[2][MAXNT / 32];
  __shared__ int s_col;

  const int tid = threadIdx.x, NT = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nwarps = NT >> 5;
  const unsigned below = (1u << lane) - 1u;    // lanes before this one
  const int nchs = (int)(p.d_in >> 2);         // chunks of a row
  const bool exact = nchs == NT * NCH;
  const bool last_slot = (tid & ~31) + NT * (NCH - 1) < nchs;   // the warp has chunks in the last slot
  const int asker = NT - 32;                   // the thread that asks for the rows: its warp has no more than the others to sweep
  const float top_q = (float)p.L, top = kMagic + top_q;

  constexpr int CHB = ROW16 ? 8 : 16;                                   // bytes of a chunk of 4 row entries
  constexpr int W0 = NCH < 8 ? NCH : 8, W1 = NCH - W0;                  // chunk slots behind the two mask words
  static_assert(NCH <= 16, "two mask words");
  const int row_span = NCH * NT * CHB;
  unsigned char* row_s = dyn_smem;                                      // [2][NCH * NT] chunks
  float4* thr_s = reinterpret_cast<float4*>(row_s + 2 * (size_t)row_span);    // [NCH * NT] thresholds of the column
  Handover* hand = reinterpret_cast<Handover*>(thr_s + NCH * NT) + kHand * warp;   // [warps][kHand]
  // H_ii and the column's group scales, if they fit beside the rows.  A coordinate that has just left its interval is scored before the
  // team can go on, and from memory they come behind the row that is on its way into the SM (18432 in groups of 128 x 296 96.1 -> 93.3 ms,
  // 9004 in groups of 4 x 296 16.4 -> 15.5, 13312 in groups of 128 x 296 46.1 -> 45.4, 14336 x 592 111.9 -> 110.3).
  unsigned char* more = reinterpret_cast<unsigned char*>(reinterpret_cast<Handover*>(thr_s + NCH * NT) + kHand * nwarps);
  constexpr Table kHd = hd_table(NCH * MAXNT, GROUPED, ROW16);
  constexpr bool kAg = GROUPED && !(ROW16 && kHd == kTableNever);   // (the group scales go with it)
  const bool hd_here = kHd == kTableAlways || (kHd == kTableIfFits && (p.tables & 1) != 0), ag_here = kAg && (p.tables & 2) != 0;
  float* hd_s = reinterpret_cast<float*>(more);
  float* ag_s = hd_s + (hd_here ? 4 * NCH * NT : 0);
  const float* hd_t = hd_here ? hd_s : p.hdiag;
  auto hd_of = [&](int i) -> float { return kHd == kTableNever ? __ldg(p.hdiag + i) : hd_t[i]; };   // H_ii
  auto hd4_of = [&](int cs) -> float4 {                                                            // those of a chunk
    return kHd == kTableNever ? __ldg(reinterpret_cast<const float4*>(p.hdiag) + cs) : reinterpret_cast<const float4*>(hd_t)[cs];
  };
  auto group_of = [&](unsigned i) -> unsigned { return p.g == 1 ? i : __umulhi(i, p.gmagic); };

  // slots past the end of the row stay zero: no copy ever writes there
  for (int t = tid; t < 2 * NCH * NT * CHB / 8; t += NT) reinterpret_cast<uint2*>(row_s)[t] = make_uint2(0u, 0u);
  if (hd_here)
    for (int t = tid; t < NCH * NT; t += NT) reinterpret_cast<float4*>(hd_s)[t] = __ldg(reinterpret_cast<const float4*>(p.hdiag) + t);
  if (tid == 0) {
    mbar_init(smem_u32(&s_bar[0]), 1);
    mbar_init(smem_u32(&s_bar[1]), 1);
    mbar_fence_init();
  }
  const uint32_t row_bytes = (uint32_t)nchs * (uint32_t)CHB;
  __syncthreads();
  fence_proxy_async_smem();  // zero fill before the first copy lands

  unsigned long long my_committed = 0, my_converged = 0;
  double my_dsum = 0.0;
  uint32_t phases = 0u;   // bit b: parity of buffer b's barrier for the next wait
  int buf = 0;            // buffer of the row being waited for
  int xbuf = 0;
  bool aborted = false;

  while (!aborted) {
    __syncthreads();  // everyone is done with the previous column
    if (tid == 0) s_col = atomicAdd(&p.ctr->next_col, 1);
    __syncthreads();
    const long long j = s_col;
    if (j >= p.d_out) break;

    // ---- column state ----
    float a_col = 1.f;
    double gscale = 1.0;
    bool frozen = false;
    if (!GROUPED) {
      a_col = p.scale[j];
      frozen = !(a_col > 0.f);   // constant column: its grid has one point, nothing can move
      gscale = frozen ? 0.0 : 1.0 / (double)a_col;
    }
    const float* scale_j = ag_here ? ag_s : p.scale + j;   // GROUPED: scale of group t at scale_j[t * scale_step]
    const long long scale_step = ag_here ? 1 : p.d_out;
    auto scale_of = [&](unsigned group) -> float {
      return kAg ? scale_j[(long long)group * scale_step] : __ldg(p.scale + j + (long long)group * p.d_out);
    };
    if (ag_here) {
      for (int t = tid; t < (int)p.ng; t += NT) ag_s[t] = p.scale[(long long)t * p.d_out + j];
      __syncthreads();
    }
    double g[4 * NCH];
    unsigned qp[NCH];
    {
      const double* gcol = p.G + j * p.ldg;
      const unsigned char* qcol = p.Qt + j * p.ldq;
#pragma unroll
      for (int k = 0; k < NCH; ++k) {
        const int cs = tid + NT * k;
        double2 g0 = make_double2(0.0, 0.0), g1 = g0;
        qp[k] = 0;
        if (exact || cs < nchs) {
          g0 = *reinterpret_cast<const double2*>(gcol + (long long)cs * 4);
          g1 = *reinterpret_cast<const double2*>(gcol + (long long)cs * 4 + 2);
          qp[k] = *reinterpret_cast<const unsigned*>(qcol + (long long)cs * 4);
        }
        g[4 * k] = g0.x * gscale; g[4 * k + 1] = g0.y * gscale; g[4 * k + 2] = g1.x * gscale; g[4 * k + 3] = g1.y * gscale;
      }
    }

    // ---- descent ----
    long long step = 0;
    double col_dsum = 0.0;
    bool done = frozen;
    unsigned theta_key = 0u;   // key of the decrease that the thresholds stand for
    float gap = kGap0;         // theta = (1 - gap) of the best decrease at the last full pass
    // The coordinate that this lane watches (its index, or -1): gradient, scale, H_ii, 0.5 / (a H_ii), kMagic + code.
    int wi = -1;
    double wg = 0.0;
    float wa = 1.f, wh = 0.f, ws = 0.f, wq = kMagic;
    unsigned wid = 0u;
    // One bit per coordinate of the thread (the first one in the highest bit of its word): it has no room upwards /
    // downwards, or is watched.
    unsigned no_up0 = 0u, no_up1 = 0u, no_dn0 = 0u, no_dn1 = 0u;
    // Outside the interval of the other side when its sign changes (see new_thresholds).
    unsigned pos0 = 0u, pos1 = 0u, neg0 = 0u, neg1 = 0u;
    unsigned e0 = 0u, e1 = 0u;    // coordinates of this thread that have left their interval and are not watched
    unsigned late_m = kNoMove, late_w = kNoMove;   // this warp's move that beats the one whose row is on its way
    unsigned cur_m = kNoMove, cur_w = kNoMove;     // the move whose row is waited for
    double c2 = 0.0;                               // twice its step (code units when per-channel)
    [[maybe_unused]] float cur_h = 0.f;            // ROW16: H_ii of its coordinate

    // What the score of a newly watched coordinate needs besides H_ii and the scale, when their loads have had time to arrive.
    auto watch_ready = [&]() {
      ws = wh > 0.f ? 0.5f / wh : 0.f;
      if (GROUPED) ws = (wa > 0.f ? 1.0f / wa : 0.f) * ws;
    };
    // Score of the watched coordinate.
    auto watch_score = [&](unsigned& key, unsigned& packed) {
      key = kNoMove; packed = kNoMove;
      if (wi >= 0) {
        const float gf = (float)wg;
        float t = fmaf(-gf, ws, wq);
        t = fminf(fmaxf(t, kMagic), top);
        const float dr = t - wq;
        const float d = GROUPED ? wa * dr : dr;
        const float dl = fmaf(d, wh, gf) * d;
        if (dl < 0.f) {
          key = ~__float_as_uint(dl);
          packed = wid | (unsigned)((int)dr + 256);
        }
      }
    };
    // Takes the move (m, w): asks for its row in buffer b.  Called behind a barrier after which nobody reads that
    // buffer any more, and as early as the move is known.  Returns the coordinate.
    auto take_move = [&](unsigned m, unsigned w, int b) -> int {
      cur_m = m; cur_w = w;
      int istar = 4 * ((int)((w >> 11) & 1023u) + NT * (int)(w >> 21)) + (int)((w >> 9) & 3u);
      if ((unsigned)istar >= (unsigned)p.d_in) {  // cannot happen; never follow a bad row index
        if (tid == 0) atomicExch(p.status, (int)kFlagBadIndex);
        istar = 0;
      }
      if (tid == asker) {
        const unsigned char* src = ROW16 ? reinterpret_cast<const unsigned char*>(p.H16 + (long long)istar * p.d_in)
                                         : reinterpret_cast<const unsigned char*>(p.H + (long long)istar * p.d_in);
        mbar_expect_tx(smem_u32(&s_bar[b]), row_bytes);
        bulk_load(smem_u32(row_s + b * row_span), src, row_bytes, smem_u32(&s_bar[b]));
      }
      return istar;
    };
    // The step of move w, and what else its sweep needs (loads: they overlap with the copy).
    auto load_step = [&](unsigned w, int istar) {
      float a = 1.f;
      if (GROUPED) a = scale_of(group_of((unsigned)istar));
      c2 = 2.0 * ((double)a * (double)((int)(w & 511u) - 256));
      if constexpr (ROW16) cur_h = hd_of(istar);
    };
    // Hands the coordinates of the two words over to idle lanes of the warp; true in the lanes that got one.
    // room: whether there were enough.
    auto watch_new = [&](bool& room) -> bool {
      bool fresh = false;
      room = true;
#pragma unroll
      for (int word = 0; word < (W1 > 0 ? 2 : 1); ++word) {
        const unsigned e = word ? e1 : e0;
        unsigned any = __reduce_or_sync(0xFFFFFFFFu, e);
        while (any && room) {
          const int bit = __ffs((int)any) - 1;
          any &= any - 1u;
          const int o = 4 * (word ? W1 : W0) - 1 - bit, k = (o >> 2) + (word ? W0 : 0), v = o & 3;
          double x[4] = {0.0, 0.0, 0.0, 0.0};
          unsigned q4 = 0u;
          pick_chunk<NCH>(k, g, qp, x, q4);
          const double x01 = v & 1 ? x[1] : x[0], x23 = v & 1 ? x[3] : x[2];
          const double xv = v & 2 ? x23 : x01;
          unsigned who = __ballot_sync(0xFFFFFFFFu, (e >> bit) & 1u);
          while (who) {
            const unsigned idle = __ballot_sync(0xFFFFFFFFu, wi < 0);
            if (!idle) { room = false; break; }
            const int rank = __popc(who & below), n = min(min(__popc(who), __popc(idle)), kHand);
            const bool give = ((who >> lane) & 1u) && rank < n;
            if (give) {
              hand[rank].g = xv;
              hand[rank].id = ((unsigned)k << 21) | ((unsigned)tid << 11) | ((unsigned)v << 9);
              hand[rank].q = (q4 >> (8 * v)) & 255u;
              if (word) { no_up1 |= 1u << bit; no_dn1 |= 1u << bit; pos1 &= ~(1u << bit); neg1 &= ~(1u << bit); }
              else { no_up0 |= 1u << bit; no_dn0 |= 1u << bit; pos0 &= ~(1u << bit); neg0 &= ~(1u << bit); }
            }
            __syncwarp();
            const int mine = __popc(idle & below);
            if (wi < 0 && mine < n) {
              wg = hand[mine].g;
              wid = hand[mine].id;
              wq = __uint_as_float(kMagicBits | hand[mine].q);
              wi = 4 * ((int)((wid >> 11) & 1023u) + NT * (int)(wid >> 21)) + (int)((wid >> 9) & 3u);
              wh = hd_of(wi);
              if (GROUPED) wa = scale_of(group_of((unsigned)wi));
              fresh = true;
            }
            who &= ~__ballot_sync(0xFFFFFFFFu, give);
            __syncwarp();
          }
        }
      }
      return fresh;
    };
    // Team-wide argmin: (decrease, lowest coordinate, lowest level).  Every thread gets the result, and the second pair
    // that warp number `lane` brought along.
    auto team_min = [&](unsigned key, unsigned packed, unsigned zm, unsigned zw, unsigned& m, unsigned& w) -> uint2 {
      m = __reduce_min_sync(0xFFFFFFFFu, key);
      w = __reduce_min_sync(0xFFFFFFFFu, key == m ? packed : kNoMove);
      if (lane == 0) s_exch[xbuf][warp] = make_uint4(m, w, zm, zw);
      __syncthreads();
      uint4 x = make_uint4(kNoMove, kNoMove, kNoMove, kNoMove);
      if (lane < nwarps) x = s_exch[xbuf][lane];
      m = __reduce_min_sync(0xFFFFFFFFu, x.x);
      w = __reduce_min_sync(0xFFFFFFFFu, x.x == m ? x.y : kNoMove);
      xbuf ^= 1;
      return make_uint2(x.z, x.w);
    };
    // Best move over all coordinates (every thread gets it; m == kNoMove: none lowers the loss).
    auto full_pass = [&](unsigned& m, unsigned& w) {
      SweepBest sb;
      sb.init();
#pragma unroll 1
      for (int k = 0; k < NCH; ++k) {
        const int cs = tid + NT * k;
        const float4 hd = hd4_of(cs);
        const float4 hs = __ldg(reinterpret_cast<const float4*>(p.hs) + cs);
        float a = 1.f, ia = 1.f;
        if (GROUPED) {
          a = cs < nchs ? scale_of(group_of(4u * (unsigned)cs)) : 0.f;
          ia = a > 0.f ? 1.0f / a : 0.f;
        }
        double x[4] = {0.0, 0.0, 0.0, 0.0};
        unsigned q4 = 0u;
        pick_chunk<NCH>(k, g, qp, x, q4);
        score_chunk<GROUPED>(x, hd, hs, q4, a, ia, top, k, sb);
      }
      unsigned key, packed;
      sweep_candidate(sb, tid, key, packed);
      team_min(key, packed, kNoMove, kNoMove, m, w);
    };
    // The intervals for the decrease theta; e0, e1: the coordinates that lie outside theirs.  A coordinate has one
    // threshold for |g|, that of a side with room enough.  If |g| is above it but within the threshold of the side it
    // is on, which has less room, it gets that one, and is flagged so that a change of sign brings it up.
    auto new_thresholds = [&](float theta) {
      theta_key = ~__float_as_uint(-theta);
      const float inv_theta = 1.0f / theta;
      wi = -1;
      no_up0 = no_up1 = no_dn0 = no_dn1 = 0u;
      pos0 = pos1 = neg0 = neg1 = 0u;
      e0 = e1 = 0u;
#pragma unroll 1
      for (int k = 0; k < NCH; ++k) {
        const int cs = tid + NT * k;
        const float4 hd = hd4_of(cs);
        float a = 1.f, ia = 1.f;
        if (GROUPED) {
          a = cs < nchs ? scale_of(group_of(4u * (unsigned)cs)) : 0.f;
          ia = a > 0.f ? 1.0f / a : 0.f;
        }
        double x[4] = {0.0, 0.0, 0.0, 0.0};
        unsigned q4 = 0u;
        pick_chunk<NCH>(k, g, qp, x, q4);
        const float ta = theta * ia;
        float t[4];
        const float h[4] = {hd.x, hd.y, hd.z, hd.w};
        unsigned up = 0u, dn = 0u, ex = 0u, ps = 0u, ns = 0u;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const float q = (float)((q4 >> (8 * v)) & 255u), r = top_q - q;   // room downwards, upwards
          const int hi = __double2hiint(x[v]);
          const unsigned mag = (unsigned)hi & 0x7FFFFFFFu;
          unsigned u = kNever;
          bool out = false, between = false;
          if (h[v] > 0.f && a > 0.f) {
            const float xk = rsqrtf(h[v] * inv_theta) * ia, ah = a * h[v];
            u = reach(xk, ta, ah, top_q);
            const float room = hi < 0 ? r : q;
            if (mag > u && room > 0.5f) {
              const unsigned side = reach(xk, ta, ah, room);
              out = mag > side;
              between = !out;
              if (between) u = side;
            }
          }
          t[v] = __uint_as_float(u);
          up = (up << 1) | (r > 0.5f ? 0u : 1u);
          dn = (dn << 1) | (q > 0.5f ? 0u : 1u);
          ex = (ex << 1) | (out ? 1u : 0u);
          ps = (ps << 1) | (between && hi >= 0 ? 1u : 0u);
          ns = (ns << 1) | (between && hi < 0 ? 1u : 0u);
        }
        thr_s[cs] = make_float4(t[0], t[1], t[2], t[3]);
        if (k < W0) {
          no_up0 = (no_up0 << 4) | up; no_dn0 = (no_dn0 << 4) | dn; e0 = (e0 << 4) | ex;
          pos0 = (pos0 << 4) | ps; neg0 = (neg0 << 4) | ns;
        } else {
          no_up1 = (no_up1 << 4) | up; no_dn1 = (no_dn1 << 4) | dn; e1 = (e1 << 4) | ex;
          pos1 = (pos1 << 4) | ps; neg1 = (neg1 << 4) | ns;
        }
      }
    };

    enum : int { kAhead, kLower, kAll };
    int how = kAll;        // where the next move comes from: it is on its way / a lower theta / a pass over all scores
    float theta = 0.f;
    bool fresh = false;    // this lane has been given a coordinate since the last argmin
    while (!done) {
      if (how == kAll) {
        unsigned m, w;
        full_pass(m, w);
        if (m == kNoMove) { done = true; break; }
        load_step(w, take_move(m, w, buf));
        theta = -__uint_as_float(~m) * (1.f - gap);
      }
      if (how != kAhead) new_thresholds(theta);
      // ---- coordinates that have left their interval get a lane that watches them ----
      bool room = true;
      if (__any_sync(0xFFFFFFFFu, (e0 | e1) != 0u)) fresh = watch_new(room);
      e0 = e1 = 0u;
      if (!room) { late_m = how == kAhead ? kFullKey : kCrowdKey; late_w = 0u; }
      if (how == kLower) {   // all that lies above theta is watched now, the best move among it
        unsigned key, packed, m, w;
        watch_ready();
        watch_score(key, packed);
        const uint2 z = team_min(key, packed, late_m, late_w, m, w);
        if (__any_sync(0xFFFFFFFFu, z.x != kNoMove) || m >= theta_key) {   // not all of it: no lane was idle
          late_m = late_w = kNoMove;
          gap = fmaxf(0.5f * gap, kGapMin);
          how = kAll;
          continue;
        }
        load_step(w, take_move(m, w, buf));
      }
      const bool chosen = how != kAhead;   // the move has been chosen with the new ones in view
      how = kAhead;

      // ---- the watched coordinates take the move first: they name the next one before the sweep ----
      const bool timed_out = !mbar_wait_clock32(smem_u32(&s_bar[buf]), (phases >> buf) & 1u, kWaitCycles);
      phases ^= 1u << buf;
      const unsigned char* row = row_s + buf * row_span;
      unsigned key, packed, m, w;
      if (__any_sync(0xFFFFFFFFu, fresh)) {   // does a new one beat the move in flight?
        watch_ready();
        watch_score(key, packed);
        const bool beats = fresh && !chosen && late_m == kNoMove && (key < cur_m || (key == cur_m && packed < cur_w));
        if (__any_sync(0xFFFFFFFFu, beats)) {
          if (!beats) key = kNoMove;
          late_m = __reduce_min_sync(0xFFFFFFFFu, key);
          late_w = __reduce_min_sync(0xFFFFFFFFu, key == late_m ? packed : kNoMove);
        }
        fresh = false;
      }
      const double wg_prev = wg;
      const bool moved = wi >= 0 && wid == (cur_w & ~511u);
      const float dri = (float)((int)(cur_w & 511u) - 256);
      if (wi >= 0) {
        float h;
        if constexpr (ROW16) {
          h = __uint_as_float((unsigned)reinterpret_cast<const unsigned short*>(row)[wi] << 16);
          if (moved) h = wh;
        } else {
          h = reinterpret_cast<const float*>(row)[wi];
        }
        wg = fma(c2, (double)h, wg);
        if (moved) wq += dri;
      }
      watch_score(key, packed);
      if (timed_out) { key = kAbortKey; packed = 0u; }
      const uint2 z = team_min(key, packed, late_m, late_w, m, w);
      if (m == kAbortKey) {   // a copy never landed: wait (bounded) for it once more, then give up
        if (tid == asker) {
          mbar_wait_clock32(smem_u32(&s_bar[buf]), ((phases >> buf) & 1u) ^ 1u, kWaitCycles);
          atomicCAS(p.status, (int)kFlagOk, (int)kFlagWaitTimeout);
        }
        aborted = true;
        break;
      }
      bool crowd = false;
      if (__any_sync(0xFFFFFFFFu, z.x != kNoMove)) {
        const unsigned bm = __reduce_min_sync(0xFFFFFFFFu, z.x);
        const unsigned bw = __reduce_min_sync(0xFFFFFFFFu, z.x == bm ? z.y : kNoMove);
        late_m = late_w = kNoMove;
        crowd = bm == kCrowdKey;
        if (bm <= kCrowdKey) gap = fmaxf(0.5f * gap, kGapMin);
        if (!crowd) {   // the last sweep found a better move than the one in flight: back to the state before it
          wg = wg_prev;
          if (moved) wq -= dri;
          if (bm == kFullKey) how = kAll;
          else load_step(bw, take_move(bm, bw, buf));
          continue;
        }
      }

      // ---- the move stands ----
      const int kcur = (int)(cur_w >> 21), vcur = (int)((cur_w >> 9) & 3u);
      const bool owner = tid == (int)((cur_w >> 11) & 1023u);
      const double c2_now = c2, c2_bits = c2 * 0x1p896;
      [[maybe_unused]] const float h_now = cur_h;
      if (owner) {
        const unsigned dq = (unsigned)(int)dri << (8 * vcur);
#pragma unroll
        for (int k = 0; k < NCH; ++k)
          if (k == kcur) qp[k] += dq;
      }
      if (tid == 0) col_dsum += (double)__uint_as_float(~cur_m);
      ++step;
      const bool last = step >= p.T;
      // A coordinate that nobody watches lowers the loss by at most theta, up to what the sweep still finds.
      const bool ahead = !last && !crowd && m < theta_key;
      int inext = 0;
      if (ahead) inext = take_move(m, w, buf ^ 1);

      // ---- sweep: g += c2 H[i*, :]; sign bits of threshold - |g| and of g ----
      // Half of the entries are widened by the conversion pipe (16 per clock and SM, which would be the sweep's bound), half
      // by moving their bits: without the exponent's bias the double is the entry times 2^-896, which the step makes up
      // for, exactly (14336 x 1184 columns 226 -> 219 ms).  (Infinities and NaN
      // would become numbers of 2^128 and more: see mark_features_kernel.)
      unsigned v0 = 0u, v1 = 0u, n0 = 0u, n1 = 0u;
#pragma unroll
      for (int k = 0; k < NCH; ++k) {
        if (k == NCH - 1 && !last_slot) break;   // (the warp's slots are past the end of the row)
        const int cs = tid + NT * k;
        float4 rv;
        if constexpr (ROW16) {
          const uint2 rr = reinterpret_cast<const uint2*>(row)[cs];
          rv = make_float4(__uint_as_float(rr.x << 16), __uint_as_float(rr.x & 0xFFFF0000u),
                           __uint_as_float(rr.y << 16), __uint_as_float(rr.y & 0xFFFF0000u));
          if (owner && k == kcur) {   // this thread holds the coordinate that moved: its own entry of the row is H_ii
            rv.x = vcur == 0 ? h_now : rv.x; rv.y = vcur == 1 ? h_now : rv.y;
            rv.z = vcur == 2 ? h_now : rv.z; rv.w = vcur == 3 ? h_now : rv.w;
          }
        } else {
          rv = reinterpret_cast<const float4*>(row)[cs];
        }
        const float4 th = thr_s[cs];
        const float hv[4] = {rv.x, rv.y, rv.z, rv.w}, tv[4] = {th.x, th.y, th.z, th.w};
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          if (v & 1) {   // widened by integer operations
            const int b = __float_as_int(hv[v]);
            g[4 * k + v] = fma(c2_bits, __hiloint2double((b >> 3) & (int)0x8FFFFFFFu, b << 29), g[4 * k + v]);
          } else {
            g[4 * k + v] = fma(c2_now, (double)hv[v], g[4 * k + v]);
          }
          const int hi = __double2hiint(g[4 * k + v]);
          const int s = __float_as_int(tv[v] - fabsf(__int_as_float(hi)));
          if (k < W0) { v0 = __funnelshift_l((unsigned)s, v0, 1); n0 = __funnelshift_l((unsigned)hi, n0, 1); }
          else { v1 = __funnelshift_l((unsigned)s, v1, 1); n1 = __funnelshift_l((unsigned)hi, n1, 1); }
        }
      }
      if (!last_slot) {
        if (NCH <= W0) { v0 <<= 4; n0 <<= 4; } else { v1 <<= 4; n1 <<= 4; }
      }
      if (last) break;   // budget used up
      if (ahead) {
        load_step(w, inext);
        e0 = (v0 & ~((n0 & no_up0) | (~n0 & no_dn0))) | (pos0 & n0) | (neg0 & ~n0);
        e1 = (v1 & ~((n1 & no_up1) | (~n1 & no_dn1))) | (pos1 & n1) | (neg1 & ~n1);
      } else if (crowd || m == kNoMove) {
        how = kAll;
      } else {   // every watched coordinate is down to theta; the best of them is a bound on the next move's decrease
        gap = fminf(kGapGrow * gap, kGapMax);
        theta = -__uint_as_float(~m) * (1.f - gap);
        how = kLower;
      }
      buf ^= 1;
    }
    if (aborted) break;
    if (tid == 0) {
      if (done) ++my_converged;
      my_committed += (unsigned long long)step;
      my_dsum += !GROUPED ? col_dsum * ((double)a_col * (double)a_col) : col_dsum;
    }

    // ---- write the codes back, and the gradient of the result (weight units) ----
    if (!frozen) {
      unsigned char* qcol = p.Qt + j * p.ldq;
      double* gcol = p.G + j * p.ldg;
      const double ga = !GROUPED ? (double)a_col : 1.0;
#pragma unroll
      for (int k = 0; k < NCH; ++k) {
        const int cs = tid + NT * k;
        if (exact || cs < nchs) {
          *reinterpret_cast<unsigned*>(qcol + (long long)cs * 4) = qp[k];
          *reinterpret_cast<double2*>(gcol + (long long)cs * 4) = make_double2(g[4 * k] * ga, g[4 * k + 1] * ga);
          *reinterpret_cast<double2*>(gcol + (long long)cs * 4 + 2) = make_double2(g[4 * k + 2] * ga, g[4 * k + 3] * ga);
        }
      }
    }
  }

  if (tid == 0) {
    if (my_dsum != 0.0) atomicAdd(&p.ctr->delta_sum, my_dsum);
    if (my_committed) atomicAdd(&p.ctr->committed, my_committed);
    if (my_converged) atomicAdd(&p.ctr->converged, my_converged);
  }
}

template <int NCH, int MAXNT, int MINB, bool GROUPED, bool ROW16>
cudaError_t launch_cfg(CdParams p, int nt, cudaStream_t st) {
  auto kern = cd_ahead_kernel<NCH, MAXNT, MINB, GROUPED, ROW16>;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // two rows, the thresholds, the handovers
  size_t smem = (size_t)NCH * nt * (ROW16 ? 16 : 32) + (size_t)NCH * nt * 16 + sizeof(Handover) * kHand * (size_t)(nt / 32);
  cudaError_t e;
  {   // H_ii and the group scales beside them where they fit (fp32 rows: up to 14336 entries)
    cudaFuncAttributes fa{};
    int optin = 0;
    e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    const size_t room = (size_t)optin - fa.sharedSizeBytes, hd = (size_t)NCH * nt * 16, ag = GROUPED ? ((size_t)p.ng * 4 + 15) / 16 * 16 : 0;
    p.tables = 0;
    constexpr Table kHd = hd_table(NCH * MAXNT, GROUPED, ROW16);
    if (kHd == kTableAlways || (kHd == kTableIfFits && smem + hd <= room)) { p.tables |= 1; smem += hd; }
    if (GROUPED && !(ROW16 && kHd == kTableNever) && smem + ag <= room) { p.tables |= 2; smem += ag; }
  }
  if (smem > 32 * 1024) {   // the 48 KB that need no opt-in include the kernel's static shared memory
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  int per_sm = 1;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, nt, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  long long blocks = (long long)sms * per_sm;
  if (blocks > p.d_out) blocks = p.d_out;
  { kern<<<(unsigned)blocks, nt, smem, st>>>(p); count_launch(); }
  return cudaGetLastError();
}

template <int NCH, int MAXNT, int MINB>
cudaError_t launch_mode(const CdParams& p, int nt, cudaStream_t st) {
  if (p.ng > 1 && (p.g & 3)) return cudaErrorNotSupported;   // one scale per chunk of 4 coordinates
  if (p.H16) return p.ng > 1 ? launch_cfg<NCH, MAXNT, MINB, true, true>(p, nt, st) : launch_cfg<NCH, MAXNT, MINB, false, true>(p, nt, st);
  return p.ng > 1 ? launch_cfg<NCH, MAXNT, MINB, true, false>(p, nt, st) : launch_cfg<NCH, MAXNT, MINB, false, false>(p, nt, st);
}

}  // namespace

cudaError_t launch_cd_ahead(const CdParams& p, cudaStream_t st) {
  if (p.d_in & 3) return cudaErrorNotSupported;
  if ((reinterpret_cast<uintptr_t>(p.H) & 15) != 0) return cudaErrorNotSupported;
  if (p.H16 && ((p.d_in & 7) != 0 || (reinterpret_cast<uintptr_t>(p.H16) & 15) != 0)) return cudaErrorNotSupported;
  const long long ch = p.d_in >> 2;
  auto team = [&](long long chunks, int nch) { return (int)((chunks + nch - 1) / nch + 31) / 32 * 32; };
  // 384 threads as long as the row fits them: three warps per scheduler hide more latency than the two of 256 threads with up to
  // 14 chunks each (14336 x 1184 columns 236 -> 226 ms, 11008 x 296 47.4 -> 43.3), and at 168 registers little spills (52 bytes at most, 12 x
  // 384 per channel).  fp32 rows of 13825 to 14336 entries per channel fill 8 x 448 slots, with room for the table of H_ii beside them
  // (13828 x 592 columns 60.1 ms against 61.1 for 10 x 384, 14336 x 592 62.6 / 62.2, x 1184 120.3 / 120.5); in groups, and as bf16 rows, 10 x 384 is
  // the quicker one (a quarter of a pass, 8 x 448 / 10 x 384: 13952 in groups of 64 x 296 14.8 / 14.5 ms, 14336 in groups of 128 x 296 15.1 / 14.8, of
  // 4 x 148 7.95 / 7.39, bf16 14336 x 296 15.8 / 14.6 and in groups of 128 17.5 / 16.6).  Rows of
  // 15361 to 16384 entries fill 8 x 512 slots (72 ms against 75 for 11 x 384 on 16384 x 296; 9 x 512 spills: 18432 x 592 226 ms
  // against 210 for 12 x 384).
  if (ch <= 2304) return launch_mode<6, 384, 1>(p, team(ch, 6), st);
  if (ch <= 3072) return launch_mode<8, 384, 1>(p, team(ch, 8), st);
  if (ch <= 3456) return launch_mode<9, 384, 1>(p, team(ch, 9), st);
  if (ch <= 3584 && p.ng == 1 && !p.H16) return launch_cfg<8, 448, 1, false, false>(p, team(ch, 8), st);
  if (ch <= 3840) return launch_mode<10, 384, 1>(p, team(ch, 10), st);
  if (ch <= 4096) return launch_mode<8, 512, 1>(p, team(ch, 8), st);
  if (ch <= 4224) return launch_mode<11, 384, 1>(p, team(ch, 11), st);
  if (ch <= 4608) return launch_mode<12, 384, 1>(p, team(ch, 12), st);
  return cudaErrorNotSupported;
}

}  // namespace cdq
