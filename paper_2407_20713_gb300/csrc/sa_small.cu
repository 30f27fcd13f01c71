// sa_small.cu -- SA of problems with few chains (one smile of 64 chains is
// the paper's case): the whole calibration in one launch, one to four warps
// per chain.
//
// Such a problem cannot fill the GPU, and its time is the latency of its
// dependent Metropolis steps plus that of its level ends.  Both are cut here:
//
//  * Speculation K steps deep.  Acceptance is the common outcome (94-97% of
//    the evaluated proposals), so a chain forms the proposals of its next K
//    steps as if every one inside the box were accepted (one outside is
//    rejected for certain) and evaluates them side by side: NW warps, KW =
//    K / NW groups of P = 32 / KW lanes each, a group a point.  The steps are
//    then decided together -- step k's Metropolis test needs the cost of the
//    step before it, which is another group's -- and the chain advances past
//    the first rejection.  Its trajectory, counters and best point are those
//    of the one-step loop bit for bit.
//  * Every warp of a chain forms all K points and takes all K decisions
//    itself, so the warps exchange nothing but the K costs (one barrier an
//    iteration).
//  * Proposal words are drawn 32 steps at a time, a Philox block a lane.
//  * The blocks of a problem stay resident (a cooperative launch) and meet at
//    each level end on one counter: every block writes its minimum, arrives,
//    and takes the argmin over the minima itself.
//
// The misfit is summed in the order of ProblemDev::G lanes, played by the P
// lanes of a group (virtual_lanes_sum).
//
// FP64: a scheduler issues one FP64 warp instruction in about 76 cycles, so
// FP64 counts what FP64 instructions cost: box tests compare the numbers'
// bits, the words are kept as FP32 (2u - 1 is exact there), and a chain's
// warps sit on different schedulers.
#include <algorithm>
#include <cmath>

#include "arrivals.h"
#include "sa_device.cuh"
#include "sa_small.cuh"

namespace sabr {

constexpr int kRing = 64;        // steps whose proposal words a warp holds
constexpr int kLevelCache = 32;  // levels whose temperatures a block holds
constexpr int kSmallBlock = 128;

// Box tests.  FP64 bounds and numbers are compared as integers that order
// like the (finite) numbers: 32-bit ALU instructions instead of FP64 compares.
template <class R> struct BoxKey;
template <> struct BoxKey<float> {
  using T = float;
  static __device__ __forceinline__ T of(float x) { return x; }
};
template <> struct BoxKey<double> {
  using T = long long;
  static __device__ __forceinline__ T of(double x) {
    const long long b = __double_as_longlong(x);
    return b >= 0 ? b : (long long)(0x8000000000000000ull - (unsigned long long)b);  // -0 is 0
  }
};

// A proposal word 2u - 1, kept as the float it exactly is (an odd multiple of
// 2^-23 in (-1, 1)), in the working precision; to FP64 by moving its bits.
__device__ __forceinline__ float word_to(float w, float) { return w; }
__device__ __forceinline__ double word_to(float w, double) {
  const uint32_t b = __float_as_uint(w);
  const uint32_t hi = (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + ((1023u - 127u) << 20));
  return __hiloint2double((int)hi, (int)(b << 29));
}

// Barrier of a chain's NW warps (they are neighbours in the block).
template <int NW> __device__ __forceinline__ void chain_sync(int chain_in_block) {
  if constexpr (NW == 1) {
    __syncwarp();
  } else if constexpr (NW == kSmallBlock / 32) {
    __syncthreads();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + chain_in_block), "r"(32 * NW) : "memory");
  }
}

// Words of steps s0 .. s0 + 31 of a chain's level into a warp's ring, a Philox
// block a lane.
__device__ __forceinline__ void draw_words(uint32_t gchain, int level, int s0, uint32_t key0, uint32_t key1,
                                           float (*w)[kRing], float* u) {
  const int s = s0 + (threadIdx.x & 31), at = s & (kRing - 1);
  const uint4 b = philox4x32_10(make_uint4(gchain, (uint32_t)level, (uint32_t)s, kTagSA), key0, key1);
  __syncwarp();  // every lane has read the entries that are replaced
  w[0][at] = 2.0f * u01<float>(b.x) - 1.0f;
  w[1][at] = 2.0f * u01<float>(b.y) - 1.0f;
  w[2][at] = 2.0f * u01<float>(b.z) - 1.0f;
  w[3][at] = 2.0f * u01<float>(b.w) - 1.0f;
  u[at] = u01<float>(sa_accept_word(b.x, b.y, b.z));
  __syncwarp();
}

// A level one step after the other, by one warp with all its lanes on one point:
// for chains that accept less than half of what they evaluate (a start
// temperature far below the costs that a step makes), whose windows would be
// points evaluated in vain.  20 levels x 50 steps at 1% accepted, ms in windows |
// so: 64 chains x 15 quotes 1.87 | 0.78, 608 x 492 4.9 | 2.0, 1216 x 492 4.9 | 2.1,
// Obloj 1216 x 246 6.2 | 2.3; FP64 (6 levels), 64 x 246 20.8 | 11.3, Obloj 152 x 42 9.0
// | 5.0.  At 20% accepted windows are still the slower by 1.3 to 2.9.
template <class R> struct ChainState {
  R x[4], bx[4];
  typename CostOf<R>::T fcur, bf;
  unsigned ev, ac;
};
template <class R, int MODEL>
__device__ __forceinline__ void single_steps(const ProblemDev& P, uint32_t gchain, int level, const R* step4, float inv_Tk,
                                          double Tk, float (*w)[kRing], float* u, ChainState<R>& z) {
  using C = typename CostOf<R>::T;
  constexpr int D = 4;
  extern __shared__ __align__(16) unsigned char smem[];
  const SmemQuotes<R> sq = staged_quotes<R>(P.n_quotes, smem);
  const R l2f = (R)P.l2f;
  const int n_quotes = P.n_quotes, G = P.G, len = P.chain_len;
  const int units = StaticPoint<R, MODEL>::kPair ? (n_quotes + 1) >> 1 : n_quotes;
  const LaneSplit ls = lane_split(G, 32);
  // lane i & 3 forms coordinate i of the proposal and tests it
  const int ci = threadIdx.x & (D - 1);
  const R step = step4[ci];
  const auto lo = BoxKey<R>::of((R)P.lo[ci]), hi = BoxKey<R>::of((R)P.hi[ci]);
  R x[D], bx[D];
#pragma unroll
  for (int i = 0; i < D; ++i) x[i] = z.x[i], bx[i] = z.bx[i];
  C fcur = z.fcur, bf = z.bf;
  unsigned ev = z.ev, ac = z.ac;
  for (int st = 0; st < len; ++st) {
    if ((st & 31) == 0) draw_words(gchain, level, st, P.key0, P.key1, w, u);
    const int at = st & (kRing - 1);
    R xi = x[0];
#pragma unroll
    for (int i = 1; i < D; ++i) xi = ci == i ? x[i] : xi;
    const R y = move_by(xi, step, word_to(w[ci][at], R{}));
    const auto v = BoxKey<R>::of(y);
    if (__any_sync(0xffffffffu, v < lo || v > hi)) continue;
    R xs[D];
#pragma unroll
    for (int i = 0; i < D; ++i) xs[i] = __shfl_sync(0xffffffffu, y, i);
    const StaticPoint<R, MODEL> pt(xs, l2f, n_quotes);
    const C f = virtual_lanes_sum<R>(pt, units, G, ls, sq, 0xffffffffu);
    ++ev;
    if (cost_less(f, bf)) {
      bf = f;
#pragma unroll
      for (int i = 0; i < D; ++i) bx[i] = xs[i];
    }
    const auto delta = cost_delta(f, fcur);
    if (delta <= 0 || metropolis(word_to(u[at], R{}), delta, inv_Tk, Tk)) {
      ++ac;
      fcur = f;
#pragma unroll
      for (int i = 0; i < D; ++i) x[i] = xs[i];
    }
  }
#pragma unroll
  for (int i = 0; i < D; ++i) z.x[i] = x[i], z.bx[i] = bx[i];
  z.fcur = fcur, z.bf = bf, z.ev = ev, z.ac = ac;
}

// FP32 calls it, so that it takes neither registers nor order from the windows
// (inlined, 152 chains x 75 quotes take 4% longer); FP64 has registers to spare.
template <class R, int MODEL>
__device__ __noinline__ void single_steps_call(const ProblemDev& P, uint32_t gchain, int level, const R* step4,
                                               float inv_Tk, double Tk, float (*w)[kRing], float* u,
                                               ChainState<R>& z) {
  single_steps<R, MODEL>(P, gchain, level, step4, inv_Tk, Tk, w, u, z);
}

// What bounds it (64 chains, 15 quotes, 4 warps x 4 points: 3.95 ms for 200
// levels x 100 steps, 15.6 two steps at a time on 8 lanes): latency.  A level of
// no steps takes 4 us (the meeting of 64 blocks), a window of 16 steps about
// 1.2 us -- one dependent chain of proposals, formula, butterfly and decision on
// a warp alone on its scheduler -- and a level waits for its slowest chain.
// FP64, 4 x 2: 33.5 ms (173.9), FP64 instructions at 76 cycles each.
//
// Block minima alternate between two buffers by the level's parity: a block
// writes the minima of level k + 2 only after every block has read those of
// level k (it arrives at k + 1 after reading them).  The costs of an iteration
// alternate likewise.
//
// A block's chains go step by step (single_steps) in the level after one in
// which they accepted less than half of the proposals that they evaluated, and
// back.  The two kinds of levels have a loop each: one loop that asks per level
// costs the windows 4 to 6% (64 chains x 15 quotes, 200 x 100: 4.01 ms without
// the single steps, 4.28 in one loop, 3.95 in two).
//
// Blocks an SM of the largest launch of a shape (small_shape,
// small_most_chains); the registers are set by it.
template <class R, int NW, int KW>
constexpr int kSmallResident = sizeof(R) == 8 ? 1 : (KW == 2 ? 4 : (NW == 1 ? 2 : 1));
template <class R, int MODEL, int NW, int KW>
__global__ void __launch_bounds__(kSmallBlock, (kSmallResident<R, NW, KW>))
    sa_small_kernel(const ProblemDev* __restrict__ probs, const int4* __restrict__ work, unsigned long long wait_ns) {
  using C = typename CostOf<R>::T;
  using Key = typename BoxKey<R>::T;
  constexpr int D = 4, P = 32 / KW, K = NW * KW, CPB = kSmallBlock / 32 / NW;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ ProblemDev Pr;
  __shared__ R s_step[kLevelCache][D];
  __shared__ double s_Tk[kLevelCache];
  __shared__ float s_invTk[kLevelCache];
  __shared__ float s_w[kSmallBlock / 32][D][kRing];  // proposal words 2u - 1 of each warp
  __shared__ float s_u[kSmallBlock / 32][kRing];     // acceptance uniforms
  __shared__ __align__(16) R s_x[kSmallBlock / 32][K][D];  // points of the window
  __shared__ C s_f[CPB][2][K];                       // their costs
  __shared__ double s_mf[CPB], s_mx[CPB][D], s_new[D + 1];
  __shared__ int s_stop;
  __shared__ float s_low[CPB];                       // evaluations less twice the acceptances of a level
  const int4 it = work[blockIdx.x];
  load_problem(probs, it.x, &Pr);
  const int blk = it.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cb = warp / NW, wc = warp % NW;  // chain in the block, warp in the chain
  const int nb = (Pr.n_chains + CPB - 1) / CPB;
  unsigned char* rest;
  const SmemQuotes<R> sq = stage_quotes<R>(Pr, smem, blockDim.x, threadIdx.x, &rest);
  if (threadIdx.x == 0) s_stop = 0;
  const int chain = blk * CPB + cb;
  const bool active = chain < Pr.n_chains;
  const uint32_t gchain = (uint32_t)(Pr.chain0 + chain);
  const int k_own = wc * KW + lane / P;  // the step (of K) this lane evaluates
  constexpr unsigned kAll = K == 32 ? 0xffffffffu : (1u << K) - 1u;
  const R l2f = (R)Pr.l2f;
  const int n_quotes = Pr.n_quotes, G = Pr.G, len = Pr.chain_len, n_levels = Pr.n_levels;
  const int units = StaticPoint<R, MODEL>::kPair ? (n_quotes + 1) >> 1 : n_quotes;
  const LaneSplit ls = lane_split(G, P);
  const uint32_t key0 = Pr.key0, key1 = Pr.key1;
  // lane i & 3 forms coordinate i of the window's points
  const int ci = lane & (D - 1);
  Key lo[D], hi[D];
  R x[D], bx[D];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    lo[i] = BoxKey<R>::of((R)Pr.lo[i]);
    hi[i] = BoxKey<R>::of((R)Pr.hi[i]);
    x[i] = (R)__ldcg(&Pr.state[i]);
    bx[i] = x[i];
  }
  const double T0 = __ldcg(&Pr.state[kMaxD + 1]);
  C fcur = cost_from(__ldcg(&Pr.state[kMaxD]), C{});
  C bf = fcur;
  unsigned long long ev_all = 0, ac_all = 0;
  unsigned target = 0;
  int parity = 0;
  __syncthreads();

  auto level_begin = [&](int level) {
    // temperatures and step widths of the next kLevelCache levels, a level a
    // lane of warp 0 (FP64 square roots and divisions, off the levels' path)
    if ((level & (kLevelCache - 1)) == 0) {
      if (warp == 0 && level + lane < n_levels) {
        const double Tk0 = __dmul_rn(T0, Pr.ck[level + lane]);
        double sk = __dmul_rn(Pr.step0, __dsqrt_rn(__ddiv_rn(Tk0, T0)));
        if (sk < Pr.step_min) sk = Pr.step_min;
        for (int i = 0; i < D; ++i) s_step[lane][i] = (R)__dmul_rn(sk, __dsub_rn(Pr.hi[i], Pr.lo[i]));
        s_Tk[lane] = Tk0;
        s_invTk[lane] = (float)(1.4426950408889634 / Tk0);
      }
      __syncthreads();
    }
  };
  bool low = false;  // few of the proposals that the block's chains evaluated in the last level were accepted
  // argmin over the chains of the problem; false when a wait gave up
  auto level_end = [&](int level, unsigned ev, unsigned ac, auto single) {
    ev_all += ev;
    ac_all += ac;
    // warps that share windows all know a lone chain's counts
    constexpr bool kShared = CPB > 1 || decltype(single)::value;
    const float excess = (float)ev - 2.0f * (float)ac;
    if (!kShared) low = ac < ev - ac;
    if (wc == 0 && lane == 0) {
      s_mf[cb] = active ? cost_to_double(fcur) : INFINITY;
#pragma unroll
      for (int i = 0; i < D; ++i) s_mx[cb][i] = (double)x[i];
    }
    __syncthreads();
    if (kShared && wc == 0 && lane == 0) s_low[cb] = active ? excess : 0.0f;
    target += (unsigned)nb;
    if (warp == 0) {
      double* mf = Pr.part_f + (size_t)(level & 1) * nb;
      int* mc = Pr.part_c + (size_t)(level & 1) * nb;
      double* mx = Pr.part_x + (size_t)(level & 1) * nb * kMaxD;
      double f = INFINITY;
      int w = 0x7fffffff;
      for (int i = 0; i < CPB; ++i) argmin_merge(f, w, s_mf[i], i);
      if (w >= CPB) w = 0;  // no cost compares
      if (lane < D) __stcg(&mx[(size_t)blk * kMaxD + lane], s_mx[w][lane]);
      if (lane == D) __stcg(&mf[blk], f);
      if (lane == D + 1) __stcg(&mc[blk], blk * CPB + w);
      __threadfence();
      __syncwarp();
      if (lane == 0) {
        atomicAdd(Pr.arrive, 1u);
        volatile unsigned int* ctr = Pr.arrive;
        volatile unsigned int* err = Pr.arrive + 1;
        bool ok = arrived(*ctr, target);
        if (!ok) {
          const unsigned long long t0 = global_ns();
          while (!(ok = arrived(*ctr, target))) {
            if (*err) break;
            if (global_ns() - t0 > wait_ns) {
              atomicExch(Pr.arrive + 1, 1u);
              break;
            }
          }
        }
        s_stop = !ok;
        __threadfence();
      }
      __syncwarp();
      if (!s_stop) {
        double g = INFINITY;
        int b = 0x7fffffff;
        for (int i = lane; i < nb; i += 32) argmin_merge(g, b, __ldcg(&mf[i]), i);
        warp_argmin(g, b);
        if (b >= nb) b = 0;
        if (lane < D) s_new[lane] = __ldcg(&mx[(size_t)b * kMaxD + lane]);
        if (lane == D) s_new[D] = g;
        if (blk == 0 && level + 1 == n_levels) {
          if (lane < kMaxD) Pr.state[lane] = lane < D ? __ldcg(&mx[(size_t)b * kMaxD + lane]) : 0.0;
          if (lane == 0) {
            Pr.state[kMaxD] = g;
            Pr.state[kStateArgChain] = (double)(Pr.chain0 + __ldcg(&mc[b]));
          }
        }
      }
    }
    __syncthreads();
    if (s_stop) return false;
#pragma unroll
    for (int i = 0; i < D; ++i) x[i] = (R)s_new[i];
    fcur = cost_from(s_new[D], C{});
    if (kShared) {
      float balance = 0.0f;
#pragma unroll
      for (int i = 0; i < CPB; ++i) balance += s_low[i];
      low = balance > 0.0f;
    }
    return true;
  };

  int level = 0;
  while (level < n_levels) {
    for (; level < n_levels && !low; ++level) {
      level_begin(level);
      unsigned ev = 0, ac = 0;
      if (active) {
        const R step = s_step[level & (kLevelCache - 1)][ci];
        const float inv_Tk = s_invTk[level & (kLevelCache - 1)];
        const double Tk = s_Tk[level & (kLevelCache - 1)];
        int filled = 0;  // steps whose words are in the ring
        int st = 0;
        while (st < len) {
          if (filled < len && filled < st + K) {
            draw_words(gchain, level, filled, key0, key1, s_w[warp], s_u[warp]);
            filled += 32;
          }
          R xi0 = x[0];
#pragma unroll
          for (int i = 1; i < D; ++i) xi0 = ci == i ? x[i] : xi0;
          const int nv = len - st < K ? len - st : K;  // steps of this window
          const unsigned window = nv == K ? kAll : (1u << nv) - 1u;
          // the window's points if every proposal inside the box is accepted;
          // one found outside (skip) is rejected for certain, and the points
          // after it start from the one before it
          unsigned skip = 0, out;
          R w[K];
#pragma unroll
          for (int j = 0; j < K; ++j) w[j] = word_to(s_w[warp][ci][(st + j) & (kRing - 1)], R{});
          do {
            R cur = xi0;
#pragma unroll
            for (int j = 0; j < K; ++j) {
              const R y = move_by(cur, step, w[j]);
              if (lane < D) s_x[warp][j][ci] = y;
              cur = (skip >> j) & 1u ? cur : y;
            }
            __syncwarp();
            const R* y = s_x[warp][K == 32 ? lane : (lane & (K - 1))];
            bool in = true;
#pragma unroll
            for (int i = 0; i < D; ++i) {
              const Key v = BoxKey<R>::of(y[i]);
              in = in && !(v < lo[i] || v > hi[i]);
            }
            out = ~__ballot_sync(0xffffffffu, in) & window & ~skip;
            skip |= out & (0u - out);
          } while (out);
          const unsigned in_mask = window & ~skip;
          unsigned rej = 0;
          if (in_mask) {
            R xs[D];
#pragma unroll
            for (int i = 0; i < D; ++i) xs[i] = s_x[warp][k_own][i];
            const StaticPoint<R, MODEL> pt(xs, l2f, n_quotes);
            const C fo = virtual_lanes_sum<R>(pt, units, G, ls, sq, 0xffffffffu);
            C* fb = s_f[cb][parity];
            parity ^= 1;
            if ((lane & (P - 1)) == 0) fb[k_own] = fo;
            chain_sync<NW>(cb);
            // lane k decides step k
            const int k = lane & (K - 1);
            const C f = fb[k];
            const unsigned before = in_mask & ((1u << k) - 1u);  // the nearest earlier step inside the box
            const C fe = fb[before ? 31 - __clz(before) : 0];
            const C fp = before ? fe : fcur;
            const auto delta = cost_delta(f, fp);
            const R u = word_to(s_u[warp][(st + k) & (kRing - 1)], R{});
            const bool acc = delta <= 0 || metropolis(u, delta, inv_Tk, Tk);
            rej = __ballot_sync(0xffffffffu, !acc) & in_mask;
            const int first = __ffs(rej) - 1;  // the first rejected step
            const unsigned eval = rej ? in_mask & ((2u << first) - 1u) : in_mask;
            const unsigned taken = rej ? eval & ~(1u << first) : eval;
            ev += __popc(eval);
            ac += __popc(taken);
            unsigned better = __ballot_sync(0xffffffffu, cost_less(f, bf)) & eval;
            if (better) {
              int at = 0;
              while (better) {
                const int l = __ffs(better) - 1;
                better &= better - 1u;
                if (cost_less(fb[l], bf)) {
                  bf = fb[l];
                  at = l;
                }
              }
#pragma unroll
              for (int i = 0; i < D; ++i) bx[i] = s_x[warp][at][i];
            }
            if (taken) {
              const int last = 31 - __clz(taken);
              fcur = fb[last];
#pragma unroll
              for (int i = 0; i < D; ++i) x[i] = s_x[warp][last][i];
            }
            st += rej ? first + 1 : nv;
          } else {
            st += nv;
          }
          __syncwarp();  // the points are read before the next window's are written
        }
      }
      if (!level_end(level, ev, ac, IntTag<0>{})) return;
    }
    // the chains' first warps run the levels step by step, and the level end hands
    // their state to the others, until acceptance is the common outcome again
    for (; level < n_levels && low; ++level) {
      level_begin(level);
      unsigned ev = 0, ac = 0;
      if (active && wc == 0) {
        ChainState<R> z;
#pragma unroll
        for (int i = 0; i < D; ++i) z.x[i] = x[i], z.bx[i] = bx[i];
        z.fcur = fcur, z.bf = bf, z.ev = 0, z.ac = 0;
        const int at = level & (kLevelCache - 1);
        if constexpr (sizeof(R) == 8)
          single_steps<R, MODEL>(Pr, gchain, level, s_step[at], s_invTk[at], s_Tk[at], s_w[warp], s_u[warp], z);
        else
          single_steps_call<R, MODEL>(Pr, gchain, level, s_step[at], s_invTk[at], s_Tk[at], s_w[warp], s_u[warp], z);
#pragma unroll
        for (int i = 0; i < D; ++i) x[i] = z.x[i], bx[i] = z.bx[i];
        fcur = z.fcur, bf = z.bf, ev = z.ev, ac = z.ac;
      }
      if (!level_end(level, ev, ac, IntTag<1>{})) return;
    }
  }
  if (n_levels > 0 && active && wc == 0 && lane == 0) {
    Pr.chain_bf[chain] = cost_to_double(bf);
    Pr.chain_ev[chain] = ev_all;
    Pr.chain_ac[chain] = ac_all;
    R* row = (R*)Pr.chain_bx + (size_t)chain * kMaxD;
#pragma unroll
    for (int i = 0; i < kMaxD; ++i) row[i] = i < D ? bx[i < D ? i : 0] : (R)0;
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
bool small_supported(int prec, int model) {
  return model == SABR_HAGAN || model == SABR_OBLOJ || (model == SABR_EXPANDED && prec == SABR_FP64);
}

// FP32, ms per calibration on 152 SMs (level kernels and queue | shapes, the
// chosen one first):
//   64 chains, 15 quotes, 200 x 100: 16.5 | 4 warps x 4 points 3.95, 4 x 2 4.21, 1 x 4 5.30
//   152 chains, 64 quotes, 50 x 50: 2.96 | 4 x 4 0.97, 4 x 2 0.91, 1 x 4 1.26
//   152 chains, 80 quotes, 50 x 50: 3.33 | 4 x 2 1.06, 4 x 4 1.23, 1 x 4 1.57
//   503 chains, 350 quotes, 28 x 97: 4.73 | 4 x 2 2.29, 1 x 4 3.00
//   600 chains, 21 quotes, 50 x 50: 3.25 | 4 x 2 1.28, 1 x 4 1.18
//   1000 chains, 11 quotes, 50 x 50: 3.26 | 1 x 4 1.04
//   1024 chains, 200 quotes, 40 x 50: 3.85 | 1 x 4 2.10
// A point too deep costs evaluations that are dropped, so few quotes take the
// deeper window.  FP64, whose time is FP64 instructions a scheduler: two
// points a warp, as many warps a chain as give every scheduler one (15 quotes, 50
// levels: 64 chains x 100 steps 47.6 | 4 x 2 8.56, 2 x 2 12.3, 1 x 2 19.9; 300 chains
// x 50 25.9 | 2 x 2 7.35, 4 x 2 8.58, 1 x 2 10.9; 600 x 50 26.8 | 1 x 2 11.3, 2 x 2 12.2).
SmallShape small_shape(int prec, int n_quotes, long long chains) {
  const long long sms = device_sms();
  if (prec == SABR_FP64) return SmallShape{chains <= sms ? 4 : (chains <= 2 * sms ? 2 : 1), 2};
  if (chains <= sms && n_quotes <= 64) return SmallShape{4, 4};
  if (chains <= 4 * sms) return SmallShape{4, 2};
  return SmallShape{1, 4};
}
long long small_most_chains(int prec) { return (prec == SABR_FP64 ? 4 : 8) * (long long)device_sms(); }

int small_blocks(const SmallShape& s, int n_chains) {
  const int cpb = kSmallBlock / 32 / s.nw;
  return (n_chains + cpb - 1) / cpb;
}

size_t small_smem_bytes(int prec, int model, int Q, int M) { return level_smem_bytes(prec, model, Q, M, 1); }

using SmallFn = void (*)(const ProblemDev*, const int4*, unsigned long long);
template <int MODEL> static SmallFn small_fn_fp32(const SmallShape& s) {
  if (s.nw == 1) return sa_small_kernel<float, MODEL, 1, 4>;
  return s.kw == 4 ? sa_small_kernel<float, MODEL, 4, 4> : sa_small_kernel<float, MODEL, 4, 2>;
}
template <int MODEL> static SmallFn small_fn_fp64(const SmallShape& s) {
  if (s.nw == 1) return sa_small_kernel<double, MODEL, 1, 2>;
  return s.nw == 2 ? sa_small_kernel<double, MODEL, 2, 2> : sa_small_kernel<double, MODEL, 4, 2>;
}
static SmallFn small_fn(int prec, int model, const SmallShape& s) {
  if (prec == SABR_FP32) return model == SABR_HAGAN ? small_fn_fp32<SABR_HAGAN>(s) : small_fn_fp32<SABR_OBLOJ>(s);
  switch (model) {
    case SABR_HAGAN: return small_fn_fp64<SABR_HAGAN>(s);
    case SABR_OBLOJ: return small_fn_fp64<SABR_OBLOJ>(s);
    default: return small_fn_fp64<SABR_EXPANDED>(s);
  }
}

int small_capacity(int prec, int model, const SmallShape& s, size_t smem) {
  const SmallFn fn = small_fn(prec, model, s);
  cudaFuncAttributes at;
  if (cudaFuncGetAttributes(&at, (const void*)fn) != cudaSuccess) return 0;
  if (smem + at.sharedSizeBytes > 227 * 1024 ||
      allow_smem((const void*)fn, smem) != cudaSuccess)
    return 0;
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (const void*)fn, kSmallBlock, smem) != cudaSuccess) return 0;
  return nb * device_sms();
}

cudaError_t launch_small(int prec, int model, const SmallShape& shape, const ProblemDev* probs, const int4* work,
                         int blocks, size_t smem, unsigned long long wait_ns, cudaStream_t s) {
  void* args[] = {&probs, &work, &wait_ns};
  return cudaLaunchCooperativeKernel((const void*)small_fn(prec, model, shape), dim3(blocks), dim3(kSmallBlock), args,
                                     smem, s);
}

}  // namespace sabr
