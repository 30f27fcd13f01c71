// mc.cuh -- fused Monte Carlo pricer of Sec. 4: one thread per path, the
// log-Euler scheme of eq. (dis_SABRd) in log space, payoffs of every option
// of a maturity accumulated when the path lands on it, eq. (payoff).
#pragma once
#include <cstdint>

#include "../../include/sabr.h"
#include "sabr_math.cuh"

namespace sabr {

constexpr int kMcBlock = 128;         // threads per MC block (4 warps)
constexpr int kMcWarps = kMcBlock / 32;
constexpr int kMaxMcQuotes = 512;     // options per pricing call
constexpr int kMaxMcSteps = 8192;     // grid points per path

// One pricing problem (quotes sorted by maturity; all pointers device).
struct McDev {
  int model;          // static models use constant nu, rho
  int n_quotes, n_mats, n_steps, n_slots;
  int64_t n_paths;
  double fwd, log_absorb;  // ln(1e-12 f)
  uint32_t key0, key1;
  PhiloxKeys rk;           // the ten round keys of (key0, key1): kernel
                           // parameters, read as constants by the path loop
  const double* step_t;    // [n_steps] dynamic models: right end t_{i+1} of
                           // step i, where its nu(t), rho(t) are taken;
                           // static models: sqrt(step_h[i])
  const double* step_h;    // [n_steps] length of step i
  const int* step_mat;     // [n_steps] maturity reached at the end of step i, or -1
  const int* mat_q0;       // [n_mats] first quote of each maturity
  const int* mat_nq;       // [n_mats] its number of quotes
  const int* mat_slot;     // [n_mats] first accumulator slot (32 values each)
  const double* K;         // [n_quotes]
  const int8_t* is_call;   // [n_quotes]
  const void* tab;         // step tables [set][n_steps] written by
                           // mc_steps_kernel, or null: each block builds its own
};

// Butterfly reduce-scatter across a warp: on entry every lane holds 32
// values v[0..31]; on exit lane l holds the warp sum of value l.  Five
// levels, 16+8+4+2+1 shuffles, fixed order (deterministic).
template <class R>
__device__ __forceinline__ R warp_reduce_scatter32(R (&v)[32], int lane) {
#pragma unroll
  for (int lvl = 0; lvl < 5; ++lvl) {
    const int half = 16 >> lvl;
    const bool upper = (lane & half) != 0;
#pragma unroll
    for (int k = 0; k < half; ++k) {
      const R keep = upper ? v[k + half] : v[k];
      const R send = upper ? v[k] : v[k + half];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, half);
    }
  }
  return v[0];
}

// Path state units: FP32 paths carry log2 F and log2 alpha, so that nu-hat =
// alpha F^(beta-1) and F come from one SFU exp2 each; FP64 paths carry the
// natural logarithms.  kLogUnit converts a natural-log increment.
template <class R> struct PathUnits;
template <> struct PathUnits<float> {
  static constexpr double kLogUnit = 1.4426950408889634;  // 1/ln 2
  __device__ static float expu(float x) { return ex2_approx(x); }
  __host__ __device__ static double logu(double x) { return log2(x); }
};
template <> struct PathUnits<double> {
  static constexpr double kLogUnit = 1.0;
  __device__ static double expu(double x) { return exp(x); }
  __host__ __device__ static double logu(double x) { return log(x); }
};

// Per-block step coefficients, in shared memory (one 16-byte load per step
// in FP32), scaled by the log unit u:
//   a_i = u nu_i sqrt(h_i)    (vol step; its drift -u nu_i^2 h_i / 2 is
//                              -a_i^2 / (2 u), formed in the step)
//   c_i = u rho_i sqrt(h_i)   d_i = u sqrt(1 - rho_i^2) sqrt(h_i)
//   e_i = -u h_i / 2
// FP32 tables hold -c_i and -d_i: the FP32 step works with the negated
// normals (path_step2).
template <class R> struct __align__(16) StepCoef {
  R a, c, d, e;
};

template <class R>
__device__ __forceinline__ StepCoef<R> step_coef(double nu, double rho_term, double orth, double h, double sh) {
  const double u = PathUnits<R>::kLogUnit, sg = sizeof(R) == 4 ? -u : u;
  StepCoef<R> s;
  s.a = (R)(u * nu * sh);
  s.c = (R)(sg * rho_term * sh);
  s.d = (R)(sg * orth * sh);
  s.e = (R)(-0.5 * u * h);
  return s;
}
// nu(t), rho(t) of a dynamic model.
__device__ __forceinline__ void dynamic_nu_rho(int model, const double* p, double t, double& nu, double& rho) {
  if (model == SABR_DYN_I) {
    rho = p[2] * exp(-p[4] * t);
    nu = p[3] * exp(-p[5] * t);
  } else {
    rho = (p[2] + p[8] * t) * exp(-p[4] * t) + p[6];
    nu = (p[3] + p[9] * t) * exp(-p[5] * t) + p[7];
  }
}
template <class R>
__device__ __forceinline__ StepCoef<R> dynamic_step_coef(const McDev& P, const double* p, int i) {
  const double h = P.step_h[i];
  double nu, rho;
  dynamic_nu_rho(P.model, p, P.step_t[i], nu, rho);
  return step_coef<R>(nu, rho, sqrt(fmax(0.0, (1.0 - rho) * (1.0 + rho))), h, sqrt(h));
}

// The block's step table: copied from P.tab, or built here; also writes
// land[m] = the step whose end is maturity m.  A static model's entry is four
// FP64 products (square roots once per thread or by the host).  A dynamic
// model's needs two FP64 exponentials and two square roots, about 80
// instructions on a pipe that takes 1.7 a clock, for every block of an SM, so
// mc_steps_kernel forms it once per set unless the launch is small
// (mc_blocks_build_steps).
template <class R>
__device__ __forceinline__ void build_steps(const McDev& P, const double* p, int set, StepCoef<R>* tab, int* land) {
  const bool dyn = P.model == SABR_DYN_I || P.model == SABR_DYN_II;
  if (P.tab != nullptr) {
    const StepCoef<R>* src = (const StepCoef<R>*)P.tab + (size_t)set * P.n_steps;
    for (int i = threadIdx.x; i < P.n_steps; i += blockDim.x) tab[i] = src[i];
  } else if (dyn) {
    for (int i = threadIdx.x; i < P.n_steps; i += blockDim.x) tab[i] = dynamic_step_coef<R>(P, p, i);
  } else {
    const double orth = sqrt(fmax(0.0, (1.0 - p[2]) * (1.0 + p[2])));
    for (int i = threadIdx.x; i < P.n_steps; i += blockDim.x)
      tab[i] = step_coef<R>(p[3], p[2], orth, P.step_h[i], P.step_t[i]);
  }
  for (int i = threadIdx.x; i < P.n_steps; i += blockDim.x) {
    const int m = P.step_mat[i];
    if (m >= 0) land[m] = i;
  }
}

// FP32: SFU forms.  -2 ln u1 = -2 ln 2 log2 u1 lies in (0, 34] for u1 in
// [2^-24, 1 - 2^-24], so sqrt = s rsqrt(s); the angle 2 pi u2 - pi lies in
// (-pi, pi), where the SFU sine and cosine keep an absolute error below
// 2^-21, and (cos, sin)(2 pi u2) = -(cos, sin)(2 pi u2 - pi).  Every operand
// is a normal number, so the flush-to-zero forms apply.
__device__ __forceinline__ void box_muller(float u1, float u2, float& z1, float& z2) {
  const float s2 = -1.38629436111989061f * lg2_approx(u1);
  const float r = s2 * rsqrt_approx(s2);
  const float ang = 6.28318530717958647692f * u2 - 3.14159265358979323846f;
  const float s = sin_approx(ang), c = cos_approx(ang);
  z1 = -r * c;
  z2 = -r * s;
}
__device__ __forceinline__ void box_muller(double u1, double u2, double& z1, double& z2) {
  const double r = sqrt(-2.0 * log(u1));
  double s, c;
  sincospi(2.0 * u2, &s, &c);
  z1 = r * c;
  z2 = r * s;
}

// State of one path in log units, and one step of the log-Euler scheme of
// eq. (dis_SABRd): the normals of steps 2m and 2m + 1 come, by Box-Muller,
// from words (x, y) and (z, w) of Philox block (path, m, 0, tag) -- see
// path_words; nu-hat uses the old alpha and the old F.  A path is absorbed
// once F < 1e-12 f (its F reads 0 from then on).
template <class R> struct PathState {
  R lnF, lnA;
  bool absorbed;
};

// Block m = i / 2 of a path, FP64 (register-heavy: the key schedule is
// stepped); the FP32 loops form the same words with path_block.
__device__ __forceinline__ uint4 path_words(const McDev& P, int64_t path, int i) {
  return philox4x32_10(make_uint4((uint32_t)path, (uint32_t)(i >> 1), 0u, kTagMC), P.key0, P.key1);
}

template <class R>
__device__ __forceinline__ void path_step(const StepCoef<R>& s, uint32_t wa, uint32_t wb, R beta_m1, R log_abs,
                                          PathState<R>& st) {
  R z1, z2;
  box_muller(u01<R>(wa), u01<R>(wb), z1, z2);
  const R nuhat = PathUnits<R>::expu(st.lnA + beta_m1 * st.lnF);
  st.lnF = st.lnF + nuhat * (s.c * z1 + s.d * z2) + nuhat * nuhat * s.e;
  const R b_over_a = s.a * (R)(-0.5 / PathUnits<R>::kLogUnit);  // b = a * b_over_a
  st.lnA = st.lnA + s.a * (z1 + b_over_a);
  st.absorbed = st.absorbed || !(st.lnF >= log_abs);
}

// Paths per thread: independent paths advance step by step together
// (independent dependency chains for the scheduler).  FP64 takes three
// (measured fastest against two and four); FP32 takes four, two pairs of
// paths stepped with the packed FP32x2 instructions (run_path_pairs).
constexpr int kMcPathsPerThread = 3;
__host__ __device__ constexpr int mc_paths_per_thread(int prec) { return prec == SABR_FP32 ? 4 : kMcPathsPerThread; }

// Simulates, with every thread of the grid, the paths path0 + k pstride
// (k = 0 .. kMcPathsPerThread - 1), then the next kMcPathsPerThread
// pstride, ... of one parameter set and adds, per warp, the sums of payoff
// and payoff^2 of every option to wacc[warp][slot * 32 + lane] (FP64).
// Values of maturity m are laid out as (option j, kind k) -> value 2 j + k,
// in chunks of 32 starting at slot mat_slot[m].  Steps go in pairs: one
// Philox block per path feeds both.
template <class R>
__device__ __forceinline__ void simulate_paths_scalar(const McDev& P, const double* p,
                                               const StepCoef<R>* tab, const int* land,
                                               const int* s_q0, const int* s_nq, const int* s_slot,
                                               const R* sK, const int8_t* scall, int64_t path0,
                                               int64_t pstride, double* wacc) {
  constexpr int NPT = kMcPathsPerThread;
  const int lane = threadIdx.x & 31;
  const R beta_m1 = (R)(p[1] - 1.0);
  const R lnf = (R)PathUnits<R>::logu(P.fwd), lna = (R)PathUnits<R>::logu(p[0]);
  const R log_abs = (R)(P.log_absorb * PathUnits<R>::kLogUnit);
  const int64_t n_paths = P.n_paths;
  const int n_steps = P.n_steps;
  // every lane of the warp runs the same trip count (idle lanes pay 0)
  const int64_t warp_path0 = path0 - lane;
  for (int64_t wp = warp_path0; wp < n_paths; wp += NPT * pstride) {
    int64_t path[NPT];
    bool live[NPT];
    PathState<R> st[NPT];
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      path[k] = wp + k * pstride + lane;
      live[k] = path[k] < n_paths;
      st[k] = PathState<R>{lnf, lna, false};
    }
    int m = 0, i_land = land[0];  // next maturity and the step it ends
    // payoffs of maturity m on the NPT paths, summed into the warp rows
    auto pay_out = [&]() {
      R F[NPT];
#pragma unroll
      for (int k = 0; k < NPT; ++k) F[k] = st[k].absorbed || !live[k] ? (R)0 : PathUnits<R>::expu(st[k].lnF);
      const int q0 = s_q0[m], nq = s_nq[m], slot0 = s_slot[m];
      for (int c0 = 0; c0 < 2 * nq; c0 += 32) {
        R v[32];
#pragma unroll
        for (int kk = 0; kk < 32; kk += 2) {
          const int j = (c0 + kk) >> 1;
          R pay = (R)0, pay2 = (R)0;
          if (j < nq) {
            const R K = sK[q0 + j];
            const bool call = scall[q0 + j] != 0;
#pragma unroll
            for (int k = 0; k < NPT; ++k) {
              const R x = call ? (F[k] > K ? F[k] - K : (R)0) : (K > F[k] ? K - F[k] : (R)0);
              const R y = live[k] ? x : (R)0;
              pay += y;
              pay2 += y * y;
            }
          }
          v[kk] = pay;
          v[kk + 1] = pay2;
        }
        const R tot = warp_reduce_scatter32<R>(v, lane);
        const int slot = slot0 + (c0 >> 5);
        wacc[slot * 32 + lane] += (double)tot;
      }
      ++m;
      i_land = m < P.n_mats ? land[m] : -1;
    };
    for (int i = 0; i < n_steps; i += 2) {
      uint4 w[NPT];
#pragma unroll
      for (int k = 0; k < NPT; ++k) w[k] = path_words(P, path[k], i);
      {
        const StepCoef<R> s = tab[i];
#pragma unroll
        for (int k = 0; k < NPT; ++k) path_step<R>(s, w[k].x, w[k].y, beta_m1, log_abs, st[k]);
      }
      if (i == i_land) pay_out();
      if (i + 1 < n_steps) {
        const StepCoef<R> s = tab[i + 1];
#pragma unroll
        for (int k = 0; k < NPT; ++k) path_step<R>(s, w[k].z, w[k].w, beta_m1, log_abs, st[k]);
        if (i + 1 == i_land) pay_out();
      }
    }
  }
}

// u01<float> of two words: the funnel shift (0x7F : w) >> 9 is 0x3F800000 |
// (w >> 9), i.e. 1 + (w >> 9) 2^-23, in one instruction, and the exact
// subtraction of 1 - 2^-24 is packed.
__device__ __forceinline__ float2 u01_pair(uint32_t w0, uint32_t w1) {
  return add2(make_float2(__uint_as_float(__funnelshift_r(w0, 0x7Fu, 9)),
                          __uint_as_float(__funnelshift_r(w1, 0x7Fu, 9))),
              f2(-0.99999994039535522f));
}

// Minimum that keeps a NaN: a path is absorbed iff its lowest ln F so far is
// not >= the threshold.  One instruction a step, where a flag per path took
// four (the flags outnumber the predicate registers and were packed and
// unpacked around every step).
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// Two FP32 paths of one log-Euler step with the packed FP32x2 instructions:
// the adds, multiplies and FMAs of both paths share an issue slot; the SFU
// operations and the absorption test stay per path.  The normals are z1 = -r
// cos, z2 = -r sin; with zr1 = r cos, zr2 = r sin the signs go into the step
// coefficients (nc = -c, nd = -d, as the FP32 table holds them).
// ORDER: how the forward's increment nuhat (c z1 + d z2) + nuhat^2 e is
// rounded; the European pricer and the cliquet keep an order each, so that
// their prices stay what they were bit for bit.
enum { kOrderEuropean = 0, kOrderCliquet = 1 };
template <int ORDER>
__device__ __forceinline__ void path_step2(const StepCoef<float>& s, uint32_t wa0, uint32_t wb0, uint32_t wa1,
                                           uint32_t wb1, float beta_m1, float2& lnF, float2& lnA, float& low0,
                                           float& low1) {
  const float2 u1 = u01_pair(wa0, wa1), u2 = u01_pair(wb0, wb1);
  const float2 s2 = mul2(f2(-1.38629436111989061f), make_float2(lg2_approx(u1.x), lg2_approx(u1.y)));
  const float2 r = mul2(s2, make_float2(rsqrt_approx(s2.x), rsqrt_approx(s2.y)));
  const float2 ang = fma2(f2(6.28318530717958647692f), u2, f2(-3.14159265358979323846f));
  const float2 zr1 = mul2(r, make_float2(cos_approx(ang.x), cos_approx(ang.y)));
  const float2 zr2 = mul2(r, make_float2(sin_approx(ang.x), sin_approx(ang.y)));
  // nu-hat from the old alpha and the old F
  const float2 arg = fma2(f2(beta_m1), lnF, lnA);
  const float2 nuhat = make_float2(ex2_approx(arg.x), ex2_approx(arg.y));
  constexpr float kDrift = (float)(-0.5 / PathUnits<float>::kLogUnit);  // vol drift / a^2
  if constexpr (ORDER == kOrderEuropean) {
    const float2 t = fma2(f2(s.d), zr2, mul2(f2(s.c), zr1));  // c z1 + d z2
    lnF = fma2(nuhat, fma2(nuhat, f2(s.e), t), lnF);
    lnA = fma2(f2(s.a), fma2(zr1, f2(-1.0f), f2(s.a * kDrift)), lnA);  // a (z1 + a kDrift)
  } else {
    const float2 t = fma2(f2(s.c), zr1, mul2(f2(s.d), zr2));
    lnF = fma2(mul2(nuhat, nuhat), f2(s.e), fma2(nuhat, t, lnF));
    lnA = fma2(f2(-s.a), fma2(f2(-s.a), f2(kDrift), zr1), lnA);
  }
  low0 = min_nan(low0, lnF.x);
  low1 = min_nan(low1, lnF.y);
}

// The part of a path's Philox blocks that no step changes.  Block m of path j
// has counter (j, m, 0, tag): its third word is 0 and m enters the second, so
// round 1 multiplies only the path (x1 = m ^ k0), round 2 the step (m ^ k0)
// and the path apart, and round 3 has one product of the path alone.  The
// path's products are formed once per path and the step's once per block for
// all paths of the thread; rounds 3 (one product) to 10 remain: 15 wide
// multiplies a block instead of 20, the same words bit for bit.
struct PathKey {
  uint32_t p1, p2, p3, p4;
};
__device__ __forceinline__ PathKey path_key(const PhiloxKeys& rk, uint32_t path) {
  const uint32_t ma = 0xD2511F53u, mb = 0xCD9E8D57u;
  const uint64_t a1 = (uint64_t)ma * path;
  const uint32_t z1 = (uint32_t)(a1 >> 32) ^ kTagMC ^ rk.k1[0];
  const uint64_t b2 = (uint64_t)mb * z1;
  const uint32_t x2 = (uint32_t)(b2 >> 32) ^ rk.k0[1];
  const uint64_t a3 = (uint64_t)ma * x2;
  return PathKey{(uint32_t)a1 ^ rk.k1[1], (uint32_t)b2 ^ rk.k0[2], (uint32_t)(a3 >> 32) ^ rk.k1[2], (uint32_t)a3};
}
// Step part of block m: both halves of round 2's product of the step.
__device__ __forceinline__ uint64_t path_step_key(const PhiloxKeys& rk, uint32_t m) {
  return (uint64_t)0xD2511F53u * (m ^ rk.k0[0]);
}
__device__ __forceinline__ uint4 path_block(const PhiloxKeys& rk, const PathKey& k, uint64_t sk) {
  const uint32_t ma = 0xD2511F53u, mb = 0xCD9E8D57u;
  const uint64_t b3 = (uint64_t)mb * ((uint32_t)(sk >> 32) ^ k.p1);
  uint4 c = make_uint4((uint32_t)(b3 >> 32) ^ k.p2, (uint32_t)b3, (uint32_t)sk ^ k.p3, k.p4);
#pragma unroll
  for (int r = 3; r < 10; ++r) {
    const uint64_t pa = (uint64_t)ma * c.x, pb = (uint64_t)mb * c.z;
    c = make_uint4((uint32_t)(pb >> 32) ^ c.y ^ rk.k0[r], (uint32_t)pb, (uint32_t)(pa >> 32) ^ c.w ^ rk.k1[r],
                   (uint32_t)pa);
  }
  return c;
}

// PAIRS pairs of FP32 paths through every step of the grid; at_land() is
// called when the step that ends at a maturity (the first: i_land) is done
// and returns the next such step, or -1.
template <int PAIRS> struct PathPairs {
  PathKey key[2 * PAIRS];
  float2 lnF[PAIRS], lnA[PAIRS];
  float low[2 * PAIRS];  // lowest ln F reached
  __device__ __forceinline__ void start(const McDev& P, float lnf, float lna, int64_t path, int64_t stride) {
#pragma unroll
    for (int k = 0; k < 2 * PAIRS; ++k) {
      key[k] = path_key(P.rk, (uint32_t)(path + k * stride));
      // opaque: the compiler would form parts of the key again in every block
      // (a wide multiply holds the FMA pipe for four cycles)
      asm volatile("" : "+r"(key[k].p1), "+r"(key[k].p2), "+r"(key[k].p3), "+r"(key[k].p4));
      low[k] = INFINITY;
    }
#pragma unroll
    for (int k = 0; k < PAIRS; ++k) {
      lnF[k] = make_float2(lnf, lnf);
      lnA[k] = make_float2(lna, lna);
    }
  }
  __device__ __forceinline__ float forward(int k, float log_abs) const {  // F, 0 once absorbed
    const float lf = (k & 1) ? lnF[k >> 1].y : lnF[k >> 1].x;
    return low[k] >= log_abs ? PathUnits<float>::expu(lf) : 0.0f;
  }
};
// Blocks of two steps without a landing between them run as straight-line
// code in which the words of one pair are formed while the other pair (or,
// with one pair, the block before) takes its steps: Philox fills the FMA pipe
// (a wide multiply holds it four cycles, a packed FP32x2 operation two) and
// Box-Muller the SFU, and neither waits for the other.  What bounds the loop: a
// path and step take about 45 cycles of a scheduler's FMA pipe (7.5 wide
// multiplies 30, packed FP32 14, the step's key and drift 1) and 36 of its SFU; 60
// are measured.  2^22 paths
// x 504 steps: 4.17 ms with 20 multiplies a block and the words formed before
// the steps, 3.87 with 15, 3.50 side by side.
template <int PAIRS, int ORDER, class Land>
__device__ __forceinline__ void run_path_pairs(const McDev& P, const StepCoef<float>* tab, float beta_m1,
                                               PathPairs<PAIRS>& st, int i_land, Land&& at_land) {
  struct Words {
    uint4 a, b;
  };
  auto words = [&](int k, int m) {
    const uint64_t sk = path_step_key(P.rk, (uint32_t)m);
    return Words{path_block(P.rk, st.key[2 * k], sk), path_block(P.rk, st.key[2 * k + 1], sk)};
  };
  auto first = [&](int k, const Words& w, const StepCoef<float>& s) {
    path_step2<ORDER>(s, w.a.x, w.a.y, w.b.x, w.b.y, beta_m1, st.lnF[k], st.lnA[k], st.low[2 * k], st.low[2 * k + 1]);
  };
  auto second = [&](int k, const Words& w, const StepCoef<float>& s) {
    path_step2<ORDER>(s, w.a.z, w.a.w, w.b.z, w.b.w, beta_m1, st.lnF[k], st.lnA[k], st.low[2 * k], st.low[2 * k + 1]);
  };
  int m = 0;
  Words w0 = words(0, 0);  // pair 0's words of block m
  while (i_land >= 0) {
    // blocks whose second step is at or before the landing
    const int mf = (i_land + 1) >> 1;
    for (; m < mf; ++m) {
      const StepCoef<float> s0 = tab[2 * m], s1 = tab[2 * m + 1];
      if constexpr (PAIRS == 2) {
        const Words w1 = words(1, m);
        first(0, w0, s0);
        second(0, w0, s1);
        w0 = words(0, m + 1);
        first(1, w1, s0);
        second(1, w1, s1);
      } else {
        const Words wn = words(0, m + 1);
        first(0, w0, s0);
        second(0, w0, s1);
        w0 = wn;
      }
    }
    if (i_land & 1) {
      i_land = at_land();
      continue;
    }
    // a landing between the two steps of block m
    Words w1 = w0;
    if constexpr (PAIRS == 2) w1 = words(1, m);
    const StepCoef<float> s0 = tab[2 * m];
    first(0, w0, s0);
    if constexpr (PAIRS == 2) first(1, w1, s0);
    i_land = at_land();
    if (2 * m + 1 < P.n_steps) {
      const StepCoef<float> s1 = tab[2 * m + 1];
      second(0, w0, s1);
      if constexpr (PAIRS == 2) second(1, w1, s1);
      if (i_land == 2 * m + 1) i_land = at_land();
    }
    ++m;
    w0 = words(0, m);
  }
}

// One option in shared memory, FP32: payoff (sgn F + c)^+ with sgn = 1,
// c = -K for a call and sgn = -1, c = K for a put: both (8 bytes), or c alone,
// whose sign bit (set for a call, at K = 0 too) gives sgn for one more instruction
// an option and maturity.
struct McOption {
  float sgn, c;
};
struct McSignedStrike {
  float c;
};
__device__ __forceinline__ void set_option(McOption& o, float K, bool call) {
  o = call ? McOption{1.0f, -K} : McOption{-1.0f, K};
}
__device__ __forceinline__ void set_option(McSignedStrike& o, float K, bool call) { o.c = call ? -K : K; }
__device__ __forceinline__ float forward_sign(const McOption& o) { return o.sgn; }
__device__ __forceinline__ float forward_sign(const McSignedStrike& o) {
  return __uint_as_float(0xBF800000u ^ (__float_as_uint(o.c) & 0x80000000u));
}

// The FP32 path loop: four paths per virtual thread as two pairs
// (path_step2); the same path numbering, Philox counters, landing steps and
// payoff accumulation as simulate_paths_scalar.
//  PAIRS = 2: a thread runs its virtual thread's four paths.
//  PAIRS = 1: two threads, t and t + kMcBlock of a block of 2 kMcBlock, run
// one pair each (launches too small to give every scheduler several warps;
// twice the warps, half the work of each).  At a maturity the two warps of a
// virtual warp exchange their forwards through fx[2][4][kMcBlock] and one of
// them, by the maturity's parity, adds the payoffs of all four paths -- the
// same FP32 sums in the same order as PAIRS = 2, so the prices are equal bit
// for bit.
template <int PAIRS, class Option>
__device__ __forceinline__ void simulate_paths_f32(const McDev& P, const double* p, const StepCoef<float>* tab,
                                                   const int* land, const int* s_q0, const int* s_nq,
                                                   const int* s_slot, const Option* opt, int64_t path0,
                                                   int64_t pstride, double* wacc, float* fx) {
  const int lane = threadIdx.x & 31;
  const int vt = threadIdx.x & (kMcBlock - 1), half = PAIRS == 1 ? threadIdx.x / kMcBlock : 0;
  const float beta_m1 = (float)(p[1] - 1.0);
  const float lnf = (float)PathUnits<float>::logu(P.fwd), lna = (float)PathUnits<float>::logu(p[0]);
  const float log_abs = (float)(P.log_absorb * PathUnits<float>::kLogUnit);
  const int64_t n_paths = P.n_paths;
  const int64_t warp_path0 = path0 - lane;
  int buf = 0;
  // one round: NP pairs of this thread's virtual thread
  auto round = [&](auto np, int64_t wp) {
    constexpr int NP = decltype(np)::value, N = 2 * NP, NF = PAIRS == 1 ? 4 : N;
    PathPairs<NP> st;
    st.start(P, lnf, lna, wp + 2 * half * pstride + lane, pstride);
    int m = 0;
    auto pay_out = [&]() {
      float F[NF];
      bool mine = true;
#pragma unroll
      for (int k = 0; k < N; ++k) F[k] = st.forward(k, log_abs);
      if constexpr (PAIRS == 1) {
        float* x = fx + buf * (4 * kMcBlock) + vt;
        x[(2 * half) * kMcBlock] = F[0];
        x[(2 * half + 1) * kMcBlock] = F[1];
        asm volatile("bar.sync %0, 64;" ::"r"(1 + vt / 32) : "memory");
        mine = (m & 1) == half;
        if (mine) {
#pragma unroll
          for (int k = 0; k < 4; ++k) F[k] = x[k * kMcBlock];
        }
        // the next maturity writes the other buffer, and the one after it is
        // written only past a barrier that follows this read
        buf ^= 1;
      }
      if (mine) {
        const int q0 = s_q0[m], nq = s_nq[m], slot0 = s_slot[m];
        // a path beyond n_paths pays 0 (the last round of the grid only)
        bool live[NF];
#pragma unroll
        for (int k = 0; k < NF; ++k) live[k] = wp + k * pstride + lane < n_paths;
        for (int c0 = 0; c0 < 2 * nq; c0 += 32) {
          float v[32];
#pragma unroll
          for (int kk = 0; kk < 32; kk += 2) {
            const int j = (c0 + kk) >> 1;
            float pay = 0.0f, pay2 = 0.0f;
            if (j < nq) {
              const Option o = opt[q0 + j];
              const float sgn = forward_sign(o);
#pragma unroll
              for (int k = 0; k < NF; ++k) {
                const float x = fmaxf(fmaf(sgn, F[k], o.c), 0.0f);
                const float y = live[k] ? x : 0.0f;
                pay += y;
                pay2 = fmaf(y, y, pay2);
              }
            }
            v[kk] = pay;
            v[kk + 1] = pay2;
          }
          const float tot = warp_reduce_scatter32<float>(v, lane);
          wacc[(slot0 + (c0 >> 5)) * 32 + lane] += (double)tot;
        }
      }
      ++m;
      return m < P.n_mats ? land[m] : -1;
    };
    run_path_pairs<NP, kOrderEuropean>(P, tab, beta_m1, st, land[0], pay_out);
  };
  for (int64_t wp = warp_path0; wp < n_paths; wp += 4 * pstride) {
    // the second pair of the grid's last round may lie wholly beyond n_paths
    // (its payoffs are zeros, which change no sum)
    if (PAIRS == 2 && wp + 2 * pstride < n_paths) {
      round(IntTag<2>{}, wp);
    } else {
      round(IntTag<1>{}, wp);
    }
  }
}

}  // namespace sabr
