// mc.cu -- sabr_mc_price: fused path simulation + deterministic reduction.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <vector>

#include "common.h"
#include "mc.cuh"
#include "mc_bessel.cuh"
#include "mc_host.h"

namespace sabr {

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------
struct McSmem {
  size_t tab, land, q0, nq, slot, K, call, wacc, fx, total;
};

// opt_bytes: an FP32 log-Euler option takes 8 or 4 (McOption, McSignedStrike; no
// call flag is read); others the strike in the working precision.  split: the
// block of 2 kMcBlock threads also needs the exchange buffer of
// simulate_paths_f32<1>.
template <class R>
__host__ __device__ inline McSmem mc_smem_layout(int n_steps, int n_quotes, int n_mats, int n_slots, int opt_bytes, bool split) {
  // (the conditional-Bessel form leaves its step table in global memory and
  // passes n_steps = 0)
  McSmem L;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    size_t r = (o + 15) & ~(size_t)15;
    o = r + bytes;
    return r;
  };
  L.wacc = take(sizeof(double) * kMcWarps * n_slots * 32);
  L.tab = take(sizeof(StepCoef<R>) * n_steps);
  L.K = take((size_t)opt_bytes * n_quotes);
  L.land = take(sizeof(int) * n_mats);
  L.q0 = take(sizeof(int) * n_mats);
  L.nq = take(sizeof(int) * n_mats);
  L.slot = take(sizeof(int) * n_mats);
  L.call = take(n_quotes);
  L.fx = take(split ? sizeof(float) * 2 * 4 * kMcBlock : 0);
  L.total = (o + 15) & ~(size_t)15;
  return L;
}
// grid = (blocks_per_set, n_sets).  Set s prices with set_params[s][0..9];
// sets whose set_valid flag is 0 are skipped.  Writes, per block, the FP64
// sums of payoff and payoff^2 of every option to
// partial[(s * blocks_per_set + block) * n_slots * 32 + value].
// block0 / grid_total (path sharding): this launch runs blocks block0 ..
// block0 + gridDim.x - 1 of a grid of grid_total blocks -- each block takes
// the paths it would take in that grid -- and writes their partials at
// positions 0 .. gridDim.x - 1; grid_total = 0 means the launch is the
// whole grid.  SCHEME: SABR_MC_LOG_EULER (eq. (dis_SABRd)) or
// SABR_MC_BESSEL (the conditional-Bessel step of mc_bessel.cuh).  SPLIT
// (FP32 log-Euler): blocks of 2 kMcBlock threads, a pair of paths each.
// Resident blocks of kMcBlock threads per SM that the grids count on (and the
// kernels' register budgets are set for).
__host__ __device__ constexpr int mc_resident_blocks(int prec, int scheme) {
  return prec == SABR_FP64 ? 3 : (scheme == SABR_MC_BESSEL ? 5 : 4);
}
template <class R, int SCHEME, bool SPLIT, class Option>
__global__ void __launch_bounds__((SPLIT ? 2 * kMcBlock : kMcBlock),
                                  (SPLIT ? 1 : mc_resident_blocks(sizeof(R) == 8 ? SABR_FP64 : SABR_FP32, SCHEME)))
    mc_paths_kernel(McDev P, const double* __restrict__ set_params, const int* __restrict__ set_valid,
                    double* __restrict__ partial, int block0, int grid_total) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int set = blockIdx.y;
  if (set_valid && !set_valid[set]) return;
  constexpr bool kPairs = sizeof(R) == 4 && SCHEME == SABR_MC_LOG_EULER;
  const McSmem L =
      mc_smem_layout<R>(SCHEME == SABR_MC_BESSEL ? 0 : P.n_steps, P.n_quotes, P.n_mats, P.n_slots, sizeof(Option), SPLIT);
  double* wacc = (double*)(smem + L.wacc);
  StepCoef<R>* tab = (StepCoef<R>*)(smem + L.tab);
  R* sK = (R*)(smem + L.K);
  Option* sopt = (Option*)(smem + L.K);
  int* land = (int*)(smem + L.land);
  int* s_q0 = (int*)(smem + L.q0);
  int* s_nq = (int*)(smem + L.nq);
  int* s_slot = (int*)(smem + L.slot);
  int8_t* scall = (int8_t*)(smem + L.call);
  double p[kMaxD];
#pragma unroll
  for (int i = 0; i < kMaxD; ++i) p[i] = set_params[(size_t)set * kMaxD + i];
  const int nv = P.n_slots * 32;
  for (int i = threadIdx.x; i < kMcWarps * nv; i += blockDim.x) wacc[i] = 0.0;
  if constexpr (SCHEME == SABR_MC_BESSEL) {
    for (int i = threadIdx.x; i < P.n_steps; i += blockDim.x) {
      const int m = P.step_mat[i];
      if (m >= 0) land[m] = i;
    }
  } else {
    build_steps<R>(P, p, set, tab, land);
  }
  for (int q = threadIdx.x; q < P.n_quotes; q += blockDim.x) {
    if constexpr (kPairs) {
      set_option(sopt[q], (float)P.K[q], P.is_call[q] != 0);
    } else {
      sK[q] = (R)P.K[q];
      scall[q] = P.is_call[q];
    }
  }
  for (int m = threadIdx.x; m < P.n_mats; m += blockDim.x) {
    s_q0[m] = P.mat_q0[m];
    s_nq[m] = P.mat_nq[m];
    s_slot[m] = P.mat_slot[m];
  }
  __syncthreads();
  const int vt = threadIdx.x & (kMcBlock - 1);  // virtual thread of the block
  const int64_t gblocks = grid_total > 0 ? grid_total : gridDim.x;
  const int64_t path0 = (int64_t)(block0 + blockIdx.x) * kMcBlock + vt, pstride = gblocks * kMcBlock;
  double* my_acc = wacc + (size_t)(vt >> 5) * nv;
  if constexpr (SCHEME == SABR_MC_BESSEL) {
    const BesselStep<R>* tb = (const BesselStep<R>*)P.tab;
    if (p[1] == 1.0) {
      simulate_paths_bessel<R, true>(P, p, tb, land, s_q0, s_nq, s_slot, sK, scall, path0, pstride, my_acc);
    } else {
      simulate_paths_bessel<R, false>(P, p, tb, land, s_q0, s_nq, s_slot, sK, scall, path0, pstride, my_acc);
    }
  } else if constexpr (kPairs) {
    simulate_paths_f32<SPLIT ? 1 : 2>(P, p, tab, land, s_q0, s_nq, s_slot, sopt, path0, pstride, my_acc,
                                      (float*)(smem + L.fx));
  } else {
    simulate_paths_scalar<R>(P, p, tab, land, s_q0, s_nq, s_slot, sK, scall, path0, pstride, my_acc);
  }
  __syncthreads();
  double* out = partial + ((size_t)set * gridDim.x + blockIdx.x) * nv;
  for (int v = threadIdx.x; v < nv; v += blockDim.x) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kMcWarps; ++w) s += wacc[(size_t)w * nv + v];
    out[v] = s;
  }
}

// The step tables of n_sets parameter sets (blockIdx.y), one thread per step:
// StepCoef entries of a dynamic model, or BesselStep entries.
template <class R, int SCHEME>
__global__ void __launch_bounds__(64) mc_steps_kernel(McDev P, const double* __restrict__ set_params,
                                                     const int* __restrict__ set_valid, void* __restrict__ out) {
  const int set = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P.n_steps || (set_valid && !set_valid[set])) return;
  double p[kMaxD];
#pragma unroll
  for (int k = 0; k < kMaxD; ++k) p[k] = set_params[(size_t)set * kMaxD + k];
  const size_t at = (size_t)set * P.n_steps + i;
  if constexpr (SCHEME == SABR_MC_BESSEL) {
    ((BesselStep<R>*)out)[at] = bessel_step_entry<R>(P, p, i);
  } else {
    ((StepCoef<R>*)out)[at] = dynamic_step_coef<R>(P, p, i);
  }
}

// L lanes per (set, option), L a power of two: lane l sums blocks l, l + L,
// ... and a fixed butterfly sums the lanes, eq. (payoff).  One lane over the
// 608 blocks of a whole-GPU launch is a chain of 608 dependent loads and FP64
// additions, which took longer than the paths of a small pricing.
__global__ void mc_reduce_kernel(McDev P, int n_sets, int blocks_per_set, int L, const double* __restrict__ partial,
                                 const int* __restrict__ q_value, const int* __restrict__ q_out,
                                 const double* __restrict__ disc, const int* __restrict__ set_valid,
                                 double* __restrict__ price, double* __restrict__ se, int out_stride) {
  const int64_t idx = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / L;
  const int lane = threadIdx.x & (L - 1);
  // (blockDim is a multiple of L: the lanes of an option leave together)
  if (idx >= (int64_t)n_sets * P.n_quotes) return;
  const int set = (int)(idx / P.n_quotes), q = (int)(idx % P.n_quotes);
  if (set_valid && !set_valid[set]) return;
  const int nv = P.n_slots * 32;
  const int v = q_value[q];
  double s = 0.0, s2 = 0.0;
#pragma unroll 4
  for (int b = lane; b < blocks_per_set; b += L) {
    const double* part = partial + ((size_t)set * blocks_per_set + b) * nv + v;
    s += part[0];
    s2 += part[1];
  }
  const unsigned mask = L == 32 ? 0xffffffffu : (((1u << L) - 1u) << ((threadIdx.x & 31) & ~(L - 1)));
  for (int off = L >> 1; off > 0; off >>= 1) {
    s += __shfl_xor_sync(mask, s, off);
    s2 += __shfl_xor_sync(mask, s2, off);
  }
  if (lane != 0) return;
  const double N = (double)P.n_paths;
  const double mean = s / N;
  double var = (s2 - s * mean) / (N - 1.0);
  if (var < 0.0) var = 0.0;
  const double D = disc[q];
  price[(size_t)set * out_stride + q_out[q]] = D * mean;
  if (se) se[(size_t)set * out_stride + q_out[q]] = D * sqrt(var / N);
}
// Lanes per option: about eight blocks a lane (a function of the grid alone,
// so a path-sharded reduction runs in the order of the unsharded one).
static int mc_reduce_lanes(int blocks_per_set) {
  int L = 1;
  while (L < 32 && 8 * L < blocks_per_set) L <<= 1;
  return L;
}
static void launch_reduce(const McDev& d, int n_sets, int blocks_per_set, const double* partial, const int* q_value,
                          const int* q_out, const double* disc, const int* set_valid, double* price, double* se,
                          int out_stride, cudaStream_t s) {
  const int L = mc_reduce_lanes(blocks_per_set);
  const int64_t threads = (int64_t)n_sets * d.n_quotes * L;
  mc_reduce_kernel<<<(unsigned)((threads + 127) / 128), 128, 0, s>>>(d, n_sets, blocks_per_set, L, partial, q_value,
                                                                     q_out, disc, set_valid, price, se, out_stride);
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
sabr_status mc_prepare(int model, double fwd, const double* T, const double* K, const int8_t* is_call,
                       const double* discount, int64_t n, int64_t n_paths, double spy, uint64_t seed,
                       int prec, McHost& h) {
  if (n_params(model) < 0) return fail(SABR_EINVAL, "unknown model");
  if (prec != SABR_FP32 && prec != SABR_FP64) return fail(SABR_EINVAL, "unknown precision");
  if (!(fwd > 0.0) || !std::isfinite(fwd)) return fail(SABR_EINVAL, "fwd must be > 0");
  if (n < 1 || n > kMaxMcQuotes) return fail(SABR_EINVAL, "number of options must lie in [1, 512]");
  if (!T || !K) return fail(SABR_EINVAL, "NULL option array");
  if (n_paths < 2 || n_paths > ((int64_t)1 << 31)) return fail(SABR_EINVAL, "n_paths must lie in [2, 2^31]");
  if (!(spy > 0.0) || !std::isfinite(spy)) return fail(SABR_EINVAL, "steps_per_year must be > 0");
  std::vector<int> order(n);
  for (int i = 0; i < n; ++i) {
    if (!(T[i] > 0.0) || !std::isfinite(T[i])) return fail(SABR_EINVAL, "maturities must be > 0");
    if (!(K[i] >= 0.0) || !std::isfinite(K[i])) return fail(SABR_EINVAL, "strikes must be >= 0");
    if (discount && !std::isfinite(discount[i])) return fail(SABR_EINVAL, "non-finite discount");
    order[i] = i;
  }
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return T[a] < T[b]; });
  h.model = model;
  h.prec = prec;
  h.fwd = fwd;
  h.n_paths = n_paths;
  h.seed = seed;
  h.n_quotes = (int)n;
  h.K.resize(n);
  h.call.resize(n);
  h.disc.resize(n);
  h.q_out.resize(n);
  h.q_value.resize(n);
  h.mats.clear();
  h.mat_q0.clear();
  h.mat_nq.clear();
  h.mat_slot.clear();
  int slots = 0;
  for (int s = 0; s < n; ++s) {
    const int i = order[s];
    if (h.mats.empty() || T[i] != h.mats.back()) {
      if (!h.mats.empty()) slots += (2 * h.mat_nq.back() + 31) / 32;
      h.mats.push_back(T[i]);
      h.mat_q0.push_back(s);
      h.mat_nq.push_back(0);
      h.mat_slot.push_back(slots);
    }
    const int pos = h.mat_nq.back()++;
    h.K[s] = K[i];
    h.call[s] = is_call ? (is_call[i] != 0) : 1;
    h.disc[s] = discount ? discount[i] : 1.0;
    h.q_out[s] = i;
    h.q_value[s] = h.mat_slot.back() * 32 + 2 * pos;
  }
  slots += (2 * h.mat_nq.back() + 31) / 32;
  h.n_slots = slots;
  if ((int)h.mats.size() > kMaxMats) return fail(SABR_EINVAL, "more than 64 distinct maturities");
  // grid: multiples of 1/spy below the last maturity with every maturity
  // inserted; a multiple within 1e-10 of a maturity is that maturity.
  h.step_t.clear();
  h.step_h.clear();
  h.step_mat.clear();
  double prev = 0.0;
  int64_t k = 1;
  for (size_t m = 0; m < h.mats.size(); ++m) {
    const double Tm = h.mats[m];
    while ((double)k / spy < Tm - 1e-10) {
      const double t = (double)k / spy;
      h.step_t.push_back(t);
      h.step_h.push_back(t - prev);
      h.step_mat.push_back(-1);
      prev = t;
      ++k;
      if ((int64_t)h.step_t.size() > kMaxMcSteps) return fail(SABR_EINVAL, "more than 8192 time steps");
    }
    h.step_t.push_back(Tm);
    h.step_h.push_back(Tm - prev);
    h.step_mat.push_back((int)m);
    prev = Tm;
    if (std::fabs((double)k / spy - Tm) <= 1e-10) ++k;
  }
  h.n_steps = (int)h.step_t.size();
  if (h.n_steps > kMaxMcSteps) return fail(SABR_EINVAL, "more than 8192 time steps");
  h.Tmax = h.mats.back();
  // what a block of the log-Euler kernel takes at its least (the
  // conditional-Bessel kernel keeps its step table in global memory; the same
  // limit holds for it)
  const int M = (int)h.mats.size();
  const size_t smem = prec == SABR_FP64
                          ? mc_smem_layout<double>(h.n_steps, h.n_quotes, M, h.n_slots, 8, false).total
                          : mc_smem_layout<float>(h.n_steps, h.n_quotes, M, h.n_slots, 4, false).total;
  if (smem > 220 * 1024) return fail(SABR_EINVAL, "too many time steps and options for one launch");
  h.smem = smem;
  return SABR_OK;
}

// Device image of an McHost: sizes and offsets in one buffer.
size_t mc_image_bytes(const McHost& h) {
  const size_t Q = h.n_quotes, M = h.mats.size(), S = h.n_steps;
  return 16 * 12 + 8 * (2 * S + 2 * Q) + 4 * (S + 3 * M + 2 * Q) + Q + 256;
}

void mc_fill_image(const McHost& h, unsigned char* host_img, unsigned char* dev_base, McDev& d, int** q_value,
                   int** q_out, double** disc) {
  size_t o = 0;
  auto put = [&](const void* src, size_t bytes) {
    o = (o + 15) & ~(size_t)15;
    std::memcpy(host_img + o, src, bytes);
    unsigned char* p = dev_base + o;
    o += bytes;
    return p;
  };
  d.model = h.model;
  d.n_quotes = h.n_quotes;
  d.n_mats = (int)h.mats.size();
  d.n_steps = h.n_steps;
  d.n_slots = h.n_slots;
  d.n_paths = h.n_paths;
  d.fwd = h.fwd;
  d.log_absorb = std::log(1e-12 * h.fwd);
  d.key0 = (uint32_t)h.seed;
  d.key1 = (uint32_t)(h.seed >> 32);
  for (int r = 0; r < 10; ++r) {  // Philox round keys (key schedule of Salmon et al.)
    d.rk.k0[r] = d.key0 + (uint32_t)r * 0x9E3779B9u;
    d.rk.k1[r] = d.key1 + (uint32_t)r * 0xBB67AE85u;
  }
  d.tab = nullptr;
  if (h.model == SABR_DYN_I || h.model == SABR_DYN_II) {
    d.step_t = (const double*)put(h.step_t.data(), 8 * h.step_t.size());
  } else {
    std::vector<double> sh(h.step_h.size());
    for (size_t i = 0; i < sh.size(); ++i) sh[i] = std::sqrt(h.step_h[i]);
    d.step_t = (const double*)put(sh.data(), 8 * sh.size());
  }
  d.step_h = (const double*)put(h.step_h.data(), 8 * h.step_h.size());
  d.step_mat = (const int*)put(h.step_mat.data(), 4 * h.step_mat.size());
  d.mat_q0 = (const int*)put(h.mat_q0.data(), 4 * h.mat_q0.size());
  d.mat_nq = (const int*)put(h.mat_nq.data(), 4 * h.mat_nq.size());
  d.mat_slot = (const int*)put(h.mat_slot.data(), 4 * h.mat_slot.size());
  d.K = (const double*)put(h.K.data(), 8 * h.K.size());
  d.is_call = (const int8_t*)put(h.call.data(), h.call.size());
  *q_value = (int*)put(h.q_value.data(), 4 * h.q_value.size());
  *q_out = (int*)put(h.q_out.data(), 4 * h.q_out.size());
  *disc = (double*)put(h.disc.data(), 8 * h.disc.size());
}

// Bytes of the step tables of n_sets sets: 0 where the blocks build their own
// (static log-Euler models, whose entries cost less than a launch).
size_t mc_step_table_bytes(const McHost& h, int n_sets) {
  const size_t rs = h.prec == SABR_FP64 ? 8 : 4;
  if (h.scheme == SABR_MC_BESSEL) return 12 * rs * (size_t)h.n_steps * n_sets;
  if (h.model != SABR_DYN_I && h.model != SABR_DYN_II) return 0;
  return 4 * rs * (size_t)h.n_steps * n_sets;
}
static_assert(sizeof(BesselStep<float>) == 48 && sizeof(BesselStep<double>) == 96, "step table entry");

using McPathsFn = void (*)(McDev, const double*, const int*, double*, int, int);

// Resident blocks of kMcBlock threads per SM that grids count on, by the
// registers and by a block's shared memory.
static int mc_blocks_per_sm(int prec, int scheme, size_t smem) {
  const size_t per_block = ((smem + 127) & ~(size_t)127) + 1024;
  return (int)std::min<size_t>(mc_resident_blocks(prec, scheme), std::max<size_t>(1, (228 * 1024) / per_block));
}

// The path kernel of a problem's precision and scheme (split: the FP32
// log-Euler form with a pair of paths a thread), with its dynamic shared
// memory allowance raised to what the problem needs.  FP32 log-Euler options
// take 8 bytes where that leaves as many blocks an SM as 4 (2^22 paths x 504
// steps, 120 options: 3.499 ms, with 4 bytes 3.512), else 4 (512 options x 1200
// steps, 600 000 paths: 1.34 ms on three blocks an SM, 1.37 where the grid counts
// four and three fit).
static McPathsFn mc_paths_fn(const McHost& h, bool split, size_t* smem) {
  const int M = (int)h.mats.size();
  if (h.prec == SABR_FP64) {
    const bool bessel = h.scheme == SABR_MC_BESSEL;
    const McPathsFn fn = bessel ? mc_paths_kernel<double, SABR_MC_BESSEL, false, double>
                                : mc_paths_kernel<double, SABR_MC_LOG_EULER, false, double>;
    *smem = mc_smem_layout<double>(bessel ? 0 : h.n_steps, h.n_quotes, M, h.n_slots, 8, false).total;
    allow_smem((const void*)fn, *smem);
    return fn;
  }
  if (h.scheme == SABR_MC_BESSEL) {
    const McPathsFn fn = mc_paths_kernel<float, SABR_MC_BESSEL, false, float>;
    *smem = mc_smem_layout<float>(0, h.n_quotes, M, h.n_slots, 4, false).total;
    allow_smem((const void*)fn, *smem);
    return fn;
  }
  McPathsFn fn = mc_paths_kernel<float, SABR_MC_LOG_EULER, true, McOption>;
  *smem = mc_smem_layout<float>(h.n_steps, h.n_quotes, M, h.n_slots, 8, split).total;
  if (!split) {
    fn = mc_paths_kernel<float, SABR_MC_LOG_EULER, false, McOption>;
    if (mc_blocks_per_sm(h.prec, h.scheme, *smem) < mc_blocks_per_sm(h.prec, h.scheme, h.smem)) {
      fn = mc_paths_kernel<float, SABR_MC_LOG_EULER, false, McSignedStrike>;
      *smem = h.smem;
    }
  }
  allow_smem((const void*)fn, *smem);
  return fn;
}

// Paths one thread takes at a time.
static int mc_thread_paths(const McHost& h) {
  return h.scheme == SABR_MC_BESSEL ? kBesselPathsPerThread : mc_paths_per_thread(h.prec);
}

// Blocks per SM that the grid of a pricing counts on.  The grid decides which
// paths share a thread and a warp, hence the order of the FP32 payoff sums,
// so it is a rule on the precision, the scheme and the table bytes and not
// what a build's register count happens to allow.
static int mc_grid_blocks_per_sm(const McHost& h) { return mc_blocks_per_sm(h.prec, h.scheme, h.smem); }

// Blocks per parameter set.  Every block of a launch does the same work
// (n_paths / blocks-per-set paths), so with R resident blocks a launch of
// n_sets x p blocks takes ceil(n_sets p / R) rounds of a block's time, which
// is proportional to 1/p: p minimises ceil(n_sets p / R) / p over p up to
// what the paths need (each thread takes kMcPathsPerThread paths at a time)
// and up to 8 rounds.  One set: p = R, one round, grid-stride.  256 sets on
// 760 resident blocks: p = 8 (3 rounds, 0.375) instead of p = 2 (one round
// with a third of the GPU idle, 0.5).
int mc_blocks_per_set(const McHost& h, int n_sets) {
  const int64_t resident = device_sms() * (int64_t)mc_grid_blocks_per_sm(h);
  const int64_t sets = std::max(1, n_sets);
  const int64_t per_block = (int64_t)kMcBlock * mc_thread_paths(h);
  const int64_t by_paths = (h.n_paths + per_block - 1) / per_block;
  const int64_t p_max = std::max<int64_t>(1, std::min(by_paths, 8 * resident / sets));
  int64_t best = 1;
  double best_cost = 1e300;
  for (int64_t p = 1; p <= p_max; ++p) {
    const double cost = (double)((sets * p + resident - 1) / resident) / (double)p;
    if (cost < best_cost * (1.0 - 1e-12)) {
      best_cost = cost;
      best = p;
    }
  }
  return (int)best;
}

// A launch of at most one block of kMcBlock threads per SM and of many steps runs
// the FP32 log-Euler form with a pair of paths a thread: two warps a scheduler
// instead of one (504 steps, us a call in a row, one pair a thread | two: 2^15
// paths 104.7 | 113.9, 2^16 105.3 | 115.2; from two blocks an SM on two pairs are
// the faster form, 2^17 171 | 160, 2^18 308 | 292).  Its larger blocks and the
// exchange at the maturities cost 1 to 2 us a launch, which the steps earn from
// about 100 on (a Technique II calibration of 30 waves, us: 3 steps 1266 | 1202,
// 50 2592 | 2592, 63 2799 | 2736, 100 4156 | 4158, 125 4600 | 4597, 250 8113 | 8175).
constexpr int kSplitSteps = 128;
static bool mc_split(const McHost& h, int64_t blocks) {
  return h.prec == SABR_FP32 && h.scheme == SABR_MC_LOG_EULER && h.n_steps >= kSplitSteps &&
         blocks <= (int64_t)device_sms();
}

// Whether the blocks of a dynamic model's launch build their step tables
// themselves: forming one entry is about 80 FP64 instructions, so a table costs
// an SM about 15 ns an entry for every block on it, and the launch that forms it
// once costs 4 to 5 us between two kernels.  The line is at 300 entries an SM
// and two entries a thread (us a call in a row, built by the blocks | by a launch;
// pricer 70 000 paths x 250 steps, 1 block an SM 67.6 | 70.4; 150 000 x 100, 2
// blocks 64.2 | 68.3; x 250 100.3 | 96.6; 300 000 x 50, 4 blocks 66.7 | 68.8; x
// 100 92.5 | 91.5; cliquet, blocks of 64: 20 000 x 100, 1 block 49.0 | 52.5; x 250
// 67.3 | 65.0; 150 000 x 50, 4 blocks 48.4 | 52.5; 300 000 x 50, 8 blocks 65.0 |
// 63.9).
bool mc_blocks_build_steps(const McHost& h, int64_t blocks, int block_threads) {
  if (h.scheme == SABR_MC_BESSEL) return false;
  if (h.model != SABR_DYN_I && h.model != SABR_DYN_II) return true;
  const int64_t sms = device_sms(), per_sm = (blocks + sms - 1) / sms;
  return per_sm * h.n_steps <= 300 && h.n_steps <= 2 * block_threads;
}

// Fills d.tab for n_sets sets.
void mc_launch_steps(const McHost& h, const McDev& d, const double* set_params, const int* set_valid, int n_sets,
                     cudaStream_t s) {
  const dim3 grid((h.n_steps + 63) / 64, n_sets);
  void* tab = const_cast<void*>(d.tab);
  if (h.scheme == SABR_MC_BESSEL) {
    if (h.prec == SABR_FP64)
      mc_steps_kernel<double, SABR_MC_BESSEL><<<grid, 64, 0, s>>>(d, set_params, set_valid, tab);
    else
      mc_steps_kernel<float, SABR_MC_BESSEL><<<grid, 64, 0, s>>>(d, set_params, set_valid, tab);
  } else if (h.prec == SABR_FP64) {
    mc_steps_kernel<double, SABR_MC_LOG_EULER><<<grid, 64, 0, s>>>(d, set_params, set_valid, tab);
  } else {
    mc_steps_kernel<float, SABR_MC_LOG_EULER><<<grid, 64, 0, s>>>(d, set_params, set_valid, tab);
  }
}

static void launch_paths(const McHost& h, const McDev& d, const double* set_params, const int* set_valid,
                         dim3 grid, double* partial, int block0, int grid_total, cudaStream_t s) {
  const int64_t blocks = (int64_t)grid.x * grid.y;
  const bool split = mc_split(h, blocks);
  const int threads = split ? 2 * kMcBlock : kMcBlock;
  McDev k = d;
  if (mc_blocks_build_steps(h, blocks, kMcBlock)) k.tab = nullptr;
  if (k.tab != nullptr) mc_launch_steps(h, k, set_params, set_valid, (int)grid.y, s);
  size_t smem = 0;
  const McPathsFn fn = mc_paths_fn(h, split, &smem);
  fn<<<grid, threads, smem, s>>>(k, set_params, set_valid, partial, block0, grid_total);
}

sabr_status mc_launch(const McHost& h, const McDev& d, const double* set_params, const int* set_valid, int n_sets,
                      int blocks_per_set, double* partial, const int* q_value, const int* q_out,
                      const double* disc, double* price, double* se, int out_stride, cudaStream_t s) {
  launch_paths(h, d, set_params, set_valid, dim3(blocks_per_set, n_sets), partial, 0, 0, s);
  launch_reduce(d, n_sets, blocks_per_set, partial, q_value, q_out, disc, set_valid, price, se, out_stride, s);
  SABR_CUDA(cudaGetLastError());
  return SABR_OK;
}

// Library-owned scratch of the pricers: two per device, taken in turn, so that a
// call's tables are laid out and copied while the kernels of the call before it
// run (2^16 paths: the GPU waited about 15 us between calls).  The calls of a
// device are serialised by its lock and by waiting, before a scratch is
// rewritten, for the kernels that last used it; calls on several streams
// therefore never share one in flight.  A scratch grows to what its calls need
// and stays.
struct McWorkspace {
  void* dev = nullptr;
  size_t dev_bytes = 0;
  unsigned char* host = nullptr;
  size_t host_bytes = 0;
  cudaEvent_t done = nullptr;
};
struct McWorkspaces {
  std::mutex mu;
  McWorkspace ws[2];
  int next = 0;
};
// The scratches of a device (map nodes stay where they are).
static McWorkspaces& mc_workspaces(int device) {
  static std::mutex mu;
  static std::map<int, McWorkspaces> all;
  std::lock_guard<std::mutex> lock(mu);
  return all[device];
}

static sabr_status ensure_ws(McWorkspace& w, size_t dev_bytes, size_t host_bytes) {
  if (!w.done) SABR_CUDA(cudaEventCreateWithFlags(&w.done, cudaEventDisableTiming));
  SABR_CUDA(cudaEventSynchronize(w.done));
  if (w.dev_bytes < dev_bytes) {
    if (w.dev) cudaFree(w.dev);
    w.dev = nullptr;
    w.dev_bytes = 0;
    SABR_CUDA(cudaMalloc(&w.dev, dev_bytes));
    w.dev_bytes = dev_bytes;
  }
  if (w.host_bytes < host_bytes) {
    if (w.host) cudaFreeHost(w.host);
    w.host = nullptr;
    w.host_bytes = 0;
    SABR_CUDA(cudaMallocHost(&w.host, host_bytes));
    w.host_bytes = host_bytes;
  }
  return SABR_OK;
}

sabr_status McScratch::acquire(size_t dev_bytes, size_t host_bytes, cudaStream_t s) {
  int d = 0;
  SABR_CUDA(cudaGetDevice(&d));
  McWorkspaces& all = mc_workspaces(d);
  lock_ = std::unique_lock<std::mutex>(all.mu);
  McWorkspace& w = all.ws[all.next];
  all.next ^= 1;
  SABR_TRY(ensure_ws(w, dev_bytes, host_bytes));
  dev = (unsigned char*)w.dev;
  host = w.host;
  done_ = w.done;
  stream_ = s;
  return SABR_OK;
}
// On every way out, errors included: what was enqueued before an error still
// uses the scratch.
McScratch::~McScratch() {
  if (done_ && cudaEventRecord(done_, stream_) != cudaSuccess) cudaStreamSynchronize(stream_);
}

}  // namespace sabr

namespace sabr {

static sabr_status mc_price(sabr_model model, const double* params, double fwd, const double* T, const double* K,
                            const int8_t* is_call, const double* discount, int64_t n, int64_t n_paths,
                            double steps_per_year, uint64_t seed, int scheme, double* price_out, double* stderr_out,
                            sabr_precision prec, void* stream) {
  SABR_TRY(check_params(model, params));
  if (!price_out) return fail(SABR_EINVAL, "price_out is NULL");
  if (scheme != SABR_MC_LOG_EULER && scheme != SABR_MC_BESSEL) return fail(SABR_EINVAL, "unknown path scheme");
  McHost h;
  SABR_TRY(mc_prepare(model, fwd, T, K, is_call, discount, n, n_paths, steps_per_year, seed, prec, h));
  h.scheme = scheme;
  if (model == SABR_DYN_II && !case2_feasible<double, double>(params, h.Tmax))
    return fail(SABR_EINVAL, "parameters violate rho(t) in [-1,1], nu(t) > 0");
  const int bps = mc_blocks_per_set(h, 1);
  const size_t img = mc_image_bytes(h);
  const size_t params_off = (img + 255) & ~(size_t)255;
  const size_t part_off = params_off + 256;
  const size_t tab_off = part_off + sizeof(double) * (size_t)bps * h.n_slots * 32;
  const size_t tab_bytes = mc_step_table_bytes(h, 1);
  const size_t dev_bytes = tab_off + tab_bytes;
  cudaStream_t s = (cudaStream_t)stream;
  McScratch w;
  SABR_TRY(w.acquire(dev_bytes, part_off, s));
  McDev d;
  int* q_value;
  int* q_out;
  double* disc;
  unsigned char* base = w.dev;
  mc_fill_image(h, w.host, base, d, &q_value, &q_out, &disc);
  if (tab_bytes) d.tab = base + tab_off;
  double p10[kMaxD];
  for (int i = 0; i < kMaxD; ++i) p10[i] = i < n_params(model) ? params[i] : 0.0;
  std::memcpy(w.host + params_off, p10, sizeof(p10));
  SABR_CUDA(cudaMemcpyAsync(w.dev, w.host, part_off, cudaMemcpyHostToDevice, s));
  return mc_launch(h, d, (const double*)(base + params_off), nullptr, 1, bps, (double*)(base + part_off), q_value,
                   q_out, disc, price_out, stderr_out, (int)n, s);
}

}  // namespace sabr

extern "C" sabr_status sabr_mc_price(sabr_model model, const double* params, double fwd, const double* T,
                                     const double* K, const int8_t* is_call, const double* discount, int64_t n,
                                     int64_t n_paths, double steps_per_year, uint64_t seed, double* price_out,
                                     double* stderr_out, sabr_precision prec, void* stream) {
  sabr::clear_error();
  return sabr::mc_price(model, params, fwd, T, K, is_call, discount, n, n_paths, steps_per_year, seed,
                        SABR_MC_LOG_EULER, price_out, stderr_out, prec, stream);
}

extern "C" sabr_status sabr_mc_price_scheme(sabr_model model, const double* params, double fwd, const double* T,
                                            const double* K, const int8_t* is_call, const double* discount,
                                            int64_t n, int64_t n_paths, double steps_per_year, uint64_t seed,
                                            sabr_mc_scheme scheme, double* price_out, double* stderr_out,
                                            sabr_precision prec, void* stream) {
  sabr::clear_error();
  return sabr::mc_price(model, params, fwd, T, K, is_call, discount, n, n_paths, steps_per_year, seed, (int)scheme,
                        price_out, stderr_out, prec, stream);
}

// ---------------------------------------------------------------------------
// Path sharding (the multi-GPU form of the Sec. 4 pricer): the grid of
// sabr_mc_price split into block ranges, one per device; the per-block FP64
// partial sums, gathered in block order, reduce to the unsharded prices bit
// for bit.
// ---------------------------------------------------------------------------
namespace sabr {

struct McShardCall {
  McHost h;
  int total_blocks = 0;
};

static sabr_status mc_shard_prepare(sabr_model model, const double* params, double fwd, const double* T,
                                    const double* K, const int8_t* is_call, const double* discount, int64_t n,
                                    int64_t n_paths, double spy, uint64_t seed, sabr_precision prec, McShardCall& c) {
  SABR_TRY(check_params(model, params));
  SABR_TRY(mc_prepare(model, fwd, T, K, is_call, discount, n, n_paths, spy, seed, prec, c.h));
  if (model == SABR_DYN_II && !case2_feasible<double, double>(params, c.h.Tmax))
    return fail(SABR_EINVAL, "parameters violate rho(t) in [-1,1], nu(t) > 0");
  c.total_blocks = mc_blocks_per_set(c.h, 1);
  return SABR_OK;
}

// Uploads the tables and parameters into a scratch; returns the device image.
static sabr_status mc_shard_upload(const McShardCall& c, const double* params, cudaStream_t s, McScratch& w, McDev& d,
                                   int** q_value, int** q_out, double** disc, const double** dparams) {
  const size_t img = mc_image_bytes(c.h);
  const size_t params_off = (img + 255) & ~(size_t)255;
  const size_t part_off = params_off + 256;
  const size_t tab_bytes = mc_step_table_bytes(c.h, 1);
  SABR_TRY(w.acquire(part_off + tab_bytes, part_off, s));
  unsigned char* base = w.dev;
  mc_fill_image(c.h, w.host, base, d, q_value, q_out, disc);
  if (tab_bytes) d.tab = base + part_off;
  double p10[kMaxD];
  for (int i = 0; i < kMaxD; ++i) p10[i] = i < n_params(c.h.model) ? params[i] : 0.0;
  std::memcpy(w.host + params_off, p10, sizeof(p10));
  SABR_CUDA(cudaMemcpyAsync(w.dev, w.host, part_off, cudaMemcpyHostToDevice, s));
  *dparams = (const double*)(base + params_off);
  return SABR_OK;
}

}  // namespace sabr

extern "C" sabr_status sabr_mc_shard_layout(sabr_model model, const double* params, double fwd, const double* T,
                                            const double* K, const int8_t* is_call, const double* discount,
                                            int64_t n, int64_t n_paths, double steps_per_year, uint64_t seed,
                                            sabr_precision prec, int32_t* total_blocks,
                                            int64_t* doubles_per_block) {
  using namespace sabr;
  clear_error();
  if (!total_blocks || !doubles_per_block) return fail(SABR_EINVAL, "NULL output");
  McShardCall c;
  SABR_TRY(mc_shard_prepare(model, params, fwd, T, K, is_call, discount, n, n_paths, steps_per_year, seed, prec, c));
  *total_blocks = c.total_blocks;
  *doubles_per_block = (int64_t)c.h.n_slots * 32;
  return SABR_OK;
}

extern "C" sabr_status sabr_mc_shard_partials(sabr_model model, const double* params, double fwd, const double* T,
                                              const double* K, const int8_t* is_call, const double* discount,
                                              int64_t n, int64_t n_paths, double steps_per_year, uint64_t seed,
                                              sabr_precision prec, int32_t total_blocks, int32_t block_begin,
                                              int32_t block_count, double* partials_out, void* stream) {
  using namespace sabr;
  clear_error();
  if (!partials_out) return fail(SABR_EINVAL, "partials_out is NULL");
  McShardCall c;
  SABR_TRY(mc_shard_prepare(model, params, fwd, T, K, is_call, discount, n, n_paths, steps_per_year, seed, prec, c));
  if (total_blocks < 1 || block_count < 1 || block_begin < 0 || (int64_t)block_begin + block_count > total_blocks)
    return fail(SABR_EINVAL, "block range outside [0, total_blocks)");
  cudaStream_t s = (cudaStream_t)stream;
  McDev d;
  int *q_value, *q_out;
  double* disc;
  const double* dp;
  McScratch w;
  SABR_TRY(mc_shard_upload(c, params, s, w, d, &q_value, &q_out, &disc, &dp));
  launch_paths(c.h, d, dp, nullptr, dim3(block_count, 1), partials_out, block_begin, total_blocks, s);
  SABR_CUDA(cudaGetLastError());
  return SABR_OK;
}

extern "C" sabr_status sabr_mc_shard_reduce(sabr_model model, const double* params, double fwd, const double* T,
                                            const double* K, const int8_t* is_call, const double* discount,
                                            int64_t n, int64_t n_paths, double steps_per_year, uint64_t seed,
                                            sabr_precision prec, int32_t total_blocks, const double* partials,
                                            double* price_out, double* stderr_out, void* stream) {
  using namespace sabr;
  clear_error();
  if (!partials || !price_out) return fail(SABR_EINVAL, "NULL partials or price_out");
  McShardCall c;
  SABR_TRY(mc_shard_prepare(model, params, fwd, T, K, is_call, discount, n, n_paths, steps_per_year, seed, prec, c));
  if (total_blocks < 1) return fail(SABR_EINVAL, "total_blocks must be >= 1");
  cudaStream_t s = (cudaStream_t)stream;
  McDev d;
  int *q_value, *q_out;
  double* disc;
  const double* dp;
  McScratch w;
  SABR_TRY(mc_shard_upload(c, params, s, w, d, &q_value, &q_out, &disc, &dp));
  launch_reduce(d, 1, total_blocks, partials, q_value, q_out, disc, nullptr, price_out, stderr_out, (int)n, s);
  SABR_CUDA(cudaGetLastError());
  return SABR_OK;
}
