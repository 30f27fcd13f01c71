// cliquet.cu -- sabr_mc_cliquet: Monte Carlo price of the cliquet option of
// Sec. 6.3, eqs. (eq_cliquet) and (cliquet_global), on the paths of the
// Sec. 4 scheme: the same Philox streams, step coefficients, absorption and
// path_step as sabr_mc_price, with the reset dates inserted into the grid as
// landing points.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <vector>

#include "common.h"
#include "mc.cuh"
#include "mc_host.h"

namespace sabr {

constexpr int kClqBlock = 64;

// Sum over the block, the same in every run: butterflies within the warps,
// then the warps' sums in order by thread 0 (which returns the total).
__device__ __forceinline__ double clq_block_sum(double v, double* row) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if ((threadIdx.x & 31) == 0) row[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += row[w];
  return t;
}

// Paths per thread.
template <class R> constexpr int kClqPaths = sizeof(R) == 4 ? 4 : kMcPathsPerThread;

// What one path pays: the returns between resets, clipped and added.
template <class R> struct ClqPath {
  R prev, sum;
  // F at reset `reset`: R_i = F(d_i)/F(d_{i-1}) - 1; a path absorbed before
  // d_{i-1} adds R_i = 0 (0 to 0)
  __device__ __forceinline__ void land(int reset, R F, R fl, R cl) {
    if (reset >= 1) {
      const R ret = prev > (R)0 ? F / prev - (R)1 : (R)0;
      const R c = ret < cl ? ret : cl;
      sum += c > fl ? c : fl;
    }
    prev = F;
  }
};

// Grid-stride over paths: thread t of the grid prices paths t, t + stride,
// ... and keeps FP64 sums of the payoff and its square; each block adds its
// threads' sums in a fixed order into partial[2 b], partial[2 b + 1].  FP32
// paths advance in two pairs a thread with the packed FP32x2 instructions
// (run_path_pairs, which says what bounds it), FP64 paths kMcPathsPerThread at a
// time.  2^20 paths x 252 steps, Case I dynamics: 693 us a call with scalar steps,
// the step table formed by every block and one thread's sum over 1064 blocks,
// 529 now.
template <class R>
__global__ void __launch_bounds__(kClqBlock) cliquet_kernel(McDev P, const double* __restrict__ params,
                                                           double floor_l, double cap_l, double floor_g,
                                                           double cap_g, double* __restrict__ partial) {
  extern __shared__ __align__(16) unsigned char smem[];
  StepCoef<R>* tab = (StepCoef<R>*)smem;
  int* land = (int*)(tab + P.n_steps);  // land[r] = the step ending at reset r
  __shared__ double red[2][kClqBlock / 32];
  double p[kMaxD];
#pragma unroll
  for (int i = 0; i < kMaxD; ++i) p[i] = params[i];
  build_steps<R>(P, p, 0, tab, land);
  __syncthreads();
  const R beta_m1 = (R)(p[1] - 1.0);
  const R lnf = (R)PathUnits<R>::logu(P.fwd), lna = (R)PathUnits<R>::logu(p[0]);
  const R log_abs = (R)(P.log_absorb * PathUnits<R>::kLogUnit);
  const R fl = (R)floor_l, cl = (R)cap_l;
  double s1 = 0.0, s2 = 0.0;
  constexpr int NPT = kClqPaths<R>;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p0 < P.n_paths; p0 += NPT * stride) {
    ClqPath<R> pay[NPT];
#pragma unroll
    for (int k = 0; k < NPT; ++k) pay[k] = ClqPath<R>{(R)0, (R)0};
    int reset = 0;
    if constexpr (sizeof(R) == 4) {
      PathPairs<2> st;
      st.start(P, lnf, lna, p0, stride);
      run_path_pairs<2, kOrderCliquet>(P, tab, beta_m1, st, land[0], [&]() {
#pragma unroll
        for (int k = 0; k < 4; ++k) pay[k].land(reset, st.forward(k, log_abs), fl, cl);
        ++reset;
        return reset < P.n_mats ? land[reset] : -1;
      });
    } else {
      PathState<R> st[NPT];
#pragma unroll
      for (int k = 0; k < NPT; ++k) st[k] = PathState<R>{lnf, lna, false};
      int i_land = land[0];
      auto at_reset = [&]() {
#pragma unroll
        for (int k = 0; k < NPT; ++k)
          pay[k].land(reset, st[k].absorbed ? (R)0 : PathUnits<R>::expu(st[k].lnF), fl, cl);
        ++reset;
        i_land = reset < P.n_mats ? land[reset] : -1;
      };
      for (int i = 0; i < P.n_steps; i += 2) {
        uint4 w[NPT];
#pragma unroll
        for (int k = 0; k < NPT; ++k) w[k] = path_words(P, p0 + k * stride, i);
#pragma unroll
        for (int k = 0; k < NPT; ++k) path_step<R>(tab[i], w[k].x, w[k].y, beta_m1, log_abs, st[k]);
        if (i == i_land) at_reset();
        if (i + 1 < P.n_steps) {
#pragma unroll
          for (int k = 0; k < NPT; ++k) path_step<R>(tab[i + 1], w[k].z, w[k].w, beta_m1, log_abs, st[k]);
          if (i + 1 == i_land) at_reset();
        }
      }
    }
#pragma unroll
    for (int k = 0; k < NPT; ++k) {
      if (p0 + k * stride < P.n_paths) {
        double g = (double)pay[k].sum;
        g = g < cap_g ? g : cap_g;
        g = g > floor_g ? g : floor_g;
        s1 += g;
        s2 += g * g;
      }
    }
  }
  const double a = clq_block_sum(s1, red[0]), b = clq_block_sum(s2, red[1]);
  if (threadIdx.x == 0) {
    partial[2 * blockIdx.x] = a;
    partial[2 * blockIdx.x + 1] = b;
  }
}

// Block sums, by one block in a fixed order -> discounted mean and its
// standard error.
__global__ void __launch_bounds__(kClqBlock) cliquet_reduce_kernel(const double* __restrict__ partial, int blocks,
                                                                  int64_t n_paths, double disc,
                                                                  double* __restrict__ price,
                                                                  double* __restrict__ se) {
  __shared__ double red[2][kClqBlock / 32];
  double v = 0.0, v2 = 0.0;
  for (int b = threadIdx.x; b < blocks; b += blockDim.x) {
    v += partial[2 * b];
    v2 += partial[2 * b + 1];
  }
  const double s = clq_block_sum(v, red[0]), s2 = clq_block_sum(v2, red[1]);
  if (threadIdx.x != 0) return;
  const double N = (double)n_paths, mean = s / N;
  double var = (s2 - s * mean) / (N - 1.0);
  if (var < 0.0) var = 0.0;
  *price = disc * mean;
  if (se) *se = disc * sqrt(var / N);
}

// Scratch of one call: a call never waits for another, whatever its stream or
// thread.  A few fixed-size scratches per device (with pinned memory for the
// upload) are kept, and a call takes one whose last use the GPU has finished;
// a call that finds none, or is being captured, takes stream-ordered memory,
// whose allocation costs a call that is waited for about 200 us.
class CliquetScratch {
 public:
  sabr_status take(size_t dev_bytes, size_t host_bytes, cudaStream_t s);
  CliquetScratch() = default;
  CliquetScratch(const CliquetScratch&) = delete;
  CliquetScratch& operator=(const CliquetScratch&) = delete;
  ~CliquetScratch();
  unsigned char* dev = nullptr;
  unsigned char* host = nullptr;

 private:
  static constexpr int kSlots = 4;
  // 8192 steps take 164 KB of image and 256 KB of table; the block sums 40 KB
  static constexpr size_t kDevBytes = 512 * 1024, kHostBytes = 192 * 1024;
  struct Slot {
    unsigned char *dev = nullptr, *host = nullptr;
    cudaEvent_t done = nullptr;
    bool taken = false;
    bool ready() const { return dev && host && done; }
  };
  static std::mutex mu_;
  static std::map<int, std::array<Slot, kSlots>> slots_;
  bool take_slot();
  Slot* slot_ = nullptr;
  cudaStream_t stream_ = nullptr;
  std::vector<unsigned char> own_;
};
std::mutex CliquetScratch::mu_;
std::map<int, std::array<CliquetScratch::Slot, CliquetScratch::kSlots>> CliquetScratch::slots_;

bool CliquetScratch::take_slot() {
  int d = 0;
  if (cudaGetDevice(&d) != cudaSuccess) return false;
  // (another thread's capture forbids queries and allocations in its mode)
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) return false;
  {
    std::lock_guard<std::mutex> lock(mu_);
    for (Slot& w : slots_[d]) {
      if (w.taken) continue;
      if (!w.ready()) {
        if (!w.done) cudaEventCreateWithFlags(&w.done, cudaEventDisableTiming);
        if (!w.dev) cudaMalloc(&w.dev, kDevBytes);
        if (!w.host) cudaMallocHost(&w.host, kHostBytes);
        if (!w.ready()) break;
      } else if (cudaEventQuery(w.done) != cudaSuccess) {
        continue;
      }
      w.taken = true;
      slot_ = &w;
      break;
    }
  }
  cudaGetLastError();  // a slot that is busy or could not be made is no error
  cudaThreadExchangeStreamCaptureMode(&mode);
  return slot_ != nullptr;
}

sabr_status CliquetScratch::take(size_t dev_bytes, size_t host_bytes, cudaStream_t s) {
  stream_ = s;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusActive;
  if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) cudaGetLastError();
  if (capture == cudaStreamCaptureStatusNone && dev_bytes <= kDevBytes && host_bytes <= kHostBytes && take_slot()) {
    dev = slot_->dev;
    host = slot_->host;
    return SABR_OK;
  }
  void* p = nullptr;
  SABR_CUDA(cudaMallocAsync(&p, dev_bytes, s));
  dev = (unsigned char*)p;
  own_.assign(host_bytes, 0);  // pageable: an upload has consumed it when it returns
  host = own_.data();
  return SABR_OK;
}

// Also after an error: what the call has enqueued may still use the memory.
CliquetScratch::~CliquetScratch() {
  if (slot_) {
    if (cudaEventRecord(slot_->done, stream_) != cudaSuccess) cudaStreamSynchronize(stream_);
    std::lock_guard<std::mutex> lock(mu_);
    slot_->taken = false;
  } else if (dev) {
    cudaFreeAsync(dev, stream_);
  }
}

}  // namespace sabr

extern "C" sabr_status sabr_mc_cliquet(sabr_model model, const double* params, double fwd, double T,
                                       int32_t n_resets, double floor_local, double cap_local, double floor_global,
                                       double cap_global, double discount, int64_t n_paths, double steps_per_year,
                                       uint64_t seed, double* price_out, double* stderr_out, sabr_precision prec,
                                       void* stream) {
  using namespace sabr;
  clear_error();
  SABR_TRY(check_params(model, params));
  if (!price_out) return fail(SABR_EINVAL, "price_out is NULL");
  if (!(T > 0.0) || !std::isfinite(T)) return fail(SABR_EINVAL, "T must be finite and > 0");
  if (n_resets < 2 || n_resets > kMaxMats) return fail(SABR_EINVAL, "n_resets must lie in [2, 64]");
  if (!(floor_local <= cap_local) || !(floor_global <= cap_global) || !std::isfinite(discount))
    return fail(SABR_EINVAL, "need floor <= cap (local and global) and a finite discount");
  if (n_paths < 2) return fail(SABR_EINVAL, "n_paths must be >= 2");
  if (model == SABR_DYN_II && !case2_feasible<double, double>(params, T))
    return fail(SABR_EINVAL, "parameters violate rho(t) in [-1,1], nu(t) > 0");
  std::vector<double> resets(n_resets), K(n_resets, fwd);
  for (int i = 0; i < n_resets; ++i) resets[i] = (double)(i + 1) * T / n_resets;
  McHost h;
  SABR_TRY(mc_prepare(model, fwd, resets.data(), K.data(), nullptr, nullptr, n_resets, n_paths, steps_per_year, seed,
                      prec, h));
  const size_t smem = (size_t)h.n_steps * (prec == SABR_FP64 ? sizeof(StepCoef<double>) : sizeof(StepCoef<float>)) +
                      (size_t)n_resets * sizeof(int);
  if (smem > 200 * 1024) return fail(SABR_EINVAL, "too many time steps for one launch");
  // The grid: as many rounds of resident threads as the paths need, then
  // only the blocks that fill these rounds evenly -- 2^20 paths are 2.2
  // rounds of the 152 x 768 threads that fit, and three rounds of 576 threads
  // an SM end together where the third of 768 would leave most SMs idle.
  // Small blocks keep the SMs' shares equal.
  int per_sm = 8;
  if (prec == SABR_FP64) {
    allow_smem((const void*)cliquet_kernel<double>, smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cliquet_kernel<double>, kClqBlock, smem);
  } else {
    allow_smem((const void*)cliquet_kernel<float>, smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cliquet_kernel<float>, kClqBlock, smem);
  }
  per_sm = std::max(per_sm, 1);
  const int64_t per_block = (int64_t)kClqBlock * mc_paths_per_thread(prec);
  const int64_t units = (n_paths + per_block - 1) / per_block, resident = device_sms() * (int64_t)per_sm;
  const int64_t rounds = (units + resident - 1) / resident;
  const int blocks = (int)((units + rounds - 1) / rounds);
  const size_t img = mc_image_bytes(h);
  const size_t params_off = (img + 255) & ~(size_t)255;
  const size_t part_off = params_off + 256;
  const size_t tab_off = (part_off + sizeof(double) * 2 * blocks + 255) & ~(size_t)255;
  const size_t tab_bytes = mc_blocks_build_steps(h, blocks, kClqBlock) ? 0 : mc_step_table_bytes(h, 1);
  const size_t bytes = tab_off + tab_bytes;
  cudaStream_t s = (cudaStream_t)stream;
  CliquetScratch w;
  SABR_TRY(w.take(bytes, part_off, s));
  unsigned char* dev = w.dev;
  McDev d;
  int *q_value, *q_out;
  double* disc;
  mc_fill_image(h, w.host, dev, d, &q_value, &q_out, &disc);
  if (tab_bytes) d.tab = dev + tab_off;
  double p10[kMaxD];
  for (int i = 0; i < kMaxD; ++i) p10[i] = i < n_params(model) ? params[i] : 0.0;
  std::memcpy(w.host + params_off, p10, sizeof(p10));
  SABR_CUDA(cudaMemcpyAsync(dev, w.host, part_off, cudaMemcpyHostToDevice, s));
  double* part = (double*)(dev + part_off);
  const double* dp = (const double*)(dev + params_off);
  if (tab_bytes) mc_launch_steps(h, d, dp, nullptr, 1, s);
  if (prec == SABR_FP64)
    cliquet_kernel<double><<<blocks, kClqBlock, smem, s>>>(d, dp, floor_local, cap_local, floor_global, cap_global,
                                                          part);
  else
    cliquet_kernel<float><<<blocks, kClqBlock, smem, s>>>(d, dp, floor_local, cap_local, floor_global, cap_global,
                                                         part);
  cliquet_reduce_kernel<<<1, kClqBlock, 0, s>>>(part, blocks, n_paths, discount, price_out, stderr_out);
  SABR_CUDA(cudaGetLastError());
  return SABR_OK;
}
