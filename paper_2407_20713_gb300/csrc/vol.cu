// vol.cu -- sabr_implied_vol: one thread per option, grid-stride.
#include <algorithm>
#include <cmath>

#include "common.h"
#include "sabr_math.cuh"

namespace sabr {

// Everything that does not depend on the option, formed once on the host: a
// thread handles a few options only, and the FP64 pipe that the conversions,
// log2 f and (in FP64) the formula's constants took on every thread issues 1.7
// operations a clock and SM (2^20 options at any forward, FP32, us a launch in a
// graph: Hagan 20.3 -> 10.9, Obloj 21.2 -> 16.5, expanded 50.3 -> 9.6, Case I 52.5 ->
// 12.0, Case II 120 -> 93; FP64 Hagan 385 -> 333; 21 options in FP64, Hagan 12.4 ->
// 8.3).  What is left on that pipe in FP32: three conversions to floats, the
// product K f, and one back.
template <class R> struct VolArgs {
  double p[kMaxD];
  double fwd;
  R f, l2f;                 // f and log2 f
  R alpha, beta, rho, nu;
  R omr, opr;               // 1 - rho, 1 + rho
  StaticConst<R> sc;        // FP64 static formulas
};

template <class R, int MODEL>
__global__ void __launch_bounds__(256) implied_vol_kernel(const __grid_constant__ VolArgs<R> a,
                                                          const double* __restrict__ T,
                                                          const double* __restrict__ K, int64_t n,
                                                          double* __restrict__ out) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  StaticConst<R> sc;
  if constexpr (MODEL == SABR_HAGAN || MODEL == SABR_OBLOJ) {
    if constexpr (sizeof(R) == 8) {
      sc = a.sc;
    } else if constexpr (MODEL == SABR_HAGAN) {
      sc = static_setup_from<R>(a.alpha, a.beta, a.rho, a.nu, zx_setup_from(a.rho, a.omr, a.opr));
    } else {
      sc = static_setup<R>(a.p);
    }
  }
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const double kd = K[i];
    const R t = (R)T[i], k = (R)kd;
    const R lfk = m_log(a.f / k);
    R v;
    if constexpr (MODEL == SABR_HAGAN) {
      v = vol_hagan<R>(sc, lfk, m_log2((R)(kd * a.fwd)), t);
    } else if constexpr (MODEL == SABR_OBLOJ) {
      v = vol_obloj<R>(sc, lfk, m_log2((R)(kd * a.fwd)), m_log2(k), t);
    } else if constexpr (MODEL == SABR_EXPANDED) {
      v = vol_poly<R>(expanded_coef<R>(a.p, a.l2f, t), lfk);
    } else {
      v = vol_poly<R>(dynamic_coef<R, MODEL == SABR_DYN_II>(a.p, a.l2f, t), lfk);
    }
    out[i] = (double)v;
  }
}

template <class R>
static void launch_vol(int model, const double* params, double fwd, const double* T, const double* K, int64_t n,
                       double* out, cudaStream_t s) {
  VolArgs<R> a;
  for (int i = 0; i < kMaxD; ++i) a.p[i] = i < n_params(model) ? params[i] : 0.0;
  a.fwd = fwd;
  a.f = (R)fwd;
  a.l2f = (R)std::log2(fwd);
  a.alpha = (R)a.p[0];
  a.beta = (R)a.p[1];
  a.rho = (R)a.p[2];
  a.nu = (R)a.p[3];
  a.omr = (R)(1.0 - a.p[2]);
  a.opr = (R)(1.0 + a.p[2]);
  if constexpr (sizeof(R) == 8)
    a.sc = static_setup_from<double>(a.p[0], a.p[1], a.p[2], a.p[3],
                                     zx_plain<double>(a.p[2], 1.0 - a.p[2], 1.0 + a.p[2]));
  // one resident grid (eight blocks an SM), options strided over it
  const int blocks = (int)std::min<int64_t>((n + 255) / 256, (int64_t)device_sms() * 8);
  switch (model) {
    case SABR_HAGAN: implied_vol_kernel<R, SABR_HAGAN><<<blocks, 256, 0, s>>>(a, T, K, n, out); break;
    case SABR_OBLOJ: implied_vol_kernel<R, SABR_OBLOJ><<<blocks, 256, 0, s>>>(a, T, K, n, out); break;
    case SABR_EXPANDED: implied_vol_kernel<R, SABR_EXPANDED><<<blocks, 256, 0, s>>>(a, T, K, n, out); break;
    case SABR_DYN_I: implied_vol_kernel<R, SABR_DYN_I><<<blocks, 256, 0, s>>>(a, T, K, n, out); break;
    default: implied_vol_kernel<R, SABR_DYN_II><<<blocks, 256, 0, s>>>(a, T, K, n, out); break;
  }
}

}  // namespace sabr

extern "C" sabr_status sabr_implied_vol(sabr_model model, const double* params, double fwd,
                                        const double* T, const double* K, int64_t n,
                                        double* vol_out, sabr_precision prec, void* stream) {
  using namespace sabr;
  clear_error();
  SABR_TRY(check_params(model, params));
  if (!(fwd > 0.0) || !std::isfinite(fwd)) return fail(SABR_EINVAL, "fwd must be > 0");
  if (prec != SABR_FP32 && prec != SABR_FP64) return fail(SABR_EINVAL, "unknown precision");
  if (n < 0) return fail(SABR_EINVAL, "n < 0");
  if (n == 0) return SABR_OK;
  if (!T || !K || !vol_out) return fail(SABR_EINVAL, "NULL array");
  cudaStream_t s = (cudaStream_t)stream;
  if (prec == SABR_FP32)
    launch_vol<float>(model, params, fwd, T, K, n, vol_out, s);
  else
    launch_vol<double>(model, params, fwd, T, K, n, vol_out, s);
  SABR_CUDA(cudaGetLastError());
  return SABR_OK;
}
