// sa_device.cuh -- device pieces shared by the SA kernels (sa.cu, sa_small.cu):
// staging of a problem's quotes, the argmin of the level ends, the proposal
// step and the Metropolis test.
#pragma once
#include <cstdint>

#include "common.h"
#include "engine.cuh"

namespace sabr {

// ---------------------------------------------------------------------------
// Shared-memory staging of a problem's quotes.
// ---------------------------------------------------------------------------
template <class R>
__device__ __forceinline__ SmemQuotes<R> stage_quotes(const ProblemDev& P, unsigned char* base,
                                                      int nthreads, int tid, unsigned char** end) {
  const int Q = P.n_quotes, M = P.n_mats;
  // Q + 1 quote slots: the pair layout of an odd count needs one more
  QuotePack<R>* pack = (QuotePack<R>*)base;  // base is 16-byte aligned
  R* l2k = (R*)(pack + Q + 1);
  R* mT = l2k + Q;
  const bool dyn = P.model == SABR_DYN_I || P.model == SABR_DYN_II;
  if (sizeof(R) == 4 && P.model == SABR_HAGAN) {
    float4* pr = (float4*)base;
    const float* lfk = (const float*)P.q_lfk;
    const float* l2kf = (const float*)P.q_l2kf;
    const float* T = (const float*)P.q_T;
    const float* w = (const float*)P.q_w;
    for (int j = tid; j < (Q + 1) / 2; j += nthreads) {
      const int i0 = 2 * j, i1 = 2 * j + 1;
      const bool two = i1 < Q;
      pr[2 * j] = make_float4(lfk[i0], two ? lfk[i1] : 0.0f, l2kf[i0], two ? l2kf[i1] : 0.0f);
      pr[2 * j + 1] = make_float4(T[i0], two ? T[i1] : 0.0f, -w[i0], two ? -w[i1] : 0.0f);
    }
  } else {
    for (int i = tid; i < Q; i += nthreads) {
      QuotePack<R> qp;
      qp.lfk = ((const R*)P.q_lfk)[i];
      qp.l2kf = dyn ? mat_in_slot(P.q_mat[i], R{}) : ((const R*)P.q_l2kf)[i];
      qp.T = ((const R*)P.q_T)[i];
      qp.w = ((const R*)P.q_w)[i];
      pack[i] = qp;
      l2k[i] = ((const R*)P.q_l2k)[i];
    }
  }
  for (int j = tid; j < M; j += nthreads) mT[j] = ((const R*)P.m_T)[j];
  // offsets from `base`, so that the compiler still knows the pointers to be
  // shared memory
  unsigned char* e = base + (((unsigned char*)(mT + M) - base + 15) & ~(ptrdiff_t)15);
  SmemQuotes<R> sq{pack, (const float4*)base, l2k, mT, nullptr, nullptr, nullptr};
  if (sizeof(R) == 4 && P.model == SABR_DYN_II) {
    // the Case II term-structure rule: nodes, sub-panels, maturity panels
    float4* nd = (float4*)e;
    float4* sb = nd + kC2Nodes * P.c2_nsub;
    int2* pn = (int2*)(sb + P.c2_nsub);
    for (int i = tid; i < kC2Nodes * P.c2_nsub; i += nthreads) nd[i] = P.c2_node[i];
    for (int i = tid; i < P.c2_nsub; i += nthreads) sb[i] = P.c2_sub[i];
    for (int i = tid; i < M; i += nthreads) pn[i] = P.c2_panel[i];
    sq.c2_node = nd;
    sq.c2_sub = sb;
    sq.c2_panel = pn;
    e = base + (((unsigned char*)(pn + M) - base + 15) & ~(ptrdiff_t)15);
  }
  *end = e;
  return sq;
}

// The quotes that stage_quotes left at `base`, for a function of its own (static
// models).
template <class R> __device__ __forceinline__ SmemQuotes<R> staged_quotes(int n_quotes, unsigned char* base) {
  QuotePack<R>* pack = (QuotePack<R>*)base;
  return SmemQuotes<R>{pack, (const float4*)base, (R*)(pack + n_quotes + 1), nullptr, nullptr, nullptr, nullptr};
}

// Lexicographic minimum of (f, i): the smaller f, then the smaller index, so
// the result does not depend on the order of merging.
__device__ __forceinline__ void argmin_merge(double& f, int& i, double f2, int i2) {
  if (f2 < f || (f2 == f && i2 < i)) {
    f = f2;
    i = i2;
  }
}
__device__ __forceinline__ void warp_argmin(double& f, int& i) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const double f2 = __shfl_xor_sync(0xffffffffu, f, off);
    const int i2 = __shfl_xor_sync(0xffffffffu, i, off);
    argmin_merge(f, i, f2, i2);
  }
}

template <int MODEL> struct Dim {
  static constexpr int value = MODEL == SABR_DYN_II ? 10 : (MODEL == SABR_DYN_I ? 6 : 4);
};

__device__ __forceinline__ unsigned group_mask(int G) {
  if (G >= 32) return 0xffffffffu;
  const int lane32 = threadIdx.x & 31;
  return ((1u << G) - 1u) << (lane32 & ~(G - 1));
}

__device__ __forceinline__ void load_problem(const ProblemDev* probs, int pid, ProblemDev* P) {
  const int words = (int)(sizeof(ProblemDev) / 4);
  for (int i = threadIdx.x; i < words; i += blockDim.x)
    ((int*)P)[i] = ((const int*)(probs + pid))[i];
  __syncthreads();
}

// Proposal step: x' = x + step (2u - 1).  The FP64 form rounds each
// operation exactly as written (no contraction into an FMA).
__device__ __forceinline__ float propose(float x, float step, float u) {
  return x + step * (2.0f * u - 1.0f);
}
__device__ __forceinline__ double propose(double x, double step, double u) {
  return __dadd_rn(x, __dmul_rn(step, __dsub_rn(__dmul_rn(2.0, u), 1.0)));
}
// The same step with w = 2u - 1 (exact in either precision) given.
__device__ __forceinline__ float move_by(float x, float step, float w) { return fmaf(step, w, x); }
__device__ __forceinline__ double move_by(double x, double step, double w) { return __dadd_rn(x, __dmul_rn(step, w)); }
// Metropolis acceptance of an uphill move (delta > 0) at temperature Tk.
// FP32 form: u < 2^(-delta log2(e)/Tk) by the SFU, with log2(e)/Tk formed
// once per level.
__device__ __forceinline__ bool metropolis(float u, float delta, float inv_Tk, double) {
  return u < ex2_approx(-delta * inv_Tk);
}
__device__ __forceinline__ bool metropolis(double u, double delta, float, double Tk) {
  return u < exp(-delta / Tk);
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

}  // namespace sabr
