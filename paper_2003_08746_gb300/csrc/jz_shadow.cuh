// FP32 shadow of an FP64 state (FP32-flux form): what the fused stage kernel's FP32 arithmetic
// reads of Q, three float2 arrays per padded node.  Shared by the stage kernel (jz_stage32.cu),
// the kernels that load a state (jz_grid.cu) and the boundary kernel (jz_bc.cu), so that every
// writer of a state leaves the same shadow bit for bit.
#pragma once

#include "jz_internal.cuh"

namespace jz {

constexpr int NSH = 3;   // float2 arrays of a shadow

struct ConstsF {
  float gamma, gm1, mu_ref, S_hat, sut_num, k_lam, k_sgs, C_s, kappa2, kappa4;
  float p_inf, ep_inf;     // p_inf, e_inf + p_inf
  double e_inf;            // p_inf / (gamma - 1), subtracted in FP64
};

// FP64 -> FP32 by bit manipulation (truncation toward zero; magnitudes below
// 2^-126 flush to signed zero).  Valid for finite |x| < 2^128.  Re-biasing the
// exponent on the high word (e - 896 fits in 8 bits) lets one funnel shift pick
// the FP32 exponent and the top 23 mantissa bits at once.
__device__ __forceinline__ float f64_to_f32(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned f = __funnelshift_l(lo, hi - (896u << 20), 3);
  const unsigned r = (f & 0x7FFFFFFFu) | (hi & 0x80000000u);
  return __uint_as_float((hi << 1) >= (897u << 21) ? r : (hi & 0x80000000u));
}

// Single MUFU approximations (relative error ~2^-22), far inside the FP32-flux
// form's error budget.
__device__ __forceinline__ float f_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The three shadow pairs of an FP64 state node (the FP32 values the stage arithmetic uses).
__device__ __forceinline__ void shadow_of(const ConstsF& c, const double q[5], float2 out[NSH]) {
  const float rp = f64_to_f32(q[0] - 1.0);
  const float m1 = f64_to_f32(q[1]), m2 = f64_to_f32(q[2]), m3 = f64_to_f32(q[3]);
  const float ep = f64_to_f32(q[4] - c.e_inf);
  const float ir = f_rcp(rp + 1.f);
  const float pp = c.gm1 * (ep - 0.5f * ir * (m1 * m1 + m2 * m2 + m3 * m3));
  out[0] = make_float2(rp, ep);
  out[1] = make_float2(m1, m2);
  out[2] = make_float2(m3, pp);
}

inline ConstsF make_constsf(const Consts& c) {
  ConstsF f;
  f.gamma = (float)c.gamma; f.gm1 = (float)c.gm1; f.mu_ref = (float)c.mu_ref; f.S_hat = (float)c.S_hat;
  f.sut_num = (float)c.sut_num; f.k_lam = (float)c.k_lam; f.k_sgs = (float)c.k_sgs; f.C_s = (float)c.C_s;
  f.kappa2 = (float)c.kappa2; f.kappa4 = (float)c.kappa4; f.p_inf = (float)c.p_inf;
  f.e_inf = c.p_inf / c.gm1;
  f.ep_inf = (float)(f.e_inf + c.p_inf);
  return f;
}

}  // namespace jz
