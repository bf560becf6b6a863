// Reductions: the CFL time step, the conservation totals and the state
// checks (minimum density and pressure, non-finite values).
#include <algorithm>

#include "jz_shadow.cuh"

namespace jz {
namespace {

constexpr int kTPB = 256;
constexpr int kStatBlocks = 1216;   // 8 x 152 SMs; fixed so the sums are reproducible

// CFL rate of the advanced nodes, max of (lambda_xi + lambda_eta + lambda_zeta) / V in FP64, found
// with FP32 bounds.  The exact rate costs ~45 FP64 instructions, an SM retires one per warp in 16
// clocks, and a plain sweep is bound by that (26 ms on 1024 x 512 x 360 where its bytes take 2.5).
// So every node gets an interval [lo, hi] around its rate in FP32, and only nodes whose interval
// reaches the largest rate known so far (this warp's lower bounds, its exact values, what other
// warps have published) are evaluated exactly: the node of the maximum is always among them, so the
// result is the plain sweep's bit for bit.  A node whose quantities leave the ranges in which the
// bounds' errors are known (values that FP32 flushes, overflows or holds as subnormals, squares of
// metrics among them; NaN) is open: it claims nothing and is always evaluated.
struct RateBounds {
  float lo, hi;
};
__device__ __forceinline__ float f32_or_inf(double x) {
  return ((unsigned)__double2hiint(x) & 0x7FFFFFFFu) < 0x45E00000u ? f64_to_f32(x) : __int_as_float(0x7F800000);   // |x| < 2^95
}
__device__ __forceinline__ RateBounds rate_bounds(const ConstsF& c, const double q[5], const float S[9], float iV) {
  const RateBounds open{0.f, __int_as_float(0x7F800000)};
  unsigned big = 0;
#pragma unroll
  for (int m = 0; m < 5; ++m) big = max(big, (unsigned)__double2hiint(q[m]) & 0x7FFFFFFFu);
  if (big >= 0x45E00000u) return open;   // some |q| >= 2^95
  // each quantity below is within kRel of its FP64 value relative to the magnitudes summed in it:
  // truncated conversions (2^-23 each), a few roundings, one hardware reciprocal and square root
  constexpr float kRel = 4e-6f;
  const float rho = f64_to_f32(q[0]);
  if (!(rho > 1e-8f && rho < 1e8f) || !(iV > 1e-30f && iV < 1e30f)) return open;
  const float ir = f_rcp(rho);
  const float m1 = f64_to_f32(q[1]), m2 = f64_to_f32(q[2]), m3 = f64_to_f32(q[3]), e = f64_to_f32(q[4]);
  const float u = m1 * ir, v = m2 * ir, w = m3 * ir;
  const float ke = 0.5f * (m1 * u + m2 * v + m3 * w);
  const float p = c.gm1 * (e - ke), dp = kRel * c.gm1 * (fabsf(e) + fabsf(ke)), p_lo = p - dp, p_hi = p + dp;
  if (!(p_hi > 1e-20f && p_hi < 1e20f)) return open;
  const float a_hi = sqrtf(c.gamma * ir * p_hi), a_lo = sqrtf(c.gamma * ir * fmaxf(p_lo, 0.f));
  float lo = 0.f, hi = 0.f, s_min = 1.f, s_max = 1.f;
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) {
    const float sx = S[3 * dir], sy = S[3 * dir + 1], sz = S[3 * dir + 2];
    const float U = fabsf(sx * u + sy * v + sz * w), dU = kRel * (fabsf(sx * u) + fabsf(sy * v) + fabsf(sz * w));
    const float s2 = sx * sx + sy * sy + sz * sz, smag = sqrtf(s2);
    s_min = fminf(s_min, s2);
    s_max = fmaxf(s_max, s2);
    lo += fmaxf(U - dU, 0.f) + a_lo * smag;
    hi += U + dU + a_hi * smag;
  }
  // |S|^2 below this holds squares of its parts that FP32 rounds as subnormals or drops
  if (!(s_min > 1e-30f && s_max < 1e30f)) return open;
  const float top = hi * iV * (1.f + kRel);
  if (!(top > 1e-25f && top < 1e30f)) return open;
  // (a node whose pressure may be negative has no rate to claim: FP64 gives NaN, which the maximum drops)
  return RateBounds{p_lo > 0.f ? lo * iV * (1.f - kRel) : 0.f, top};
}

// Mf: FP32 metric records where the solver or the grid has them, else the FP64 metrics.
__global__ void __launch_bounds__(kTPB) k_cfl_rate(Dims d, GridDev g, State q, Consts c, ConstsF cf, const float* Mf,
                                                   Scalars* sc) {
  const volatile double* known = &sc->rate_max;
  const unsigned lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (kTPB / 32);
  // rows of the advanced nodes in turns of 32 along i
  const bool jet = d.topo == JZ_TOPO_JET;
  const int i0 = jet ? 1 : 0, i1 = jet ? d.ni - 1 : d.ni, j0 = jet ? 1 : 0, ej = jet ? d.nj - 2 : d.nj;
  const int segs = (i1 - i0 + 31) / 32;
  const long long n = (long long)segs * ej * d.nk;
  double rate = 0.0, cut = 0.0;            // this thread's largest exact rate; no node below cut is the maximum
  for (long long t = blockIdx.x * (long long)(kTPB / 32) + threadIdx.x / 32; t < n; t += warps) {
    const int sgm = (int)(t % segs);
    const long long r = t / segs;
    const int i = i0 + sgm * 32 + (int)lane, j = j0 + (int)(r % ej), k = (int)(r / ej);
    const bool in = i < i1;
    const long long p = pidx(d, in ? i : i0, j, k);
    double v[5];
    float S[9], iV;
#pragma unroll
    for (int m = 0; m < 5; ++m) v[m] = q.q[m][p];
    if (Mf) {
      const float4* M = reinterpret_cast<const float4*>(Mf + p * kMF);
      const float4 a = __ldg(M), b = __ldg(M + 1), e = __ldg(M + 2);
      S[0] = a.x; S[1] = a.y; S[2] = a.z; S[3] = a.w; S[4] = b.x; S[5] = b.y; S[6] = b.z; S[7] = b.w;
      S[8] = e.x;
      iV = e.z;
    } else {
#pragma unroll
      for (int m = 0; m < 9; ++m) S[m] = f32_or_inf(g.S[m][p]);
      iV = f32_or_inf(g.invV[p]);
    }
    cut = fmax(cut, *known);
    const RateBounds b = rate_bounds(cf, v, S, iV);
    float best = in && b.lo > 0.f ? b.lo : 0.f;            // (a NaN bound claims nothing)
    for (int o = 16; o > 0; o >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, o));
    // compared in FP32: the cut rounded down
    const float cutf = fmaxf(best, __double2float_rd(cut));
    if (in && !(b.hi < cutf)) rate = fmax(rate, node_rate(g, c, p, v[0], v[1], v[2], v[3], v[4]));
    double x = rate;
    if (__any_sync(0xffffffffu, x > cut)) {
      for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
      // non-negative doubles order like their bit patterns
      if (lane == 0)
        atomicMax(reinterpret_cast<unsigned long long*>(&sc->rate_max), (unsigned long long)__double_as_longlong(x));
      cut = x;
    }
  }
}

// Coefficients of the entrance shapes at the five stage times of the step (t, dt), one thread for a
// sine and then one for a coefficient; a step evaluates them once instead of once per entrance
// block and stage.
struct Forcing {
  double amp[kNF], psi[kNF], cphi[kNF], sphi[kNF], omega[JZ_N_FREQ];
  double* co;                    // null off the jet
};
constexpr int kForcing = 5 * kNF;
__device__ __forceinline__ void stage_forcing(const Forcing& f, double t, double dt) {
  const double alpha[5] = {0.25, 1.0 / 6.0, 0.375, 0.5, 1.0};
  __shared__ double am[kForcing];
  const int th = threadIdx.x, l = th / kNF, mf = th % kNF;
  if (f.co) am[th] = f.amp[mf] * sin(f.omega[mf % JZ_N_FREQ] * (t + alpha[l] * dt) + f.psi[mf]);
  __syncthreads();
  if (f.co && th < 5 * kNT) f.co[th] = shape_coef(th % kNT, am + th / kNT * kNF, f.cphi, f.sphi);
}

__global__ void __launch_bounds__(kForcing) k_set_dt(Consts c, const __grid_constant__ Forcing f, Scalars* sc) {
  const double dt = c.dt_fixed > 0.0 ? c.dt_fixed : c.cfl / sc->rate_max;
  stage_forcing(f, sc->t, dt);
  __syncthreads();
  if (threadIdx.x != 0) return;
  sc->dt = dt;
  sc->rate_max = 0.0;
  sc->res_sum = 0.0;
}

__global__ void __launch_bounds__(kForcing) k_set_time(const __grid_constant__ Forcing f, Scalars* sc, double t, double dt) {
  stage_forcing(f, t, dt);
  if (threadIdx.x == 0) {
    sc->t = t;
    sc->dt = dt;
  }
}

Forcing forcing_of(const Inflow& in) {
  Forcing f;
  f.co = in.co;
  for (int mf = 0; mf < kNF; ++mf) {
    f.amp[mf] = in.amp[mf];
    f.psi[mf] = in.psi[mf];
    f.cphi[mf] = in.cphi[mf];
    f.sphi[mf] = in.sphi[mf];
  }
  for (int q = 0; q < JZ_N_FREQ; ++q) f.omega[q] = in.omega[q];
  return f;
}

// Totals sum Q_m V, min rho, min p, non-finite flag; grid-stride with a fixed
// grid, per-block partials reduced by one block in a fixed order.
__global__ void k_stats_partial(Dims d, GridDev g, State q, Consts c, double* part) {
  const long long n = (long long)d.ni * d.nj * d.nk;
  double tot[5] = {0, 0, 0, 0, 0};
  double mn_r = 1e300, mn_p = 1e300, bad = 0.0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % d.ni);
    const long long r = t / d.ni;
    const int j = (int)(r % d.nj), k = (int)(r / d.nj);
    const long long p = pidx(d, i, j, k);
    const double V = g.compact ? (double)g.Mf[p * kMF + MF_V] : g.V[p];
    double qq[5];
    for (int m = 0; m < 5; ++m) {
      qq[m] = q.q[m][p];
      tot[m] += qq[m] * V;
      if (!isfinite(qq[m])) bad = 1.0;
    }
    const double pr = c.gm1 * (qq[4] - 0.5 * (qq[1] * qq[1] + qq[2] * qq[2] + qq[3] * qq[3]) / qq[0]);
    mn_r = fmin(mn_r, qq[0]);
    mn_p = fmin(mn_p, pr);
    if (!(qq[0] > 0.0) || !(pr > 0.0)) bad = 1.0;
  }
  __shared__ double red[8][kTPB];
  red[0][threadIdx.x] = tot[0]; red[1][threadIdx.x] = tot[1]; red[2][threadIdx.x] = tot[2];
  red[3][threadIdx.x] = tot[3]; red[4][threadIdx.x] = tot[4];
  red[5][threadIdx.x] = mn_r; red[6][threadIdx.x] = mn_p; red[7][threadIdx.x] = bad;
  __syncthreads();
  for (int s = kTPB / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      for (int m = 0; m < 5; ++m) red[m][threadIdx.x] += red[m][threadIdx.x + s];
      red[5][threadIdx.x] = fmin(red[5][threadIdx.x], red[5][threadIdx.x + s]);
      red[6][threadIdx.x] = fmin(red[6][threadIdx.x], red[6][threadIdx.x + s]);
      red[7][threadIdx.x] = fmax(red[7][threadIdx.x], red[7][threadIdx.x + s]);
    }
    __syncthreads();
  }
  if (threadIdx.x < 8) part[blockIdx.x * 8 + threadIdx.x] = red[threadIdx.x][0];
}

__global__ void k_stats_final(const double* part, int nblk, Scalars* sc) {
  __shared__ double red[8][kTPB];
  double v[8] = {0, 0, 0, 0, 0, 1e300, 1e300, 0};
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) {
    for (int m = 0; m < 5; ++m) v[m] += part[b * 8 + m];
    v[5] = fmin(v[5], part[b * 8 + 5]);
    v[6] = fmin(v[6], part[b * 8 + 6]);
    v[7] = fmax(v[7], part[b * 8 + 7]);
  }
  for (int m = 0; m < 8; ++m) red[m][threadIdx.x] = v[m];
  __syncthreads();
  for (int s = kTPB / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      for (int m = 0; m < 5; ++m) red[m][threadIdx.x] += red[m][threadIdx.x + s];
      red[5][threadIdx.x] = fmin(red[5][threadIdx.x], red[5][threadIdx.x + s]);
      red[6][threadIdx.x] = fmin(red[6][threadIdx.x], red[6][threadIdx.x + s]);
      red[7][threadIdx.x] = fmax(red[7][threadIdx.x], red[7][threadIdx.x + s]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    for (int m = 0; m < 5; ++m) sc->tot[m] = red[m][0];
    sc->min_rho = red[5][0];
    sc->min_p = red[6][0];
    sc->nonfinite = red[7][0] > 0.0 ? 1 : 0;
  }
}

}  // namespace

int stat_partial_count() { return kStatBlocks; }

cudaError_t cfl_rate(const Dims& d, const Consts& c, const GridDev& g, const float* Mf, const State& q, Scalars* sc,
                     cudaStream_t st) {
  // eight blocks per SM keep the sweep going; fewer where the grid has fewer turns of 32 nodes
  const long long turns = (long long)((d.ni + 31) / 32) * d.nj * d.nk;
  const unsigned blocks = (unsigned)std::min<long long>(8 * 152, (turns + kTPB / 32 - 1) / (kTPB / 32));
  k_cfl_rate<<<blocks, kTPB, 0, st>>>(d, g, q, c, make_constsf(c), Mf, sc);
  return cudaGetLastError();
}

cudaError_t set_dt(const Consts& c, const Inflow& in, Scalars* sc, cudaStream_t st) {
  k_set_dt<<<1, kForcing, 0, st>>>(c, forcing_of(in), sc);
  return cudaGetLastError();
}

cudaError_t set_time(const Inflow& in, Scalars* sc, double t, double dt, cudaStream_t st) {
  k_set_time<<<1, kForcing, 0, st>>>(forcing_of(in), sc, t, dt);
  return cudaGetLastError();
}

cudaError_t stats_with(const Dims& d, const Consts& c, const GridDev& g, const State& q, Scalars* sc,
                       double* part, cudaStream_t st) {
  k_stats_partial<<<kStatBlocks, kTPB, 0, st>>>(d, g, q, c, part);
  k_stats_final<<<1, kTPB, 0, st>>>(part, kStatBlocks, sc);
  return cudaGetLastError();
}

}  // namespace jz
