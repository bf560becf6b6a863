// FP32-flux form of one Runge-Kutta stage: fluxes, dissipation and SGS terms
// in FP32; the state Q, the stage combination Q^n - alpha dt RHS and the
// totals in FP64.  One fused kernel per stage, one HBM sweep:
//
//   read the FP32 shadow of Q^(l-1) (halo 2, by TMA), Q^n (FP64, own node),
//   metrics (FP32, halo 1); write Q^(l) (FP64) and its FP32 shadow.
//
// The shadow of a state is what the stage's FP32 arithmetic reads of it, kept
// beside the FP64 state in three float2 arrays per padded node:
// (rho - 1, e - e_inf), (rho u, rho v), (rho w, p - p_inf).  The offsets keep
// the FP32 values small in the ambient flow.  The stage that writes Q^(l)
// writes its shadow, and the kernels that set boundary nodes, fill ghosts or
// load a state write the shadow of what they set.
//
// Each CTA owns a TX x TY tile of (i, j) columns and marches in k; a thread
// owns the column of one node of the tile or of its one-node halo, a warp one
// row of them.  Shared memory holds a ring of four planes of the shadow (tile +
// 2-node halo; each plane is one 4-D TMA box of 34 x 12 x 1 x 3 float2 landing
// on an mbarrier) with 1/rho beside them, and the eta quantities that rows
// exchange (H^eta, Lambda^eta, nu^eta of one plane, two planes in turn).
// Everything else stays with its thread.  Per plane p:
//   (a) wait for the shadow of plane p+2 (requested one plane earlier) and
//       form 1/rho on its points;
//   (b) the node of plane p+1 gets its gradients, viscous and inviscid
//       transformed fluxes H^dir, spectral radii Lambda^dir and pressure
//       sensors nu^dir; its eta quantities go to shared memory, its xi faces
//       and the xi part of its RHS are formed from the neighbouring lanes
//       (shuffles);
//       one barrier; one thread requests plane p+3;
//   (c) the node of plane p gets its zeta face, which completes its RHS (xi
//       and eta part from the iteration before), and its update;
//   (d) the eta faces below and above the node of plane p+1 (each face formed
//       by both its nodes: cheaper than a second exchange) and the eta part.
//
// On a GB300 the FP64 pipe (DADD/DFMA, and also the F2F conversions between
// FP64 and FP32) issues ~2 instructions per SM per clock against 128 for
// FP32, so FP64 -> FP32 conversions are done with integer bit operations
// (truncation), and FP32 -> FP64 exactly, also with integer operations.
// Only the offsets rho - 1, e - e_inf and the final Q^n - dQ are FP64
// additions.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cstring>

#include "jz_mbar.cuh"
#include "jz_shadow.cuh"

namespace jz {
namespace {

constexpr int TX = 30, TY = 8;
constexpr int H1X = TX + 2, H1Y = TY + 2, NP1 = H1X * H1Y;   // 32 x 10
constexpr int H2X = TX + 4, H2Y = TY + 4, NP2 = H2X * H2Y;   // 34 x 12
constexpr int NT = NP1;                                      // threads per CTA
static_assert(TX == 30, "a warp holds a row of the tile and its halo");
constexpr int NIR = (NP2 + NT - 1) / NT;                     // halo-2 points per thread (1/rho pass)

// shadow ring: per halo-2 point three float2 pairs, as in global memory
// (rho' = rho - 1, e' = e - e_inf), (m1, m2), (m3, p' = p - p_inf), and 1/rho beside them
// (u = m/rho and T = gamma p/rho are formed where they are used)
constexpr int NRING = 4;           // planes k-1 .. k+2: the next plane's request needs no barrier
constexpr int BOX_BYTES = NSH * NP2 * 8;                       // one TMA box (34 x 12 x 1 x 3 float2)
constexpr int SLOT = ((BOX_BYTES + 127) / 128) * 128 / 8;      // float2 per ring slot, 128-byte aligned
// eta exchange between rows, two planes in turn: H^eta(5), Lambda^eta, nu^eta
constexpr int E_H = 0, E_L = 5, E_N = 6, NEF = 7;

struct Smem {
  float2 sh[NRING][SLOT];          // TMA destinations (first member: 128-byte aligned)
  float ir[NRING][NP2];
  float eta[2][NEF][NP1];
  float carry[5][NP1];             // H^zeta(p-1) of each thread's column
  unsigned long long bar[NRING];   // one mbarrier per ring slot
  int fail;                        // a bounded wait ran out in this CTA
};

// FP32 -> FP64, exact (subnormals flush to zero; Inf/NaN kept).
__device__ __forceinline__ double f32_to_f64(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned s = b & 0x80000000u, e8 = (b >> 23) & 0xFFu, m = b & 0x7FFFFFu;
  if (e8 == 0) return __hiloint2double((int)s, 0);
  const unsigned e11 = e8 == 0xFFu ? 0x7FFu : e8 + 896u;
  return __hiloint2double((int)(s | (e11 << 20) | (m >> 3)), (int)(m << 29));
}

// Single MUFU approximations as f_rcp (relative error ~2^-22).
__device__ __forceinline__ float f_sqrt(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float f_ex2(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float f_lg2(float x) {
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float cbrt_pos(float x) {   // x >= 0; 0 -> 0
  return x > 0.f ? f_ex2(f_lg2(x) * (1.f / 3.f)) : 0.f;
}

__device__ __forceinline__ int ring(int k) { return (k + 8) & (NRING - 1); }   // k >= -8

__device__ __forceinline__ bool in_padded(const Dims& d, int i, int j) {
  return i >= -kG && i <= d.ni + 1 && j >= -kG && j <= d.nj + 1;
}

// Turkel-Vatsa face flux between nodes a and b = a + s (d = Lambda_f [eps2 dQ - eps4 d3Q]).
__device__ __forceinline__ void face_flux(const ConstsF& c, float La, float Lb, float na, float nb,
                                          const float qm[5], const float q0[5], const float q1[5],
                                          const float q2[5], float out[5]) {
  const float eps2 = c.kappa2 * fmaxf(na, nb);
  const float eps4 = fmaxf(0.f, c.kappa4 - eps2);
  const float Lf = 0.5f * (La + Lb);
  // Lf (eps2 d1 - eps4 d3) with d3 = (q2 - qm) - 3 d1, as (Lf eps2 + 3 Lf eps4) d1 - Lf eps4 (q2 - qm)
  const float b = Lf * eps4;
  const float a3 = fmaf(3.f, b, Lf * eps2);
#pragma unroll
  for (int m = 0; m < 5; ++m) out[m] = fmaf(a3, q1[m] - q0[m], -b * (q2[m] - qm[m]));
}

struct Args {
  CUtensorMap tm;            // shadow of Q^(l-1): 4-D (Pi, Pj, Pk, 3) of float2, box 34 x 12 x 1 x 3
  Dims d;
  ConstsF c;
  const float* M;            // FP32 metric records, kMF floats per padded node
  const double* qin[5];      // FP64 Q^(l-1): copied on the nodes the stage does not advance
  const double* qn[5];
  double* qout[5];
  float2* sout[NSH];         // shadow of Q^(l) (not used with rhs)
  double* rhs;               // non-null: write RHS [5][N] instead of updating
  Scalars* sc;
  double alpha;
  int kchunk;
  int want_res;
  int want_rate;
};

// ---- TMA (inline PTX) ----
// Request the shadow of plane k (padded plane k + 2) of this CTA's halo-2 box into a ring slot;
// the mbarrier completes when its BOX_BYTES have landed.  Called by one thread.
__device__ __forceinline__ void request_plane(const Args& A, Smem& sm, int slot, int x0, int y0, int k) {
  unsigned long long* b = &sm.bar[slot];
  // the slot's previous contents were read through the generic proxy before the last barrier
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(BOX_BYTES)
               : "memory");
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
      "%5}], [%6];" ::"r"(smem_u32(&sm.sh[slot][0])),
      "l"(reinterpret_cast<unsigned long long>(&A.tm)), "r"(x0), "r"(y0), "r"(k + kG), "r"(0), "r"(smem_u32(b))
      : "memory");
}
__device__ __forceinline__ bool wait_slot(Smem& sm, int slot, unsigned parity) { return wait_bar(&sm.bar[slot], parity); }

// Plane k of the CTA starting at k0 - 2 uses ring slot ring(k) for the ((k - k0 + 2) / 4)-th time.
__device__ __forceinline__ unsigned plane_parity(int k, int k0) { return (unsigned)((k - k0 + 2) >> 2) & 1u; }

// 1/rho on the halo-2 points of a landed shadow plane (rho = rho' + 1).
__device__ __forceinline__ void inv_rho(Smem& sm, int slot) {
#pragma unroll
  for (int r = 0; r < NIR; ++r) {
    const int t = threadIdx.x + r * NT;
    if (t < NP2) sm.ir[slot][t] = f_rcp(sm.sh[slot][t].x + 1.f);
  }
}

// Metric record of one node (three 16-byte loads).
__device__ __forceinline__ void load_record(const float* M, unsigned p, float met[kMF]) {
  const float4* r = reinterpret_cast<const float4*>(M) + (unsigned long long)p * (kMF / 4);
  const float4 a = __ldg(r), b = __ldg(r + 1), c = __ldg(r + 2);
  met[0] = a.x; met[1] = a.y; met[2] = a.z; met[3] = a.w;
  met[4] = b.x; met[5] = b.y; met[6] = b.z; met[7] = b.w;
  met[8] = c.x; met[9] = c.y; met[10] = c.z; met[11] = c.w;
}

// Ask L2 to fetch the sector holding p (no register, no wait).
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// A landed ring slot: the shadow pairs and 1/rho of its halo-2 points.
struct Plane {
  const float2* s;
  const float* ir;
};
__device__ __forceinline__ Plane plane(const Smem& sm, int slot) { return Plane{sm.sh[slot], sm.ir[slot]}; }
__device__ __forceinline__ float2 P_re(const Plane& P, int c) { return P.s[c]; }              // rho', e'
__device__ __forceinline__ float2 P_m12(const Plane& P, int c) { return P.s[NP2 + c]; }       // m1, m2
__device__ __forceinline__ float2 P_m3p(const Plane& P, int c) { return P.s[2 * NP2 + c]; }   // m3, p'
// The five conserved offsets (rho', m1, m2, m3, e') of a ring point: what the dissipation acts on.
__device__ __forceinline__ void load_q(const Plane& P, int c, float q[5]) {
  const float2 a = P_re(P, c), b = P_m12(P, c), d = P_m3p(P, c);
  q[0] = a.x; q[1] = b.x; q[2] = b.y; q[3] = d.x; q[4] = a.y;
}

// Transformed fluxes, anisotropic spectral radii and pressure sensors of one node, and 1/V.
struct Node {
  float H[3][5], lam[3], nu[3], iV;
};

// ... of one node of plane q (slots s_m, s_0, s_p of planes q-1, q, q+1) at halo-2 index c2.
__device__ __forceinline__ void nodal(const Args& A, const Smem& sm, const float met[kMF], int s_m, int s_0, int s_p,
                                      int c2, Node& N) {
  const ConstsF& c = A.c;
  float S[3][3];
#pragma unroll
  for (int dir = 0; dir < 3; ++dir)
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) S[dir][cc] = met[3 * dir + cc];
  const float iV = met[MF_IV];
  const Plane P0 = plane(sm, s_0), Pm = plane(sm, s_m), Pp = plane(sm, s_p);
  // u, v, w, T at a node of the ring (plane P, halo-2 index cc, 1/rho there; that of plane q+1 is only
  // being written by others and formed again)
  auto uvwT = [&](const Plane& P, int cc, float ir, float f[4]) {
    const float2 a = P_m12(P, cc), b = P_m3p(P, cc);
    f[0] = a.x * ir;
    f[1] = a.y * ir;
    f[2] = b.x * ir;
    f[3] = c.gamma * (b.y + c.p_inf) * ir;
  };
  // gradients of u, v, w, T: L[n][j] = sum_dir (S^dir_j / (2V)) (f_{+} - f_{-})
  const float h = 0.5f * iV;
  float fxp[4], fxm[4], fyp[4], fym[4], fzp[4], fzm[4];
  uvwT(P0, c2 + 1, P0.ir[c2 + 1], fxp);
  uvwT(P0, c2 - 1, P0.ir[c2 - 1], fxm);
  uvwT(P0, c2 + H2X, P0.ir[c2 + H2X], fyp);
  uvwT(P0, c2 - H2X, P0.ir[c2 - H2X], fym);
  uvwT(Pp, c2, f_rcp(P_re(Pp, c2).x + 1.f), fzp);
  uvwT(Pm, c2, Pm.ir[c2], fzm);
  float L[4][3];
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    const float dx = fxp[n] - fxm[n], dy = fyp[n] - fym[n], dz = fzp[n] - fzm[n];
#pragma unroll
    for (int jj = 0; jj < 3; ++jj) L[n][jj] = h * (S[0][jj] * dx + S[1][jj] * dy + S[2][jj] * dz);
  }
  const float2 re0 = P_re(P0, c2), m12 = P_m12(P0, c2), m3p = P_m3p(P0, c2);
  const float rho = re0.x + 1.f;
  const float m1 = m12.x, m2 = m12.y, m3 = m3p.x;
  float f0[4];
  uvwT(P0, c2, P0.ir[c2], f0);
  const float u = f0[0], v = f0[1], w = f0[2], T = f0[3];
  const float pp = m3p.y;
  const float ep = re0.y;
  const float a = f_sqrt(T);
  const float mu = c.mu_ref * (T * a) * c.sut_num * f_rcp(T + c.S_hat);
  // strain rate (symmetric), eddy viscosity, stresses
  const float s11 = L[0][0], s22 = L[1][1], s33 = L[2][2];
  const float s12 = 0.5f * (L[0][1] + L[1][0]), s13 = 0.5f * (L[0][2] + L[2][0]), s23 = 0.5f * (L[1][2] + L[2][1]);
  const float div = s11 + s22 + s33;
  const float SS = s11 * s11 + s22 * s22 + s33 * s33 + 2.f * (s12 * s12 + s13 * s13 + s23 * s23);
  const float Smod = f_sqrt(2.f * SS);
  const float csd = c.C_s * met[MF_D];
  const float mu_sgs = rho * (csd * csd) * Smod;
  const float m2e = 2.f * (mu + mu_sgs);
  const float k_eff = mu * c.k_lam + mu_sgs * c.k_sgs;
  const float d3 = div * (1.f / 3.f);
  const float t11 = m2e * (s11 - d3), t22 = m2e * (s22 - d3), t33 = m2e * (s33 - d3);
  const float t12 = m2e * s12, t13 = m2e * s13, t23 = m2e * s23;
  // Cartesian viscous fluxes F_x, F_y, F_z (momentum x, y, z; energy)
  const float F[3][4] = {{t11, t12, t13, u * t11 + v * t12 + w * t13 + k_eff * L[3][0]},
                         {t12, t22, t23, u * t12 + v * t22 + w * t23 + k_eff * L[3][1]},
                         {t13, t23, t33, u * t13 + v * t23 + w * t33 + k_eff * L[3][2]}};
  const float h0 = ep + pp + c.ep_inf;   // e + p
  float lam[3];
  float (*H)[5] = N.H;
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) {
    const float U = S[dir][0] * u + S[dir][1] * v + S[dir][2] * w;
    const float smag = f_sqrt(S[dir][0] * S[dir][0] + S[dir][1] * S[dir][1] + S[dir][2] * S[dir][2]);
    lam[dir] = fabsf(U) + a * smag;
    H[dir][0] = rho * U;
    H[dir][1] = m1 * U + pp * S[dir][0] - (S[dir][0] * F[0][0] + S[dir][1] * F[1][0] + S[dir][2] * F[2][0]);
    H[dir][2] = m2 * U + pp * S[dir][1] - (S[dir][0] * F[0][1] + S[dir][1] * F[1][1] + S[dir][2] * F[2][1]);
    H[dir][3] = m3 * U + pp * S[dir][2] - (S[dir][0] * F[0][2] + S[dir][1] * F[1][2] + S[dir][2] * F[2][2]);
    H[dir][4] = h0 * U - (S[dir][0] * F[0][3] + S[dir][1] * F[1][3] + S[dir][2] * F[2][3]);
  }
  const float r0 = cbrt_pos(lam[0]), r1 = cbrt_pos(lam[1]), r2 = cbrt_pos(lam[2]);
  // pressure sensors (p' = p - p_inf; denominators add 4 p_inf back)
  const float pxm = P_m3p(P0, c2 - 1).y, pxp = P_m3p(P0, c2 + 1).y;
  const float pym = P_m3p(P0, c2 - H2X).y, pyp = P_m3p(P0, c2 + H2X).y;
  const float pzm = P_m3p(Pm, c2).y, pzp = P_m3p(Pp, c2).y;
  const float p4 = 4.f * c.p_inf;
  N.lam[0] = lam[0] + r0 * (r1 * r1 + r2 * r2);
  N.lam[1] = lam[1] + r1 * (r0 * r0 + r2 * r2);
  N.lam[2] = lam[2] + r2 * (r0 * r0 + r1 * r1);
  N.nu[0] = fabsf(pxp - 2.f * pp + pxm) * f_rcp(pxp + 2.f * pp + pxm + p4);
  N.nu[1] = fabsf(pyp - 2.f * pp + pym) * f_rcp(pyp + 2.f * pp + pym + p4);
  N.nu[2] = fabsf(pzp - 2.f * pp + pzm) * f_rcp(pzp + 2.f * pp + pzm + p4);
  N.iV = iV;
}

// Latency and issue bound it (56% of the cycles issue, 20 warps per SM): 9.9 ms per launch on
// 1024 x 512 x 360, 2.9 TB/s of algorithmic bytes, against 13.0 with the zeta and xi quantities and
// the faces in shared memory too and two barriers per plane.  Rows per tile: 8 (96 registers, two
// CTAs per SM); 6: 11.7, 9 (88 registers, spills): 17.5, 12 at one CTA: 12.8.  H^zeta(p-1) in shared
// memory instead of registers (spills): 10.8 against 12.0; metric records and Q^n a plane ahead by
// cp.async: 11.8 against 10.3.
__global__ void __launch_bounds__(NT, 2) k_fused32(const __grid_constant__ Args A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // TMA destinations need 128-byte alignment; the launch adds 128 bytes of room for it
  Smem& sm = *reinterpret_cast<Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~(uintptr_t)127);
  const Dims& d = A.d;
  const ConstsF& c = A.c;
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
  const int k0 = blockIdx.z * A.kchunk;
  const int k1 = min(k0 + A.kchunk, d.nk);          // output planes [k0, k1)
  const int t = threadIdx.x;
  // this thread's node: one row of the tile and its one-node halo per warp
  const int x1 = t & 31, y1 = t >> 5;
  const int oi = i0 - 1 + x1, oj = j0 - 1 + y1;
  const int c2 = (y1 + 1) * H2X + (x1 + 1);         // its halo-2 index
  const bool valid = in_padded(d, oi, oj);
  const bool rowt = y1 >= 1 && y1 <= TY;            // (uniform in a warp)
  const bool outv = rowt && x1 >= 1 && x1 <= TX && oi < d.ni && oj < d.nj;   // an output node
  const bool adv = outv && (d.topo != JZ_TOPO_JET || (oi >= 1 && oi <= d.ni - 2 && oj >= 1 && oj <= d.nj - 2));
  // the halo-2 box starts at real (i0 - 2, j0 - 2): padded (i0, j0); x0 * 8 bytes is a multiple
  // of 16 because TX is even
  const int x0 = i0, y0 = j0;
  // its element in plane p of a padded field (32 bits: a field's Np nodes at 240 bytes each, three
  // states with their shadows and the metric records, reach the GPU's memory before 2^32), here for p = k0 - 2
  const unsigned sk = (unsigned)d.sk;
  unsigned pp = (unsigned)(valid ? pidx(d, oi, oj, k0 - 2) : 0);
  // prime: mbarriers, then planes k0-2 .. k0 requested; k0-2 and k0-1 waited for
  int last_req = k0 - 3;                           // thread 0: last plane requested
  if (t == 0) {
    for (int s = 0; s < NRING; ++s) bar_init(&sm.bar[s], 1);
    sm.fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (t == 0) {
    for (int q = k0 - 2; q <= k0; ++q) request_plane(A, sm, ring(q), x0, y0, q);
    last_req = k0;
  }
  for (int q = k0 - 2; q <= k0 - 1; ++q) {
    if (!wait_slot(sm, ring(q), plane_parity(q, k0))) sm.fail = q + 1000000;
    inv_rho(sm, ring(q));
  }
  __syncthreads();                                 // 1/rho of the first two planes

  // marching state of the thread's column: plane p-1 (fluxes, Q, face p-1/2) and plane p (zeta
  // quantities, and the xi and eta part of its RHS)
  float Hz_0[5] = {0, 0, 0, 0, 0};      // H^zeta(p); H^zeta(p-1) is kept in shared memory
  float Dz_prev[5] = {0, 0, 0, 0, 0};   // d^zeta(p-1/2)
  for (int m = 0; m < 5; ++m) sm.carry[m][t] = 0.f;
  float Qz_prev[5] = {0, 0, 0, 0, 0};   // Q(p-1), FP32
  float acc[5] = {0, 0, 0, 0, 0};       // xi and eta part of plane p
  float Lz = 0.f, Nz = 0.f, iV0 = 0.f;  // Lambda^zeta(p), nu^zeta(p), 1/V(p)
  const float adt = f64_to_f32(A.alpha * A.sc->dt);
  float res = 0.f, rate = 0.f;

  for (int p = k0 - 2; p < k1; ++p, pp += sk) {
    const Plane P0 = plane(sm, ring(p)), P1 = plane(sm, ring(p + 1)), P2 = plane(sm, ring(p + 2));
    // (a) metrics of plane p+1; the shadow of plane p+2 (requested one plane earlier) and its 1/rho
    float met[kMF] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (valid) {
      load_record(A.M, pp + sk, met);
      if (p + 2 <= k1) {
        // the next plane's record: it spans two 32-byte sectors, and with the neighbours' requests
        // every sector of the row is asked for
        const float* pm = A.M + (unsigned long long)(pp + 2 * sk) * kMF;
        prefetch_l2(pm);
        prefetch_l2(pm + 8);
      }
    }
    // after a wait ran out no plane is requested or waited for any more (the CTA finishes on
    // stale data and the host reports the error)
    if (sm.fail == 0 && !wait_slot(sm, ring(p + 2), plane_parity(p + 2, k0))) sm.fail = p + 2 + 1000000;
    inv_rho(sm, ring(p + 2));                      // (neighbours read it one plane later)
    // (b) the node of plane p+1; its eta quantities for the rows above and below
    // Q^n of the output node of plane p, requested before the work that hides its latency
    double qn_r[5];
    if (p >= k0 && adv && !A.rhs) {
#pragma unroll
      for (int m = 0; m < 5; ++m) qn_r[m] = __ldg(A.qn[m] + pp);
    }
    Node N;                                        // (zeros outside the padded box, as its metrics)
    nodal(A, sm, met, ring(p), ring(p + 1), ring(p + 2), c2, N);
    float* E = &sm.eta[p & 1][0][0];
    const bool inplane = p + 1 >= k0 && p + 1 < k1;   // plane p+1 is an output plane
    float ax[5] = {0.f, 0.f, 0.f, 0.f, 0.f};          // its xi (and then eta) part
    if (inplane) {
#pragma unroll
      for (int m = 0; m < 5; ++m) E[(E_H + m) * NP1 + t] = N.H[1][m];
      E[E_L * NP1 + t] = N.lam[1];
      E[E_N * NP1 + t] = N.nu[1];
      if (rowt) {
        // xi faces: each lane the face to its right neighbour, the left one from the lane before
        float qm[5], q0[5], q1[5], q2[5], out[5];
        load_q(P1, c2 - 1, qm);
        load_q(P1, c2, q0);
        load_q(P1, c2 + 1, q1);
        load_q(P1, c2 + 2, q2);
        const unsigned all = 0xffffffffu;
        face_flux(c, N.lam[0], __shfl_down_sync(all, N.lam[0], 1), N.nu[0], __shfl_down_sync(all, N.nu[0], 1), qm, q0, q1,
                  q2, out);
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          const float hp = __shfl_down_sync(all, N.H[0][m], 1), hm = __shfl_up_sync(all, N.H[0][m], 1);
          ax[m] = 0.5f * (hp - hm) - (out[m] - __shfl_up_sync(all, out[m], 1));
        }
      }
    }
    // The one barrier of a plane: 1/rho of plane p+2 and the eta quantities of plane p+1 are there;
    // every thread is done with plane p-1 of the ring and with the eta quantities of plane p.
    __syncthreads();
    if (t == 0 && p + 3 <= k1 + 1 && sm.fail == 0) {
      request_plane(A, sm, ring(p + 3), x0, y0, p + 3);
      last_req = p + 3;
    }
    if (rowt) {
      // (c) zeta face p+1/2, RHS and update of plane p
      float q0[5], q1[5], q2[5], Dz[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
      load_q(P0, c2, q0);
      load_q(P1, c2, q1);
      load_q(P2, c2, q2);
      if (p >= k0 - 1) face_flux(c, Lz, N.lam[2], Nz, N.nu[2], Qz_prev, q0, q1, q2, Dz);
      if (p >= k0 && outv) {
        float R[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          float a = acc[m];
          a += 0.5f * (N.H[2][m] - sm.carry[m][t]) - (Dz[m] - Dz_prev[m]);
          R[m] = a * iV0;
        }
        if (A.rhs) {
          const long long Nr = (long long)d.ni * d.nj * d.nk;
          const long long ridx = ((long long)p * d.nj + oj) * d.ni + oi;
#pragma unroll
          for (int m = 0; m < 5; ++m) A.rhs[m * Nr + ridx] = adv ? f32_to_f64(R[m]) : 0.0;
        } else if (adv) {
          double qnew[5];
#pragma unroll
          for (int m = 0; m < 5; ++m) {
            qnew[m] = qn_r[m] - f32_to_f64(adt * R[m]);
            A.qout[m][pp] = qnew[m];
          }
          float2 shn[NSH];
          shadow_of(c, qnew, shn);
#pragma unroll
          for (int m = 0; m < NSH; ++m) A.sout[m][pp] = shn[m];
          if (A.want_rate) {
            const float rho = f64_to_f32(qnew[0]);
            const float ir = f_rcp(rho);
            const float m1 = f64_to_f32(qnew[1]), m2 = f64_to_f32(qnew[2]), m3 = f64_to_f32(qnew[3]);
            const float u = m1 * ir, v = m2 * ir, w = m3 * ir;
            const float pr = c.gm1 * (f64_to_f32(qnew[4] - c.e_inf) - 0.5f * (m1 * u + m2 * v + m3 * w)) + c.p_inf;
            const float a = f_sqrt(c.gamma * pr * ir);
            float ls = 0.f;
            float mr[kMF];
            load_record(A.M, pp, mr);
#pragma unroll
            for (int dir = 0; dir < 3; ++dir) {
              const float sx = mr[3 * dir], sy = mr[3 * dir + 1], sz = mr[3 * dir + 2];
              ls += fabsf(sx * u + sy * v + sz * w) + a * f_sqrt(sx * sx + sy * sy + sz * sz);
            }
            rate = fmaxf(rate, ls * iV0);
          }
        } else {
#pragma unroll
          for (int m = 0; m < 5; ++m) A.qout[m][pp] = A.qin[m][pp];
          A.sout[0][pp] = P_re(P0, c2);
          A.sout[1][pp] = P_m12(P0, c2);
          A.sout[2][pp] = P_m3p(P0, c2);
        }
        if (adv) res += R[0] * R[0];
      }
      // (d) eta faces of plane p+1, both of the node's, and its xi and eta part
      if (inplane) {
        float qa[5], qb[5], qc[5], qd[5], lo[5], hi[5];
        load_q(P1, c2 - 2 * H2X, qa);
        load_q(P1, c2 - H2X, qb);
        load_q(P1, c2 + H2X, qc);
        load_q(P1, c2 + 2 * H2X, qd);
        face_flux(c, E[E_L * NP1 + t - 32], N.lam[1], E[E_N * NP1 + t - 32], N.nu[1], qa, qb, q1, qc, lo);
        face_flux(c, N.lam[1], E[E_L * NP1 + t + 32], N.nu[1], E[E_N * NP1 + t + 32], qb, q1, qc, qd, hi);
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          float a = ax[m];
          a += 0.5f * (E[(E_H + m) * NP1 + t + 32] - E[(E_H + m) * NP1 + t - 32]) - (hi[m] - lo[m]);
          ax[m] = a;
        }
      }
      // rotate the marching state
#pragma unroll
      for (int m = 0; m < 5; ++m) {
        sm.carry[m][t] = Hz_0[m];
        Hz_0[m] = N.H[2][m];
        Dz_prev[m] = Dz[m];
        Qz_prev[m] = q0[m];
        acc[m] = ax[m];
      }
      Lz = N.lam[2];
      Nz = N.nu[2];
      iV0 = N.iV;
    }
  }
  if (t == 0 && sm.fail != 0) {
    // a wait ran out: give the copies still in flight a bounded time to land before the CTA's
    // shared memory is released, then report
    for (int q = sm.fail - 1000000; q <= last_req; ++q) wait_slot(sm, ring(q), plane_parity(q, k0));
    atomicOr(&A.sc->wait_timeout, 1);
  }
  if (A.want_res || A.want_rate) {
    __shared__ float red[2][NT / 32];
    float r1 = res, r2 = rate;
    for (int o = 16; o > 0; o >>= 1) {
      r1 += __shfl_xor_sync(0xffffffffu, r1, o);
      r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
    }
    if ((t & 31) == 0) { red[0][t >> 5] = r1; red[1][t >> 5] = r2; }
    __syncthreads();
    if (t == 0) {
      float s1 = 0.f, s2 = 0.f;
      for (int w = 0; w < NT / 32; ++w) { s1 += red[0][w]; s2 = fmaxf(s2, red[1][w]); }
      if (A.want_res) atomicAdd(&A.sc->res_sum, (double)s1);
      if (A.want_rate && s2 > 0.f)
        atomicMax(reinterpret_cast<unsigned long long*>(&A.sc->rate_max),
                  (unsigned long long)__double_as_longlong((double)s2));
    }
  }
}


// Self-check of the bounded wait: one warp initialises an mbarrier that nothing ever arrives at
// and waits for it with the stage kernel's bounded poll; the wait must run out and return.
__global__ void k_wait_check(int* timed_out, long long* cycles) {
  __shared__ unsigned long long bar;
  if (threadIdx.x == 0) {
    bar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const long long t0 = clock64();
  const bool ok = wait_bar(&bar, 0);
  const long long t1 = clock64();
  if (threadIdx.x == 0) {
    *timed_out = ok ? 0 : 1;
    *cycles = t1 - t0;
  }
}

constexpr int kSmemBytes = (int)sizeof(Smem) + 128;    // + room to align the ring to 128 bytes
static_assert(TX % 2 == 0, "the TMA box must start on a 16-byte boundary (x0 = i0 padded, 8-byte elements)");

// The dynamic shared-memory size above 48 KB must be allowed once per device.
cudaError_t allow_smem() {
  static std::atomic<bool> attr[64];
  int dev = 0;
  cudaError_t e0 = cudaGetDevice(&dev);
  if (e0 != cudaSuccess) return e0;
  if (dev < 0 || dev >= 64 || !attr[dev].load(std::memory_order_relaxed)) {
    cudaError_t e = cudaFuncSetAttribute(k_fused32, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) attr[dev].store(true, std::memory_order_relaxed);
  }
  return cudaSuccess;
}

}  // namespace

// Resident CTAs of the fused kernel on the whole device (SMs x CTAs per SM).
cudaError_t fused32_slots(int* slots) {
  cudaError_t e = allow_smem();
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_fused32, NT, kSmemBytes);
  if (e != cudaSuccess) return e;
  *slots = sms * (per > 0 ? per : 1);
  return cudaSuccess;
}

cudaError_t make_shadow_map(const Dims& d, float2* sh, void* tmap128) {
  static std::atomic<PFN_cuTensorMapEncodeTiled_v12000> known{nullptr};
  PFN_cuTensorMapEncodeTiled_v12000 encode = known.load(std::memory_order_relaxed);
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess) return e;
    if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorInvalidValue;
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    known.store(encode, std::memory_order_relaxed);
  }
  // 8-byte elements (one float2 pair each); rows of Pi, planes of Pi x Pj, three arrays of Np
  const cuuint64_t dims[4] = {(cuuint64_t)d.Pi, (cuuint64_t)d.Pj, (cuuint64_t)d.Pk, (cuuint64_t)NSH};
  const cuuint64_t strides[3] = {(cuuint64_t)d.Pi * 8, (cuuint64_t)d.sk * 8, (cuuint64_t)d.Np * 8};
  const cuuint32_t box[4] = {(cuuint32_t)H2X, (cuuint32_t)H2Y, 1, (cuuint32_t)NSH};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = encode(static_cast<CUtensorMap*>(tmap128), CU_TENSOR_MAP_DATA_TYPE_UINT64, 4, sh, dims, strides,
                            box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t fused32(const Dims& d, const Consts& c, const float* Mf, const State& qin, const void* tm_in,
                    const State& qn, const State& qout, Scalars* sc, double alpha, int want_res, int want_rate,
                    double* rhs_flat, int kchunk, cudaStream_t st) {
  cudaError_t e0 = allow_smem();
  if (e0 != cudaSuccess) return e0;
  Args A;
  std::memcpy(&A.tm, tm_in, sizeof(CUtensorMap));
  A.d = d;
  A.c = make_constsf(c);
  A.M = Mf;
  for (int m = 0; m < 5; ++m) {
    A.qin[m] = qin.q[m];
    A.qn[m] = qn.q[m];
    A.qout[m] = qout.q[m];
  }
  if (d.Np >= (1LL << 32)) return cudaErrorInvalidValue;
  for (int m = 0; m < NSH; ++m) A.sout[m] = qout.sh + m * d.Np;
  A.rhs = rhs_flat;
  A.sc = sc;
  A.alpha = alpha;
  A.kchunk = kchunk > 0 ? kchunk : d.nk;
  A.want_res = want_res;
  A.want_rate = want_rate;
  dim3 grid((d.ni + TX - 1) / TX, (d.nj + TY - 1) / TY, (d.nk + A.kchunk - 1) / A.kchunk);
  k_fused32<<<grid, NT, kSmemBytes, st>>>(A);
  return cudaGetLastError();
}

cudaError_t wait_check(int* dev_timed_out, long long* dev_cycles, cudaStream_t st) {
  k_wait_check<<<1, 32, 0, st>>>(dev_timed_out, dev_cycles);
  return cudaGetLastError();
}

int fused32_tile_x() { return TX; }
int fused32_tile_y() { return TY; }

}  // namespace jz
