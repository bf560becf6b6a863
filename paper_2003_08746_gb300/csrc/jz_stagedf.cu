// Pair form of the FP64 stage: the work of the four passes of jz_stage64.cu (nodal, viscous,
// faces, update; Algorithm 2's inviscid flux, dissipation, viscous flux, RHS and
// Update(Cons, alpha_l)) in two kernels, with every flux, dissipation and SGS operation in
// double-float arithmetic (jz_df.cuh: pairs of FP32 numbers, ~48 significant bits) and the stage
// combination Q^n - alpha dt RHS in FP64.  The state stays FP64; the flux kernel reads it once and
// leaves a double-float copy for the dissipation; the fields it hands on are double-float pairs
// (float2) in the FP64 form's work arrays (same size); the metrics are a double-float copy made
// when the solver is created.  The second kernel forms the dissipative face fluxes, sums them and
// the flux differences into the RHS of each node, and updates the state.
//
// The adjoint of a pair-form solver regenerates the primitives, spectral radii and sensors of a
// stage with the nodal and sensor passes below, on 3-D launches (64 x 4 threads per block along i
// and j, one block row per k), so that no pass divides a flat index.
#include <atomic>

#include "jz_dfconsts.cuh"

namespace jz {
namespace {

constexpr int BX = 64, BY = 4;

// node of a 3-D launch over the box [i0, i0 + ei) x [j0, j0 + ej) x [k0, k0 + ek)
__device__ __forceinline__ bool node3(int i0, int j0, int k0, int ei, int ej, int& i, int& j, int& k) {
  const int x = blockIdx.x * BX + threadIdx.x, y = blockIdx.y * BY + threadIdx.y;
  if (x >= ei || y >= ej) return false;
  i = i0 + x;
  j = j0 + y;
  k = k0 + (int)blockIdx.z;
  return true;
}

__device__ __forceinline__ bool advanced(const Dims& d, int i, int j) {
  return d.topo != JZ_TOPO_JET || (i >= 1 && i <= d.ni - 2 && j >= 1 && j <= d.nj - 2);
}


// Every padded node: primitives, Sutherland mu, spectral radii and their anisotropic scaling, the
// double-float copy of Q.  Five blocks per SM (48 registers): the pass is bound by DRAM traffic and
// gains from the extra warps (11.3 against 12.8 ms per launch on 1000 x 400 x 500).
__global__ void __launch_bounds__(BX* BY, 5) k_nodal_df(Dims d, ConstsDF c, DFMetrics M, Work64 w, State q,
                                                     QDF qdf) {
  int i, j, k;
  if (!node3(-kG, -kG, -kG, d.ni + 2 * kG, d.nj + 2 * kG, i, j, k)) return;
  const long long p = pidx(d, i, j, k);
  const dfl rho = df_of(q.q[0][p]), m1 = df_of(q.q[1][p]), m2 = df_of(q.q[2][p]), m3 = df_of(q.q[3][p]),
            e = df_of(q.q[4][p]);
  st(qdf.q[0], p, rho); st(qdf.q[1], p, m1); st(qdf.q[2], p, m2); st(qdf.q[3], p, m3); st(qdf.q[4], p, e);
  const dfl ir = df_rcp(rho);
  const dfl u = df_mul(m1, ir), v = df_mul(m2, ir), ww = df_mul(m3, ir);
  const dfl ke = df_fma(m3, ww, df_fma(m2, v, df_mul(m1, u)));            // rho |u|^2
  const dfl pr = df_sub(df_mul(e, c.gm1), df_mul(ke, c.gm1_half));    // (gamma-1)(e - rho|u|^2/2)
  const dfl T = df_mul(df_mul(pr, c.gamma), ir);
  const dfl a = df_sqrt(T);
  // Sutherland, eq. (sutherland), with T_inf = 1
  const dfl mu = df_mul(df_mul(c.mu_sut, df_mul(T, a)), df_rcp(df_add(T, c.S_hat)));
  st(w.u, p, u); st(w.v, p, v); st(w.w, p, ww); st(w.T, p, T); st(w.p, p, pr); st(w.mu, p, mu);
  dfl lam[3];
  for (int dir = 0; dir < 3; ++dir) {
    const dfl sx = df_load(M.S[3 * dir], p), sy = df_load(M.S[3 * dir + 1], p), sz = df_load(M.S[3 * dir + 2], p);
    const dfl U = df_fma(sz, ww, df_fma(sy, v, df_mul(sx, u)));
    lam[dir] = df_fma(a, df_load(M.Smag[dir], p), df_abs(U));
  }
  dfl Lam[3];
  aniso_df(c, lam, Lam);
  st(w.Lam[0], p, Lam[0]); st(w.Lam[1], p, Lam[1]); st(w.Lam[2], p, Lam[2]);
}

// Pressure sensors |p+ - 2p + p-| / (p+ + 2p + p-) of the nodes within one layer of the real region,
// from the nodal pass's pressures: with that pass, what the adjoint's transposed kernels read of a
// stage (they form the gradients and stresses again themselves).
__device__ __forceinline__ dfl sensor_df(dfl pc, dfl pm, dfl pp) {
  const dfl pc2 = df_scale(pc, 2.f), sum = df_add_l(pp, pm);
  return df_n(df_mul_l(df_abs(df_n(df_sub_l(sum, pc2))), df_rcp(df_n(df_add_l(sum, pc2)))));
}
__global__ void __launch_bounds__(BX* BY) k_sensor_df(Dims d, Work64 w) {
  int i, j, k;
  if (!node3(-1, -1, -1, d.ni + 2, d.nj + 2, i, j, k)) return;
  const long long p = pidx(d, i, j, k);
  const long long s[3] = {1, d.sj, d.sk};
  const dfl pc = ld(w.p, p);
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) st(w.nu[dir], p, sensor_df(pc, ld(w.p, p - s[dir]), ld(w.p, p + s[dir])));
}

// Fluxes of a stage: primitives, Sutherland's viscosity, spectral radii and their anisotropic scaling,
// gradients by the chain rule, Smagorinsky eddy viscosity, stresses and heat flux, the transformed
// fluxes H^dir = E^dir - S^dir_j F_j and the pressure sensors of the nodes within one layer of the
// real region, and the pair copy of Q on every padded node; at stage 1 also the CFL rate of Q^n
// (block max, one atomic per block).  A block of VY - 2 warps marches along k; per plane every thread
// forms u, v, w, T, p of its node into shared memory (three planes in turn; the first and the last
// warp also of the tile's halo rows), and 30 x (VY - 2) nodes form their fluxes from the neighbours
// there, so the primitives and the viscosity never reach HBM (360 bytes per node against 568 for a
// nodal and a viscous pass).
// The momentum and energy fluxes are contracted as H_m = m_m U + S_j P_jm, P = p I - tau, and
// H_e = e U + S_j (u_m P_jm - k dT/dx_j).
// FP32 issue bounds it: 9.5 ms per launch on 512 x 512 x 360 (the two passes before: 11.4) with 8 rows
// at three blocks per SM (80 registers); at four (64, spills) 10% slower, at two (128) 12%; 14 rows at
// two the same, but slower on small grids.  Warps for the halo rows that then idle through the fluxes:
// 5% slower.  Split arrivals instead of a barrier per plane (warps drifting by a plane): 12%.
// Sums and products inside a chain are unnormalized pairs (every pair normalized: 6% slower); U, H, the
// sensors, what seeds a root or reciprocal, and in the dissipation the difference over a face (where
// the leading parts cancel) are normalized.  The residual's error against 64 bits: 9.6e-13 on a
// 333 x 177 x 90 jet, 1.1e-13 on 40 x 20 x 16; with every pair normalized but face sums of H instead of
// differences 1.1e-12 and 1.2e-13, without the two last normalizations 1.07e-12 and 1.2e-13 (and 0.6% faster).
constexpr int VX = 32, VY = 10;      // nodes of the tile with its one-node halo

// Element of a field at a 32-bit byte offset (every field of a pair solver is below 4 GB: its 632
// bytes per padded node reach the GPU's memory first): the address is a uniform base plus one
// register, and the offsets of a node's neighbours are shared by all fields.
__device__ __forceinline__ dfl ldo(const float2* f, unsigned off) {
  const float2 v = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(f) + off);
  return df_make(v.x, v.y);
}
__device__ __forceinline__ double ldo(const double* f, unsigned off) {
  return *reinterpret_cast<const double*>(reinterpret_cast<const char*>(f) + off);
}
__device__ __forceinline__ void sto(float2* f, unsigned off, dfl v) {
  *reinterpret_cast<float2*>(reinterpret_cast<char*>(f) + off) = make_float2(v.hi, v.lo);
}
inline cudaError_t offsets_fit(const Dims& d) { return d.Np < (1LL << 29) ? cudaSuccess : cudaErrorInvalidValue; }

struct StageArgs {
  Dims d;
  ConstsDF c;
  const float2* S[9];
  const float2* Smag[3];
  const float2* invV;
  const float2* Delta;
  const double* q[5];
  float2* qdf[5];
  float2* H[3][5];
  float2* nu[3];
  float2* Lam[3];
  double* rate_max;      // non-null: also the CFL rate of q over the advanced nodes
  int kchunk;
  unsigned nbx;
};

struct PlaneDF {
  float2 f[5][VY][VX];   // u, v, w, T, p
};
__device__ __forceinline__ dfl sm(const PlaneDF& P, int n, int y, int x) {
  const float2 t = P.f[n][y][x];
  return df_make(t.x, t.y);
}

__global__ void __launch_bounds__(VX*(VY - 2), 3) k_flux_df(const __grid_constant__ StageArgs A) {
  __shared__ PlaneDF pl[3];
  const Dims& d = A.d;
  const ConstsDF& c = A.c;
  const int x = threadIdx.x, y = threadIdx.y + 1;           // column and row of the tile
  const unsigned by = blockIdx.x / A.nbx, bx = blockIdx.x - by * A.nbx;
  const int i = (int)bx * (VX - 2) - 2 + x, j0 = (int)by * (VY - 2) - 2, j = j0 + y;
  const int k0 = (int)blockIdx.y * A.kchunk - 1, k1 = min(k0 + A.kchunk, d.nk + 1);   // planes [k0, k1) of -1 .. nk
  const bool out = x > 0 && x < VX - 1 && i <= d.ni && j <= d.nj;   // a node this block forms the fluxes of
  // the halo row whose primitives the first and the last warp form beside their own
  const int extra = y == 1 ? 0 : (y == VY - 2 ? VY - 1 : -1);
  double rate = 0.0;
  const unsigned sk = (unsigned)d.sk * 8u;                  // bytes
  const unsigned sj = (unsigned)d.sj * 8u;
  unsigned p = (unsigned)pidx(d, i, j, k0) * 8u;
  // the thread's node in tile row `row` of a plane: Q at offset pn, and from it the primitives into a slot and the
  // pair copy of Q (written for the block's own nodes and the outermost ghosts)
  auto load_row = [&](unsigned pn, double q[5]) {
#pragma unroll
    for (int m = 0; m < 5; ++m) q[m] = ldo(A.q[m], pn);
  };
  auto primitives = [&](const double q[5], unsigned pn, int row, int kp, PlaneDF& P) {
    const int jr = j0 + row;
    const dfl rho = df_of(q[0]), m1 = df_of(q[1]), m2 = df_of(q[2]), m3 = df_of(q[3]), e = df_of(q[4]);
    if ((x > 0 || i == -2) && (x < VX - 1 || i == d.ni + 1) && (row > 0 || jr == -2) && (row < VY - 1 || jr == d.nj + 1) &&
        ((kp >= k0 && kp < k1) || kp == -2 || kp == d.nk + 1)) {
      sto(A.qdf[0], pn, rho);
      sto(A.qdf[1], pn, m1);
      sto(A.qdf[2], pn, m2);
      sto(A.qdf[3], pn, m3);
      sto(A.qdf[4], pn, e);
    }
    const dfl ir = df_rcp(rho);
    const dfl u = df_mul(m1, ir), v = df_mul(m2, ir), w = df_mul(m3, ir);
    const dfl ke = df_fma_l(m3, w, df_fma_l(m2, v, df_mul_l(m1, u)));                   // rho |u|^2
    const dfl pr = df_n(df_sub_l(df_mul_l(e, c.gm1), df_mul_l(ke, c.gm1_half)));        // (gamma-1)(e - rho|u|^2/2)
    const dfl T = df_n(df_mul_l(df_mul_l(pr, c.gamma), ir));
    P.f[0][row][x] = make_float2(u.hi, u.lo);
    P.f[1][row][x] = make_float2(v.hi, v.lo);
    P.f[2][row][x] = make_float2(w.hi, w.lo);
    P.f[3][row][x] = make_float2(T.hi, T.lo);
    P.f[4][row][x] = make_float2(pr.hi, pr.lo);
  };
  int s0 = 0, s1 = 1, s2 = 2;                               // slots of planes k - 1, k, k + 1
  // the first two planes together: their loads and their chains overlap (a block of a small grid
  // marches one plane: the launch takes 1.3 us less on 32 x 24 x 16)
#pragma unroll 1
  for (int row = y;; row = extra) {
    if (i <= d.ni + 1 && j0 + row <= d.nj + 1) {           // i, j >= -2 by construction
      const unsigned pn = p + (unsigned)(row - y) * sj;
      double qa[5], qb[5];
      load_row(pn - sk, qa);
      load_row(pn, qb);
      primitives(qa, pn - sk, row, k0 - 1, pl[s0]);
      primitives(qb, pn, row, k0, pl[s1]);
    }
    if (row != y || extra < 0) break;
  }
  for (int k = k0; k < k1; ++k, p += sk) {
    dfl S[3][3] = {}, Smag[3] = {}, iV = {}, Delta = {};
    if (out) {
      // the metrics of plane k, requested before the primitives of plane k + 1 that hide their latency (a load
      // that follows a store to another array waits for it: |S| read beside its use cost 2.7%)
#pragma unroll
      for (int dir = 0; dir < 3; ++dir) {
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) S[dir][cc] = ldo(A.S[3 * dir + cc], p);
        Smag[dir] = ldo(A.Smag[dir], p);
      }
      iV = ldo(A.invV, p);
      Delta = ldo(A.Delta, p);
    }
    // primitives of plane k + 1 in the thread's row and, at the tile's edge, in the halo row
#pragma unroll 1
    for (int row = y;; row = extra) {
      if (i <= d.ni + 1 && j0 + row <= d.nj + 1) {
        const unsigned pn = p + sk + (unsigned)(row - y) * sj;
        double q[5];
        load_row(pn, q);
        primitives(q, pn, row, k + 1, pl[s2]);
      }
      if (row != y || extra < 0) break;
    }
    {
      // plane k + 1 before its neighbours read it one iteration later, and every thread done with
      // plane k - 1 as neighbours; planes k - 1 and k + 1 are read by their own column only
      __syncthreads();
      if (out) {
        const PlaneDF &Pm = pl[s0], &P0 = pl[s1], &Pp = pl[s2];
        // G[n][j] = sum_dir S^dir_j (f_n[+dir] - f_n[-dir]); the gradient is h G with h = 1/(2V)
        dfl G[4][3];
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const dfl dx = df_sub_l(sm(P0, n, y, x + 1), sm(P0, n, y, x - 1));
          const dfl dy = df_sub_l(sm(P0, n, y + 1, x), sm(P0, n, y - 1, x));
          const dfl dz = df_sub_l(sm(Pp, n, y, x), sm(Pm, n, y, x));
#pragma unroll
          for (int jj = 0; jj < 3; ++jj)
            G[n][jj] = df_fma_l(S[2][jj], dz, df_fma_l(S[1][jj], dy, df_mul_l(S[0][jj], dx)));
        }
        const dfl h = df_scale(iV, 0.5f);
        // |S| = h sqrt(2 sum G_ii^2 + sum_{i<j} A_ij^2), A_ij = G_ij + G_ji
        const dfl A12 = df_add_l(G[0][1], G[1][0]), A13 = df_add_l(G[0][2], G[2][0]), A23 = df_add_l(G[1][2], G[2][1]);
        const dfl Gd = df_add_l(df_add_l(G[0][0], G[1][1]), G[2][2]);
        const dfl DG = df_fma_l(G[2][2], G[2][2], df_fma_l(G[1][1], G[1][1], df_mul_l(G[0][0], G[0][0])));
        const dfl AA = df_fma_l(A23, A23, df_fma_l(A13, A13, df_mul_l(A12, A12)));
        const dfl csd = df_mul_l(Delta, c.C_s);
        const dfl rho = ldo(A.qdf[0], p);
        // Smagorinsky eddy viscosity rho (C_s Delta)^2 |S|
        const dfl mu_sgs = df_n(df_mul_l(df_mul_l(rho, df_mul_l(csd, csd)),
                                         df_mul_l(h, df_sqrt(df_n(df_add_l(df_scale(DG, 2.f), AA))))));
        // Sutherland, eq. (sutherland), with T_inf = 1
        const dfl T = sm(P0, 3, y, x), a = df_sqrt(T);
        const dfl mu = df_mul_l(df_mul_l(c.mu_sut, df_mul_l(T, a)), df_rcp(df_n(df_add_l(T, c.S_hat))));
        const dfl mt = df_add_l(mu, mu_sgs);
        const dfl mV = df_mul_l(mt, iV), mh = df_neg(df_mul_l(mt, h));
        const dfl kh = df_neg(df_mul_l(df_add_l(df_mul_l(mu, c.k_lam), df_mul_l(mu_sgs, c.k_sgs)), h));  // -k_eff h
        const dfl d3 = df_mul_l(Gd, c.third);                                                              // Gd / 3
        // P_jm = p delta_jm - tau_jm (symmetric)
        const dfl pc = sm(P0, 4, y, x);
        const dfl P11 = df_fma_l(mV, df_sub_l(d3, G[0][0]), pc), P22 = df_fma_l(mV, df_sub_l(d3, G[1][1]), pc),
                  P33 = df_fma_l(mV, df_sub_l(d3, G[2][2]), pc);
        const dfl P12 = df_mul_l(mh, A12), P13 = df_mul_l(mh, A13), P23 = df_mul_l(mh, A23);
        const dfl u = sm(P0, 0, y, x), v = sm(P0, 1, y, x), w = sm(P0, 2, y, x);
        // X_j = sum_m u_m P_jm - k dT/dx_j: what remains of the energy flux beside e U
        const dfl X1 = df_fma_l(kh, G[3][0], df_fma_l(w, P13, df_fma_l(v, P12, df_mul_l(u, P11))));
        const dfl X2 = df_fma_l(kh, G[3][1], df_fma_l(w, P23, df_fma_l(v, P22, df_mul_l(u, P12))));
        const dfl X3 = df_fma_l(kh, G[3][2], df_fma_l(w, P33, df_fma_l(v, P23, df_mul_l(u, P13))));
        const dfl m1 = ldo(A.qdf[1], p), m2 = ldo(A.qdf[2], p), m3 = ldo(A.qdf[3], p),
                  e = ldo(A.qdf[4], p);
        dfl lam[3];
#pragma unroll
        for (int dir = 0; dir < 3; ++dir) {
          const dfl sx = S[dir][0], sy = S[dir][1], sz = S[dir][2];
          const dfl U = df_n(df_fma_l(sz, w, df_fma_l(sy, v, df_mul_l(sx, u))));
          lam[dir] = df_fma(a, Smag[dir], df_abs(U));
          // H^dir = [rho U, m_i U + S_j P_ji, e U + S_j X_j]
          auto flux = [&](dfl q, dfl f1, dfl f2, dfl f3) {
            return df_n(df_fma_l(q, U, df_fma_l(sz, f3, df_fma_l(sy, f2, df_mul_l(sx, f1)))));
          };
          sto(A.H[dir][0], p, df_mul(rho, U));
          sto(A.H[dir][1], p, flux(m1, P11, P12, P13));
          sto(A.H[dir][2], p, flux(m2, P12, P22, P23));
          sto(A.H[dir][3], p, flux(m3, P13, P23, P33));
          sto(A.H[dir][4], p, flux(e, X1, X2, X3));
        }
        if (A.rate_max && i >= 0 && i < d.ni && j >= 0 && j < d.nj && k >= 0 && k < d.nk && advanced(d, i, j))
          rate = fmax(rate, df_to_f64(df_mul(df_add(df_add(lam[0], lam[1]), lam[2]), iV)));
        dfl L[3];
        aniso_df(c, lam, L);
        sto(A.nu[0], p, sensor_df(pc, sm(P0, 4, y, x - 1), sm(P0, 4, y, x + 1)));
        sto(A.nu[1], p, sensor_df(pc, sm(P0, 4, y - 1, x), sm(P0, 4, y + 1, x)));
        sto(A.nu[2], p, sensor_df(pc, sm(Pm, 4, y, x), sm(Pp, 4, y, x)));
#pragma unroll
        for (int dir = 0; dir < 3; ++dir) sto(A.Lam[dir], p, L[dir]);
      }
    }
    const int t = s0;
    s0 = s1;
    s1 = s2;
    s2 = t;
  }
  if (A.rate_max) {
    // block max -> one atomic per block (non-negative doubles order like their bits)
    __shared__ double redm[VY - 2];
    for (int o = 16; o > 0; o >>= 1) rate = fmax(rate, __shfl_xor_sync(0xffffffffu, rate, o));
    if (x == 0) redm[y - 1] = rate;
    __syncthreads();
    if (x == 0 && y == 1) {
      for (int n = 1; n < VY - 2; ++n) rate = fmax(rate, redm[n]);
      if (rate > 0.0)
        atomicMax(reinterpret_cast<unsigned long long*>(A.rate_max), (unsigned long long)__double_as_longlong(rate));
    }
  }
}

// C + D: Turkel-Vatsa dissipation, RHS and stage update in one kernel.  Per node and variable
//   2 V RHS = sum_dir [ H(n+1) - H(n-1) - (D(n+1/2) - D(n-1/2)) ],  D = 2 d,
// in double-float, then Q^n - alpha dt RHS in FP64 (mode 0; mode 2: a periodic box, with its ghosts) or
// the RHS itself (mode 1).  Neither the faces nor their sums leave the SM.
// 2 d = a32 d1 - b2 e3 on the face between p and p + sd, with d1 and e3 the differences of Q over the
// face (one and three spacings): Ls = 2 L_f, b2 = Ls eps4, a32 = 3 b2 + Ls eps2, as (a32, b2).
__device__ __forceinline__ float4 face_coef(const ConstsDF& c, const float2* nu, const float2* Lam, long long p,
                                            long long sd) {
  const dfl eps2 = df_mul(df_max(df_load(nu, p), df_load(nu, p + sd)), c.kappa2);
  const dfl k4 = df_sub(c.kappa4, eps2);
  const dfl eps4 = df_gt0(k4) ? k4 : df_make(0.f, 0.f);
  const dfl Ls = df_add(df_load(Lam, p), df_load(Lam, p + sd));
  const dfl b2 = df_mul(Ls, eps4);
  const dfl a32 = df_fma(Ls, eps2, df_mul_f(b2, 3.f));
  return make_float4(a32.hi, a32.lo, b2.hi, b2.lo);
}
__device__ __forceinline__ dfl face_diss(float4 k, dfl qm, dfl q0, dfl q1, dfl q2) {
  const dfl d1 = df_n(df_sub_l(q1, q0)), e3 = df_sub_l(q2, qm);
  return df_fma_l(df_make(-k.z, -k.w), e3, df_mul_l(df_make(k.x, k.y), d1));
}

struct FacesArgs {
  Dims d;
  ConstsDF c;
  const float2* nu[3];
  const float2* Lam[3];
  const float2* H[3][5];
  const float2* Q[5];
  const double* invV;
  const double* qin[5];
  const double* qn[5];
  double* qout[5];
  Scalars* sc;
  double alpha;
  int last;              // t += dt (mode 2)
  double* rhs;           // [5][N] (mode 1)
  double* res_sum;       // non-null: add the sum of RHS_rho^2
  int kchunk;
  unsigned nbx;          // blocks along i (blockIdx.x = by * nbx + bx)
};


// A block of 32 x FY nodes marches along k over a chunk of planes; a thread forms the faces i + 1/2,
// j + 1/2, k + 1/2 of its node for the five variables, takes i - 1/2 from the lane below it (shuffle),
// j - 1/2 from the row below it (shared memory) and k - 1/2 from its own previous plane.  Column 0
// and row 0 of the block are that halo (31 x (FY - 1) nodes updated per plane).  The fluxes enter as
// the difference of their neighbours, not as face sums: fewer operations and a smaller rounding
// error (H(n+1) - H(n-1) cancels before anything is rounded), and the dissipation, small beside the
// flux, is summed in unnormalized pairs.
// Issue-bound (62%) with load latency behind it: 7.6 ms per launch on 512 x 512 x 360 with 32 x 8
// blocks at four per SM (when it took 8.1: 8.3 for 32 x 16 at two, 8.1 for 32 x 12 at three; 9.2 with face sums).
// One variable per thread (five times the threads, coefficients through shared memory) took 16.9.
// PER blocks per SM: 4, or 2 where every plane of every tile is resident at two: load latency alone is left
// then, and 108 to 119 registers (of the 128 that two blocks leave) hold more loads in flight than 64 (32 x 24 x 16: 0.9 us per launch less,
// ten steps 0.98 -> 0.92 ms; with 360 blocks on 304 places 70 x 40 x 20 would take 18.9 us instead of 15.6).
constexpr int FX = 32, FY = 8;
template <int MODE, int PER>
__global__ void __launch_bounds__(FX* FY, PER) k_faces_update_df(const __grid_constant__ FacesArgs A) {
  const Dims& d = A.d;
  const ConstsDF& c = A.c;
  __shared__ float2 g1s[2][5][FY][FX];   // faces j + 1/2 of the plane, two planes in turn
  __shared__ float2 g2s[5][FY][FX];      // each thread's face k - 1/2
  const int x = threadIdx.x, y = threadIdx.y;
  const unsigned by = blockIdx.x / A.nbx, bx = blockIdx.x - by * A.nbx;
  const int i = (int)bx * (FX - 1) - 1 + x, j = (int)by * (FY - 1) - 1 + y;
  const int k0 = (int)blockIdx.y * A.kchunk, k1 = min(k0 + A.kchunk, d.nk);
  const bool inside = i <= d.ni - 1 && j <= d.nj - 1;
  const bool need0 = inside && y > 0, need1 = inside && x > 0, node = need0 && x > 0;
  const bool adv = advanced(d, i, j);
  const long long sj = d.sj, sk = d.sk;
  long long p = pidx(d, i, j, k0);
  const double adt = MODE != 1 ? A.alpha * A.sc->dt : 0.0;
  double r2 = 0.0;
  if (node) {
    const float4 cf = face_coef(c, A.nu[2], A.Lam[2], p - sk, sk);
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      const float2* Q = A.Q[m] + p;
      const dfl D = face_diss(cf, df_load(Q, -2 * sk), df_load(Q, -sk), df_load(Q, 0), df_load(Q, sk));
      g2s[m][y][x] = make_float2(D.hi, D.lo);
    }
  }
  for (int k = k0; k < k1; ++k, p += sk) {
    const int b = k & 1;
    dfl R[5];
    float4 cf = make_float4(0.f, 0.f, 0.f, 0.f);
    if (need0) cf = face_coef(c, A.nu[0], A.Lam[0], p, 1);
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      dfl D = df_make(0.f, 0.f);
      if (need0) {
        const float2* Q = A.Q[m] + p;
        D = face_diss(cf, df_load(Q, -1), df_load(Q, 0), df_load(Q, 1), df_load(Q, 2 * 1));
      }
      const float mh = __shfl_up_sync(0xffffffffu, D.hi, 1), ml = __shfl_up_sync(0xffffffffu, D.lo, 1);
      R[m] = df_sub_l(df_make(mh, ml), D);
    }
    if (need1) {
      cf = face_coef(c, A.nu[1], A.Lam[1], p, sj);
#pragma unroll
      for (int m = 0; m < 5; ++m) {
        const float2* Q = A.Q[m] + p;
        const dfl D = face_diss(cf, df_load(Q, -sj), df_load(Q, 0), df_load(Q, sj), df_load(Q, 2 * sj));
        g1s[b][m][y][x] = make_float2(D.hi, D.lo);
      }
    }
    if (node) {
      cf = face_coef(c, A.nu[2], A.Lam[2], p, sk);
#pragma unroll
      for (int m = 0; m < 5; ++m) {
        const float2* Q = A.Q[m] + p;
        const dfl D = face_diss(cf, df_load(Q, -sk), df_load(Q, 0), df_load(Q, sk), df_load(Q, 2 * sk));
        const float2 o = g2s[m][y][x];
        g2s[m][y][x] = make_float2(D.hi, D.lo);
        const float2 *H0 = A.H[0][m] + p, *H1 = A.H[1][m] + p, *H2 = A.H[2][m] + p;
        R[m] = df_add_l(R[m], df_sub_l(df_load(H0, 1), df_load(H0, -1)));
        R[m] = df_add_l(R[m], df_sub_l(df_sub_l(df_load(H2, sk), df_load(H2, -sk)), df_sub_l(D, df_make(o.x, o.y))));
        R[m] = df_add_l(R[m], df_sub_l(df_load(H1, sj), df_load(H1, -sj)));
      }
    }
    __syncthreads();
    if (node) {
      // all of Q^n before the first store (behind it each load would wait for the one before: 5% of the
      // kernel)
      double qn[5] = {};
      if (MODE != 1) {
#pragma unroll
        for (int m = 0; m < 5; ++m) qn[m] = A.qn[m][p];
      }
      const double hV = 0.5 * A.invV[p];
#pragma unroll
      for (int m = 0; m < 5; ++m) {
        const float2 t1 = g1s[b][m][y][x], t0 = g1s[b][m][y - 1][x];
        const double R64 = df_to_f64(df_sub_l(R[m], df_sub_l(df_make(t1.x, t1.y), df_make(t0.x, t0.y))));
        if (MODE != 1) {
          A.qout[m][p] = adv ? fma(-(adt * hV), R64, qn[m]) : A.qin[m][p];
        } else {
          const long long N = (long long)d.ni * d.nj * d.nk, t = ((long long)k * d.nj + j) * d.ni + i;
          A.rhs[m * N + t] = adv ? R64 * hV : 0.0;
        }
        if (adv && m == 0) {
          const double r0 = R64 * hV;
          r2 += r0 * r0;
        }
      }
      // (values read back from what this thread has just written: registers for them would cost
      // every node)
      if (MODE == 2 && has_images(d, i, j, k)) {
        double v[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) v[m] = A.qout[m][p];
        for_images(d, i, j, k, [&](long long g) {
#pragma unroll
          for (int m = 0; m < 5; ++m) A.qout[m][g] = v[m];
        });
      }
    }
  }
  if (MODE == 2 && A.last && blockIdx.x == 0 && blockIdx.y == 0 && x == 0 && y == 0) A.sc->t = A.sc->t + A.sc->dt;
  if (A.res_sum) {
    __shared__ double red[FY];
    for (int o = 16; o > 0; o >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, o);
    if (x == 0) red[y] = r2;
    __syncthreads();
    if (x == 0 && y == 0) {
      double t = 0.0;
      for (int q = 0; q < FY; ++q) t += red[q];
      atomicAdd(A.res_sum, t);
    }
  }
}

// FP64 metrics -> double-float copies (every padded node).
__global__ void k_metrics_df(Dims d, GridDev g, DFMetrics M) {
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= d.Np) return;
  for (int c = 0; c < 9; ++c) df_store(M.S[c], p, df_of(g.S[c][p]));
  for (int c = 0; c < 3; ++c) df_store(M.Smag[c], p, df_of(g.Smag[c][p]));
  df_store(M.invV, p, df_of(g.invV[p]));
  df_store(M.Delta, p, df_of(g.Delta[p]));
}


dim3 grid3(int ei, int ej, int ek) { return dim3((ei + BX - 1) / BX, (ej + BY - 1) / BY, ek); }

}  // namespace

cudaError_t metrics_to_df(const Dims& d, const GridDev& g, const DFMetrics& M, cudaStream_t st) {
  k_metrics_df<<<blocks_for(d.Np, 256), 256, 0, st>>>(d, g, M);
  return cudaGetLastError();
}

cudaError_t nodal_df(const Dims& d, const Consts& c, const DFMetrics& M, const Work64& w, const QDF& qdf,
                     const State& qin, cudaStream_t st) {
  k_nodal_df<<<grid3(d.ni + 2 * kG, d.nj + 2 * kG, d.nk + 2 * kG), dim3(BX, BY), 0, st>>>(d, make_cdf(c), M, w, qin,
                                                                                          qdf);
  return cudaGetLastError();
}

cudaError_t sensor_df_pass(const Dims& d, const Work64& w, cudaStream_t st) {
  k_sensor_df<<<grid3(d.ni + 2, d.nj + 2, d.nk + 2), dim3(BX, BY), 0, st>>>(d, w);
  return cudaGetLastError();
}

// Resident blocks of a kernel on the current device, asked for once per device (by any host thread: all
// store the same value).
using SlotCache = std::atomic<int>[64];
template <class K>
int resident_blocks(K kernel, int threads, SlotCache& cache) {
  int dev = 0, sms = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 304;
  int n = cache[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, 0) != cudaSuccess || per < 1)
      return 304;
    n = sms * per;
    cache[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

// Planes per block of the marching kernels, from r = planes of all tiles per resident block.  Fitted to
// sweeps of 1 .. 45 planes over eight jets from 64 x 48 x 32 to 512 x 512 x 360 (each choice within a few per cent
// of its sweep's best).  Flux kernel: two planes are primed per block, so long blocks, but three
// waves of them; small grids take the blocks that just fill the device (96 x 64 x 32: 42 us with 3 planes,
// 48 with 1, 58 with 8).  Faces kernel: one face is primed per block and its loads want many blocks
// out of step: twenty waves where that leaves three planes or more (512 x 256 x 128: 1.48 ms with 6, 1.64
// with 32), then three planes, two, one (128 x 96 x 64: 104 us with 2, 132 with 6).
int flux_chunk(double r) {
  if (r <= 3.0) return r <= 1.0 ? 1 : (r <= 2.0 ? 2 : 3);
  return r < 9.0 ? 3 : (r < 96.0 ? (int)(r / 3.0) : 32);
}
int faces_chunk(double r) {
  if (r >= 60.0) return r < 640.0 ? (int)(r / 20.0) : 32;
  return r >= 13.5 ? 3 : (r >= 6.0 ? 2 : 1);
}

cudaError_t flux_df(const Dims& d, const Consts& c, const DFMetrics& M, const Work64& w, const QDF& qdf,
                    const State& qin, Scalars* sc, cudaStream_t st, int want_rate) {
  const cudaError_t fit = offsets_fit(d);
  if (fit != cudaSuccess) return fit;
  StageArgs A;
  A.d = d;
  A.c = make_cdf(c);
  auto f2 = [](double* x) { return reinterpret_cast<float2*>(x); };
  for (int n = 0; n < 9; ++n) A.S[n] = M.S[n];
  for (int dir = 0; dir < 3; ++dir) {
    A.Smag[dir] = M.Smag[dir];
    A.nu[dir] = f2(w.nu[dir]);
    A.Lam[dir] = f2(w.Lam[dir]);
    for (int m = 0; m < 5; ++m) A.H[dir][m] = f2(w.H[dir][m]);
  }
  A.invV = M.invV;
  A.Delta = M.Delta;
  for (int m = 0; m < 5; ++m) {
    A.q[m] = qin.q[m];
    A.qdf[m] = f2(qdf.q[m]);
  }
  A.rate_max = want_rate ? &sc->rate_max : nullptr;
  A.nbx = (d.ni + VX - 1) / (VX - 2);
  const long long tiles = (long long)A.nbx * ((d.nj + VY - 1) / (VY - 2));
  static SlotCache slots;
  A.kchunk = flux_chunk((double)tiles * (d.nk + 2) / resident_blocks(k_flux_df, VX * (VY - 2), slots));
  const dim3 gr((unsigned)tiles, (d.nk + 1 + A.kchunk) / A.kchunk);
  k_flux_df<<<gr, dim3(VX, VY - 2), 0, st>>>(A);
  return cudaGetLastError();
}

cudaError_t faces_update_df(const Dims& d, const Consts& c, const GridDev& g, const Work64& w, const QDF& qdf,
                            const State& qin, const State& qn, const State& qout, Scalars* sc, double alpha,
                            int want_res, double* rhs_flat, cudaStream_t st, Finish finish) {
  FacesArgs A;
  A.d = d;
  A.c = make_cdf(c);
  auto f2 = [](const double* x) { return reinterpret_cast<const float2*>(x); };
  for (int dir = 0; dir < 3; ++dir) {
    A.nu[dir] = f2(w.nu[dir]);
    A.Lam[dir] = f2(w.Lam[dir]);
    for (int m = 0; m < 5; ++m) A.H[dir][m] = f2(w.H[dir][m]);
  }
  for (int m = 0; m < 5; ++m) {
    A.Q[m] = f2(qdf.q[m]);
    A.qin[m] = qin.q[m];
    A.qn[m] = qn.q[m];
    A.qout[m] = qout.q[m];
  }
  A.invV = g.invV;
  A.sc = sc;
  A.alpha = alpha;
  A.last = finish == FINISH_STEP;
  A.rhs = rhs_flat;
  A.res_sum = want_res && !rhs_flat ? &sc->res_sum : nullptr;
  A.nbx = (d.ni + FX - 2) / (FX - 1);
  const long long tiles = (long long)A.nbx * ((d.nj + FY - 2) / (FY - 1));
  static SlotCache slots, slots2;
  const long long planes = tiles * d.nk;
  const bool small = planes <= resident_blocks(k_faces_update_df<0, 2>, FX * FY, slots2);
  A.kchunk = small ? 1 : faces_chunk((double)planes / resident_blocks(k_faces_update_df<0, 4>, FX * FY, slots));
  const dim3 gr((unsigned)tiles, (d.nk + A.kchunk - 1) / A.kchunk), blk(FX, FY);
  const int mode = rhs_flat ? 1 : finish == FINISH_NONE ? 0 : 2;
  const auto kernel = mode == 0   ? (small ? k_faces_update_df<0, 2> : k_faces_update_df<0, 4>)
                      : mode == 1 ? (small ? k_faces_update_df<1, 2> : k_faces_update_df<1, 4>)
                                  : (small ? k_faces_update_df<2, 2> : k_faces_update_df<2, 4>);
  kernel<<<gr, blk, 0, st>>>(A);
  return cudaGetLastError();
}

}  // namespace jz
