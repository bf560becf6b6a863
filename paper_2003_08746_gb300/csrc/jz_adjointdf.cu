// Transposed passes of the discrete adjoint for a pair-form solver (see jz_adjoint.cu for the
// FP64 form and the structure of the reverse sweep): the face, viscous-and-sensor and nodal
// passes in double-float arithmetic on the pair intermediates that the pair nodal and sensor
// passes regenerated (u, v, w, T, p, mu, the sensors, Lambda, the pair copies of Q and of the
// metrics).  The running adjoint lambda and Q^n's adjoint stay FP64 (as do the boundary-condition
// adjoints and the observer); the intermediate adjoint arrays the transposed passes pass to one
// another (alpha dt lambda / V, the face coefficients and sensor adjoints, the adjoints of the
// gradients, of u, mu and rho) are double-float pairs in the same arrays, so the gathers of the
// transposed nodal pass run on the FP32 pipes.  Sums and products inside a chain are unnormalized
// pairs (jz_df.cuh), normalized before they are stored or seed a root or reciprocal.
#include "jz_adjgather.cuh"
#include "jz_dfconsts.cuh"

namespace jz {
namespace {
// an element of an array that the kernel does not write: the load may move before stores to others
__device__ __forceinline__ dfl ldc(const double* f, long long p) {
  const float2 v = __ldg(reinterpret_cast<const float2*>(f) + p);
  return df_make(v.x, v.y);
}

// Node of a launch over the box [o, o + ei) x [o, o + ej) x [o, o + ek): the plane's nodes in a row
// along blockIdx.x (no lanes lost to tiles that overhang it: 64 x 4 tiles cost the 130 nodes along i
// of a 128-node grid a third), k along blockIdx.y; one 32-bit division.
__device__ __forceinline__ bool plane_node(int o, int ei, int ej, int& i, int& j, int& k) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x, y = t / (unsigned)ei;
  i = o + (int)(t - y * (unsigned)ei);
  j = o + (int)y;
  k = o + (int)blockIdx.y;
  return y < (unsigned)ej;
}
dim3 plane_grid(int ei, int ej, int ek, int tpb) { return dim3(blocks_for((long long)ei * ej, tpb), ek); }

// Adjoint of the stage update: Qn_bar += lambda (FP64), acc = -alpha dt lambda / V as a pair, on
// advanced real nodes (acc stays 0 elsewhere).
__global__ void k_adj_update_df(Dims d, GridDev g, Adj64 a, double adt) {
  int i, j, k;
  if (!plane_node(0, d.ni, d.nj, i, j, k)) return;
  const long long p = pidx(d, i, j, k);
  const bool adv = d.topo != JZ_TOPO_JET || (i >= 1 && i <= d.ni - 2 && j >= 1 && j <= d.nj - 2);
  const double f = -adt * g.invV[p];
  // (every load before the first store: behind it each would wait for the one before)
  double l[5], qb[5];
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    l[m] = a.lam[m][p];
    qb[m] = a.qnbar[m][p];
  }
#pragma unroll
  for (int m = 0; m < 5; ++m) {
    if (adv) a.qnbar[m][p] = qb[m] + l[m];
    st(a.acc[m], p, adv ? df_of(f * l[m]) : df_from(0.f));
  }
}

// Transposed dissipation faces of the discrete adjoint (jz_adjoint.cu, k_adj_faces) for a
// pair-form solver, in double-float arithmetic on the pair copies of Q, the sensors and Lambda.
// Faces n + 1/2, n in [-1, n_dir - 1].
__global__ void k_adj_faces_df(Dims d, ConstsDF c, Work64 w, QDF qdf, Adj64 a) {
  int i, j, k;
  if (!plane_node(-1, d.ni + 1, d.nj + 1, i, j, k)) return;
  const long long p = pidx(d, i, j, k);
  const long long s[3] = {1, d.sj, d.sk};
  for (int dir = 0; dir < 3; ++dir) {
    const long long sd = s[dir];
    const dfl nu0 = ld(w.nu[dir], p), nu1 = ld(w.nu[dir], p + sd);
    const bool first = df_ge(nu0, nu1);
    const dfl eps2 = df_mul_l(c.kappa2, first ? nu0 : nu1);
    const dfl k4 = df_n(df_sub_l(c.kappa4, eps2));
    const bool pos4 = df_gt0(k4);
    const dfl eps4 = pos4 ? k4 : df_from(0.f);
    const dfl Lf = df_scale(df_add_l(ld(w.Lam[dir], p), ld(w.Lam[dir], p + sd)), 0.5f);
    dfl lf = df_from(0.f), e2b = df_from(0.f), e4b = df_from(0.f);
    for (int m = 0; m < 5; ++m) {
      const double* Q = qdf.q[m];
      const dfl q0 = ld(Q, p), q1 = ld(Q, p + sd), q2 = ld(Q, p + 2 * sd), qm = ld(Q, p - sd);
      const dfl d1 = df_sub_l(q1, q0);
      const dfl d3 = df_sub_l(df_add_l(df_sub_l(q2, df_mul_f(q1, 3.f)), df_mul_f(q0, 3.f)), qm);
      const dfl Db = df_sub_l(ld(a.acc[m], p + sd), ld(a.acc[m], p));
      lf = df_fma_l(Db, df_sub_l(df_mul_l(eps2, d1), df_mul_l(eps4, d3)), lf);
      const dfl DL = df_mul_l(Db, Lf);
      e2b = df_fma_l(DL, d1, e2b);
      e4b = df_sub_l(e4b, df_mul_l(DL, d3));
    }
    st(a.ca2[dir], p, df_n(df_mul_l(Lf, eps2)));
    st(a.ca4[dir], p, df_n(df_mul_l(Lf, eps4)));
    if (pos4) e2b = df_sub_l(e2b, e4b);
    const dfl nub = df_n(df_mul_l(c.kappa2, e2b));
    st(a.nb0[dir], p, first ? nub : df_from(0.f));
    st(a.nb1[dir], p, first ? df_from(0.f) : nub);
    st(a.lfh[dir], p, df_scale(df_n(lf), 0.5f));
  }
}

// Transposed viscous pass and pressure sensor of the discrete adjoint (jz_adjoint.cu, k_adj_visc)
// for a pair-form solver: the same reverse sweep through gradients, strain rate, eddy viscosity,
// stresses, heat flux and sensors, in double-float arithmetic on the pair intermediates the pair
// passes regenerated (u, v, w, T, p, mu, the pair copies of Q and of the metrics).  Nodes within
// one layer of the real region.
// Four 128-thread blocks per SM (128 registers); three (168) or six (80) are 3% slower.  Loads that may not
// move before the stores: 2% slower.
constexpr int kTPBV = 128;
__global__ void __launch_bounds__(kTPBV, 4) k_adj_visc_df(Dims d, ConstsDF c, DFMetrics M, Work64 w, QDF qdf, Adj64 a) {
  int i, j, k;
  if (!plane_node(-1, d.ni + 2, d.nj + 2, i, j, k)) return;
  const long long p = pidx(d, i, j, k);
  const long long s[3] = {1, d.sj, d.sk};
  // adjoint of H^dir (components 1..4 carry the viscous flux)
  dfl Hb[3][4];
  for (int dir = 0; dir < 3; ++dir)
    for (int m = 0; m < 4; ++m) Hb[dir][m] = df_scale(df_sub_l(ldc(a.acc[m + 1], p - s[dir]), ldc(a.acc[m + 1], p + s[dir])), 0.5f);
  // forward viscous quantities
  const double* f[4] = {w.u, w.v, w.w, w.T};
  dfl S[3][3];
  for (int dir = 0; dir < 3; ++dir)
    for (int cc = 0; cc < 3; ++cc) S[dir][cc] = df_load(M.S[3 * dir + cc], p);
  const dfl iV = df_load(M.invV, p);
  dfl L[4][3];
  for (int n = 0; n < 4; ++n) {
    dfl dd[3];
    for (int dir = 0; dir < 3; ++dir) dd[dir] = df_scale(df_sub_l(ldc(f[n], p + s[dir]), ldc(f[n], p - s[dir])), 0.5f);
    for (int jj = 0; jj < 3; ++jj)
      L[n][jj] = df_n(df_mul_l(iV, df_fma_l(S[2][jj], dd[2], df_fma_l(S[1][jj], dd[1], df_mul_l(S[0][jj], dd[0])))));
  }
  dfl Sij[3][3];
  for (int x = 0; x < 3; ++x)
    for (int y = 0; y < 3; ++y) Sij[x][y] = df_scale(df_add_l(L[x][y], L[y][x]), 0.5f);
  const dfl div = df_add_l(df_add_l(Sij[0][0], Sij[1][1]), Sij[2][2]);
  dfl SS = df_from(0.f);
  for (int x = 0; x < 3; ++x)
    for (int y = 0; y < 3; ++y) SS = df_fma_l(Sij[x][y], Sij[x][y], SS);
  const dfl Smod = df_sqrt(df_n(df_scale(SS, 2.f)));
  const dfl mu = ldc(w.mu, p);
  const dfl csd = df_mul_l(c.C_s, df_load(M.Delta, p));
  const dfl cs2 = df_mul_l(csd, csd);
  const dfl rho = ldc(qdf.q[0], p);
  const dfl mu_sgs = df_n(df_mul_l(df_mul_l(rho, cs2), Smod));
  const dfl mu_eff = df_add_l(mu, mu_sgs);
  const dfl k_eff = df_add_l(df_mul_l(mu, c.k_lam), df_mul_l(mu_sgs, c.k_sgs));
  const dfl d3 = df_mul_l(div, c.third);
  const dfl m2 = df_scale(mu_eff, 2.f);
  dfl dev[3][3];                                       // S_ij - delta_ij div/3
  for (int x = 0; x < 3; ++x)
    for (int y = 0; y < 3; ++y) dev[x][y] = x == y ? df_sub_l(Sij[x][y], d3) : Sij[x][y];
  const dfl vel[3] = {ldc(w.u, p), ldc(w.v, p), ldc(w.w, p)};
  // reverse: F^dir_m = S^dir_j F_j,m ; H = E - F
  dfl taub[3][3], ubd[3], keb = df_from(0.f), L3b[3];
  for (int x = 0; x < 3; ++x) {
    ubd[x] = df_from(0.f);
    L3b[x] = df_from(0.f);
    for (int y = 0; y < 3; ++y) taub[x][y] = df_from(0.f);
  }
  for (int jj = 0; jj < 3; ++jj) {
    dfl Fb[4];
    for (int m = 0; m < 4; ++m)
      Fb[m] = df_neg(df_fma_l(S[2][jj], Hb[2][m], df_fma_l(S[1][jj], Hb[1][m], df_mul_l(S[0][jj], Hb[0][m]))));
    for (int x = 0; x < 3; ++x) taub[x][jj] = df_add_l(taub[x][jj], Fb[x]);
    const dfl e = Fb[3];
    for (int x = 0; x < 3; ++x) {
      ubd[x] = df_fma_l(e, df_mul_l(m2, dev[x][jj]), ubd[x]);         // e tau_x,jj
      taub[x][jj] = df_fma_l(e, vel[x], taub[x][jj]);
    }
    keb = df_fma_l(e, L[3][jj], keb);
    L3b[jj] = df_fma_l(e, k_eff, L3b[jj]);
  }
  dfl mueb = df_from(0.f), Sijb[3][3], tr = df_from(0.f);
  for (int x = 0; x < 3; ++x)
    for (int y = 0; y < 3; ++y) {
      mueb = df_fma_l(taub[x][y], df_scale(dev[x][y], 2.f), mueb);
      Sijb[x][y] = df_mul_l(m2, taub[x][y]);
    }
  for (int x = 0; x < 3; ++x) tr = df_add_l(tr, taub[x][x]);
  const dfl divb = df_neg(df_mul_l(df_mul_l(mu_eff, df_scale(c.third, 2.f)), tr));
  for (int x = 0; x < 3; ++x) Sijb[x][x] = df_add_l(Sijb[x][x], divb);
  const dfl mub = df_add_l(df_mul_l(keb, c.k_lam), mueb);
  const dfl musb = df_add_l(df_mul_l(keb, c.k_sgs), mueb);
  const dfl rhob = df_mul_l(df_mul_l(musb, cs2), Smod);
  const dfl Smodb = df_mul_l(df_mul_l(musb, rho), cs2);
  const dfl SSb = df_gt0(Smod) ? df_mul_l(Smodb, df_rcp(Smod)) : df_from(0.f);
  for (int x = 0; x < 3; ++x)
    for (int y = 0; y < 3; ++y) Sijb[x][y] = df_fma_l(df_scale(Sij[x][y], 2.f), SSb, Sijb[x][y]);
  dfl Lb[4][3];
  for (int x = 0; x < 3; ++x)
    for (int y = 0; y < 3; ++y) Lb[x][y] = df_scale(df_add_l(Sijb[x][y], Sijb[y][x]), 0.5f);
  for (int y = 0; y < 3; ++y) Lb[3][y] = L3b[y];
  for (int n = 0; n < 4; ++n)
    for (int dir = 0; dir < 3; ++dir)
      st(a.G[n][dir], p, df_n(df_mul_l(iV, df_fma_l(S[dir][2], Lb[n][2], df_fma_l(S[dir][1], Lb[n][1], df_mul_l(S[dir][0], Lb[n][0]))))));
  for (int x = 0; x < 3; ++x) st(a.ubd[x], p, df_n(ubd[x]));
  st(a.mub, p, df_n(mub));
  st(a.rhob, p, df_n(rhob));
  // pressure sensor nu = |N| / Dn
  const dfl pc2 = df_scale(ldc(w.p, p), 2.f);
  for (int dir = 0; dir < 3; ++dir) {
    const dfl nub = df_add_l(ldc(a.nb0[dir], p), ldc(a.nb1[dir], p - s[dir]));
    const dfl sum = df_add_l(ldc(w.p, p + s[dir]), ldc(w.p, p - s[dir]));
    const dfl N = df_n(df_sub_l(sum, pc2)), Dn = df_n(df_add_l(sum, pc2));
    const dfl iD = df_rcp(Dn);
    const dfl nu = df_mul_l(df_abs(N), iD);
    const float sg = N.hi > 0.f ? 1.f : (N.hi < 0.f ? -1.f : 0.f);
    const dfl nbD = df_mul_l(nub, iD);
    st(a.cpm[dir], p, df_n(df_mul_l(nbD, df_sub_l(df_from(sg), nu))));
    st(a.c0[dir], p, df_n(df_mul_l(nbD, df_scale(df_add_l(df_from(sg), nu), -2.f))));
  }
}


// Neighbours of a padded node in the pair adjoint arrays, `off` nodes along `dir` (up to two), read by
// offset.  Beyond the padded box along i or j the offset lands in the next or previous row or plane,
// on elements that no pass writes: acc is 0 off the real nodes, the face arrays off [-1, n), the
// viscous and sensor arrays off [-1, n], and what an offset of one or two can reach from the outer
// ghosts lies outside those ranges at the other end (padding columns, i = -2, -1 or i >= n, and the
// same for j); before the first and after the last row of an array stand rows of zeros
// (jz_adjoint_step).  Along k the neighbour is tested.
struct PaddedNode {
  int p, sj, sk;
  bool m2, m1, p1, p2;             // k - 2, k - 1, k + 1, k + 2 lie in the padded box
  __device__ __forceinline__ PaddedNode(const Dims& d, int i, int j, int k)
      : p((int)pidx(d, i, j, k)), sj((int)d.sj), sk((int)d.sk), m2(k >= 0), m1(k >= -1), p1(k <= d.nk), p2(k < d.nk) {}
  __device__ __forceinline__ dfl operator()(const double* f, int dir, int off) const {
    if (dir < 2 || off == 0) return ld(f, p + off * (dir == 0 ? 1 : sj));
    const bool in = off == -2 ? m2 : (off == -1 ? m1 : (off == 1 ? p1 : p2));
    return in ? ld(f, p + off * sk) : df_from(0.f);
  }
};

// The gathers of the transposed nodal pass (as nodal_gathers, jz_adjgather.cuh) on the pair
// adjoint arrays, summed in double-float.
struct NodalGathersDF {
  dfl fb[4], pb, Eb[3][5], Lamb[3], qb[5], mub;
};
__device__ __forceinline__ void nodal_gathers_df(const Adj64& a, const PaddedNode& nb, NodalGathersDF& G) {
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    dfl v = n < 3 ? nb(a.ubd[n], 0, 0) : df_from(0.f);
#pragma unroll
    for (int dir = 0; dir < 3; ++dir)
      v = df_add_l(v, df_scale(df_sub_l(nb(a.G[n][dir], dir, -1), nb(a.G[n][dir], dir, 1)), 0.5f));
    G.fb[n] = v;
  }
  G.pb = df_from(0.f);
#pragma unroll
  for (int dir = 0; dir < 3; ++dir)
    G.pb = df_add_l(G.pb, df_add_l(df_add_l(nb(a.c0[dir], 0, 0), nb(a.cpm[dir], dir, -1)),
                               nb(a.cpm[dir], dir, 1)));
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) {
#pragma unroll
    for (int m = 0; m < 5; ++m)
      G.Eb[dir][m] = df_scale(df_sub_l(nb(a.acc[m], dir, -1), nb(a.acc[m], dir, 1)), 0.5f);
    G.Lamb[dir] = df_add_l(nb(a.lfh[dir], 0, 0), nb(a.lfh[dir], dir, -1));
  }
#pragma unroll
  for (int m = 0; m < 5; ++m) G.qb[m] = df_from(0.f);
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) {
    dfl c2[4], c4[4];              // faces n-2, n-1, n, n+1
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      c2[o] = nb(a.ca2[dir], dir, o - 2);
      c4[o] = nb(a.ca4[dir], dir, o - 2);
    }
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      const dfl am2 = nb(a.acc[m], dir, -2), am1 = nb(a.acc[m], dir, -1),
                a0 = nb(a.acc[m], 0, 0), ap1 = nb(a.acc[m], dir, 1),
                ap2 = nb(a.acc[m], dir, 2);
      const dfl D0 = df_sub_l(am1, am2), D1 = df_sub_l(a0, am1), D2 = df_sub_l(ap1, a0), D3 = df_sub_l(ap2, ap1);
      // -D0 c4(n-2) + D1 (c2(n-1) + 3 c4(n-1)) - D2 (c2(n) + 3 c4(n)) + D3 c4(n+1)
      dfl v = df_sub_l(df_mul_l(D3, c4[3]), df_mul_l(D0, c4[0]));
      v = df_fma_l(D1, df_add_l(c2[1], df_mul_f(c4[1], 3.f)), v);
      v = df_sub_l(v, df_mul_l(D2, df_add_l(c2[2], df_mul_f(c4[2], 3.f))));
      G.qb[m] = df_add_l(G.qb[m], v);
    }
  }
  G.qb[0] = df_add_l(G.qb[0], nb(a.rhob, 0, 0));
  G.mub = nb(a.mub, 0, 0);
}

// Transposed nodal pass (jz_adjoint.cu, k_adj_nodal) for a pair-form solver: the gathers, then
// the reverse of the anisotropic spectral radii, the inviscid fluxes, Sutherland's law and the
// primitives, all in double-float arithmetic (the gathers on the pair adjoint arrays).
// Every padded node.  Issue and load latency bound it at the 16 warps per SM that 128 registers
// leave (a few spilled; three blocks at 168 registers 4% slower, two at 224 20%): 0.17 ms per launch on
// 128 x 96 x 64, against 0.29 with a bounds check and 64-bit indices for each of the ~140 gathers (more
// than half of its 6770 instructions per node) and every pair normalized.
constexpr int kTPBN = 128;
__global__ void __launch_bounds__(kTPBN, 4) k_adj_nodal_df(const __grid_constant__ Dims d, const __grid_constant__ ConstsDF c,
                                                           const __grid_constant__ DFMetrics M,
                                                           const __grid_constant__ QDF qdf,
                                                           const __grid_constant__ Adj64 a) {
  int i, j, k;
  if (!plane_node(-kG, d.ni + 2 * kG, d.nj + 2 * kG, i, j, k)) return;
  const PaddedNode nb(d, i, j, k);
  const int p = nb.p;
  NodalGathersDF G;
  nodal_gathers_df(a, nb, G);
  dfl ub[3] = {G.fb[0], G.fb[1], G.fb[2]};
  dfl Tb = G.fb[3];
  dfl pb = G.pb;
  dfl qb[5];
#pragma unroll
  for (int m = 0; m < 5; ++m) qb[m] = G.qb[m];
  const dfl mub = G.mub;
  // forward nodal quantities
  dfl Q[5];
#pragma unroll
  for (int m = 0; m < 5; ++m) Q[m] = ld(qdf.q[m], p);
  const dfl rho = Q[0];
  const dfl ir = df_rcp(rho);
  const dfl u[3] = {df_mul_l(Q[1], ir), df_mul_l(Q[2], ir), df_mul_l(Q[3], ir)};
  const dfl pr = df_mul_l(c.gm1, df_sub_l(Q[4], df_scale(df_fma_l(Q[3], u[2], df_fma_l(Q[2], u[1], df_mul_l(Q[1], u[0]))), 0.5f)));
  const dfl T = df_n(df_mul_l(df_mul_l(c.gamma, pr), ir));
  const dfl aa = df_sqrt(T);
  const dfl iTS = df_rcp(df_n(df_add_l(T, c.S_hat)));
  const dfl mu = df_mul_l(df_mul_l(c.mu_sut, df_mul_l(T, aa)), iTS);
  dfl Sv[3][3], Smag[3], U[3], lam[3];
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) {
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) Sv[dir][cc] = df_load(M.S[3 * dir + cc], p);
    Smag[dir] = df_load(M.Smag[dir], p);
    U[dir] = df_n(df_fma_l(Sv[dir][2], u[2], df_fma_l(Sv[dir][1], u[1], df_mul_l(Sv[dir][0], u[0]))));
    lam[dir] = df_n(df_fma_l(aa, Smag[dir], df_abs(U[dir])));
  }
  // anisotropic scaling Lambda_d = lam_d + lo_d (hi_e + hi_f)
  const dfl Lamb[3] = {G.Lamb[0], G.Lamb[1], G.Lamb[2]};
  dfl lamb[3] = {Lamb[0], Lamb[1], Lamb[2]};
  {
    dfl lo[3], hi[3], dlo[3], dhi[3];
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) {
      if (c.sigma_is_two_thirds) {
        df_cbrt_pair(lam[dd], lo[dd], hi[dd]);                       // lam^(1/3), lam^(2/3)
        dlo[dd] = df_gt0(lo[dd]) ? df_rcp(df_mul_f(hi[dd], 3.f)) : df_from(0.f);   // d lo / d lam
        dhi[dd] = df_mul_l(df_scale(lo[dd], 2.f), dlo[dd]);          // d hi / d lam
      } else {
        // a general exponent through FP64 pow (not on the benchmark path)
        const double l = df_to_f64(lam[dd]);
        const bool pos = l > 0.0;
        const double lo64 = pos ? pow(l, 1.0 - c.sigma) : 0.0, hi64 = pos ? pow(l, c.sigma) : 0.0;
        lo[dd] = df_of(lo64);
        hi[dd] = df_of(hi64);
        dlo[dd] = df_of(pos ? (1.0 - c.sigma) * lo64 / l : 0.0);
        dhi[dd] = df_of(pos ? c.sigma * hi64 / l : 0.0);
      }
    }
    dfl lob[3], hib[3];
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) lob[dd] = hib[dd] = df_from(0.f);
    const int e1[3] = {1, 0, 0}, e2[3] = {2, 2, 1};
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) {
      lob[dd] = df_fma_l(Lamb[dd], df_add_l(hi[e1[dd]], hi[e2[dd]]), lob[dd]);
      const dfl Ll = df_mul_l(Lamb[dd], lo[dd]);
      hib[e1[dd]] = df_add_l(hib[e1[dd]], Ll);
      hib[e2[dd]] = df_add_l(hib[e2[dd]], Ll);
    }
#pragma unroll
    for (int dd = 0; dd < 3; ++dd) lamb[dd] = df_fma_l(hib[dd], dhi[dd], df_fma_l(lob[dd], dlo[dd], lamb[dd]));
  }
  dfl ab = df_from(0.f);
  const dfl h0 = df_add_l(Q[4], pr);
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) {
    const dfl E[5] = {G.Eb[dir][0], G.Eb[dir][1], G.Eb[dir][2], G.Eb[dir][3], G.Eb[dir][4]};
    const float sg = U[dir].hi > 0.f ? 1.f : (U[dir].hi < 0.f ? -1.f : 0.f);
    dfl Ub = df_mul_f(lamb[dir], sg);
    ab = df_fma_l(lamb[dir], Smag[dir], ab);
    // E = [rho U, m_i U + p S_i, (e + p) U]
    qb[0] = df_fma_l(E[0], U[dir], qb[0]);
    Ub = df_fma_l(E[0], rho, Ub);
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      qb[1 + x] = df_fma_l(E[1 + x], U[dir], qb[1 + x]);
      Ub = df_fma_l(E[1 + x], Q[1 + x], Ub);
      pb = df_fma_l(E[1 + x], Sv[dir][x], pb);
    }
    qb[4] = df_fma_l(E[4], U[dir], qb[4]);
    pb = df_fma_l(E[4], U[dir], pb);
    Ub = df_fma_l(E[4], h0, Ub);
#pragma unroll
    for (int x = 0; x < 3; ++x) ub[x] = df_fma_l(Ub, Sv[dir][x], ub[x]);
  }
  // Sutherland mu(T): d mu / dT = mu (1.5/T - 1/(T + S))
  Tb = df_fma_l(mub, df_mul_l(mu, df_sub_l(df_mul_f(df_rcp(T), 1.5f), iTS)), Tb);
  Tb = df_fma_l(ab, df_scale(df_rcp(aa), 0.5f), Tb);
  pb = df_fma_l(Tb, df_mul_l(c.gamma, ir), pb);
  qb[0] = df_sub_l(qb[0], df_mul_l(df_mul_l(Tb, T), ir));
  // reverse of u_i = m_i / rho, p = (gamma-1)(e - m.u/2)
  qb[4] = df_fma_l(c.gm1, pb, qb[4]);
  const dfl keb = df_scale(df_neg(df_mul_l(c.gm1, pb)), 0.5f);      // half the adjoint of m.u
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    qb[1 + x] = df_fma_l(keb, u[x], qb[1 + x]);
    ub[x] = df_fma_l(keb, Q[1 + x], ub[x]);
  }
  dfl sum = df_from(0.f);
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    qb[1 + x] = df_fma_l(ub[x], ir, qb[1 + x]);
    sum = df_fma_l(ub[x], u[x], sum);
  }
  qb[0] = df_sub_l(qb[0], df_mul_l(sum, ir));
#pragma unroll
  for (int m = 0; m < 5; ++m) a.lam[m][p] = df_to_f64(qb[m]);
}

}  // namespace

cudaError_t adj_update_df(const Dims& d, const GridDev& g, const Adj64& a, double adt, cudaStream_t st) {
  k_adj_update_df<<<plane_grid(d.ni, d.nj, d.nk, 256), 256, 0, st>>>(d, g, a, adt);
  return cudaGetLastError();
}

cudaError_t adj_nodal_df(const Dims& d, const Consts& c, const DFMetrics& M, const QDF& qdf, const Adj64& a,
                         cudaStream_t st) {
  if (d.Np >= (1LL << 31)) return cudaErrorInvalidValue;      // (the adjoint's arrays reach the memory long before)
  k_adj_nodal_df<<<plane_grid(d.ni + 2 * kG, d.nj + 2 * kG, d.nk + 2 * kG, kTPBN), kTPBN, 0, st>>>(d, make_cdf(c), M,
                                                                                                    qdf, a);
  return cudaGetLastError();
}

cudaError_t adj_faces_df(const Dims& d, const Consts& c, const Work64& w, const QDF& qdf, const Adj64& a,
                         cudaStream_t st) {
  k_adj_faces_df<<<plane_grid(d.ni + 1, d.nj + 1, d.nk + 1, 256), 256, 0, st>>>(d, make_cdf(c), w, qdf, a);
  return cudaGetLastError();
}

cudaError_t adj_visc_df(const Dims& d, const Consts& c, const DFMetrics& M, const Work64& w, const QDF& qdf,
                        const Adj64& a, cudaStream_t st) {
  k_adj_visc_df<<<plane_grid(d.ni + 2, d.nj + 2, d.nk + 2, kTPBV), kTPBV, 0, st>>>(d, make_cdf(c), M, w, qdf, a);
  return cudaGetLastError();
}

}  // namespace jz
