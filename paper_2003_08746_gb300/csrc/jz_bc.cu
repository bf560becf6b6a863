// Boundary conditions of the jet (paper Sec. "Large Eddy Simulation
// Formulation": entrance, far field, exit, azimuthal periodicity, centerline)
// and its ghost points, applied after every Runge-Kutta stage (Algorithm 2:
// Update(B.C., Visc.), Create(Ghost)) by one kernel.
//
// In order the conditions are: far field (j = nj-1), entrance (i = 0) and exit
// (i = ni-1), axis average (j = 0), then every ghost copies its source node.
// Each reads only nodes the stage advanced or the condition before it, and the
// values that are read across conditions are few (the far field at i = 1 and
// i = ni-2 by the corners of the entrance and exit planes, the corners of the
// ring j = 1 by the axis ends), so each thread forms those again and the whole
// shell needs no order between blocks: a thread that owns a boundary node
// computes it and writes it with all its ghost images, and the ghosts of
// advanced nodes (across the axis, around the azimuth) are copied beside them.
#include <cmath>

#include "jz_shadow.cuh"

namespace jz {
namespace {

constexpr int kTPB = 128;
constexpr int AXI = 8;                     // lines of i per axis block

// What the kernel needs of the state: the FP64 fields and, for the FP32-flux form, the shadow.
struct ShellArgs {
  Dims d;
  Consts c;
  ConstsF cf;
  const double* Sb;      // far-field unit normals [3][nk][ni]
  const double* u0;      // entrance profile [nk][nj]
  const double* T;       // forcing shapes [15][nk][nj]
  const double* co;      // their coefficients at this stage's time
  double ink;            // 1 / nk
  State q;
  Scalars* sc;
  int advance;           // last stage of a step: t += dt
  unsigned bA, bE, bX, bF, bR;   // first block after the axis, entrance, exit, far-field and row roles
};

struct Prim {
  double u[3], p, ir, rho;
};
__device__ __forceinline__ Prim prim_of(const Consts& c, const double q[5]) {
  Prim r;
  r.rho = q[0];
  r.ir = rcp64(q[0]);
  for (int a = 0; a < 3; ++a) r.u[a] = q[a + 1] * r.ir;
  r.p = fma(-c.gm1_half, q[1] * r.u[0] + q[2] * r.u[1] + q[3] * r.u[2], c.gm1 * q[4]);
  return r;
}
__device__ __forceinline__ void cons_of(const Consts& c, double rho, double u, double v, double w, double pr,
                                        double out[5]) {
  out[0] = rho;
  out[1] = rho * u;
  out[2] = rho * v;
  out[3] = rho * w;
  out[4] = fma(pr, c.Cp, 0.5 * (out[1] * u + out[2] * v + out[3] * w));   // p / (gamma-1) + rho |u|^2 / 2
}
__device__ __forceinline__ void load_q(const State& q, long long p, double v[5]) {
#pragma unroll
  for (int m = 0; m < 5; ++m) v[m] = q.q[m][p];
}

// Riemann-invariant far field of the node (i, nj-1, k) from its inner neighbour qi = Q(i, nj-2, k).
__device__ void farfield_value(const ShellArgs& A, int i, int k, const double qi[5], double out[5]) {
  const Consts& c = A.c;
  const long long nb = (long long)A.d.nk * A.d.ni, sb = (long long)k * A.d.ni + i;
  const double n[3] = {A.Sb[sb], A.Sb[nb + sb], A.Sb[2 * nb + sb]};
  const Prim r = prim_of(c, qi);
  const double a_i = sqrt64(c.gamma * r.p * r.ir);
  const double un_i = r.u[0] * n[0] + r.u[1] * n[1] + r.u[2] * n[2];
  const double two = 2.0 * c.Cp;                           // 2 / (gamma - 1)
  const double Rp = fma(two, a_i, un_i), Rm = -two;
  const double un = 0.5 * (Rp + Rm), ab = 0.25 * c.gm1 * (Rp - Rm);
  const bool outflow = un > 0.0;
  // density of the isentrope through (rho_s, a_s), interior or ambient, at sound speed ab:
  // rho_s |ab / a_s|^(2 / (gamma-1))
  const double rho = outflow ? r.rho * isentrope(c, fabs(ab) * rcp64(a_i)) : isentrope(c, fabs(ab));
  const double pr = rho * ab * ab * c.p_inf;               // rho a^2 / gamma
  double v[3];
  for (int x = 0; x < 3; ++x) v[x] = outflow ? fma(un - un_i, n[x], r.u[x]) : un * n[x];
  cons_of(c, rho, v[0], v[1], v[2], pr, out);
}

// Entrance node (0, j, k) by 1-D characteristics: tanh profile + forcing at the stage time,
// q1 = Q(1, j, k).
__device__ void entrance_value(const ShellArgs& A, int j, int k, const double q1[5], double out[5]) {
  const Consts& c = A.c;
  const long long tab = (long long)k * A.d.nj + j, plane = (long long)A.d.nk * A.d.nj;
  // five partial sums: the FP64 latency of one chain of 15 would set the kernel's time
  double f[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int n = 0; n < kNT; ++n) f[n % 5] = fma(__ldg(A.co + n), __ldg(A.T + n * plane + tab), f[n % 5]);
  const double ut = fma(c.jet_mach, ((f[0] + f[1]) + (f[2] + f[3])) + f[4], A.u0[tab]);
  if (ut >= 1.0) {                                          // supersonic: all imposed
    cons_of(c, 1.0, ut, 0.0, 0.0, c.p_inf, out);
    return;
  }
  const Prim r = prim_of(c, q1);
  const double two = 2.0 * c.Cp;
  const double Rm = fma(-two, sqrt64(c.gamma * r.p * r.ir), r.u[0]), Rp = ut + two;
  const double ub = 0.5 * (Rp + Rm), ab = 0.25 * c.gm1 * (Rp - Rm);
  const double rho = isentrope(c, fabs(ab));
  cons_of(c, rho, ub, 0.0, 0.0, rho * ab * ab * c.p_inf, out);
}

// Exit node (ni-1, j, k): ambient pressure, velocity and internal energy of qi = Q(ni-2, j, k).
__device__ void exit_value(const ShellArgs& A, const double qi[5], double out[5]) {
  const Prim r = prim_of(A.c, qi);
  cons_of(A.c, A.c.p_inf * r.rho * rcp64(r.p), r.u[0], r.u[1], r.u[2], A.c.p_inf, out);
}

// The inner neighbour of an entrance or exit node (i = 1 or ni-2): an advanced node, or for
// j = nj-1 the far-field node formed from the one below it.
__device__ __forceinline__ void inner_neighbour(const ShellArgs& A, int i, int j, int k, double q[5]) {
  if (j < A.d.nj - 1) {
    load_q(A.q, pidx(A.d, i, j, k), q);
  } else {
    double t[5];
    load_q(A.q, pidx(A.d, i, j - 1, k), t);
    farfield_value(A, i, k, t, q);
  }
}

// Write the value of a boundary node at row (j, k), with every ghost that copies it, as NC nodes along
// i from ia: the entrance and exit with their ghosts beyond (zero order in i), one node elsewhere.  Beyond
// the far field two more rows take it (zero order in j), across the axis row -j holds it at k + nk/2,
// and each row has images around the azimuth where k is within two of its ends.
template <bool SH, int NC>
__device__ __forceinline__ void put_node(const ShellArgs& A, const double v[5], int ia, int j, int k) {
  const Dims& d = A.d;
  float2 s[NSH];
  if (SH) shadow_of(A.cf, v, s);
  const bool far = j == d.nj - 1, mirror = j >= 1 && j <= kG;
  const long long turn = (long long)d.nk * d.sk;
  const int half = d.nk / 2, kf = far ? kG : 0, rows = 1 + kf + (mirror ? 1 : 0);
#pragma unroll 1
  for (int r = 0; r < rows; ++r) {
    const bool m = r > kf;                                 // the row across the axis
    const int kk = m ? (k >= half ? k - half : k + half) : k;
    long long p = pidx(d, ia, m ? -j : j + r, kk);
    const int before = kk >= d.nk - kG, after = kk < kG;   // images at kk - nk and kk + nk
    if (before) p -= turn;
#pragma unroll 1
    for (int n = 0; n < 1 + before + after; ++n, p += turn) {
#pragma unroll
      for (int q = 0; q < 5; ++q)
#pragma unroll
        for (int x = 0; x < NC; ++x) A.q.q[q][p + x] = v[q];
      if (SH) {
#pragma unroll
        for (int q = 0; q < NSH; ++q)
#pragma unroll
          for (int x = 0; x < NC; ++x) A.q.sh[q * d.Np + p + x] = s[q];
      }
    }
  }
}

// Copy a source node to a ghost (state and shadow as they are), all loads before the first store.
template <bool SH>
__device__ __forceinline__ void copy_node(const ShellArgs& A, long long p, long long src) {
  double v[5];
  float2 s[NSH];
  load_q(A.q, src, v);
  if (SH) {
#pragma unroll
    for (int m = 0; m < NSH; ++m) s[m] = A.q.sh[m * A.d.Np + src];
  }
#pragma unroll
  for (int m = 0; m < 5; ++m) A.q.q[m][p] = v[m];
  if (SH) {
#pragma unroll
    for (int m = 0; m < NSH; ++m) A.q.sh[m * A.d.Np + p] = s[m];
  }
}

// Boundary nodes and ghosts of the jet, by block roles: axis, entrance, exit, far field, ghost rows across the
// axis, ghost planes around the azimuth.  Every stage waits for it.  On small grids latency bounds it, a chain of
// dependent FP64 operations per node: 6.6 us per launch on 70 x 33 x 18 (a launch that does nothing 0.7, the
// copies alone 2.6, the far field 3.9, the exit 5.0, the entrance 6.6), where three kernels for the conditions and
// one for the ghosts took 4 launches and 57 us; 11 with 32 forcing shapes, the far field's normals normalized at
// each use, and corner nodes among the others.  On large grids the ghosts' traffic does: 1024 x 512 x 360
// with the FP32 shadow 0.25 ms (0.32 when each copied value was stored before the next was loaded; 0.64 by the
// separate kernels).
template <bool SH>
__global__ void __launch_bounds__(kTPB) k_jet_shell(const __grid_constant__ ShellArgs A) {
  const Dims& d = A.d;
  const unsigned b = blockIdx.x, th = threadIdx.x;
  if (b < A.bA) {
    // axis: the ring j = 1 averaged over the azimuth; the two ends, whose ring is entrance and exit
    // nodes, by a block each with all its threads along k, the lines between AXI to a block
    const bool end = b < 2;
    const int nx = end ? 1 : AXI, ix = end ? 0 : (int)(th % AXI), ky = end ? (int)th : (int)(th / AXI), nky = kTPB / nx;
    const int i = end ? (b == 0 ? 0 : d.ni - 1) : (int)((b - 2) * AXI) + 1 + ix;
    const bool in = end || i < d.ni - 1;
    double s[5] = {0, 0, 0, 0, 0};
    if (in) {
      for (int k = ky; k < d.nk; k += nky) {
        double v[5], t[5];
        if (b == 0) {
          inner_neighbour(A, 1, 1, k, t);
          entrance_value(A, 1, k, t, v);
        } else if (b == 1) {
          inner_neighbour(A, i - 1, 1, k, t);
          exit_value(A, t, v);
        } else {
          load_q(A.q, pidx(d, i, 1, k), v);
        }
#pragma unroll
        for (int m = 0; m < 5; ++m) s[m] += v[m];
      }
    }
    __shared__ double red[5][kTPB / 32][AXI];
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      double x = s[m];
      for (int o = 16; o >= nx; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if ((th & 31) < nx) red[m][th >> 5][th & 31] = x;
    }
    __syncthreads();
    double mean[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      double x = 0.0;
      for (int w = 0; w < kTPB / 32; ++w) x += red[m][w][ix];
      mean[m] = x * A.ink;
    }
    if (end)
      for (int k = ky; k < d.nk; k += nky) put_node<SH, 1 + kG>(A, mean, b == 0 ? -kG : i, 0, k);
    else if (in)
      for (int k = ky; k < d.nk; k += nky) put_node<SH, 1>(A, mean, i, 0, k);
    if (b == 0 && th == 0 && A.advance) A.sc->t = A.sc->t + A.sc->dt;
    return;
  }
  if (b < A.bX) {
    // entrance (i = 0) and exit (i = ni-1), 1 <= j <= nj-1; the nodes at j = nj-1, which take the
    // longest (a far-field value first, three rows of images), last and by warps of their own
    const bool ent = b < A.bE;
    const unsigned t = (b - (ent ? A.bA : A.bE)) * kTPB + th, nj2 = d.nj - 2, n = nj2 * (unsigned)d.nk;
    if (t >= n + (unsigned)d.nk) return;
    const int k = t < n ? (int)(t / nj2) : (int)(t - n), j = t < n ? 1 + (int)(t - k * nj2) : d.nj - 1;
    double qi[5], v[5];
    inner_neighbour(A, ent ? 1 : d.ni - 2, j, k, qi);
    if (ent)
      entrance_value(A, j, k, qi, v);
    else
      exit_value(A, qi, v);
    put_node<SH, 1 + kG>(A, v, ent ? -kG : d.ni - 1, j, k);
    return;
  }
  const unsigned ni2 = d.ni - 2;
  if (b < A.bF) {
    // far field j = nj-1, 1 <= i <= ni-2
    const unsigned t = (b - A.bX) * kTPB + th;
    if (t >= ni2 * (unsigned)d.nk) return;
    const int i = 1 + (int)(t % ni2), k = (int)(t / ni2);
    double qi[5], v[5];
    load_q(A.q, pidx(d, i, d.nj - 2, k), qi);
    farfield_value(A, i, k, qi, v);
    put_node<SH, 1>(A, v, i, d.nj - 1, k);
    return;
  }
  if (b < A.bR) {
    // ghost rows across the axis, 1 <= i <= ni-2, every padded k
    const unsigned t = (b - A.bF) * kTPB + th, ek = d.nk + 2 * kG;
    if (t >= 2 * ni2 * ek) return;
    const int i = 1 + (int)(t % ni2);
    const unsigned r = t / ni2;
    const int m = 1 + (int)(r & 1), k = (int)(r >> 1) - kG;
    int ks = k + d.nk / 2;
    ks = ks < 0 ? ks + d.nk : (ks >= d.nk ? ks - d.nk : ks);
    copy_node<SH>(A, pidx(d, i, -m, k), pidx(d, i, m, ks));
    return;
  }
  // ghost planes around the azimuth, 1 <= i <= ni-2, 1 <= j <= nj-2
  const unsigned t = (b - A.bR) * kTPB + th, nj2 = d.nj - 2;
  if (t >= 4 * ni2 * nj2) return;
  const int i = 1 + (int)(t % ni2);
  const unsigned r = t / ni2;
  const int j = 1 + (int)(r % nj2), s = (int)(r / nj2);    // k = -2, -1, nk, nk+1
  const int k = s < 2 ? s - kG : d.nk + s - kG;
  copy_node<SH>(A, pidx(d, i, j, k), pidx(d, i, j, s < 2 ? k + d.nk : k - d.nk));
}

// Entrance tables at i = 0: u0 = U_j/2 [1 + tanh((0.5 - r)/(2 theta))] and the forcing shapes
// g(r) cos m theta, g(r) sin m theta, g(r) = exp(-((r - 0.5)/0.1)^2), with r and theta from the node
// coordinates.
__global__ void k_build_inflow(Dims d, Consts c, GridDev g, double* u0, double* T) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)d.nj * d.nk) return;
  const double y = g.Xin[t], z = g.Xin[(long long)d.nj * d.nk + t];   // t = k nj + j
  const double r = sqrt(y * y + z * z);
  const double th = atan2(z, y);
  u0[t] = 0.5 * c.jet_mach * (1.0 + tanh((0.5 - r) / (2.0 * c.theta_mom)));
  const double x = (r - 0.5) / 0.1;
  const double gr = exp(-(x * x));
  const long long plane = (long long)d.nk * d.nj;
  for (int n = 0; n < kNT; ++n) {
    const double a = shape_mode(n) * th;
    T[n * plane + t] = gr * (shape_sine(n) ? sin(a) : cos(a));
  }
}

}  // namespace

cudaError_t jet_shell(const Dims& d, const Consts& c, const GridDev& g, const Inflow& in, const State& q,
                      Scalars* sc, int stage, int advance, cudaStream_t st) {
  ShellArgs A;
  A.d = d;
  A.c = c;
  A.cf = make_constsf(c);
  A.Sb = g.Sb;
  A.u0 = in.u0;
  A.T = in.T;
  A.co = in.co + stage * kNT;
  A.ink = 1.0 / d.nk;
  A.q = q;
  A.sc = sc;
  A.advance = advance;
  const long long ni2 = d.ni - 2;
  const unsigned nio = blocks_for((long long)(d.nj - 1) * d.nk, kTPB);
  A.bA = 2 + blocks_for(ni2, AXI);
  A.bE = A.bA + nio;
  A.bX = A.bE + nio;
  A.bF = A.bX + blocks_for(ni2 * d.nk, kTPB);
  A.bR = A.bF + blocks_for(2 * ni2 * (d.nk + 2 * kG), kTPB);
  const unsigned n = A.bR + blocks_for(4 * ni2 * (d.nj - 2), kTPB);
  if (q.sh)
    k_jet_shell<true><<<n, kTPB, 0, st>>>(A);
  else
    k_jet_shell<false><<<n, kTPB, 0, st>>>(A);
  return cudaGetLastError();
}

cudaError_t build_inflow(const Dims& d, const Consts& c, const GridDev& g, const jz_params& p, Inflow& in,
                         cudaStream_t st) {
  for (int mf = 0; mf < kNF; ++mf) {
    in.cphi[mf] = std::cos(p.forcing_phi[mf]);
    in.sphi[mf] = std::sin(p.forcing_phi[mf]);
    in.amp[mf] = p.forcing_amp[mf];
    in.psi[mf] = p.forcing_psi[mf];
  }
  for (int f = 0; f < JZ_N_FREQ; ++f) in.omega[f] = 2.0 * 3.141592653589793 * p.strouhal[f] * p.jet_mach;
  const long long n = (long long)d.nj * d.nk;
  k_build_inflow<<<blocks_for(n, kTPB), kTPB, 0, st>>>(d, c, g, in.u0, in.T);
  return cudaGetLastError();
}

}  // namespace jz
