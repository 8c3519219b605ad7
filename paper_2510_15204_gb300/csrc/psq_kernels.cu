// FP64 kernels of the PS quadrature path: grid points and weights (Section 2.1, eqs 2-11;
// Algorithm 2), STO and aux-potential evaluation (eq 1, eqs 15-16), the weighted
// contraction of eq 9, the deterministic per-element reduction of its chunk partial sums,
// and the assembly of molecule matrices from per-grid blocks (Section 4).
#include "psq_internal.h"
#include "psq_fx.cuh"

#include <cstdio>

namespace psq {

__constant__ double c_glx[kMaxQ + 1][kMaxQ];  // Gauss-Legendre nodes on [-1,1], rule q
__constant__ double c_glw[kMaxQ + 1][kMaxQ];  // and weights
__constant__ double c_klm[(kMaxL + 1) * (kMaxL + 1)];  // harmonic norms, sqrt2 for m != 0
__constant__ double c_fact[2 * kMaxN + 4];             // k!
constexpr int kRcpD = 128;
__constant__ double c_rcpd[kRcpD];                     // 1/k (c_rcpd[0] unused)

void upload_gl_tables(const double* x, const double* w, const double* klm) {
  cudaMemcpyToSymbol(c_glx, x, sizeof(double) * (kMaxQ + 1) * kMaxQ);
  cudaMemcpyToSymbol(c_glw, w, sizeof(double) * (kMaxQ + 1) * kMaxQ);
  cudaMemcpyToSymbol(c_klm, klm, sizeof(double) * (kMaxL + 1) * (kMaxL + 1));
  double f[2 * kMaxN + 4];
  f[0] = 1.0;
  for (int k = 1; k < 2 * kMaxN + 4; ++k) f[k] = f[k - 1] * k;
  cudaMemcpyToSymbol(c_fact, f, sizeof(f));
  double r[kRcpD];
  r[0] = 0.0;
  for (int k = 1; k < kRcpD; ++k) r[k] = 1.0 / k;
  cudaMemcpyToSymbol(c_rcpd, r, sizeof(r));
}

// x / k for a positive integer k: a multiply by the rounded reciprocal from a table (one
// rounding more than a division, a relative 2^-52 per term; FP64 division is a long
// instruction sequence on this GPU's FP64 pipe), a division past the table.
__device__ __forceinline__ double div_int(double x, int k) { return k < kRcpD ? x * c_rcpd[k] : x / k; }

struct Pt {
  double P[3], dA[3], dB[3];
  double w, rA, rB, mu, nu;
};

// Point p of grid g.  The cell layout follows DevGrid's numbering; the node is the
// Gauss-Legendre node of each dimension mapped onto the cell, the weight is eq 10-11 with
// the Jacobian at the node, and r_A, r_B and the offsets from A and B use the forms
// 2a(sinh^2(mu/2) + sin^2(nu/2)) etc. that do not cancel near the foci.
__device__ __forceinline__ void ps_point(const DevGrid& g, const double* __restrict__ edges,
                                         int64_t p, Pt& o) {
  const int q3 = g.q_mu * g.q_nu * g.q_phi;
  const double* emu = edges + g.edge_off;
  const double* enu = emu + g.n_mu + 1;
  const double* eph = enu + g.n_nu + 1;
  int qi, qj, qk;
  double m0, m1, n0, n1, p0, p1;
  bool dead = false;
  if (p < g.K_reg) {
    const int64_t cell = p / q3;
    const int r = (int)(p - cell * q3);
    const int k = (int)(cell % g.n_phi);
    const int j = (int)((cell / g.n_phi) % g.n_nu);
    const int i = (int)(cell / ((int64_t)g.n_phi * g.n_nu));
    m0 = emu[i]; m1 = emu[i + 1];
    n0 = enu[j]; n1 = enu[j + 1];
    p0 = eph[k]; p1 = eph[k + 1];
    if (g.n_touch > 0 && i >= g.t_mu0 && i <= g.t_mu1 && j >= g.t_nu0 && j <= g.t_nu1 &&
        (g.t_phi_all || k == 0 || k == g.n_phi - 1))
      dead = true;
    qi = r / (g.q_nu * g.q_phi);
    qj = (r / g.q_phi) % g.q_nu;
    qk = r % g.q_phi;
  } else {
    const int64_t s = (p - g.K_reg) / q3;
    const int r = (int)((p - g.K_reg) - s * q3);
    const int ns = g.n_sp, ns3 = ns * ns * ns;
    const int tc = (int)(s / ns3), sub = (int)(s % ns3);
    const int ntp = g.t_phi_all ? g.n_phi : (g.n_phi == 1 ? 1 : 2);
    const int nnu = g.t_nu1 - g.t_nu0 + 1;
    const int ti = tc / (nnu * ntp), tj = (tc / ntp) % nnu, tk = tc % ntp;
    const int i = g.t_mu0 + ti, j = g.t_nu0 + tj;
    const int k = g.t_phi_all ? tk : (tk == 0 ? 0 : g.n_phi - 1);
    const int si = sub / (ns * ns), sj = (sub / ns) % ns, sk = sub % ns;
    const double M0 = emu[i], M1 = emu[i + 1], N0 = enu[j], N1 = enu[j + 1];
    const double P0 = eph[k], P1 = eph[k + 1];
    m0 = M0 + (M1 - M0) * si / ns; m1 = M0 + (M1 - M0) * (si + 1) / ns;
    n0 = N0 + (N1 - N0) * sj / ns; n1 = N0 + (N1 - N0) * (sj + 1) / ns;
    p0 = P0 + (P1 - P0) * sk / ns; p1 = P0 + (P1 - P0) * (sk + 1) / ns;
    qi = r / (g.q_nu * g.q_phi);
    qj = (r / g.q_phi) % g.q_nu;
    qk = r % g.q_phi;
  }
  const double hm = 0.5 * (m1 - m0), hn = 0.5 * (n1 - n0), hp = 0.5 * (p1 - p0);
  const double mu = 0.5 * (m0 + m1) + hm * c_glx[g.q_mu][qi];
  const double nu = 0.5 * (n0 + n1) + hn * c_glx[g.q_nu][qj];
  const double ph = 0.5 * (p0 + p1) + hp * c_glx[g.q_phi][qk];
  const double wq = (hm * c_glw[g.q_mu][qi]) * (hn * c_glw[g.q_nu][qj]) * (hp * c_glw[g.q_phi][qk]);
  const double a = g.a;
  const double sh = sinh(mu), ch = cosh(mu);
  double sn, cs, sp, cp;
  sincos(nu, &sn, &cs);
  sincos(ph, &sp, &cp);
  o.w = dead ? 0.0 : wq * (a * a * a) * sh * sn * (sh * sh + sn * sn);
  const double x = a * sh * sn * cp, y = a * sh * sn * sp, z = a * ch * cs;
  const double shm = sinh(0.5 * mu);
  double sn2, cs2;
  sincos(0.5 * nu, &sn2, &cs2);
  const double s2m = shm * shm, s2n = sn2 * sn2, c2n = cs2 * cs2;
  o.rA = 2.0 * a * (s2m + s2n);
  o.rB = 2.0 * a * (s2m + c2n);
  const double zA = 2.0 * a * (s2m * cs - s2n);
  const double zB = 2.0 * a * (s2m * cs + c2n);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double r0 = g.R[c * 3 + 0], r1 = g.R[c * 3 + 1], r2 = g.R[c * 3 + 2];
    o.P[c] = g.M[c] + (r0 * x + r1 * y + r2 * z);
    o.dA[c] = r0 * x + r1 * y + r2 * zA;
    o.dB[c] = r0 * x + r1 * y + r2 * zB;
  }
  o.mu = mu;
  o.nu = nu;
}

// Real orthonormal spherical harmonics Y_lm(u), |u| = 1, l <= lmax, index l*l + l + m:
// Y_lm = K_lm Q_l^|m|(u_z) {Re, Im}(u_x + i u_y)^|m|, with Q_m^m = (2m-1)!!,
// Q_{m+1}^m = (2m+1) u_z Q_m^m, (l-m) Q_l^m = (2l-1) u_z Q_{l-1}^m - (l+m-1) Q_{l-2}^m (unrolled: the
// coefficients are constants, a conversion or division would run on the FP64 pipe).
__device__ __forceinline__ void real_ylm(int lmax, double ux, double uy, double uz, double* Y) {
  double C = 1.0, S = 0.0, dfact = 1.0;  // Re, Im of (u_x + i u_y)^m; (2m-1)!!
#pragma unroll
  for (int m = 0; m <= kMaxL; ++m) {
    if (m > lmax) break;
    if (m > 0) {
      const double c = ux * C - uy * S;
      S = ux * S + uy * C;
      C = c;
      dfact *= 2 * m - 1;
    }
    double q2 = 0.0, q1 = dfact;  // Q_{l-2}, Q_{l-1} as l climbs
#pragma unroll
    for (int l = m; l <= kMaxL; ++l) {
      if (l > lmax) break;
      double q = dfact;
      if (l > m) {
        q = l == m + 1 ? (double)(2 * m + 1) * dfact * uz
                       : ((double)(2 * l - 1) / (l - m)) * (uz * q1) - ((double)(l + m - 1) / (l - m)) * q2;
        q2 = q1;
        q1 = q;
      }
      const int base = l * l + l;
      const double kq = c_klm[base + m] * q;
      if (m == 0) {
        Y[base] = kq;
      } else {
        Y[base + m] = kq * C;
        Y[base - m] = kq * S;
      }
    }
  }
}

__device__ __forceinline__ double ipow(double x, int n) {
  double r = 1.0;
  for (int i = 0; i < n; ++i) r *= x;
  return r;
}

// 1 + x/a (1 + x/(a+1) (1 + ... x/b)): a finite exponential-type sum, from its last term.
__device__ __forceinline__ double nested(double x, int a, int b) {
  double s = 1.0;
#pragma unroll 1
  for (int j = b; j >= a; --j) s = fma(s, div_int(x, j), 1.0);
  return s;
}

// Radial factor of V^P (eq 16 written out by the Laplace expansion of 1/r12) as a function of
// x = zeta r, without its constant 4 pi/(2l+1) N zeta^-(n+1):
// gamma(n+l+2, x)/x^(l+1) + Gamma(n-l+1, x) x^l, ex = e^-x.
// gamma by its positive series below x = k (no cancellation), by (k-1)! - Gamma above; the number of
// terms of the series comes from an FP32 run of it.
__device__ __forceinline__ double aux_pot_radial(int n, int l, double x, double ex) {
  const int k1 = n + l + 2, k2 = n - l + 1;
  double inner;
  if (x < (double)k1) {
    const float xf = (float)x;
    float t = 1.0f, s = 1.0f;
    int m = 0;
#pragma unroll 1
    while (t > 3e-18f * s && m < kRcpD - 1 - k1) {
      ++m;
      t *= __fdividef(xf, (float)(k1 + m));
      s += t;
    }
    inner = ipow(x, n + 1) * ex * (c_rcpd[k1] * nested(x, k1 + 1, k1 + m));  // x^k1 / x^(l+1) = x^(n+1)
  } else {
    const double f = c_fact[k1 - 1];
    inner = (f - f * ex * nested(x, 1, k1 - 1)) * ipow(1.0 / x, l + 1);
  }
  return inner + c_fact[k2 - 1] * ex * nested(x, 1, k2 - 1) * ipow(x, l);
}

// Radial factor of one row kind (0 chi, 1 lap chi (kinetic operand), 2 V^P) of a shell at distance
// r: x = zeta r, ex = e^-x, ir = 1/r.
__device__ __forceinline__ double radial_value(const DevShell& q, int kind, double r, double ir, double ex) {
  if (kind == 2) return q.vnorm * aux_pot_radial(q.n, q.l, q.zeta * r, ex);
  double v = q.norm * ipow(r, q.n - 1) * ex;
  if (kind == 1) v *= (q.n * (q.n - 1) - q.l * (q.l + 1)) * (ir * ir) - 2.0 * q.n * q.zeta * ir + q.zeta * q.zeta;
  return v;
}

__device__ __forceinline__ int shells_lmax(const DevShell* sh, int s0, int s1) {
  int l = 0;
  for (int s = s0; s < s1; ++s) l = max(l, sh[s].l);
  return l;
}

// One row kind of a shell at one point: the radial value v times the harmonics.
__device__ __forceinline__ void store_shell(const DevShell& q, double v, const double* Y, double* __restrict__ out, int64_t rs,
                                            int64_t p, int row) {
  const int base = q.l * q.l + q.l;
  int64_t o = (int64_t)(row + q.fn0) * rs + p;
  for (int m = -q.l; m <= q.l; ++m, o += rs) out[o] = v * Y[base + m];
}

// Evaluation, FP64: one CTA per PointBlock, the operand rows of its points (ps_point's forms of the
// weight, the distances and the offsets).  GB300's FP64 pipe is the bound (two operations per clock
// and SM), so nothing is computed twice on it: the trigonometric functions once per node, the radial
// factors of A and B (exponentials, incomplete gamma series) once per (mu, nu) node pair for all phi,
// those of a third centre for half of the phi nodes (phi -> -phi is a symmetry of the grid).  A point
// is then its harmonics and one product per function.  Row layout: F/L rows are A's basis functions
// then B's (fn0 counted within each atom), G/U rows the aux functions of the grid's aux centres.
// Measured (a thread per point -> now): bent triatomic (963,072 points) 4.5 -> 1.1 ms, H2 (57,600
// points) 0.22 -> 0.06 ms.
struct EvalNodes {
  double mu[kMaxQ][4];             // sinh, cosh, sinh^2(v/2), weight
  double nu[kMaxQ][5];             // sin, cos, sin^2(v/2), cos^2(v/2), weight
  double ph[2 * kEvalMaxNodes][3];  // sin, cos, weight: the rows [u0, u1), then their mirrors
  int meta[4];                     // lmax of A, B, C; functions of the first aux centre
  CentreShells shells[3];
};
constexpr int kEvalFp64Smem = (int)sizeof(EvalNodes) + kEvalTabBytes;

__global__ void __launch_bounds__(kEvalThreads, 3) eval_fp64_kernel(LaunchTables t, double* __restrict__ ops) {
  extern __shared__ __align__(16) uint8_t raw[];
  EvalNodes& nd = *reinterpret_cast<EvalNodes*>(raw);
  const int tid = threadIdx.x;
  const PointBlock pb = t.pblocks[blockIdx.x];
  const DevGrid& g = t.grids[pb.grid];
  const bool third = g.C >= 0;
  const int np = pb.pr1 - pb.pr0, nu = pb.u1 - pb.u0, nn = nu * g.q_phi;  // node pairs; phi rows, nodes of the half
  const int nbA = g.shb_A1 - g.shb_A0, nbB = g.shb_B1 - g.shb_B0, na0 = g.sha_1 - g.sha_0, na1 = g.sha_3 - g.sha_2;
  const bool basis = g.row_F >= 0 || g.row_L >= 0, aux = g.row_G >= 0 || g.row_U >= 0;
  const int n_pair = nbA + nbB + (third ? 0 : na0 + na1);  // shells with a value per node pair
  double* tp = reinterpret_cast<double*>(raw + sizeof(EvalNodes));  // [2 shell + kind][pair]
  const int p0 = min(pb.s0, n_pair), p1 = min(pb.s1, n_pair);       // this CTA's shells: of those,
  const int q0 = third ? max(pb.s0 - n_pair, 0) : 0, q1 = third ? max(pb.s1 - n_pair, 0) : 0;  // and of C
  double* tr = tp + 2 * (p1 - p0) * np;                             // [phi node][pair]: distance from C
  double* tc = tr + (third ? nn * np : 0);                          // [shell of C][phi node][pair]
  // the column: its element rows, its points, its phi rows
  const int nreg = g.n_mu * g.n_nu, ns = g.n_sp, q3 = g.q_mu * g.q_nu * g.q_phi;
  const bool reg = pb.col < nreg;
  int i, j, si = 0, sj = 0, nu_rows;
  int64_t cell0, cell_s1, cell_s2 = 0;  // first point; point strides of phi cells and of their sub-rows
  bool touch = false;
  if (reg) {
    i = pb.col / g.n_nu;
    j = pb.col - i * g.n_nu;
    nu_rows = g.n_phi;
    cell0 = (int64_t)pb.col * g.n_phi * q3;
    cell_s1 = q3;
    touch = g.n_touch > 0 && i >= g.t_mu0 && i <= g.t_mu1 && j >= g.t_nu0 && j <= g.t_nu1;
  } else {
    const int c = pb.col - nreg, sub = c % (ns * ns), tij = c / (ns * ns);
    i = g.t_mu0 + tij / g.nt_nu;
    j = g.t_nu0 + tij % g.nt_nu;
    si = sub / ns;
    sj = sub - si * ns;
    nu_rows = g.nt_phi * ns;
    cell0 = g.K_reg + ((int64_t)tij * g.nt_phi * ns * ns * ns + (si * ns + sj) * ns) * q3;
    cell_s1 = (int64_t)ns * ns * ns * q3;
    cell_s2 = q3;
  }
  // nodes: mu, nu, and the phi rows of the half and their mirrors
  const double* emu = t.edges + g.edge_off;
  const double* enu = emu + g.n_mu + 1;
  const double* eph = enu + g.n_nu + 1;
  for (int e = tid; e < g.q_mu + g.q_nu + 2 * nn; e += kEvalThreads) {
    const int dim = e < g.q_mu ? 0 : (e < g.q_mu + g.q_nu ? 1 : 2);
    int q, Q, s = 0;
    double m0, m1;
    if (dim == 0) {
      q = e; Q = g.q_mu; s = si; m0 = emu[i]; m1 = emu[i + 1];
    } else if (dim == 1) {
      q = e - g.q_mu; Q = g.q_nu; s = sj; m0 = enu[j]; m1 = enu[j + 1];
    } else {
      const int f = e - g.q_mu - g.q_nu, ul = f / g.q_phi;
      const int uh = pb.u0 + (ul < nu ? ul : ul - nu), u = ul < nu ? uh : nu_rows - 1 - uh;
      q = f - ul * g.q_phi;
      Q = g.q_phi;
      int k = u;
      if (!reg) {
        s = u % ns;
        k = u / ns;
        if (!g.t_phi_all && k > 0) k = g.n_phi - 1;
      }
      m0 = eph[k]; m1 = eph[k + 1];
    }
    if (!reg) {
      const double M0 = m0, M1 = m1;
      m0 = M0 + (M1 - M0) * s / ns;
      m1 = M0 + (M1 - M0) * (s + 1) / ns;
    }
    const double h = 0.5 * (m1 - m0), v = 0.5 * (m0 + m1) + h * c_glx[Q][q], w = h * c_glw[Q][q];
    if (dim == 0) {
      const double s2 = sinh(0.5 * v);
      nd.mu[q][0] = sinh(v); nd.mu[q][1] = cosh(v); nd.mu[q][2] = s2 * s2; nd.mu[q][3] = w;
    } else {
      double sn, cs;
      sincos(v, &sn, &cs);
      if (dim == 1) {
        double s2, c2;
        sincos(0.5 * v, &s2, &c2);
        nd.nu[q][0] = sn; nd.nu[q][1] = cs; nd.nu[q][2] = s2 * s2; nd.nu[q][3] = c2 * c2; nd.nu[q][4] = w;
      } else {
        double* d = nd.ph[e - g.q_mu - g.q_nu];
        d[0] = sn; d[1] = cs; d[2] = w;
      }
    }
  }
  if (tid == 0) {
    nd.meta[0] = max(basis ? shells_lmax(t.bshell, g.shb_A0, g.shb_A1) : 0, aux && !third ? shells_lmax(t.ashell, g.sha_0, g.sha_1) : 0);
    nd.meta[1] = max(basis ? shells_lmax(t.bshell, g.shb_B0, g.shb_B1) : 0, aux && !third ? shells_lmax(t.ashell, g.sha_2, g.sha_3) : 0);
    nd.meta[2] = third && aux ? shells_lmax(t.ashell, g.sha_0, g.sha_1) : 0;
    int nf = 0;
    for (int s = g.sha_0; s < g.sha_1; ++s) nf += 2 * t.ashell[s].l + 1;
    nd.meta[3] = nf;
    for (int c = 0; c < 3; ++c) nd.shells[c] = centre_shells(g, pb, c);
  }
  __syncthreads();
  const double a = g.a;
  if (third)
    for (int e = tid; e < nn * np; e += kEvalThreads) {
      const int f = e / np, pr = pb.pr0 + e - f * np, qi = pr / g.q_nu, qj = pr - qi * g.q_nu;
      const double ss = a * nd.mu[qi][0] * nd.nu[qj][0];
      const double x = ss * nd.ph[f][1] - g.xc, y = ss * nd.ph[f][0], z = a * nd.mu[qi][1] * nd.nu[qj][1] - g.zc;
      tr[e] = sqrt(x * x + y * y + z * z);
    }
  // radial factors per node pair
  for (int e = tid; e < (p1 - p0) * np; e += kEvalThreads) {
    const int i = e / np, s = p0 + i, pq = e - i * np, pr = pb.pr0 + pq, qi = pr / g.q_nu, qj = pr - qi * g.q_nu;
    const bool isb = s < nbA + nbB, onA = isb ? s < nbA : s < nbA + nbB + na0;
    if (isb ? !basis : !aux) continue;
    const DevShell& q = isb ? t.bshell[s < nbA ? g.shb_A0 + s : g.shb_B0 + s - nbA]
                            : t.ashell[onA ? g.sha_0 + s - nbA - nbB : g.sha_2 + s - nbA - nbB - na0];
    const double r = 2.0 * a * (nd.mu[qi][2] + nd.nu[qj][onA ? 2 : 3]), ex = exp(-q.zeta * r), ir = 1.0 / r;
    const bool ka = isb ? g.row_F >= 0 : g.row_G >= 0, kb = isb ? g.row_L >= 0 : g.row_U >= 0;
    if (ka) tp[2 * i * np + pq] = radial_value(q, 0, r, ir, ex);
    if (kb) tp[(2 * i + 1) * np + pq] = radial_value(q, isb ? 1 : 2, r, ir, ex);
  }
  if (third && aux) {
    __syncthreads();
    const int kind = g.row_U >= 0 ? 2 : 0;  // (a refined grid has one aux kind)
    for (int e = tid; e < (q1 - q0) * nn * np; e += kEvalThreads) {
      const int i = e / (nn * np);
      const DevShell& q = t.ashell[g.sha_0 + q0 + i];
      const double r = tr[e - i * nn * np];
      tc[e] = radial_value(q, kind, r, 0.0, exp(-q.zeta * r));
    }
  }
  __syncthreads();
  // the points: phi rows u0 .. u1 - 1 and their mirrors
  double* base = ops + g.op_off;
  const int64_t rs = g.rs;
  const int per = np * g.q_phi;
  double Y[(kMaxL + 1) * (kMaxL + 1)];
  for (int e = tid; e < 2 * nu * per; e += kEvalThreads) {
    const int c = e / per, r = e - c * per, pq = r / g.q_phi, qk = r - pq * g.q_phi;
    const bool mirror = c >= nu;
    const int uh = pb.u0 + (mirror ? c - nu : c), u = mirror ? nu_rows - 1 - uh : uh;
    if (mirror && u == uh) continue;  // the middle row is its own mirror
    const int pr = pb.pr0 + pq, qi = pr / g.q_nu, qj = pr - qi * g.q_nu;
    const int f = (uh - pb.u0) * g.q_phi + (mirror ? g.q_phi - 1 - qk : qk);  // node of the half
    const int64_t pt = cell0 + (reg ? u * cell_s1 : (u / ns) * cell_s1 + (u % ns) * cell_s2) + (int64_t)pr * g.q_phi + qk;
    const int64_t p = (pt >> 7) * g.ws + (pt & 127);  // its element in row 0
    const bool dead = touch && (g.t_phi_all || u == 0 || u == g.n_phi - 1);
    const double sh = nd.mu[qi][0], ch = nd.mu[qi][1], s2m = nd.mu[qi][2];
    const double sn = nd.nu[qj][0], cs = nd.nu[qj][1], s2n = nd.nu[qj][2], c2n = nd.nu[qj][3];
    const double* ph = nd.ph[c * g.q_phi + qk];
    const double rA = 2.0 * a * (s2m + s2n), rB = 2.0 * a * (s2m + c2n), rC = third ? tr[f * np + pq] : 1.0;
    // The operand rows of a contraction carry the weight: chi and lap chi sqrt(w), aux chi w, so that
    // a product of two basis rows is w chi_i chi_j and V^P, which varies slowly, stays as it is.
    double wg = 1.0, wf = 1.0;
    if (g.row_W >= 0) {
      wg = dead ? 0.0 : nd.mu[qi][3] * nd.nu[qj][4] * ph[2] * (a * a * a) * sh * sn * (sh * sh + sn * sn);
      wf = sqrt(wg);
      // the nuclear weights that V_ne elements of this grid are summed with: on a pair grid those of the
      // A x B elements and the square roots of those of the A x A and B x B elements (an atom's own
      // nucleus only on its one-centre grid), on a refined grid the third nucleus's
      // (written with the first shells)
      if (g.n_W == 3 && pb.s0 == 0) {
        const double wa = g.zA / rA, wb = g.zB / rB;
        base[(int64_t)(g.row_W + 0) * rs + p] = wa + wb;
        base[(int64_t)(g.row_W + 1) * rs + p] = sqrt(g.own_A ? wa + wb : wb);
        base[(int64_t)(g.row_W + 2) * rs + p] = sqrt(g.own_B ? wa + wb : wa);
      } else if (g.n_W == 1 && pb.s0 == 0) {
        base[(int64_t)g.row_W * rs + p] = g.zC / rC;
      }
    }
    const double x = a * sh * sn * ph[1], y = a * sh * sn * ph[0];
#pragma unroll 1
    for (int ctr = 0; ctr < 3; ++ctr) {  // A, B, C
      const CentreShells& own = nd.shells[ctr];
      const int b0 = own.b0, b1 = own.b1, a0 = own.a0, a1 = own.a1;
      const bool hb = basis && ctr < 2 && b1 > b0, ha = aux && (ctr == 2) == third && a1 > a0;
      if (!hb && !ha) continue;
      const double ir = 1.0 / (ctr == 0 ? rA : (ctr == 1 ? rB : rC));
      const double dx = (ctr == 2 ? x - g.xc : x) * ir, dy = y * ir;
      const double dz = (ctr == 0 ? 2.0 * a * (s2m * cs - s2n) : (ctr == 1 ? 2.0 * a * (s2m * cs + c2n) : a * ch * cs - g.zc)) * ir;
      real_ylm(nd.meta[ctr], g.R[0] * dx + g.R[1] * dy + g.R[2] * dz, g.R[3] * dx + g.R[4] * dy + g.R[5] * dz,
               g.R[6] * dx + g.R[7] * dy + g.R[8] * dz, Y);
      if (hb) {
        const int roff = ctr == 0 ? 0 : g.nFA;
        for (int s = b0; s < b1; ++s) {
          const DevShell& q = t.bshell[s];
          const double* tv = tp + 2 * (s + own.bt) * np + pq;
          if (g.row_F >= 0) store_shell(q, wf * tv[0], Y, base, rs, p, g.row_F + roff);
          if (g.row_L >= 0) store_shell(q, wf * tv[np], Y, base, rs, p, g.row_L + roff);
        }
      }
      if (ha) {
        const int roff = ctr == 1 ? nd.meta[3] : 0;
        for (int s = a0; s < a1; ++s) {
          const DevShell& q = t.ashell[s];
          if (ctr == 2) {
            const double v = tc[((s + own.at) * nn + f) * np + pq];
            store_shell(q, g.row_U >= 0 ? v : wg * v, Y, base, rs, p, g.row_U >= 0 ? g.row_U : g.row_G);
          } else {
            const double* tv = tp + 2 * (s + own.at) * np + pq;
            if (g.row_G >= 0) store_shell(q, wg * tv[0], Y, base, rs, p, g.row_G + roff);
            if (g.row_U >= 0) store_shell(q, tv[np], Y, base, rs, p, g.row_U + roff);
          }
        }
      }
    }
  }
}

cudaError_t launch_eval_fp64(const LaunchTables& t, double* ops, int /*kinds*/, cudaStream_t s) {
  if (t.n_pblocks == 0) return cudaSuccess;
  eval_fp64_kernel<<<t.n_pblocks, kEvalThreads, kEvalFp64Smem, s>>>(t, ops);
  return cudaGetLastError();
}

// Weighted contraction, FP64 (eq 9): one CTA per (block, output tile, range of 64-point windows);
// partial sums go to their own slot, so the result does not depend on scheduling.
//
// GB300's FP64 pipe (two FMAs per clock and SM) bounds every FP64 sum, so the (P|Q) and (P|ij) sums
// run on the tensor cores in exact digits.  There one factor (V^P) mostly varies slowly over a window and
// the other (w times an aux function or a pair product, formed before it is cut) is scaled by
// its own largest value; an element whose factors are large at different points of a window (a window
// that runs across cells, a steep V^P of high l) takes the window's FP64 chain instead, so that every
// element keeps the precision of its own terms (psq_fx.cuh).  The overlap,
// kinetic and V_ne sums multiply two steep functions of different atoms, whose largest values in a
// window can lie at its opposite ends, where an element would take the chain all the same.
// They stay on the FP64 pipe, with less to do: the nuclear weights of a
// grid are summed first, and symmetric blocks are summed once.
//
// Measured on a bent triatomic (26 basis / 82 aux functions, 963,072 points; all sums on the FP64
// pipe before -> now): 11.82 -> 4.08 ms ((P|ij) alone 2.45, (P|Q) 0.97, the three others 0.89).
// One-electron matrices alone (90 functions, 4.5 M points): 36.0 -> 30.7 ms, 0.79 TFLOP/s on the FP64
// pipe, its bound; H2 (57,600 points): 249 -> 113 us (launch and window latency).
//
// The FMA part: the warps of the CTA share the tile and take every eighth group of 8 points each, so
// that no barrier stands between a warp's loads and its FMAs; a lane holds one column and up to 16
// rows, 16 independent chains, and the pipe stays fed by the two CTAs of an SM (16 warps).  Sub-sums
// of 32 points join the running sums (small outer-region terms are not absorbed one by one); the
// warps' sums are added in order at the end.
constexpr int kFpPts = 8;
struct FmaSmem {
  double v[8][kFpPts][kFpFmaRegs + kFpFmaLanes];   // per warp: [point][register side, then lane side]
  int64_t x[kFpFmaRegs + kFpFmaLanes], y[kFpFmaRegs + kFpFmaLanes];  // operand rows (element offsets; y = -1: no factor)
  double sum[8][kFpFmaRegs][kFpFmaLanes];
};
static_assert(sizeof(FmaSmem) <= fx::kSmemBytes, "the FMA part shares the digits part's shared memory");

// A whole symmetric tile of side n <= 31 in ceil(n / 2) rows of n + 1 lanes: row r and row n - 1 - r
// share a register row, lanes c >= r (c < n) take (r, c), lanes c < r (n - 1 - r, n - 1 - c) and lane
// n the diagonal (n - 1 - r, n - 1 - r).
__device__ __forceinline__ void sym_entry(int n, int r, int lane, int& row, int& col) {
  const bool first = lane >= r && lane < n;
  row = first ? r : n - 1 - r;
  col = first ? lane : (lane < r ? n - 1 - lane : n - 1 - r);
}

// One warp's share of a tile of nr register-side and nl lane-side operand rows (SYM: of a whole
// symmetric tile of nl rows, all on the lane side), into sm.sum[warp].  Narrow tiles: the lanes make
// 1 << gs groups of 32 >> gs, each taking every (1 << gs)-th point.
template <int R, bool SYM>
__device__ __noinline__ void fma_warp(FmaSmem& sm, const double* __restrict__ base, int64_t ws, int k0, int k1, int nr, int nl,
                                      int gs) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double(&v)[kFpPts][kFpFmaRegs + kFpFmaLanes] = sm.v[warp];
  const int gl = lane & ((32 >> gs) - 1), grp = lane >> (5 - gs);
  double acc[R], sq[R];
  int ra[R], rb[R];  // staged operand rows of each entry
#pragma unroll
  for (int r = 0; r < R; ++r) {
    acc[r] = sq[r] = 0.0;
    ra[r] = min(r, nr - 1);
    rb[r] = kFpFmaRegs + min(gl, nl - 1);
    if (SYM) {
      sym_entry(nl, min(r, (nl - 1) / 2), min(gl, nl), ra[r], rb[r]);
      ra[r] += kFpFmaRegs;
      rb[r] += kFpFmaRegs;
    }
  }
  const int pp = lane & (kFpPts - 1), e0 = lane >> 3;
  for (int k = k0 + kFpPts * warp, n = 1; k < k1; k += 8 * kFpPts, ++n) {
    const double* at = base + (int64_t)(k >> 7) * ws + (k & 127) + pp;
#pragma unroll
    for (int i = SYM ? kFpFmaRegs / 4 : 0; i < (kFpFmaRegs + kFpFmaLanes) / 4; ++i) {
      const int e = e0 + 4 * i;
      if (e < kFpFmaRegs ? e < nr : e - kFpFmaRegs < nl) {
        double x = 0.0;
        if (k + pp < k1) {
          x = __ldg(at + sm.x[e]);
          if (sm.y[e] >= 0) x *= __ldg(at + sm.y[e]);
        }
        v[pp][e] = x;
      }
    }
    __syncwarp();
#pragma unroll 1
    for (int p = grp; p < kFpPts; p += 1 << gs)
#pragma unroll
      for (int r = 0; r < R; ++r) sq[r] = fma(v[p][ra[r]], v[p][rb[r]], sq[r]);
    if ((n & 3) == 0) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        acc[r] += sq[r];
        sq[r] = 0.0;
      }
    }
    __syncwarp();
  }
#pragma unroll
  for (int r = 0; r < R; ++r) sm.sum[warp][r][lane] = acc[r] + sq[r];
}

__device__ __forceinline__ void contract_fma(const LaunchTables& t, const GemmItem& it, const GemmBlock& b, const DevGrid& g,
                                             const double* __restrict__ base, double* __restrict__ part, uint8_t* raw) {
  FmaSmem& sm = *reinterpret_cast<FmaSmem*>(raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, K = (int)g.K;
  const int k0 = it.chunk * b.win_per * kFpWin, k1 = (int)min((int64_t)K, (int64_t)k0 + (int64_t)b.win_per * kFpWin);
  const int r0 = it.tm * b.tile_m, c0 = it.tn * b.tile_n;
  const int rows = min(b.tile_m, b.m - r0), cols = min(b.tile_n, b.n - c0);
  const bool sym = b.kind == kFpFmaSym && it.tm == it.tn;
  // register side and lane side: rows and columns, or (swap) columns and rows
  const int nr = sym ? 0 : (b.swap ? cols : rows), nl = b.swap ? rows : cols;
  const int roff = b.swap ? b.b_off + c0 : b.a_off + r0, loff = b.swap ? b.a_off + r0 : b.b_off + c0;
  if (tid < kFpFmaRegs + kFpFmaLanes) {
    const bool rs = tid < kFpFmaRegs;
    const int i = rs ? tid : tid - kFpFmaRegs;
    if (i < (rs ? nr : nl)) {
      const int2 q = t.pairs[(rs ? roff : loff) + i];
      sm.x[tid] = q.x * g.rs;
      sm.y[tid] = q.y >= 0 ? q.y * g.rs : -1;
    }
  }
  __syncthreads();
  const int R = sym ? (nl + 1) / 2 : nr;
  const int width = sym ? nl + 1 : nl, gs = width <= 4 ? 3 : (width <= 8 ? 2 : (width <= 16 ? 1 : 0));
  if (sym) {
    if (R <= 2) fma_warp<2, true>(sm, base, g.ws, k0, k1, nr, nl, gs);
    else if (R <= 4) fma_warp<4, true>(sm, base, g.ws, k0, k1, nr, nl, gs);
    else if (R <= 8) fma_warp<8, true>(sm, base, g.ws, k0, k1, nr, nl, gs);
    else if (R <= 12) fma_warp<12, true>(sm, base, g.ws, k0, k1, nr, nl, gs);
    else fma_warp<16, true>(sm, base, g.ws, k0, k1, nr, nl, gs);
  } else {
    if (R <= 2) fma_warp<2, false>(sm, base, g.ws, k0, k1, nr, nl, gs);
    else if (R <= 4) fma_warp<4, false>(sm, base, g.ws, k0, k1, nr, nl, gs);
    else if (R <= 6) fma_warp<6, false>(sm, base, g.ws, k0, k1, nr, nl, gs);
    else if (R <= 8) fma_warp<8, false>(sm, base, g.ws, k0, k1, nr, nl, gs);
    else if (R <= 10) fma_warp<10, false>(sm, base, g.ws, k0, k1, nr, nl, gs);
    else if (R <= 12) fma_warp<12, false>(sm, base, g.ws, k0, k1, nr, nl, gs);
    else if (R <= 14) fma_warp<14, false>(sm, base, g.ws, k0, k1, nr, nl, gs);
    else fma_warp<16, false>(sm, base, g.ws, k0, k1, nr, nl, gs);
  }
  __syncthreads();
  double* out = part + b.part_off + (int64_t)it.chunk * b.m * b.n;
  for (int r = warp; r < R; r += 8) {
    if (lane >= 32 >> gs) continue;
    double s = 0.0;
    for (int w = 0; w < 8; ++w)
      for (int g2 = lane; g2 < 32; g2 += 32 >> gs) s += sm.sum[w][r][g2];
    int row = b.swap ? lane : r, col = b.swap ? r : lane;
    bool live = lane < nl;
    if (sym) {
      sym_entry(nl, r, lane, row, col);
      live = lane < nl || (lane == nl && 2 * r != nl - 1);
    }
    if (live) {
      out[(int64_t)(r0 + row) * b.n + c0 + col] = s;
      if (b.kind == kFpFmaSym) out[(int64_t)(c0 + col) * b.n + r0 + row] = s;
    }
  }
}

// The plain sums of an item's points [from, to) for element (r, c) of its tile and the next columns:
// fx::window's chain.
struct ItemChain {
  const GemmItem* item;
  const GemmBlock* blocks;
  const DevGrid* grids;
  const int2* pairs;
  const double* ops;
  int from, to;
  template <int N>
  __device__ __forceinline__ void operator()(int r, int c, int p0, int step, double (&s)[N]) const {
    const GemmBlock& b = blocks[item->block];
    const DevGrid& g = grids[b.grid];
    const int row = item->tm * kFpDigitRows + r, col = item->tn * kFpDigitCols + c;
    if (row >= b.m || col >= b.n) return;
    const int2 qa = pairs[b.a_off + row];
    int2 qb[N];
#pragma unroll
    for (int j = 0; j < N; ++j) qb[j] = pairs[b.b_off + min(col + j, b.n - 1)];
    const int64_t rs = g.rs, ws = g.ws;
#pragma unroll 4
    for (int p = from + p0; p < to; p += step) {
      const double* at = ops + g.op_off + (int64_t)(p >> 7) * ws + (p & 127);
      double x = at[qa.x * rs];
      if (qa.y >= 0) x *= at[qa.y * rs];
#pragma unroll
      for (int j = 0; j < N; ++j) {
        double y = at[qb[j].x * rs];
        if (qb[j].y >= 0) y *= at[qb[j].y * rs];
        s[j] = fma(x, y, s[j]);
      }
    }
  }
};

__global__ void __launch_bounds__(fx::kThreads, 2) contract_fp64_kernel(LaunchTables t, const double* __restrict__ ops,
                                                                        double* __restrict__ part, int* __restrict__ status,
                                                                        uint64_t wait_ns, const int* hold) {
  extern __shared__ __align__(1024) uint8_t raw[];
  const GemmItem it = t.items[blockIdx.x];
  const GemmBlock b = t.gblocks[it.block];
  const DevGrid& g = t.grids[b.grid];
  const double* base = ops + g.op_off;
  if (b.kind != kFpDigits) {
    // a CTA that may still allocate TMEM keeps the next one of its kernel off the SM
    if (threadIdx.x < 32) asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    contract_fma(t, it, b, g, base, part, raw);
    return;
  }
  fx::Smem& sm = fx::smem_at(raw);
  const uint32_t tmem = fx::open(sm);
  const int rs = (int)g.rs;  // (128: offsets within a block of points fit 32 bits)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = it.tm * kFpDigitRows, c0 = it.tn * kFpDigitCols;
  const int rows = min(kFpDigitRows, b.m - r0), cols = min(kFpDigitCols, b.n - c0);
  const int K = (int)g.K;  // below 2^31 - 256 (the planner checks)
  const int k0 = it.chunk * b.win_per * kFpWin, k1 = (int)min((int64_t)K, (int64_t)k0 + (int64_t)b.win_per * kFpWin);
  // this thread's operand rows (element offsets from base; the second one -1: none)
  int ax[2], ay[2], bx, by;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int2 q = t.pairs[b.a_off + r0 + min(fx::a_row(u), rows - 1)];
    ax[u] = q.x * rs;
    ay[u] = q.y >= 0 ? q.y * rs : -1;
  }
  {
    const int2 q = t.pairs[b.b_off + c0 + min(fx::b_col(), cols - 1)];
    bx = q.x * rs;
    by = q.y >= 0 ? q.y * rs : -1;
  }
  double acc[16] = {};
  uint32_t phase = 0, win = 0;
  bool ok = true, run = true;
  bool issued = true;  // (no MMA in flight where none was)
  if (hold) {  // failure-detection test: a raised flag holds the CTA back until the wait limit runs out
    if (threadIdx.x == 0) {
      const uint64_t t0 = mma::global_ns();
      while ((ok = *(volatile const int*)hold == 0) == false && mma::global_ns() - t0 <= wait_ns) {
      }
    }
    issued = run = __syncthreads_and(ok);
  }
  // A window ends where a mu row of cells does as well: its last points lie at one nucleus, the next ones
  // at the other, and two to ten times as many elements would take the chain (psq_fx.cuh).  Points
  // [from, to) of an aligned window.
  const uint32_t row_pts = (uint32_t)(g.n_nu * g.n_phi * g.q_mu * g.q_nu * g.q_phi);
  uint32_t cut = ((uint32_t)k0 / row_pts + 1) * row_pts;  // (below 2^32)
  for (int from = k0; from < k1 && run; ++win) {
    if (cut > g.K_reg) cut = ~0u;
    const int k = from & -kFpWin, to = (int)min(cut, (uint32_t)min(k + kFpWin, k1));
    const bool whole = to - from == kFpWin;
    double va[4][8], vb[2][4];
    const double* win0 = base + (int64_t)(k >> 7) * g.ws + (k & 127);  // the window's first point (row 0)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        double(&v)[8] = va[2 * c + u];
        const double* at = win0 + fx::a_pt(c);
        if (whole && 64 * u + 8 * warp < rows) {
          const double2* x = reinterpret_cast<const double2*>(at + ax[u]);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const double2 q = __ldg(x + i);
            v[2 * i] = q.x;
            v[2 * i + 1] = q.y;
          }
          if (ay[u] >= 0) {
            const double2* y = reinterpret_cast<const double2*>(at + ay[u]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const double2 q = __ldg(y + i);
              v[2 * i] *= q.x;
              v[2 * i + 1] *= q.y;
            }
          }
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            v[i] = 0.0;
            const int p = k + fx::a_pt(c) + i;
            if (64 * u + 8 * warp < rows && p >= from && p < to) v[i] = at[ax[u] + i] * (ay[u] >= 0 ? at[ay[u] + i] : 1.0);
          }
        }
      }
      const double* at = win0 + fx::b_pt(c);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        vb[c][i] = 0.0;
        const int p = k + fx::b_pt(c) + i;
        if (fx::b_col() < cols && (whole || (p >= from && p < to))) vb[c][i] = __ldg(at + bx + i) * (by >= 0 ? __ldg(at + by + i) : 1.0);
      }
    }
    run = fx::window(sm, tmem, va, vb, acc, phase, win, rows, cols, ok,
                     ItemChain{t.items + blockIdx.x, t.gblocks, t.grids, t.pairs, ops, from, to}, wait_ns);
    if ((uint32_t)to == cut) cut += row_pts;
    from = to;
  }
  if (run) run = __syncthreads_and(ok);
  if (!run && threadIdx.x == 0) atomicCAS(status, 0, 9);  // a wait that ran out (the first failure's code stays)
  double* out = part + b.part_off + (int64_t)it.chunk * b.m * b.n;
  const int r = 32 * (warp & 3) + lane;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int c = 16 * (warp >> 2) + j;
    // a wait that ran out leaves NaN as well: no result is better than a wrong one
    if (r < rows && c < cols) out[(int64_t)(r0 + r) * b.n + c0 + c] = run ? acc[j] : __longlong_as_double(0x7ff8000000000000ll);
  }
  fx::close(sm, tmem, run || !issued, phase);
}

cudaError_t prepare_kernels_fp64() {
  cudaError_t e = cudaFuncSetAttribute(eval_fp64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kEvalFp64Smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(contract_fp64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fx::kSmemBytes);
  // room for two CTAs per SM (of 228 KB), the rest L1
  return e != cudaSuccess ? e : cudaFuncSetAttribute(contract_fp64_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 80);
}

cudaError_t launch_contract_fp64(const LaunchTables& t, const double* ops, double* part, int* status, uint64_t wait_ns,
                                 const int* hold, cudaStream_t s) {
  if (t.n_items == 0) return cudaSuccess;
  contract_fp64_kernel<<<t.n_items, fx::kThreads, fx::kSmemBytes, s>>>(t, ops, part, status, wait_ns, hold);
  return cudaGetLastError();
}

// Per-element reduction of chunk partials: one warp per output element, lanes stride the
// chunks in a fixed order and combine by a shuffle tree (deterministic).
__global__ void __launch_bounds__(256) reduce_kernel(LaunchTables t, const double* __restrict__ part,
                                                      double* __restrict__ res) {
  const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (wid >= t.n_elems) return;
  int lo = 0, hi = t.n_gblocks;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (t.elem_begin[mid] <= wid) lo = mid; else hi = mid;
  }
  const GemmBlock b = t.gblocks[lo];
  const int64_t e = wid - t.elem_begin[lo];
  const int64_t mn = (int64_t)b.m * b.n;
  double s = 0.0;
  for (int c = lane; c < b.n_chunks; c += 32) s += part[b.part_off + c * mn + e];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) res[b.res_off + e] = s;
}

cudaError_t launch_reduce(const LaunchTables& t, const double* part, double* res, cudaStream_t s) {
  if (t.n_elems == 0) return cudaSuccess;
  const int64_t threads = t.n_elems * 32;
  reduce_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(t, part, res);
  return cudaGetLastError();
}

// k! / z^(k+1) = int_0^inf r^k e^(-z r) dr (k >= 0), as a product of k + 1 factors.
__device__ double radial_moment(int k, double z) {
  double v = 1.0 / z;
  for (int i = 1; i <= k; ++i) v *= (double)i / z;
  return v;
}

// One-centre overlap (cls 1) or kinetic (cls 2) element of two basis functions of one atom,
// from the closed forms of eq 1's functions: with I(k) = k! / (zeta_a + zeta_b)^(k+1), for the
// same l and m S = N_a N_b I(n_a + n_b) and T = -1/2 N_a N_b [(n_b (n_b - 1) - l (l + 1))
// I(n_a + n_b - 2) - 2 n_b zeta_b I(n_a + n_b - 1) + zeta_b^2 I(n_a + n_b)] (the radial
// Laplacian written out), symmetrised; 0 for different l or m.
__device__ double one_centre_st(int cls, const DevShell& A, int ma, const DevShell& B, int mb) {
  if (A.l != B.l || ma != mb) return 0.0;
  const double z = A.zeta + B.zeta, nn = A.norm * B.norm;
  const int k = A.n + B.n;
  if (cls == 1) return nn * radial_moment(k, z);
  const double ll = (double)(A.l * (A.l + 1));
  const double i2 = radial_moment(k - 2, z), i1 = radial_moment(k - 1, z), i0 = radial_moment(k, z);
  const double tab = (B.n * (B.n - 1) - ll) * i2 - 2.0 * B.n * B.zeta * i1 + B.zeta * B.zeta * i0;
  const double tba = (A.n * (A.n - 1) - ll) * i2 - 2.0 * A.n * A.zeta * i1 + A.zeta * A.zeta * i0;
  return -0.25 * nn * (tab + tba);
}

// Molecule matrices from per-grid blocks.  cls: 1 S, 2 T, 4 V, 8 J2 (two-index), 16 J3.
// With `shells`, one-centre elements take their closed forms (S and T).
//
// The matrices do not depend on one another, and each kernel is a short chain of dependent loads: from
// the second on, a kernel is launched as the programmatic dependent of the one before it (it starts
// when that one has started, so after the sums it reads are complete) and ends after it, so that
// whatever follows the last one follows them all.
// Measured: H2 (five matrices of 10 and 20 functions) 210.7 -> 193.8 us a call in FP64, 170.4 -> 160.1 us as a
// graph; bent triatomic, mixed, 1.422 -> 1.401 ms.
__device__ __forceinline__ void assemble_begin() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void assemble_end() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void assemble2_element(int64_t idx, int cls, int nat, int nfn, const int* __restrict__ fn_atom,
                                                  const int* __restrict__ fn_local, const SrcEntry* __restrict__ src,
                                                  const int* __restrict__ src_ptr, const DevShell* __restrict__ shells,
                                                  const int* __restrict__ fn_shell, const double* __restrict__ res,
                                                  double* __restrict__ out) {
  const int a = (int)(idx / nfn), b = (int)(idx % nfn);
  int X = fn_atom[a], Y = fn_atom[b], la = fn_local[a], lb = fn_local[b];
  if (shells && X == Y) {
    const DevShell& A = shells[fn_shell[a]];
    const DevShell& B = shells[fn_shell[b]];
    out[idx] = one_centre_st(cls, A, la - A.fn0, B, lb - B.fn0);
    return;
  }
  if (X > Y) { int t = X; X = Y; Y = t; t = la; la = lb; lb = t; }
  double v = 0.0;
  for (int e = src_ptr[X * nat + Y]; e < src_ptr[X * nat + Y + 1]; ++e) {
    const SrcEntry s = src[e];
    const double* M = res + s.off;
    if (s.mode == 0) {
      const double m1 = M[(int64_t)(s.rX + la) * s.ld + s.cY + lb];
      if (cls == 2 || cls == 8 || X == Y) {
        const double* M2 = s.ld2 > 0 ? res + s.off2 : M;
        const double m2 = M2[(int64_t)(s.rY + lb) * (s.ld2 > 0 ? s.ld2 : s.ld) + s.cX + la];
        v += (cls == 2 ? -0.25 : s.z * 0.5) * (m1 + m2);
      } else {
        v += s.z * m1;
      }
    } else {
      int64_t p;
      if (s.mode == 1) {
        const int i = min(s.rX + la, s.cY + lb), j = max(s.rX + la, s.cY + lb);
        p = (int64_t)i * s.nloc - (int64_t)i * (i - 1) / 2 + (j - i);
      } else {
        p = (int64_t)la * s.nloc + lb;
      }
      v += s.z * M[p * s.ld + (int64_t)s.cX * s.cs];
    }
  }
  out[idx] = v;
}

__global__ void assemble2_kernel(int cls, int nat, int nfn, const int* __restrict__ fn_atom,
                                 const int* __restrict__ fn_local, const SrcEntry* __restrict__ src,
                                 const int* __restrict__ src_ptr, const DevShell* __restrict__ shells,
                                 const int* __restrict__ fn_shell, const double* __restrict__ res,
                                 double* __restrict__ out) {
  assemble_begin();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < (int64_t)nfn * nfn) assemble2_element(idx, cls, nat, nfn, fn_atom, fn_local, src, src_ptr, shells, fn_shell, res, out);
  assemble_end();
}

__device__ __forceinline__ void assemble3_element(int64_t idx, int64_t nn, int nat, int nfn, const int* __restrict__ fn_atom,
                                                  const int* __restrict__ fn_local, const int* __restrict__ aux_atom,
                                                  const int* __restrict__ aux_local, const J3Src* __restrict__ j3,
                                                  const double* __restrict__ res, double* __restrict__ out) {
  const int P = (int)(idx / nn);
  const int a = (int)((idx / nfn) % nfn), b = (int)(idx % nfn);
  const int X = aux_atom[P], lp = aux_local[P];
  int Y = fn_atom[a], W = fn_atom[b], la = fn_local[a], lb = fn_local[b];
  if (Y > W) { int t = Y; Y = W; W = t; t = la; la = lb; lb = t; }
  const J3Src s = j3[((int64_t)X * nat + Y) * nat + W];
  int64_t pidx;
  const int i0 = s.offY + la, j0 = s.offW + lb;
  if (s.mode == 1) {
    const int i = min(i0, j0), j = max(i0, j0);
    pidx = (int64_t)i * s.nloc - (int64_t)i * (i - 1) / 2 + (j - i);
  } else {
    pidx = (int64_t)i0 * s.nloc + j0;
  }
  out[idx] = res[s.off + pidx * s.s_pair + (int64_t)lp * s.s_aux];
}

__global__ void assemble3_kernel(int nat, int nfn, int naux, const int* __restrict__ fn_atom,
                                 const int* __restrict__ fn_local, const int* __restrict__ aux_atom,
                                 const int* __restrict__ aux_local, const J3Src* __restrict__ j3,
                                 const double* __restrict__ res, double* __restrict__ out) {
  assemble_begin();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nn = (int64_t)nfn * nfn;
  if (idx < nn * naux) assemble3_element(idx, nn, nat, nfn, fn_atom, fn_local, aux_atom, aux_local, j3, res, out);
  assemble_end();
}

cudaError_t launch_assemble(int cls, int nat, int nfn, int naux, const int* fn_atom,
                            const int* fn_local, const int* aux_atom, const int* aux_local,
                            const SrcEntry* src, const int* src_ptr, const J3Src* j3,
                            const DevShell* shells, const int* fn_shell, const double* res, double* out,
                            bool dependent, cudaStream_t s) {
  const int64_t n = cls == 16 ? (int64_t)naux * nfn * nfn : (int64_t)nfn * nfn;
  if (n == 0) return cudaSuccess;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)((n + 255) / 256));
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = dependent ? 1 : 0;
  return cls == 16 ? cudaLaunchKernelEx(&cfg, assemble3_kernel, nat, nfn, naux, fn_atom, fn_local, aux_atom, aux_local, j3, res, out)
                   : cudaLaunchKernelEx(&cfg, assemble2_kernel, cls, nat, nfn, fn_atom, fn_local, src, src_ptr, shells, fn_shell,
                                        res, out);
}

// Diagnostics: the points of one grid (8 rows: x, y, z, w, r_A, r_B, mu, nu).
__global__ void grid_points_kernel(const DevGrid* grids, int gi, const double* edges, double* out) {
  const DevGrid& g = grids[gi];
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= g.K) return;
  Pt pt;
  ps_point(g, edges, p, pt);
  const int64_t K = g.K;
  out[0 * K + p] = pt.P[0];
  out[1 * K + p] = pt.P[1];
  out[2 * K + p] = pt.P[2];
  out[3 * K + p] = pt.w;
  out[4 * K + p] = pt.rA;
  out[5 * K + p] = pt.rB;
  out[6 * K + p] = pt.mu;
  out[7 * K + p] = pt.nu;
}

cudaError_t launch_grid_points(const LaunchTables& t, int g, double* out, cudaStream_t s) {
  // the point count is on the device; the host passes it through n_elems
  const int64_t K = t.n_elems;
  if (K == 0) return cudaSuccess;
  grid_points_kernel<<<(unsigned)((K + 255) / 256), 256, 0, s>>>(t.grids, g, t.edges, out);
  return cudaGetLastError();
}

}  // namespace psq
