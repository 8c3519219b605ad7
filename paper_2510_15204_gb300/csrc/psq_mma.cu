// Mixed-precision path of the PS quadrature on sm_103a:
//  * node tables: the PS grid is a tensor product in (mu, nu, phi) per volume element, so the
//    per-node trigonometric factors (Section 2.1, eqs 2-6, 10-11) are computed once per grid
//    row in FP64 (nodes_kernel) and stored with double-float (FP32 hi + lo) copies;
//  * eval_mixed_kernel: point weights, focal distances and offsets in double-float from the
//    node tables (the cancellation-free forms), the third-centre offset in FP64 (it cancels
//    near that centre), STOs (eq 1), their kinetic operand and the aux potentials (eq 16,
//    incomplete gamma by its positive series below x = k) as double-float functions of
//    x = zeta r and the direction (psq_df.cuh); every constant factor of a row is left to FP64;
//  * pack_kernel: every operand row that a contraction tile reads whole is scaled by a power
//    of two per 128-point window (from the window's maximum) and cut into five integer slices
//    of at most 8 bits (exact in BF16; 39 bits of the window's largest value), stored as the
//    tcgen05 shared-memory image (64-byte rows of 32 points, 64-byte swizzle);
//  * contract_ws_kernel: the weighted contraction of eq 9 on tcgen05 tensor cores.  Packed
//    tiles arrive by bulk copies; the 3-index operand chi_i chi_j is formed (double-float
//    products) and sliced in shared memory from staged basis rows.  Per K step of 16 points
//    five MMAs (A slice i against B slices 0..4-i, contiguous in shared memory) accumulate
//    the slice products of orders 0..4 into five FP32 TMEM accumulators; all partial sums are
//    integers below 2^24, so the FP32 accumulation is exact.  After each window the
//    accumulators are scaled back and added into double-float registers; each work item
//    writes its point range's (hi, lo) sums, and reduce_mixed_kernel adds the ranges in FP64
//    and applies the FP64 constants of each row and column (normalisations, powers of zeta,
//    a^3), which the values omit.
#include "psq_internal.h"
#include "psq_df.cuh"
#include "psq_tc.cuh"
#include "psq_f2.cuh"

#include <cuda_bf16.h>

#include <cmath>
#include <cstdint>

namespace psq {

// ------------------------------------------------------------------ node tables

__constant__ double c_glx2[kMaxQ + 1][kMaxQ];
__constant__ double c_glw2[kMaxQ + 1][kMaxQ];
__constant__ float c_rcpf[128];           // 1/n (FP32 tails of the incomplete-gamma series)
__constant__ float2 c_factd[2 * kMaxN + 4];  // k! as (hi, lo)
__constant__ float2 c_exp_tab[64];        // 2^(-j/64) as (hi, lo)
__constant__ dfa::ExpConsts c_expc;

__host__ __device__ __forceinline__ float2 split_f(double v) {
  const float hi = (float)v;
  return make_float2(hi, (float)(v - (double)hi));
}

void upload_mixed_tables(const double* x, const double* w, const double* klm) {
  (void)klm;
  cudaMemcpyToSymbol(c_glx2, x, sizeof(double) * (kMaxQ + 1) * kMaxQ);
  cudaMemcpyToSymbol(c_glw2, w, sizeof(double) * (kMaxQ + 1) * kMaxQ);
  float2 f[2 * kMaxN + 4];
  double fd = 1.0;
  f[0] = split_f(1.0);
  for (int i = 1; i < 2 * kMaxN + 4; ++i) {
    fd *= i;
    f[i] = split_f(fd);
  }
  cudaMemcpyToSymbol(c_factd, f, sizeof(f));
  float r[128];
  r[0] = 0.0f;
  for (int i = 1; i < 128; ++i) r[i] = (float)(1.0 / i);
  cudaMemcpyToSymbol(c_rcpf, r, sizeof(r));
  float2 t[64];
  for (int j = 0; j < 64; ++j) t[j] = split_f(std::exp2(-j / 64.0));
  cudaMemcpyToSymbol(c_exp_tab, t, sizeof(t));
  // ln2/64 = c1 + c2 + c3, c1 rounded to 10 significant bits
  const double l64 = 0.693147180559945309417232121458 / 64.0;
  int e2 = 0;
  std::frexp(l64, &e2);
  const double c1 = std::ldexp(std::nearbyint(std::ldexp(l64, 10 - e2)), e2 - 10);
  const float c2 = (float)(l64 - c1);
  const float c3 = (float)(l64 - c1 - (double)c2);
  dfa::ExpConsts ec{(float)(64.0 / 0.693147180559945309417232121458), (float)c1, c2, c3};
  cudaMemcpyToSymbol(c_expc, &ec, sizeof(ec));
}

// Entry (row, node) of one dimension: rows 0..N-1 are the volume-element rows, then
// N_SP sub-rows of each touching row.  dim 0 = mu, 1 = nu, 2 = phi.
__global__ void nodes_kernel(const DevGrid* __restrict__ grids, const double* __restrict__ edges,
                             NodeEntry* __restrict__ tab) {
  const DevGrid& g = grids[blockIdx.y];
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  const int nmu = (g.n_mu + g.nt_mu * g.n_sp) * g.q_mu;
  const int nnu = (g.n_nu + g.nt_nu * g.n_sp) * g.q_nu;
  const int nph = (g.n_phi + g.nt_phi * g.n_sp) * g.q_phi;
  if (e >= nmu + nnu + nph) return;
  int dim, idx, N, Q, t0;
  const double* ed = edges + g.edge_off;
  if (e < nmu) {
    dim = 0; idx = e; N = g.n_mu; Q = g.q_mu; t0 = g.t_mu0;
  } else if (e < nmu + nnu) {
    dim = 1; idx = e - nmu; N = g.n_nu; Q = g.q_nu; t0 = g.t_nu0; ed += g.n_mu + 1;
  } else {
    dim = 2; idx = e - nmu - nnu; N = g.n_phi; Q = g.q_phi; t0 = 0; ed += g.n_mu + 1 + g.n_nu + 1;
  }
  const int row = idx / Q, q = idx % Q;
  double m0, m1;
  if (row < N) {
    m0 = ed[row];
    m1 = ed[row + 1];
  } else {
    const int t = (row - N) / g.n_sp, s = (row - N) % g.n_sp;
    int base;
    if (dim < 2) base = t0 + t;
    else base = g.t_phi_all ? t : (t == 0 ? 0 : g.n_phi - 1);
    const double M0 = ed[base], M1 = ed[base + 1];
    const int ns = g.n_sp;
    m0 = M0 + (M1 - M0) * s / ns;
    m1 = M0 + (M1 - M0) * (s + 1) / ns;
  }
  const double h = 0.5 * (m1 - m0);
  const double v = 0.5 * (m0 + m1) + h * c_glx2[Q][q];
  double s, c, h2, g2;
  if (dim == 0) {
    s = sinh(v);
    c = cosh(v);
    const double sh2 = sinh(0.5 * v);
    h2 = sh2 * sh2;
    g2 = 0.0;
  } else {
    sincos(v, &s, &c);
    double s2, c2;
    sincos(0.5 * v, &s2, &c2);
    h2 = s2 * s2;
    g2 = c2 * c2;
  }
  NodeEntry o;
  o.v = v;
  o.s = s;
  o.c = c;
  o.fs = split_f(s);
  o.fc = split_f(c);
  o.fh2 = split_f(h2);
  o.fg2 = split_f(g2);
  o.fw = split_f(h * c_glw2[Q][q]);
  tab[g.nt_off + e] = o;
}

// ------------------------------------------------------------------ mixed evaluation
//
// Every value is a double-float (hi, lo) pair (about 48 bits): the slices the contraction
// keeps reach 39 bits of each 128-point window's largest value, so the function values must
// carry more than that.

using dfa::df;

__device__ __forceinline__ df ld2(float2 v) { return df{v.x, v.y}; }

// Highest l and number of functions of the shells [s0, s1).
__device__ __forceinline__ int shells_lmax_f(const DevShell* sh, int s0, int s1) {
  int l = 0;
  for (int s = s0; s < s1; ++s) l = max(l, sh[s].l);
  return l;
}

// One row kind of a shell at one point: the radial value times the harmonics, to the hi and lo planes.
__device__ __forceinline__ void store_shell(const DevShell& q, df r, const df* Y, float* __restrict__ oh,
                                            float* __restrict__ ol, int64_t rs, int64_t p, int row) {
  const int base = q.l * q.l + q.l;
  int64_t o = (int64_t)(row + q.fn0) * rs + p;
#pragma unroll 1
  for (int m = -q.l; m <= q.l; ++m, o += rs) {
    const df v = dfa::mul(r, Y[base + m]);
    oh[o] = v.h;
    ol[o] = v.l;
  }
}

// u = R v / len (R as a double-float matrix), the unit vector of the offset v of length len.
__device__ __forceinline__ void rotate_unit_df(const DevGrid& g, df vx, df vy, df vz, df inv_len, df* u) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const df r0{g.Rh[c * 3], g.Rl[c * 3]}, r1{g.Rh[c * 3 + 1], g.Rl[c * 3 + 1]}, r2{g.Rh[c * 3 + 2], g.Rl[c * 3 + 2]};
    const df d = dfa::add(dfa::add(dfa::mul(r0, vx), dfa::mul(r1, vy)), dfa::mul(r2, vz));
    u[c] = dfa::mul(d, inv_len);
  }
}

__device__ __forceinline__ df split_d(double v) {
  const float hi = (float)v;
  return df{hi, (float)(v - (double)hi)};
}

// One CTA per PointBlock.  The weight w = a^3 [G G G sinh mu sin nu (sinh^2 mu + sin^2 nu)]
// and r_A = 2a rho_A, r_B = 2a rho_B are written without their per-grid constants (a^3,
// a^2/2), which are applied in FP64 after the contraction; functions likewise.  The offsets
// from A and B (in units of a) are (sinh mu sin nu cos phi, sinh mu sin nu sin phi,
// 2(sinh^2(mu/2) cos nu -+ {sin^2, cos^2}(nu/2))), of length 2 rho; the offset from a third
// centre is formed in FP64 (it cancels near that centre).
//
// The radial factors (e^-x, powers, incomplete gamma series) are most of the arithmetic, and those of
// A and B depend on (mu, nu) only: they are computed once per node pair and kept in shared memory for
// all phi nodes (32 points share one on an 8-cell grid with Q = 4); those of a third centre are
// computed for half of the phi nodes.  A point is then its harmonics and one product per function.
// FP32 issue bounds it.  Measured (radial factors per point -> shared): bent triatomic (963,072 points)
// 0.58 -> 0.36 ms, nine atoms (55.7 M points) 45.0 -> 33.2 ms.
__global__ void __launch_bounds__(kEvalThreads) eval_mixed_kernel(LaunchTables t, const NodeEntry* __restrict__ tab,
                                                                  const float2* __restrict__ xi_tab,
                                                                  float* __restrict__ ops, float* __restrict__ ops_lo) {
  extern __shared__ __align__(16) uint8_t raw[];
  __shared__ float2 etab[64];
  __shared__ int meta[5];  // lmax of A, B, C; functions of the first aux centre
  __shared__ CentreShells shells[3];
  const int tid = threadIdx.x;
  if (tid < 64) etab[tid] = c_exp_tab[tid];
  const PointBlock pb = t.pblocks[blockIdx.x];
  const DevGrid& g = t.grids[pb.grid];
  const bool third = g.C >= 0;
  const int np = pb.pr1 - pb.pr0, nn = (pb.u1 - pb.u0) * g.q_phi;  // node pairs, phi nodes of the half
  const int nbA = g.shb_A1 - g.shb_A0, nbB = g.shb_B1 - g.shb_B0, na0 = g.sha_1 - g.sha_0, na1 = g.sha_3 - g.sha_2;
  const bool basis = g.row_F >= 0 || g.row_L >= 0, aux = g.row_G >= 0 || g.row_U >= 0;
  const int n_pair = nbA + nbB + (third ? 0 : na0 + na1);  // shells with a value per node pair
  float2* tp = reinterpret_cast<float2*>(raw);             // [2 shell + kind][pair]
  const int p0 = min(pb.s0, n_pair), p1 = min(pb.s1, n_pair);  // this CTA's shells: of those,
  const int q0 = third ? max(pb.s0 - n_pair, 0) : 0, q1 = third ? max(pb.s1 - n_pair, 0) : 0;  // and of C
  float2* tr = tp + 2 * (p1 - p0) * np;                    // [phi node][pair]: distance from C
  float2* tc = tr + (third ? nn * np : 0);                 // [shell of C][phi node][pair]
  // the column's node rows
  const int nreg = g.n_mu * g.n_nu, ns = g.n_sp;
  const bool reg = pb.col < nreg;
  int ri, rj, nu_rows;
  int64_t cell0;       // first point of the column's phi row 0
  int64_t cell_s1, cell_s2;  // point strides of phi cells and of their sub-rows
  const int q3 = g.q_mu * g.q_nu * g.q_phi;
  bool touch = false;
  if (reg) {
    ri = pb.col / g.n_nu;
    rj = pb.col - ri * g.n_nu;
    nu_rows = g.n_phi;
    cell0 = (int64_t)pb.col * g.n_phi * q3;
    cell_s1 = q3;
    cell_s2 = 0;
    touch = g.n_touch > 0 && ri >= g.t_mu0 && ri <= g.t_mu1 && rj >= g.t_nu0 && rj <= g.t_nu1;
  } else {
    const int c = pb.col - nreg, sub = c % (ns * ns), tij = c / (ns * ns);
    const int ti = tij / g.nt_nu, tj = tij - ti * g.nt_nu, si = sub / ns, sj = sub - si * ns;
    ri = g.n_mu + ti * ns + si;
    rj = g.n_nu + tj * ns + sj;
    nu_rows = g.nt_phi * ns;
    cell0 = g.K_reg + ((int64_t)tij * g.nt_phi * ns * ns * ns + (si * ns + sj) * ns) * q3;
    cell_s1 = (int64_t)ns * ns * ns * q3;
    cell_s2 = q3;
  }
  const NodeEntry* Mu = tab + g.nt_off + ri * g.q_mu;
  const NodeEntry* Nu = tab + g.nt_off + (g.n_mu + g.nt_mu * ns) * g.q_mu + rj * g.q_nu;
  const NodeEntry* Ph = tab + g.nt_off + (g.n_mu + g.nt_mu * ns) * g.q_mu + (g.n_nu + g.nt_nu * ns) * g.q_nu +
                        (reg ? 0 : g.n_phi * g.q_phi);  // rows of the column's phi rows, in order
  if (tid == 0) {
    const bool auxA = !third;
    meta[0] = max(basis ? shells_lmax_f(t.bshell, g.shb_A0, g.shb_A1) : 0, aux && auxA ? shells_lmax_f(t.ashell, g.sha_0, g.sha_1) : 0);
    meta[1] = max(basis ? shells_lmax_f(t.bshell, g.shb_B0, g.shb_B1) : 0, aux && auxA ? shells_lmax_f(t.ashell, g.sha_2, g.sha_3) : 0);
    meta[2] = third && aux ? shells_lmax_f(t.ashell, g.sha_0, g.sha_1) : 0;
    int nf = 0;
    for (int s = g.sha_0; s < g.sha_1; ++s) nf += 2 * t.ashell[s].l + 1;
    meta[3] = nf;
    for (int c = 0; c < 3; ++c) shells[c] = centre_shells(g, pb, c);
  }
  // third centre: distances at the phi nodes of the half, FP64 offsets
  if (third) {
    for (int e = tid; e < nn * np; e += kEvalThreads) {
      const int f = e / np, pr = pb.pr0 + e - f * np, qi = pr / g.q_nu, qj = pr - qi * g.q_nu;
      const NodeEntry &M = Mu[qi], &N = Nu[qj], &F = Ph[pb.u0 * g.q_phi + f];
      const df dX = split_d(g.a * M.s * N.s * F.c - g.xc), dY = split_d(g.a * M.s * N.s * F.s), dZ = split_d(g.a * M.c * N.c - g.zc);
      const df r = dfa::sqrt(dfa::add_same(dfa::add_same(dfa::mul(dX, dX), dfa::mul(dY, dY)), dfa::mul(dZ, dZ)));
      tr[e] = make_float2(r.h, r.l);
    }
  }
  __syncthreads();
  const float2* xi = xi_tab + g.xi_off;  // basis A, basis B, aux c0, aux c1 shells
  for (int e = tid; e < (p1 - p0) * np; e += kEvalThreads) {
    const int i = e / np, s = p0 + i, pq = e - i * np, pr = pb.pr0 + pq, qi = pr / g.q_nu, qj = pr - qi * g.q_nu;
    const bool isb = s < nbA + nbB, onA = isb ? s < nbA : s < nbA + nbB + na0;
    if (isb ? !basis : !aux) continue;
    const DevShell& q = isb ? t.bshell[s < nbA ? g.shb_A0 + s : g.shb_B0 + s - nbA]
                            : t.ashell[onA ? g.sha_0 + s - nbA - nbB : g.sha_2 + s - nbA - nbB - na0];
    const df rho = dfa::add_same(ld2(Mu[qi].fh2), onA ? ld2(Nu[qj].fh2) : ld2(Nu[qj].fg2));
    const df x = dfa::mul(ld2(xi[s]), rho), ex = dfa::exp_neg(x, c_expc, etab), ix = dfa::rcp(x);
    const bool ka = isb ? g.row_F >= 0 : g.row_G >= 0, kb = isb ? g.row_L >= 0 : g.row_U >= 0;
    if (ka) {
      const df r = dfa::radial(0, q.n, q.l, x, ex, ix, c_factd, c_rcpf);
      tp[2 * i * np + pq] = make_float2(r.h, r.l);
    }
    if (kb) {
      const df r = dfa::radial(isb ? 1 : 2, q.n, q.l, x, ex, ix, c_factd, c_rcpf);
      tp[(2 * i + 1) * np + pq] = make_float2(r.h, r.l);
    }
  }
  if (third && aux) {
    const int kind = g.row_U >= 0 ? 2 : 0;  // (a refined grid has one aux kind)
    for (int e = tid; e < (q1 - q0) * nn * np; e += kEvalThreads) {
      const int i = e / (nn * np);
      const DevShell& q = t.ashell[g.sha_0 + q0 + i];
      const df x = dfa::mul(ld2(xi[n_pair + q0 + i]), ld2(tr[e - i * nn * np]));
      const df r = dfa::radial(kind, q.n, q.l, x, dfa::exp_neg(x, c_expc, etab), dfa::rcp(x), c_factd, c_rcpf);
      tc[e] = make_float2(r.h, r.l);
    }
  }
  __syncthreads();
  // the points: phi rows u0 .. u1 - 1 and their mirrors
  float* bh = ops + g.op_off;
  float* bl = ops_lo + g.op_off;
  const int64_t rs = g.rs;
  const int per = np * g.q_phi, nu = pb.u1 - pb.u0;
  df Y[(kMaxL + 1) * (kMaxL + 1)];
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
    const NodeEntry &M = Mu[qi], &N = Nu[qj], &F = Ph[u * g.q_phi + qk];
    const df sh = ld2(M.fs), s2m = ld2(M.fh2), sn = ld2(N.fs), s2n = ld2(N.fh2), c2n = ld2(N.fg2);
    const df shsn = dfa::mul(sh, sn);
    const df rhoA = dfa::add_same(s2m, s2n), rhoB = dfa::add_same(s2m, c2n);
    df rC = dfa::mk(1.0f);
    if (third) rC = ld2(tr[f * np + pq]);
    if (g.row_W >= 0 && pb.s0 == 0) {
      df w = dfa::mk(0.0f);
      if (!dead) {
        const df gw = dfa::mul(dfa::mul(ld2(M.fw), ld2(N.fw)), ld2(F.fw));
        w = dfa::mul(dfa::mul(gw, shsn), dfa::add_same(dfa::mul(sh, sh), dfa::mul(sn, sn)));
      }
      const df wv[4] = {w, dfa::div(w, rhoA), dfa::div(w, rhoB), third ? dfa::div(w, rC) : dfa::mk(0.0f)};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        bh[(int64_t)(g.row_W + k) * rs + p] = wv[k].h;
        bl[(int64_t)(g.row_W + k) * rs + p] = wv[k].l;
      }
    }
    const df xs = dfa::mul(shsn, ld2(F.fc)), ys = dfa::mul(shsn, ld2(F.fs)), s2mc = dfa::mul(s2m, ld2(N.fc));
#pragma unroll 1
    for (int ctr = 0; ctr < 3; ++ctr) {  // A, B, C
      const CentreShells& own = shells[ctr];
      const int b0 = own.b0, b1 = own.b1, a0 = own.a0, a1 = own.a1;
      const bool hb = basis && ctr < 2 && b1 > b0, ha = aux && (ctr == 2) == third && a1 > a0;
      if (!hb && !ha) continue;
      df u3[3];
      if (ctr < 2) {
        const df z = ctr == 0 ? dfa::sub(s2mc, s2n) : dfa::add(s2mc, c2n);
        rotate_unit_df(g, xs, ys, dfa::scale2(z, 2.0f), dfa::rcp(dfa::scale2(ctr == 0 ? rhoA : rhoB, 2.0f)), u3);
      } else {
        rotate_unit_df(g, split_d(g.a * M.s * N.s * F.c - g.xc), split_d(g.a * M.s * N.s * F.s),
                       split_d(g.a * M.c * N.c - g.zc), dfa::rcp(rC), u3);
      }
      dfa::real_ylm(meta[ctr], u3[0], u3[1], u3[2], Y, c_rcpf);
      if (hb) {
        const int roff = ctr == 0 ? 0 : g.nFA;
#pragma unroll 1
        for (int s = b0; s < b1; ++s) {
          const DevShell& q = t.bshell[s];
          const float2* tv = tp + 2 * (s + own.bt) * np + pq;
          if (g.row_F >= 0) store_shell(q, ld2(tv[0]), Y, bh, bl, rs, p, g.row_F + roff);
          if (g.row_L >= 0) store_shell(q, ld2(tv[np]), Y, bh, bl, rs, p, g.row_L + roff);
        }
      }
      if (ha) {
        const int roff = ctr == 1 ? meta[3] : 0;
#pragma unroll 1
        for (int s = a0; s < a1; ++s) {
          const DevShell& q = t.ashell[s];
          if (ctr == 2) {
            store_shell(q, ld2(tc[((s + own.at) * nn + f) * np + pq]), Y, bh, bl, rs, p, g.row_U >= 0 ? g.row_U : g.row_G);
          } else {
            const float2* tv = tp + 2 * (s + own.at) * np + pq;
            if (g.row_G >= 0) store_shell(q, ld2(tv[0]), Y, bh, bl, rs, p, g.row_G + roff);
            if (g.row_U >= 0) store_shell(q, ld2(tv[np]), Y, bh, bl, rs, p, g.row_U + roff);
          }
        }
      }
    }
  }
}

// ------------------------------------------------------------------ tcgen05 contraction

namespace mma {

constexpr int kM = kMmaM;
constexpr int kTileN = kMmaN;
constexpr int kChunk = kChunkPts;
constexpr int kRowB = 2 * kChunkPts;            // bytes of one operand row of a stage (64)
constexpr int kARingBytes = 147456;             // A ring: 3 chunks of 128 rows (40 KB each), more of fewer rows
constexpr int kMaxStages = 8;
constexpr int kStagesB = 3;                     // B ring depth (chunks, 15 KB each)
constexpr int kChunksPerWin = kWinPts / kChunkPts;

// Instruction descriptor: kind::f16, A = B = BF16, D = F32, both K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t make_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
}

__device__ __forceinline__ float pow2f(int k) {
  if (k < -126) return 0.0f;
  if (k > 127) k = 127;
  return __int_as_float((k + 127) << 23);
}

}  // namespace mma

// ------------------------------------------------------------------ operand packing
//
// Every operand row that a tile reads as a whole (weighted aux potentials, weighted kinetic
// operands, basis and aux functions) is sliced once per job into the tcgen05 shared-memory
// image by pack_kernel; the contraction then moves it with bulk copies.  Only the 3-index
// operand chi_i chi_j, whose rows are products of two basis rows, is formed inside the
// contraction, from basis rows staged in shared memory.
//
// Slicing.  A row's values in a 128-point window are scaled by 2^(7-e) (|v| < 2^e over the
// window) and cut into five digits v ~ s0 + s1/256 + ... + s4/256^4 of integers (each the
// nearest integer of what the previous digits left, times 256), exact in BF16: 39 bits of the
// window's largest value.  Values are double-float pairs, products of two pairs left
// unnormalised (|lo| <= 3 2^-24 |hi|); the first two digits come from the hi part (exactly),
// then the lo part joins the remainder, which rounds once, at 2^-17 of the third digit's unit
// (2^-40 of the window's largest value); s2 can reach 130.  Accumulation bound: the order-k
// sum sum_{i+j=k} s_i t_j over 128 points stays below 128 x 114688 < 2^24 for every k <= 4,
// so the FP32 tensor-core accumulators hold it exactly.

namespace mma {

// The lo parts join the remainder after digit kJoin = 1: products are left unnormalised (|lo| <= 3 2^-24
// |hi|: the join adds at most 1.5 to s2, which stays <= 130, and rounds at 2^-17 of s2's unit,
// 2^-40 of the window's largest value).
//
// Each digit takes three full-rate FP32 instructions (packed: for two values).  With M = 1.5 x 2^23 and |x| < 2^22,
// t = x + M rounds x to its nearest integer s (ties to even): t lies in [2^23, 2^24), where the
// spacing is 1, so t = M + s exactly.  Then fma(t, -256, 256 M) = -256 s and
// fma(x, 256, -256 s) = 256 (x - s) are exact (|x - s| <= 1/2 is a multiple of x's spacing).
// The stored digit is -256 s, exact in BF16 like s (at most 8 significant bits); every operand
// is stored this way, so a slice product carries 2^16, which keeps the order sums exact in FP32
// (multiples of 2^16 below 2^40) and which the fold removes with the window scales.
constexpr float kRneMagic = 12582912.0f;         // 1.5 x 2^23
constexpr float kRneMagic256 = 3221225472.0f;    // 256 x 1.5 x 2^23 = 1.5 x 2^31
constexpr int kDigitScaleExp = 8;                // |stored digit| = 2^8 |s|
constexpr int kJoin = 1;

// BF16x2 bits of two floats that are exact in BF16 (at most 8 significant bits: their low 16
// bits are zero), first value in the low half.
__device__ __forceinline__ uint32_t pack_bf16_exact(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}

// The window scale of a row whose largest |value| is below 2^e, for the hi words (sc) and
// for the lo words joining after digit kJoin (sc 256^(kJoin + 1), capped at 2^127: rows below
// 2^-96, whose lo parts are below 2^-120, join them at a smaller weight).
__device__ __forceinline__ void window_scales(int e, float& sc, float& scj) {
  sc = e == kZeroExp ? 0.0f : pow2f(7 - e);
  scj = e == kZeroExp ? 0.0f : pow2f(7 - e + 8 * (kJoin + 1));
}

// The planes of 2 NP consecutive points (NP = 4: a 16-byte group) given as pairs, NP words each; the
// values are sgn vh + vl (sgn: the sign the hi words' scale sc carries).
template <int NP>
__device__ __forceinline__ void slice_f2(const f2 (&vh)[NP], const f2 (&vl)[NP], float sc, float scj, uint32_t (&o)[kSlices][NP]) {
  const f2 s0 = f2_both(sc), s256 = f2_both(sc * 256.0f), sj = f2_both(scj);  // |sc 256| at most 2^125
  const f2 magic = f2_both(kRneMagic), magic256 = f2_both(kRneMagic256), m256 = f2_both(-256.0f), p256 = f2_both(256.0f);
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    f2 r{};
    const f2 l = f2_mul(vl[q], sj);
#pragma unroll
    for (int k = 0; k < kSlices; ++k) {
      // digit 0 rounds v sc (exact: sc is a power of two) inside its first FMA
      const f2 t = k == 0 ? f2_fma(vh[q], s0, magic) : f2_add(r, magic);
      const f2 d = f2_fma(t, m256, magic256);
      float d0, d1;
      f2_unpack(d, d0, d1);
      o[k][q] = pack_bf16_exact(d0, d1);
      if (k + 1 < kSlices) {
        r = k == 0 ? f2_fma(vh[q], s256, d) : f2_fma(r, p256, d);
        if (k == kJoin) r = f2_add(r, l);
      }
    }
  }
}

// Exponent e with mx < 2^e <= 2 mx (frexp's), read from the exponent bits, or kZeroExp for
// a row that is zero (or below 2^-110; subnormal maxima count as zero).
__device__ __forceinline__ int row_exponent(float mx) {
  const int e = (int)(__float_as_uint(mx) >> 23) - 126;  // mx >= 0
  return e < -110 ? kZeroExp : e;
}

}  // namespace mma

// (xh + xl)(yh + yl) as hi = fl(xh yh) and the unnormalised lo = the exact error of that
// product plus the cross terms (|lo| <= 3 2^-24 |hi|; the lo lo term, below 2^-48, dropped).  The hi
// words come negated (the error of a product is one FMA from its negative).
__device__ __forceinline__ void prod_unnorm(f2 xh, f2 xl, f2 yh, f2 yl, f2& nh, f2& l) {
  nh = f2_mul(xh, f2_mul(yh, f2_both(-1.0f)));
  l = f2_fma(xl, yh, f2_fma(xh, yl, f2_fma(xh, yh, nh)));
}

// Decodes packing job `job` (panel, tile, window, 16-row group) for this thread: 8 threads per
// row, thread qq holding points [4 qq, 4 qq + 4) of each of the window's four chunks (half qq % 2 of
// 16-byte group qq / 2 of its row), so that the eight read 128 contiguous bytes and write whole
// 64-byte rows, four of them one after the other.
struct PackPos {
  int pn, t, w, r, qq;
};

// The panel of a job: from hint[job / kPackHintJobs] (the panel of that block's first job) by
// a short forward scan, or by bisection when there is no hint.
__device__ __forceinline__ PackPos pack_pos(int64_t job, const Panel* __restrict__ panels, int n_panels,
                                            const int* __restrict__ hint) {
  int lo = 0;
  if (hint) {
    lo = __ldg(hint + (job / kPackHintJobs));
    while (lo + 1 < n_panels && panels[lo + 1].job_begin <= job) ++lo;
  } else {
    int hi = n_panels;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (panels[mid].job_begin <= job) lo = mid; else hi = mid;
    }
  }
  const Panel& pn = panels[lo];
  const int G = pn.tr / kPackRows;
  const int lj = (int)(job - pn.job_begin);  // jobs of one panel < 2^31 (one launch's grid)
  const int tw = lj / G, grp = lj - tw * G;
  PackPos P;
  P.pn = lo;
  P.t = tw / pn.nwin;
  P.w = tw - P.t * pn.nwin;
  P.r = kPackRows * grp + (threadIdx.x >> 3);
  P.qq = threadIdx.x & 7;
  return P;
}

// The row's window exponent (the eight threads of the row share it) and the five planes of
// this thread's 4 x 4 points, sgn h + l (sgn = 1 or -1).
__device__ __forceinline__ void pack_store(const PackPos& P, const Panel& pn, const f2 (&h)[4][2], const f2 (&l)[4][2], float sgn,
                                           uint8_t* __restrict__ packed) {
  using namespace mma;
  float mx = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float a, b;
    f2_unpack(h[i >> 1][i & 1], a, b);
    mx = fmaxf(mx, fmaxf(fabsf(a), fabsf(b)));
  }
  const unsigned m8 = 0xffu << ((threadIdx.x & 31) & ~7u);
  mx = fmaxf(mx, __shfl_xor_sync(m8, mx, 1));
  mx = fmaxf(mx, __shfl_xor_sync(m8, mx, 2));
  mx = fmaxf(mx, __shfl_xor_sync(m8, mx, 4));
  const int e = row_exponent(mx);
  if (P.qq == 0)
    *reinterpret_cast<int*>(packed + pn.exp_off + (((int64_t)P.t * pn.nwin + P.w) * pn.tr + P.r) * 4) = e;
  const int rt = min(pn.tr, pn.nrows - P.t * pn.tr);
  if (P.r >= rt) return;
  float sc, scj;
  window_scales(e, sc, scj);
  const int plane = rt * kRowB, left = pn.nch - kChunksPerWin * P.w;  // chunks of the window that exist
  uint8_t* dst = packed + pn.pack_off + (int64_t)P.t * pn.nch * (kSlices * pn.tr * kRowB) +
                 (int64_t)kChunksPerWin * P.w * (kSlices * plane) + swz(P.r, P.qq >> 1) + 8 * (P.qq & 1);
#pragma unroll
  for (int c = 0; c < kChunksPerWin; ++c) {
    if (c >= left) break;
    uint32_t wv[kSlices][2];
    slice_f2<2>(h[c], l[c], sgn * sc, scj, wv);
#pragma unroll
    for (int k = 0; k < kSlices; ++k) *reinterpret_cast<uint2*>(dst + (c * kSlices + k) * plane) = make_uint2(wv[k][0], wv[k][1]);
  }
}

// One CTA of 128 threads per packing job.  Values: source row times its weight row
// (double-float products), zeros past K.  Bound by HBM and by the sectors its loads and stores touch:
// with 16 consecutive points per thread every access of a warp touched 32 sectors of which it used
// half; with four points of each chunk it uses them whole (and 64 registers instead of 70: eight CTAs
// per SM).  Whole steps before -> after: bent triatomic 1.503 -> 1.421 ms, C3H6 225.2 -> 219.9 ms.
__global__ void __launch_bounds__(128) pack_kernel(const DevGrid* __restrict__ grids, const Panel* __restrict__ panels,
                                                   int n_panels, const int* __restrict__ hint, const int2* __restrict__ rows,
                                                   const float* __restrict__ ops, const float* __restrict__ ops_lo,
                                                   uint8_t* __restrict__ packed) {
  using namespace mma;
  const PackPos P = pack_pos(blockIdx.x, panels, n_panels, hint);
  const Panel& pn = panels[P.pn];
  const DevGrid& g = grids[pn.grid];
  const int row = P.t * pn.tr + P.r;
  const int64_t k0 = (int64_t)kWinPts * P.w + 4 * P.qq;
  const int64_t blk = g.op_off + (int64_t)P.w * g.ws + 4 * P.qq;  // (kWinPts = 128: one block)
  int64_t src = -1, mul = -1;
  if (row < pn.nrows) {
    const int2 q = rows[pn.rows_off + row];
    src = blk + q.x * g.rs;
    if (q.y >= 0) mul = blk + q.y * g.rs;
  }
  const int64_t left = src >= 0 ? g.K - k0 : 0;
  f2 h[kChunksPerWin][2], l[kChunksPerWin][2];
#pragma unroll
  for (int c = 0; c < kChunksPerWin; ++c) {
    const int p = kChunk * c;  // this chunk's four points, from the thread's first
    ulonglong2 ah = make_ulonglong2(0, 0), al = ah, bh = ah, bl = ah;
    if (left >= p + 4) {
      ah = __ldg(reinterpret_cast<const ulonglong2*>(ops + src + p));
      al = __ldg(reinterpret_cast<const ulonglong2*>(ops_lo + src + p));
      if (mul >= 0) {
        bh = __ldg(reinterpret_cast<const ulonglong2*>(ops + mul + p));
        bl = __ldg(reinterpret_cast<const ulonglong2*>(ops_lo + mul + p));
      }
    } else if (left > p) {
      float v[4][4] = {};
      for (int i = 0; i < 4 && p + i < left; ++i) {
        v[0][i] = ops[src + p + i];
        v[1][i] = ops_lo[src + p + i];
        if (mul >= 0) {
          v[2][i] = ops[mul + p + i];
          v[3][i] = ops_lo[mul + p + i];
        }
      }
      ah = make_ulonglong2(f2_pack(v[0][0], v[0][1]).v, f2_pack(v[0][2], v[0][3]).v);
      al = make_ulonglong2(f2_pack(v[1][0], v[1][1]).v, f2_pack(v[1][2], v[1][3]).v);
      bh = make_ulonglong2(f2_pack(v[2][0], v[2][1]).v, f2_pack(v[2][2], v[2][3]).v);
      bl = make_ulonglong2(f2_pack(v[3][0], v[3][1]).v, f2_pack(v[3][2], v[3][3]).v);
    }
    f2 &h0 = h[c][0], &h1 = h[c][1], &l0 = l[c][0], &l1 = l[c][1];
    if (mul >= 0) {
      prod_unnorm(f2{ah.x}, f2{al.x}, f2{bh.x}, f2{bl.x}, h0, l0);
      prod_unnorm(f2{ah.y}, f2{al.y}, f2{bh.y}, f2{bl.y}, h1, l1);
    } else {
      h0 = f2{ah.x}; h1 = f2{ah.y};
      l0 = f2{al.x}; l1 = f2{al.y};
    }
  }
  pack_store(P, pn, h, l, mul >= 0 ? -1.0f : 1.0f, packed);
}

// The same packed-panel image from FP64 operand rows (row-major, stride n): used for the
// RI 4-index product, whose operand rows are the (P|ij) columns after the forward solve.
// Panel k's rows start at src[k]; jobs as in pack_kernel, both panels' jobs in one launch.
// Each FP64 value is split into a double-float pair first (48 bits, beyond the 39 that the
// digits keep).
__global__ void __launch_bounds__(128) ri_pack_kernel(const Panel* __restrict__ panels, const double* __restrict__ srcA,
                                                      const double* __restrict__ srcB, int n, uint8_t* __restrict__ packed) {
  using namespace mma;
  const PackPos P = pack_pos(blockIdx.x, panels, 2, nullptr);
  const Panel& pn = panels[P.pn];
  const double* src = P.pn ? srcB : srcA;
  const int row = P.t * pn.tr + P.r;
  const int k0 = kWinPts * P.w + 4 * P.qq;
  f2 h[kChunksPerWin][2], l[kChunksPerWin][2];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float hv[2], lv[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      double v = 0.0;
      if (row < pn.nrows && k0 + kChunk * (i >> 1) + 2 * (i & 1) + k < n) v = src[(int64_t)row * n + k0 + kChunk * (i >> 1) + 2 * (i & 1) + k];
      hv[k] = (float)v;
      lv[k] = (float)(v - (double)hv[k]);
    }
    h[i >> 1][i & 1] = f2_pack(hv[0], hv[1]);
    l[i >> 1][i & 1] = f2_pack(lv[0], lv[1]);
  }
  pack_store(P, pn, h, l, 1.0f, packed);
}

// ------------------------------------------------------------------ warp-specialised contraction
//
// One persistent CTA per SM, 512 threads, working through tiles (128 A rows x <= 48 B
// columns x a range of 128-point windows):
//   warp 4       loader: two ordered streams of bulk copies, each served as soon as its next
//                buffer is free: the packed A tile of every 32-point chunk into the A ring
//                of three to eight chunks (and, for a packed B, its B tile into the B ring), and the staged basis
//                rows (hi and lo planes) of every formed window into two buffers;
//   warps 0-3, 6, 7  producers: for a formed B, column c of the tile = product of two staged
//                rows (a double-float product); each warp owns 8 columns, four lanes per
//                column, lane g the 16-byte group g of every chunk; per window they form the
//                products, find each column's scale, then slice chunk by chunk into the B ring,
//                so that the MMAs of one chunk overlap the slicing of the next (for a packed B
//                they only pass each chunk on);
//   warp 5       MMA issue: per chunk 2 K-steps x 5 MMAs (A plane i against B planes
//                0..4-i, contiguous in shared memory: one MMA of N = 48 (5 - i) whose columns
//                land on the order accumulators i..4) into the window's TMEM accumulator set
//                (5 orders x 48 columns; two sets);
//   warps 8-15   fold: per window, the five order sums of their TMEM lane quadrant and column
//                half, scaled by the window's row and column exponents, into double-float
//                registers (orders 0 and 1 join the sum exactly through TwoSums, orders 2-4
//                as one FP32 term); at the end of the tile, (hi, lo) partials to global memory.
// What bounds it: the tensor pipe (62% of the measured BF16 rate on nine atoms) and, about even with
// it, the producers' slicing and the fold.  Measured (MMAs issued from a divergent branch, scalar
// slicing and folding, a bulk copy per plane and row -> now): nine-atom quadruple-zeta job (288 grids)
// 250 -> 163 ms, quintuple-zeta diatomic 98 -> 68 ms, bent triatomic 0.97 -> 0.64 ms.
//
// Every wait is bounded (wait_ns in the main loops, the fixed kWaitNs for the drains); a
// timeout sets *status and the CTA's abort flag, and each role leaves its loops at its next
// wait; the loader then waits for its copies in flight and the MMA lane for its MMAs before
// the TMEM is released.

namespace ws {

constexpr int kThreads = 512;
constexpr int kLoadWarp = 4, kMmaWarp = 5, kFoldWarp0 = 8;
// Staged basis rows lie 512 bytes apart, as in memory, so that a run of consecutive rows is one copy (a
// bulk copy takes the loader about 100 cycles to issue; rows spread over the banks, one copy each,
// cost more than the two-way conflicts of this layout's reads).
constexpr int kRawStride = kWinPts;

struct Smem {
  alignas(1024) uint8_t a[mma::kARingBytes];
  alignas(1024) uint8_t b[mma::kStagesB][kSlices][mma::kTileN * mma::kRowB];
  alignas(16) float raw[2][2][kPairTileRows][kRawStride];  // [buffer][hi, lo][row][point]
  int eb[2][mma::kTileN];
  alignas(8) float sbw[8][mma::kTileN];  // fold warp k: the column scales of the current window
  alignas(8) uint64_t a_full[mma::kMaxStages], a_free[mma::kMaxStages], b_ready[mma::kStagesB], b_free[mma::kStagesB];
  uint64_t tmem_full[2], tmem_free[2], raw_full[2], raw_free[2], eb_free[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};

__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(mma::smem_u32(b))
               : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(
                   mma::smem_u32(b)),
               "r"(bytes)
               : "memory");
}

// Bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16), completing
// on mbarrier b.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* b) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   mma::smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(mma::smem_u32(b))
               : "memory");
}

__device__ __forceinline__ bool wait(uint64_t* b, uint32_t parity, const int* abort, uint64_t limit_ns) {
  return mma::mbar_wait(mma::smem_u32(b), parity, abort, limit_ns);
}

// The A ring.  A tile's chunk takes its real rows (rounded up to eight) times 64 bytes per plane, so a
// tile of 72 rows has six chunks in flight where one of 128 rows has three: the ring must cover the
// latency of the copies (2 us under load, about three chunks' MMAs).  The MMAs read 128 rows per
// plane; what lies past the real ones (other planes, the B ring) only reaches result rows that are
// never read.  Loader and MMA lane step through the stages alike; when the rows per tile change, the
// loader waits for the ring to empty and both start again at stage 0.
struct ARing {
  uint32_t par;   // loader: parity of each stage's next a_free phase; MMA lane: of its next a_full phase
  uint32_t used;  // loader: stages whose last use is not yet known to be over
  int s, n, plane;  // stage, stages, bytes of a plane
  __device__ __forceinline__ void open() { par = used = 0; s = n = plane = 0; }
  __device__ __forceinline__ bool fits(int rows) const { return plane == ((rows + 7) & ~7) * mma::kRowB; }
  __device__ __forceinline__ void layout(int rows) {
    plane = ((rows + 7) & ~7) * mma::kRowB;
    n = min(mma::kMaxStages, mma::kARingBytes / (kSlices * plane));
    s = 0;
  }
  __device__ __forceinline__ uint32_t offset() const { return (uint32_t)(s * kSlices * plane); }
  __device__ __forceinline__ void next() { s = s + 1 == n ? 0 : s + 1; }
};
// Stage k free again (loader)
__device__ __forceinline__ bool wait_a_free(Smem& sm, ARing& r, int k, uint64_t ns) {
  if (!((r.used >> k) & 1u)) return true;
  if (!mma::mbar_wait(mma::smem_u32(&sm.a_free[k]), (r.par >> k) & 1u, &sm.abort, ns)) return false;
  r.par ^= 1u << k;
  r.used &= ~(1u << k);
  return true;
}
// B stage of chunk c: c % kStagesB after c / kStagesB completed rounds
__device__ __forceinline__ int bstage_of(uint32_t c) { return (int)(c % mma::kStagesB); }
__device__ __forceinline__ uint32_t bround_of(uint32_t c) { return c / mma::kStagesB; }
// B stage of chunk c free again (its MMAs of chunk c - kStagesB complete)
__device__ __forceinline__ bool wait_b_free(Smem& sm, uint32_t c, uint64_t ns) {
  return c < (uint32_t)mma::kStagesB ||
         mma::mbar_wait(mma::smem_u32(&sm.b_free[bstage_of(c)]), (bround_of(c) - 1) & 1, &sm.abort, ns);
}

// What every role needs to know about an item.
struct Geo {
  const MmaBlock* blk;
  int64_t K;
  int nch, nwin, w0, w1;
  int nt;  // B columns of the tile
  bool formed;
  const PairTile* pt;
};

__device__ __forceinline__ Geo geo(const GemmItem& it, const MmaBlock* blocks, const DevGrid* grids,
                                   const PairTile* ptiles) {
  Geo q;
  q.blk = blocks + it.block;
  const MmaBlock& b = *q.blk;
  q.K = grids[b.grid].K;
  q.nch = (int)((q.K + mma::kChunk - 1) / mma::kChunk);
  q.nwin = (q.nch + mma::kChunksPerWin - 1) / mma::kChunksPerWin;
  q.w0 = it.chunk * b.win_per;
  q.w1 = min(q.nwin, q.w0 + b.win_per);
  q.formed = b.b_panel < 0;
  q.pt = q.formed ? ptiles + b.ptile_off + it.tn : nullptr;
  q.nt = q.formed ? q.pt->ncols : min(mma::kTileN, b.n - it.tn * mma::kTileN);
  return q;
}

__device__ __forceinline__ int chunks_in(const Geo& q, int win) { return min(mma::kChunksPerWin, q.nch - mma::kChunksPerWin * win); }

__device__ __forceinline__ void fail(Smem& sm, int* status, int code) {
  *(volatile int*)&sm.abort = 1;
  atomicCAS(status, 0, code);  // the first failure's code stays
}

__device__ __forceinline__ bool aborted(Smem& sm) { return *(volatile int*)&sm.abort != 0; }

// The loader's stream of staged-row requests: the formed windows of the CTA's items in the
// order the producers form them, with the current item's tile rows and grid offsets cached
// (one lookup per item, not per window).
struct RowStream {
  int ii, ie, win, w1;  // current item, end, next window, the item's window end
  int nr;               // staged rows of the item's pair tile (<= kPairTileRows)
  unsigned runs;        // bit r: row r does not follow row r - 1 in memory
  int64_t src, ws;      // this lane's row (lane & 15), window 0, in floats; window stride
  bool more;

  __device__ __forceinline__ void open(int i0, int i1, const GemmItem* items, const MmaBlock* blocks,
                                       const DevGrid* grids, const PairTile* ptiles, int lane) {
    ii = i0;
    ie = i1;
    win = -1;
    more = false;
    seek(items, blocks, grids, ptiles, lane, false);
  }
  // Advances to the next formed window (the next window of the current item when `step`).
  __device__ __forceinline__ void seek(const GemmItem* items, const MmaBlock* blocks, const DevGrid* grids,
                                       const PairTile* ptiles, int lane, bool step) {
    if (step && ++win < w1) return;
    if (step) ++ii;
    for (; ii < ie; ++ii) {
      const Geo q = geo(items[ii], blocks, grids, ptiles);
      if (!q.formed) continue;
      const DevGrid& g = grids[q.blk->grid];
      win = q.w0;
      w1 = q.w1;
      nr = q.pt->nrows;
      const int row = q.pt->rows[max(0, min(lane & 15, nr - 1))];
      const int before = __shfl_up_sync(0xffffffffu, row, 1);
      runs = __ballot_sync(0xffffffffu, lane < nr && (lane == 0 || row != before + 1));
      src = g.op_off + row * g.rs;
      ws = g.ws;
      more = win < w1;
      if (more) return;
    }
    more = false;
  }
  // Bulk copies of the current window's rows (hi and lo planes, 512 bytes per row and plane, one copy
  // per run of consecutive rows) into raw buffer rb, completing on raw_full[rb]; one warp, one lane
  // issuing on uniform addresses.
  __device__ __forceinline__ void request(Smem& sm, int rb, const float* ops, const float* ops_lo) const {
    const int n = __shfl_sync(0xffffffffu, nr, 0);
    if (mma::elect_one()) mbar_expect_tx(&sm.raw_full[rb], (uint32_t)n * 2u * 512u);
    __syncwarp();
    const int64_t w0 = ws * win;
    for (unsigned m = runs; m != 0;) {
      const int r = __ffs(m) - 1;
      m &= m - 1;
      const uint32_t bytes = (uint32_t)((m ? __ffs(m) - 1 : n) - r) * 512u;
      const int64_t at = __shfl_sync(0xffffffffu, src, r) + w0;
      if (mma::elect_one()) {
        bulk_g2s(sm.raw[rb][0][r], ops + at, bytes, &sm.raw_full[rb]);
        bulk_g2s(sm.raw[rb][1][r], ops_lo + at, bytes, &sm.raw_full[rb]);
      }
      __syncwarp();
    }
  }
};

}  // namespace ws

__global__ void __launch_bounds__(ws::kThreads, 1)
    contract_ws_kernel(const DevGrid* __restrict__ grids, const MmaBlock* __restrict__ blocks,
                       const GemmItem* __restrict__ items, const int* __restrict__ cta_begin,
                       const Panel* __restrict__ panels, const PairTile* __restrict__ ptiles,
                       const float* __restrict__ ops, const float* __restrict__ ops_lo,
                       const uint8_t* __restrict__ packed, float2* __restrict__ part, int* __restrict__ status,
                       uint64_t wait_ns, const int* __restrict__ hold) {
  using namespace mma;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  ws::Smem& sm = *reinterpret_cast<ws::Smem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;  // (a warp-uniform index)
  if (warp == ws::kMmaWarp) tmem_alloc(&sm.tmem_base, 512);
  if (tid == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(&sm.a_full[s], 1);
      mbar_init(&sm.a_free[s], 1);
    }
    for (int s = 0; s < kStagesB; ++s) {
      mbar_init(&sm.b_ready[s], 6);
      mbar_init(&sm.b_free[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sm.tmem_full[s], 1);
      mbar_init(&sm.tmem_free[s], 8);
      mbar_init(&sm.raw_full[s], 1);
      mbar_init(&sm.raw_free[s], 6);
      mbar_init(&sm.eb_free[s], 8);
    }
    mbar_init(&sm.drain, 1);
    sm.abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = sm.tmem_base;
  uint32_t c = 0, w = 0, rw = 0;  // chunks, windows and formed windows of this CTA so far

  constexpr unsigned kFull = 0xffffffffu;
  if (warp == ws::kLoadWarp) {
    // ------------------------------------------------------------------ loader
    bool run = true;  // warp-uniform
    ws::ARing ar;
    ar.open();
    bool was_formed = false;
    uint32_t loads = 0, loaded = 0;  // parity of each stage's loads so far; stages ever loaded (for the drain)
    if (hold) {
      // failure-detection test: a raised flag that nothing clears holds the first copy back
      // until the wait limit runs out
      int held = 0;
      if (lane == 0) {
        const uint64_t t0 = global_ns();
        while ((held = *(volatile const int*)hold) != 0 && global_ns() - t0 <= wait_ns) {
        }
      }
      if (__shfl_sync(kFull, held, 0) != 0) {
        ws::fail(sm, status, 8);
        run = false;
      }
    }
    // Two ordered streams: the packed A (and packed B) tiles of every chunk into the rings, and
    // the staged basis rows of every formed window into two buffers (the rows of formed window
    // k + 1 are in flight while the producers form window k).  The warp waits for the chunk
    // stream's buffers and, before each of those waits, requests every window of rows whose
    // buffer is already free.
    const int ie = cta_begin[blockIdx.x + 1];
    ws::RowStream rs;
    rs.open(cta_begin[blockIdx.x], ie, items, blocks, grids, ptiles, lane);
    uint32_t rq = 0;  // formed windows requested
    auto request_free = [&]() {
      while (rs.more) {
        // buffer rq & 1 last held formed window rq - 2, released after its products
        const int rb = (int)(rq & 1);
        int free_ = 1;
        if (lane == 0) free_ = rq < 2 || mbar_test(smem_u32(&sm.raw_free[rb]), ((rq - 2) >> 1) & 1);
        if (!__shfl_sync(kFull, free_, 0)) return;
        rs.request(sm, rb, ops, ops_lo);
        ++rq;
        rs.seek(items, blocks, grids, ptiles, lane, true);
      }
    };
    for (int ii = cta_begin[blockIdx.x]; ii < ie && run; ++ii) {
      const GemmItem it = items[ii];
      const ws::Geo q = ws::geo(it, blocks, grids, ptiles);
      const MmaBlock& b = *q.blk;
      const Panel& pa = panels[b.a_panel];
      const Panel* pb = q.formed ? nullptr : panels + b.b_panel;
      // the stored rows of the tiles, and their first chunk
      const int ra = __shfl_sync(kFull, min(kM, pa.nrows - it.tm * kM), 0);
      const int rbw = __shfl_sync(kFull, pb ? min(kTileN, pb->nrows - it.tn * kTileN) : 0, 0);
      const uint8_t* pk_a = packed + __shfl_sync(kFull, pa.pack_off + (int64_t)it.tm * pa.nch * (kSlices * kM * kRowB), 0);
      const uint8_t* pk_b = packed + __shfl_sync(kFull, pb ? pb->pack_off + (int64_t)it.tn * pb->nch * (kSlices * kTileN * kRowB) : 0, 0);
      // The ring empties before another row count's layout, and before a packed B after formed ones (the
      // B ring's phases are then known to be over up to this item's first chunk).
      if (!ar.fits(ra) || (pb && was_formed)) {
        // The rows of the formed windows still in the ring may have to be requested meanwhile: the
        // ring holds up to eight chunks of as many windows, the staged buffers two windows.
        const uint64_t t0 = global_ns();
        for (int k = 0; k < kMaxStages && run; ++k) {
          if (!((ar.used >> k) & 1u)) continue;
          while (run && !__all_sync(kFull, mbar_test(smem_u32(&sm.a_free[k]), (ar.par >> k) & 1u))) {
            request_free();
            run = __all_sync(kFull, !ws::aborted(sm) && global_ns() - t0 <= wait_ns);
          }
          ar.par ^= 1u << k;
          ar.used &= ~(1u << k);
        }
        if (!run) { ws::fail(sm, status, 4); break; }
        if (!ar.fits(ra)) ar.layout(ra);
      }
      was_formed = !pb;
      for (int win = q.w0; win < q.w1 && run; ++win) {
        const int nck = ws::chunks_in(q, win);
        for (int j = 0; j < nck; ++j, ++c) {
          request_free();
          const int s = ar.s, sb = ws::bstage_of(c), ch = kChunksPerWin * win + j;
          const bool ok = ws::wait_a_free(sm, ar, s, wait_ns) && (!pb || ws::wait_b_free(sm, c, wait_ns));
          run = __all_sync(kFull, ok && !ws::aborted(sm));
          if (!run) { ws::fail(sm, status, 4); break; }
          // one bulk copy, or one per plane, issued by one lane on uniform addresses
          if (elect_one()) {
            ws::mbar_expect_tx(&sm.a_full[s], (uint32_t)(kSlices * kRowB * (ra + rbw)));
            const uint8_t* src = pk_a + (int64_t)ch * (kSlices * ra * kRowB);
            uint8_t* dst = sm.a + ar.offset();
            if (ar.plane == ra * kRowB) {  // whole groups of eight rows: the planes follow one another
              ws::bulk_g2s(dst, src, (uint32_t)(kSlices * kRowB * ra), &sm.a_full[s]);
            } else {
#pragma unroll
              for (int k = 0; k < kSlices; ++k)
                ws::bulk_g2s(dst + k * ar.plane, src + k * (ra * kRowB), (uint32_t)(kRowB * ra), &sm.a_full[s]);
            }
            if (pb) {
              const uint8_t* srcb = pk_b + (int64_t)ch * (kSlices * rbw * kRowB);
              if (rbw == kTileN) {
                ws::bulk_g2s(sm.b[sb][0], srcb, (uint32_t)(kSlices * kTileN * kRowB), &sm.a_full[s]);
              } else {
#pragma unroll
                for (int k = 0; k < kSlices; ++k)
                  ws::bulk_g2s(sm.b[sb][k], srcb + k * (rbw * kRowB), (uint32_t)(kRowB * rbw), &sm.a_full[s]);
              }
            }
          }
          __syncwarp();
          ar.used |= 1u << s;
          loads ^= 1u << s;
          loaded |= 1u << s;
          ar.next();
        }
      }
    }
    // the rows of the last formed windows, as their buffers free up
    while (run && rs.more) {
      const int rb = (int)(rq & 1);
      const bool ok = rq < 2 || ws::wait(&sm.raw_free[rb], ((rq - 2) >> 1) & 1, &sm.abort, wait_ns);
      run = __all_sync(kFull, ok && !ws::aborted(sm));
      if (!run) { ws::fail(sm, status, 4); break; }
      request_free();
    }
    // drain: nothing may still be copying into shared memory when the CTA exits (another
    // role may have given up after this loop ended; the phases waited for here are the last
    // ones issued on each barrier, complete at once when the copies were consumed)
    for (int k = 0; k < kMaxStages; ++k)
      if ((loaded >> k) & 1u) ws::wait(&sm.a_full[k], ((loads >> k) & 1u) ^ 1u, nullptr, kWaitNs);
    for (int k = (int)rq - 1; k >= 0 && k > (int)rq - 3; --k)
      ws::wait(&sm.raw_full[k & 1], (k >> 1) & 1, nullptr, kWaitNs);
  } else if (warp < 4 || warp == 6 || warp == 7) {
    // ------------------------------------------------------------------ producers
    // A lane forms columns col[0] and col[1], which mostly share their first row (the pairs of a tile
    // are listed row by row), four points of each per chunk: its eight lanes read 128 contiguous bytes
    // of a row, and the shared row once.
    const int pw = warp < 4 ? warp : warp - 2;  // 0..5
    const int col[2] = {8 * pw + (lane >> 3), 8 * pw + 4 + (lane >> 3)};
    const int g = lane & 7;                     // points [4 g, 4 g + 4) of each chunk
    const unsigned col_mask = 0xffu << (lane & 24);
    bool run = true;  // warp-uniform
    for (int ii = cta_begin[blockIdx.x], ie = cta_begin[blockIdx.x + 1]; ii < ie && run; ++ii) {
      const GemmItem it = items[ii];
      const ws::Geo q = ws::geo(it, blocks, grids, ptiles);
      if (!q.formed) {
        // packed B: the loader brings it; b_ready still completes one phase per chunk
        for (int win = q.w0; win < q.w1 && run; ++win, ++w) {
          const int nck = ws::chunks_in(q, win);
          // every phase of eb_free is waited for, so that a formed window's wait cannot take an older
          // phase of the same parity for its own where windows of one chunk follow one another
          const bool oke = w < 2 || ws::wait(&sm.eb_free[w & 1], ((w - 2) >> 1) & 1, &sm.abort, wait_ns);
          run = __all_sync(kFull, oke && !ws::aborted(sm));
          if (!run) { ws::fail(sm, status, 5); break; }
          for (int j = 0; j < nck; ++j, ++c) {
            const int sb = ws::bstage_of(c);
            const bool ok = ws::wait_b_free(sm, c, wait_ns);
            run = __all_sync(kFull, ok && !ws::aborted(sm));
            if (!run) { ws::fail(sm, status, 5); break; }
            if (lane == 0) ws::mbar_arrive(&sm.b_ready[sb]);
          }
        }
        continue;
      }
      int dx[2], dy[2];
      bool valid[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        valid[u] = col[u] < q.nt;
        dx[u] = valid[u] ? q.pt->dx[col[u]] : 0;
        dy[u] = valid[u] ? q.pt->dy[col[u]] : 0;
      }
      for (int win = q.w0; win < q.w1 && run; ++win, ++w, ++rw) {
        const int nck = ws::chunks_in(q, win);
        const int rb = rw & 1, set = w & 1;
        bool ok = ws::wait(&sm.raw_full[rb], (rw >> 1) & 1, &sm.abort, wait_ns);
        run = __all_sync(kFull, ok && !ws::aborted(sm));
        if (!run) { ws::fail(sm, status, 5); break; }
        const int wleft = (int)(q.K - (int64_t)kWinPts * win);  // points of the window that exist
        f2 vh[kChunksPerWin][2][2], vl[kChunksPerWin][2][2];  // products, hi words negated
        float mx[2] = {0.0f, 0.0f};
#pragma unroll
        for (int cc = 0; cc < kChunksPerWin; ++cc) {
          const int p0 = kChunk * cc + 4 * g;
          ulonglong2 a = *reinterpret_cast<const ulonglong2*>(sm.raw[rb][0][dx[0]] + p0);
          ulonglong2 al = *reinterpret_cast<const ulonglong2*>(sm.raw[rb][1][dx[0]] + p0);
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if (u == 1 && dx[1] != dx[0]) {
              a = *reinterpret_cast<const ulonglong2*>(sm.raw[rb][0][dx[1]] + p0);
              al = *reinterpret_cast<const ulonglong2*>(sm.raw[rb][1][dx[1]] + p0);
            }
            const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(sm.raw[rb][0][dy[u]] + p0);
            const ulonglong2 bl = *reinterpret_cast<const ulonglong2*>(sm.raw[rb][1][dy[u]] + p0);
            prod_unnorm(f2{a.x}, f2{al.x}, f2{b.x}, f2{bl.x}, vh[cc][u][0], vl[cc][u][0]);
            prod_unnorm(f2{a.y}, f2{al.y}, f2{b.y}, f2{bl.y}, vh[cc][u][1], vl[cc][u][1]);
            const int left = valid[u] ? wleft - p0 : 0;  // a short last window, or no such column: zeros
            if (left < 4) {
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                float h0, h1, l0, l1;
                f2_unpack(vh[cc][u][i], h0, h1);
                f2_unpack(vl[cc][u][i], l0, l1);
                if (2 * i >= left) h0 = l0 = 0.0f;
                if (2 * i + 1 >= left) h1 = l1 = 0.0f;
                vh[cc][u][i] = f2_pack(h0, h1);
                vl[cc][u][i] = f2_pack(l0, l1);
              }
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              float h0, h1;
              f2_unpack(vh[cc][u][i], h0, h1);
              mx[u] = fmaxf(mx[u], fmaxf(fabsf(h0), fabsf(h1)));
            }
          }
        }
        // the staged rows are read: release the buffer for the window after next
        __syncwarp();
        if (lane == 0) ws::mbar_arrive(&sm.raw_free[rb]);
        // the columns' window maxima over their eight lanes
        int e[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) mx[u] = fmaxf(mx[u], __shfl_xor_sync(col_mask, mx[u], o));
          e[u] = row_exponent(mx[u]);
        }
        // the column exponents of this set were last read by the fold of window w - 2, which
        // releases them (eb_free) as soon as it has copied them: the fold stays off this path
        const bool okb = w < 2 || ws::wait(&sm.eb_free[set], ((w - 2) >> 1) & 1, &sm.abort, wait_ns);
        run = __all_sync(kFull, okb && !ws::aborted(sm));
        if (!run) { ws::fail(sm, status, 5); break; }
        float sc[2], scj[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (g == 0) sm.eb[set][col[u]] = e[u];
          window_scales(e[u], sc[u], scj[u]);
        }
#pragma unroll
        for (int cc = 0; cc < kChunksPerWin; ++cc) {
          if (cc < nck && run) {
            const int sb = ws::bstage_of(c);
            const bool okc = ws::wait_b_free(sm, c, wait_ns);
            run = __all_sync(kFull, okc && !ws::aborted(sm));
            if (!run) {
              ws::fail(sm, status, 5);
            } else {
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                uint32_t wv[kSlices][2];
                slice_f2<2>(vh[cc][u], vl[cc][u], -sc[u], scj[u], wv);
#pragma unroll
                for (int k = 0; k < kSlices; ++k)
                  *reinterpret_cast<uint2*>(sm.b[sb][k] + swz(col[u], g >> 1) + 8 * (g & 1)) = make_uint2(wv[k][0], wv[k][1]);
              }
              fence_async_smem();
              __syncwarp();
              if (lane == 0) ws::mbar_arrive(&sm.b_ready[sb]);
              ++c;
            }
          }
        }
        if (!run) break;
      }
    }
  } else if (warp == ws::kMmaWarp) {
    // ------------------------------------------------------------------ MMA issue
    // The whole warp runs the loop on warp-uniform values and one lane issues: issued from a divergent
    // branch, an MMA took about 90 cycles to issue, more than the smaller ones of a K step run.
    bool ok = true;
    ws::ARing ar;
    ar.open();
    for (int ii = cta_begin[blockIdx.x], ie = cta_begin[blockIdx.x + 1]; ii < ie && ok; ++ii) {
      const GemmItem it = items[ii];
      const ws::Geo q = ws::geo(it, blocks, grids, ptiles);
      const int ra = __shfl_sync(kFull, min(kM, panels[q.blk->a_panel].nrows - it.tm * kM), 0);
      if (!ar.fits(ra)) ar.layout(ra);
      const int w0 = __shfl_sync(kFull, q.w0, 0), w1 = __shfl_sync(kFull, q.w1, 0), nch = __shfl_sync(kFull, q.nch, 0);
      for (int win = w0; win < w1 && ok; ++win, ++w) {
        const int nck = min(kChunksPerWin, nch - kChunksPerWin * win);
        const int set = w & 1;
        if (w >= 2) ok = __all_sync(kFull, ws::wait(&sm.tmem_free[set], ((w - 2) >> 1) & 1, &sm.abort, wait_ns));
        const uint32_t tset = tmem + (uint32_t)set * 256u;
        for (int j = 0; j < nck && ok; ++j, ++c) {
          const uint32_t s = ar.s, sb = c % kStagesB;
          ok = ws::wait(&sm.a_full[s], (ar.par >> s) & 1u, &sm.abort, wait_ns) &&
               ws::wait(&sm.b_ready[sb], ws::bround_of(c) & 1, &sm.abort, wait_ns);
          ok = __all_sync(kFull, ok);
          if (!ok) break;
          fence_after();
          // The B planes of a stage are contiguous (48 rows each), so plane i of A against
          // planes 0..4-i of B is one MMA of N = 48 (5 - i) whose columns land on the order
          // accumulators i..4 (order k at TMEM columns 48k..48k+47 of the set).
          const uint32_t da = desc_lo(smem_u32(sm.a)) + (ar.offset() >> 4), dp = (uint32_t)ar.plane >> 4;
          const uint32_t db = desc_lo(smem_u32(sm.b[0][0])) + sb * (uint32_t)(sizeof(sm.b[0]) >> 4);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < kChunk / 16; ++k)
#pragma unroll
              for (int i = 0; i < kSlices; ++i)
                mma_f16_lo(tset + (uint32_t)(kTileN * i), da + i * dp + 2u * k, db + 2u * k,
                           make_idesc(kTileN * (kSlices - i)), (j > 0 || k > 0 || i > 0) ? 1u : 0u);
            mma_commit(smem_u32(&sm.a_free[s]));
            mma_commit(smem_u32(&sm.b_free[sb]));
            if (j + 1 == nck) mma_commit(smem_u32(&sm.tmem_full[set]));
          }
          __syncwarp();
          ar.par ^= 1u << s;
          ar.next();
        }
      }
    }
    if (!ok) ws::fail(sm, status, 6);
    // drain: every issued MMA must be complete before the TMEM is released (also when
    // another role gave up after this loop ended)
    if (elect_one()) mma_commit(smem_u32(&sm.drain));
    ws::wait(&sm.drain, 0, nullptr, kWaitNs);
    __syncwarp();
  } else if (warp >= ws::kFoldWarp0) {
    // ------------------------------------------------------------------ fold
    const int ew = warp - ws::kFoldWarp0;  // 0..7
    const int quad = warp & 3;             // TMEM lane quadrant this warp may access
    const int half = ew >> 2;              // columns [24 half, 24 half + 24)
    const int row_in_tile = quad * 32 + lane;
    const int my_col = 24 * half + lane;   // lanes 0-23: the column whose scale this lane loads
    bool run = true;  // warp-uniform
    for (int ii = cta_begin[blockIdx.x], ie = cta_begin[blockIdx.x + 1]; ii < ie && run; ++ii) {
      const GemmItem it = items[ii];
      const ws::Geo q = ws::geo(it, blocks, grids, ptiles);
      const MmaBlock& b = *q.blk;
      const Panel& pa = panels[b.a_panel];
      const Panel* pb = q.formed ? nullptr : panels + b.b_panel;
      const int rows_valid = min(kM, b.m - it.tm * kM);  // real rows of the A tile
      f2 H[12], L[12];  // pairs of columns
#pragma unroll
      for (int j = 0; j < 12; ++j) H[j] = L[j] = f2_both(0.0f);
      // the window's exponents (A rows from the packed panel; B columns from the packed panel,
      // one per lane for this warp's 24 columns, or from the producers), loaded one window ahead
      const int* ea_src = reinterpret_cast<const int*>(packed + pa.exp_off) + (int64_t)it.tm * pa.nwin * kM + row_in_tile;
      const int* eb_src = (pb && lane < 24)
                              ? reinterpret_cast<const int*>(packed + pb->exp_off) + (int64_t)it.tn * pb->nwin * kTileN + my_col
                              : nullptr;
      int ea_next = __ldg(ea_src + (int64_t)q.w0 * kM);
      int eb_next = eb_src ? __ldg(eb_src + (int64_t)q.w0 * kTileN) : 0;
      for (int win = q.w0; win < q.w1; ++win, ++w) {
        const int set = w & 1;
        const int ea = ea_next, eb_lane = eb_next;
        if (win + 1 < q.w1) {
          ea_next = __ldg(ea_src + (int64_t)(win + 1) * kM);
          if (eb_src) eb_next = __ldg(eb_src + (int64_t)(win + 1) * kTileN);
        }
        const bool ok = ws::wait(&sm.tmem_full[set], (w >> 1) & 1, &sm.abort, wait_ns);
        run = __all_sync(kFull, ok && !ws::aborted(sm));
        if (!run) { ws::fail(sm, status, 7); break; }
        fence_after();
        // column scales 2^(e_b - 7 - 8) for this warp, row scale 2^(e_a - 7 - 8) for this
        // thread (each stored digit carries 2^8)
        float* sbw = sm.sbw[ew];
        if (lane < 24) sbw[my_col] = pow2f((pb ? eb_lane : sm.eb[set][my_col]) - 7 - kDigitScaleExp);
        const float sa = pow2f(ea - 7 - kDigitScaleExp);
        __syncwarp();
        if (lane == 0) ws::mbar_arrive(&sm.eb_free[set]);  // the producers may refill eb[set]
        const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)set * 256u;
        // a warp whose 32 rows are all past the tile's last real row has nothing to fold
        if (quad * 32 < rows_valid) {
#pragma unroll
          for (int gi = 0; gi < 3; ++gi) {
            const int c0 = 24 * half + 8 * gi;  // first of 8 columns
            if (c0 < q.nt) {
              float o[kSlices][8];
#pragma unroll
              for (int k = 0; k < kSlices; ++k) tmem_ld8(lane_base + (uint32_t)(kTileN * k + c0), o[k]);
              tmem_wait_ld();
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                f2 &h = H[4 * gi + j], &lo = L[4 * gi + j];
                const f2 sc = f2_mul(f2_both(sa), *reinterpret_cast<const f2*>(sbw + c0 + 2 * j));  // 2^(e_a + e_b - 30)
                const f2 o0 = f2_pack(o[0][2 * j], o[0][2 * j + 1]), o1 = f2_pack(o[1][2 * j], o[1][2 * j + 1]),
                         o2 = f2_pack(o[2][2 * j], o[2][2 * j + 1]), o3 = f2_pack(o[3][2 * j], o[3][2 * j + 1]),
                         o4 = f2_pack(o[4][2 * j], o[4][2 * j + 1]);
                // Orders 0 and 1 as a sum t and its exact error e (Dekker's Fast2Sum on the FMA; the
                // orders are multiples of 2^16 below 2^40, so o0 - t is exact also where o0 is the
                // smaller); t, times the power of two sc, enters the double-float sum through one
                // TwoSum; e and orders 2-4 (at most 2^-15 of order 0) join the lo word as one FP32
                // term, rounded at 2^-16 of order 0's unit (2^-37 of the window's largest sum).
                const f2 c8 = f2_both(0.00390625f);
                const f2 t = f2_fma(o1, c8, o0);
                const f2 e = f2_fma(o1, c8, f2_rsub(t, o0));
                const f2 tail = f2_fma(f2_fma(f2_fma(o4, c8, o3), c8, o2), f2_both(1.52587890625e-5f), e);
                const f2 p = f2_mul(t, sc);
                const f2 s = f2_add(h, p), bb = f2_rsub(h, s);
                const f2 er = f2_add(f2_rsub(f2_rsub(bb, s), h), f2_rsub(bb, p));
                const f2 l2 = f2_add(lo, f2_fma(tail, sc, er));
                h = f2_add(s, l2);
                lo = f2_rsub(f2_rsub(s, h), l2);
              }
            }
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) ws::mbar_arrive(&sm.tmem_free[set]);
      }
      if (!run) break;
      // (hi, lo) partial sums of this tile's window range
      const int grow = it.tm * kM + row_in_tile;
      if (grow < b.m) {
        float2* out = part + b.part_off + (int64_t)it.chunk * b.m * b.n + (int64_t)grow * b.n;
#pragma unroll
        for (int j = 0; j < 12; ++j) {
          float h[2], l[2];
          f2_unpack(H[j], h[0], h[1]);
          f2_unpack(L[j], l[0], l[1]);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const int cc = 24 * half + 2 * j + k;
            if (cc < q.nt) {
              const int ocol = q.formed ? q.pt->col[cc] : it.tn * kTileN + cc;
              out[ocol] = make_float2(h[k], l[k]);
            }
          }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == ws::kMmaWarp) {
    fence_after();
    tmem_free(tmem, 512);
  }
}

// FP64 reduction of the (hi, lo) range partials of the tensor-core blocks, times the FP64
// constants of each element's row and column (rowc NULL: all of them 1); one thread per element, ranges
// added in order (consecutive threads read consecutive partials).  The FP64 pipe (two operations per clock
// and SM) is what bounds it, so nothing is multiplied by one or added to zero.  Whole calls, before -> after: a
// 4096 x 4096 RI block 705 -> 547 us, 2-centre Coulomb of a dense grid 9.03 -> 8.66 ms, H2 graph 160 -> 153 us.
__global__ void __launch_bounds__(256) reduce_mixed_kernel(const DevGrid* __restrict__ grids,
                                                           const MmaBlock* __restrict__ blocks, int n_blocks,
                                                           const int64_t* __restrict__ elem_begin, int64_t e0,
                                                           int64_t e1, const int2* __restrict__ rows,
                                                           const double* __restrict__ rowc,
                                                           const float2* __restrict__ part, double* __restrict__ res) {
  const int64_t idx = e0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= e1) return;
  int lo = 0, hi = n_blocks;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (elem_begin[mid] <= idx) lo = mid; else hi = mid;
  }
  const MmaBlock b = blocks[lo];
  const int64_t e = idx - elem_begin[lo];
  const int64_t mn = (int64_t)b.m * b.n;
  const float2* p = part + b.part_off + e;
  const float2 v0 = __ldg(p);
  double s = (double)v0.x + (double)v0.y;
  for (int c = 1; c < b.n_ranges; ++c) {
    const float2 v = __ldg(p + c * mn);
    s += (double)v.x + (double)v.y;
  }
  if (rowc) {
    const int r = mn <= 0x7fffffff ? (int)((uint32_t)e / (uint32_t)b.n) : (int)(e / b.n), col = (int)(e - (int64_t)r * b.n);
    const double* rc = rowc + grids[b.grid].rc_off;
    const int2 qa = rows[b.a_off + r], qb = rows[b.b_off + col];
    double ca = rc[qa.x], cb = rc[qb.x];
    if (qa.y >= 0) ca *= rc[qa.y];
    if (qb.y >= 0) cb *= rc[qb.y];
    s = s * ca * cb;
  }
  res[b.res_off + e] = s;
}

// Diagnostics: operand rows (hi + lo) times their FP64 row constants, as FP64 rows of K values.
__global__ void combine_rows_kernel(const float* __restrict__ h, const float* __restrict__ l,
                                    const double* __restrict__ rc, int nrows, int64_t K, int64_t ld,
                                    double* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)nrows * K) return;
  const int r = (int)(i / K);
  const int64_t p = i - (int64_t)r * K;
  out[i] = ((double)h[r * ld + p] + (double)l[r * ld + p]) * rc[r];
}

// ------------------------------------------------------------------ launchers

cudaError_t launch_combine_rows(const float* h, const float* l, const double* rc, int nrows, int64_t K, int64_t ld,
                                double* out, cudaStream_t s) {
  const int64_t n = (int64_t)nrows * K;
  if (n == 0) return cudaSuccess;
  combine_rows_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(h, l, rc, nrows, K, ld, out);
  return cudaGetLastError();
}

cudaError_t launch_nodes(const DevGrid* grids, int n_grids, int max_entries, const double* edges, NodeEntry* tab,
                         cudaStream_t s) {
  if (n_grids == 0) return cudaSuccess;
  dim3 grid((max_entries + 127) / 128, n_grids);
  nodes_kernel<<<grid, 128, 0, s>>>(grids, edges, tab);
  return cudaGetLastError();
}

cudaError_t launch_eval_mixed(const LaunchTables& t, const NodeEntry* tab, const float2* xi, float* ops,
                              float* ops_lo, cudaStream_t s) {
  if (t.n_pblocks == 0) return cudaSuccess;
  eval_mixed_kernel<<<t.n_pblocks, kEvalThreads, kEvalTabBytes, s>>>(t, tab, xi, ops, ops_lo);
  return cudaGetLastError();
}

// the ring, staging buffers and barriers, plus 1 KB to align the ring's start
static_assert(sizeof(ws::Smem) + 1024 <= 232448, "contraction shared memory above the 227 KB a CTA may use");
size_t ws_smem_bytes() { return sizeof(ws::Smem) + 1024; }

cudaError_t prepare_kernels() {
  const cudaError_t e = cudaFuncSetAttribute(eval_mixed_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kEvalTabBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(contract_ws_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ws_smem_bytes());
}

cudaError_t launch_pack(const DevGrid* grids, const Panel* panels, int n_panels, const int* hint, int64_t n_jobs,
                        const int2* rows, const float* ops, const float* ops_lo, uint8_t* packed, cudaStream_t s) {
  if (n_jobs == 0) return cudaSuccess;
  pack_kernel<<<(unsigned)n_jobs, 128, 0, s>>>(grids, panels, n_panels, hint, rows, ops, ops_lo, packed);
  return cudaGetLastError();
}

cudaError_t launch_contract_ws(const DevGrid* grids, const MmaBlock* blocks, const GemmItem* items,
                               const int* cta_begin, int n_ctas, const Panel* panels, const PairTile* ptiles,
                               const float* ops, const float* ops_lo, const uint8_t* packed, float2* part, int* status,
                               uint64_t wait_ns, const int* hold, cudaStream_t s) {
  if (n_ctas == 0) return cudaSuccess;
  contract_ws_kernel<<<n_ctas, ws::kThreads, ws_smem_bytes(), s>>>(grids, blocks, items, cta_begin, panels, ptiles, ops,
                                                                   ops_lo, packed, part, status, wait_ns, hold);
  return cudaGetLastError();
}

cudaError_t launch_ri_pack(const Panel* panels, int64_t n_jobs, const double* srcA, const double* srcB, int n,
                           uint8_t* packed, cudaStream_t s) {
  if (n_jobs == 0) return cudaSuccess;
  ri_pack_kernel<<<(unsigned)n_jobs, 128, 0, s>>>(panels, srcA, srcB, n, packed);
  return cudaGetLastError();
}

cudaError_t launch_reduce_mixed(const DevGrid* grids, const MmaBlock* blocks, int n_blocks, const int64_t* elem_begin,
                                int64_t e0, int64_t e1, const int2* rows, const double* rowc, const float2* part,
                                double* res, cudaStream_t s) {
  if (e1 <= e0) return cudaSuccess;
  reduce_mixed_kernel<<<(unsigned)((e1 - e0 + 255) / 256), 256, 0, s>>>(grids, blocks, n_blocks, elem_begin, e0, e1,
                                                                         rows, rowc, part, res);
  return cudaGetLastError();
}


}  // namespace psq
