// lbcollide.cuh -- the per-node part of a fluid iteration shared by the
// fluid kernels: moments, forces, equilibrium velocity, BGK collision and
// the stores (collide_store), and the inlet/outlet rules on opening nodes
// (apply_openings).  The kernels differ only in where the pulled
// populations come from.
#pragma once

#include "lbarith.cuh"

namespace lbk {

namespace {

// random word for (node, component, direction, step)
__device__ __forceinline__ uint32_t rnd(uint32_t seed, int self, int c, int i) {
  return mix32(((uint32_t)self * 0x9e3779b1u) ^ (seed + 0x632be5abu * (uint32_t)c) ^
               (0x85ebca6bu * (uint32_t)(i + 1)));
}

// moments, forces, equilibrium velocity, BGK and the stores of one node of a
// single-component lattice.  PM: the momentum as an exact hi + lo sum (the
// storage flag LB_PRECISE_MOMENTUM).  FOLD (scaled 16-bit storage): h
// arrives and leaves in the stored units 2^s h, so the loads and stores skip
// their scale factors; the moments are unscaled once and the equilibrium is
// formed directly in stored units.  SR: 1 round to nearest, 2 stochastic
// rounding.
template <class S, bool PM, bool FOLD, int SR, int RX = 0>
__device__ __forceinline__ void collide_store(const FluidArgs &p, int x, int y, uint32_t bits, float (&h)[9],
                                              float *uo = nullptr) {
  const Geometry &g = p.g;
  const int self = y * g.pitch + x;
  // the node's slot in the whole lattice: the random words are the same
  // whether the lattice is held whole or in slabs
  const int hself = self + g.yoff * g.pitch;
  const int P = (int)g.plane;
  Node1<float> n;
  // stored units -> physical units (a power of two: exact)
  const float un = FOLD ? p.inv_scale : 1.0f;
  moments1<float, PM, FOLD>(h, p.rho_ref[0], un, n);
  n.Fx = vfma(n.rho, p.ax[0], p.fx[0]);
  n.Fy = vfma(n.rho, p.ay[0], p.fy[0]);
  if (p.ads[0]) {
    float sx, sy;
    wall_sum(bits, sx, sy);
    const float psi = p.ads_psi0[0] * expf(-p.ads_rho0[0] / n.rho);
    n.Fx -= p.Gads[0] * psi * sx;
    n.Fy -= p.Gads[0] * psi * sy;
  }
  shift1<float, PM, sizeof(S) == 2>(p.tau[0], n);
  S *out = (S *)p.fout;
  float heq[9];
  equilibrium1<float, PM, FOLD, sizeof(S) == 2>(n, p.scale, p.wa[0], p.wd[0], heq);
  relax<sizeof(S) == 2 ? 2 : RX>(h, heq, p.omega[0], p.keep);
  // in stored units: FP16 is folded, the other types have no scale
  if (SR == 2) {
    // stochastic rounding: one hash per node, then a linear congruential
    // sequence, one step per pair of stores (each state is uniform for a
    // uniformly random start, so both dithers of the paired conversion are
    // uniform: unbiased rounding); the ninth store takes the single
    // conversion's high bits
    uint32_t r = rnd(p.sr_seed, hself, 0, 0);
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      r = r * 1664525u + 1013904223u;
      Store<S>::st2_dither(out, i * P + self, (i + 1) * P + self, h[i], h[i + 1], r);
    }
    r = r * 1664525u + 1013904223u;
    Store<S>::st_dither(out, 8 * P + self, h[8], r);
  } else {
#pragma unroll
    for (int i = 0; i < 9; i++) Store<S>::st(out, i * P + self, h[i], 1.0f);
  }
  const float px = vadd(n.jx, vfma(0.5f, n.Fx, n.jxl)), py = vadd(n.jy, vfma(0.5f, n.Fy, n.jyl));
  if (p.fields) {
    p.fields[self] = n.drho;
    p.fields[P + self] = px;
    p.fields[2 * P + self] = py;
    p.fields[3 * P + self] = equilibrium_sum(heq, un);
  }
  if (p.uout || uo) {
    // the solvent velocity of Eq. (4)
    const float vx = px / n.rho, vy = py / n.rho;
    if (uo) {
      uo[0] = vx;
      uo[1] = vy;
    }
    if (p.uout) {
      p.uout[self] = vx;
      p.uout[P + self] = vy;
    }
  }
}

// the equilibrium of lbarith.cuh for the mass-exact collision, in plain
// expressions
__device__ __forceinline__ void equilibrium_pairs(float drho, float rho, float ux, float uy,
                                                  float mx, float my, float wa, float wd,
                                                  float (&heq)[9]) {
  const float q = rho * (ux * ux + uy * uy);
  const float sp = ux + uy, sm = uy - ux;  // e5.u and e6.u
  const float d9 = drho * wa, d36 = drho * wd;
  const float A1 = d9 + 0.5f * rho * ux * ux - q * (1.0f / 6.0f);
  const float A2 = d9 + 0.5f * rho * uy * uy - q * (1.0f / 6.0f);
  const float A5 = d36 + 0.125f * rho * sp * sp - q * (1.0f / 24.0f);
  const float A6 = d36 + 0.125f * rho * sm * sm - q * (1.0f / 24.0f);
  const float B5 = rho * sp * (1.0f / 12.0f);
  const float B6 = rho * sm * (1.0f / 12.0f);
  const float B1 = 0.5f * mx - B5 + B6;
  const float B2 = 0.5f * my - B5 - B6;
  heq[1] = A1 + B1;
  heq[3] = A1 - B1;
  heq[2] = A2 + B2;
  heq[4] = A2 - B2;
  heq[5] = A5 + B5;
  heq[7] = A5 - B5;
  heq[6] = A6 + B6;
  heq[8] = A6 - B6;
  heq[0] = drho - 2.0f * ((A1 + A2) + (A5 + A6));
}

// the same node update with the mass-exact collision (see below): two
// components, or interforce.  Fsc: interforce already evaluated (zero when
// off).
template <class S, int NC>
__device__ __forceinline__ void collide_store_me(const FluidArgs &p, int x, int y, uint32_t bits,
                                                 float (&h)[NC][9], const float (&Fsc)[NC][2]) {
  const Geometry &g = p.g;
  const int self = y * g.pitch + x;
  // the node's slot in the whole lattice: the random words are the same
  // whether the lattice is held whole or in slabs
  const int hself = self + g.yoff * g.pitch;
  const int P = (int)g.plane;
  float drho[NC], rho[NC], jx[NC], jy[NC], Fx[NC], Fy[NC];
#pragma unroll
  for (int c = 0; c < NC; c++) {
    const float(&f)[9] = h[c];
    drho[c] = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
    rho[c] = p.rho_ref[c] + drho[c];
    jx[c] = (f[1] - f[3]) + (f[5] - f[7]) + (f[8] - f[6]);
    jy[c] = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
    Fx[c] = p.fx[c] + rho[c] * p.ax[c] + Fsc[c][0];
    Fy[c] = p.fy[c] + rho[c] * p.ay[c] + Fsc[c][1];
    if (p.ads[c]) {
      float sx, sy;
      wall_sum(bits, sx, sy);
      const float psi = (NC == 1) ? p.ads_psi0[c] * expf(-p.ads_rho0[c] / rho[c]) : rho[c];
      Fx[c] -= p.Gads[c] * psi * sx;
      Fy[c] -= p.Gads[c] * psi * sy;
    }
  }
  // equilibrium velocity (velocity shift) and the momentum rho u_eq it
  // carries, the latter formed without a division
  float uex[NC], uey[NC], mxt[NC], myt[NC];
  if (NC == 1) {
    mxt[0] = jx[0] + p.tau[0] * Fx[0];
    myt[0] = jy[0] + p.tau[0] * Fy[0];
    const float ir = 1.0f / rho[0];
    uex[0] = mxt[0] * ir;
    uey[0] = myt[0] * ir;
  } else {
    // common velocity sum(j/tau) / sum(rho/tau), shifted per component
    float nxs = 0.f, nys = 0.f, den = 0.f;
#pragma unroll
    for (int c = 0; c < NC; c++) {
      nxs += jx[c] * p.omega[c];
      nys += jy[c] * p.omega[c];
      den += rho[c] * p.omega[c];
    }
    const float upx = nxs / den, upy = nys / den;
#pragma unroll
    for (int c = 0; c < NC; c++) {
      mxt[c] = rho[c] * upx + p.tau[c] * Fx[c];
      myt[c] = rho[c] * upy + p.tau[c] * Fy[c];
      uex[c] = upx + p.tau[c] * Fx[c] / rho[c];
      uey[c] = upy + p.tau[c] * Fy[c] / rho[c];
    }
  }
#pragma unroll
  for (int c = 0; c < NC; c++) {
    S *out = (S *)p.fout + (size_t)c * 9 * P;
    float heq[9];
    equilibrium_pairs(drho[c], rho[c], uex[c], uey[c], mxt[c], myt[c], p.wa[c], p.wd[c], heq);
    const float om = p.omega[c];
    // Mass-exact collision: when |h| is large (two components, or one far
    // from rho_ref) the rounding of nine stored values of a slowly
    // changing state repeats every step and drifts the mass.  Here the
    // exact sum D of the pulled values and the exact sum S of the eight
    // stored moving populations are formed with error-free sums, and the
    // rest population is set to D - S -- the BGK value in exact
    // arithmetic -- rounded stochastically, so the node's mass is kept
    // up to an unbiased last-bit step.
    float Dh = h[c][0], Dl = 0.f;
#pragma unroll
    for (int i = 1; i < 9; i++) {
      float s, e;
      two_sum(Dh, h[c][i], s, e);
      Dh = s;
      Dl += e;
    }
    float Sh = 0.f, Sl = 0.f;
#pragma unroll
    for (int i = 1; i < 9; i++) {
      // 16-bit dither: an independent hash per store (a linear
      // congruential sequence per node, as in the plain collision, was
      // measurably worse for the two-component runs)
      const uint32_t r = p.sr_seed ? (rnd(p.sr_seed, hself, c, i) | 1u) : 0u;
      const float v = Store<S>::st_ret(out, i * P + self, h[c][i] + om * (heq[i] - h[c][i]),
                                       p.scale, p.inv_scale, r);
      float s, e;
      two_sum(Sh, v, s, e);
      Sh = s;
      Sl += e;
    }
    float rh, rl;
    two_sum(Dh, -Sh, rh, rl);
    rl += Dl - Sl;
    float h0, rem;
    two_sum(rh, rl, h0, rem);
    if (rem != 0.f && h0 != 0.f) {
      const int step = ((rem > 0.f) == (h0 > 0.f)) ? 1 : -1;
      const float nxt = __int_as_float(__float_as_int(h0) + step);
      // |nxt - h0| is a power of two, so the quotient is exact up to the
      // fast division's last bit: a probability, compared with a uniform
      // variate
      const float pr = __fdividef(fabsf(rem), fabsf(nxt - h0));
      const float u01 = (float)(rnd(p.step_seed, hself, c, 9) >> 8) * (1.0f / 16777216.0f);
      if (u01 < pr) h0 = nxt;
    }
    const uint32_t r0 = p.sr_seed ? (rnd(p.sr_seed, hself, c, 0) | 1u) : 0u;
    Store<S>::st(out, self, h0, p.scale, r0);
    if (p.fields) {
      float *fl = p.fields + (size_t)c * NFIELD * P;
      fl[self] = drho[c];
      fl[P + self] = jx[c] + 0.5f * Fx[c];
      fl[2 * P + self] = jy[c] + 0.5f * Fy[c];
      // sum of the equilibrium populations (Mass_eq of the thermo command)
      fl[3 * P + self] = (heq[0] + ((heq[1] + heq[3]) + (heq[2] + heq[4])) +
                          ((heq[5] + heq[7]) + (heq[6] + heq[8])));
    }
  }
  if (p.uout) {
    // the solvent velocity of Eq. (4)
    float pxs = 0.f, pys = 0.f, rs = 0.f;
#pragma unroll
    for (int c = 0; c < NC; c++) {
      pxs += jx[c] + 0.5f * Fx[c];
      pys += jy[c] + 0.5f * Fy[c];
      rs += rho[c];
    }
    p.uout[self] = pxs / rs;
    p.uout[P + self] = pys / rs;
  }
}

__device__ __forceinline__ f2 both(const float (&a)[2]) { return mk2(a[0], a[1]); }
__device__ __forceinline__ f2 swapped(f2 a) { return mk2(hi(a), lo(a)); }

// the rest population D - S of the mass-exact collision, rounded
// stochastically in its last bit (rem: what h0 leaves out)
__device__ __forceinline__ float last_bit(float h0, float rem, uint32_t word) {
  if (rem == 0.f || h0 == 0.f) return h0;
  const int step = ((rem > 0.f) == (h0 > 0.f)) ? 1 : -1;
  const float nxt = __int_as_float(__float_as_int(h0) + step);
  // |nxt - h0| is a power of two, so the quotient is exact up to the fast
  // division's last bit: a probability, compared with a uniform variate
  const float pr = __fdividef(fabsf(rem), fabsf(nxt - h0));
  const float u01 = (float)(word >> 8) * (1.0f / 16777216.0f);
  return u01 < pr ? nxt : h0;
}

// the equilibrium of lbarith.cuh for two components, in the order of
// operations their runs were validated with (B's from (mx, my); populations'
// error 0.98 of collide_store_me's; in the other order the Shan-Chen ring's
// mass, a random walk of last bits, ended 1.6e-9 off after 300 iterations)
__device__ __forceinline__ void equilibrium_two(f2 drho, f2 ux, f2 uy, f2 mx, f2 my, f2 wa, f2 wd, f2 (&heq)[9]) {
  const f2 xx = vmul(mx, ux), yy = vmul(my, uy), xy = vmul(mx, uy);
  const f2 da = vmul(drho, wa), dd = vmul(drho, wd);
  const f2 third = vset<f2>(1.0f / 3.0f), sixth = vset<f2>(-1.0f / 6.0f);
  const f2 c12 = vset<f2>(1.0f / 12.0f), n12 = vset<f2>(-1.0f / 12.0f), half = vset<f2>(0.5f);
  const f2 A1 = vfma(third, xx, vfma(sixth, yy, da));
  const f2 A2 = vfma(third, yy, vfma(sixth, xx, da));
  const f2 e = vfma(c12, vfma(mx, ux, yy), dd);
  const f2 A5 = vfma(vset<f2>(0.25f), xy, e), A6 = vfma(vset<f2>(-0.25f), xy, e);
  const f2 s = vadd(mx, my), t = vsub(my, mx);
  const f2 B1 = vfma(n12, vsub(s, t), vmul(half, mx));
  const f2 B2 = vfma(n12, vadd(s, t), vmul(half, my));
  heq[1] = vadd(A1, B1);
  heq[3] = vsub(A1, B1);
  heq[2] = vadd(A2, B2);
  heq[4] = vsub(A2, B2);
  heq[5] = vfma(c12, s, A5);
  heq[7] = vfma(n12, s, A5);
  heq[6] = vfma(c12, t, A6);
  heq[8] = vfma(n12, t, A6);
  heq[0] = vfma(vset<f2>(-2.0f), vadd(vadd(A1, A2), vadd(A5, A6)), drho);
}

// collide_store_me for two components, both in every packed operation (low
// half: component 1), its error-free sums included.  h: the pulled
// populations; d their sum; F: the interforce.
template <class S>
__device__ __forceinline__ void collide_store_two(const FluidArgs &p, int x, int y, uint32_t bits,
                                                  const f2 (&h)[9], f2 d, f2 Fx, f2 Fy) {
  const Geometry &g = p.g;
  const int self = y * g.pitch + x;
  const int hself = self + g.yoff * g.pitch;
  const int P = (int)g.plane;
  const f2 rho = vadd(both(p.rho_ref), d), tau = both(p.tau), om = both(p.omega);
  f2 jx, jy;
  momentum_sum(h, jx, jy);
  Fx = vadd(Fx, vfma(rho, both(p.ax), both(p.fx)));
  Fy = vadd(Fy, vfma(rho, both(p.ay), both(p.fy)));
  constexpr uint32_t NB = 0x1efu;
  if ((p.ads[0] | p.ads[1]) && (bits & NB)) {
    float sx, sy;
    wall_sum(bits, sx, sy);
    const f2 a = vmul(mk2(p.ads[0] ? -p.Gads[0] : 0.f, p.ads[1] ? -p.Gads[1] : 0.f), rho);
    Fx = vfma(a, vset<f2>(sx), Fx);
    Fy = vfma(a, vset<f2>(sy), Fy);
  }
  // common velocity sum(j/tau) / sum(rho/tau)
  const f2 nx = vmul(jx, om), ny = vmul(jy, om), nd = vmul(rho, om);
  const f2 num = mk2(lo(nx) + hi(nx), lo(ny) + hi(ny)), den = vset<f2>(lo(nd) + hi(nd));
  const f2 up = vdiv_rn(num, den);
  const f2 tx = vmul(tau, Fx), ty = vmul(tau, Fy);
  const f2 upx = vset<f2>(lo(up)), upy = vset<f2>(hi(up));
  const f2 mx = vfma(rho, upx, tx), my = vfma(rho, upy, ty);
  f2 heq[9];
  equilibrium_two(d, vadd(upx, vdiv_rn(tx, rho)), vadd(upy, vdiv_rn(ty, rho)), mx, my, both(p.wa), both(p.wd),
                  heq);
  if (p.fields || p.uout) {
    const f2 half = vset<f2>(0.5f), px = vfma(half, Fx, jx), py = vfma(half, Fy, jy);
    if (p.fields) {
      const f2 e = equilibrium_sum(heq, 1.0f);
      float *a = p.fields + self, *b = a + NFIELD * P;
      a[0] = lo(d);
      a[P] = lo(px);
      a[2 * P] = lo(py);
      a[3 * P] = lo(e);
      b[0] = hi(d);
      b[P] = hi(px);
      b[2 * P] = hi(py);
      b[3 * P] = hi(e);
    }
    if (p.uout) {
      // the solvent velocity of Eq. (4)
      const float rs = lo(rho) + hi(rho);
      p.uout[self] = (lo(px) + hi(px)) / rs;
      p.uout[P + self] = (lo(py) + hi(py)) / rs;
    }
  }
  // mass-exact collision (collide_store_me): the exact sum D of the pulled
  // values less the exact sum S of the eight stored moving populations
  f2 Dh = h[0], Dl = vset<f2>(0.f), Sh, Sl = vset<f2>(0.f);
#pragma unroll
  for (int i = 1; i < 9; i++) {
    f2 s, e;
    two_sum(Dh, h[i], s, e);
    Dh = s;
    Dl = vadd(Dl, e);
  }
  S *f0 = (S *)p.fout, *f1 = f0 + 9 * P;
#pragma unroll
  for (int i = 1; i < 9; i++) {
    f2 v = vfma(om, vsub(heq[i], h[i]), h[i]);
    if constexpr (sizeof(S) == 4) {
      f0[i * P + self] = lo(v);
      f1[i * P + self] = hi(v);
    } else {
      // 16-bit dither: an independent hash per store
      const uint32_t r0 = p.sr_seed ? (rnd(p.sr_seed, hself, 0, i) | 1u) : 0u;
      const uint32_t r1 = p.sr_seed ? (rnd(p.sr_seed, hself, 1, i) | 1u) : 0u;
      v = mk2(Store<S>::st_ret(f0, i * P + self, lo(v), p.scale, p.inv_scale, r0),
              Store<S>::st_ret(f1, i * P + self, hi(v), p.scale, p.inv_scale, r1));
    }
    if (i == 1) {
      Sh = v;
    } else {
      f2 s, e;
      two_sum(Sh, v, s, e);
      Sh = s;
      Sl = vadd(Sl, e);
    }
  }
  f2 rh, rl, h0, rem;
  two_sum(Dh, vsub(vset<f2>(0.f), Sh), rh, rl);
  rl = vadd(rl, vsub(Dl, Sl));
  two_sum(rh, rl, h0, rem);
  Store<S>::st(f0, self, last_bit(lo(h0), lo(rem), rnd(p.step_seed, hself, 0, 9)), p.scale,
               p.sr_seed ? (rnd(p.sr_seed, hself, 0, 0) | 1u) : 0u);
  Store<S>::st(f1, self, last_bit(hi(h0), hi(rem), rnd(p.step_seed, hself, 1, 9)), p.scale,
               p.sr_seed ? (rnd(p.sr_seed, hself, 1, 0) | 1u) : 0u);
}

// ---------------------------------------------------------------------
// inlet/outlet rules in one rotated form.
//
// Every wall is mapped onto a canonical one whose inward normal n is e1 and
// tangent t is e2; canonical slot k then holds direction PERM[wall][k]:
//   k: 0  1=n  2=t  3=-n  4=-t  5=n+t  6=-n+t  7=-n-t  8=n-t
// With u_n the velocity along n, S = h0 + h2 + h4 + 2 (h3 + h6 + h7) and
// a = rho u_n:
//   velocity styles:  rho = (rho_ref + S)/(1 - u_n), so
//                     a = (rho_ref + S) u_n/(1 - u_n)
//   dirichlet:        u_n = (rho - rho_ref - S)/rho, so a = rho - rho_ref - S
//   h1 = h3 + 2/3 a
//   h5 = h7 - (h2 - h4)/2 + a/6
//   h8 = h6 + (h2 - h4)/2 + a/6
// which is the set of printed rules for each wall and style (inlet: u_n =
// +v, outlet: u_n = -v), written for deviations h = f - w rho_ref.  Either
// way a = m S + b with m and b fixed by the opening (and, for a Poiseuille
// profile, the node's place along it).  16-bit storage forms the dirichlet
// a as rho u_n by the quotient (equilibrium_16 says why): r is then the
// density held, else 0.
// ---------------------------------------------------------------------
template <int WALL> __device__ __forceinline__ constexpr int PERM(int k) {
  // xlo: n=+x t=+y; xhi: n=-x t=+y; ylo: n=+y t=+x; yhi: n=-y t=-x
  return WALL == 0 ? k
       : WALL == 1 ? (k == 1 ? 3 : k == 3 ? 1 : k == 5 ? 6 : k == 6 ? 5 : k == 7 ? 8 : k == 8 ? 7 : k)
       : WALL == 2 ? (k == 1 ? 2 : k == 2 ? 1 : k == 3 ? 4 : k == 4 ? 3 : k == 6 ? 8 : k == 8 ? 6 : k)
                   : (k == 1 ? 4 : k == 2 ? 3 : k == 3 ? 2 : k == 4 ? 1 : k == 5 ? 7 : k == 7 ? 5 : k);
}

__device__ __forceinline__ float hold(float a, float r) { return r != 0.f ? __fmul_rn(r, __fdiv_rn(a, r)) : a; }
__device__ __forceinline__ f2 hold(f2 a, f2 r) { return mk2(hold(lo(a), lo(r)), hold(hi(a), hi(r))); }

template <int WALL, bool S16, class V>
__device__ __forceinline__ void zou_he(const V (&h)[9], V m, V b, V r, V &h1, V &h5, V &h8) {
  constexpr int c0 = PERM<WALL>(0), c2 = PERM<WALL>(2), c3 = PERM<WALL>(3), c4 = PERM<WALL>(4), c6 = PERM<WALL>(6),
                c7 = PERM<WALL>(7);
  const V S = vfma(vset<V>(2.0f), vadd(vadd(h[c3], h[c6]), h[c7]), vadd(vadd(h[c0], h[c2]), h[c4]));
  V a = vfma(S, m, b);
  if (S16) a = hold(a, r);
  const V d = vsub(h[c2], h[c4]), sixth = vset<V>(1.0f / 6.0f);
  h1 = vfma(vset<V>(2.0f / 3.0f), a, h[c3]);
  h5 = vfma(sixth, a, vfma(vset<V>(-0.5f), d, h[c7]));
  h8 = vfma(sixth, a, vfma(vset<V>(0.5f), d, h[c6]));
}

template <int WALL, bool S16>
__device__ __forceinline__ void zou_he_node(float (&h)[9], float m, float b, float r) {
  float h1, h5, h8;
  zou_he<WALL, S16>(h, m, b, r, h1, h5, h8);
  h[PERM<WALL>(1)] = h1;
  h[PERM<WALL>(5)] = h5;
  h[PERM<WALL>(8)] = h8;
}

// m, b and r of component c's rule at coordinate coord along the wall; false
// if the component has no velocity or density style there.  sc: the units
// of h (the rule is homogeneous of degree one in h, drho and rho_ref, so
// scaled storage units take sc = 2^s)
__device__ __forceinline__ bool opening_mb(const OpenSpan &s, const OpenRule &r, int c, int coord, float rho_ref,
                                           float sc, float &m, float &b, float &rho) {
  const int st = (r.bits >> (3 * c)) & 7;
  rho = 0.f;
  if (st == OPEN_DIRICHLET) {
    m = -1.0f;
    b = vmul(r.val[c], sc);
    rho = vadd(vmul(rho_ref, sc), b);
    return true;
  }
  if (st != OPEN_POISEUILLE && st != OPEN_UNIFORM) return false;
  const float v = (st == OPEN_UNIFORM) ? r.val[c] : poiseuille(r.val[c], s.wa0 >> 2, s.a1, coord);
  const float un = ((r.bits >> 6) & 1) == 0 ? v : -v;
  m = __fdiv_rn(un, vsub(1.0f, un));
  b = vmul(vmul(rho_ref, sc), m);
  return true;
}

// apply the velocity/dirichlet rule r of the opening at s to component c's
// h (in units sc)
template <bool S16>
__device__ __forceinline__ void apply_opening(const OpenSpan &s, const OpenRule &r, int c, float (&h)[9],
                                              int x, int y, float rho_ref, float sc = 1.0f) {
  const int wall = span_wall(s);
  float m, b, rho;
  if (!opening_mb(s, r, c, wall <= 1 ? y : x, rho_ref, sc, m, b, rho)) return;
  switch (wall) {
    case 0: zou_he_node<0, S16>(h, m, b, rho); break;
    case 1: zou_he_node<1, S16>(h, m, b, rho); break;
    case 2: zou_he_node<2, S16>(h, m, b, rho); break;
    default: zou_he_node<3, S16>(h, m, b, rho); break;
  }
}

// component c's opening rule at node (x, y) if an opening holds it (the
// rule of a component reads only that component's populations, so the
// interforce kernel applies it per component, to its own node and to the
// ring nodes whose densities it stages); h in unscaled units
template <bool S16>
__device__ __forceinline__ void apply_opening_c(const FluidArgs &p, int c, int x, int y, float (&h)[9]) {
  const Geometry &g = p.g;
  const int gy = grow(g, y);
  if (!(x == 0 || gy == 0 || x == g.nx - 1 || gy == g.gny - 1)) return;
#pragma unroll 1
  for (int k = 0; k < p.nopen; k++) {
    if (!opening_has(p.span[k], x, gy, g.nx, g.gny)) continue;
    apply_opening<S16>(p.span[k], p.rule[k], c, h, x, gy, p.rho_ref[c]);
    return;
  }
}

template <int NC, bool S16>
__device__ __forceinline__ void apply_openings(const FluidArgs &p, int x, int y,
                                               float (&h)[NC][9], float sc = 1.0f) {
  const Geometry &g = p.g;
  const int gy = grow(g, y);  // openings are placed on the whole lattice
  if (!(x == 0 || gy == 0 || x == g.nx - 1 || gy == g.gny - 1)) return;
#pragma unroll 1
  for (int k = 0; k < p.nopen; k++) {
    if (!opening_has(p.span[k], x, gy, g.nx, g.gny)) continue;
#pragma unroll
    for (int c = 0; c < NC; c++) apply_opening<S16>(p.span[k], p.rule[k], c, h[c], x, gy, p.rho_ref[c], sc);
    break;
  }
}

}  // namespace

}  // namespace lbk
