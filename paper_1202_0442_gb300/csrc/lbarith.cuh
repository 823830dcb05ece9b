// lbarith.cuh -- the arithmetic of a single-component collision, written
// once for one node (V = float) and for two nodes at a time (V = f2, packed
// FP32 instructions).
//
// Every operation is spelled out (add, multiply, fused multiply-add), so the
// compiler has no choice in contracting them and the two forms give the same
// bits: a node's update does not depend on the kernel that makes it.
//
// The packed form issues one instruction for two nodes.  The streaming
// kernel issues some 285 instructions per node and sits on the issue limit
// whenever its data comes from L2, so the packed form is what the kernels
// that keep two nodes per thread are built on (k_march.cuh, k_tile.cuh).
#pragma once

#include "lbdev.cuh"

namespace lbk {

namespace {

// two FP32 values in one 64-bit register pair
struct f2 {
  unsigned long long v;
};

__device__ __forceinline__ f2 mk2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float lo(f2 a) { return __uint_as_float((uint32_t)a.v); }
__device__ __forceinline__ float hi(f2 a) { return __uint_as_float((uint32_t)(a.v >> 32)); }

__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ f2 vadd(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 vsub(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 vmul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 vfma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// the same constant in every value
template <class V> __device__ __forceinline__ V vset(float a);
template <> __device__ __forceinline__ float vset<float>(float a) { return a; }
template <> __device__ __forceinline__ f2 vset<f2>(float a) { return mk2(a, a); }

// 1/a, correctly rounded: the hardware's approximation (within one unit in the last
// place, subnormal a included) and one Newton step in fused multiply-adds,
// which rounds correctly from such a start (P. Markstein, IBM J. Res. Dev.
// 34, 1990).  The same bits as __frcp_rn for every a whose reciprocal is a
// normal number (all significands of exponents -126 to 125 compared; one
// unit off at some of 2^126 and 2^127), and unlike it packed but for the
// approximation: porous 1024^2 FP32 9.5 us per iteration against 9.9, 256
// lattices 193 against 216.
__device__ __forceinline__ float vrcp_approx(float a) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ f2 vrcp_approx(f2 a) { return mk2(vrcp_approx(lo(a)), vrcp_approx(hi(a))); }
template <class V>
__device__ __forceinline__ V vrcp(V a) {
  const V r = vrcp_approx(a);
  return vfma(r, vfma(vsub(vset<V>(0.f), a), r, vset<V>(1.0f)), r);
}

__device__ __forceinline__ float vrcp_rn(float a) { return __frcp_rn(a); }
__device__ __forceinline__ f2 vrcp_rn(f2 a) { return mk2(__frcp_rn(lo(a)), __frcp_rn(hi(a))); }
__device__ __forceinline__ f2 vdiv_rn(f2 a, f2 b) { return mk2(__fdiv_rn(lo(a), lo(b)), __fdiv_rn(hi(a), hi(b))); }
// a rounded product that may feed a sum.  Of two nodes: one multiplication
// each, which the compiler does not fuse with the packed sum (it does fuse a
// packed product, one written as a multiply-add with zero as well)
__device__ __forceinline__ float vprod(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ f2 vprod(f2 a, f2 b) {
  return mk2(__fmul_rn(lo(a), lo(b)), __fmul_rn(hi(a), hi(b)));
}

// error-free sum: s + e == a + b exactly (Knuth)
template <class V>
__device__ __forceinline__ void two_sum(V a, V b, V &s, V &e) {
  s = vadd(a, b);
  const V bb = vsub(s, a);
  e = vadd(vsub(a, vsub(s, bb)), vsub(b, bb));
}

// momentum sum_i e_i f_i of one component as an unevaluated sum hi + lo,
// every addition error-free (two_sum): a moment rounded to FP32 feeds its
// rounding error back into the state as a spurious force (the collision
// relaxes toward the computed momentum), which in slow force-driven flows
// is comparable with the force itself
template <class V>
__device__ __forceinline__ void momentum_exact(const V (&f)[9], V &jx, V &jxl, V &jy, V &jyl) {
  V a, ea, b, eb, d, ed, s, es, t, et;
  two_sum(f[1], vsub(vset<V>(0.f), f[3]), a, ea);
  two_sum(f[5], vsub(vset<V>(0.f), f[7]), b, eb);
  two_sum(f[8], vsub(vset<V>(0.f), f[6]), d, ed);
  two_sum(a, b, s, es);
  two_sum(s, d, t, et);
  jx = t;
  jxl = vadd(vadd(vadd(ea, eb), vadd(ed, es)), et);
  two_sum(f[2], vsub(vset<V>(0.f), f[4]), a, ea);
  two_sum(f[6], vsub(vset<V>(0.f), f[8]), d, ed);
  two_sum(a, b, s, es);
  two_sum(s, d, t, et);
  jy = t;
  jyl = vadd(vadd(vadd(ea, eb), vadd(ed, es)), et);
}

// sum_i f_i
template <class V>
__device__ __forceinline__ V density_sum(const V (&f)[9]) {
  return vadd(vadd(vadd(vadd(f[0], f[1]), vadd(f[2], f[3])), vadd(vadd(f[4], f[5]), vadd(f[6], f[7]))), f[8]);
}

// sum_i e_i f_i
template <class V>
__device__ __forceinline__ void momentum_sum(const V (&f)[9], V &jx, V &jy) {
  const V a = vsub(f[1], f[3]), b = vsub(f[2], f[4]), c = vsub(f[5], f[7]), d = vsub(f[6], f[8]);
  jx = vsub(vadd(a, c), d);
  jy = vadd(vadd(b, c), d);
}

// ---------------------------------------------------------------------
// Equilibrium of Eq. (2), generalised by the fluids command to
// f_eq,i = w_i rho [A_i + 3 e.u + 9/2 (e.u)^2 - 3/2 u.u] with A_0 = 9/4 alpha,
// A_{1..8} = 9/5 (1 - alpha), as deviations h_eq,i = f_eq,i - s_i rho_ref
// from the rest state s_i = w_i A_i (s_0 = alpha, wa = s_{1..4} =
// (1 - alpha)/5, wd = s_{5..8} = (1 - alpha)/20; 4/9, 1/9, 1/36 at
// alpha = 4/9), drho = rho - rho_ref, in symmetric/antisymmetric pairs
// (i, opp(i)):
//   A_i = s_i drho + w_i rho (9/2 (e_i.u)^2 - 3/2 u.u),  B_i = 3 w_i rho e_i.u
//   h_eq,i = A_i + B_i,  h_eq,opp(i) = A_i - B_i
// (sum_i s_i = 1, so h_eq,0 = drho - the other eight holds for any alpha).
// With (mx, my) = rho u and the products xx = mx ux, yy = my uy, xy = mx uy
//   A_1 = wa drho + xx/3 - yy/6,   A_2 = wa drho + yy/3 - xx/6
//   A_5 = wd drho + (xx + yy)/12 + xy/4,   A_6 = the same with - xy/4
//   B_5 = rho (ux + uy)/12,   B_6 = rho (uy - ux)/12
// The rounded FP32 weights would make sum h_eq and sum h_eq e miss drho and
// rho u by a fixed relative 1e-8..1e-7, repeated by every collision (a
// spurious force proportional to the momentum).  So the two moments are
// imposed instead: the axis B's come from the target momentum (mx, my)
// minus the diagonal B's (B_1 = mx/2 - (B_5 - B_6) = mx/2 - rho ux/6, B_2 =
// my/2 - (B_5 + B_6)), and h_eq,0 from drho minus the other eight; in exact
// arithmetic both are the formula above.  No plain product feeds a plain sum
// here: the compiler may fuse such a pair in the packed form.
//
// The order of the operations decides the noise.  s_i drho, the largest term
// of a slow flow's A_i, enters by a fused multiply-add (no rounding of its
// own), and the B's come from rho/12 and u rather than from (mx + my)/12,
// whose roundings follow those of the momentum and so repeat along a smooth
// flow.  Error of the FP32 populations against FP64 (2-norm): reactive
// channel 1024 x 512, 200 iterations 1.2e-7 (B's from fused (mx + my)/12 and
// s_i drho rounded 2.2e-7, equilibrium_16's order 1.6e-7); porous 512 x 333,
// 100 iterations 1.4e-7 (2.1e-7, 2.8e-7).
// ---------------------------------------------------------------------
// PM (exact momentum): the products unrounded.  There the rounded ones, which
// repeat at a node of a steady flow, are the largest error left: slow porous
// lattice 64 x 288, 5000 iterations, largest velocity error 1.4e-6 against
// 6.0e-6 rounded (equilibrium_16's order: 1.7e-6).  Without PM they are the
// lower at openings: porous 1024^2, 30 iterations from rest, largest velocity
// error, mean of six media, 0.97e-5 against 1.04e-5 unrounded (1.04e-5).
template <bool PM, class V>
__device__ __forceinline__ void equilibrium(V drho, V rho, V ux, V uy, V mx, V my, V wa, V wd, V (&heq)[9]) {
  const V xx = vmul(mx, ux), yy = vmul(my, uy), xy = vmul(mx, uy);
  const V third = vset<V>(1.0f / 3.0f), sixth = vset<V>(-1.0f / 6.0f);
  const V c12 = vset<V>(1.0f / 12.0f), half = vset<V>(0.5f), nhalf = vset<V>(-0.5f);
  const V A1 = vfma(third, xx, vfma(drho, wa, vmul(sixth, yy)));
  const V A2 = vfma(third, yy, vfma(drho, wa, vmul(sixth, xx)));
  const V e = vfma(drho, wd, vmul(c12, vfma(mx, ux, yy)));
  const V A5 = vfma(vset<V>(0.25f), xy, e), A6 = vfma(vset<V>(-0.25f), xy, e);
  const V r12 = vmul(rho, c12), s = vadd(ux, uy), t = vsub(uy, ux);
  if (PM) {
    const V n12 = vmul(rho, vset<V>(-1.0f / 12.0f)), n6 = vmul(rho, sixth);
    const V B1 = vfma(n6, ux, vmul(half, mx)), B2 = vfma(n6, uy, vmul(half, my));
    heq[1] = vadd(A1, B1);
    heq[3] = vsub(A1, B1);
    heq[2] = vadd(A2, B2);
    heq[4] = vsub(A2, B2);
    heq[5] = vfma(r12, s, A5);
    heq[7] = vfma(n12, s, A5);
    heq[6] = vfma(r12, t, A6);
    heq[8] = vfma(n12, t, A6);
  } else {
    const V B5 = vprod(r12, s), B6 = vprod(r12, t), k = vsub(B5, B6), l = vadd(B5, B6);
    heq[1] = vfma(half, mx, vsub(A1, k));
    heq[3] = vfma(nhalf, mx, vadd(A1, k));
    heq[2] = vfma(half, my, vsub(A2, l));
    heq[4] = vfma(nhalf, my, vadd(A2, l));
    heq[5] = vadd(A5, B5);
    heq[7] = vsub(A5, B5);
    heq[6] = vadd(A6, B6);
    heq[8] = vsub(A6, B6);
  }
  heq[0] = vfma(vset<V>(-2.0f), vadd(vadd(A1, A2), vadd(A5, A6)), drho);
}

// The same equilibrium in the operations that 16-bit storage keeps: its long
// runs were validated with them, and there a single changed rounding moves
// a dither's decision and with it, within some tens of iterations, the
// whole noise pattern.  u is a rounded quotient, the quadratic terms are
// formed from u and rho.
template <class V>
__device__ __forceinline__ void equilibrium_16(V drho, V rho, V ux, V uy, V mx, V my, V wa, V wd, V (&heq)[9]) {
  const V q = vmul(rho, vfma(ux, ux, vmul(uy, uy)));
  const V sp = vadd(ux, uy), sm = vsub(uy, ux);  // e5.u and e6.u
  const V c12 = vset<V>(1.0f / 12.0f), n12 = vset<V>(-1.0f / 12.0f), half = vset<V>(0.5f);
  const V n6 = vset<V>(-1.0f / 6.0f), n24 = vset<V>(-1.0f / 24.0f);
  const V rh = vmul(half, rho), re = vmul(vset<V>(0.125f), rho);
  const V A1 = vfma(q, n6, vfma(drho, wa, vmul(vmul(rh, ux), ux)));
  const V A2 = vfma(q, n6, vfma(drho, wa, vmul(vmul(rh, uy), uy)));
  const V A5 = vfma(q, n24, vfma(drho, wd, vmul(vmul(re, sp), sp)));
  const V A6 = vfma(q, n24, vfma(drho, wd, vmul(vmul(re, sm), sm)));
  const V B5 = vprod(vmul(rho, sp), c12), t6 = vmul(rho, sm);
  const V B1 = vfma(t6, c12, vsub(vmul(half, mx), B5));
  const V B2 = vfma(t6, n12, vsub(vmul(half, my), B5));
  heq[1] = vadd(A1, B1);
  heq[3] = vsub(A1, B1);
  heq[2] = vadd(A2, B2);
  heq[4] = vsub(A2, B2);
  heq[5] = vadd(A5, B5);
  heq[7] = vsub(A5, B5);
  heq[6] = vfma(t6, c12, A6);
  heq[8] = vfma(t6, n12, A6);
  heq[0] = vfma(vset<V>(-2.0f), vadd(vadd(A1, A2), vadd(A5, A6)), drho);
}

// sum of the equilibrium deviations (Mass_eq of the thermo command); un:
// stored units -> physical units
template <class V>
__device__ __forceinline__ V equilibrium_sum(const V (&heq)[9], float un) {
  const V axis = vadd(vadd(heq[1], heq[3]), vadd(heq[2], heq[4]));
  const V diag = vadd(vadd(heq[5], heq[7]), vadd(heq[6], heq[8]));
  return vmul(vadd(vadd(heq[0], axis), diag), vset<V>(un));
}

// Moments and shifted equilibrium momentum of one single-component node
// (or two): j = sum e f (PM: as hi + lo), F the force of the node, mt =
// j + tau F, u = mt / rho.  un: stored units -> physical units (a power of
// two).
template <class V>
struct Node1 {
  V drho, rho, jx, jy, jxl, jyl, Fx, Fy, mx, my, ux, uy;
};

template <class V, bool PM, bool FOLD>
__device__ __forceinline__ void moments1(const V (&h)[9], float rho_ref, float un, Node1<V> &n) {
  n.drho = density_sum(h);
  if (PM) {
    momentum_exact(h, n.jx, n.jxl, n.jy, n.jyl);
  } else {
    momentum_sum(h, n.jx, n.jy);
    n.jxl = n.jyl = vset<V>(0.f);
  }
  if (FOLD) {
    const V u = vset<V>(un);
    n.drho = vmul(n.drho, u);
    n.jx = vmul(n.jx, u);
    n.jy = vmul(n.jy, u);
    if (PM) {
      n.jxl = vmul(n.jxl, u);
      n.jyl = vmul(n.jyl, u);
    }
  }
  n.rho = vadd(vset<V>(rho_ref), n.drho);
}

// S16: 16-bit storage
template <class V, bool PM, bool S16>
__device__ __forceinline__ void shift1(float tau, Node1<V> &n) {
  const V t = vset<V>(tau);
  if (PM) {
    n.mx = vadd(n.jx, vfma(t, n.Fx, n.jxl));
    n.my = vadd(n.jy, vfma(t, n.Fy, n.jyl));
  } else {
    n.mx = vfma(t, n.Fx, n.jx);
    n.my = vfma(t, n.Fy, n.jy);
  }
  const V ir = S16 ? vrcp_rn(n.rho) : vrcp(n.rho);
  n.ux = vprod(n.mx, ir);
  n.uy = vprod(n.my, ir);
}

// h_eq of the node; FOLD: in stored units (it is linear in drho and rho u
// at fixed u), sc = 2^s
template <class V, bool PM, bool FOLD, bool S16>
__device__ __forceinline__ void equilibrium1(const Node1<V> &n, float sc, float wa, float wd, V (&heq)[9]) {
  V d = n.drho, r = n.rho, mx = n.mx, my = n.my;
  if (FOLD) {
    const V s = vset<V>(sc);
    d = vmul(d, s);
    r = vmul(r, s);
    mx = vmul(mx, s);
    my = vmul(my, s);
  }
  if (S16) equilibrium_16(d, r, n.ux, n.uy, mx, my, vset<V>(wa), vset<V>(wd), heq);
  else equilibrium<PM>(d, r, n.ux, n.uy, mx, my, vset<V>(wa), vset<V>(wd), heq);
}

// BGK: h becomes (1 - omega) h + omega h_eq.  For omega >= 1 in that form
// (keep = 1 - omega is exact): its intermediate rounding is that of (1 - omega) h,
// none at tau = 1 and tau = 0.8, where h + omega (h_eq - h) rounds the
// difference at the size of h; a channel started far from equilibrium
// (f = 4 and 1) carries 3.5 times less momentum noise after 150 iterations;
// flows near equilibrium (porous 256^2, 100 iterations) have the same error at
// tau = 0.75 and 1, 1.15 times the other form's at 0.6, 1.01 at 0.52 (0.5 to 0.8 of
// equilibrium_16's with that form).  For omega < 1 as h + omega (h_eq - h):
// the error is the lower there (tau = 1.5: by 3), and the
// node's sums are kept although 1 - omega may be rounded; 16-bit storage
// always takes that form (equilibrium_16).  RX: 0 decided here, 1 the first
// form, 2 the second (decided by the launch: both forms in one
// kernel cost the 32-register streaming kernel 12 bytes of spills and 1.5 %
// at 1024^2).
template <int RX = 0, class V>
__device__ __forceinline__ void relax(V (&h)[9], const V (&heq)[9], float omega, float keep) {
  const V om = vset<V>(omega);
  if (RX == 1 || (RX == 0 && omega >= 1.0f)) {
    const V k = vset<V>(keep);
#pragma unroll
    for (int i = 0; i < 9; i++) h[i] = vfma(om, heq[i], vmul(k, h[i]));
  } else {
#pragma unroll
    for (int i = 0; i < 9; i++) h[i] = vfma(om, vsub(heq[i], h[i]), h[i]);
  }
}

}  // namespace

}  // namespace lbk
