// Hand-written reverse mode (adjoints) of the FP64 point and node arithmetic
// of fdcgks_math.cuh: the GENO interface and node reconstructions (Sec. 3.1,
// Sec. 3.2, App. C), the kinetic interface solve (App. A1-A2, Eq. eq:W-model)
// and the nodal flux (Sec. 2.1).
//
// Each *_adj function recomputes its forward values, then runs the forward
// statements backwards, adding to the adjoints of its inputs the transposed
// partial derivatives times the adjoints of its outputs.  Readings of the
// non-smooth points: the branch the forward took (GENO saturation, chi == 1, the positivity safeguard); at an
// exact tie of min/max the mean of the two one-sided derivatives (what a
// central difference sees), and at |x| = 0 derivative 0; a vanishing
// derivative factor times an infinite one (the time coefficients at tau = 0)
// counts as 0.  __host__ __device__ so that the CPU test suite checks it
// against forward-mode dual numbers on the same arithmetic without a GPU.
#pragma once

#include "fdcgks_math.cuh"

namespace fdk {
namespace rev {

typedef double R;

// sign of x, 0 at x = 0 (the derivative of |x| there, as for the dual numbers)
FD_HD R sgn0(R x) { return x > 0.0 ? 1.0 : x < 0.0 ? -1.0 : 0.0; }

// y = max(a, b) / min(a, b) with the dual numbers' tie rule
FD_HD void max_adj(R a, R b, R yb, R& ab, R& bb) {
  if (b > a) bb += yb;
  else if (a > b) ab += yb;
  else { ab += 0.5 * yb; bb += 0.5 * yb; }
}
FD_HD void min_adj(R a, R b, R yb, R& ab, R& bb) {
  if (b < a) bb += yb;
  else if (a < b) ab += yb;
  else { ab += 0.5 * yb; bb += 0.5 * yb; }
}

// ---------------------------------------------------------------------------
// GENO (Sec. 3.2)
// ---------------------------------------------------------------------------
// adjoint of geno_chi (FP64 product form) with the floor fl added to eps_a:
// chib -> ISb[3], flb
FD_HD void geno_chi_adj(const GenoK<R>& g, const R IS[3], R fl, R chib, R ISb[3], R& flb) {
  if (g.linear || chib == 0.0) return;
  const R m_lo = s_min(IS[1], IS[2]), ISL = s_min(IS[0], m_lo);
  const R m_hi = s_max(IS[1], IS[2]), ISH = s_max(IS[0], m_hi);
  const R D = 0.5 * (IS[1] + IS[2]) - IS[0];
  const R tau = s_abs(D);
  R ea = g.eps_a;
  if (fl != 0.0) ea = ea + fl;
  const R H = ISH + ea, Lo = ISL + ea;
  const R hr = rpow(H, g.r), lr = rpow(Lo, g.r), tr = rpow(tau, g.r);
  const R A = (hr + tr) * lr, B = (lr + tr) * hr, den = A + B;
  const R z = (2.0 * g.C) * (A * (1.0 / den));
  if (z > R(GENO_SAT64)) return;   // saturated: chi constant
  const R e = s_exp(-2.0 * z), ie = 1.0 / (1.0 + e);
  const R alphab = chib * (4.0 * e * ie * ie) * g.C;
  // alpha = 2 A / (A + B)
  const R Ab = alphab * 2.0 * B / (den * den), Bb = -alphab * 2.0 * A / (den * den);
  const R hrb = Ab * lr + Bb * (lr + tr), lrb = Ab * (hr + tr) + Bb * hr, trb = (Ab * lr + Bb * hr);
  const R dpow = g.r == 3 ? 3.0 : 2.0;
  const R Hb = hrb * dpow * (g.r == 3 ? H * H : H), Lob = lrb * dpow * (g.r == 3 ? Lo * Lo : Lo);
  const R taub = trb * dpow * (g.r == 3 ? tau * tau : tau);
  const R Db = taub * sgn0(D);
  if (fl != 0.0) flb += Hb + Lob;
  ISb[0] -= Db;
  ISb[1] += 0.5 * Db;
  ISb[2] += 0.5 * Db;
  R mb = 0.0;
  max_adj(IS[0], m_hi, Hb, ISb[0], mb);
  max_adj(IS[1], IS[2], mb, ISb[1], ISb[2]);
  mb = 0.0;
  min_adj(IS[0], m_lo, Lob, ISb[0], mb);
  min_adj(IS[1], IS[2], mb, ISb[1], ISb[2]);
}

// adjoint of geno_weights (FP64 product form): wb[3] -> ISb[3]
FD_HD void geno_weights_adj(const GenoK<R>& g, const R d[3], const R IS[3], const R wb[3], R ISb[3]) {
  const R e0 = IS[0] + g.eps_w, e1 = IS[1] + g.eps_w, e2 = IS[2] + g.eps_w;
  const R s0 = e0 * e0, s1 = e1 * e1, s2 = e2 * e2;
  const R t0 = d[0] * s1 * s2, t1 = d[1] * s0 * s2, t2 = d[2] * s0 * s1;
  const R S = t0 + t1 + t2, inv = 1.0 / S;
  const R w0 = t0 * inv, w1 = t1 * inv, w2 = t2 * inv;
  const R dot = wb[0] * w0 + wb[1] * w1 + wb[2] * w2;
  const R t0b = (wb[0] - dot) * inv, t1b = (wb[1] - dot) * inv, t2b = (wb[2] - dot) * inv;
  const R s0b = d[1] * s2 * t1b + d[2] * s1 * t2b;
  const R s1b = d[0] * s2 * t0b + d[2] * s0 * t2b;
  const R s2b = d[0] * s1 * t0b + d[1] * s0 * t1b;
  ISb[0] += 2.0 * e0 * s0b;
  ISb[1] += 2.0 * e1 * s1b;
  ISb[2] += 2.0 * e2 * s2b;
}

// The GENO blend of one side: value v = chi PH + (1 - chi) PL, derivative
// d = chi PHx + (1 - chi) PLx, PL = sum w_k q_k, PLx = w0 qx0 + (w1 + w2) dq12.
// Given vb, db and the adjoint of chi, returns the adjoints of PH, PHx, q[3],
// qx0, dq12, IS[3] and the floor fl of the path function.
FD_HD void geno_blend_adj(const GenoK<R>& g, const R dk[3], const R IS[3], R fl, R PH, R PHx, const R q[3], R qx0,
                          R dq12, R vb, R db, R chib, R& PHb, R& PHxb, R qb[3], R& qx0b, R& dq12b, R ISb[3],
                          R& flb) {
  const R chi = geno_chi(g, IS[0], IS[1], IS[2], fl);
  if (chi == 1.0) {
    // the forward skips the blend; chi's derivative is zero there
    PHb += vb;
    PHxb += db;
    return;
  }
  R w[3];
  const R inv = geno_weights(g, dk, IS[0], IS[1], IS[2], w);
  for (int k = 0; k < 3; ++k) w[k] *= inv;
  const R PL = w[0] * q[0] + w[1] * q[1] + w[2] * q[2];
  const R PLx = w[0] * qx0 + (w[1] + w[2]) * dq12;
  const R chib_t = chib + vb * (PH - PL) + db * (PHx - PLx);
  PHb += chi * vb;
  PHxb += chi * db;
  const R PLb = (1.0 - chi) * vb, PLxb = (1.0 - chi) * db;
  R wb[3];
  wb[0] = PLb * q[0] + PLxb * qx0;
  wb[1] = PLb * q[1] + PLxb * dq12;
  wb[2] = PLb * q[2] + PLxb * dq12;
  qb[0] += PLb * w[0];
  qb[1] += PLb * w[1];
  qb[2] += PLb * w[2];
  qx0b += PLxb * w[0];
  dq12b += PLxb * (w[1] + w[2]);
  geno_weights_adj(g, dk, IS, wb, ISb);
  geno_chi_adj(g, IS, fl, chib_t, ISb, flb);
}

// floor of the path function from max |Q| (geno_floor_of with fscale): its
// adjoint flb goes to the entry of largest magnitude (ties: shared, as for
// the dual numbers' nested max)
FD_HD void floor_adj4(const R Q[4], R fscale, R flb, R Qb[4]) {
  if (flb == 0.0 || fscale == 0.0) return;
  const R a0 = s_abs(Q[0]), a1 = s_abs(Q[1]), a2 = s_abs(Q[2]), a3 = s_abs(Q[3]);
  const R m01 = s_max(a0, a1), m23 = s_max(a2, a3), qmax = s_max(m01, m23);
  const R qb = flb * 2.0 * fscale * fscale * qmax;
  R m01b = 0.0, m23b = 0.0, ab[4] = {0.0, 0.0, 0.0, 0.0};
  max_adj(m01, m23, qb, m01b, m23b);
  max_adj(a0, a1, m01b, ab[0], ab[1]);
  max_adj(a2, a3, m23b, ab[2], ab[3]);
  for (int k = 0; k < 4; ++k) Qb[k] += ab[k] * sgn0(Q[k]);
}
FD_HD void floor_adj3(const R Q[3], R fscale, R flb, R Qb[3]) {
  if (flb == 0.0 || fscale == 0.0) return;
  // qmax = max(|Q1|, max(|Q0|, |Q2|)) as in recon_node
  const R a0 = s_abs(Q[0]), a1 = s_abs(Q[1]), a2 = s_abs(Q[2]);
  const R m02 = s_max(a0, a2), qmax = s_max(a1, m02);
  const R qb = flb * 2.0 * fscale * fscale * qmax;
  R m02b = 0.0, ab[3] = {0.0, 0.0, 0.0};
  max_adj(a1, m02, qb, ab[1], m02b);
  max_adj(a0, a2, m02b, ab[0], ab[2]);
  for (int k = 0; k < 3; ++k) Qb[k] += ab[k] * sgn0(Q[k]);
}

// 13/12 t^2 + u^2 / 4 for given t and u: returns (tb, ub)
FD_HD void is_three_adj(R t, R u, R ISb, R& tb, R& ub) {
  tb = (13.0 / 6.0) * t * ISb;
  ub = 0.5 * u * ISb;
}

// 13/3 t^2 + u^2 with t = b - xh, u = 2 b - xh (the sub-stencil with an
// averaged gradient, App. C): adds to bb, xhb
FD_HD void is_grad_adj(R b, R xh, R ISb, R& bb, R& xhb) {
  const R t = b - xh, u = 2.0 * b - xh;
  const R tb = (26.0 / 3.0) * t * ISb, ub = 2.0 * u * ISb;
  bb += tb + 2.0 * ub;
  xhb -= tb + ub;
}

// adjoint of recon_interface (FP64, path-function floor from fscale as in
// geno_floor_of): output adjoints vlb, dlb, chilb, vrb, drb, chirb -> Qb[4],
// Qxb[4] (added).  As the forward: everything in the differences b_k, and no
// indicators on a side that the FP32 screen finds saturated.
FD_HD void recon_interface_adj(const GenoK<R>& g, const R Q[4], const R Qx[4], R h, R ih, R vlb, R dlb, R chilb,
                               R vrb, R drb, R chirb, R Qb[4], R Qxb[4], R fscale = 0.0) {
  const R c64 = 1.0 / 64.0, c30 = 1.0 / 30.0;
  const R b0 = Q[1] - Q[0], b1 = Q[2] - Q[1], b2 = Q[3] - Q[2];
  bool smooth_l = g.linear, smooth_r = g.linear;
  if (!g.linear && fscale == 0.0) screen_iface(g, b0, b1, b2, Qx[0], Qx[3], screen_h(h), smooth_l, smooth_r);
  R b0b = 0.0, b1b = 0.0, b2b = 0.0, PHxb = 0.0, PHlb = 0.0, PHrb = 0.0;
  if (smooth_l) {
    PHlb = vlb;
    PHxb += dlb;
  }
  if (smooth_r) {
    PHrb = vrb;
    PHxb += drb;
  }
  if (!smooth_l || !smooth_r) {
    const R PHx = (b0 + b2 + 46.0 * b1) * (ih * c30) - 0.3 * (Qx[1] + Qx[2]);
    const R fl = geno_floor_of(s_max(s_max(s_abs(Q[0]), s_abs(Q[1])), s_max(s_abs(Q[2]), s_abs(Q[3]))), fscale);
    const R dq12 = b1 * ih, t01 = b1 - b0, t12 = b2 - b1;
    const R s01 = (13.0 / 12.0) * t01 * t01, s12 = (13.0 / 12.0) * t12 * t12;
    R flb = 0.0, dq12b = 0.0, t01b = 0.0, t12b = 0.0, tb, ub;
    // ---- left (App. C1) ----
    if (!smooth_l) {
      const R PH = (22.0 * b1 + b2 - 7.0 * b0 + (Qx[0] + 22.0 * Qx[1] - 7.0 * Qx[2]) * h) * c64;
      const R xh = Qx[0] * h, u1 = b0 + b1, u2 = b2 - 3.0 * b1;
      const R q[3] = {1.25 * b0 - 0.75 * xh, 0.125 * b0 + 0.375 * b1, 0.625 * b1 - 0.125 * b2};
      const R t = b0 - xh, u = 2.0 * b0 - xh;
      const R IS[3] = {(13.0 / 3.0) * t * t + u * u, s01 + 0.25 * u1 * u1, s12 + 0.25 * u2 * u2};
      R qb[3] = {0.0, 0.0, 0.0}, qx0b = 0.0, ISb[3] = {0.0, 0.0, 0.0}, xhb = 0.0;
      geno_blend_adj(g, g.d_iface, IS, fl, PH, PHx, q, 3.0 * b0 * ih - 2.0 * Qx[0], dq12, vlb, dlb, chilb, PHlb,
                     PHxb, qb, qx0b, dq12b, ISb, flb);
      b0b += 1.25 * qb[0] + 0.125 * qb[1] + 3.0 * ih * qx0b;
      b1b += 0.375 * qb[1] + 0.625 * qb[2];
      b2b -= 0.125 * qb[2];
      xhb -= 0.75 * qb[0];
      is_grad_adj(b0, xh, ISb[0], b0b, xhb);
      is_three_adj(t01, u1, ISb[1], tb, ub);
      t01b += tb; b0b += ub; b1b += ub;
      is_three_adj(t12, u2, ISb[2], tb, ub);
      t12b += tb; b2b += ub; b1b -= 3.0 * ub;
      Qxb[0] += h * xhb - 2.0 * qx0b;
    }
    // ---- right (App. C2, formulas for interface j+1/2) ----
    if (!smooth_r) {
      const R PH = (7.0 * b2 - 22.0 * b1 - b0 + (7.0 * Qx[1] - 22.0 * Qx[2] - Qx[3]) * h) * c64;
      const R xh = Qx[3] * h, u1 = b1 + b2, u2 = b0 - 3.0 * b1;
      const R q[3] = {0.75 * xh - 1.25 * b2, -(0.125 * b2 + 0.375 * b1), 0.125 * b0 - 0.625 * b1};
      const R t = b2 - xh, u = 2.0 * b2 - xh;
      const R IS[3] = {(13.0 / 3.0) * t * t + u * u, s12 + 0.25 * u1 * u1, s01 + 0.25 * u2 * u2};
      R qb[3] = {0.0, 0.0, 0.0}, qx0b = 0.0, ISb[3] = {0.0, 0.0, 0.0}, xhb = 0.0;
      geno_blend_adj(g, g.d_iface, IS, fl, PH, PHx, q, 3.0 * b2 * ih - 2.0 * Qx[3], dq12, vrb, drb, chirb, PHrb,
                     PHxb, qb, qx0b, dq12b, ISb, flb);
      b2b += 3.0 * ih * qx0b - 1.25 * qb[0] - 0.125 * qb[1];
      b1b -= 0.375 * qb[1] + 0.625 * qb[2];
      b0b += 0.125 * qb[2];
      xhb += 0.75 * qb[0];
      is_grad_adj(b2, xh, ISb[0], b2b, xhb);
      is_three_adj(t12, u1, ISb[1], tb, ub);
      t12b += tb; b1b += ub; b2b += ub;
      is_three_adj(t01, u2, ISb[2], tb, ub);
      t01b += tb; b0b += ub; b1b -= 3.0 * ub;
      Qxb[3] += h * xhb - 2.0 * qx0b;
    }
    b1b += t01b - t12b + ih * dq12b;
    b0b -= t01b;
    b2b += t12b;
    floor_adj4(Q, fscale, flb, Qb);
  }
  // values relative to Q1 (left) and Q2 (right), shared derivative
  const R hl = c64 * PHlb, hr = c64 * PHrb, hx = ih * c30 * PHxb;
  b0b += hx - 7.0 * hl - hr;
  b1b += 46.0 * hx + 22.0 * (hl - hr);
  b2b += hx + hl + 7.0 * hr;
  Qxb[0] += h * hl;
  Qxb[1] += h * (22.0 * hl + 7.0 * hr) - 0.3 * PHxb;
  Qxb[2] -= h * (7.0 * hl + 22.0 * hr) + 0.3 * PHxb;
  Qxb[3] -= h * hr;
  Qb[0] -= b0b;
  Qb[1] += vlb + b0b - b1b;
  Qb[2] += vrb + b1b - b2b;
  Qb[3] += b2b;
}

// adjoint of recon_node (FP64, floor from fscale): rb -> Qb[3], Qxb[3] (added)
FD_HD void recon_node_adj(const GenoK<R>& g, const R Q[3], const R Qx[3], R h, R ih, R rb, R Qb[3], R Qxb[3],
                          R fscale = 0.0) {
  const R c30 = 1.0 / 30.0;
  const R b0 = Q[1] - Q[0], b1 = Q[2] - Q[1], b = b0 + b1;
  R PHxb = rb, b0b = 0.0, b1b = 0.0, bb = 0.0;
  if (!g.linear && !(fscale == 0.0 && screen_node(g, b0, b1, Qx[0], Qx[2], screen_h(h)))) {
    const R x0 = Qx[0] * h, x2 = Qx[2] * h, t = b1 - b0;
    const R t1 = b0 - x0, u1 = 2.0 * b0 - x0, t2 = b1 - x2, u2 = 2.0 * b1 - x2;
    const R IS[3] = {(13.0 / 12.0) * t * t + 0.25 * b * b, (13.0 / 3.0) * t1 * t1 + u1 * u1,
                     (13.0 / 3.0) * t2 * t2 + u2 * u2};
    const R fl = geno_floor_of(s_max(s_abs(Q[1]), s_max(s_abs(Q[0]), s_abs(Q[2]))), fscale);
    const R chi = geno_chi(g, IS[0], IS[1], IS[2], fl);
    if (chi != 1.0) {
      R ISb[3] = {0.0, 0.0, 0.0}, flb = 0.0, w[3], x0b = 0.0, x2b = 0.0, tb, ub;
      const R PHx = (Qx[0] + 46.0 * Qx[1] + Qx[2]) * c30 - (0.3 * ih) * b;
      const R qx[3] = {0.5 * b * ih, 2.0 * b0 * ih - Qx[0], 2.0 * b1 * ih - Qx[2]};
      const R inv = geno_weights(g, g.d_node, IS[0], IS[1], IS[2], w);
      for (int k = 0; k < 3; ++k) w[k] *= inv;
      const R PLx = w[0] * qx[0] + w[1] * qx[1] + w[2] * qx[2];
      PHxb = chi * rb;
      const R PLxb = (1.0 - chi) * rb;
      const R wb[3] = {PLxb * qx[0], PLxb * qx[1], PLxb * qx[2]};
      geno_weights_adj(g, g.d_node, IS, wb, ISb);
      geno_chi_adj(g, IS, fl, rb * (PHx - PLx), ISb, flb);
      floor_adj3(Q, fscale, flb, Qb);
      bb += 0.5 * ih * PLxb * w[0];
      b0b += 2.0 * ih * PLxb * w[1];
      b1b += 2.0 * ih * PLxb * w[2];
      Qxb[0] -= PLxb * w[1];
      Qxb[2] -= PLxb * w[2];
      is_three_adj(t, b, ISb[0], tb, ub);
      b1b += tb; b0b -= tb; bb += ub;
      is_grad_adj(b0, x0, ISb[1], b0b, x0b);
      is_grad_adj(b1, x2, ISb[2], b1b, x2b);
      Qxb[0] += h * x0b;
      Qxb[2] += h * x2b;
    }
  }
  bb -= 0.3 * ih * PHxb;
  Qxb[0] += c30 * PHxb; Qxb[1] += 46.0 * c30 * PHxb; Qxb[2] += c30 * PHxb;
  b0b += bb;
  b1b += bb;
  Qb[0] -= b0b;
  Qb[1] += b0b - b1b;
  Qb[2] += b1b;
}

// Adjoint of the reconstruction of one 4-point line in conservative
// components with the positivity safeguard (recon_line_ld): x[e * 8 + f] the
// line's inputs (entry e, field f: 0-3 W, 4-7 the averaged gradient along the
// line); vb[0..3][c] the adjoints of the left value, left derivative, right
// value and right derivative of component c; chib that of the line's chi
// (the smaller of the two sides' chi of rho, 0 where the safeguard acts).
// Adds to xb[32].  radj(Q, Qx, vlb, dlb, chilb, vrb, drb, chirb, Qb, Qxb)
// runs recon_interface_adj for one component (an out-of-line copy on the GPU)
// with the same fscale (the path-function floor, geno_floor_of).
// The forward of that line (recon_line_ld's arithmetic, with the floor):
// v[0..3][c] = left value, left derivative, right value, right derivative;
// chi of the flux; cl0, cr0 the two sides' chi of rho; fixl / fixr whether
// the safeguard replaced a side.
FD_HD void recon_line_fwd(const GenoK<R>& g, const R* x, R h, R ih, R fscale, R v[4][4], R& chi, R& cl0, R& cr0,
                          bool& fixl, bool& fixr) {
  for (int c = 0; c < 4; ++c) {
    const R Q[4] = {x[c], x[8 + c], x[16 + c], x[24 + c]};
    const R Qx[4] = {x[4 + c], x[12 + c], x[20 + c], x[28 + c]};
    R cl, cr;
    recon_interface(g, Q, Qx, h, ih, v[0][c], v[1][c], cl, v[2][c], v[3][c], cr, fscale);
    if (c == 0) { cl0 = cl; cr0 = cr; }
  }
  chi = s_min(cl0, cr0);
  fixl = !physical_state(v[0]);
  fixr = !physical_state(v[2]);
  for (int c = 0; c < 4; ++c) {
    if (fixl) { v[0][c] = x[8 + c]; v[1][c] = 0.0; }
    if (fixr) { v[2][c] = x[16 + c]; v[3][c] = 0.0; }
  }
  if (fixl || fixr) chi = 0.0;
}

template <class RADJ>
FD_HD void recon_line_adj(const GenoK<R>& g, const R* x, R h, R ih, const R vb[4][4], R chib, R* xb, RADJ radj,
                          R fscale = 0.0) {
  R v[4][4], chi, cl0, cr0;
  bool fixl, fixr;
  recon_line_fwd(g, x, h, ih, fscale, v, chi, cl0, cr0, fixl, fixr);
  R chilb = 0.0, chirb = 0.0;
  if (!fixl && !fixr) min_adj(cl0, cr0, chib, chilb, chirb);
  for (int c = 0; c < 4; ++c) {
    // a replaced side takes the value of its node (entry 1 left, 2 right) and a zero slope
    if (fixl) xb[8 + c] += vb[0][c];
    if (fixr) xb[16 + c] += vb[2][c];
    const R Q[4] = {x[c], x[8 + c], x[16 + c], x[24 + c]};
    const R Qx[4] = {x[4 + c], x[12 + c], x[20 + c], x[28 + c]};
    R Qb[4] = {0.0, 0.0, 0.0, 0.0}, Qxb[4] = {0.0, 0.0, 0.0, 0.0};
    radj(Q, Qx, fixl ? 0.0 : vb[0][c], fixl ? 0.0 : vb[1][c], c == 0 ? chilb : 0.0, fixr ? 0.0 : vb[2][c],
         fixr ? 0.0 : vb[3][c], c == 0 ? chirb : 0.0, Qb, Qxb);
    for (int e = 0; e < 4; ++e) {
      xb[e * 8 + c] += Qb[e];
      xb[e * 8 + 4 + c] += Qxb[e];
    }
  }
}

// ---------------------------------------------------------------------------
// Closed-form moments (gas_state, prim_grad, prim_rate, cons_rate, euler_flux,
// euler_flux_rate, stress_flux, half_moments, half_side, half_flux): each
// reverse adds the adjoints of its inputs, given those of its outputs.  A
// state's or gradient's adjoint is kept in the struct of the value itself.
// ---------------------------------------------------------------------------
typedef GasState<R> Gas;
typedef PrimGrad<R> Grad;
FD_HD Gas gas_zero() { return Gas{0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0}; }
FD_HD Grad grad_zero() { return Grad{0.0, 0.0, 0.0, 0.0}; }

FD_HD void gas_state_adj(const R W[4], R gm1, const Gas& g, const Gas& gb, R Wb[4]) {
  const R pb = gm1 * (gb.p + gb.th * g.ir);                    // th = p ir, p = gm1 (W3 - W0 (U^2 + V^2)/2)
  const R Ub = gb.U - W[0] * g.U * pb, Vb = gb.V - W[0] * g.V * pb;
  const R irb = gb.ir + gb.th * g.p + gb.en * W[3] + Ub * W[1] + Vb * W[2];
  Wb[0] += gb.rho - 0.5 * (g.U * g.U + g.V * g.V) * pb - irb * g.ir * g.ir;
  Wb[1] += Ub * g.ir;
  Wb[2] += Vb * g.ir;
  Wb[3] += pb + gb.en * g.ir;
}

FD_HD void prim_grad_adj(const Gas& g, R gm1, const R D[4], const Grad& q, const Grad& qb, Gas& gb, R Db[4]) {
  const R tb = gm1 * qb.t, ub = qb.u - g.U * tb, vb = qb.v - g.V * tb;
  gb.en -= D[0] * tb;
  gb.U -= q.u * tb + D[0] * ub;
  gb.V -= q.v * tb + D[0] * vb;
  Db[0] += qb.d - g.en * tb - g.V * vb - g.U * ub;
  Db[1] += ub;
  Db[2] += vb;
  Db[3] += tb;
}

FD_HD void prim_rate_adj(const Gas& g, R gm1, const Grad& x, const Grad& y, const Grad& qb, Gas& gb, Grad& xb,
                         Grad& yb) {
  const R div = x.u + y.v, divb = qb.d + gm1 * g.th * qb.t;
  gb.U -= qb.d * x.d + qb.u * x.u + qb.v * x.v + qb.t * x.t;
  gb.V -= qb.d * y.d + qb.u * y.u + qb.v * y.v + qb.t * y.t;
  gb.th -= qb.u * x.d + qb.v * y.d + gm1 * div * qb.t;
  xb.d -= g.U * qb.d + g.th * qb.u;
  xb.u -= g.U * qb.u + divb;
  xb.v -= g.U * qb.v;
  xb.t -= g.U * qb.t + qb.u;
  yb.d -= g.V * qb.d + g.th * qb.v;
  yb.u -= g.V * qb.u;
  yb.v -= g.V * qb.v + divb;
  yb.t -= g.V * qb.t + qb.v;
}

FD_HD void cons_rate_adj(const Gas& g, R hN, const Grad& q, const R Wb[4], Gas& gb, Grad& qb) {
  gb.U += q.d * Wb[1] + q.u * Wb[3];
  gb.V += q.d * Wb[2] + q.v * Wb[3];
  gb.en += q.d * Wb[3];
  qb.d += Wb[0] + g.U * Wb[1] + g.V * Wb[2] + g.en * Wb[3];
  qb.u += Wb[1] + g.U * Wb[3];
  qb.v += Wb[2] + g.V * Wb[3];
  qb.t += hN * Wb[3];
}

FD_HD void euler_flux_adj(const Gas& g, const R W[4], const R Fb[4], Gas& gb, R Wb[4]) {
  Wb[1] += Fb[0] + g.U * Fb[1] + g.V * Fb[2];
  Wb[3] += g.U * Fb[3];
  gb.U += W[1] * Fb[1] + (W[3] + g.p) * Fb[3];
  gb.V += W[1] * Fb[2];
  gb.p += Fb[1] + g.U * Fb[3];
}

FD_HD void euler_flux_rate_adj(const Gas& g, const Grad& q, const R Wq[4], const R Fb[4], Gas& gb, Grad& qb,
                               R Wqb[4]) {
  const R pq = g.th * q.d + q.t, pqb = Fb[1] + g.U * Fb[3], quFb = q.u * Fb[3];
  gb.U += (Wq[1] + q.u) * Fb[1] + q.v * Fb[2] + (Wq[3] + pq) * Fb[3];
  gb.V += Wq[1] * Fb[2];
  gb.en += quFb;
  gb.th += quFb + q.d * pqb;
  qb.d += g.th * pqb;
  qb.t += pqb;
  qb.u += g.U * Fb[1] + (g.en + g.th) * Fb[3];
  qb.v += g.U * Fb[2];
  Wqb[1] += Fb[0] + g.U * Fb[1] + g.V * Fb[2];
  Wqb[3] += g.U * Fb[3];
}

FD_HD void stress_flux_adj(const Gas& g, R K, R gm1, const Grad& x, const Grad& y, const R Sb[4], Gas& gb, Grad& xb,
                           Grad& yb) {
  const R A = 2.0 * x.u - gm1 * (x.u + y.v), B = x.v + y.u, c = 0.5 * K + 2.0;
  const R s1 = Sb[1] + g.U * Sb[3], s2 = Sb[2] + g.V * Sb[3], s1p = g.th * s1, s2p = g.th * s2;
  gb.U += g.th * A * Sb[3];
  gb.V += g.th * B * Sb[3];
  gb.th += A * s1 + B * s2 + c * x.t * Sb[3];
  xb.u += (2.0 - gm1) * s1p;
  yb.v -= gm1 * s1p;
  xb.v += s2p;
  yb.u += s2p;
  xb.t += c * g.th * Sb[3];
}

// half_moments with sl = 1/sqrt(2 theta): Mb -> U, theta (Mb is used up)
FD_HD void half_moments_adj(const Gas& g, int sign, R sl, const R M[7], R Mb[7], Gas& gb) {
  for (int n = 4; n >= 0; --n) {
    const R b = Mb[n + 2], nb = R(n + 1) * b;
    Mb[n + 1] += g.U * b;
    Mb[n] += g.th * nb;
    gb.U += M[n + 1] * b;
    gb.th += M[n] * nb;
  }
  // M1 = U M0 + sign e sl theta/sqrt(pi), M0 = erfc(-sign x)/2, e = exp(-x^2), x = sl U
  const R x = sl * g.U, sg = R(sign), c = 0.56418958354775628695, b1 = Mb[1];
  R e, ec;
  exp_erfc(x, e, ec);
  const R ce = c * e, m0b = Mb[0] + g.U * b1;
  const R xb = sg * (ce * m0b - 2.0 * x * ce * (sl * g.th) * b1);
  const R slb = sg * ce * g.th * b1 + g.U * xb;
  gb.U += M[0] * b1 + sl * xb;
  gb.th += sg * ce * sl * b1 - sl * sl * sl * slb;
}

// one slope s0, s1, s3 = t/theta (t = q.t/theta) of half_side: the adjoints of
// t, s0 (its integrated form), s1 and s3
FD_HD void slope_adj(const Gas& g, R ith, R cU, const Grad& q, R t, R s1, R s3, R tb, R s0b, R s1b, R s3b, Gas& gb,
                     R& cUb, R& ithb, Grad& qb) {
  qb.d += s0b;
  tb -= 0.5 * s0b;
  s1b -= g.U * s0b;
  s3b -= cU * s0b + g.U * s1b;
  cUb -= s3 * s0b;
  gb.U -= s1 * s0b + s3 * s1b;
  qb.u += ith * s1b;
  tb += ith * s3b;
  qb.t += ith * tb;
  ithb += q.u * s1b + t * s3b + q.t * tb;
}

// sb: adjoints of half_side's outputs (M unused; rho and V go to the state)
FD_HD void half_side_adj(const Gas& g, R N, R ith, const Grad& gx, const Grad& gy, const Grad& gt,
                         const HalfSide<R>& s, const HalfSide<R>& sb, Gas& gb, Grad& xb, Grad& yb, Grad& tb) {
  const R cU = 0.5 * g.U * g.U, V = g.V, th = g.th, Nh = s.Nh;
  const R ta = gx.t * ith, a3 = ta * ith, a1 = s.e2 - 0.5 * V * (gy.t * ith * ith);
  const R tb_ = gy.t * ith, b3 = tb_ * ith, b1 = gy.u * ith - g.U * b3;
  const R b0 = gy.d - 0.5 * tb_ - g.U * b1 - cU * b3;
  const R tA = gt.t * ith, A3 = tA * ith;
  R cUb = 0.0, ithb = 0.0;
  const R Nhb = sb.Nh + tA * sb.AX0 + V * tb_ * sb.X0 + ta * sb.X1;
  gb.rho += sb.rho;
  gb.V += sb.V + b0 * sb.e0 + b1 * sb.e1 + 0.5 * b3 * sb.e2 + Nh * tb_ * sb.X0 + gy.v * sb.c0;
  gb.th += gy.v * sb.X0 + (b0 + tb_) * sb.c0 + b1 * sb.c1 + 0.5 * N * Nhb;
  xb.v += sb.c1;
  yb.v += sb.e0 + th * sb.X0 + V * sb.c0;
  tb.v += sb.Ac0;
  slope_adj(g, ith, cU, gt, tA, s.Ae1, A3, Nh * sb.AX0, sb.Ae0, sb.Ae1, 0.5 * sb.Ae2, gb, cUb, ithb, tb);
  slope_adj(g, ith, cU, gx, ta, a1, a3, Nh * sb.X1, sb.e1, sb.e2, 0.5 * sb.e3, gb, cUb, ithb, xb);
  slope_adj(g, ith, cU, gy, tb_, b1, b3, V * Nh * sb.X0 + th * sb.c0 + 0.5 * sb.c2, V * sb.e0 + th * sb.c0,
            V * sb.e1 + th * sb.c1, 0.5 * V * sb.e2, gb, cUb, ithb, yb);
  gb.U += g.U * cUb;
  gb.th -= ith * ith * ithb;
}

// half_flux for the weights k[0..2] = (k3, k4, k5): the adjoints Fb, Wb of the
// sums it adds to -> those of the side (into sb, M's included) and of k
FD_HD void half_flux_adj(const HalfSide<R>& s, const R k[3], const R Fb[4], const R Wb[4], HalfSide<R>& sb, R kb[3]) {
  const R q3 = s.rho * k[0], q4 = k[1], q5 = k[2];
  const R e[4] = {q3 + q4 * s.e0 + q5 * s.Ae0, q4 * s.e1 + q5 * s.Ae1, q4 * s.e2 + q5 * s.Ae2, q4 * s.e3};
  const R X0 = q4 * s.X0 + q5 * s.AX0, X1 = q4 * s.X1;
  const R c0 = q4 * s.c0 + q5 * s.Ac0, c1 = q4 * s.c1, c2 = q4 * s.c2;
  const R* M = s.M;
  const R V = s.V, hV2 = 0.5 * V * V;
  const R T0 = e[0] * M[0] + e[1] * M[1] + e[2] * M[2] + e[3] * M[3];
  const R T1 = e[0] * M[1] + e[1] * M[2] + e[2] * M[3] + e[3] * M[4];
  const R C0 = c0 * M[0] + c1 * M[1] + c2 * M[2], C1 = c0 * M[1] + c1 * M[2] + c2 * M[3];
  const R E0b = Wb[3], E1b = Fb[3], C0b = Wb[2] + V * Wb[3], C1b = Fb[2] + V * Fb[3];
  const R Tb[4] = {Wb[0] + V * Wb[2] + hV2 * Wb[3] + s.Nh * E0b,
                   Wb[1] + Fb[0] + V * Fb[2] + hV2 * Fb[3] + s.Nh * E1b, Fb[1] + 0.5 * E0b, 0.5 * E1b};
  sb.V += T0 * Wb[2] + (C0 + V * T0) * Wb[3] + T1 * Fb[2] + (C1 + V * T1) * Fb[3];
  sb.Nh += T0 * E0b + T1 * E1b;
  const R X0b = M[0] * E0b + M[1] * E1b, X1b = M[1] * E0b + M[2] * E1b;
  const R c0b = M[0] * C0b + M[1] * C1b, c1b = M[1] * C0b + M[2] * C1b, c2b = M[2] * C0b + M[3] * C1b;
  sb.M[0] += X0 * E0b + c0 * C0b;
  sb.M[1] += X1 * E0b + X0 * E1b + c1 * C0b + c0 * C1b;
  sb.M[2] += X1 * E1b + c2 * C0b + c1 * C1b;
  sb.M[3] += c2 * C1b;
  R eb[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int t = 0; t < 4; ++t)
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      eb[m] += M[t + m] * Tb[t];
      sb.M[t + m] += e[m] * Tb[t];
    }
  sb.e0 += q4 * eb[0];
  sb.e1 += q4 * eb[1];
  sb.e2 += q4 * eb[2];
  sb.e3 += q4 * eb[3];
  sb.X0 += q4 * X0b;
  sb.X1 += q4 * X1b;
  sb.c0 += q4 * c0b;
  sb.c1 += q4 * c1b;
  sb.c2 += q4 * c2b;
  sb.Ae0 += q5 * eb[0];
  sb.Ae1 += q5 * eb[1];
  sb.Ae2 += q5 * eb[2];
  sb.AX0 += q5 * X0b;
  sb.Ac0 += q5 * c0b;
  const R q4b = s.e0 * eb[0] + s.e1 * eb[1] + s.e2 * eb[2] + s.e3 * eb[3] + s.X0 * X0b + s.X1 * X1b + s.c0 * c0b +
                s.c1 * c1b + s.c2 * c2b;
  const R q5b = s.Ae0 * eb[0] + s.Ae1 * eb[1] + s.Ae2 * eb[2] + s.AX0 * X0b + s.Ac0 * c0b;
  sb.rho += k[0] * eb[0];
  kb[0] += s.rho * eb[0];
  kb[1] += q4b;
  kb[2] += q5b;
}

FD_HD void half_side_zero(HalfSide<R>& s) {
  for (int n = 0; n < 7; ++n) s.M[n] = 0.0;
  s.rho = s.V = s.Nh = s.e0 = s.e1 = s.e2 = s.e3 = s.X0 = s.X1 = s.c0 = s.c1 = s.c2 = 0.0;
  s.Ae0 = s.Ae1 = s.Ae2 = s.AX0 = s.Ac0 = 0.0;
}

// one side of the interface solve: everything that hangs on W (state), D (its
// normal derivative) and Dt (the tangential one)
struct SideFwd {
  Gas g;
  Grad x, y, t;
  R sl, Wq[4];
  HalfSide<R> s;
};
FD_HD void side_fwd(const R W[4], const R D[4], const R Dt[4], int sign, R K, R gm1, SideFwd& f) {
  f.g = gas_state(W, gm1);
  f.sl = s_rsqrt(2.0 * f.g.th);
  half_moments(f.g, sign, f.sl, f.s.M);
  f.x = prim_grad(f.g, gm1, D);
  f.y = prim_grad(f.g, gm1, Dt);
  f.t = prim_rate(f.g, gm1, f.x, f.y);
  half_side(f.g, K + 1.0, 2.0 * f.sl * f.sl, f.x, f.y, f.t, f.s);
  cons_rate(f.g, 0.5 * K + 1.0, f.t, f.Wq);
}
// sb: adjoint of the half-space quantities, Wqb of W_t, W0b of the equilibrium
// state rho (M0, M1, V M0, (M2 + (N theta + V^2) M0)/2) summed over the sides
FD_HD void side_adj(const R W[4], const R D[4], const R Dt[4], int sign, R K, R gm1, const SideFwd& f, HalfSide<R>& sb,
                    const R Wqb[4], const R W0b[4], Gas& gb, R Wb[4], R Db[4], R Dtb[4]) {
  const Gas& g = f.g;
  const R* M = f.s.M;
  const R N = K + 1.0, h = N * g.th + g.V * g.V, r0 = g.rho * M[0];
  gb.rho += M[0] * W0b[0] + M[1] * W0b[1] + g.V * M[0] * W0b[2] + 0.5 * (M[2] + h * M[0]) * W0b[3];
  gb.V += r0 * (W0b[2] + g.V * W0b[3]);
  gb.th += 0.5 * N * r0 * W0b[3];
  sb.M[0] += g.rho * (W0b[0] + g.V * W0b[2] + 0.5 * h * W0b[3]);
  sb.M[1] += g.rho * W0b[1];
  sb.M[2] += 0.5 * g.rho * W0b[3];
  Grad xb = grad_zero(), yb = grad_zero(), tb = grad_zero();
  half_side_adj(g, N, 2.0 * f.sl * f.sl, f.x, f.y, f.t, f.s, sb, gb, xb, yb, tb);
  cons_rate_adj(g, 0.5 * K + 1.0, f.t, Wqb, gb, tb);
  prim_rate_adj(g, gm1, f.x, f.y, tb, gb, xb, yb);
  prim_grad_adj(g, gm1, D, f.x, xb, gb, Db);
  prim_grad_adj(g, gm1, Dt, f.y, yb, gb, Dtb);
  half_moments_adj(g, sign, f.sl, M, sb.M, gb);
  gas_state_adj(W, gm1, g, gb, Wb);
}

// heat flux of the energy flux relative to (U0, V0), x-normal:
// adds hb times its partial derivatives to Fb, Wb, U0b, V0b
FD_HD void heat_flux_x_adj(const R F[4], const R W[4], R U0, R V0, R hb, R Fb[4], R Wb[4], R& U0b, R& V0b) {
  Fb[3] += hb;
  Wb[3] -= U0 * hb;
  Fb[1] -= U0 * hb;
  Fb[2] -= V0 * hb;
  Wb[1] += (1.5 * U0 * U0 + 0.5 * V0 * V0) * hb;
  Wb[2] += U0 * V0 * hb;
  Wb[0] -= 0.5 * U0 * (U0 * U0 + V0 * V0) * hb;
  U0b += hb * (-W[3] - F[1] + 3.0 * U0 * W[1] + V0 * W[2] - 0.5 * (3.0 * U0 * U0 + V0 * V0) * W[0]);
  V0b += hb * (-F[2] + V0 * W[1] + U0 * W[2] - U0 * V0 * W[0]);
}
// time coefficients of the interface distribution (time_coef): the adjoints
// of cn[6], ct[6], E, e1 -> d/dtau
FD_HD R time_coef_adj(R tau, R dt, R inv_dt, const R cnb_in[6], const R ctb_in[6], R Eb, R e1b) {
  const R em = s_expm1(-0.5 * dt / tau);
  const R Eh = 1.0 + em, e1h = -em, E = Eh * Eh, e1 = -em * (em + 2.0);
  R cnb[3], ctb[3], taub = 0.0;
  // cn3 = 1 - cn0, ct3 = -ct0, cn4 = -tau - cn1, ct4 = -ct1, cn5 = -tau - cn2, ct5 = 1 - ct2
  cnb[0] = cnb_in[0] - cnb_in[3];
  ctb[0] = ctb_in[0] - ctb_in[3];
  cnb[1] = cnb_in[1] - cnb_in[4];
  ctb[1] = ctb_in[1] - ctb_in[4];
  cnb[2] = cnb_in[2] - cnb_in[5];
  ctb[2] = ctb_in[2] - ctb_in[5];
  taub -= cnb_in[4] + cnb_in[5];
  R Ehb = 0.0, e1hb = 0.0;
  for (int half = 0; half < 2; ++half) {
    // Ch (d = dt/2, with Eh, e1h) and Cf (d = dt, with E, e1)
    const R d = half ? 0.5 * dt : dt;
    const R EE = half ? Eh : E, ee = half ? e1h : e1;
    R Cb[3];
    for (int k = 0; k < 3; ++k)
      Cb[k] = half ? 4.0 * inv_dt * cnb[k] - 8.0 * inv_dt * inv_dt * ctb[k]
                   : -inv_dt * cnb[k] + 4.0 * inv_dt * inv_dt * ctb[k];
    // C0 = d - tau ee, C1 = -tau d (1 + EE) + 2 tau^2 ee, C2 = d^2/2 - tau d + tau^2 ee
    taub += -ee * Cb[0] + (-d * (1.0 + EE) + 4.0 * tau * ee) * Cb[1] + (-d + 2.0 * tau * ee) * Cb[2];
    const R eeb = -tau * Cb[0] + 2.0 * tau * tau * Cb[1] + tau * tau * Cb[2];
    const R EEb = -tau * d * Cb[1];
    if (half) { Ehb += EEb; e1hb += eeb; }
    else { Eb += EEb; e1b += eeb; }
  }
  // E = Eh^2, e1 = -em (em + 2), Eh = 1 + em, e1h = -em
  Ehb += 2.0 * Eh * Eb;
  const R emb = Ehb - e1hb - (2.0 * em + 2.0) * e1b;
  // em = expm1(-dt / (2 tau)): d em / d tau = (em + 1) dt / (2 tau^2); zero when em + 1 is
  if (emb != 0.0 && em + 1.0 != 0.0) taub += emb * (em + 1.0) * 0.5 * dt / (tau * tau);
  return taub;
}

// ---------------------------------------------------------------------------
// kinetic interface solve, x-normal (iface_solve_x): output adjoints ob ->
// input adjoints (added)
// ---------------------------------------------------------------------------
FD_HD void iface_solve_x_adj(const GasK<R>& gas, const R Wl[4], const R Wr[4], const R Wln[4], const R Wrn[4],
                             const R Wt[4], bool want_n, const IfaceOut<R>& ob, R Wlb[4], R Wrb[4], R Wlnb[4],
                             R Wrnb[4], R Wtb[4]) {
  const R K = gas.K, gm1 = gas.gm1, N = K + 1.0, hN = 0.5 * K + 1.0;
  // ---- forward ----
  SideFwd l, r;
  side_fwd(Wl, Wln, Wt, +1, K, gm1, l);
  side_fwd(Wr, Wrn, Wt, -1, K, gm1, r);
  R W0[4], x1[4], W0q[4], FE[4], FQ[4], FS[4];
  {
    const R ml = l.g.rho * l.s.M[0], mr = r.g.rho * r.s.M[0];
    W0[0] = ml + mr;
    W0[1] = l.g.rho * l.s.M[1] + r.g.rho * r.s.M[1];
    W0[2] = l.g.V * ml + r.g.V * mr;
    W0[3] = 0.5 * (l.g.rho * (l.s.M[2] + N * l.g.th * l.s.M[0] + l.g.V * l.g.V * l.s.M[0]) +
                   r.g.rho * (r.s.M[2] + N * r.g.th * r.s.M[0] + r.g.V * r.g.V * r.s.M[0]));
  }
  const Gas g0 = gas_state(W0, gm1);
  for (int k = 0; k < 4; ++k) x1[k] = 0.5 * (Wln[k] + Wrn[k]);
  const Grad gx = prim_grad(g0, gm1, x1), gy = prim_grad(g0, gm1, Wt), gt = prim_rate(g0, gm1, gx, gy);
  cons_rate(g0, hN, gt, W0q);
  euler_flux(g0, W0, FE);
  euler_flux_rate(g0, gt, W0q, FQ);
  stress_flux(g0, K, gm1, gx, gy, FS);
  const R ip0 = 1.0 / g0.p, dp = l.g.p - r.g.p, sp = l.g.p + r.g.p;
  const R tau = gas.c1 * gas.dt + gas.mu * ip0 + gas.c2 * gas.dt * s_abs(dp) / sp;
  const TimeCoef<R> tc = time_coef(tau, gas.dt, gas.inv_dt);
  const R E = tc.E, e1 = tc.e1;

  // ---- reverse ----
  HalfSide<R> lb, rb;
  half_side_zero(lb);
  half_side_zero(rb);
  Gas g0b = gas_zero();
  R W0b[4] = {0.0, 0.0, 0.0, 0.0}, W0qb[4] = {0.0, 0.0, 0.0, 0.0};
  R FEb[4] = {0.0, 0.0, 0.0, 0.0}, FQb[4] = {0.0, 0.0, 0.0, 0.0}, FSb[4] = {0.0, 0.0, 0.0, 0.0};
  R cnb[6] = {0, 0, 0, 0, 0, 0}, ctb[6] = {0, 0, 0, 0, 0, 0}, Eb = 0.0, e1b = 0.0, Wlqb[4], Wrqb[4];
  // set 0: the values (cn), set 1: the time derivatives (ct)
  for (int set = want_n ? 0 : 1; set < 2; ++set) {
    const R* c = set ? tc.ct : tc.cn;
    R* cb = set ? ctb : cnb;
    const R kq = c[2] - c[1];
    R F[4], We[4], Fb[4], Web[4];
    for (int k = 0; k < 4; ++k) {
      F[k] = c[0] * FE[k] + kq * FQ[k] + c[1] * FS[k];
      We[k] = c[0] * W0[k] + kq * W0q[k];
    }
    half_flux(l.s, c[3], c[4], c[5], F, We);
    half_flux(r.s, c[3], c[4], c[5], F, We);
    for (int k = 0; k < 4; ++k) {
      // o.F = F, o.W(l,r) = e1 We + E W(l,r); for set 1 o.Ft, o.W(l,r)t with W(l,r)_t
      const R ol = set ? ob.Wlt[k] : ob.Wl[k], orr = set ? ob.Wrt[k] : ob.Wr[k];
      Fb[k] = set ? ob.Ft[k] : ob.F[k];
      Web[k] = e1 * (ol + orr);
      e1b += We[k] * (ol + orr);
      if (set) {
        Eb += l.Wq[k] * ol + r.Wq[k] * orr;
        Wlqb[k] = E * ol;
        Wrqb[k] = E * orr;
      } else {
        Eb += Wl[k] * ol + Wr[k] * orr;
        Wlb[k] += E * ol;
        Wrb[k] += E * orr;
      }
    }
    // Prandtl correction F3 += prfix q(F, We) (F above is the sum before it)
    if (gas.prfix != 0.0) heat_flux_x_adj(F, We, g0.U, g0.V, gas.prfix * Fb[3], Fb, Web, g0b.U, g0b.V);
    R kqb = 0.0;
    for (int k = 0; k < 4; ++k) {
      cb[0] += FE[k] * Fb[k] + W0[k] * Web[k];
      cb[1] += FS[k] * Fb[k];
      kqb += FQ[k] * Fb[k] + W0q[k] * Web[k];
      FEb[k] += c[0] * Fb[k];
      FQb[k] += kq * Fb[k];
      FSb[k] += c[1] * Fb[k];
      W0b[k] += c[0] * Web[k];
      W0qb[k] += kq * Web[k];
    }
    cb[1] -= kqb;
    cb[2] += kqb;
    half_flux_adj(l.s, c + 3, Fb, Web, lb, cb + 3);
    half_flux_adj(r.s, c + 3, Fb, Web, rb, cb + 3);
  }
  // time coefficients and the collision time
  Gas glb = gas_zero(), grb = gas_zero();
  {
    const R taub = time_coef_adj(tau, gas.dt, gas.inv_dt, cnb, ctb, Eb, e1b);
    g0b.p -= gas.mu * ip0 * ip0 * taub;
    // |dp| / sp with d|x|/dx = sign(x), 0 at x = 0
    const R s = sgn0(dp), adp = s_abs(dp), c = gas.c2 * gas.dt * taub / (sp * sp);
    glb.p += c * (s * sp - adp);
    grb.p += c * (-s * sp - adp);
  }
  // equilibrium state: stress, Euler flux and its time derivative, gradients
  {
    Grad xb = grad_zero(), yb = grad_zero(), tb = grad_zero();
    R x1b[4] = {0.0, 0.0, 0.0, 0.0};
    stress_flux_adj(g0, K, gm1, gx, gy, FSb, g0b, xb, yb);
    euler_flux_rate_adj(g0, gt, W0q, FQb, g0b, tb, W0qb);
    euler_flux_adj(g0, W0, FEb, g0b, W0b);
    cons_rate_adj(g0, hN, gt, W0qb, g0b, tb);
    prim_rate_adj(g0, gm1, gx, gy, tb, g0b, xb, yb);
    prim_grad_adj(g0, gm1, x1, gx, xb, g0b, x1b);
    prim_grad_adj(g0, gm1, Wt, gy, yb, g0b, Wtb);
    gas_state_adj(W0, gm1, g0, g0b, W0b);
    for (int k = 0; k < 4; ++k) {
      Wlnb[k] += 0.5 * x1b[k];
      Wrnb[k] += 0.5 * x1b[k];
    }
  }
  side_adj(Wl, Wln, Wt, +1, K, gm1, l, lb, Wlqb, W0b, glb, Wlb, Wlnb, Wtb);
  side_adj(Wr, Wrn, Wt, -1, K, gm1, r, rb, Wrqb, W0b, grb, Wrb, Wrnb, Wtb);
}

// any normal: the x <-> y transposition of iface_solve, transposed
FD_HD void iface_solve_adj(const GasK<R>& gas, int normal, const R Wl[4], const R Wr[4], const R Wln[4], const R Wrn[4],
                           const R Wt[4], bool want_n, const IfaceOut<R>& ob, R Wlb[4], R Wrb[4], R Wlnb[4],
                           R Wrnb[4], R Wtb[4]) {
  const bool sw = normal != 0;
  R a[4], b[4], c[4], d[4], e[4];
  swap_uv(Wl, a, sw); swap_uv(Wr, b, sw); swap_uv(Wln, c, sw); swap_uv(Wrn, d, sw); swap_uv(Wt, e, sw);
  IfaceOut<R> obs;
  swap_uv(ob.Ft, obs.Ft, sw); swap_uv(ob.Wlt, obs.Wlt, sw); swap_uv(ob.Wrt, obs.Wrt, sw);
  if (want_n) { swap_uv(ob.F, obs.F, sw); swap_uv(ob.Wl, obs.Wl, sw); swap_uv(ob.Wr, obs.Wr, sw); }
  R ab[4] = {0, 0, 0, 0}, bb[4] = {0, 0, 0, 0}, cb[4] = {0, 0, 0, 0}, db[4] = {0, 0, 0, 0}, eb[4] = {0, 0, 0, 0};
  iface_solve_x_adj(gas, a, b, c, d, e, want_n, obs, ab, bb, cb, db, eb);
  R t[4];
  swap_uv(ab, t, sw); for (int k = 0; k < 4; ++k) Wlb[k] += t[k];
  swap_uv(bb, t, sw); for (int k = 0; k < 4; ++k) Wrb[k] += t[k];
  swap_uv(cb, t, sw); for (int k = 0; k < 4; ++k) Wlnb[k] += t[k];
  swap_uv(db, t, sw); for (int k = 0; k < 4; ++k) Wrnb[k] += t[k];
  swap_uv(eb, t, sw); for (int k = 0; k < 4; ++k) Wtb[k] += t[k];
}

// ---------------------------------------------------------------------------
// nodal flux (Sec. 2.1): adjoints of F, G, F_t, G_t -> of W, W_x, W_y (added)
// ---------------------------------------------------------------------------
// the x <-> y transposition of a state and of a gradient (its own inverse)
FD_HD Gas swap_gas(const Gas& g) { return Gas{g.rho, g.ir, g.V, g.U, g.p, g.th, g.en}; }
FD_HD Grad swap_grad(const Grad& q) { return Grad{q.d, q.v, q.u, q.t}; }

// x-flux and its time derivative: Fb, Ftb -> the adjoints of the state, W, the
// gradients and W_t
FD_HD void nodal_dir_adj(R K, R gm1, R prfix, R tau, const Gas& g, const R W[4], const Grad& x, const Grad& y,
                         const Grad& t, const R Wq[4], const R Fb[4], const R Ftb[4], Gas& gb, R Wb[4], Grad& xb,
                         Grad& yb, Grad& tb, R Wqb[4], R& taub) {
  const R c = prfix * (0.5 * K + 2.0);
  // Ft = Euler rate, Ft3 += c theta rho U_t
  euler_flux_rate_adj(g, t, Wq, Ftb, gb, tb, Wqb);
  gb.th += c * t.u * Ftb[3];
  tb.u += c * g.th * Ftb[3];
  // F = Euler - tau S, S3 += c theta rho theta_x
  euler_flux_adj(g, W, Fb, gb, Wb);
  R S[4], Sb[4];
  stress_flux(g, K, gm1, x, y, S);
  S[3] += c * g.th * x.t;
  for (int k = 0; k < 4; ++k) {
    taub -= S[k] * Fb[k];
    Sb[k] = -tau * Fb[k];
  }
  stress_flux_adj(g, K, gm1, x, y, Sb, gb, xb, yb);
  gb.th += c * x.t * Sb[3];
  xb.t += c * g.th * Sb[3];
}

FD_HD void nodal_flux_adj(const GasK<R>& gas, const R W[4], const R Wx[4], const R Wy[4], const R Fb_in[4],
                          const R Gb_in[4], const R Ftb_in[4], const R Gtb_in[4], R Wb[4], R Wxb[4], R Wyb[4]) {
  const R K = gas.K, gm1 = gas.gm1, hN = 0.5 * K + 1.0;
  const Gas g = gas_state(W, gm1);
  const Grad x = prim_grad(g, gm1, Wx), y = prim_grad(g, gm1, Wy), t = prim_rate(g, gm1, x, y);
  R Wq[4];
  cons_rate(g, hN, t, Wq);
  const R ip = 1.0 / g.p, tau = gas.c1_r * gas.dt_r + gas.mu_r * ip;
  Gas gb = gas_zero(), sgb = gas_zero();
  Grad xb = grad_zero(), yb = grad_zero(), tb = grad_zero(), sxb = grad_zero(), syb = grad_zero(), stb = grad_zero();
  R Wqb[4] = {0, 0, 0, 0}, sWqb[4] = {0, 0, 0, 0}, sWb[4] = {0, 0, 0, 0}, taub = 0.0;
  nodal_dir_adj(K, gm1, gas.prfix, tau, g, W, x, y, t, Wq, Fb_in, Ftb_in, gb, Wb, xb, yb, tb, Wqb, taub);
  const R sW[4] = {W[0], W[2], W[1], W[3]}, sWq[4] = {Wq[0], Wq[2], Wq[1], Wq[3]};
  const R sG[4] = {Gb_in[0], Gb_in[2], Gb_in[1], Gb_in[3]}, sGt[4] = {Gtb_in[0], Gtb_in[2], Gtb_in[1], Gtb_in[3]};
  nodal_dir_adj(K, gm1, gas.prfix, tau, swap_gas(g), sW, swap_grad(y), swap_grad(x), swap_grad(t), sWq, sG, sGt,
                sgb, sWb, syb, sxb, stb, sWqb, taub);
  const int sw[4] = {0, 2, 1, 3};
  for (int k = 0; k < 4; ++k) {
    Wb[k] += sWb[sw[k]];
    Wqb[k] += sWqb[sw[k]];
  }
  auto addg = [](Grad& a, const Grad& b) { a.d += b.d; a.u += b.v; a.v += b.u; a.t += b.t; };
  addg(xb, sxb);
  addg(yb, syb);
  addg(tb, stb);
  gb.rho += sgb.rho;
  gb.ir += sgb.ir;
  gb.U += sgb.V;
  gb.V += sgb.U;
  gb.p += sgb.p - gas.mu_r * ip * ip * taub;   // tau = c1 dt + mu/p
  gb.th += sgb.th;
  gb.en += sgb.en;
  cons_rate_adj(g, hN, t, Wqb, gb, tb);
  prim_rate_adj(g, gm1, x, y, tb, gb, xb, yb);
  prim_grad_adj(g, gm1, Wx, x, xb, gb, Wxb);
  prim_grad_adj(g, gm1, Wy, y, yb, gb, Wyb);
  gas_state_adj(W, gm1, g, gb, Wb);
}

}  // namespace rev
}  // namespace fdk
