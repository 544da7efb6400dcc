// Templated CUDA kernels of the FD-CGKS stage (Sec. 4 of the paper): nodal
// reconstruction + flux, virtual-interface points (two line reconstructions
// shared by the primary-grid and dual-grid solves), and the fused compact
// finite-difference + S2O4 update.  Included by one translation unit per
// compute precision.
#pragma once

#include <type_traits>

#include "fdcgks_internal.cuh"

// Tuning knobs (defaults are the tuned values).  Figures: ms per step of a fixed
// time loop, all builds of this source; points and nodal are the class's time.
// FDK_NODAL_MINB_F32  minimum resident blocks per SM in the launch bounds (caps
//                  registers per thread) of the FP32 nodal kernel (the FP64
//                  kernels are FP64-pipe bound and are left uncapped): 5, 6, 8
//                  give 0.111, 0.106, 0.108 (nodal, 1024^2 vortex)
#ifndef FDK_NODAL_MINB_F32
#define FDK_NODAL_MINB_F32 6
#endif
// FDK_POINT_PAIR_MINB_F32 / _F64  the same for the stage kernel in its forms with
//                  the nodes or with characteristic reconstruction: FP32 3, 4, 5
//                  give 0.0363, 0.0342, 0.0350 (128^2 vortex) and 0.296, 0.277,
//                  0.279 (double Mach 960x240, characteristic); FP64 holds 8
//                  one-warp blocks at its 248 registers
#ifndef FDK_POINT_PAIR_MINB_F32
#define FDK_POINT_PAIR_MINB_F32 4
#endif
#ifndef FDK_POINT_PAIR_MINB_F64
#define FDK_POINT_PAIR_MINB_F64 1
#endif
// FDK_POINT_ALONE_MINB_F32  the same for the FP32 stage kernel of points alone and
//                  conservative reconstruction, which needs fewer registers and
//                  spills 36 bytes at 96: 4, 5, 6 give 0.912, 0.878, 0.886
//                  (1024^2 vortex) and 0.517, 0.509, 0.516 (tube 1000x500)
#ifndef FDK_POINT_ALONE_MINB_F32
#define FDK_POINT_ALONE_MINB_F32 5
#endif
// FDK_STAGE_THREADS_F64  block size of the FP64 stage kernel: 32 and 128 give 0.177
//                  and 0.190 (33^2), 0.458 and 0.454 (128^2), 3.90 and 3.94 (512^2)
#ifndef FDK_STAGE_THREADS_F64
#define FDK_STAGE_THREADS_F64 32
#endif
// FDK_PAIR_PRELOAD_F32  1: a thread of the FP32 stage kernel loads its line's 32
//                  values (4 entries x W and the gradient along the line) into
//                  registers before the first reconstruction, so the loads are
//                  not issued between the reconstructions: 0 and 1 give points
//                  0.570 and 0.480 (1024^2 vortex).  The reconstruction is inlined:
//                  in differences and without indicators on smooth data it is
//                  short enough
#ifndef FDK_PAIR_PRELOAD_F32
#define FDK_PAIR_PRELOAD_F32 1
#endif

namespace fdk {

template <class R> struct PointTune;
template <> struct PointTune<double> {
  static constexpr int nodal_minb = 1;
  static constexpr int pair_minb = FDK_POINT_PAIR_MINB_F64, alone_minb = pair_minb;
};
template <> struct PointTune<float> {
  static constexpr int nodal_minb = FDK_NODAL_MINB_F32;
  static constexpr int pair_minb = FDK_POINT_PAIR_MINB_F32, alone_minb = FDK_POINT_ALONE_MINB_F32;
};

// ---------------------------------------------------------------------------
// nodal reconstruction and flux (Sec. 4 item 2; Sec. 2.1 nodal fluxes)
// one thread per node, nodes i in [-1, n_x], j in [-1, n_y] of grid blockIdx.z
// ---------------------------------------------------------------------------
// One node: GENO node derivatives along x and y, then the nodal flux.
// ld(e, f): field f (0-3 W, 4-7 x-gradient, 8-11 y-gradient) of node e (0 the
// node, 1/2 its x neighbours -/+, 3/4 its y neighbours -/+); st(k, v): output
// k (F[4], G[4], F_t[4], G_t[4]); want_n = false (second S2O4 stage): F_t and
// G_t only, F and G are neither computed nor stored.
// FP32: bound by the latency of its 44 loads (DRAM 16 % busy), so all of them
// are issued before the first component's branches: 1024^2 mixed 0.160 -> 0.115
// ms per step (one component ahead 0.123), 512^2 0.0458 -> 0.0392.  FP64 is
// bound by its pipe and keeps the registers.
template <class R, class LD, class ST>
FD_HD void nodal_compute(const GenoK<R>& geno, const GasK<R>& gas, const R h[2], const R ih[2], LD ld, ST st,
                         bool want_n = true) {
  constexpr int AHEAD = IsF32<R>::v ? 4 : 1;   // components loaded at once
  R W[4], Wx[4], Wy[4], qx[AHEAD][3], gx[AHEAD][3], qy[AHEAD][3], gy[AHEAD][3];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    if (c % AHEAD == 0) {
#pragma unroll
      for (int k = 0; k < AHEAD; ++k)
#pragma unroll
        for (int e = 0; e < 3; ++e) {   // the lower neighbour, the node, the upper one
          const int ex = e == 1 ? 0 : e == 0 ? 1 : 2, ey = e == 1 ? 0 : e == 0 ? 3 : 4;
          qx[k][e] = ld(ex, c + k);
          gx[k][e] = ld(ex, 4 + c + k);
          qy[k][e] = e == 1 ? qx[k][1] : ld(ey, c + k);
          gy[k][e] = ld(ey, 8 + c + k);
        }
    }
    const int k = c % AHEAD;
    W[c] = qx[k][1];
    Wx[c] = recon_node(geno, qx[k], gx[k], h[0], ih[0]);
    Wy[c] = recon_node(geno, qy[k], gy[k], h[1], ih[1]);
  }
  R F[4], G[4], Ft[4], Gt[4];
  nodal_flux(gas, W, Wx, Wy, F, G, Ft, Gt, want_n);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    if (want_n) {
      st(c, F[c]);
      st(4 + c, G[c]);
    }
    st(8 + c, Ft[c]);
    st(12 + c, Gt[c]);
  }
}

// offset of node e of the nodal stencil (see nodal_compute) from the node
FD_HD long nodal_offset(const Layout& L, int e) {
  return e == 0 ? 0 : e == 1 ? -1 : e == 2 ? 1 : e == 3 ? -(long)L.pitch : (long)L.pitch;
}

template <class R>
__device__ __forceinline__ void nodal_body(const KArgs<R>& a, int g, int i, int j) {
  const Layout& L = a.L;
  const int nxg = g == 0 ? L.nx : L.nxd, nyg = g == 0 ? L.ny : L.nyd;
  if (i < -1 || j < -1 || i > nxg || j > nyg) return;
  const R* S = a.Sr + (long)g * NFLD * L.plane;
  const long c0 = cell(L, i, j);
  R* NF = a.NF + (long)g * NNF * L.plane + c0;
  nodal_compute<R>(
      a.geno, a.gas, a.h, a.ih, [&](int e, int f) -> R { return S[(long)f * L.plane + c0 + nodal_offset(L, e)]; },
      [&](int k, R v) { NF[(long)k * L.plane] = v; }, a.want_n != 0);
}

template <class R>
__global__ void __launch_bounds__(128, PointTune<R>::nodal_minb) nodal_kernel(KArgs<R> a) {
  if constexpr (IsF32<R>::v) step_begin();
  nodal_body(a, blockIdx.z, blockIdx.x * blockDim.x + threadIdx.x - 1, blockIdx.y * blockDim.y + threadIdx.y - 1);
}

// Positivity safeguard of the interface states (the paper describes none): a
// reconstructed state with non-positive or non-finite density or pressure
// (physical_state, fdcgks_math.cuh) is replaced by the state of the node on
// its side (line entries 1 and 2) with zero normal slope, and the interface's
// chi by 0, so its compact flux takes the low-order form.  Never triggered by
// smooth data.
// the safeguard applied to the left/right states of line l
template <class R, class LD>
FD_HD void positivity_fix(LD ld, int l, R vl[4], R dl[4], R vr[4], R dr[4], R& chi) {
  if (!physical_state(vl)) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      vl[c] = ld(l, 1, c);
      dl[c] = R(0);
    }
    chi = R(0);
  }
  if (!physical_state(vr)) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      vr[c] = ld(l, 2, c);
      dr[c] = R(0);
    }
    chi = R(0);
  }
}

// Reconstruct one 4-point line at its virtual interface (between entries 1
// and 2), with the safeguard above.  ld(l, e, f) = field f (0-3 W, 4-7 the
// averaged gradient along the line) of entry e (0-3) of line l.
// D1: component 2 is 0 throughout (the one-dimensional gas).
template <bool D1 = false, class R, class LD>
FD_HD void recon_line_ld(const GenoK<R>& geno, LD ld, int l, R h, R ih, R vl[4], R dl[4], R vr[4], R dr[4],
                         R& chi) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    if (D1 && c == 2) {
      vl[c] = dl[c] = vr[c] = dr[c] = R(0);
      continue;
    }
    R Q[4] = {ld(l, 0, c), ld(l, 1, c), ld(l, 2, c), ld(l, 3, c)};
    R Qx[4] = {ld(l, 0, 4 + c), ld(l, 1, 4 + c), ld(l, 2, 4 + c), ld(l, 3, 4 + c)};
    R cl, cr;
    recon_interface(geno, Q, Qx, h, ih, vl[c], dl[c], cl, vr[c], dr[c], cr);
    if (c == 0) chi = s_min(cl, cr);   // chi_{j+1/2} = min(chi^{l,rho}, chi^{r,rho})
  }
  positivity_fix(ld, l, vl, dl, vr, dr, chi);
}

// The same on characteristic components (Sec. 3.1, "characteristic component
// of W"; recon_vars = 1): the eigenvectors of the Euler flux Jacobian along
// the line's normal, frozen at the mean of entries 1 and 2, in the order
// (rho, m_n, m_t, E); rows of L / columns of R: U - c, entropy, shear, U + c.
// Values and gradients are projected with L, each component reconstructed,
// values and derivatives mapped back with R; chi of the flux is the smaller
// of the two acoustic fields' (Sec. 3.2).  A non-physical mean state falls
// back to conservative components.
template <bool D1 = false, class R, class LD>
FD_HD void recon_line_char(const GenoK<R>& geno, R gm1, int normal, LD ld, int l, R h, R ih, R vl[4], R dl[4],
                           R vr[4], R dr[4], R& chi) {
  // component j of (rho, m_n, m_t, E) of an entry's values (f0 = 0) or
  // gradients (f0 = 4): a select between the two momenta, not an index, so that
  // values held in registers stay there
  const bool sw = normal != 0;
  auto comp = [&](int e, int f0, int j) -> R {
    return j == 1 ? (sw ? ld(l, e, f0 + 2) : ld(l, e, f0 + 1))
                  : j == 2 ? (sw ? ld(l, e, f0 + 1) : ld(l, e, f0 + 2)) : ld(l, e, f0 + j);
  };
  const R r = R(0.5) * (ld(l, 1, 0) + ld(l, 2, 0));
  const R mn = R(0.5) * (comp(1, 0, 1) + comp(2, 0, 1)), mt = R(0.5) * (comp(1, 0, 2) + comp(2, 0, 2));
  const R E = R(0.5) * (ld(l, 1, 3) + ld(l, 2, 3));
  const R ir = s_div(R(1), r), u = mn * ir, v = mt * ir;
  const R q2 = u * u + v * v;
  const R p = gm1 * (E - R(0.5) * r * q2);
  if (!(r > R(0)) || !(p > R(0))) {
    recon_line_ld<D1>(geno, ld, l, h, ih, vl, dl, vr, dr, chi);
    return;
  }
  const R c = s_sqrt((gm1 + R(1)) * p * ir), ic = s_div(R(1), c), H = (E + p) * ir;
  const R b1 = gm1 * ic * ic, b2 = R(0.5) * b1 * q2;
  const R Lm[4][4] = {{R(0.5) * (b2 + u * ic), -R(0.5) * (b1 * u + ic), -R(0.5) * b1 * v, R(0.5) * b1},
                      {R(1) - b2, b1 * u, b1 * v, -b1},
                      {-v, R(0), R(1), R(0)},
                      {R(0.5) * (b2 - u * ic), -R(0.5) * (b1 * u - ic), -R(0.5) * b1 * v, R(0.5) * b1}};
  const R Rm[4][4] = {{R(1), R(1), R(0), R(1)},
                      {u - c, u, R(0), u + c},
                      {v, v, R(1), v},
                      {H - u * c, R(0.5) * q2, v, H + u * c}};
  R cvl[4], cdl[4], cvr[4], cdr[4], cl[4], cr[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (D1 && k == 2) {   // shear
      cvl[k] = cdl[k] = cvr[k] = cdr[k] = R(0);
      continue;
    }
    R Q[4], Qx[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      R a = R(0), b = R(0);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (D1 && j == 2) continue;
        a += Lm[k][j] * comp(m, 0, j);
        b += Lm[k][j] * comp(m, 4, j);
      }
      Q[m] = a;
      Qx[m] = b;
    }
    recon_interface(geno, Q, Qx, h, ih, cvl[k], cdl[k], cl[k], cvr[k], cdr[k], cr[k]);
  }
  R tvl[4], tdl[4], tvr[4], tdr[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    tvl[j] = tdl[j] = tvr[j] = tdr[j] = R(0);
    if (D1 && j == 2) continue;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (D1 && k == 2) continue;
      tvl[j] += Rm[j][k] * cvl[k];
      tvr[j] += Rm[j][k] * cvr[k];
      tdl[j] += Rm[j][k] * cdl[k];
      tdr[j] += Rm[j][k] * cdr[k];
    }
  }
  swap_uv(tvl, vl, sw);
  swap_uv(tdl, dl, sw);
  swap_uv(tvr, vr, sw);
  swap_uv(tdr, dr, sw);
  chi = s_min(s_min(cl[0], cr[0]), s_min(cl[3], cr[3]));
  positivity_fix(ld, l, vl, dl, vr, dr, chi);
}

// Where the lines of point (i, j) lie in the padded state: entry e of line l
// is at base[l] + e * stride[l] of grid l (primary 0, dual 1), its gradient
// along the line in fields gfield[l]..gfield[l] + 3.
struct PointLines {
  long base[2], stride[2];
  int gfield[2];
};
FD_HD PointLines point_lines(const Layout& L, int type, int i, int j) {
  PointLines p;
  if (type == 0) {
    // primary nodes (i-1..i+2, j) along x; dual nodes (i+1, j-1..j+2) along y
    p.base[0] = cell(L, i - 1, j); p.stride[0] = 1; p.gfield[0] = 4;
    p.base[1] = cell(L, i + 1, j - 1); p.stride[1] = L.pitch; p.gfield[1] = 8;
  } else {
    // primary nodes (i, j-1..j+2) along y; dual nodes (i-1..i+2, j+1) along x
    p.base[0] = cell(L, i, j - 1); p.stride[0] = L.pitch; p.gfield[0] = 8;
    p.base[1] = cell(L, i - 1, j + 1); p.stride[1] = 1; p.gfield[1] = 4;
  }
  return p;
}

// ---------------------------------------------------------------------------
// virtual-interface points (Sec. 4 item 1; App. A3).
// TYPE 0 = point A (i+1/2, j): primary x-interface, dual y-interface of dual column i+1
// TYPE 1 = point B (i, j+1/2): primary y-interface, dual x-interface of dual row j+1
// ---------------------------------------------------------------------------
// Two threads per point (lanes 2k and 2k + 1 of a warp): lane parity l
// reconstructs line l and runs solve l (l = 0 the primary-grid line and solve
// with normal `type`, spacing h[type]; l = 1 the dual-grid ones with the other
// normal).  What couples the two solves of a point travels between the
// partner lanes by warp shuffles: the tangential derivative of each solve (the
// mean of the other line's l/r derivatives) and the other solve's quarter in
// W~ (Eq. eq:W-model-2d).  One thread with both solves needs a call frame in
// local memory (1024^2 vortex, point phase per step: 1.019 ms mixed and
// 32.06 ms FP64 against 0.903 and 31.41 ms for the pair when it was brought
// in).  ld(l, e, f) as for recon_line_ld; st(k, v): output k of this lane's
// solve (PO_*; F and W~ values only when wn).  mask: the lanes of the warp
// that take part (pairs are valid together).
// ---------------------------------------------------------------------------
template <class R, bool CHAR, class LD, class ST>
__device__ __forceinline__ void point_compute_pair(const GenoK<R>& geno, const GasK<R>& gas, const R h[2],
                                                   const R ih[2], bool wn, int type, int l, unsigned mask, LD ld,
                                                   ST st) {
  const int n = l == 0 ? type : 1 - type;   // normal of this lane's solve
  R lv[4], ldv[4], rv[4], rdv[4], chi;
  if constexpr (CHAR)
    recon_line_char(geno, gas.gm1, n, ld, l, h[n], ih[n], lv, ldv, rv, rdv, chi);
  else
    recon_line_ld(geno, ld, l, h[n], ih[n], lv, ldv, rv, rdv, chi);
  R t[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) t[c] = R(0.5) * __shfl_xor_sync(mask, ldv[c] + rdv[c], 1);
  IfaceOut<R> o;
  iface_solve(gas, n, lv, rv, ldv, rdv, t, wn, o);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const R mt = R(0.25) * __shfl_xor_sync(mask, o.Wlt[c] + o.Wrt[c], 1);
    st(PO_FT + c, o.Ft[c]);
    st(PO_WLT + c, R(0.5) * o.Wlt[c] + mt);
    st(PO_WRT + c, R(0.5) * o.Wrt[c] + mt);
    if (wn) {
      const R m = R(0.25) * __shfl_xor_sync(mask, o.Wl[c] + o.Wr[c], 1);
      st(PO_F + c, o.F[c]);
      st(PO_WL + c, R(0.5) * o.Wl[c] + m);
      st(PO_WR + c, R(0.5) * o.Wr[c] + m);
    }
  }
  st(PO_CHI, chi);
}

// one thread of a point pair: point (i, j) of the type, line / solve l
template <class R, bool CHAR>
__device__ __forceinline__ void point_pair_body(const KArgs<R>& a, int type, int i, int j, int l) {
  const Layout& L = a.L;
  const int imax = type == 0 ? L.nx : L.nxd;
  const int jmax = type == 0 ? L.nyd : L.ny;
  const bool valid = !(i < -2 || j < -2 || i > imax || j > jmax);
  const unsigned mask = __ballot_sync(0xffffffffu, valid);
  if (!valid) return;
  const PointLines pl = point_lines(L, type, i, j);
  const R* S = a.Sr;
  R* P = (type == 0 ? a.PA : a.PB) + pcell(L, i, j) + (long)l * NPS * L.pplane;
  const long pp = L.pplane;
  auto st = [&](int k, R v) { P[(long)k * pp] = v; };
  auto gl = [&](int ll, int e, int f) -> R {
    const int field = f < 4 ? f : pl.gfield[ll] + (f - 4);
    return S[((long)ll * NFLD + field) * L.plane + pl.base[ll] + e * pl.stride[ll]];
  };
#if FDK_PAIR_PRELOAD_F32
  if constexpr (IsF32<R>::v) {
  R xl[32];
#pragma unroll
  for (int e = 0; e < 4; ++e)
#pragma unroll
    for (int f = 0; f < 8; ++f) xl[e * 8 + f] = gl(l, e, f);
  point_compute_pair<R, CHAR>(a.geno, a.gas, a.h, a.ih, a.want_n != 0, type, l, mask,
                              [&](int, int e, int f) -> R { return xl[e * 8 + f]; }, st);
  } else {
    point_compute_pair<R, CHAR>(a.geno, a.gas, a.h, a.ih, a.want_n != 0, type, l, mask, gl, st);
  }
#else
  point_compute_pair<R, CHAR>(a.geno, a.gas, a.h, a.ih, a.want_n != 0, type, l, mask, gl, st);
#endif
}

// Both point types and, if `nodal` is set, the nodal work of a stage in one
// launch (the three are independent).  FP64: items are dealt out linearly
// (A pairs, B pairs, nodes) to blocks of one warp, since the FP64 pipe needs
// one warp per scheduler and nothing else: no tile is partly empty, the last
// wave is one warp deep, and the short nodal items fill it.  Mixed: tiles of
// 16 x 4 points (32 x 4 nodes) in blocks of 128, whose rows share lines in L1.
struct StageGrid {
  int nA, nB, nN0, nN1;   // items (FP64) or blocks (mixed) of each kind
  int wA, wB, w0, w1;     // items or blocks per row
};

template <class R> struct StageTune;
template <> struct StageTune<double> { static constexpr int threads = FDK_STAGE_THREADS_F64; };
template <> struct StageTune<float> { static constexpr int threads = 128; };

template <class R, bool CHAR, bool NODAL>
__global__ void __launch_bounds__(StageTune<R>::threads,
                                  (CHAR || NODAL ? PointTune<R>::pair_minb : PointTune<R>::alone_minb) * 128 /
                                      StageTune<R>::threads)
    stage_kernel(KArgs<R> a, StageGrid G) {
  if constexpr (IsF32<R>::v) step_begin();
  const int T = StageTune<R>::threads;
  if constexpr (IsF32<R>::v) {
    int b = blockIdx.x;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    if (b < G.nA + G.nB) {
      const int type = b < G.nA ? 0 : 1;
      if (type) b -= G.nA;
      const int w = type ? G.wB : G.wA, by = b / w, bx = b - by * w;
      point_pair_body<R, CHAR>(a, type, bx * 16 + (tx >> 1) - 2, by * 4 + ty - 2, tx & 1);
    } else if constexpr (NODAL) {
      b -= G.nA + G.nB;
      const int g = b < G.nN0 ? 0 : 1;
      if (g) b -= G.nN0;
      const int w = g ? G.w1 : G.w0, by = b / w, bx = b - by * w;
      nodal_body(a, g, bx * 32 + tx - 1, by * 4 + ty - 1);
    }
  } else {
    // whole warps take points or nodes: the point items are padded to a warp
    const int q = blockIdx.x * T + threadIdx.x;
    const int np = 2 * (G.nA + G.nB), npp = (np + 31) / 32 * 32;
    if (q < npp) {
      int p = q >> 1;
      const int type = p < G.nA ? 0 : 1;
      if (type) p -= G.nA;
      const int w = type ? G.wB : G.wA, j = p / w;
      point_pair_body<R, CHAR>(a, type, q < np ? p - j * w - 2 : -3, j - 2, q & 1);
    } else if constexpr (NODAL) {
      int n = q - npp;
      if (n >= G.nN0 + G.nN1) return;
      const int g = n < G.nN0 ? 0 : 1;
      if (g) n -= G.nN0;
      const int w = g ? G.w1 : G.w0, j = n / w;
      nodal_body(a, g, n - j * w - 1, j - 1);
    }
  }
}

// ---------------------------------------------------------------------------
// compact FD + S2O4 update (Eqs. eq-conservation-law-2d, fd-conservative-flux*,
// define-averaged-gradient, eq-nodal-update, eq-interface-update).
// One thread per interior node of grid blockIdx.z.
// ---------------------------------------------------------------------------

// one node's stage operator: L, dL/dt (per component), the averaged gradients
// re-evaluated from the interface solution (node's own side) and their time
// derivatives
struct NodeOp {
  double L[4], Lt[4], gbx[4], gby[4], gtx[4], gty[4];
};

__device__ __forceinline__ void node_operator(const KArgs<double>& a, int g, int i, int j, bool want_n, NodeOp& o) {
  using R = double;
  const Layout& L = a.L;
  const long pp = L.pplane;
  // x-interface k+1/2 of this grid's row and y-interface k+1/2 of its column
  const R* PX = g == 0 ? a.PA : a.PB + NPS * pp;   // primary: A points solve 0; dual: B points solve 1
  const R* PY = g == 0 ? a.PB : a.PA + NPS * pp;   // primary: B points solve 0; dual: A points solve 1
  auto xi = [&](int k) { return g == 0 ? pcell(L, k, j) : pcell(L, k, j - 1); };
  auto yi = [&](int k) { return g == 0 ? pcell(L, i, k) : pcell(L, i - 1, k); };
  const R* NF = a.NF + (long)g * NNF * L.plane;
  const long cN = cell(L, i, j);
  const int fv = a.flux_variant;
  const R ihx = a.ih[0], ihy = a.ih[1];
  const long xm2 = xi(i - 2), xm1 = xi(i - 1), x0 = xi(i), xp1 = xi(i + 1);
  const long ym2 = yi(j - 2), ym1 = yi(j - 1), y0 = yi(j), yp1 = yi(j + 1);
  const R chixm = PX[PO_CHI * pp + xm1], chix0 = PX[PO_CHI * pp + x0];
  const R chiym = PY[PO_CHI * pp + ym1], chiy0 = PY[PO_CHI * pp + y0];
  // bound by the FP64 pipe: the short form of the flux difference where all
  // four interfaces are smooth (1024^2 vortex: 2.77 -> 1.39 ms per step)
  {
    auto components = [&](auto sm) {
      constexpr bool SMOOTH = decltype(sm)::value;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        auto div = [&](const R* f, const R* fn, const R* q, const R* qn) {
          return -compact_flux_diff<SMOOTH>(fv, chixm, chix0, f[xm2], f[xm1], f[x0], f[xp1], fn[cN - 1], fn[cN],
                                            fn[cN + 1]) * ihx -
                 compact_flux_diff<SMOOTH>(fv, chiym, chiy0, q[ym2], q[ym1], q[y0], q[yp1], qn[cN - L.pitch], qn[cN],
                                           qn[cN + L.pitch]) * ihy;
        };
        o.Lt[c] = div(PX + (PO_FT + c) * pp, NF + (8 + c) * L.plane, PY + (PO_FT + c) * pp, NF + (12 + c) * L.plane);
        o.L[c] = R(0);
        o.gbx[c] = R(0);
        o.gby[c] = R(0);
        if (want_n) {
          o.L[c] = div(PX + (PO_F + c) * pp, NF + c * L.plane, PY + (PO_F + c) * pp, NF + (4 + c) * L.plane);
          o.gbx[c] = (PX[(PO_WL + c) * pp + x0] - PX[(PO_WR + c) * pp + xm1]) * ihx;
          o.gby[c] = (PY[(PO_WL + c) * pp + y0] - PY[(PO_WR + c) * pp + ym1]) * ihy;
        }
        o.gtx[c] = (PX[(PO_WLT + c) * pp + x0] - PX[(PO_WRT + c) * pp + xm1]) * ihx;
        o.gty[c] = (PY[(PO_WLT + c) * pp + y0] - PY[(PO_WRT + c) * pp + ym1]) * ihy;
      }
    };
    if (chixm == R(1) && chix0 == R(1) && chiym == R(1) && chiy0 == R(1)) components(std::true_type());
    else components(std::false_type());
  }
}

// float-float (double-word) accumulation for the mixed path: Knuth's TwoSum
// gives s + e = a + b exactly; Dekker's FastTwoSum renormalises hi + lo
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  float v = s - a;
  e = (a - (s - v)) + (b - v);
}
__device__ __forceinline__ void ff_add(float& hi, float& lo, float b) {
  float s, e;
  two_sum(hi, b, s, e);
  e += lo;
  hi = s + e;
  lo = e - (hi - s);
}

__device__ __forceinline__ void update_body(const KArgs<double>& a, int mode, int g, int i, int j) {
  const Layout& L = a.L;
  const int nxg = g == 0 ? L.nx : L.nxd, nyg = g == 0 ? L.ny : L.nyd;
  if (i < 0 || j < 0 || i >= nxg || j >= nyg) return;
  NodeOp o;
  node_operator(a, g, i, j, mode != UPD_STAGE2, o);
  const long c0 = cell(L, i, j);
  if (mode == UPD_OPERATOR) {
    const long NN = (long)nxg * nyg, oi = (long)j * nxg + i;
    double* const* op = a.op + 4 * g;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      op[0][c * NN + oi] = (double)o.L[c];
      op[1][c * NN + oi] = (double)o.Lt[c];
      op[2][c * NN + oi] = (double)o.gbx[c];
      op[2][(4 + c) * NN + oi] = (double)o.gby[c];
      op[3][c * NN + oi] = (double)o.gtx[c];
      op[3][(4 + c) * NN + oi] = (double)o.gty[c];
    }
    return;
  }
  // dual nodes on a no-slip wall: velocity set to zero (internal energy kept),
  // and, as U = V = 0 along the whole wall, the momentum gradients along it too
  const bool xwall = g == 1 && ((a.bc[0] == 3 && i == 0) || (a.bc[1] == 3 && i == nxg - 1));
  const bool ywall = g == 1 && ((a.bc[2] == 3 && j == 0) || (a.bc[3] == 3 && j == nyg - 1));
  const long P = L.plane;

  {
    const double dt = a.dt;
    const double* Sng = a.Sn + (long)g * NFLD * P;
    double* Og = a.Sout + (long)g * NFLD * P;
    double* Ag = a.Wacc + (long)g * 4 * P;
    double* Bg = a.gB + (long)g * 8 * P;
    double Wnew[4], Gnew[8];
    // every input is loaded before the first store, so that the loads are
    // issued together (the stores could alias them for the compiler)
    if (mode == UPD_STAGE1) {
      double Wn[4], Gb[8];
#pragma unroll
      for (int c = 0; c < 4; ++c) Wn[c] = Sng[(long)c * P + c0];
#pragma unroll
      for (int f = 0; f < 8; ++f)
        Gb[f] = a.grad_base ? Sng[(long)(4 + f) * P + c0] : (double)(f < 4 ? o.gbx[f] : o.gby[f - 4]);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const double dL = (double)o.L[c], dLt = (double)o.Lt[c];
        Wnew[c] = Wn[c] + a.dtk[0] * dL + a.dtk[1] * dLt;
        Ag[(long)c * P + c0] = Wn[c] + dt * dL + a.dtk[2] * dLt;
      }
#pragma unroll
      for (int f = 0; f < 8; ++f) {
        Bg[(long)f * P + c0] = Gb[f];
        Gnew[f] = Gb[f] + a.dtk[0] * (double)(f < 4 ? o.gtx[f] : o.gty[f - 4]);
      }
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) Wnew[c] = Ag[(long)c * P + c0];
#pragma unroll
      for (int f = 0; f < 8; ++f) Gnew[f] = Bg[(long)f * P + c0];
#pragma unroll
      for (int c = 0; c < 4; ++c) Wnew[c] = Wnew[c] + a.dtk[3] * (double)o.Lt[c];
#pragma unroll
      for (int f = 0; f < 8; ++f) Gnew[f] = Gnew[f] + dt * (double)(f < 4 ? o.gtx[f] : o.gty[f - 4]);
    }
    if (xwall || ywall) {
      double ke = 0.5 * (Wnew[1] * Wnew[1] + Wnew[2] * Wnew[2]) / Wnew[0];
      Wnew[1] = 0.0;
      Wnew[2] = 0.0;
      Wnew[3] -= ke;
    }
    if (xwall) { Gnew[5] = 0.0; Gnew[6] = 0.0; }   // y-gradients of rho U, rho V
    if (ywall) { Gnew[1] = 0.0; Gnew[2] = 0.0; }   // x-gradients of rho U, rho V
#pragma unroll
    for (int c = 0; c < 4; ++c) Og[(long)c * P + c0] = Wnew[c];
#pragma unroll
    for (int f = 0; f < 8; ++f) Og[(long)(4 + f) * P + c0] = Gnew[f];
    // positivity of density and pressure (no trap: a flag the host reads), p > 0
    // as 2 E rho > m^2, without a division unless it fails (products out of range)
    const double m2 = Wnew[1] * Wnew[1] + Wnew[2] * Wnew[2];
    if (!(Wnew[0] > 0.0) || (!(2.0 * Wnew[3] * Wnew[0] > m2) && !(Wnew[3] - 0.5 * m2 / Wnew[0] > 0.0)))
      atomicOr(a.flag, 1);
  }
}

static __global__ void __launch_bounds__(128) update_kernel(KArgs<double> a, int mode) {
  update_body(a, mode, blockIdx.z, blockIdx.x * blockDim.x + threadIdx.x, blockIdx.y * blockDim.y + threadIdx.y);
}

// ---------------------------------------------------------------------------
// The mixed update: one thread per component and column of ROWS nodes, the
// component the index of the warp in its block of four, which covers 32 ROWS
// nodes.  It is bound by the latency and number of its loads (148 a node, DRAM
// 46 % busy), not by arithmetic: a thread of one component needs few enough
// registers to have a column's loads in flight together, and its rows share
// the interfaces between them (20 loads a component and node of 4 rows where
// one node takes 28).  ms per step of the update against one thread per node
// with all four components:
//             33^2    128^2   512^2   1024^2
//   by node   0.0195  0.0215  0.104   0.345
//   1 row     0.0147  0.0166  0.126   0.447   (40 registers: 0.106, 0.363)
//   2 rows    0.0188  0.0204  0.0988  0.325   (40 registers; 64: 0.0996, 0.334)
//   4 rows    0.0198  0.0216  0.0964  0.312   (64 registers; 48: 0.1135, 0.369)
//   8 rows    0.0376  0.0358  0.147   0.438   (80 registers)
// ---------------------------------------------------------------------------
// Rows a thread: 1 where the whole grid is then one wave of blocks (12 an SM,
// 152 SMs, two grids in blocks of 32 nodes), 4 where it fills the GPU anyway
// (the table above), 2 between (200^2 nodes, step: 1, 2, 4 rows 0.0742, 0.0692,
// 0.0700 ms; 256^2 0.0966, 0.0946, 0.0944).
template <int ROWS> struct UpdRows { static constexpr int minb = 12; };
template <> struct UpdRows<4> { static constexpr int minb = 8; };
const long UPD_SMALL_NODES = 29000, UPD_LARGE_NODES = 100000;

// what one component of one node of the mixed update hands to its second half
struct CompOut {
  float Wh, Wl, gxh, gxl, gyh, gyl;
};

// component c of rows j..j + ROWS - 1 of column i, `rows` >= 1 of which exist
template <int ROWS>
__device__ __forceinline__ void update_comp(const KArgs<float>& a, int mode, int g, int c, int i, int j, int rows,
                                            CompOut o[ROWS]) {
  const Layout& L = a.L;
  const long pp = L.pplane, P = L.plane;
  const bool want_n = mode != UPD_STAGE2;
  const int fv = a.flux_variant;
  const float ihx = a.ih[0], ihy = a.ih[1];
  const long xc = g == 0 ? pcell(L, i, j) : pcell(L, i, j - 1), yc = g == 0 ? pcell(L, i, j) : pcell(L, i - 1, j);
  const float* PX = (g == 0 ? a.PA : a.PB + NPS * pp) + xc;
  const float* PY = (g == 0 ? a.PB : a.PA + NPS * pp) + yc;
  const float* PXc = PX + (long)c * pp;
  const float* PYc = PY + (long)c * pp;
  const long c0 = cell(L, i, j);
  const float* NF = a.NF + ((long)g * NNF + c) * P + c0;
  const int sp = L.ppitch, sn = L.pitch;
  auto rr = [&](int r) { return ROWS > 1 ? min(r, rows - 1) : r; };   // rows past the grid: its last one
  float chx[2 * ROWS], chy[ROWS + 1];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    chx[2 * r] = PX[PO_CHI * pp + rr(r) * sp - 1];
    chx[2 * r + 1] = PX[PO_CHI * pp + rr(r) * sp];
  }
#pragma unroll
  for (int r = 0; r <= ROWS; ++r) chy[r] = PY[PO_CHI * pp + (ROWS > 1 ? min(r, rows) - 1 : r - 1) * sp];
  // compact_flux with its roundings spelled out, as every sum of products below:
  // the kernels that inline this for other ROWS give the same bits
  auto flux = [&](float chi, float Fm, float F0, float Fp, float N0, float N1) {
    const float hi = __fmul_rn(__fmaf_rn(-9.0f, N0 + N1, __fmaf_rn(46.0f, F0, Fm) + Fp), 1.0f / 30.0f);
    const float lo = fv == 62 ? F0 : __fmul_rn(__fmaf_rn(8.0f, F0, -N0) - N1, 1.0f / 6.0f);
    return __fmaf_rn(chi, hi, __fmul_rn(1.0f - chi, lo));
  };
  float Ll[2][ROWS];
#pragma unroll
  for (int d = 0; d < 2; ++d) {   // F_t, then F
    if (d == 1 && !want_n) {
#pragma unroll
      for (int r = 0; r < ROWS; ++r) Ll[1][r] = 0.0f;
      continue;
    }
    const int po = d == 0 ? PO_FT : PO_F, no = d == 0 ? 8 : 0;
    const float* f = PXc + po * pp;
    const float* q = PYc + po * pp;
    const float* n = NF + no * P;
    const float* m = NF + (no + 4) * P;
    float y[ROWS + 3], ny[ROWS + 2];
#pragma unroll
    for (int r = 0; r < ROWS + 3; ++r) y[r] = q[(ROWS > 1 ? min(r, rows + 2) - 2 : r - 2) * sp];
#pragma unroll
    for (int r = 0; r < ROWS + 2; ++r) ny[r] = m[(ROWS > 1 ? min(r, rows + 1) - 1 : r - 1) * sn];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const float* fr = f + rr(r) * sp;
      const float* nr = n + rr(r) * sn;
      const float x0 = fr[-2], x1 = fr[-1], x2 = fr[0], x3 = fr[1], n0 = nr[-1], n1 = nr[0], n2 = nr[1];
      const float fp = flux(chx[2 * r + 1], x1, x2, x3, n1, n2);
      const float fm = flux(chx[2 * r], x0, x1, x2, n0, n1);
      const float gp = flux(chy[r + 1], y[r + 1], y[r + 2], y[r + 3], ny[r + 1], ny[r + 2]);
      const float gm = flux(chy[r], y[r], y[r + 1], y[r + 2], ny[r], ny[r + 1]);
      Ll[d][r] = __fmaf_rn(gm - gp, ihy, __fmul_rn(fm - fp, ihx));
    }
  }
  float gbx[ROWS], gby[ROWS], gtx[ROWS], gty[ROWS];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const float* x = PXc + rr(r) * sp;
    const float* y = PYc + rr(r) * sp;
    gtx[r] = __fmul_rn(x[PO_WLT * pp] - x[PO_WRT * pp - 1], ihx);
    gty[r] = __fmul_rn(y[PO_WLT * pp] - y[PO_WRT * pp - sp], ihy);
    gbx[r] = gby[r] = 0.0f;
    if (want_n && (!a.grad_base || mode == UPD_OPERATOR)) {
      gbx[r] = __fmul_rn(x[PO_WL * pp] - x[PO_WR * pp - 1], ihx);
      gby[r] = __fmul_rn(y[PO_WL * pp] - y[PO_WR * pp - sp], ihy);
    }
  }
  if (mode == UPD_OPERATOR) {
    const int nxg = g == 0 ? L.nx : L.nxd, nyg = g == 0 ? L.ny : L.nyd;
    const long NN = (long)nxg * nyg, oi = (long)j * nxg + i;
    double* const* op = a.op + 4 * g;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      if (r >= rows) break;
      const long k = oi + (long)r * nxg;
      op[0][c * NN + k] = (double)Ll[1][r];
      op[1][c * NN + k] = (double)Ll[0][r];
      op[2][c * NN + k] = (double)gbx[r];
      op[2][(4 + c) * NN + k] = (double)gby[r];
      op[3][c * NN + k] = (double)gtx[r];
      op[3][(4 + c) * NN + k] = (double)gty[r];
    }
    return;
  }
  // state and accumulators are float-float pairs; increments are formed in
  // FP32 and added exactly (two_sum) to the pairs
  const float dtr = a.gas.dt_r;
  const long sc = ((long)g * NFLD + c) * P + c0, ac = ((long)g * 4 + c) * P + c0, bc = ((long)g * 8 + c) * P + c0;
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    if (r >= rows) break;
    CompOut& v = o[r];
    const long k = (long)r * sn;
    if (mode == UPD_STAGE1) {
      v.Wh = a.Sn_hi[sc + k];
      v.Wl = a.Sn_lo[sc + k];
      v.gxh = gbx[r]; v.gxl = 0.0f;
      v.gyh = gby[r]; v.gyl = 0.0f;
      if (a.grad_base) {
        v.gxh = a.Sn_hi[sc + 4 * P + k]; v.gxl = a.Sn_lo[sc + 4 * P + k];
        v.gyh = a.Sn_hi[sc + 8 * P + k]; v.gyl = a.Sn_lo[sc + 8 * P + k];
      }
      float ah = v.Wh, al = v.Wl;
      ff_add(v.Wh, v.Wl, __fmaf_rn(0.125f * dtr * dtr, Ll[0][r], __fmul_rn(0.5f * dtr, Ll[1][r])));
      ff_add(ah, al, __fmaf_rn(dtr * dtr * (1.0f / 6.0f), Ll[0][r], __fmul_rn(dtr, Ll[1][r])));
      a.Acc_hi[ac + k] = ah;
      a.Acc_lo[ac + k] = al;
      // the gradient base: re-evaluated gradients are FP32 values (low part 0,
      // not stored); a base taken from the state keeps its low part
      a.Gb_hi[bc + k] = v.gxh;
      a.Gb_hi[bc + 4 * P + k] = v.gyh;
      if (a.grad_base) {
        a.Gb_lo[bc + k] = v.gxl;
        a.Gb_lo[bc + 4 * P + k] = v.gyl;
      }
      ff_add(v.gxh, v.gxl, __fmul_rn(0.5f * dtr, gtx[r]));
      ff_add(v.gyh, v.gyl, __fmul_rn(0.5f * dtr, gty[r]));
    } else {
      v.Wh = a.Acc_hi[ac + k];
      v.Wl = a.Acc_lo[ac + k];
      v.gxh = a.Gb_hi[bc + k];
      v.gyh = a.Gb_hi[bc + 4 * P + k];
      v.gxl = a.grad_base ? a.Gb_lo[bc + k] : 0.0f;
      v.gyl = a.grad_base ? a.Gb_lo[bc + 4 * P + k] : 0.0f;
      ff_add(v.Wh, v.Wl, __fmul_rn(dtr * dtr * (1.0f / 3.0f), Ll[0][r]));
      ff_add(v.gxh, v.gxl, __fmul_rn(dtr, gtx[r]));
      ff_add(v.gyh, v.gyl, __fmul_rn(dtr, gty[r]));
    }
  }
}

// second half: the walls, the stores and the positivity flag; W[comp] are the
// four components' high parts of the node (before the walls)
__device__ __forceinline__ void update_comp_store(const KArgs<float>& a, int g, int c, int i, int j, CompOut v,
                                                  float w0, float w1, float w2) {
  const Layout& L = a.L;
  const int nxg = g == 0 ? L.nx : L.nxd, nyg = g == 0 ? L.ny : L.nyd;
  // dual nodes on a no-slip wall: velocity set to zero (internal energy kept),
  // and, as U = V = 0 along the whole wall, the momentum gradients along it too
  const bool xwall = g == 1 && ((a.bc[0] == 3 && i == 0) || (a.bc[1] == 3 && i == nxg - 1));
  const bool ywall = g == 1 && ((a.bc[2] == 3 && j == 0) || (a.bc[3] == 3 && j == nyg - 1));
  if (xwall || ywall) {
    if (c == 3) ff_add(v.Wh, v.Wl, __fmul_rn(-0.5f, __fmaf_rn(w2, w2, __fmul_rn(w1, w1))) / w0);
    if (c == 1 || c == 2) {
      v.Wh = v.Wl = 0.0f;
      if (xwall) v.gyh = v.gyl = 0.0f;   // y-gradients of rho U, rho V
      if (ywall) v.gxh = v.gxl = 0.0f;   // x-gradients of rho U, rho V
    }
    w1 = w2 = 0.0f;
  }
  const long k = ((long)g * NFLD + c) * L.plane + cell(L, i, j);
  a.Out_hi[k] = v.Wh;
  a.Out_hi[k + 4 * L.plane] = v.gxh;
  a.Out_hi[k + 8 * L.plane] = v.gyh;
  if (a.Out_lo) {
    a.Out_lo[k] = v.Wl;
    a.Out_lo[k + 4 * L.plane] = v.gxl;
    a.Out_lo[k + 8 * L.plane] = v.gyl;
  }
  if (c == 3) {
    const float pr = v.Wh - 0.5f * (w1 * w1 + w2 * w2) / w0;
    if (!(w0 > 0.0f) || !(pr > 0.0f)) atomicOr(a.flag, 1);
  }
}

// A block's nodes: lane l takes ROWS rows from column and row `at`.  The
// components meet in shared memory for the walls and the positivity test.
template <int ROWS>
__device__ __forceinline__ void update_block(const KArgs<float>& a, int mode, int g, int2 at, float (*sw)[4][32]) {
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nxg = g == 0 ? a.L.nx : a.L.nxd, nyg = g == 0 ? a.L.ny : a.L.nyd;
  const bool in = at.x < nxg && at.y < nyg;
  CompOut o[ROWS];
  if (in) {
    update_comp<ROWS>(a, mode, g, c, at.x, at.y, nyg - at.y, o);
#pragma unroll
    for (int r = 0; r < ROWS; ++r) sw[r][c][lane] = o[r].Wh;
  }
  if (mode == UPD_OPERATOR) return;
  __syncthreads();
  if (!in) return;
#pragma unroll
  for (int r = 0; r < ROWS; ++r)
    if (at.y + r < nyg)
      update_comp_store(a, g, c, at.x, at.y + r, o[r], sw[r][0][lane], sw[r][1][lane], sw[r][2][lane]);
}

template <int ROWS>
__global__ void __launch_bounds__(128, UpdRows<ROWS>::minb) update_comp_kernel(KArgs<float> a, int mode) {
  __shared__ float sw[ROWS][4][32];
  step_begin();
  update_block<ROWS>(a, mode, blockIdx.z, make_int2(blockIdx.x * 32 + (threadIdx.x & 31), blockIdx.y * ROWS), sw);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
inline dim3 grid2(int nxp, int nyp, dim3 b, int z) {
  return dim3((unsigned)((nxp + b.x - 1) / b.x), (unsigned)((nyp + b.y - 1) / b.y), (unsigned)z);
}

template <class R>
cudaError_t launch_nodal(const KArgs<R>& a, cudaStream_t s) {
  dim3 b(32, 4);
  int mx = (a.L.nx > a.L.nxd ? a.L.nx : a.L.nxd) + 2, my = (a.L.ny > a.L.nyd ? a.L.ny : a.L.nyd) + 2;
  return launch_step(a.overlap, nodal_kernel<R>, grid2(mx, my, b, 2), b, s, a);
}

// interface points, with the nodal work in the same launch if nodal is set
template <class R>
cudaError_t launch_points(const KArgs<R>& a, bool nodal, cudaStream_t s) {
  const Layout& L = a.L;
  StageGrid G;
  const int T = StageTune<R>::threads;
  long blocks;
  if (IsF32<R>::v) {
    auto up = [](int n, int b) { return (n + b - 1) / b; };
    G.wA = up(L.nx + 3, 16); G.nA = G.wA * up(L.nyd + 3, 4);
    G.wB = up(L.nxd + 3, 16); G.nB = G.wB * up(L.ny + 3, 4);
    G.w0 = up(L.nx + 2, 32); G.nN0 = G.w0 * up(L.ny + 2, 4);
    G.w1 = up(L.nxd + 2, 32); G.nN1 = G.w1 * up(L.nyd + 2, 4);
    blocks = (long)G.nA + G.nB + (nodal ? G.nN0 + G.nN1 : 0);
  } else {
    G.wA = L.nx + 3; G.nA = G.wA * (L.nyd + 3);
    G.wB = L.nxd + 3; G.nB = G.wB * (L.ny + 3);
    G.w0 = L.nx + 2; G.nN0 = G.w0 * (L.ny + 2);
    G.w1 = L.nxd + 2; G.nN1 = G.w1 * (L.nyd + 2);
    const long np = (2L * G.nA + 2L * G.nB + 31) / 32 * 32;
    blocks = (np + (nodal ? (long)G.nN0 + G.nN1 : 0) + T - 1) / T;
  }
  auto kernel = a.recon_vars ? (nodal ? stage_kernel<R, true, true> : stage_kernel<R, true, false>)
                             : (nodal ? stage_kernel<R, false, true> : stage_kernel<R, false, false>);
  return launch_step(a.overlap, kernel, dim3((unsigned)blocks), dim3(T), s, a, G);
}

template <class R>
cudaError_t launch_update(const KArgs<R>& a, int mode, cudaStream_t s) {
  const int mx = a.L.nx > a.L.nxd ? a.L.nx : a.L.nxd, my = a.L.ny > a.L.nyd ? a.L.ny : a.L.nyd;
  if constexpr (IsF32<R>::v) {
    const long nn = (long)mx * my;
    const int rows = nn > UPD_LARGE_NODES ? 4 : nn > UPD_SMALL_NODES ? 2 : 1;
    auto kernel = rows == 4 ? update_comp_kernel<4> : rows == 2 ? update_comp_kernel<2> : update_comp_kernel<1>;
    return launch_step(a.overlap, kernel, grid2(mx, my, dim3(32, rows), 2), dim3(128), s, a, mode);
  } else {
    const dim3 b(32, 4);
    update_kernel<<<grid2(mx, my, b, 2), b, 0, s>>>(a, mode);
    return cudaGetLastError();
  }
}

// ---------------------------------------------------------------------------
// component batches
// ---------------------------------------------------------------------------
template <class R>
__global__ void iface_batch_kernel(GasK<R> gas, int normal, int n, const double* in, double* out) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  R v[20];
  for (int k = 0; k < 20; ++k) v[k] = (R)in[(long)t * 20 + k];
  IfaceOut<R> o;
  iface_solve(gas, normal, v, v + 4, v + 8, v + 12, v + 16, true, o);
  double* q = out + (long)t * 24;
  for (int k = 0; k < 4; ++k) {
    q[k] = o.F[k]; q[4 + k] = o.Ft[k]; q[8 + k] = o.Wl[k];
    q[12 + k] = o.Wr[k]; q[16 + k] = o.Wlt[k]; q[20 + k] = o.Wrt[k];
  }
}

template <class R>
__global__ void nodal_batch_kernel(GasK<R> gas, int n, const double* in, double* out) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  R v[12];
  for (int k = 0; k < 12; ++k) v[k] = (R)in[(long)t * 12 + k];
  R F[4], G[4], Ft[4], Gt[4];
  nodal_flux(gas, v, v + 4, v + 8, F, G, Ft, Gt);
  double* q = out + (long)t * 16;
  for (int k = 0; k < 4; ++k) { q[k] = F[k]; q[4 + k] = G[k]; q[8 + k] = Ft[k]; q[12 + k] = Gt[k]; }
}

template <class R>
__global__ void recon_batch_kernel(GenoK<R> g, int kind, R h, R ih, int n, const double* in, double* out) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  if (kind == 0) {
    R Q[4], Qx[4];
    for (int k = 0; k < 4; ++k) { Q[k] = (R)in[(long)t * 8 + k]; Qx[k] = (R)in[(long)t * 8 + 4 + k]; }
    R vl, dl, cl, vr, dr, cr;
    recon_interface(g, Q, Qx, h, ih, vl, dl, cl, vr, dr, cr);
    double* q = out + (long)t * 6;
    q[0] = vl; q[1] = dl; q[2] = cl; q[3] = vr; q[4] = dr; q[5] = cr;
  } else {
    R Q[3], Qx[3];
    for (int k = 0; k < 3; ++k) { Q[k] = (R)in[(long)t * 6 + k]; Qx[k] = (R)in[(long)t * 6 + 3 + k]; }
    out[(long)t * 6] = recon_node(g, Q, Qx, h, ih);
    for (int k = 1; k < 6; ++k) out[(long)t * 6 + k] = 0.0;
  }
}

template <class R>
cudaError_t launch_iface_batch(const GasK<R>& gas, int normal, int n, const double* in, double* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  iface_batch_kernel<R><<<(n + 63) / 64, 64, 0, s>>>(gas, normal, n, in, out);
  return cudaGetLastError();
}
template <class R>
cudaError_t launch_nodal_batch(const GasK<R>& gas, int n, const double* in, double* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  nodal_batch_kernel<R><<<(n + 63) / 64, 64, 0, s>>>(gas, n, in, out);
  return cudaGetLastError();
}
template <class R>
cudaError_t launch_recon_batch(const GenoK<R>& g, int kind, double h, int n, const double* in, double* out,
                               cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  recon_batch_kernel<R><<<(n + 127) / 128, 128, 0, s>>>(g, kind, (R)h, (R)(1.0 / h), n, in, out);
  return cudaGetLastError();
}

#define FDK_INSTANTIATE(R)                                                                                  \
  template cudaError_t launch_nodal<R>(const KArgs<R>&, cudaStream_t);                                     \
  template cudaError_t launch_points<R>(const KArgs<R>&, bool, cudaStream_t);                                    \
  template cudaError_t launch_update<R>(const KArgs<R>&, int, cudaStream_t);                               \
  template cudaError_t launch_iface_batch<R>(const GasK<R>&, int, int, const double*, double*, cudaStream_t); \
  template cudaError_t launch_nodal_batch<R>(const GasK<R>&, int, const double*, double*, cudaStream_t);   \
  template cudaError_t launch_recon_batch<R>(const GenoK<R>&, int, double, int, const double*, double*,     \
                                             cudaStream_t);

}  // namespace fdk
