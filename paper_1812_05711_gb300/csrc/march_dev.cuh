// march_dev.cuh -- the FP32 collision of the fused collide-and-stream kernels
// (Eqs. 5-15), shared by the march forms (k_march.cu) and the kernel that keeps
// a whole run on chip (k_resident.cu).
#pragma once

#include "ehd_dev.cuh"

namespace ehd {

template <class R>
__device__ __forceinline__ void trt_f2(R& fi, R& fo, R w, R drho, R rho, R cu, R usq15, R cF, R uF3, R wp, R wm, R cp,
                                       R cm) {
  const R ep = w * (drho + rho * (R(4.5) * cu * cu - usq15));
  const R em = w * rho * R(3) * cu;
  const R Fp = w * (R(9) * cu * cF - uF3);
  const R Fm = w * R(3) * cF;
  const R sp = R(0.5) * (fi + fo), sm = R(0.5) * (fi - fo);
  const R A = cp * Fp - wp * (sp - ep);
  const R B = cm * Fm - wm * (sm - em);
  fi = fi + A + B;
  fo = fo + A - B;
}

// trt_f2 for a pair that crosses rows (fi moves up, fo down) in storage
// shifted by a density ramp r(y) = r(0) + dr y: with dq = -dr / omega- the
// antisymmetric part hands fi its storage offset change -w dr and fo +w dr,
// at no extra instruction (dq is added inside the product w (3 rho cu + dq)).
template <class R>
__device__ __forceinline__ void trt_f2y(R& fi, R& fo, R w, R drho, R rho, R cu, R usq15, R cF, R uF3, R wp, R wm,
                                        R cp, R cm, R dq) {
  const R ep = w * (drho + rho * (R(4.5) * cu * cu - usq15));
  const R em = w * (rho * R(3) * cu + dq);
  const R Fp = w * (R(9) * cu * cF - uF3);
  const R Fm = w * R(3) * cF;
  const R sp = R(0.5) * (fi + fo), sm = R(0.5) * (fi - fo);
  const R A = cp * Fp - wp * (sp - ep);
  const R B = cm * Fm - wm * (sm - em);
  fi = fi + A + B;
  fo = fo + A - B;
}

template <class R>
__device__ __forceinline__ void trt_g2(R& gi, R& go, R w, R drc, R rc, R cv, R vsq15, R wp, R wm) {
  const R ep = w * (drc + rc * (R(4.5) * cv * cv - vsq15));
  const R em = w * rc * R(3) * cv;
  const R sp = R(0.5) * (gi + go), sm = R(0.5) * (gi - go);
  const R A = -wp * (sp - ep);
  const R B = -wm * (sm - em);
  gi = gi + A + B;
  go = go + A - B;
}

template <class S, class R>
__device__ __forceinline__ void collide_node(R (&f)[9], R (&g)[9], R Ex, R Ey, R sy, R sf, R dq, R mub, R wp, R wm,
                                             R cp, R cm, R gwp, R gwm, bool& bad) {
  if constexpr (sizeof(R) == 8) {  // unshifted: sy, sf and dq are zero
    collide_f64(f, g, Ex, Ey, mub, collide_f64_constants(wp, wm, gwp, gwm), bad);
    return;
  }
  const R W0 = (R)kW0, W1 = (R)kW1, W2 = (R)kW2;
  const R drho = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
  const R rho = sf + drho;
  const R jx = (f[1] - f[3]) + (f[5] - f[7]) + (f[8] - f[6]);
  const R jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
  const R drc = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8];
  const R rc = sy + drc;
  bad = !isfinite(drho) || !isfinite(drc);
  const R Fx = rc * Ex, Fy = rc * Ey;
  const R irho = R(1) / rho;
  const R ux = (jx + R(0.5) * Fx) * irho;
  const R uy = (jy + R(0.5) * Fy) * irho;
  const R vx = ux + mub * Ex, vy = uy + mub * Ey;
  const R usq15 = R(1.5) * (ux * ux + uy * uy);
  const R uF3 = R(3) * (ux * Fx + uy * Fy);
  f[0] = f[0] - wp * (f[0] - W0 * (drho - rho * usq15)) - cp * W0 * uF3;
  trt_f2<R>(f[1], f[3], W1, drho, rho, ux, usq15, Fx, uF3, wp, wm, cp, cm);
  trt_f2y<R>(f[2], f[4], W1, drho, rho, uy, usq15, Fy, uF3, wp, wm, cp, cm, dq);
  trt_f2y<R>(f[5], f[7], W2, drho, rho, ux + uy, usq15, Fx + Fy, uF3, wp, wm, cp, cm, dq);
  trt_f2y<R>(f[6], f[8], W2, drho, rho, uy - ux, usq15, Fy - Fx, uF3, wp, wm, cp, cm, dq);
  const R vsq15 = R(1.5) * (vx * vx + vy * vy);
  g[0] = g[0] - gwp * (g[0] - W0 * (drc - rc * vsq15));
  trt_g2<R>(g[1], g[3], W1, drc, rc, vx, vsq15, gwp, gwm);
  trt_g2<R>(g[2], g[4], W1, drc, rc, vy, vsq15, gwp, gwm);
  trt_g2<R>(g[5], g[7], W2, drc, rc, vx + vy, vsq15, gwp, gwm);
  trt_g2<R>(g[6], g[8], W2, drc, rc, vy - vx, vsq15, gwp, gwm);
}

// Charge density of one node from its new populations z(0) .. z(8) and the
// shift s of its row, summed as the march form leaves it: a slab's last row
// lacks the populations pushed down into it, its first row those pushed up,
// until the forward transform adds their shares.
template <class Z>
__device__ __forceinline__ float march_charge(float s, bool first, bool last, Z&& z) {
  const float h = (z(0) + z(1)) + z(3), u = (z(2) + z(5)) + z(6), d = (z(4) + z(7)) + z(8);
  const float hu = first ? h : h + u;
  float r = last ? s + hu : s + (hu + d);
  if (last) r += d;
  if (first) r += u;
  return r;
}
// row y opens / closes a slab of S rows
__device__ __forceinline__ bool slab_first(int y, int S) { return y > 0 && y % S == 0; }
__device__ __forceinline__ bool slab_last(int y, int Ny, int S) { return y + 1 < Ny && (y + 1) % S == 0; }

}  // namespace ehd
