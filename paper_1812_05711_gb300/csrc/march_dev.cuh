// march_dev.cuh -- the FP32 collision of the fused collide-and-stream kernels
// (Eqs. 5-15), shared by the march forms (k_march.cu) and the kernel that keeps
// a whole run on chip (k_resident.cu).
#pragma once

#include "ehd_dev.cuh"

namespace ehd {

// A product that is rounded, and a multiply-add that is rounded once: below,
// every product that meets a sum is written as one of the two (FP32; products
// by 1/2 are exact), so that a node has the same bits in the march forms, one
// node per thread, on chip and in a batch whatever the compiler would make of
// each.  Which of two products is rounded follows what it made of them before this
// was written down (each choice tried against it on 3.3e4 nodes, all populations).
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_(double a, double b) { return a * b; }
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_(double a, double b) { return a + b; }
__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return a * b + c; }

template <class R>
__device__ __forceinline__ void trt_f2(R& fi, R& fo, R w, R drho, R rho, R cu, R usq15, R cF, R uF3, R wp, R wm, R cp,
                                       R cm) {
  const R ep = mul_(w, fma_(rho, fma_(R(4.5) * cu, cu, -usq15), drho));
  const R em = mul_(w * rho * R(3), cu);
  const R Fp = mul_(w, fma_(R(9) * cu, cF, -uF3));
  const R Fm = mul_(w * R(3), cF);
  const R sp = R(0.5) * (fi + fo), sm = R(0.5) * (fi - fo);
  const R A = fma_(cp, Fp, -mul_(wp, sp - ep));
  const R B = fma_(cm, Fm, -mul_(wm, sm - em));
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
  const R ep = mul_(w, fma_(rho, fma_(R(4.5) * cu, cu, -usq15), drho));
  const R em = mul_(w, fma_(rho * R(3), cu, dq));
  const R Fp = mul_(w, fma_(R(9) * cu, cF, -uF3));
  const R Fm = mul_(w * R(3), cF);
  const R sp = R(0.5) * (fi + fo), sm = R(0.5) * (fi - fo);
  const R A = fma_(cp, Fp, -mul_(wp, sp - ep));
  const R B = fma_(cm, Fm, -mul_(wm, sm - em));
  fi = fi + A + B;
  fo = fo + A - B;
}

template <class R>
__device__ __forceinline__ void trt_g2(R& gi, R& go, R w, R drc, R rc, R cv, R vsq15, R wp, R wm) {
  const R ep = mul_(w, fma_(rc, fma_(R(4.5) * cv, cv, -vsq15), drc));
  const R em = mul_(w * rc * R(3), cv);
  const R sp = R(0.5) * (gi + go), sm = R(0.5) * (gi - go);
  const R dp = sp - ep, dm = sm - em;
  gi = fma_(-wm, dm, fma_(-wp, dp, gi));
  go = fma_(wm, dm, fma_(-wp, dp, go));
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
  const R Fx = mul_(rc, Ex), Fy = mul_(rc, Ey);
  const R irho = R(1) / rho;
  const R ux = mul_(fma_(R(0.5), Fx, jx), irho);
  const R uy = mul_(fma_(R(0.5), Fy, jy), irho);
  const R vx = ux + mul_(mub, Ex), vy = uy + mul_(mub, Ey);
  const R usq15 = mul_(R(1.5), fma_(ux, ux, mul_(uy, uy)));
  const R uF3 = mul_(R(3), fma_(ux, Fx, mul_(uy, Fy)));
  f[0] = fma_(-mul_(cp, W0), uF3, fma_(-wp, fma_(-W0, fma_(-rho, usq15, drho), f[0]), f[0]));
  trt_f2<R>(f[1], f[3], W1, drho, rho, ux, usq15, Fx, uF3, wp, wm, cp, cm);
  trt_f2y<R>(f[2], f[4], W1, drho, rho, uy, usq15, Fy, uF3, wp, wm, cp, cm, dq);
  trt_f2y<R>(f[5], f[7], W2, drho, rho, ux + uy, usq15, Fx + Fy, uF3, wp, wm, cp, cm, dq);
  trt_f2y<R>(f[6], f[8], W2, drho, rho, uy - ux, usq15, Fy - Fx, uF3, wp, wm, cp, cm, dq);
  const R vsq15 = mul_(R(1.5), fma_(vx, vx, mul_(vy, vy)));
  g[0] = fma_(-gwp, fma_(-W0, fma_(-rc, vsq15, drc), g[0]), g[0]);
  trt_g2<R>(g[1], g[3], W1, drc, rc, vx, vsq15, gwp, gwm);
  trt_g2<R>(g[2], g[4], W1, drc, rc, vy, vsq15, gwp, gwm);
  trt_g2<R>(g[5], g[7], W2, drc, rc, vx + vy, vsq15, gwp, gwm);
  trt_g2<R>(g[6], g[8], W2, drc, rc, vy - vx, vsq15, gwp, gwm);
}

// Injector: anti-bounce-back of g imposing rho_c = rho0 with the wall drift mu_b E
// (fluid at rest on the wall): the new populations 2, 5, 6 from 4, 7, 8.
template <class R>
__device__ __forceinline__ void inject(R g4, R g7, R g8, R Ex, R Ey, R sy, R mub, R rho0, R& n2, R& n5, R& n6) {
  // (plain products, which meet no plain sum: the collision's mul_(mub, E) would
  // be kept in a register for them, 128 x 104 6.7 us per step against 6.3)
  const R wx = mub * Ex, wy = mub * Ey, w2 = fma_(wx, wx, mul_(wy, wy));
  auto one = [&](R g, R W, R c) {
    const R even = fma_(R(-1.5), w2, fma_(R(4.5) * c, c, R(1)));
    return fma_(mul_(R(2) * W, rho0), even, -fma_(R(2) * W, sy, g));
  };
  n2 = one(g4, (R)kW1, wy);
  n5 = one(g7, (R)kW2, add_(wx, wy));
  n6 = one(g8, (R)kW2, add_(wy, -wx));
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
