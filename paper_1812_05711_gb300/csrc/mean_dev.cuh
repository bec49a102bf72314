// mean_dev.cuh -- the m = 0 mode of the Poisson solve (the row means), shared by
// the kernels that solve it (k_poisson.cu) and the one that keeps a whole run
// on chip (k_resident.cu).
#pragma once

#include <algorithm>

#include "ehd_dev.cuh"

namespace ehd {

// Float-float ("double-single") numbers for the FP32 path: value = hi + lo
// with |lo| <= ulp(hi)/2, about 48 significant bits, on the FP32 pipes (scalar
// FP64 is slow on this part).  Error-free transformations: Knuth's two-sum
// and the FMA two-product.
struct ff {
  float hi, lo;
};
__device__ __forceinline__ ff ff_from(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}
__device__ __forceinline__ double ff_to(ff a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  const float s = a.hi + b.hi;
  const float bb = s - a.hi;
  const float e = (a.hi - (s - bb)) + (b.hi - bb) + a.lo + b.lo;
  const float h = s + e;
  return {h, e - (h - s)};
}
__device__ __forceinline__ ff ff_neg(ff a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = a.hi * b.hi;
  const float e = fmaf(a.hi, b.hi, -p) + (a.hi * b.lo + a.lo * b.hi);
  const float h = p + e;
  return {h, e - (h - p)};
}
__device__ __forceinline__ ff ff_shfl_up(ff a, int o) {
  return {__shfl_up_sync(0xffffffffu, a.hi, o), __shfl_up_sync(0xffffffffu, a.lo, o)};
}
__device__ __forceinline__ ff ff_shfl_down(ff a, int o) {
  return {__shfl_down_sync(0xffffffffu, a.hi, o), __shfl_down_sync(0xffffffffu, a.lo, o)};
}

// Mean-mode arithmetic: native double, or float-float.
template <class R>
struct MeanNum;
template <>
struct MeanNum<double> {
  using T = double;
  __device__ static T from(double v) { return v; }
  __device__ static T from_f(float v) { return (double)v; }
  __device__ static T from_i(int v) { return (double)v; }
  __device__ static T pair(double d, float, float) { return d; }
  __device__ static double to(T v) { return v; }
  __device__ static T add(T a, T b) { return a + b; }
  __device__ static T mul(T a, T b) { return a * b; }
  __device__ static T neg(T a) { return -a; }
  __device__ static T up(T a, int o) { return __shfl_up_sync(0xffffffffu, a, o); }
  __device__ static T down(T a, int o) { return __shfl_down_sync(0xffffffffu, a, o); }
};
template <>
struct MeanNum<float> {
  using T = ff;
  __device__ static T from(double v) { return ff_from(v); }
  __device__ static T from_f(float v) { return {v, 0.0f}; }
  // exact for |v| <= 2^24, and then equal to ff_from((double)v)
  __device__ static T from_i(int v) { return {(float)v, 0.0f}; }
  // a constant the host split into (hi, lo): equal to ff_from(d)
  __device__ static T pair(double, float hi, float lo) { return {hi, lo}; }
  __device__ static double to(T v) { return ff_to(v); }
  __device__ static T add(T a, T b) { return ff_add(a, b); }
  __device__ static T mul(T a, T b) { return ff_mul(a, b); }
  __device__ static T neg(T a) { return ff_neg(a); }
  __device__ static T up(T a, int o) { return ff_shfl_up(a, o); }
  __device__ static T down(T a, int o) { return ff_shfl_down(a, o); }
};

// m = 0 (the row means) + the step's wall fluxes.  For m = 0 the system of
// Eq. 25 is the 1-D discrete Poisson equation phi_{j-1} - 2 phi_j + phi_{j+1}
// = s_j with the wall ghosts of the closure, whose solution is a double
// prefix sum: with D_j = phi_{j+1} - phi_j (j = -1 .. Ny-1),
//   D_j = D_{-1} + S_j,  S_j = sum_{k<=j} s_k,
//   phi_j = phi_{-1} + (j+1) D_{-1} + T_j,  T_j = sum_{k<j} S_k,
// and the two wall conditions fix phi_{-1} and D_{-1}.  Both sums are block
// scans (per-thread chunks, warp shuffles, one warp over the warp totals).
// Arithmetic: FP64 on the plain FP64 path, float-float on the FP32 path.
// Barrier among the first NT threads of the CTA (all of it when the CTA has
// NT threads): the mean mode may run on a sub-block of a larger CTA.
template <int NT>
__device__ __forceinline__ void sub_sync() {
  asm volatile("bar.sync 1, %0;\n" ::"n"(NT) : "memory");
}

template <class R, int NT>
struct MeanScratch {
  static constexpr int NW = NT / 32;
  typename MeanNum<R>::T wsum[NW], woff[NW], tot[2];
  double fq[2][NW];
};

// Inclusive prefix sum of v[0..Ny) in place (all NT threads; chunk [j0, j1)
// per thread); returns the total.
template <class R, int NT>
__device__ __forceinline__ typename MeanNum<R>::T block_prefix_sum(typename MeanNum<R>::T* v, int j0, int j1,
                                                                   MeanScratch<R, NT>& ms, int t) {
  using N = MeanNum<R>;
  using T = typename N::T;
  constexpr int NW = NT / 32;
  const int lane = t & 31, warp = t >> 5;
  T acc = N::from_f(0.0f);
  for (int j = j0; j < j1; ++j) {
    acc = N::add(acc, v[j]);
    v[j] = acc;
  }
  T incl = acc;  // inclusive scan of the chunk totals over the warp
  for (int o = 1; o < 32; o <<= 1) {
    const T u = N::up(incl, o);
    if (lane >= o) incl = N::add(incl, u);
  }
  if (lane == 31) ms.wsum[warp] = incl;
  sub_sync<NT>();
  if (warp == 0) {
    T w = lane < NW ? ms.wsum[lane] : N::from_f(0.0f);
    for (int o = 1; o < NW; o <<= 1) {
      const T u = N::up(w, o);
      if (lane >= o) w = N::add(w, u);
    }
    T ex = N::up(w, 1);
    if (lane == 0) ex = N::from_f(0.0f);
    if (lane < NW) ms.woff[lane] = ex;
    if (lane == NW - 1) ms.tot[0] = w;
  }
  sub_sync<NT>();
  T ex = N::up(incl, 1);  // chunks of the earlier lanes of this warp
  if (lane == 0) ex = N::from_f(0.0f);
  const T off = N::add(ms.woff[warp], ex);
  for (int j = j0; j < j1; ++j) v[j] = N::add(v[j], off);
  const T total = ms.tot[0];
  sub_sync<NT>();
  return total;
}

// The solve itself by threads t < NT: v[0 .. Ny) holds the row sums (v[Ny ..
// 2 Ny) is scratch); put(j, phi_j, E_j) takes the rows' results.
template <class R, int NT, class Put>
__device__ __forceinline__ void mean_mode_core(const PoissonArgs& a, typename MeanNum<R>::T* v,
                                               MeanScratch<R, NT>& ms, int t, Put&& put) {
  using N = MeanNum<R>;
  using T = typename N::T;
  const int Ny = a.Ny;
  const int C = (Ny + NT - 1) / NT;
  const int j0 = min(t * C, Ny), j1 = min(j0 + C, Ny);
  T* Sv = v + Ny;  // [Ny]: copy of S
  // S_j (inclusive), kept in Sv; then v[j] = sum_{k<=j} S_k = T_{j+1}
  block_prefix_sum<R, NT>(v, j0, j1, ms, t);
  for (int j = j0; j < j1; ++j) Sv[j] = v[j];
  const T T_all = block_prefix_sum<R, NT>(v, j0, j1, ms, t);   // T_Ny
  const T T_last = (Ny >= 2) ? v[Ny - 2] : N::from_f(0.0f);  // T_{Ny-1}
  // wall values in spectral units: W = Nx phi0 at the injector, 0 at the
  // collector; W and the closure factor come from the host
  const T W = N::pair(a.mW, a.mWf[0], a.mWf[1]);
  T Dm, Pm;  // D_{-1}, phi_{-1}
  if (a.wall_mode == 0) {
    // phi_{-1} + phi_0 = 2W, phi_Ny + phi_{Ny-1} = 0: D_{-1} = -(2W + T_Ny + T_{Ny-1}) / (2 Ny)
    const T num = N::add(N::add(W, W), N::add(T_all, T_last));
    Dm = N::mul(N::neg(num), N::pair(a.mC, a.mCf[0], a.mCf[1]));
    Pm = N::add(W, N::neg(N::mul(Dm, N::from_f(0.5f))));
  } else {
    // phi_{-1} = W, phi_Ny = 0: D_{-1} = -(W + T_Ny) / (Ny + 1)
    Dm = N::mul(N::neg(N::add(W, T_all)), N::pair(a.mC, a.mCf[0], a.mCf[1]));
    Pm = W;
  }
  // phi_j = phi_{-1} + (j+1) D_{-1} + T_j,  E_j = -(2 D_{-1} + S_j + S_{j-1}) / 2
  const T inN = N::from_f(1.0f / (float)a.Nx);
  const T mhalf = N::from_f(-0.5f);
  for (int j = j0; j < j1; ++j) {
    const T Tj = (j > 0) ? v[j - 1] : N::from_f(0.0f);
    const T Sj = Sv[j], Sjm1 = (j > 0) ? Sv[j - 1] : N::from_f(0.0f);
    const T phi = N::add(N::add(Pm, N::mul(N::from_i(j + 1), Dm)), Tj);
    const T ey = N::mul(mhalf, N::add(N::add(Dm, Dm), N::add(Sj, Sjm1)));
    put(j, N::mul(phi, inN), N::mul(ey, inN));
  }
}

// The step's wall fluxes, added to the run's FP64 totals by threads t < NT: a
// shuffle tree over the strips, in the warps that hold partials (the others'
// totals would be +0, whose addition changes nothing; FP64 issue is slow on
// this part).
template <int NT>
__device__ __forceinline__ void wall_flux_totals(const PoissonArgs& a, double (*fq)[NT / 32], int t) {
  constexpr int NW = NT / 32;
  const int lane = t & 31, warp = t >> 5;
  const int nfw = min(NW, (a.nflux + 31) / 32);
  double qi = 0.0, qo = 0.0;
  if (warp < nfw) {
    for (int b = t; b < a.nflux; b += NT) {
      qi += __ldcg(a.flux_part + b);
      qo += __ldcg(a.flux_part + a.nflux + b);
    }
    for (int o = 16; o > 0; o >>= 1) {
      qi += __shfl_down_sync(0xffffffffu, qi, o);
      qo += __shfl_down_sync(0xffffffffu, qo, o);
    }
  }
  if (lane == 0 && warp < nfw) {
    fq[0][warp] = qi;
    fq[1][warp] = qo;
  }
  sub_sync<NT>();
  if (t == 0) {
    double si = 0.0, so = 0.0;
    for (int w = 0; w < nfw; ++w) {
      si += fq[0][w];
      so += fq[1][w];
    }
    a.flux_acc[0] += si;
    a.flux_acc[1] += so;
  }
}

// The mean mode of a run by threads t < NT (v: 2 Ny numbers), from its row sums.
template <class R, int NT>
__device__ __forceinline__ void mean_mode_solve(const PoissonArgs& a, typename MeanNum<R>::T* v,
                                                MeanScratch<R, NT>& ms, int t) {
  using T = typename MeanNum<R>::T;
  for (int j = t; j < a.Ny; j += NT) {
    if constexpr (sizeof(R) == 8) {
      v[j] = __ldcg(static_cast<const double*>(a.spec0) + j);
    } else {
      const float2 s = __ldcg(static_cast<const float2*>(a.spec0) + j);
      v[j] = {s.x, s.y};
    }
  }
  sub_sync<NT>();
  mean_mode_core<R, NT>(a, v, ms, t, [&](int j, T pc, T ec) {
    R* Ebar = static_cast<R*>(a.Ebar);
    if constexpr (sizeof(R) == 8) {
      static_cast<double*>(a.phibar)[j] = pc;
      Ebar[j] = ec;
    } else {
      static_cast<float2*>(a.phibar)[j] = make_float2(pc.hi, pc.lo);
      Ebar[j] = ec.hi + ec.lo;
    }
  });
}

template <class R, int NT>
__device__ __forceinline__ void mean_mode_body(const PoissonArgs& a, unsigned char* smem_raw,
                                               MeanScratch<R, NT>& ms) {
  if (a.flux_part) wall_flux_totals<NT>(a, ms.fq, threadIdx.x);
  mean_mode_solve<R, NT>(a, reinterpret_cast<typename MeanNum<R>::T*>(smem_raw), ms, threadIdx.x);
}

// threads of the mean mode: 128 up to 1024 rows (shorter scans over the
// warps), 512 above (shorter per-thread chunks)
constexpr int kMeanThreads = 512;
constexpr int kMeanThreadsSmall = 128;
constexpr int kMeanSmallRows = 1024;

}  // namespace ehd
