// ehd_dev.cuh -- device-side types shared by the kernels and the host code of
// the GB300 electroconvection library (D2Q9 TRT lattice Boltzmann for fluid f
// and charge g, FFT/tridiagonal Poisson solve; arXiv:1812.05711).
//
// Memory layout of one run in HBM (all planes row-major, x fastest, rows
// padded to a pitch P that is a multiple of 32 elements = 128 B for FP32):
//   f[2], g[2]   population ping-pong buffers, [9][Ny][P] of the storage type
//   dphi         potential minus its row mean, [Ny][P] of the compute type R
//   phibar       row mean of the potential (the m = 0 mode), [Ny] FP64
//   Ebar         mean-mode field E_y per row, [Ny] of R
//   spec         half spectrum of every row, [Ny][Mh] complex R, Mh = Nx/2+1
//   spec0        mean-mode right-hand side / solution, [Ny] FP64
//   rfac         reciprocal Thomas pivots, mode-major [Mh][Ny] of R
//   rfac0        the same for m = 0, [Ny] FP64
//   tw           twiddles exp(-2 pi i k / Nx), k < Nx/2, complex R
//   rch          per-row charge shift (hydrostatic rho_c rounded to FP32), [Ny]
#pragma once

#include <cuda.h>  // CUtensorMap (types only; the encoder is reached through the runtime)
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ehd {

// D2Q9 numbering: c0=(0,0) c1=(1,0) c2=(0,1) c3=(-1,0) c4=(0,-1)
// c5=(1,1) c6=(-1,1) c7=(-1,-1) c8=(1,-1); weights 4/9, 1/9, 1/36.
constexpr double kW0 = 4.0 / 9.0;
constexpr double kW1 = 1.0 / 9.0;
constexpr double kW2 = 1.0 / 36.0;

// ------------------------------------------------------------ storage ---
template <class S> struct Store;
template <> struct Store<double> {
  template <class R> __device__ __forceinline__ static R ld(const double* p) { return (R)__ldg(p); }
  template <class R> __device__ __forceinline__ static void st(double* p, R v) { *p = (double)v; }
  template <class R> __device__ __forceinline__ static R rt(R v) { return v; }
};
template <> struct Store<float> {
  template <class R> __device__ __forceinline__ static R ld(const float* p) { return (R)__ldg(p); }
  template <class R> __device__ __forceinline__ static void st(float* p, R v) { *p = (float)v; }
  template <class R> __device__ __forceinline__ static R rt(R v) { return (R)(float)v; }
};
template <> struct Store<__nv_bfloat16> {
  template <class R> __device__ __forceinline__ static R ld(const __nv_bfloat16* p) {
    return (R)__bfloat162float(__ldg(p));
  }
  template <class R> __device__ __forceinline__ static void st(__nv_bfloat16* p, R v) {
    *p = __float2bfloat16_rn((float)v);
  }
  template <class R> __device__ __forceinline__ static R rt(R v) {
    return (R)__bfloat162float(__float2bfloat16_rn((float)v));
  }
};
// FP16 keeps the shifted populations scaled by 2^12: they are small (of the
// order of the flow's departure from the hydrostatic state, 1e-7 .. 1e-2)
// and would otherwise fall below FP16's normal range (6.1e-5); the scaled
// values stay far below its largest finite value.  Powers of two scale exactly.
constexpr float kHalfScale = 4096.0f, kHalfUnscale = 1.0f / 4096.0f;
template <> struct Store<__half> {
  template <class R> __device__ __forceinline__ static R ld(const __half* p) {
    return (R)(__half2float(__ldg(p)) * kHalfUnscale);
  }
  template <class R> __device__ __forceinline__ static void st(__half* p, R v) {
    *p = __float2half_rn((float)v * kHalfScale);
  }
  template <class R> __device__ __forceinline__ static R rt(R v) {
    return (R)(__half2float(__float2half_rn((float)v * kHalfScale)) * kHalfUnscale);
  }
};

template <class R> struct Cplx { R re, im; };

// ----------------------------------------------------------- kernel args ---
// Programmatic dependent launch.  A kernel launched with pdl = true may
// start while the previous kernel of its stream is still running.  The step's
// kernels keep these rules:
//  1. Before grid_dep_wait() a kernel reads nothing that its predecessor
//     writes, and writes nothing that its predecessor reads or writes.
//  2. The forward row transforms and the y solves release their successor
//     (grid_dep_launch, or by ending) only after their own grid_dep_wait().
//     So when an inverse transform starts, the forward transform and the step
//     kernel before it have completed, and when a step kernel starts, so have
//     the solve and all before it.
//  3. On the strength of 2, and only of 2: the step kernels (k_push, k_march2,
//     k_step64) read the populations before their wait, and the mean mode's
//     CTAs of k_irfft_warp read the m = 0 coefficients and the wall-flux
//     partials without one.  A step kernel is therefore launched with pdl only
//     where a Poisson solve lies between it and the populations' last writer;
//     behind k_resident, which is that writer itself, it is not.
//  4. The step kernels and the mean mode's CTAs may release before their wait:
//     their successor (the forward transform; the next step kernel) touches
//     what they write after its own wait only.
//  5. What a predecessor may still write while the kernel is resident is read
//     with plain loads, not through the non-coherent path (__ldg, or a const
//     __restrict__ pointer), whose data must not change in the kernel's life.
// Both instructions are no-ops in a kernel launched without the attribute.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_ex(bool pdl, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                      A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = at;
  c.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, static_cast<A&&>(args)...);
}

// Tensor maps of a run's spectrum [Ny][Mp] complex and pivots [Ny][Mp] (FP32)
// for staging a tile of 8 wavenumbers: boxes of 256 rows and one box of the
// last Ny % 256 rows.
struct ModesTma {
  CUtensorMap spec_full, spec_tail, rf_full, rf_tail;
  int nfull, tail;
};
// a 2-D FP32 tensor map: inner x outer elements, rows row_bytes apart
cudaError_t tma_encode_2d(CUtensorMap* m, const void* base, unsigned long long inner, unsigned long long outer,
                          unsigned long long row_bytes, unsigned box_inner, unsigned box_outer);
cudaError_t modes_tma_encode(ModesTma* t, const void* spec, const void* rfac, int Ny, int Mp);

// Constants of the FP64 collision (collide_f64).  The one-node-per-thread step
// takes them from the host: an FP64 instruction reads its constant operand from
// the kernel parameters, and no thread spends FP64 issue slots on forming one.
struct CollideF64 {
  double hp, hm;        // (1 - omega+) / 2, (1 - omega-) / 2
  double rw;            // W1 omega+
  double gj, gF;        // 4.5 W1 omega+, 4.5 W1 (2 - omega+ / 2)
  double jj, jF;        // 3 W1 omega-, 3 W1
  double ghp, ghm;      // (1 - omega_g+) / 2, (1 - omega_g-) / 2
  double grw, gg, gjm;  // W1 omega_g+, 4.5 W1 omega_g+, 3 W1 omega_g-
};
__host__ __device__ inline CollideF64 collide_f64_constants(double wp, double wm, double gwp, double gwm) {
  CollideF64 k;
  k.hp = 0.5 * (1.0 - wp);
  k.hm = 0.5 * (1.0 - wm);
  k.rw = kW1 * wp;
  k.gj = 4.5 * kW1 * wp;
  k.gF = 4.5 * kW1 * (2.0 - 0.5 * wp);
  k.jj = 3.0 * kW1 * wm;
  k.jF = 3.0 * kW1;
  k.ghp = 0.5 * (1.0 - gwp);
  k.ghm = 0.5 * (1.0 - gwm);
  k.grw = kW1 * gwp;
  k.gg = 4.5 * kW1 * gwp;
  k.gjm = 3.0 * kW1 * gwm;
  return k;
}

struct StepArgs {
  int Nx, Ny, P;
  long long plane;           // elements per population plane (Ny * P)
  const void* fin;
  const void* gin;
  void* fout;
  void* gout;
  const void* dphi;          // R [Ny][P]
  const void* Ebar;          // R [Ny]
  const float* rch;          // [Ny] charge shift, nullptr for unshifted storage
  double* flux_part;         // [2][nxb] per-CTA injected / collected charge
  int* err;                  // bit 0: non-finite density or charge
  double wp, wm, gwp, gwm;   // omega+, omega-, omega_g+, omega_g-
  double mub, rho0;          // ion mobility, injected density
  double fb, fd, fdq;        // f shift r(y) = fb + fd y (fd an FP32 value), and -fd / omega- (0 when unshifted)
  const void* ex;            // R [Ny][P]: spectral E_x, or nullptr for central differences of dphi
  int wall_mode;
  // march form only
  void* rhoc_out;            // R [Ny][P]: rho_c of the new state (slab-boundary rows: partial, see rhoc_dn)
  void* rhoc_dn;             // R [nslab][P]: row y0(b) - 1, charge of the populations pushed down by slab b
  void* rhoc_up;             // R [nslab][P]: row y0(b), charge of the populations pushed up by slab b - 1
  int slab_rows;             // rows per warp slab
  int slab_off;              // slab b covers rows [b*slab_rows - slab_off, (b+1)*slab_rows - slab_off) within
                             // [0, Ny), 0 <= slab_off < slab_rows (cp.async march, two columns per lane only)
  int nstrips;               // 32-column strips (30 owned columns each)
  int ring_depth;            // rows staged ahead by cp.async (2, 3, 4 or 6)
  int cols_per_lane;         // 1: 32-column strips (30 owned); 2: 64-column strips (60 owned)
  int pdl;                   // launch with programmatic dependent launch (see launch_ex)
  const float* base_tab;     // perturbation form: the march table of time t ([Ny][4]); nullptr otherwise
};

// -------------------------------------------------- FP64 TRT collision ---
// Scalar FP64 issues two lanes per clock and SM on this part (a warp's FP64
// instruction takes the unit 16 cycles), so the FP64 step is bound by its FP64
// instruction count and nothing else.  This is the collision of Eqs. 5-15
// with that count at about 130 per node (226 when every population's
// equilibrium, force and relaxation were formed one by one as in the FP32
// kernels):
//   - sums s and differences d of each pair of opposite populations serve the
//     moments and the relaxation alike;
//   - the post-collision pair is P + D, P - D with P = (1 - omega+) s / 2 +
//     E, D = (1 - omega-) d / 2 + J; since rho u = j + F / 2 (Eq. 7), the
//     equilibrium and the force enter E and J only through
//     G = 4.5 W1 (omega+ j + (2 - omega+ / 2) F) and 3 W1 (omega- j + F):
//     with C = W1 omega+ rho - u.G / 3 the axis pairs get C + u_x G_x and
//     C + u_y G_y, and the diagonal pairs a quarter of
//     C + u.G +- (u_x G_y + u_y G_x);
//   - the rest population takes what the pairs leave of the density, so the
//     mass and charge of a node are conserved to a rounding that has no
//     preferred sign, whatever the rounding of the constants;
//   - 1 / rho by two Newton-Raphson steps x' = x + x (1 - rho x) from the
//     hardware's approximation (see recip_f64).
// 1 / v for 2^-1000 < |v| < 2^1000.  The approximation takes and gives 20
// mantissa bits, so 1 - v x is below 2^-18; a step squares it, so after the
// second the truncation is below 2^-72 and the error that of the last rounding:
// half an ulp and 2^-19 of one, as the correctly rounded division's but for
// quotients that lie that close to a tie.
__device__ __forceinline__ double recip_f64(double v) {
  double x;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(v));
  x = fma(x, fma(-v, x, 1.0), x);
  return fma(x, fma(-v, x, 1.0), x);
}
// finite: the exponent bits are not all ones (an integer test: an FP64
// compare would take an FP64 slot)
__device__ __forceinline__ bool finite_f64(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

__device__ __forceinline__ void collide_f64(double (&f)[9], double (&g)[9], double Ex, double Ey, double mub,
                                            const CollideF64& k, bool& bad) {
  constexpr double third = -1.0 / 3.0;
  // fluid
  const double s1 = f[1] + f[3], s2 = f[2] + f[4], s5 = f[5] + f[7], s6 = f[6] + f[8];
  const double d1 = f[1] - f[3], d2 = f[2] - f[4], d5 = f[5] - f[7], d6 = f[6] - f[8];
  const double rho = ((s1 + s2) + (s5 + s6)) + f[0];
  const double jx = d1 + (d5 - d6), jy = d2 + (d5 + d6);
  // charge
  const double p1 = g[1] + g[3], p2 = g[2] + g[4], p5 = g[5] + g[7], p6 = g[6] + g[8];
  const double e1 = g[1] - g[3], e2 = g[2] - g[4], e5 = g[5] - g[7], e6 = g[6] - g[8];
  const double rc = ((p1 + p2) + (p5 + p6)) + g[0];
  bad = !finite_f64(rho) || !finite_f64(rc);
  const double Fx = rc * Ex, Fy = rc * Ey;
  const double irho = recip_f64(rho);
  const double ux = fma(0.5, Fx, jx) * irho, uy = fma(0.5, Fy, jy) * irho;
  {
    const double Gx = fma(k.gj, jx, k.gF * Fx), Gy = fma(k.gj, jy, k.gF * Fy);
    const double Q = fma(uy, Gy, ux * Gx), X = fma(ux, Gy, uy * Gx);
    const double C = fma(third, Q, k.rw * rho), t = 0.25 * (C + Q);
    const double P1 = fma(k.hp, s1, fma(ux, Gx, C)), P2 = fma(k.hp, s2, fma(uy, Gy, C));
    const double P5 = fma(k.hp, s5, fma(0.25, X, t)), P6 = fma(k.hp, s6, fma(-0.25, X, t));
    const double Jx = fma(k.jj, jx, k.jF * Fx), Jy = fma(k.jj, jy, k.jF * Fy);
    const double D1 = fma(k.hm, d1, Jx), D2 = fma(k.hm, d2, Jy);
    const double q = 0.25 * Jy;
    const double D5 = fma(k.hm, d5, fma(0.25, Jx, q)), D6 = fma(k.hm, d6, fma(-0.25, Jx, q));
    f[0] = fma(-2.0, (P1 + P2) + (P5 + P6), rho);
    f[1] = P1 + D1;
    f[3] = P1 - D1;
    f[2] = P2 + D2;
    f[4] = P2 - D2;
    f[5] = P5 + D5;
    f[7] = P5 - D5;
    f[6] = P6 + D6;
    f[8] = P6 - D6;
  }
  {
    const double vx = fma(mub, Ex, ux), vy = fma(mub, Ey, uy);
    const double h = k.gg * rc, Gx = h * vx, Gy = h * vy, X = vx * Gy;  // v_x G_y = v_y G_x
    const double Q = fma(vy, Gy, vx * Gx);
    const double C = fma(third, Q, k.grw * rc), t = 0.25 * (C + Q);
    const double P1 = fma(k.ghp, p1, fma(vx, Gx, C)), P2 = fma(k.ghp, p2, fma(vy, Gy, C));
    const double P5 = fma(k.ghp, p5, fma(0.5, X, t)), P6 = fma(k.ghp, p6, fma(-0.5, X, t));
    const double m = k.gjm * rc, Jx = m * vx, Jy = m * vy;
    const double D1 = fma(k.ghm, e1, Jx), D2 = fma(k.ghm, e2, Jy);
    const double q = 0.25 * Jy;
    const double D5 = fma(k.ghm, e5, fma(0.25, Jx, q)), D6 = fma(k.ghm, e6, fma(-0.25, Jx, q));
    g[0] = fma(-2.0, (P1 + P2) + (P5 + P6), rc);
    g[1] = P1 + D1;
    g[3] = P1 - D1;
    g[2] = P2 + D2;
    g[4] = P2 - D2;
    g[5] = P5 + D5;
    g[7] = P5 - D5;
    g[6] = P6 + D6;
    g[8] = P6 - D6;
  }
}

struct PoissonArgs {
  int Nx, Ny, P, Mh, log2Nx;
  int Mp;                    // row pitch of the spectrum and pivot tables (Mh rounded up to 4)
  const void* rhoc;          // charge density, R [Ny][P]
  const void* g;             // charge populations that the forward transform sums (rhoc then unused), or nullptr
  long long gplane;          // elements per plane of g
  int gstorage;              // FP32 compute after k_push: g's storage type, and its shift
  const float* rch;
  const float* flux_lo;      // wall rows' charge populations of k_push, [6][P] each
  const float* flux_hi;
  double* flux_strip;        // the strips' wall fluxes formed from them: flux_part
  const void* rhoc_dn;       // slab-boundary partials of the march form (see StepArgs), added to rhoc
  const void* rhoc_up;
  int xslab;                 // slab height of those partials; 0: rhoc is complete
  int xoff;                  // slab_off of the step kernel that wrote them
  double inv_eps;            // 1 / eps
  void* spec;                // half spectrum, complex R [Ny][Mp]
  void* spec0;               // row sums (m = 0), [Ny]: double, or float (hi, lo) pairs when R = float
  const void* rfac;          // reciprocal pivots, R [Ny][Mp] (m >= 1 used)
  const void* rfac0;         // reciprocal pivots of m = 0, [Ny]: double, or float (hi, lo) pairs
  const void* tw;            // complex R [Nx]: exp(-2 pi i q / Nx)
  void* dphi;                // R [Ny][P]
  void* phibar;              // row-mean potential [Ny]: double, or float (hi, lo) pairs when R = float
  void* Ebar;                // R [Ny]
  double phi0;               // injector potential (collector is 0)
  // mean-mode (m = 0) constants, formed on the host: the injector wall value
  // W = Nx phi0 in spectral units and the closure factor 1 / (2 Ny) (walls
  // halfway) or 1 / (Ny + 1) (walls on nodes); in FP64 and split into
  // float-float (hi, lo) pairs, hi = fl32(v), lo = fl32(v - hi)
  double mW, mC;
  float mWf[2], mCf[2];
  int wall_mode;
  const double* flux_part;   // [2][nflux] wall-flux partials of the last step, or nullptr
  int nflux;
  double* flux_acc;          // [2] FP64 totals of injected / collected charge
  int tile_modes;            // wavenumbers per CTA of the mode solve (8, 4, 2, 1; 0 = largest that fits)
  int tile_threads;          // threads per CTA of the mode solve (FP32: 256, 512, 1024; 0 = 256)
  int tile_cluster;          // FP32, 8 wavenumbers per tile: two-CTA clusters per tile (same bits)
  int tile_tma;              // FP32, 8 wavenumbers per tile: tiles staged by tensor copies (same bits)
  const struct ModesTma* mtma;  // host pointer to the run's tensor maps of spec and rfac (or nullptr)
  int* err;                  // device error word (bit 2: a bounded wait gave up)
  int pdl;                   // programmatic dependent launch, a mask: 1 forward transform, 2 wavenumber
                             // solve, 4 inverse transform
  int fft_cta;               // rows of 2048: one CTA of 64 threads per row (else one warp per row)
  // y solve of the wavenumbers m >= 1: 0 per-wavenumber tridiagonal (k_modes_tile),
  // 1 odd-extension transform of length NE (k_modes_oddext, Eqs. 21-25)
  int y_solver;
  int NE, nfac;              // odd-extension length, number of its radices
  int fac[16];               // radices of NE in stage order
  const void* twy;           // complex R [NE]: exp(-2 pi i t / NE)
  const void* symy;          // R [NE]: 4 sin^2(pi k / NE)
  const void* kap;           // R [Mh]: kappa_m, the x symbol of wavenumber m
  void* ex;                  // R [Ny][P]: spectral E_x written after phi, or nullptr
};

// Charge density of row y as the Poisson solve sees it: the step kernel's
// march form leaves, at each slab boundary, the populations that cross it to
// the slab that computed them, together with their share of the new charge
// density (rhoc_dn for the row below the boundary, rhoc_up for the row
// above).  The readers add main + dn + up, in this order.
template <class R>
__device__ __forceinline__ void rhoc_partials(const PoissonArgs& a, int y, const R*& dn, const R*& up) {
  dn = nullptr;
  up = nullptr;
  if (a.xslab > 0) {
    // slab b starts at row b S - off (b >= 1): row y closes a slab when
    // y + 1 + off is a multiple of S and opens one when y + off is
    const int S = a.xslab, yd = y + 1 + a.xoff, yu = y + a.xoff;
    if (yd % S == 0 && y + 1 < a.Ny) dn = static_cast<const R*>(a.rhoc_dn) + (long long)(yd / S) * a.P;
    if (yu % S == 0 && y > 0) up = static_cast<const R*>(a.rhoc_up) + (long long)(yu / S) * a.P;
  }
}

struct FieldArgs {
  int Nx, Ny, P;
  long long plane;
  const void* f;
  const void* g;
  const void* dphi;
  const void* phibar;        // double, or float (hi, lo) pairs when R = float
  const void* Ebar;
  const float* rch;
  const void* ex;            // R [Ny][P]: spectral E_x, or nullptr
  double fb, fd;             // f shift r(y) = fb + fd y
  double mub;
  int wall_mode;
  const double* base_g;      // perturbation form: [9][Ny] base g added to the stored departures (else nullptr)
  const double* phiB;        // [Ny] base potential and field added to the departure's
  const double* EB;
};

// Row-mean potential as stored: a double, or a float-float (hi, lo) pair on
// the FP32 path (kept off the slow scalar FP64 units during the step).
template <class R>
__device__ __forceinline__ double load_phibar(const void* p, int j) {
  if constexpr (sizeof(R) == 8) {
    return static_cast<const double*>(p)[j];
  } else {
    const float2 v = static_cast<const float2*>(p)[j];
    return (double)v.x + (double)v.y;
  }
}

// ------------------------------------------------ perturbation form ---
// FP32-compute runs may advance the charge populations as departures from an
// x-uniform base state that is advanced exactly, in FP64: g = B_g(y, t) + d.
// The base (both population sets, [9][Ny] FP64 each) follows the method's
// own dynamics restricted to x-uniform fields -- collision, streaming in y,
// the wall rules and the mean mode of the Poisson equation -- so the
// departure d carries only what varies in x (a roll and its consequences)
// and its FP32 arithmetic is relative to that.  The step kernel needs, per
// row, the base charge, the base fluid velocity u_y and the base field E_y:
// the march table, FP32 [Ny][4] = {rho_c, u_y, E_y, 0}.
struct BaseArgs {
  int Nx, Ny;
  const double* fin;   // [9][Ny] base f at time t
  const double* gin;   // [9][Ny] base g at time t
  double* fout;        // [9][Ny] at t + 1
  double* gout;
  const double* EB;    // [Ny] base E_y at time t
  const double* mom;   // [7][Ny] rho_c, rho, u_x, u_y, u_y + mu_b E_y, j_x, j_y at time t
  double wp, gwp, mub, rho0;
  double rhs_scale;    // -Nx / eps
  CollideF64 k64;
  double* flux_acc;    // [2] FP64 totals of the base's injected / collected charge
  double* sums;        // [4][Ny] rho_c, rho, j_y, j_x of the state at t + 1 (out)
  double* rhs;         // [Ny] its mean-mode right-hand side -Nx rho_c / eps (out)
  double* loc;         // [2][Ny] chunk-local prefix sums of rhs (out)
  double* chunk;       // [2][base_chunks(Ny)] chunk totals (out)
};
struct BasePoissonArgs {
  int Nx, Ny, wall_mode;
  double W, closure, inN;  // Nx phi0, 1 / (2 Ny) (walls halfway) or 1 / (Ny + 1), 1 / Nx
  double mub;
  const double* rhs;   // [Ny] mean-mode right-hand side of the state
  const double* sums;  // [4][Ny] its rho_c, rho, j_y, j_x
  const double* loc;   // [2][Ny] and the chunk sums of the right-hand side
  const double* chunk;
  double* phiB;        // [Ny] base potential (out)
  double* EB;          // [Ny] base E_y (out)
  float* table;        // [Ny][4] march table (out)
  double* mom;         // [7][Ny] moments for the state's base step (out)
};
// rows per chunk of the base kernels: chunks of a run's base state
int base_chunks(int Ny);
cudaError_t launch_base_step(const BaseArgs& a, cudaStream_t s);
// row sums and right-hand side of the state fin / gin (fout, gout unused)
cudaError_t launch_base_sums(const BaseArgs& a, cudaStream_t s);
cudaError_t launch_base_poisson(const BasePoissonArgs& a, cudaStream_t s);

// ------------------------------------------------------------- batches ---
// A batch advances many runs (FP32 storage and compute, march form) together:
// each phase of the step is one persistent kernel over a work list that
// covers every member run; the lists live in device memory, so membership
// changes need no new launch configuration.
struct BatchRunDesc {
  StepArgs sa[2];    // [p]: step from buffer p to 1 - p
  PoissonArgs pa;    // Poisson solve of the run (with its wall fluxes)
  BaseArgs ba[2];    // perturbation form: the base step from buffer p (ba[p].fin == nullptr otherwise)
  BasePoissonArgs bp[2];  // and the potential of its result (bp[p].sums == nullptr otherwise)
  int cur0;          // buffer holding the state at the start of the tick
  int remaining;     // steps the run still takes in this tick
  int E;             // Nx / 64: warp-FFT shape
  int pad;
};
struct BatchTables {
  const BatchRunDesc* runs;
  const int4* march_items;  // (run, strip, slab, 0)
  const int2* row_items;    // (run, rows: row_item)
  const int2* tile_items;   // (run, first wavenumber)
  const int* counts;        // device: [0] runs, [1] march items, [2] rows, [3] tiles
  int* work;                // device: [0] march items and [1] y solves taken from the step's counters (each
                            // zeroed, for the next step, by the transform that follows its phase)
  int mean_in_modes;        // the mean modes are items of the wavenumber kernel (all runs of at most 1024 rows)
  int modes_smem;           // tile bytes for the largest admissible Ny (fixed per batch)
  int pdl;                  // programmatic dependent launch: 1 forward transforms, 2 tiles, 4 inverse
  int emax;                 // largest admissible Nx / 64: the widest warp-FFT shape compiled in
};

// Rows of a row-transform item: first row and how many (Ny <= 4096).
__host__ __device__ __forceinline__ int row_item(int y, int count) { return y | (count << 16); }
__device__ __forceinline__ int row_item_row(int v) { return v & 0xffff; }
__device__ __forceinline__ int row_item_count(int v) { return v >> 16; }

// Dynamic scheduling of a batch phase's items (largest first in the lists):
// one lane or thread takes the next index from the phase's counter.
__device__ __forceinline__ int next_item_warp(int* counter) {
  int it = 0;
  if ((threadIdx.x & 31) == 0) it = atomicAdd(counter, 1);
  return __shfl_sync(0xffffffffu, it, 0);
}
// one launch of each phase for step t (0-based) of a tick
// pert: the graph has perturbation-form members (the march branches per run)
cudaError_t launch_batch_march(const BatchTables& t, int step, int grid, bool pert, cudaStream_t s);
cudaError_t launch_batch_rfft(const BatchTables& t, int step, int grid, cudaStream_t s);
cudaError_t launch_batch_irfft(const BatchTables& t, int step, int grid, cudaStream_t s);
cudaError_t launch_batch_modes(const BatchTables& t, int step, int grid, cudaStream_t s);
cudaError_t launch_batch_mean(const BatchTables& t, int step, int grid, cudaStream_t s);
// wavenumber-tile CTAs of the batch that fit one SM with `smem` bytes of tile
int batch_modes_ctas_per_sm(int smem);
// perturbation-form members: the FP64 base step and its potential
cudaError_t launch_batch_base(const BatchTables& t, int step, int max_runs, int max_ny, cudaStream_t s);
constexpr int kBatchTileModes = 8;
// From here an SM holds one tile of the wavenumber solve and no longer two (96
// bytes a row and 5 KB of scratch), and launching the solve ahead of its
// predecessor's end starts to pay for rows of 1024 (measured on both sides of
// the line: see default_pdl).
constexpr int kTallRows = 1140;



// Tensor maps of the TMA form of the march kernel (FP32 storage and compute,
// Nx >= 128): the pre-collision populations as 3-D tensors {Nx, Ny, 9}
// loaded in boxes of {68, 1, 9} (a strip's 64 columns and the 4-column
// alignment margin, every plane of one row), the potential fluctuation
// {Nx, Ny} in boxes of {68, 1}, and the post-collision populations stored in
// boxes of {60, 1, 9} (a strip's owned columns).  One set per buffer parity.
constexpr int kTmaLoadCols = 68;
constexpr int kTmaStoreCols = 60;
struct MarchTma {
  CUtensorMap f, g, dphi, fo, go;
};
// Encode the maps of a run (f[cur], g[cur] in, f[1-cur], g[1-cur] out).
cudaError_t march_tma_encode(MarchTma* m, const void* fin, const void* gin, const void* dphi, void* fout, void* gout,
                             int Nx, int Ny, int P);
bool march_tma_supported(int Nx);
cudaError_t launch_march_tma(const StepArgs& a, const MarchTma& m, int form, cudaStream_t s);

// Launchers (defined in the .cu files); storage: 0 F64, 1 F32, 2 BF16, 3 F16;
// real_f64: compute type (true = double).
cudaError_t launch_step(const StepArgs& a, int storage, bool real_f64, int rows_per_cta, cudaStream_t s);
int step_flux_blocks(int Nx, bool real_f64);
cudaError_t launch_march(const StepArgs& a, int storage, bool real_f64, cudaStream_t s);
int march_strips(int Nx, int cols_per_lane);
int march_warps_per_sm(int storage, bool real_f64, int cols_per_lane, int ring_depth);
// attributes of all march kernels, on the current device
cudaError_t march_set_attributes();
// Poisson solve from the charge plane (or, with a.g, from the populations):
// forward row FFTs, wavenumber systems and inverse FFTs on s.  The mean mode and
// the wall-flux totals are in the launch of the wavenumber systems (FP64) or of
// the inverse FFTs (FP32 rows of 64 to 1024, up to 1024 rows); otherwise a kernel
// of their own, on `side` between the fork and join events when side != nullptr.
cudaError_t launch_poisson(const PoissonArgs& a, bool real_f64, cudaStream_t s, cudaStream_t side, cudaEvent_t fork,
                           cudaEvent_t join, const cudaEvent_t* marks = nullptr);
// row transforms of the FP64 path (k_fft64.cu); the spectrum they keep is S / Nx
cudaError_t launch_rfft64(const PoissonArgs& a, cudaStream_t s);
cudaError_t launch_irfft64(const PoissonArgs& a, bool dx, cudaStream_t s);
// Odd-extension y solve (k_oddext.cu): radices of n (4, 2, 3, 5, 7, 11, 13;
// at most cap of them) into fac, their count, or -1 if n has another factor;
// the shared memory one CTA needs; the launch over m = 1 .. Mh - 1.
int oddext_factors(int n, int* fac, int cap);
size_t oddext_smem_bytes(int NE, bool real_f64);
cudaError_t launch_modes_oddext(const PoissonArgs& a, bool real_f64, cudaStream_t s);
cudaError_t oddext_set_attributes();
// One node per thread (k_push.cu): FP32-compute runs without a base state;
// the wall rows' charge populations go to rhoc_dn and rhoc_up
cudaError_t launch_push(const StepArgs& a, int storage, int log2Nx, cudaStream_t s);
// Many steps of a small FP32 run in one launch with its state on chip
// (k_resident.cu): whether the size fits a cluster of this GPU (also sets the
// kernel's attributes), and `steps` steps from a.fin / a.gin back into them.
bool resident_supported(int Nx, int Ny, int storage);
cudaError_t launch_resident(const StepArgs& a, const PoissonArgs& pa, int storage, int steps, cudaStream_t s);
// rho_c = sum_i g_i (+ the row shift) into the charge plane (FP32 compute).
cudaError_t launch_rhoc(const void* g, long long plane, int storage, int Nx, int Ny, int P,
                        const float* rch, void* rhoc, cudaStream_t s);
cudaError_t poisson_set_attributes();
// warp-per-row real FFTs (FP32 path, Nx = 64 ... 2048)
bool fftw_supported(int Nx);
cudaError_t launch_rfft_warp(const PoissonArgs& a, cudaStream_t s);
cudaError_t launch_irfft_warp(const PoissonArgs& a, cudaStream_t s);
// the forward transform after k_push (rows of 64 to 1024)
cudaError_t launch_rfft_push(const PoissonArgs& a, cudaStream_t s);
// the inverse transform and, beside it and the wavenumber solve, the mean mode
bool irfft_mean_supported(int Nx, int Ny);
cudaError_t launch_irfft_mean(const PoissonArgs& a, cudaStream_t s);
// The same transform of -i k_m phi_m (spectral E_x) into a.ex.
cudaError_t launch_irfft_warp_dx(const PoissonArgs& a, cudaStream_t s);
cudaError_t launch_fields(const FieldArgs& a, int storage, bool real_f64, unsigned mask, double* out,
                          cudaStream_t s);
cudaError_t launch_reduce_state(const FieldArgs& a, int storage, bool real_f64, double* part, int nblk,
                                double* out, int* err, cudaStream_t s);
int reduce_state_blocks();
// shift per row: shift_w (rch[y] + c0 + c1 y) + (brow ? brow[y] : 0)
cudaError_t launch_load_plane(const double* src, void* dst, int storage, int Nx, int Ny, int P, double shift_w,
                              const float* rch, double c0, double c1, const double* brow, cudaStream_t s);
cudaError_t launch_save_plane(const void* src, double* dst, int storage, int Nx, int Ny, int P, double shift_w,
                              const float* rch, double c0, double c1, const double* brow, cudaStream_t s);
// base_g (perturbation form): [9][Ny] subtracted from g instead of w_i rch[y]
cudaError_t launch_init(const double* rho_h, const double* rc_h, const double* Eh, const double* sY,
                        const double* cY, const double* Sx, const double* Cy, double Fh, double mub,
                        void* f, void* g, int storage, int Nx, int Ny, int P, const float* rch, double fb,
                        double fd, const double* base_g, cudaStream_t s);

}  // namespace ehd
