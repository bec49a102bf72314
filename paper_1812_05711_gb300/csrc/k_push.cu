// k_push.cu -- the collide-and-stream kernel of small and medium FP32-compute
// runs: one node per thread.
//
// The march form (k_march.cu) moves the fewest bytes, with one warp walking
// four rows or more of a strip; a run whose populations live in L2 has no use
// for that, and its step waited for the walk: 256 x 205 gave it 260 warps on
// 152 SMs, each with five L2 round trips and row collisions one after another
// (6.9 us).  Here every node is its own thread -- one round trip, one
// collision -- and pushes its post-collision populations to their nodes.  The
// charge density is left to the forward transform, which sums the nine
// populations of a node as it loads them (k_rfft_push), in the order and with
// the slab boundaries of the march form, so a run's results are the same bit
// for bit in either form and in a batch.  The two wall rows' six charge
// populations go to two small planes that the flux totals are formed from.
#include "march_dev.cuh"

namespace ehd {

template <class S>
__global__ void __launch_bounds__(128) k_push(StepArgs a, int log2Nx) {
  using R = float;
  grid_dep_launch();  // the forward transform waits for this whole grid before it reads
  const int Nx = a.Nx, Ny = a.Ny, P = a.P;
  const int n = blockIdx.x * 128 + threadIdx.x;
  const int y = n >> log2Nx, x = n & (Nx - 1);
  if (y >= Ny) return;  // whole warps: a row is 64 nodes or more
  const long long pl = a.plane, c = (long long)y * P + x;
  const S* __restrict__ fin = static_cast<const S*>(a.fin) + c;
  const S* __restrict__ gin = static_cast<const S*>(a.gin) + c;
  R f[9], g[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    f[i] = Store<S>::template ld<R>(fin + i * pl);
    g[i] = Store<S>::template ld<R>(gin + i * pl);
  }
  const R sy = (R)__ldg(a.rch + y);
  const R s_up = (y + 1 < Ny) ? (R)__ldg(a.rch + y + 1) : sy;
  const R s_dn = (y > 0) ? (R)__ldg(a.rch + y - 1) : sy;
  grid_dep_wait();  // the populations are the step's before; the potential's kernels end here
  const int xl = (x - 1) & (Nx - 1), xr = (x + 1) & (Nx - 1);
  const R* ph = static_cast<const R*>(a.dphi) + (long long)y * P;
  const R gwall = (a.wall_mode == 0) ? R(-1) : R(0);
  const R pc = ph[x];
  const R pm = (y > 0) ? ph[x - P] : gwall * pc;
  const R pn = (y + 1 < Ny) ? ph[x + P] : gwall * pc;
  const R Ex = R(-0.5) * (ph[xr] - ph[xl]);
  const R Ey = static_cast<const R*>(a.Ebar)[y] - R(0.5) * (pn - pm);
  const R wp = (R)a.wp, wm = (R)a.wm, gwp = (R)a.gwp, gwm = (R)a.gwm;
  const R cp = R(1) - R(0.5) * wp, cm = R(1) - R(0.5) * wm;
  const R mub = (R)a.mub, rho0 = (R)a.rho0;
  const R W1 = (R)kW1, W2 = (R)kW2;
  const R fb = (R)a.fb, fd = (R)a.fd, fdq = (R)a.fdq;
  const R wd1 = W1 * fd, wd2 = W2 * fd;
  const R sf = fb + fd * (R)y;
  bool bad;
  collide_node<S, R>(f, g, Ex, Ey, sy, sf, fdq, mub, wp, wm, cp, cm, gwp, gwm, bad);
  if (bad) atomicOr(a.err, 1);
  S* __restrict__ fo = static_cast<S*>(a.fout) + (long long)y * P;
  S* __restrict__ go = static_cast<S*>(a.gout) + (long long)y * P;
  auto put = [](S* p, R v) { Store<S>::st(p, v); };
  auto rt = [](R v) { return Store<S>::template rt<R>(v); };
  put(fo + x, f[0]);
  put(go + x, g[0]);
  put(fo + pl + xr, f[1]);
  put(go + pl + xr, g[1]);
  put(fo + 3 * pl + xl, f[3]);
  put(go + 3 * pl + xl, g[3]);
  // c_y = +1
  if (y + 1 < Ny) {
    const R sh = sy - s_up;
    S *u = fo + P, *v = go + P;
    put(u + 2 * pl + x, f[2]);
    put(u + 5 * pl + xr, f[5]);
    put(u + 6 * pl + xl, f[6]);
    put(v + 2 * pl + x, g[2] + W1 * sh);
    put(v + 5 * pl + xr, g[5] + W2 * sh);
    put(v + 6 * pl + xl, g[6] + W2 * sh);
  } else {
    // collector: f bounces back; g leaves and re-enters from its own row
    put(fo + 4 * pl + x, f[2] + wd1);
    put(fo + 7 * pl + x, f[5] + wd2);
    put(fo + 8 * pl + x, f[6] + wd2);
    put(go + 4 * pl + x, g[4]);
    put(go + 7 * pl + xl, g[7]);
    put(go + 8 * pl + xr, g[8]);
    R* w = static_cast<R*>(a.rhoc_up) + x;
    w[0] = rt(g[2]);
    w[P] = rt(g[5]);
    w[2 * P] = rt(g[6]);
    w[3 * P] = rt(g[4]);
    w[4 * P] = rt(g[7]);
    w[5 * P] = rt(g[8]);
  }
  // c_y = -1
  if (y > 0) {
    const R sh = sy - s_dn;
    S *d = fo - P, *e = go - P;
    put(d + 4 * pl + x, f[4]);
    put(d + 7 * pl + xl, f[7]);
    put(d + 8 * pl + xr, f[8]);
    put(e + 4 * pl + x, g[4] + W1 * sh);
    put(e + 7 * pl + xl, g[7] + W2 * sh);
    put(e + 8 * pl + xr, g[8] + W2 * sh);
  } else {
    // injector: bounce-back of f, anti-bounce-back of g
    R n2, n5, n6;
    inject<R>(g[4], g[7], g[8], Ex, Ey, sy, mub, rho0, n2, n5, n6);
    put(fo + 2 * pl + x, f[4] - wd1);
    put(fo + 5 * pl + x, f[7] - wd2);
    put(fo + 6 * pl + x, f[8] - wd2);
    put(go + 2 * pl + x, n2);
    put(go + 5 * pl + x, n5);
    put(go + 6 * pl + x, n6);
    R* w = static_cast<R*>(a.rhoc_dn) + x;
    w[0] = rt(n2);
    w[P] = rt(n5);
    w[2 * P] = rt(n6);
    w[3 * P] = rt(g[4]);
    w[4 * P] = rt(g[7]);
    w[5 * P] = rt(g[8]);
  }
}

cudaError_t launch_push(const StepArgs& a, int storage, int log2Nx, cudaStream_t s) {
  const dim3 grid((unsigned)(((long long)a.Nx * a.Ny + 127) / 128)), block(128);
  const bool pdl = (a.pdl & 8) != 0;
  switch (storage) {
    case 0: return launch_ex(pdl, k_push<double>, grid, block, 0, s, a, log2Nx);
    case 1: return launch_ex(pdl, k_push<float>, grid, block, 0, s, a, log2Nx);
    case 2: return launch_ex(pdl, k_push<__nv_bfloat16>, grid, block, 0, s, a, log2Nx);
    case 3: return launch_ex(pdl, k_push<__half>, grid, block, 0, s, a, log2Nx);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ehd
