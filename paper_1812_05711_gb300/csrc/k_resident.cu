// k_resident.cu -- many coupled steps of a small FP32 run in one launch, the
// whole state on chip.
//
// A small channel's step moves next to nothing (128 x 104: 2 MB, 0.3 us at
// the copy bandwidth) but took 14.5 us as four kernels: each is a launch, a
// chain of L2 round trips and a few hundred dependent instructions on a part
// of the SMs.  Here one cluster of 16 CTAs (one GPC) holds the run's
// populations, potential and spectrum in shared memory; a CTA owns a band of
// rows, and what crosses bands -- populations streaming up or down, the
// spectrum's columns on their way to the wavenumber solves and back, the
// potential rows next to a band -- is written straight into the owner's
// shared memory.  A step is four phases, each ended by a hardware cluster
// barrier:
//   march     one node per thread: E, moments, collisions (collide_node), the
//             post-collision populations pushed to their nodes; wall rules
//   forward   a warp per row: charge density, LaneFft, each wavenumber's value
//             to the CTA that solves it
//   solve     a warp per wavenumber: the two sweeps as scans over 32 chunks of
//             rows (one chunk per lane, its rows in registers); the mean mode
//             by four warps of one CTA, which has until the end of the next
//             phase, since only the march reads its result
//   inverse   a warp per row -> potential, its band's edge rows to both
//             neighbours
// Every value is formed as the multi-kernel step forms it (same chunking, same
// order of sums, slab boundaries included, by the functions of march_dev.cuh,
// fft_dev.cuh and sweep_dev.cuh, whose rounding is stated), so the results are
// the same bit for bit; FP64 wall fluxes are summed by spare warps of the two wall CTAs.
//
// Why 16 CTAs: the march needs the SMs (13 K nodes x 260 instructions), and
// two copies of the populations (36 floats a node) must fit beside the rest;
// a cluster spans at most one GPC.  Larger runs keep the multi-kernel step,
// which has all SMs.
#include "cluster_dev.cuh"
#include "fft_dev.cuh"
#include "march_dev.cuh"
#include "mean_dev.cuh"
#include "sweep_dev.cuh"

namespace ehd {

namespace {

constexpr int kThreads = 512;
constexpr int kRowWarps = 8;    // a CTA owns at most 8 rows
constexpr int kMaxRows = kClusterCtas * kRowWarps;
constexpr int kChunkRows = 4;   // rows per lane in the wavenumber solve (Ny <= 128)
constexpr int kMeanCta = 8;     // neither wall's CTA
constexpr int kMeanWarp = 8;    // its first warp of the mean mode (four of them)
constexpr int kFluxWarp = 8;    // first flux warp of the wall CTAs, one per 60-column strip

// four populations of the storage type, as floats (see Store)
template <class S>
struct Four;
template <>
struct Four<float> {
  __device__ static float4 ld(const float* p) { return *reinterpret_cast<const float4*>(p); }
  __device__ static void st(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
};
template <>
struct Four<__nv_bfloat16> {
  __device__ static float4 ld(const __nv_bfloat16* p) {
    const __nv_bfloat162* q = reinterpret_cast<const __nv_bfloat162*>(p);
    const float2 a = __bfloat1622float2(q[0]), b = __bfloat1622float2(q[1]);
    return make_float4(a.x, a.y, b.x, b.y);
  }
  __device__ static void st(__nv_bfloat16* p, float4 v) {
    __nv_bfloat162* q = reinterpret_cast<__nv_bfloat162*>(p);
    q[0] = __floats2bfloat162_rn(v.x, v.y);
    q[1] = __floats2bfloat162_rn(v.z, v.w);
  }
};
template <>
struct Four<__half> {
  __device__ static float4 ld(const __half* p) {
    const __half2* q = reinterpret_cast<const __half2*>(p);
    const float2 a = __half22float2(q[0]), b = __half22float2(q[1]);
    return make_float4(a.x * kHalfUnscale, a.y * kHalfUnscale, b.x * kHalfUnscale, b.y * kHalfUnscale);
  }
  __device__ static void st(__half* p, float4 v) {
    __half2* q = reinterpret_cast<__half2*>(p);
    q[0] = __floats2half2_rn(v.x * kHalfScale, v.y * kHalfScale);
    q[1] = __floats2half2_rn(v.z * kHalfScale, v.w * kHalfScale);
  }
};

// Shared memory of a CTA (floats from its start), RM rows at most per band.
template <int E>
struct Layout {
  static constexpr int Nx = 64 * E, L = 32 * E;
  static constexpr int kModes = L / kClusterCtas;  // wavenumbers per CTA: m = rank kModes + 1 ...
  static constexpr int kSpecRow = 2 * (L + 2);
  static constexpr int kStrips = (Nx + 59) / 60;
  int pop, phi, spec, col, col_row, row, mean, ebar, shift, flux, total;
  __host__ __device__ Layout(int RM, int Ny) {
    auto up = [](int v) { return (v + 3) & ~3; };
    pop = 0;
    phi = pop + 2 * 18 * RM * Nx;
    spec = phi + (RM + 2) * Nx;
    col = up(spec + RM * kSpecRow);
    col_row = 2 * (Ny + 1);
    row = up(col + kModes * col_row);
    mean = row + kRowWarps * 2 * kLaneRow<E>;
    ebar = up(mean + 4 * Ny);
    shift = ebar + up(RM);
    flux = shift + up(RM + 2);
    total = flux + 2 * 6 * Nx;
  }
};

}  // namespace

template <class S, int E>
__global__ void __launch_bounds__(kThreads, 1) k_resident(StepArgs a, PoissonArgs pa, int steps, int RM) {
  using Lay = Layout<E>;
  constexpr int Nx = Lay::Nx, L = Lay::L, ML = Lay::kModes;
  extern __shared__ __align__(16) float sm[];
  __shared__ MeanScratch<float, kMeanThreadsSmall> ms;
  __shared__ double fpart[Lay::kStrips];
  const Lay lay(RM, a.Ny);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int Ny = a.Ny, P = a.P, slab = a.slab_rows;
  int rank;
  asm("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(rank));
  const int r0 = band_start(rank, Ny), nr = band_start(rank + 1, Ny) - r0;
  const int RN = RM * Nx;
  float* const phi = sm + lay.phi;  // row ly at (ly + 1) Nx, the rows beside the band at 0 and (nr + 1) Nx
  float2* const spec = reinterpret_cast<float2*>(sm + lay.spec);
  float2* const col = reinterpret_cast<float2*>(sm + lay.col);
  float2* const rowbuf = reinterpret_cast<float2*>(sm + lay.row) + (warp & 7) * kLaneRow<E>;
  ff* const mean_v = reinterpret_cast<ff*>(sm + lay.mean);
  float* const ebar = sm + lay.ebar;
  float* const shift = sm + lay.shift;  // shift of row r0 - 1 + k at k (the wall rows' own where there is no neighbour)

  // ---- the run's state into shared memory
  for (int i = 0; i < 18; ++i) {
    const S* src = static_cast<const S*>(i < 9 ? a.fin : a.gin) + (i % 9) * a.plane + (long long)r0 * P;
    for (int k = 4 * tid; k < nr * Nx; k += 4 * kThreads)  // P == Nx
      *reinterpret_cast<float4*>(sm + lay.pop + i * RN + k) = Four<S>::ld(src + k);
  }
  for (int k = tid; k < (nr + 2) * Nx; k += kThreads) {
    const int y = r0 - 1 + k / Nx;
    if (y >= 0 && y < Ny) phi[k] = static_cast<const float*>(a.dphi)[(long long)y * P + (k & (Nx - 1))];
  }
  if (tid < nr) ebar[tid] = static_cast<const float*>(a.Ebar)[r0 + tid];
  if (tid < nr + 2) shift[tid] = a.rch[min(max(r0 - 1 + tid, 0), Ny - 1)];

  // ---- constants of the warps' roles
  const float2* __restrict__ tw = static_cast<const float2*>(pa.tw);
  LaneFft<E> fft;
  float2 wkf[E], wki[E];
  fft.init(tw, lane);
  untangle_factors<E>(tw, lane, wkf);
#pragma unroll
  for (int n2 = 0; n2 < E; ++n2) wki[n2] = cmf1(tw[lane], tw[32 * n2]);
  // wavenumber solve: lane = chunk of C rows, reciprocal pivots in registers
  const int C = (Ny + 31) / 32, j0 = min(lane * C, Ny), nj = min(j0 + C, Ny) - j0;
  const int mode = rank * ML + warp + 1;
  float piv[kChunkRows];
  unsigned home[kChunkRows];  // where the solved value of row j0 + q goes
#pragma unroll
  for (int q = 0; q < kChunkRows; ++q) {
    piv[q] = 0.0f;
    home[q] = 0;
    if (warp < ML && q < nj) {
      const int j = j0 + q, o = band_owner(j, Ny);
      piv[q] = static_cast<const float*>(pa.rfac)[(long long)j * pa.Mp + mode];
      home[q] = peer_addr(spec + (j - band_start(o, Ny)) * (Lay::kSpecRow / 2) + mode, o);
    }
  }
  // forward transform: where wavenumber lane + 32 q (and the Nyquist one) of this warp's row goes
  const int myrow = r0 + warp;
  unsigned to_col[E], to_nyq = 0;
#pragma unroll
  for (int q = 0; q < E; ++q) {
    const int m = lane + 32 * q - 1;
    to_col[q] = (m >= 0 && warp < nr) ? peer_addr(col + (m % ML) * (lay.col_row / 2) + myrow, m / ML) : 0u;
  }
  if (warp < nr) to_nyq = peer_addr(col + (ML - 1) * (lay.col_row / 2) + myrow, kClusterCtas - 1);
  const unsigned to_mean = warp < nr ? peer_addr(mean_v + myrow, kMeanCta) : 0u;
  const bool wall_lo = rank == 0, wall_hi = rank == kClusterCtas - 1;
  const int strip = warp - kFluxWarp;
  const bool flux_warp = (wall_lo || wall_hi) && strip >= 0 && strip < Lay::kStrips;
  double flux_total = (flux_warp && strip == 0) ? pa.flux_acc[wall_hi ? 1 : 0] : 0.0;

  const float wp = (float)a.wp, wm = (float)a.wm, gwp = (float)a.gwp, gwm = (float)a.gwm;
  const float cp = 1.0f - 0.5f * wp, cm_ = 1.0f - 0.5f * wm;
  const float mub = (float)a.mub, rho0 = (float)a.rho0;
  const float gwall = (a.wall_mode == 0) ? -1.0f : 0.0f;
  const float W1 = (float)kW1, W2 = (float)kW2;
  const float fb = (float)a.fb, fd = (float)a.fd, fdq = (float)a.fdq;
  const float wd1 = W1 * fd, wd2 = W2 * fd;
  const float nieps = -(float)pa.inv_eps;
  bool bad = false;

  // totals of a wall's strips, added in the order of the mean-mode kernel
  auto add_flux = [&]() {
    double v = lane < Lay::kStrips ? fpart[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    flux_total += v;
  };

  __syncthreads();
  cluster_sync();  // every CTA of the cluster runs and holds its state

  int cur = 0;
  for (int t = 0; t < steps; ++t) {
    // ------------------------------------------------------------- march
    const float* const p = sm + lay.pop + cur * 18 * RN;
    float* const q = sm + lay.pop + (cur ^ 1) * 18 * RN;
    float* const flux = sm + lay.flux + cur * 6 * Nx;
    for (int idx = tid; idx < nr * Nx; idx += kThreads) {
      const int ly = idx / Nx, x = idx & (Nx - 1), y = r0 + ly;
      const int xl = (x - 1) & (Nx - 1), xr = (x + 1) & (Nx - 1);
      float f[9], g[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        f[i] = p[i * RN + idx];
        g[i] = p[(9 + i) * RN + idx];
      }
      const float* ph = phi + (ly + 1) * Nx;
      const float pc = ph[x];
      const float pm = (y > 0) ? ph[x - Nx] : gwall * pc;
      const float pn = (y + 1 < Ny) ? ph[x + Nx] : gwall * pc;
      const float Ex = -0.5f * (ph[xr] - ph[xl]);
      const float Ey = ebar[ly] - 0.5f * (pn - pm);
      const float sy = shift[ly + 1], s_dn = shift[ly], s_up = shift[ly + 2];
      const float sf = fb + fd * (float)y;
      bool b;
      collide_node<S, float>(f, g, Ex, Ey, sy, sf, fdq, mub, wp, wm, cp, cm_, gwp, gwm, b);
      bad = bad || b;
      // a population is rounded to its storage type when it reaches its node
      // (rt); what changes on the way there changes first
      auto rt = [](float v) { return Store<S>::template rt<float>(v); };
      q[idx] = rt(f[0]);
      q[9 * RN + idx] = rt(g[0]);
      const int rowb = ly * Nx;
      q[1 * RN + rowb + xr] = rt(f[1]);
      q[10 * RN + rowb + xr] = rt(g[1]);
      q[3 * RN + rowb + xl] = rt(f[3]);
      q[12 * RN + rowb + xl] = rt(g[3]);
      // c_y = +1
      if (y + 1 < Ny) {
        const float sh = sy - s_up;
        const float n2 = g[2] + W1 * sh, n5 = g[5] + W2 * sh, n6 = g[6] + W2 * sh;
        if (ly + 1 < nr) {
          float* d = q + rowb + Nx;
          d[2 * RN + x] = rt(f[2]);
          d[5 * RN + xr] = rt(f[5]);
          d[6 * RN + xl] = rt(f[6]);
          d[11 * RN + x] = rt(n2);
          d[14 * RN + xr] = rt(n5);
          d[15 * RN + xl] = rt(n6);
        } else {
          const unsigned d = peer_addr(q, rank + 1);
          st_peer(d + 4 * (2 * RN + x), rt(f[2]));
          st_peer(d + 4 * (5 * RN + xr), rt(f[5]));
          st_peer(d + 4 * (6 * RN + xl), rt(f[6]));
          st_peer(d + 4 * (11 * RN + x), rt(n2));
          st_peer(d + 4 * (14 * RN + xr), rt(n5));
          st_peer(d + 4 * (15 * RN + xl), rt(n6));
        }
      } else {
        // collector: f bounces back; g leaves and re-enters from its own row
        float* d = q + rowb;
        d[4 * RN + x] = rt(f[2] + wd1);
        d[7 * RN + x] = rt(f[5] + wd2);
        d[8 * RN + x] = rt(f[6] + wd2);
        d[13 * RN + x] = rt(g[4]);
        d[16 * RN + xl] = rt(g[7]);
        d[17 * RN + xr] = rt(g[8]);
        flux[x] = rt(g[2]);
        flux[Nx + x] = rt(g[5]);
        flux[2 * Nx + x] = rt(g[6]);
        flux[3 * Nx + x] = rt(g[4]);
        flux[4 * Nx + x] = rt(g[7]);
        flux[5 * Nx + x] = rt(g[8]);
      }
      // c_y = -1
      if (y > 0) {
        const float sh = sy - s_dn;
        const float n4 = g[4] + W1 * sh, n7 = g[7] + W2 * sh, n8 = g[8] + W2 * sh;
        if (ly > 0) {
          float* d = q + rowb - Nx;
          d[4 * RN + x] = rt(f[4]);
          d[7 * RN + xl] = rt(f[7]);
          d[8 * RN + xr] = rt(f[8]);
          d[13 * RN + x] = rt(n4);
          d[16 * RN + xl] = rt(n7);
          d[17 * RN + xr] = rt(n8);
        } else {
          const int last = r0 - 1 - band_start(rank - 1, Ny);
          const unsigned d = peer_addr(q + last * Nx, rank - 1);
          st_peer(d + 4 * (4 * RN + x), rt(f[4]));
          st_peer(d + 4 * (7 * RN + xl), rt(f[7]));
          st_peer(d + 4 * (8 * RN + xr), rt(f[8]));
          st_peer(d + 4 * (13 * RN + x), rt(n4));
          st_peer(d + 4 * (16 * RN + xl), rt(n7));
          st_peer(d + 4 * (17 * RN + xr), rt(n8));
        }
      } else {
        // injector: bounce-back of f, anti-bounce-back of g
        float n2, n5, n6;
        inject<float>(g[4], g[7], g[8], Ex, Ey, sy, mub, rho0, n2, n5, n6);
        float* d = q + rowb;
        d[2 * RN + x] = rt(f[4] - wd1);
        d[5 * RN + x] = rt(f[7] - wd2);
        d[6 * RN + x] = rt(f[8] - wd2);
        d[11 * RN + x] = rt(n2);
        d[14 * RN + x] = rt(n5);
        d[15 * RN + x] = rt(n6);
        flux[x] = rt(n2);
        flux[Nx + x] = rt(n5);
        flux[2 * Nx + x] = rt(n6);
        flux[3 * Nx + x] = rt(g[4]);
        flux[4 * Nx + x] = rt(g[7]);
        flux[5 * Nx + x] = rt(g[8]);
      }
    }
    cur ^= 1;
    cluster_sync();

    // ----------------------------------------------------------- forward
    double wall = 0.0;  // this lane's share of the strip's wall flux
    if (warp < nr) {
      const float* g = q + 9 * RN + warp * Nx;
      const float s = shift[warp + 1];
      const bool first = slab_first(myrow, slab), last = slab_last(myrow, Ny, slab);
      float2 v[E];
#pragma unroll
      for (int n2 = 0; n2 < E; ++n2) {
        float2 c[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) c[i] = *reinterpret_cast<const float2*>(g + i * RN + 2 * (lane + 32 * n2));
        v[n2] = make_float2(march_charge(s, first, last, [&](int i) { return c[i].x; }),
                            march_charge(s, first, last, [&](int i) { return c[i].y; }));
      }
      const float c0 = __shfl_sync(0xffffffffu, v[0].x, 0);
      float re[E], im[E];
#pragma unroll
      for (int n2 = 0; n2 < E; ++n2) {
        re[n2] = (v[n2].x - c0) * nieps;
        im[n2] = (v[n2].y - c0) * nieps;
      }
      fft.run(re, im, lane);
      if (lane == 0) {
        st_peer(to_mean, mean_coefficient(make_float2(re[0], im[0]), c0, nieps, (float)Nx));
        st_peer(to_nyq, make_float2(re[0] - im[0], 0.0f));
      }
      lane_fft_store<E>(re, im, rowbuf, lane);
#pragma unroll
      for (int n = 0; n < E; ++n) {
        const int k = lane + 32 * n;
        if (k > 0) st_peer(to_col[n], untangle<E>(rowbuf, k, wkf[n]));
      }
      cluster_sync();
    } else if (flux_warp) {
      if (strip == 0 && t > 0) add_flux();  // the step before
      __syncwarp();
      cluster_arrive();
      const int x = 60 * strip + 2 * (lane - 1);
      if (lane >= 1 && lane <= 30 && x < Nx) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          double z[6];
#pragma unroll
          for (int i = 0; i < 6; ++i) z[i] = (double)flux[i * Nx + x + j];
          if (wall_lo) {
            wall += ((z[0] - z[3]) + (z[1] - z[4])) + (z[2] - z[5]);
          } else {
            wall += (z[0] + z[1]) + z[2];
            wall -= (z[3] + z[4]) + z[5];
          }
        }
      }
      __syncwarp();
      cluster_wait();
    } else {
      cluster_sync();
    }

    // ------------------------------------------------------------- solve
    if (rank == kMeanCta && warp >= kMeanWarp && warp < kMeanWarp + kMeanThreadsSmall / 32) {
      cluster_arrive();  // nothing of this is read before the next march
      const bool final_step = t + 1 == steps;
      mean_mode_core<float, kMeanThreadsSmall>(pa, mean_v, ms, tid - 32 * kMeanWarp, [&](int j, ff pc, ff ec) {
        const int o = band_owner(j, Ny);
        st_peer(peer_addr(ebar + (j - band_start(o, Ny)), o), ec.hi + ec.lo);
        if (final_step) static_cast<float2*>(pa.phibar)[j] = make_float2(pc.hi, pc.lo);
      });
      __syncwarp();
      cluster_wait();
    } else if (flux_warp) {
      cluster_arrive();
      for (int o = 16; o > 0; o >>= 1) wall += __shfl_down_sync(0xffffffffu, wall, o);
      if (lane == 0) fpart[strip] = wall;
      __syncwarp();
      cluster_wait();
    } else {
      if (warp < ML) {
        float2 d[kChunkRows];
        const float2* c = col + warp * (lay.col_row / 2) + j0;
#pragma unroll
        for (int k = 0; k < kChunkRows; ++k) d[k] = k < nj ? c[k] : make_float2(0.0f, 0.0f);
        // forward sweep: the chunk's affine map, the scan over chunks, values
        ChunkMap cm;
#pragma unroll
        for (int k = 0; k < kChunkRows; ++k)
          if (k < nj) cm.row(piv[k], d[k].x, d[k].y, tail_row_fused(k, nj));
        float al = cm.al;
        float2 br = cm.br;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const float a2 = __shfl_up_sync(0xffffffffu, al, o);
          const float bx = __shfl_up_sync(0xffffffffu, br.x, o), by = __shfl_up_sync(0xffffffffu, br.y, o);
          if (lane >= o) {
            br = make_float2(map_apply(al, bx, br.x), map_apply(al, by, br.y));
            al = al * a2;
          }
        }
        float2 x = make_float2(__shfl_up_sync(0xffffffffu, br.x, 1), __shfl_up_sync(0xffffffffu, br.y, 1));
        if (lane == 0) x = make_float2(0.0f, 0.0f);
        al = 1.0f;
        br = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int k = 0; k < kChunkRows; ++k)
          if (k < nj) {
            const float r = piv[k];
            x = make_float2(sweep_value(r, d[k].x, x.x), sweep_value(r, d[k].y, x.y));
            d[k] = x;
            br = make_float2(map_apply(al, x.x, br.x), map_apply(al, x.y, br.y));
            al = -al * r;
          }
        // backward sweep, from the last chunk down
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const float a2 = __shfl_down_sync(0xffffffffu, al, o);
          const float bx = __shfl_down_sync(0xffffffffu, br.x, o), by = __shfl_down_sync(0xffffffffu, br.y, o);
          if (lane + o < 32) {
            br = make_float2(map_apply(al, bx, br.x), map_apply(al, by, br.y));
            al = al * a2;
          }
        }
        x = make_float2(__shfl_down_sync(0xffffffffu, br.x, 1), __shfl_down_sync(0xffffffffu, br.y, 1));
        if (lane == 31) x = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int k = kChunkRows - 1; k >= 0; --k)
          if (k < nj) {
            const float r = piv[k];
            x = make_float2(sweep_back(r, d[k].x, x.x), sweep_back(r, d[k].y, x.y));
            st_peer(home[k], x);
          }
      }
      cluster_sync();
    }

    // ----------------------------------------------------------- inverse
    if (warp < nr) {
      const float2* s = spec + warp * (Lay::kSpecRow / 2);
      float re[E], im[E];
#pragma unroll
      for (int n2 = 0; n2 < E; ++n2) {
        const int k = lane + 32 * n2;
        const float2 sk = (k == 0) ? make_float2(0.0f, 0.0f) : s[k];
        const float2 z = entangle(sk, s[L - k], wki[n2]);
        re[n2] = z.x;
        im[n2] = z.y;
      }
      fft.run(re, im, lane);
      lane_fft_store<E>(re, im, rowbuf, lane);
      const float inL = 1.0f / (float)L;
      float* out = phi + (warp + 1) * Nx;
      const bool to_dn = warp == 0 && !wall_lo, to_up = warp == nr - 1 && !wall_hi;
      const unsigned dn = to_dn ? peer_addr(phi + (r0 - band_start(rank - 1, Ny) + 1) * Nx, rank - 1) : 0u;
      const unsigned upr = to_up ? peer_addr(phi, rank + 1) : 0u;
#pragma unroll
      for (int n = 0; n < E; ++n) {
        const int k = lane + 32 * n;
        const float2 w = rowbuf[lpad(k)];
        const float2 v = make_float2(w.x * inL, -w.y * inL);
        reinterpret_cast<float2*>(out)[k] = v;
        if (to_dn) st_peer(dn + 8 * k, v);
        if (to_up) st_peer(upr + 8 * k, v);
      }
    }
    cluster_sync();
  }

  // ---- back to the run's buffers
  if (bad) atomicOr(a.err, 1);
  for (int i = 0; i < 18; ++i) {
    S* dst = static_cast<S*>(const_cast<void*>(i < 9 ? a.fin : a.gin)) + (i % 9) * a.plane + (long long)r0 * P;
    for (int k = 4 * tid; k < nr * Nx; k += 4 * kThreads)
      Four<S>::st(dst + k, *reinterpret_cast<const float4*>(sm + lay.pop + (cur * 18 + i) * RN + k));
  }
  for (int k = 4 * tid; k < nr * Nx; k += 4 * kThreads)
    *reinterpret_cast<float4*>(static_cast<float*>(pa.dphi) + (long long)r0 * P + k) =
        *reinterpret_cast<const float4*>(phi + Nx + k);
  if (tid < nr) static_cast<float*>(pa.Ebar)[r0 + tid] = ebar[tid];
  if (flux_warp && strip == 0) {
    add_flux();
    if (lane == 0) pa.flux_acc[wall_hi ? 1 : 0] = flux_total;
  }
}

namespace {

using ResidentKernel = void (*)(StepArgs, PoissonArgs, int, int);

int max_rows(int Ny) { return (Ny + kClusterCtas - 1) / kClusterCtas; }

template <int E>
bool resident_config_n(int storage, int Ny, ResidentKernel* k, size_t* smem) {
  *smem = sizeof(float) * (size_t)Layout<E>(max_rows(Ny), Ny).total;
  switch (storage) {
    case 1: *k = k_resident<float, E>; return true;
    case 2: *k = k_resident<__nv_bfloat16, E>; return true;
    case 3: *k = k_resident<__half, E>; return true;
  }
  return false;
}
bool resident_config(int Nx, int Ny, int storage, ResidentKernel* k, size_t* smem) {
  if (Ny < kClusterCtas || Ny > kMaxRows) return false;
  switch (Nx) {
    case 64: return resident_config_n<1>(storage, Ny, k, smem);
    case 128: return resident_config_n<2>(storage, Ny, k, smem);
    case 256: return resident_config_n<4>(storage, Ny, k, smem);
  }
  return false;
}

}  // namespace

// Whether this GPU can hold a run of this size in one cluster; sets the
// kernel's attributes on the current device (no copies, no synchronisation:
// ehd_step asks).
bool resident_supported(int Nx, int Ny, int storage) {
  ResidentKernel k = nullptr;
  size_t smem = 0;
  if (!resident_config(Nx, Ny, storage, &k, &smem)) return false;
  return cluster_fits(k, kThreads, smem);
}

cudaError_t launch_resident(const StepArgs& a, const PoissonArgs& pa, int storage, int steps, cudaStream_t s) {
  ResidentKernel k = nullptr;
  size_t smem = 0;
  if (!resident_config(a.Nx, a.Ny, storage, &k, &smem)) return cudaErrorInvalidValue;
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t c;
  cluster_launch_config(&c, at, kThreads, smem, s);
  return cudaLaunchKernelEx(&c, k, a, pa, steps, max_rows(a.Ny));
}

}  // namespace ehd
