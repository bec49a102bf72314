// ehd_noalloc.cu -- a Poisson solve that allocates no device memory.
//
// Some callers cannot call cudaMalloc once they are running: a process whose
// device memory is entirely reserved up front by a framework's own pool, or a
// latency-critical loop where the implicit device synchronisation of
// cudaMalloc / cudaFree is not acceptable.  ehd_poisson_noalloc gives them the
// Poisson solve of the library (row FFT, one tridiagonal per wavenumber with
// the mean mode in FP64, inverse row FFT) on their own device buffers, with
// every intermediate (half spectrum, pivots, twiddles, mean profile) kept in
// one file-scope __device__ array of fixed size.  That array is part of the
// library image: every GPU that loads the library holds it until the process
// exits.
//
// In host code the array's name is only a host-side stand-in; its device
// address is looked up with cudaGetSymbolAddress on every call, with the
// calling device current, and passed to the kernels.
//
// The twiddle and pivot tables for a grid are rebuilt only when the sizes
// change, which the host tracks per device.  A call made while its stream is
// being captured cannot rely on that record (the captured work may run any
// number of times, interleaved with direct calls for other sizes), so it
// always enqueues the table build, and from then on every call on that
// device rebuilds the tables.
#include <cuda_runtime.h>

#include <mutex>

#include "cluster_dev.cuh"
#include "ehd.h"
#include "fft_dev.cuh"
#include "mean_dev.cuh"

namespace ehd {
void set_error(const char* msg);
}

namespace {

using ehd::Cplx;

constexpr size_t kScratchBytes = size_t(8) << 20;  // 8 MiB
constexpr int kMaxNx = 2048;
constexpr int kMaxNy = 4096;
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

struct Layout {
  size_t spec, spec0, piv, piv0, tw, phibar, total;
};

size_t up256(size_t b) { return (b + 255) & ~size_t(255); }

Layout layout_for(int Nx, int Ny) {
  const size_t Mh = (size_t)Nx / 2 + 1;
  Layout L{};
  size_t o = 0;
  L.spec = o;   o += up256(Mh * Ny * sizeof(Cplx<float>));  // [Ny][Mh]
  L.spec0 = o;  o += up256((size_t)Ny * sizeof(double));
  L.piv = o;    o += up256(Mh * Ny * sizeof(float));        // [Mh][Ny]
  L.piv0 = o;   o += up256((size_t)Ny * sizeof(double));
  L.tw = o;     o += up256((size_t)(Nx / 2) * sizeof(Cplx<float>));
  L.phibar = o; o += up256((size_t)Ny * sizeof(double));
  L.total = o;
  return L;
}

struct DeviceSlot {
  unsigned char* base = nullptr;  // device address of g_scratch at the last call
  int Nx = 0, Ny = 0, wall_mode = -1;  // sizes the tables were built for
  bool always_rebuild = false;    // set once a call was made during stream capture
  // the cluster kernel of 64, 128, 256, 512 columns: most shared memory known
  // to fit, least known not to
  size_t fits[4] = {0, 0, 0, 0}, too_big[4] = {~size_t(0), ~size_t(0), ~size_t(0), ~size_t(0)};
};
std::mutex g_mu;
DeviceSlot g_slots[kMaxDevices];

struct Ptrs {
  Cplx<float>* spec;
  double* spec0;
  float* piv;
  double* piv0;
  Cplx<float>* tw;
  double* phibar;
};

Ptrs ptrs(unsigned char* base, const Layout& L) {
  return {reinterpret_cast<Cplx<float>*>(base + L.spec), reinterpret_cast<double*>(base + L.spec0),
          reinterpret_cast<float*>(base + L.piv),        reinterpret_cast<double*>(base + L.piv0),
          reinterpret_cast<Cplx<float>*>(base + L.tw),   reinterpret_cast<double*>(base + L.phibar)};
}

// Twiddles exp(-2 pi i k / Nx) and reciprocal Thomas pivots of every
// wavenumber (diagonal -(2 + kappa_m), unit off-diagonals, wall corners).
__global__ void k_na_tables(int Nx, int Ny, int wall_mode, Ptrs p) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < Nx / 2) {
    double s, c;
    sincospi(2.0 * (double)t / (double)Nx, &s, &c);
    p.tw[t] = {(float)c, (float)-s};
  }
  const int Mh = Nx / 2 + 1;
  if (t < Mh) {
    const double kx = 2.0 * 3.141592653589793238462643383279502884 * (double)t / (double)Nx;
    const double diag = -(2.0 + kx * kx);
    const double corner = diag - (wall_mode == 0 ? 1.0 : 0.0);
    double prev = 0.0;
    for (int j = 0; j < Ny; ++j) {
      const double b = (j == 0 || j == Ny - 1) ? corner : diag;
      prev = 1.0 / ((j == 0) ? b : b - prev);
      if (t == 0)
        p.piv0[j] = prev;
      else
        p.piv[(size_t)t * Ny + j] = (float)prev;
    }
  }
}

__device__ Cplx<float>* na_fft(Cplx<float>* a, Cplx<float>* b, int N, const Cplx<float>* tw, bool inverse) {
  const int half = N >> 1;
  for (int Ns = 1; Ns < N; Ns <<= 1) {
    const int tstride = N / (2 * Ns);
    for (int j = threadIdx.x; j < half; j += blockDim.x) {
      const int k = j & (Ns - 1);
      Cplx<float> w = tw[k * tstride];
      if (inverse) w.im = -w.im;
      const Cplx<float> u = a[j], x = a[j + half];
      const Cplx<float> v = {x.re * w.re - x.im * w.im, x.re * w.im + x.im * w.re};
      const int idx = ((j - k) << 1) + k;
      b[idx] = {u.re + v.re, u.im + v.im};
      b[idx + Ns] = {u.re - v.re, u.im - v.im};
    }
    __syncthreads();
    Cplx<float>* t = a;
    a = b;
    b = t;
  }
  return a;
}

// One CTA per row: s = -rho_c / eps, FP64 row sum (mean mode), FFT of the rest.
__global__ void __launch_bounds__(256) k_na_fwd(int Nx, int Ny, double inv_eps, const float* __restrict__ rhoc,
                                                Ptrs p) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[8];
  Cplx<float>* A = reinterpret_cast<Cplx<float>*>(smem);
  Cplx<float>* B = A + Nx;
  const int y = blockIdx.x;
  double sum = 0.0;
  for (int x = threadIdx.x; x < Nx; x += blockDim.x) {
    const float s = -rhoc[(size_t)y * Nx + x] * (float)inv_eps;
    A[x].re = s;
    sum += (double)s;
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    red[0] = t;
    p.spec0[y] = t;
  }
  __syncthreads();
  const float mean = (float)(red[0] / (double)Nx);
  for (int x = threadIdx.x; x < Nx; x += blockDim.x) {
    A[x].re -= mean;
    A[x].im = 0.0f;
  }
  __syncthreads();
  const Cplx<float>* res = na_fft(A, B, Nx, p.tw, false);
  const int Mh = Nx / 2 + 1;
  for (int m = threadIdx.x; m < Mh; m += blockDim.x)
    p.spec[(size_t)y * Mh + m] = (m == 0) ? Cplx<float>{0.0f, 0.0f} : res[m];
}

// Thomas recurrences of one wavenumber as a warp scan over 32 row chunks.
template <class R, class V, class Ops>
__device__ void na_thomas(V* d, const R* r, int Ny, int lane) {
  const int C = (Ny + 31) >> 5;
  const int j0 = min(lane * C, Ny), j1 = min(j0 + C, Ny);
  R al = R(1);
  V br = Ops::zero();
  for (int j = j0; j < j1; ++j) {
    al = -r[j] * al;
    br = Ops::scl(r[j], Ops::sub(d[j], br));
  }
  for (int o = 1; o < 32; o <<= 1) {
    const R a2 = __shfl_up_sync(0xffffffffu, al, o);
    const V b2 = Ops::up(br, o);
    if (lane >= o) {
      br = Ops::axpy(al, b2, br);
      al *= a2;
    }
  }
  V x = Ops::up(br, 1);
  if (lane == 0) x = Ops::zero();
  for (int j = j0; j < j1; ++j) {
    x = Ops::scl(r[j], Ops::sub(d[j], x));
    d[j] = x;
  }
  __syncwarp();
  al = R(1);
  br = Ops::zero();
  for (int j = j1 - 1; j >= j0; --j) {
    al = -r[j] * al;
    br = Ops::axpy(-r[j], br, d[j]);
  }
  for (int o = 1; o < 32; o <<= 1) {
    const R a2 = __shfl_down_sync(0xffffffffu, al, o);
    const V b2 = Ops::down(br, o);
    if (lane + o < 32) {
      br = Ops::axpy(al, b2, br);
      al *= a2;
    }
  }
  x = Ops::down(br, 1);
  if (lane == 31) x = Ops::zero();
  for (int j = j1 - 1; j >= j0; --j) {
    x = Ops::axpy(-r[j], x, d[j]);
    d[j] = x;
  }
  __syncwarp();
}

struct RealOps {
  __device__ static double zero() { return 0.0; }
  __device__ static double up(double v, int o) { return __shfl_up_sync(0xffffffffu, v, o); }
  __device__ static double down(double v, int o) { return __shfl_down_sync(0xffffffffu, v, o); }
  __device__ static double axpy(double a, double x, double b) { return a * x + b; }
  __device__ static double sub(double x, double y) { return x - y; }
  __device__ static double scl(double a, double x) { return a * x; }
};

struct CplxOps {
  using V = Cplx<float>;
  __device__ static V zero() { return {0.0f, 0.0f}; }
  __device__ static V up(V v, int o) {
    return {__shfl_up_sync(0xffffffffu, v.re, o), __shfl_up_sync(0xffffffffu, v.im, o)};
  }
  __device__ static V down(V v, int o) {
    return {__shfl_down_sync(0xffffffffu, v.re, o), __shfl_down_sync(0xffffffffu, v.im, o)};
  }
  __device__ static V axpy(float a, V x, V b) { return {a * x.re + b.re, a * x.im + b.im}; }
  __device__ static V sub(V x, V y) { return {x.re - y.re, x.im - y.im}; }
  __device__ static V scl(float a, V x) { return {a * x.re, a * x.im}; }
};

__global__ void __launch_bounds__(128) k_na_modes(int Nx, int Ny, int wall_mode, double phi0, int wpc, Ptrs p) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m = blockIdx.x * wpc + warp;
  const int Mh = Nx / 2 + 1;
  if (warp >= wpc || m >= Mh) return;
  if (m == 0) {
    double* d = reinterpret_cast<double*>(smem) + (size_t)warp * Ny;
    const double wc = (wall_mode == 0) ? 2.0 : 1.0;
    for (int j = lane; j < Ny; j += 32) d[j] = p.spec0[j] - ((j == 0) ? wc * (double)Nx * phi0 : 0.0);
    __syncwarp();
    na_thomas<double, double, RealOps>(d, p.piv0, Ny, lane);
    for (int j = lane; j < Ny; j += 32) p.phibar[j] = d[j] / (double)Nx;
    return;
  }
  Cplx<float>* d = reinterpret_cast<Cplx<float>*>(smem) + (size_t)warp * Ny;
  for (int j = lane; j < Ny; j += 32) d[j] = p.spec[(size_t)j * Mh + m];
  __syncwarp();
  na_thomas<float, Cplx<float>, CplxOps>(d, p.piv + (size_t)m * Ny, Ny, lane);
  for (int j = lane; j < Ny; j += 32) p.spec[(size_t)j * Mh + m] = d[j];
}

// One CTA per row: inverse FFT of the modes m >= 1 plus the FP64 mean profile.
__global__ void __launch_bounds__(256) k_na_inv(int Nx, int Ny, float* __restrict__ phi, Ptrs p) {
  extern __shared__ __align__(16) unsigned char smem[];
  Cplx<float>* A = reinterpret_cast<Cplx<float>*>(smem);
  Cplx<float>* B = A + Nx;
  const int y = blockIdx.x, half = Nx >> 1, Mh = Nx / 2 + 1;
  const Cplx<float>* spec = p.spec + (size_t)y * Mh;
  for (int m = threadIdx.x; m < Nx; m += blockDim.x) {
    Cplx<float> v = {0.0f, 0.0f};
    if (m > 0 && m <= half) {
      v = spec[m];
    } else if (m > half) {
      const Cplx<float> s = spec[Nx - m];
      v = {s.re, -s.im};
    }
    A[m] = v;
  }
  __syncthreads();
  const Cplx<float>* res = na_fft(A, B, Nx, p.tw, true);
  const double pb = p.phibar[y];
  for (int x = threadIdx.x; x < Nx; x += blockDim.x)
    phi[(size_t)y * Nx + x] = (float)(pb + (double)(res[x].re / (float)Nx));
}

// ---------------------------------------------------------------- one launch
// The whole solve by one cluster of 16 CTAs, for grids whose spectrum fits
// their shared memory (64 to 512 columns, up to 2^18 nodes).  A small solve is
// bound by its launches and by the chain of each kernel, not by the work: the
// three kernels above take 24.7 to 26.7 us a call at 256 x 208 (radix-2 rows with
// a barrier a stage, an FP64 elimination of the mean mode), of which the data
// would take 0.1; this one takes 12.4 (64 x 56: 16.5 -> 8.3; 512 x 416: 32.9 ->
// 28.2; 512 x 512: 41 -> 35.6; calls back to back, on one machine -- a call that
// the caller waits for takes 34 -> 22 us at 256 x 208).  Here a warp transforms a
// row (LaneFft), the wavenumbers' columns are written into the CTA that solves
// them and back into the rows' owners, and the mean mode is the FP64 double
// prefix sum of the run's solver.
namespace na {
using namespace ehd;
constexpr int kThreads = 512, kWarps = kThreads / 32;
constexpr int kMeanCta = 8, kMeanWarp = kWarps - 4;  // the mean mode's CTA and its first warp there
constexpr int kMeanNT = 128;

template <int E>
struct Lay {
  static constexpr int Nx = 64 * E, L = 32 * E, kModes = L / kClusterCtas;
  int rows, spec, col, row, mean, pb;  // float2 offsets
  // A wavenumber's column: 32 chunks of `chunk` rows (a lane each), an odd
  // number of float2 apart -- with the rows packed, the lanes of a solve met in
  // one or two banks whenever the chunk's length was a multiple of 16 or 8 (512
  // x 512: 48.9 us a call, three kernels 41.2) -- and the columns too.
  int chunk, chunk_pitch, col_pitch;
  size_t bytes;
  __host__ __device__ explicit Lay(int Ny) {
    rows = (Ny + kClusterCtas - 1) / kClusterCtas;
    chunk = (Ny + 31) / 32;
    chunk_pitch = chunk | 1;
    col_pitch = 32 * chunk_pitch + 1;
    spec = 0;
    col = spec + rows * (L + 2);
    row = col + kModes * col_pitch;
    mean = row + kWarps * kLaneRow<E>;
    pb = mean + 2 * Ny;
    bytes = sizeof(float2) * (size_t)(pb + rows);
  }
  // row y's place in a column; inv = 2^32 / chunk + 1 (y / chunk exactly for y
  // below 2^25), as a division costs a row 0.3 us
  __device__ int in_col(int y, unsigned inv) const { return y + (int)__umulhi(y, inv) * (chunk_pitch - chunk); }
};
unsigned chunk_inverse(int Ny) { return (unsigned)((1ull << 32) / ((Ny + 31) / 32) + 1); }  // (chunk 1: unused)

// A sum as three FP32 numbers a + b + c, the error of each addition carried into
// the next part (Knuth's two-sum).
struct Sum3 {
  float a = 0.0f, b = 0.0f, c = 0.0f;
  __device__ void add(float v) {
    float e;
    two_sum_f(a, v, a, e);
    two_sum_f(b, e, b, e);
    c += e;
  }
  __device__ void add(float a2, float b2, float c2) {
    float e, f;
    two_sum_f(a, a2, a, e);
    two_sum_f(b, b2, b, f);
    c += c2 + f;
    two_sum_f(b, e, b, f);
    c += f;
  }
};

// hieps: 1 / (2 eps)
template <int E>
__global__ void __launch_bounds__(kThreads, 1) k_solve(int Ny, unsigned inv, float hieps, const float* __restrict__ rhoc,
                                                       float* __restrict__ phi, Ptrs p, PoissonArgs pa) {
  using La = Lay<E>;
  constexpr int Nx = La::Nx, L = La::L, ML = La::kModes;
  extern __shared__ __align__(16) float2 sm[];
  __shared__ MeanScratch<double, kMeanNT> ms;
  const La la(Ny);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int rank;
  asm("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(rank));
  const int r0 = band_start(rank, Ny), nr = band_start(rank + 1, Ny) - r0;
  float2* const spec = sm + la.spec;
  float2* const col = sm + la.col;
  float2* const rowbuf = sm + la.row + warp * kLaneRow<E>;
  double* const mean_v = reinterpret_cast<double*>(sm + la.mean);
  double* const pb = reinterpret_cast<double*>(sm + la.pb);

  const float2* __restrict__ tw = reinterpret_cast<const float2*>(p.tw);  // W_Nx^k, k < Nx / 2
  auto W = [&](int k) {
    const float2 v = tw[k & (Nx / 2 - 1)];
    return (k & (Nx / 2)) ? make_float2(-v.x, -v.y) : v;
  };
  LaneFft<E, true> fft;
#pragma unroll
  for (int k2 = 0; k2 < E; ++k2) fft.w[k2] = W((2 * lane * k2) & (Nx - 1));
  fft.init_stages(lane);
  float2 wk[E];  // W_Nx^(lane + 32 j)
#pragma unroll
  for (int j = 0; j < E; ++j) wk[j] = tw[lane + 32 * j];
  cluster_sync();  // every CTA runs: its shared memory may be written

  // ---- rows: half of s = -rho_c / eps, the row's sum, and the transform of what
  // differs from the row's first value.  The sum is held in three FP32 numbers
  // whose rounding errors are carried on (FP64 additions, 16 cycles of the SM
  // each, would be most of a small solve): over values spread across 2^60 it is
  // within 3e-21 of the largest, an FP64 sum within 9e-16, two FP32 numbers
  // within 2e-14.  Its terms are s / Nx, so that it is finite where every s is.
  for (int r = warp; r < nr; r += kWarps) {
    const int y = r0 + r, yc = la.in_col(y, inv);
    const float2* src = reinterpret_cast<const float2*>(rhoc + (size_t)y * Nx);
    float re[E], im[E];
    Sum3 sum;
#pragma unroll
    for (int j = 0; j < E; ++j) {
      const float2 v = src[lane + 32 * j];
      re[j] = -v.x * hieps;
      im[j] = -v.y * hieps;
    }
    const float c0 = __shfl_sync(0xffffffffu, re[0], 0);
#pragma unroll
    for (int j = 0; j < E; ++j) {
      sum.add(re[j] * (2.0f / Nx));
      sum.add(im[j] * (2.0f / Nx));
      re[j] -= c0;
      im[j] -= c0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      sum.add(__shfl_xor_sync(0xffffffffu, sum.a, o), __shfl_xor_sync(0xffffffffu, sum.b, o),
              __shfl_xor_sync(0xffffffffu, sum.c, o));
    fft.run(re, im, lane);
    if (lane == 0) {
      // (the third part waits in the mean mode's scratch half of the array)
      st_peer(peer_addr(mean_v + y, kMeanCta), make_float2(sum.a, sum.b));
      st_peer(peer_addr(mean_v + Ny + y, kMeanCta), make_float2(sum.c, 0.0f));
      st_peer(peer_addr(col + (ML - 1) * la.col_pitch + yc, kClusterCtas - 1), make_float2(2.0f * (re[0] - im[0]), 0.0f));
    }
    lane_fft_store<E>(re, im, rowbuf, lane);
    // S[k] = E + W^k O from E = Z[k] + Z*[L - k], O = (Z[k] - Z*[L - k]) / i
    // (the halves are in the values transformed)
#pragma unroll
    for (int j = 0; j < E; ++j) {
      const int k = lane + 32 * j;
      const float2 zk = rowbuf[lpad(k)], zp = rowbuf[lpad((L - k) & (L - 1))];
      const float Er = zk.x + zp.x, Ei = zk.y - zp.y, Dr = zk.x - zp.x, Di = zk.y + zp.y;
      const int m = k - 1;
      if (m >= 0)
        st_peer(peer_addr(col + (m % ML) * la.col_pitch + yc, m / ML),
                make_float2(fmaf(wk[j].x, Di, fmaf(wk[j].y, Dr, Er)), fmaf(wk[j].y, Di, fmaf(-wk[j].x, Dr, Ei))));
    }
    __syncwarp();
  }
  cluster_sync();

  // ---- y solves: a warp per wavenumber, 32 chunks of rows
  const bool mean_warp = rank == kMeanCta && warp >= kMeanWarp;
  if (mean_warp) {
    const int t = tid - 32 * kMeanWarp;
    for (int j = t; j < Ny; j += kMeanNT) {
      const float2 v = reinterpret_cast<const float2*>(mean_v)[j];
      mean_v[j] = (double)Nx * ((double)v.x + ((double)v.y + (double)reinterpret_cast<const float2*>(mean_v)[Ny + j].x));
    }
    sub_sync<kMeanNT>();
    mean_mode_core<double, kMeanNT>(pa, mean_v, ms, t, [&](int j, double pc, double) {
      const int o = band_owner(j, Ny);
      const unsigned long long b = __double_as_longlong(pc);
      st_peer(peer_addr(pb + (j - band_start(o, Ny)), o),
              make_float2(__uint_as_float((unsigned)b), __uint_as_float((unsigned)(b >> 32))));
    });
  } else {
    const int nw = rank == kMeanCta ? kMeanWarp : kWarps;
    const int C = la.chunk, j0 = min(lane * C, Ny), j1 = min(j0 + C, Ny);
    for (int q = warp; q < ML; q += nw) {
      const int m = rank * ML + q + 1;
      const float* __restrict__ r = p.piv + (size_t)m * Ny;
      float2* d = col + q * la.col_pitch + lane * (la.chunk_pitch - C);  // d[j]: row j of this lane's chunk
      float al = 1.0f;
      float2 br = make_float2(0.0f, 0.0f);
      for (int j = j0; j < j1; ++j) {
        const float rj = r[j];
        const float2 v = d[j];
        al = -rj * al;
        br = make_float2(rj * (v.x - br.x), rj * (v.y - br.y));
      }
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float a2 = __shfl_up_sync(0xffffffffu, al, o);
        const float bx = __shfl_up_sync(0xffffffffu, br.x, o), by = __shfl_up_sync(0xffffffffu, br.y, o);
        if (lane >= o) {
          br = make_float2(fmaf(al, bx, br.x), fmaf(al, by, br.y));
          al *= a2;
        }
      }
      float2 x = make_float2(__shfl_up_sync(0xffffffffu, br.x, 1), __shfl_up_sync(0xffffffffu, br.y, 1));
      if (lane == 0) x = make_float2(0.0f, 0.0f);
      al = 1.0f;
      br = make_float2(0.0f, 0.0f);
      for (int j = j0; j < j1; ++j) {
        const float rj = r[j];
        const float2 v = d[j];
        x = make_float2(rj * (v.x - x.x), rj * (v.y - x.y));
        d[j] = x;
        br = make_float2(fmaf(al, x.x, br.x), fmaf(al, x.y, br.y));
        al = -al * rj;
      }
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float a2 = __shfl_down_sync(0xffffffffu, al, o);
        const float bx = __shfl_down_sync(0xffffffffu, br.x, o), by = __shfl_down_sync(0xffffffffu, br.y, o);
        if (lane + o < 32) {
          br = make_float2(fmaf(al, bx, br.x), fmaf(al, by, br.y));
          al *= a2;
        }
      }
      x = make_float2(__shfl_down_sync(0xffffffffu, br.x, 1), __shfl_down_sync(0xffffffffu, br.y, 1));
      if (lane == 31) x = make_float2(0.0f, 0.0f);
      int o = j1 > j0 ? band_owner(j1 - 1, Ny) : 0, b0 = band_start(o, Ny);
      for (int j = j1 - 1; j >= j0; --j) {
        const float2 v = d[j];
        x = make_float2(fmaf(-r[j], x.x, v.x), fmaf(-r[j], x.y, v.y));
        if (j < b0) b0 = band_start(--o, Ny);  // (every band has a row)
        st_peer(peer_addr(spec + (j - b0) * (L + 2) + m, o), x);
      }
    }
  }
  cluster_sync();

  // ---- rows back: phi = mean + inverse transform.  The FP64 mean as a pair of
  // FP32 numbers: the sum rounds as the FP64 one (error of 4e6 random sums at
  // most 0.5 ulp in both, not one different).
  const float scale = 0.5f / (float)L;  // the halves and 1 / L
  for (int r = warp; r < nr; r += kWarps) {
    const float2* s = spec + r * (L + 2);
    float re[E], im[E];
#pragma unroll
    for (int j = 0; j < E; ++j) {
      const int k = lane + 32 * j;
      const float2 sk = (k == 0) ? make_float2(0.0f, 0.0f) : s[k], sp = s[L - k];
      const float Er = sk.x + sp.x, Ei = sk.y - sp.y, Dr = sk.x - sp.x, Di = sk.y + sp.y;
      const float Or = fmaf(Dr, wk[j].x, Di * wk[j].y), Oi = fmaf(Di, wk[j].x, -Dr * wk[j].y);
      re[j] = Er - Oi;
      im[j] = -(Ei + Or);
    }
    fft.run(re, im, lane);
    lane_fft_store<E>(re, im, rowbuf, lane);
    const ff b = ff_from(pb[r]);
    float2* out = reinterpret_cast<float2*>(phi + (size_t)(r0 + r) * Nx);
#pragma unroll
    for (int j = 0; j < E; ++j) {
      const float2 v = rowbuf[lpad(lane + 32 * j)];
      float hx, ex, hy, ey;
      two_sum_f(b.hi, v.x * scale, hx, ex);
      two_sum_f(b.hi, -v.y * scale, hy, ey);
      out[lane + 32 * j] = make_float2(hx + (ex + b.lo), hy + (ey + b.lo));
    }
    __syncwarp();
  }
}

// The cluster kernel of a grid, nullptr where it does not apply.
using Kernel = void (*)(int, unsigned, float, const float*, float*, Ptrs, PoissonArgs);
Kernel pick(int Nx, int Ny, size_t* smem) {
  if (Ny < kClusterCtas || (long long)Nx * Ny > (1LL << 18)) return nullptr;
  switch (Nx) {
    case 64: *smem = Lay<1>(Ny).bytes; return k_solve<1>;
    case 128: *smem = Lay<2>(Ny).bytes; return k_solve<2>;
    case 256: *smem = Lay<4>(Ny).bytes; return k_solve<4>;
    case 512: *smem = Lay<8>(Ny).bytes; return k_solve<8>;
  }
  return nullptr;
}
}  // namespace na

ehd_status na_fail(ehd_status st, const char* msg) {
  ehd::set_error(msg);
  return st;
}

}  // namespace

extern "C" ehd_status ehd_poisson_noalloc(int Nx, int Ny, double eps, double phi0, int wall_mode,
                                          const float* rhoc, float* phi, void* stream) {
  if (Nx < 16 || Nx > kMaxNx || (Nx & (Nx - 1)))
    return na_fail(EHD_EINVAL, "ehd_poisson_noalloc: Nx must be a power of two in [16, 2048]");
  if (Ny < 2 || Ny > kMaxNy) return na_fail(EHD_EINVAL, "ehd_poisson_noalloc: Ny must be in [2, 4096]");
  if (!(eps > 0)) return na_fail(EHD_EINVAL, "ehd_poisson_noalloc: eps must be positive");
  if (wall_mode != 0 && wall_mode != 1) return na_fail(EHD_EINVAL, "ehd_poisson_noalloc: wall_mode must be 0 or 1");
  if (!rhoc || !phi) return na_fail(EHD_EINVAL, "ehd_poisson_noalloc: rhoc and phi must be device pointers");
  const Layout L = layout_for(Nx, Ny);
  if (L.total > kScratchBytes)
    return na_fail(EHD_EINVAL,
                   "ehd_poisson_noalloc: this grid needs more than the 8 MiB static scratch "
                   "(about 1024 x 840 nodes is the largest channel that fits)");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) return na_fail(EHD_ECUDA, "ehd_poisson_noalloc: no CUDA device");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  std::lock_guard<std::mutex> lk(g_mu);
  DeviceSlot& slot = g_slots[dev];
  void* addr = nullptr;
  e = cudaGetSymbolAddress(&addr, g_scratch);
  if (e != cudaSuccess || !addr)
    return na_fail(EHD_ECUDA, "ehd_poisson_noalloc: cudaGetSymbolAddress of the static scratch failed");
  if (static_cast<unsigned char*>(addr) != slot.base) {
    // first call on this device, or the module was loaded again (e.g. after
    // cudaDeviceReset): nothing in the array can be trusted
    slot = DeviceSlot{};
    slot.base = static_cast<unsigned char*>(addr);
  }
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
    (void)cudaGetLastError();
    cap = cudaStreamCaptureStatusActive;  // unknown: take the safe path
  }
  if (cap != cudaStreamCaptureStatusNone) slot.always_rebuild = true;
  const Ptrs p = ptrs(slot.base, L);
  if (slot.always_rebuild || slot.Nx != Nx || slot.Ny != Ny || slot.wall_mode != wall_mode) {
    const int n = Nx / 2 + 1;
    k_na_tables<<<(n + 127) / 128, 128, 0, s>>>(Nx, Ny, wall_mode, p);
    if ((e = cudaGetLastError()) != cudaSuccess) return na_fail(EHD_ECUDA, "ehd_poisson_noalloc: table kernel launch failed");
    slot.Nx = Nx;
    slot.Ny = Ny;
    slot.wall_mode = wall_mode;
  }
  size_t smem = 0;
  na::Kernel kernel = na::pick(Nx, Ny, &smem);
  // rows are read and written as pairs
  if (kernel && ((reinterpret_cast<uintptr_t>(rhoc) | reinterpret_cast<uintptr_t>(phi)) & 7) == 0) {
    const int i = Nx == 64 ? 0 : Nx == 128 ? 1 : Nx == 256 ? 2 : 3;
    if (smem > slot.fits[i] && smem < slot.too_big[i]) {
      if (ehd::cluster_fits(kernel, na::kThreads, smem))
        slot.fits[i] = smem;
      else
        slot.too_big[i] = smem;
    }
    if (smem <= slot.fits[i]) {
      ehd::PoissonArgs pa{};
      pa.Nx = Nx;
      pa.Ny = Ny;
      pa.wall_mode = wall_mode;
      pa.mW = (double)Nx * phi0;
      pa.mC = (wall_mode == 0) ? 1.0 / (2.0 * Ny) : 1.0 / (double)(Ny + 1);
      cudaLaunchAttribute at[1];
      cudaLaunchConfig_t c;
      ehd::cluster_launch_config(&c, at, na::kThreads, smem, s);
      if (cudaLaunchKernelEx(&c, kernel, Ny, na::chunk_inverse(Ny), 0.5f * (float)(1.0 / eps), rhoc, phi, p, pa) != cudaSuccess)
        return na_fail(EHD_ECUDA, "ehd_poisson_noalloc: kernel launch failed");
      return EHD_OK;
    }
  }
  const size_t row_smem = 2 * (size_t)Nx * sizeof(Cplx<float>);
  k_na_fwd<<<Ny, 256, row_smem, s>>>(Nx, Ny, 1.0 / eps, rhoc, p);
  int wpc = (int)((48u * 1024u) / ((size_t)Ny * sizeof(Cplx<float>)));
  wpc = wpc < 1 ? 1 : (wpc > 4 ? 4 : wpc);
  k_na_modes<<<(Nx / 2 + 1 + wpc - 1) / wpc, 32 * wpc, (size_t)wpc * Ny * sizeof(Cplx<float>), s>>>(
      Nx, Ny, wall_mode, phi0, wpc, p);
  k_na_inv<<<Ny, 256, row_smem, s>>>(Nx, Ny, phi, p);
  if ((e = cudaGetLastError()) != cudaSuccess) return na_fail(EHD_ECUDA, "ehd_poisson_noalloc: kernel launch failed");
  return EHD_OK;
}
