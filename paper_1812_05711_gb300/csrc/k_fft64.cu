// k_fft64.cu -- row transforms of the plain FP64 path (Sec. IV.3 of
// arXiv:1812.05711, Eq. 19), rows of N = 16 ... 2048 reals.
//
// A row is packed as L = N / 2 complex values and transformed by a radix-4
// Stockham FFT, four values per thread (T = L / 4 threads), through two
// padded shared-memory buffers.
//
// What bounds them: scalar FP64 issues two lanes per clock and SM on this
// part, so both the number of FP64 instructions and the number of SMs that
// share them count.  Hence one row per CTA (rows below 128 values: as many
// as fill one warp) -- 128 x 104 runs on 52 SMs, where 16 rows per CTA left
// it to seven -- and per value
//   - the first stage without twiddles, straight from the loads;
//   - the row constant c0 (any value near the row's mean) taken out in the
//     same fused multiply-add that applies -1 / eps and every power-of-two
//     scale of both transforms (the stored spectrum is S / N); the m = 0
//     coefficient gets it back exactly as it was taken out;
//   - values k and L - k untangled together: 12 instructions a pair.
// The plain FP64 step has no charge plane: its forward transform sums the
// nine populations of each node as it loads them.
#include <type_traits>

#include "ehd_dev.cuh"

namespace ehd {

namespace {

__device__ __forceinline__ double2 cmul64(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 add64(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 sub64(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

template <int LG>
struct Row64 {
  static constexpr int L = 1 << LG, N = 2 * L, T = L / 4;
  static constexpr int kRows = T < 32 ? 32 / T : 1;  // rows per CTA
  static constexpr int kThreads = T * kRows;
  static constexpr int kPad = L + L / 8;              // one of padding every 8 values (128 bytes)
  static constexpr size_t kSmem = (size_t)2 * kRows * kPad * sizeof(double2);
};
__device__ __forceinline__ int pad64(int c) { return c + (c >> 3); }

// 4-point DFT of v, natural order (INV: the inverse sign)
template <bool INV>
__device__ __forceinline__ void dft4_64(double2 (&v)[4]) {
  const double2 t0 = add64(v[0], v[2]), t1 = sub64(v[0], v[2]), t2 = add64(v[1], v[3]), d = sub64(v[1], v[3]);
  const double2 t3 = INV ? make_double2(-d.y, d.x) : make_double2(d.y, -d.x);
  v[0] = add64(t0, t2);
  v[1] = add64(t1, t3);
  v[2] = sub64(t0, t2);
  v[3] = sub64(t1, t3);
}

// One radix-4 stage with sub-transform length NS and the ones after it; the
// last stage's values (t + q T in v[q]) are returned in registers.
template <int LG, bool INV, int NS>
__device__ __forceinline__ void stages64(double2 (&v)[4], double2* a, double2* b, const double2* __restrict__ tw,
                                         int t) {
  using C = Row64<LG>;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = a[pad64(t + q * C::T)];
  const int k = t & (NS - 1);
#pragma unroll
  for (int q = 1; q < 4; ++q) {
    double2 w = __ldg(tw + q * k * (C::N / (4 * NS)));
    if (INV) w.y = -w.y;
    v[q] = cmul64(v[q], w);
  }
  dft4_64<INV>(v);
  if constexpr (4 * NS < C::L) {
    const int idx = (t - k) * 4 + k;
#pragma unroll
    for (int q = 0; q < 4; ++q) b[pad64(idx + q * NS)] = v[q];
    stages64<LG, INV, 4 * NS>(v, b, a, tw, t);
  }
}

// Transform of the L values t + q T (in v[q]); returns the same positions of
// the result.  Row buffers a and b; a thread may still be reading either on
// return.
template <int LG, bool INV>
__device__ __forceinline__ void fft64(double2 (&v)[4], double2* a, double2* b, const double2* __restrict__ tw, int t) {
  using C = Row64<LG>;
  if constexpr (LG & 1) {  // radix 2, no twiddles: pairs (j, j + L / 2) for j = t and t + T
    const double2 a0 = add64(v[0], v[2]), a1 = sub64(v[0], v[2]), b0 = add64(v[1], v[3]), b1 = sub64(v[1], v[3]);
    a[pad64(2 * t)] = a0;
    a[pad64(2 * t + 1)] = a1;
    a[pad64(2 * (t + C::T))] = b0;
    a[pad64(2 * (t + C::T) + 1)] = b1;
    stages64<LG, INV, 2>(v, a, b, tw, t);
  } else {
    dft4_64<INV>(v);
#pragma unroll
    for (int q = 0; q < 4; ++q) a[pad64(4 * t + q)] = v[q];
    stages64<LG, INV, 4>(v, a, b, tw, t);
  }
}

}  // namespace

// Forward transform of -rho_c / eps (Eqs. 4, 19).  FROMG: rho_c is summed
// from the populations; else read from the charge plane (with the step
// kernel's slab-boundary partials).
template <int LG, bool FROMG>
__global__ void __launch_bounds__(Row64<LG>::kThreads) k_rfft64(PoissonArgs a) {
  using C = Row64<LG>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lr = threadIdx.x / C::T, t = threadIdx.x % C::T;
  const int y = blockIdx.x * C::kRows + lr;
  const bool live = y < a.Ny;
  double2* A = reinterpret_cast<double2*>(smem_raw) + (size_t)lr * 2 * C::kPad;
  double2* B = A + C::kPad;
  const double2* __restrict__ tw = static_cast<const double2*>(a.tw);
  grid_dep_wait();
  // -1 / eps, 1/2 of the untangling and 1 / N of the inverse
  const double s = -a.inv_eps * (0.5 / C::N);
  double2 v[4];
  double cs = 0.0;
  const long long row = (long long)(live ? y : 0) * a.P;
  if constexpr (FROMG) {
    const double* g = static_cast<const double*>(a.g) + row;
    cs = 2.25 * s * g[0];  // near the row's mean: g_0 is about 4/9 rho_c
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double* p = g + 2 * (t + q * C::T);
      double2 r = *reinterpret_cast<const double2*>(p);
#pragma unroll
      for (int i = 1; i < 9; ++i) r = add64(r, *reinterpret_cast<const double2*>(p + i * a.gplane));
      v[q] = make_double2(fma(r.x, s, -cs), fma(r.y, s, -cs));
    }
  } else {
    const double* rc = static_cast<const double*>(a.rhoc) + row;
    const double *rdn, *rup;
    rhoc_partials<double>(a, live ? y : 0, rdn, rup);
    cs = s * rc[0];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int n = t + q * C::T;
      double2 r = reinterpret_cast<const double2*>(rc)[n];
      if (rdn) r = add64(r, reinterpret_cast<const double2*>(rdn)[n]);
      if (rup) r = add64(r, reinterpret_cast<const double2*>(rup)[n]);
      v[q] = make_double2(fma(r.x, s, -cs), fma(r.y, s, -cs));
    }
  }
  fft64<LG, false>(v, A, B, tw, t);
  // the last stage was read from one of the buffers: all threads are past it
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) A[pad64(t + q * C::T)] = v[q];
  __syncthreads();
  if (!live) return;
  // S[k] = E + W^k D / i with E = Z[k] + Z*[L - k], D = Z[k] - Z*[L - k] (the
  // halves are in the scale); for L - k: conj(E), -conj(D) and -conj(W^k)
  double2* spec = static_cast<double2*>(a.spec) + (long long)y * a.Mp;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int k = t + h * C::T;  // 0 .. L / 2 - 1
    const double2 zk = A[pad64(k)], zp = A[pad64((C::L - k) & (C::L - 1))];
    if (k == 0) {
      static_cast<double*>(a.spec0)[y] = (2.0 * C::N) * fma((double)C::N, cs, zk.x + zk.y);
      spec[0] = make_double2(0.0, 0.0);
      spec[C::L] = make_double2(2.0 * (zk.x - zk.y), 0.0);  // Nyquist
      const double2 zm = A[pad64(C::L / 2)];                 // its own partner
      spec[C::L / 2] = make_double2(2.0 * zm.x, -2.0 * zm.y);
    } else {
      const double2 w = __ldg(tw + k);
      const double Er = zk.x + zp.x, Ei = zk.y - zp.y, Dr = zk.x - zp.x, Di = zk.y + zp.y;
      spec[k] = make_double2(fma(w.x, Di, fma(w.y, Dr, Er)), fma(w.y, Di, fma(-w.x, Dr, Ei)));
      spec[C::L - k] = make_double2(fma(-w.x, Di, fma(-w.y, Dr, Er)), fma(w.y, Di, fma(-w.x, Dr, -Ei)));
    }
  }
}

// Inverse transform -> phi minus its row mean (DX: E_x, the transform of
// -i k_m phi_m with the Nyquist coefficient dropped).
template <int LG, bool DX>
__global__ void __launch_bounds__(Row64<LG>::kThreads) k_irfft64(PoissonArgs a) {
  using C = Row64<LG>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lr = threadIdx.x / C::T, t = threadIdx.x % C::T;
  const int y = blockIdx.x * C::kRows + lr;
  const bool live = y < a.Ny;
  double2* A = reinterpret_cast<double2*>(smem_raw) + (size_t)lr * 2 * C::kPad;
  double2* B = A + C::kPad;
  const double2* __restrict__ tw = static_cast<const double2*>(a.tw);
  double2 w[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) w[h] = __ldg(tw + t + h * C::T);
  grid_dep_wait();
  const double2* spec = static_cast<const double2*>(a.spec) + (long long)(live ? y : 0) * a.Mp;
  auto coef = [&](int k) {
    const double2 c = spec[k];
    if constexpr (!DX) {
      return c;
    } else {
      if (k == C::L) return make_double2(0.0, 0.0);
      const double kk = (3.141592653589793238462643383279502884 / C::L) * (double)k;
      return make_double2(kk * c.y, -kk * c.x);
    }
  };
  // Z[k] = E + i O, Z[L - k] = conj(E) + i conj(O), E = S[k] + S*[L - k],
  // O = (S[k] - S*[L - k]) / W^k; the mean S[0] is left out
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int k = t + h * C::T;
    const double2 sp = coef(C::L - k), sk = (k == 0) ? make_double2(0.0, 0.0) : coef(k);
    const double Er = sk.x + sp.x, Ei = sk.y - sp.y, Dr = sk.x - sp.x, Di = sk.y + sp.y;
    const double Or = fma(Dr, w[h].x, Di * w[h].y), Oi = fma(Di, w[h].x, -Dr * w[h].y);
    A[pad64(k)] = make_double2(Er - Oi, Ei + Or);
    if (k > 0) {
      A[pad64(C::L - k)] = make_double2(Er + Oi, Or - Ei);
    } else {
      const double2 sm = coef(C::L / 2);
      A[pad64(C::L / 2)] = make_double2(2.0 * sm.x, -2.0 * sm.y);
    }
  }
  __syncthreads();
  double2 v[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = A[pad64(t + q * C::T)];
  fft64<LG, true>(v, B, A, tw, t);
  if (!live) return;
  double2* out = reinterpret_cast<double2*>(static_cast<double*>(DX ? a.ex : a.dphi) + (long long)y * a.P);
#pragma unroll
  for (int q = 0; q < 4; ++q) out[t + q * C::T] = v[q];
}

namespace {
template <int LG>
cudaError_t rfft64_n(const PoissonArgs& a, cudaStream_t s) {
  using C = Row64<LG>;
  const dim3 grid((a.Ny + C::kRows - 1) / C::kRows), block(C::kThreads);
  const bool pdl = (a.pdl & 1) != 0;
  return a.g ? launch_ex(pdl, k_rfft64<LG, true>, grid, block, C::kSmem, s, a)
             : launch_ex(pdl, k_rfft64<LG, false>, grid, block, C::kSmem, s, a);
}
template <int LG, bool DX>
cudaError_t irfft64_n(const PoissonArgs& a, cudaStream_t s) {
  using C = Row64<LG>;
  return launch_ex((a.pdl & 4) != 0, k_irfft64<LG, DX>, dim3((a.Ny + C::kRows - 1) / C::kRows), dim3(C::kThreads),
                   C::kSmem, s, a);
}
template <class F>
cudaError_t by_row64(int Nx, F&& f) {
  switch (Nx) {
    case 16: return f(std::integral_constant<int, 3>());
    case 32: return f(std::integral_constant<int, 4>());
    case 64: return f(std::integral_constant<int, 5>());
    case 128: return f(std::integral_constant<int, 6>());
    case 256: return f(std::integral_constant<int, 7>());
    case 512: return f(std::integral_constant<int, 8>());
    case 1024: return f(std::integral_constant<int, 9>());
    case 2048: return f(std::integral_constant<int, 10>());
  }
  return cudaErrorInvalidValue;
}
}  // namespace

cudaError_t launch_rfft64(const PoissonArgs& a, cudaStream_t s) {
  return by_row64(a.Nx, [&](auto lg) { return rfft64_n<lg.value>(a, s); });
}
cudaError_t launch_irfft64(const PoissonArgs& a, bool dx, cudaStream_t s) {
  return by_row64(a.Nx, [&](auto lg) { return dx ? irfft64_n<lg.value, true>(a, s) : irfft64_n<lg.value, false>(a, s); });
}

}  // namespace ehd
