// fft_dev.cuh -- device pieces of the FP32 row transforms, shared by the
// kernels that transform rows (k_fftw.cu) and the one that keeps a whole run
// on chip (k_resident.cu).
#pragma once

#include "ehd_dev.cuh"

namespace ehd {

// exp(-2 pi i k / 32) and exp(-2 pi i k / 64) rounded to FP32.  The tables are
// part of the module's image: nothing has to be copied before a kernel that
// reads them may run.
#define EHD_W32 \
  {1.0f, -0.0f}, {0.980785251f, -0.195090324f}, {0.923879504f, -0.382683426f}, {0.831469595f, -0.555570245f}, \
  {0.707106769f, -0.707106769f}, {0.555570245f, -0.831469595f}, {0.382683426f, -0.923879504f}, \
  {0.195090324f, -0.980785251f}, {6.12323426e-17f, -1.0f}, {-0.195090324f, -0.980785251f}, \
  {-0.382683426f, -0.923879504f}, {-0.555570245f, -0.831469595f}, {-0.707106769f, -0.707106769f}, \
  {-0.831469595f, -0.555570245f}, {-0.923879504f, -0.382683426f}, {-0.980785251f, -0.195090324f}, \
  {-1.0f, -1.22464685e-16f}, {-0.980785251f, 0.195090324f}, {-0.923879504f, 0.382683426f}, \
  {-0.831469595f, 0.555570245f}, {-0.707106769f, 0.707106769f}, {-0.555570245f, 0.831469595f}, \
  {-0.382683426f, 0.923879504f}, {-0.195090324f, 0.980785251f}, {-1.83697015e-16f, 1.0f}, \
  {0.195090324f, 0.980785251f}, {0.382683426f, 0.923879504f}, {0.555570245f, 0.831469595f}, \
  {0.707106769f, 0.707106769f}, {0.831469595f, 0.555570245f}, {0.923879504f, 0.382683426f}, \
  {0.980785251f, 0.195090324f}
#define EHD_W64 \
  {1.0f, -0.0f}, {0.99518472f, -0.0980171412f}, {0.980785251f, -0.195090324f}, {0.956940353f, -0.290284663f}, \
  {0.923879504f, -0.382683426f}, {0.881921291f, -0.471396744f}, {0.831469595f, -0.555570245f}, \
  {0.773010433f, -0.634393275f}, {0.707106769f, -0.707106769f}, {0.634393275f, -0.773010433f}, \
  {0.555570245f, -0.831469595f}, {0.471396744f, -0.881921291f}, {0.382683426f, -0.923879504f}, \
  {0.290284663f, -0.956940353f}, {0.195090324f, -0.980785251f}, {0.0980171412f, -0.99518472f}, \
  {6.12323426e-17f, -1.0f}, {-0.0980171412f, -0.99518472f}, {-0.195090324f, -0.980785251f}, \
  {-0.290284663f, -0.956940353f}, {-0.382683426f, -0.923879504f}, {-0.471396744f, -0.881921291f}, \
  {-0.555570245f, -0.831469595f}, {-0.634393275f, -0.773010433f}, {-0.707106769f, -0.707106769f}, \
  {-0.773010433f, -0.634393275f}, {-0.831469595f, -0.555570245f}, {-0.881921291f, -0.471396744f}, \
  {-0.923879504f, -0.382683426f}, {-0.956940353f, -0.290284663f}, {-0.980785251f, -0.195090324f}, \
  {-0.99518472f, -0.0980171412f}, {-1.0f, -1.22464685e-16f}, {-0.99518472f, 0.0980171412f}, \
  {-0.980785251f, 0.195090324f}, {-0.956940353f, 0.290284663f}, {-0.923879504f, 0.382683426f}, \
  {-0.881921291f, 0.471396744f}, {-0.831469595f, 0.555570245f}, {-0.773010433f, 0.634393275f}, \
  {-0.707106769f, 0.707106769f}, {-0.634393275f, 0.773010433f}, {-0.555570245f, 0.831469595f}, \
  {-0.471396744f, 0.881921291f}, {-0.382683426f, 0.923879504f}, {-0.290284663f, 0.956940353f}, \
  {-0.195090324f, 0.980785251f}, {-0.0980171412f, 0.99518472f}, {-1.83697015e-16f, 1.0f}, \
  {0.0980171412f, 0.99518472f}, {0.195090324f, 0.980785251f}, {0.290284663f, 0.956940353f}, \
  {0.382683426f, 0.923879504f}, {0.471396744f, 0.881921291f}, {0.555570245f, 0.831469595f}, \
  {0.634393275f, 0.773010433f}, {0.707106769f, 0.707106769f}, {0.773010433f, 0.634393275f}, \
  {0.831469595f, 0.555570245f}, {0.881921291f, 0.471396744f}, {0.923879504f, 0.382683426f}, \
  {0.956940353f, 0.290284663f}, {0.980785251f, 0.195090324f}, {0.99518472f, 0.0980171412f}
static __constant__ float2 c_w32[32] = {EHD_W32};  // for indices known at compile time
static __constant__ float2 c_w64[64] = {EHD_W64};
static __device__ float2 g_w64[64] = {EHD_W64};  // for lane-dependent ones
#undef EHD_W32
#undef EHD_W64

__host__ __device__ constexpr int bitrev(int i, int n) {
  int r = 0;
  for (int b = 1; b < n; b <<= 1) {
    r = (r << 1) | (i & 1);
    i >>= 1;
  }
  return r;
}

// in-register radix-2 FFT of length M <= 32 (forward, natural order in/out);
// every index is a compile-time constant so the arrays stay in registers
template <int M, int LEN>
struct FftStage {
  __device__ __forceinline__ static void run(float (&re)[M], float (&im)[M]) {
#pragma unroll
    for (int b = 0; b < M / LEN; ++b) {
#pragma unroll
      for (int k = 0; k < LEN / 2; ++k) {
        const float2 w = c_w32[k * (32 / LEN)];
        const int u = b * LEN + k, v = u + LEN / 2;
        // cmf0, without the multiplications by W^0 = 1 (an eighth to a half of
        // them: with the rounding stated, 1024 x 840 BF16 35.3 us per step
        // against 36.0)
        const float tr = k == 0 ? re[v] : fmaf(re[v], w.x, -(im[v] * w.y));
        const float ti = k == 0 ? im[v] : fmaf(re[v], w.y, im[v] * w.x);
        // the pair's sum and difference as packed two-float adds
        const float2 a = make_float2(re[u], im[u]);
        const float2 lo = __fadd2_rn(a, make_float2(-tr, -ti)), hi = __fadd2_rn(a, make_float2(tr, ti));
        re[v] = lo.x;
        im[v] = lo.y;
        re[u] = hi.x;
        im[u] = hi.y;
      }
    }
    FftStage<M, LEN * 2>::run(re, im);
  }
};
template <int M>
struct FftStage<M, M * 2> {
  __device__ __forceinline__ static void run(float (&)[M], float (&)[M]) {}
};

template <int M>
__device__ __forceinline__ void fft_reg(float (&re)[M], float (&im)[M]) {
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const int j = bitrev(i, M);
    if (j > i) {
      const float tr = re[i], ti = im[i];
      re[i] = re[j];
      im[i] = im[j];
      re[j] = tr;
      im[j] = ti;
    }
  }
  FftStage<M, 2>::run(re, im);
}

__device__ __forceinline__ float2 cm(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// The same product with its rounding stated: which product of the imaginary
// part is rounded before the fused multiply-add.
__device__ __forceinline__ float2 cmf0(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -(a.y * b.y)), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cmf1(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -(a.y * b.y)), fmaf(a.y, b.x, a.x * b.y));
}

__device__ __forceinline__ void two_sum_f(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// the first stage's twiddles of lane n1: powers of W_N^(2 n1), resynchronised
// from the table every 4 steps
template <int E>
__device__ __forceinline__ void four_step_twiddles(const float2* __restrict__ tw, int lane, float2 (&w)[E]) {
  constexpr int N = 64 * E;
  const float2 base = tw[(2 * lane) & (N - 1)];
  float2 c = make_float2(1.0f, 0.0f);
#pragma unroll
  for (int k2 = 0; k2 < E; ++k2) {
    if (k2 > 0) c = ((k2 & 3) == 0) ? tw[(2 * lane * k2) & (N - 1)] : k2 == 1 ? base : cmf0(c, base);
    w[k2] = c;
  }
}

// ---------------------------------------------------------------------------
// One row of N = 64 E reals (L = 32 E complex values, E <= 8) by one warp with
// every lane at work in every stage.  The four-step factorisation of
// k_fftw.cu, L = 32 x E: lane n1 transforms its E values over n2, multiplies
// by W_L^(n1 k2), and for each k2 the 32 lanes hold one value each of a
// 32-point transform over n1, which runs across the lanes: position p =
// bitrev(lane) of the radix-2 network, so its five stages exchange with lane
// xor 16, 8, 4, 2, 1.  The butterflies are those of fft_reg, value for value.
// (With the 32-point transforms in registers of E lanes, the other lanes only
// repeated them: for E = 2 a warp issued 640 instructions where 110 do.)
// On return (re[k2], im[k2]) of a lane is X[k2 + E bitrev(lane)].
//
// Every product sum here and in the wide transforms (rfft_warp_rows,
// irfft_warp_rows in k_fftw.cu) is written with its fused multiply-add, so that
// a row has the same bits in every kernel that transforms it: the step of one
// node per thread sends rows of 1024 through LaneFft, the march form and the
// batch through the wide form.
// LIT: the E-point transform by literal factors (fft_lit), for a kernel that
// owes no other its bits.
template <int E>
__device__ __forceinline__ void fft_lit(float (&re)[E], float (&im)[E]) {
  if constexpr (E == 2) {
    const float r = re[0], i = im[0];
    re[0] = r + re[1];
    im[0] = i + im[1];
    re[1] = r - re[1];
    im[1] = i - im[1];
  } else if constexpr (E > 2) {  // even and odd halves, then W_E^k
    float er[E / 2], ei[E / 2], orr[E / 2], oi[E / 2];
#pragma unroll
    for (int k = 0; k < E / 2; ++k) {
      er[k] = re[2 * k];
      ei[k] = im[2 * k];
      orr[k] = re[2 * k + 1];
      oi[k] = im[2 * k + 1];
    }
    fft_lit<E / 2>(er, ei);
    fft_lit<E / 2>(orr, oi);
    constexpr float h = 0.70710678118654752440f;
#pragma unroll
    for (int k = 0; k < E / 2; ++k) {
      // W_E^k for E = 4 and 8: k (8 / E) eighths of a turn
      const int q = k * (8 / E);
      const float c = q == 0 ? 1.0f : (q == 1 ? h : (q == 2 ? 0.0f : -h));
      const float s = q == 0 ? 0.0f : (q == 2 ? -1.0f : -h);
      const float tr = orr[k] * c - oi[k] * s, ti = orr[k] * s + oi[k] * c;
      re[k] = er[k] + tr;
      im[k] = ei[k] + ti;
      re[k + E / 2] = er[k] - tr;
      im[k + E / 2] = ei[k] - ti;
    }
  }
}
template <int E, bool LIT = false>
struct LaneFft {
  float2 w[E];   // W_L^(lane k2)
  float2 ws[5];  // this lane's butterfly factor in each stage
  __device__ __forceinline__ void init(const float2* __restrict__ tw, int lane) {
    // as four_step_twiddles
    const float2 base = tw[(2 * lane) & (64 * E - 1)];
    w[0] = make_float2(1.0f, 0.0f);
#pragma unroll
    for (int k2 = 1; k2 < E; ++k2)
      w[k2] = k2 == 1 ? base : ((k2 & 3) == 0) ? tw[(2 * lane * k2) & (64 * E - 1)] : cmf0(w[k2 - 1], base);
    init_stages(lane);
  }
  __device__ __forceinline__ void init_stages(int lane) {
    const int p = __brev((unsigned)lane) >> 27;
#pragma unroll
    for (int s = 0; s < 5; ++s) {
      const int len = 2 << s;
      ws[s] = g_w64[2 * (p & (len / 2 - 1)) * (32 / len)];
    }
  }
  __device__ __forceinline__ void run(float (&re)[E], float (&im)[E], int lane) const {
    if constexpr (LIT)
      fft_lit<E>(re, im);
    else
      fft_reg<E>(re, im);
#pragma unroll
    for (int k2 = 0; k2 < E; ++k2) {
      const float2 v = cmf1(make_float2(re[k2], im[k2]), w[k2]);
      re[k2] = v.x;
      im[k2] = v.y;
    }
#pragma unroll
    for (int s = 0; s < 5; ++s) {
      const int m = 16 >> s;
      const bool up = (lane & m) != 0;  // the pair's second element: times the factor, then u - w v
      const float sg = up ? -1.0f : 1.0f;
#pragma unroll
      for (int k2 = 0; k2 < E; ++k2) {
        const float2 t = cmf0(make_float2(re[k2], im[k2]), ws[s]);
        const float vr = up ? t.x : re[k2], vi = up ? t.y : im[k2];
        const float ur = __shfl_xor_sync(0xffffffffu, vr, m), ui = __shfl_xor_sync(0xffffffffu, vi, m);
        re[k2] = fmaf(sg, vr, ur);
        im[k2] = fmaf(sg, vi, ui);
      }
    }
  }
};
// shared-memory index of value k: one float2 of padding every 16
__device__ __forceinline__ int lpad(int k) { return k + (k >> 4); }
template <int E>
constexpr int kLaneRow = 32 * E + 2 * E;  // float2 per row buffer

// The transform's values into the row buffer in natural order.
template <int E>
__device__ __forceinline__ void lane_fft_store(const float (&re)[E], const float (&im)[E], float2* sm, int lane) {
  const int p = __brev((unsigned)lane) >> 27;
#pragma unroll
  for (int k2 = 0; k2 < E; ++k2) sm[lpad(k2 + E * p)] = make_float2(re[k2], im[k2]);
  __syncwarp();
}

// Untangling factors of the forward transform, W_N^k for k = lane + 32 j.
template <int E>
__device__ __forceinline__ void untangle_factors(const float2* __restrict__ tw, int lane, float2 (&wk)[E]) {
#pragma unroll
  for (int j = 0; j < E; ++j) {
    const int k = lane + 32 * j;
    wk[j] = cmf1(tw[k & (E - 1)], g_w64[k / E]);
  }
}
// Half-spectrum value S[k], k = lane + 32 j (k >= 1), of the row in the buffer
template <int E>
__device__ __forceinline__ float2 untangle(const float2* sm, int k, float2 wk) {
  constexpr int L = 32 * E;
  const float2 zk = sm[lpad(k)], zp = sm[lpad((L - k) & (L - 1))];
  const float2 zc = make_float2(zp.x, -zp.y);
  const float2 Ev = make_float2(0.5f * (zk.x + zc.x), 0.5f * (zk.y + zc.y));
  const float2 Dv = make_float2(0.5f * (zk.x - zc.x), 0.5f * (zk.y - zc.y));
  const float2 O = make_float2(Dv.y, -Dv.x);
  const float2 wO = cmf0(wk, O);
  return make_float2(Ev.x + wO.x, Ev.y + wO.y);
}
// The m = 0 coefficient in float-float: (Re Z0 + Im Z0) + N c0 (-1 / eps), the
// product exact by the FMA two-product, N a power of two.
__device__ __forceinline__ float2 mean_coefficient(float2 z0, float c0, float nieps, float N) {
  float s, e;
  two_sum_f(z0.x, z0.y, s, e);
  const float p = c0 * nieps, pe = fmaf(c0, nieps, -p);
  const float P = p * N, PE = pe * N;
  float h, l;
  two_sum_f(s, P, h, l);
  l += e + PE;
  two_sum_f(h, l, s, e);
  return make_float2(s, e);
}
// conj(Z[k]) of the inverse's packed spectrum from S[k] and S[L - k] (S[0]
// taken as 0): Z[k] = E_k + i O_k, E_k = (S[k] + S*[L-k]) / 2,
// O_k = (S[k] - S*[L-k]) / (2 W_N^k)
__device__ __forceinline__ float2 entangle(float2 sk, float2 sp, float2 wk) {
  const float2 sc = make_float2(sp.x, -sp.y);
  const float2 Ev = make_float2(0.5f * (sk.x + sc.x), 0.5f * (sk.y + sc.y));
  const float2 Dv = make_float2(0.5f * (sk.x - sc.x), 0.5f * (sk.y - sc.y));
  const float2 O = cmf1(Dv, make_float2(wk.x, -wk.y));  // D / W^k
  return make_float2(Ev.x - O.y, -(Ev.y + O.x));      // Re(E + i O), -Im: conjugate
}

}  // namespace ehd
