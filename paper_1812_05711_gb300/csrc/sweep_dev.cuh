// sweep_dev.cuh -- the FP32 sweeps of a wavenumber's tridiagonal solve over one
// chunk of rows, with their rounding stated: the tile kernels (k_poisson.cu) and
// the on-chip form (k_resident.cu) give a run the same bits because both follow
// these, whatever a compiler makes of the loops around them.
#pragma once

namespace ehd {

// The chunk's forward map x -> al x + br composes, row by row,
//   al' = -r al,  br' = r (d - br),
// walked in groups of eight rows and, for the rows left over, of four, two and
// one.  Within a group the product of the row before is not rounded: d - br is
// one fused multiply-add (a shorter chain than multiply and subtract).  Row i of
// the `rem` < 8 rows left over:
__host__ __device__ constexpr bool tail_row_fused(int i, int rem) { return (i & 1) != 0 || (i == 2 && rem >= 4); }

struct ChunkMap {
  float al = 1.0f;
  float2 br = make_float2(0.0f, 0.0f);
  float2 df = make_float2(0.0f, 0.0f);  // the last row's difference and
  float rp = 0.0f;                       // pivot
  __device__ __forceinline__ void row(float r, float dx, float dy, bool fused) {
    al = -r * al;
    df = fused ? make_float2(fmaf(-rp, df.x, dx), fmaf(-rp, df.y, dy))
               : make_float2(__fsub_rn(dx, br.x), __fsub_rn(dy, br.y));
    br = make_float2(__fmul_rn(r, df.x), __fmul_rn(r, df.y));
    rp = r;
  }
};
// The map of n rows, pivot(k) and value(k) of row k.  Every group's loads go
// ahead of its chain, the last one's ahead of all (2048 x 300: 30.8 us per step
// against 31.4 with loads and chain row by row).
template <class P, class V>
__device__ __forceinline__ ChunkMap chunk_map(int n, P&& pivot, V&& value) {
  ChunkMap m;
  const int rem = n & 7, whole = n - rem;
  float r[8], dx[8], dy[8], rr[7], rx[7], ry[7];
#pragma unroll
  for (int i = 0; i < 7; ++i)
    if (i < rem) {
      rr[i] = pivot(whole + i);
      const auto v = value(whole + i);
      rx[i] = v.re;
      ry[i] = v.im;
    }
  for (int k = 0; k < whole; k += 8) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      r[i] = pivot(k + i);
      const auto v = value(k + i);
      dx[i] = v.re;
      dy[i] = v.im;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) m.row(r[i], dx[i], dy[i], i > 0);
  }
#pragma unroll
  for (int i = 0; i < 7; ++i)
    if (i < rem) m.row(rr[i], rx[i], ry[i], tail_row_fused(i, rem));
  return m;
}

// value of a row from the row before: r (d - x), both operations rounded
__device__ __forceinline__ float sweep_value(float r, float d, float x) { return __fmul_rn(r, __fsub_rn(d, x)); }
// back substitution d - r x, and the maps' composition al x + b: one rounding
__device__ __forceinline__ float sweep_back(float r, float d, float x) { return fmaf(-r, x, d); }
__device__ __forceinline__ double sweep_back(double r, double d, double x) { return d - r * x; }
__device__ __forceinline__ float map_apply(float al, float x, float b) { return fmaf(al, x, b); }
__device__ __forceinline__ double map_apply(double al, double x, double b) { return al * x + b; }

}  // namespace ehd
