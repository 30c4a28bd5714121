// sdpd_f64.cuh -- float64 arithmetic with few float64 instructions: elementary
// functions, and the pieces shared by the float64 pair passes (density,
// forces, reverse passes).
#pragma once
#include "sdpd_internal.cuh"

namespace sdpd {

// Elementary functions with few float64 instructions.  Each starts from a
// hardware approximation or a float32 evaluation of its small terms.
namespace f64 {
// Conversions on the integer pipe (a conversion instruction costs a float64
// issue): |x| truncated to float32, 0 below float32's normal range (|x| must
// be below 2^127), and a non-negative float32 to float64 (0 becomes 2^-127).
__device__ __forceinline__ float trunc_abs(double x) {
  const int hi = max(__double2hiint(x) & 0x7fffffff, 0x38000000) - 0x38000000;
  return __int_as_float(hi << 3 | (int)((unsigned)__double2loint(x) >> 29));
}
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f);
  return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}
__device__ __forceinline__ double widen_signed(float f) {
  const unsigned u = __float_as_uint(f);
  return __hiloint2double((int)((((u & 0x7fffffffu) >> 3) + 0x38000000u) | (u & 0x80000000u)), (int)(u << 29));
}
__device__ __forceinline__ double rcp_seed(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}
__device__ __forceinline__ double rsqrt_seed(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}
// 1/x: one third-order (Householder) step y (1 + e + e^2), e = 1 - x y.
__device__ __forceinline__ double rcp(double x) {
  const double y = rcp_seed(x), e = __fma_rn(-x, y, 1.0);
  return __fma_rn(y, __fma_rn(e, e, e), y);
}
// sqrt(x) and 1/sqrt(x): one third-order step, (1 - e)^(-1/2) =
// 1 + e/2 + 3 e^2/8 + O(e^3) with e = 1 - x y^2.  The reciprocal root takes the
// seed's upper 21 bits, whose square is exact, so that e has one rounding (0.58
// ulp; e from a rounded x y: 1.01, 1 / sqrt: 1.49).  Arguments whose seed could
// be flushed take the library functions.
__device__ __forceinline__ bool rsqrt_tiny(double x) { return __double2hiint(x) < 0x03f00000; }  // below 2^-960, <= 0
__device__ __forceinline__ double sqrt_(double x) {
  if (rsqrt_tiny(x)) return ::sqrt(x);
  const double y = rsqrt_seed(x), h = __dmul_rn(x, y), e = __fma_rn(-h, y, 1.0);
  return __fma_rn(__dmul_rn(h, e), __fma_rn(e, 0.375, 0.5), h);
}
__device__ __forceinline__ double rsqrt_(double x) {
  if (rsqrt_tiny(x)) return ::rsqrt(x);
  const double y = __hiloint2double(__double2hiint(rsqrt_seed(x)), 0), e = __fma_rn(-x, __dmul_rn(y, y), 1.0);
  return __fma_rn(__dmul_rn(y, e), __fma_rn(e, 0.375, 0.5), y);
}
__device__ __forceinline__ bool below(double x, int hi) { return (__double2hiint(x) & 0x7fffffff) < hi; }
constexpr int kHi2m6 = 0x3f900000, kHi2m3 = 0x3fc00000, kHi2m2 = 0x3fd00000;  // high words of 2^-6, 1/8, 1/4
// expm1: Taylor series; below 2^-6 the terms from x^6/720 on, 2^-39 of the
// result, in float32; below 1/4 those from x^9/362880 on, 2^-34 of it.  Within
// 0.51, 0.54, 0.58 and 0.65 ulp up to 2^-6, 2^-4, 1/8 and 1/4, as the
// library's function is.
__device__ __forceinline__ double expm1(double x) {
  if (below(x, kHi2m2)) {
    const float f = copysignf(trunc_abs(x), __int_as_float(__double2hiint(x)));
    double p;
    if (below(x, kHi2m6)) {
      const float t = f * (1.0f / 720.0f + f * (1.0f / 5040.0f + f * (1.0f / 40320.0f)));
      p = 1.0 / 120.0 + widen_signed(t);
    } else {
      const float t =
          f * (1.0f / 362880.0f +
               f * (1.0f / 3628800.0f +
                    f * (1.0f / 39916800.0f + f * (1.0f / 479001600.0f + f * (1.0f / 6227020800.0f)))));
      p = 1.0 / 40320.0 + widen_signed(t);
      p = __fma_rn(p, x, 1.0 / 5040.0);
      p = __fma_rn(p, x, 1.0 / 720.0);
      p = __fma_rn(p, x, 1.0 / 120.0);
    }
    p = __fma_rn(p, x, 1.0 / 24.0);
    p = __fma_rn(p, x, 1.0 / 6.0);
    p = __fma_rn(p, x, 0.5);
    return __fma_rn(__dmul_rn(p, x), x, x);
  }
  return ::expm1(x);
}
// log1p: below 2^-6 the alternating series, its terms from x^7/7 on (2^-39 of
// the result) in float32; below 1/8 2 atanh(u) with u = x / (2 + x) and the
// rounding errors of the sum and the quotient carried along, its terms from
// u^9/9 on (2^-34 of it) in float32.  Within 0.53 ulp (the library's
// function: 0.52 below 2^-6, 0.66 below 1/8).
__device__ __forceinline__ double log1p(double x) {
  if (below(x, kHi2m6)) {
    const float f = copysignf(trunc_abs(x), __int_as_float(__double2hiint(x)));
    const float t = f * (1.0f / 7.0f + f * (-1.0f / 8.0f + f * (1.0f / 9.0f + f * (-1.0f / 10.0f))));
    double p = -1.0 / 6.0 + widen_signed(t);
    p = __fma_rn(p, x, 0.2);
    p = __fma_rn(p, x, -0.25);
    p = __fma_rn(p, x, 1.0 / 3.0);
    p = __fma_rn(p, x, -0.5);
    return __fma_rn(__dmul_rn(p, x), x, x);
  }
  if (below(x, kHi2m3)) {
    const double d = __dadd_rn(2.0, x), dl = __dadd_rn(x, -__dadd_rn(d, -2.0));  // d + dl = 2 + x
    const double r = rcp(d), u = __dmul_rn(x, r);
    const double ul = __dmul_rn(__fma_rn(-u, dl, __fma_rn(-u, d, x)), r);  // u + ul: the quotient
    const double w = __dmul_rn(u, u);
    const float f = trunc_abs(w);
    const float t = f * (1.0f / 9.0f + f * (1.0f / 11.0f + f * (1.0f / 13.0f + f * (1.0f / 15.0f))));
    double p = 1.0 / 7.0 + widen(t);
    p = __fma_rn(p, w, 0.2);
    p = __fma_rn(p, w, 1.0 / 3.0);
    const double v = __dadd_rn(u, __fma_rn(__dmul_rn(p, w), u, ul));
    return __dadd_rn(v, v);
  }
  return ::log1p(x);
}
// comparisons with zero on the bits (a float64 comparison costs an issue)
__device__ __forceinline__ bool positive(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool negative(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return b > 0x8000000000000000ull && b <= 0xfff0000000000000ull;
}
}  // namespace f64

// ---------------------------------------------------------------------------
// Float64 pair passes.  GB300 issues one float64 instruction per 64 cycles on
// each quarter of an SM whether 1 or 32 lanes are active, so a pass costs its
// float64 instructions per warp.  With one thread per particle the kept
// neighbour's branch ran on nearly every candidate of the 27 cells (one lane
// in six keeps one): ~500 evaluations instead of ~80.  Here kLanes64 lanes
// share a particle (a whole warp where particles are few).  The search is
// float32: r^2 from the float32 positions decides a candidate unless it lies
// within its rounding bound of h^2 (then the float64 predicate does), and the
// kept ones are appended in walk order (ballot and prefix count) to a list in
// shared memory.  Only list entries see float64 arithmetic, with all lanes at
// work.
// ---------------------------------------------------------------------------
constexpr int kLanes64 = 8;

// r of r^2: y = 1/sqrt(r^2) and the root H = r^2 y in float32, then
// H + (r^2 - H^2) y / 2 with float64 only in the residual and the sum (Heron's
// step; the error is about the product of those of H and y).  y takes a Newton
// step in float32, which costs no float64 issue: 1.4e-14 relative at most (rms
// 2.0e-15) instead of 3.7e-14 (3.7e-15); the float64 Newton step of pair_r has
// 3.2e-14 (3.5e-15).  r^2 outside float32's range takes the library square root.
__device__ __forceinline__ double pair_r64(double r2) {
  const float f = f64::trunc_abs(r2);
  if (!(f > 1e-30f)) return sqrt(r2);
  float y = rsqrtf(f);
  y = __fmaf_rn(0.5f * y, __fmaf_rn(-f * y, y, 1.0f), y);
  const double H = f64::widen(f * y);
  return __fma_rn(__fma_rn(-H, H, r2), f64::widen(0.5f * y), H);
}
// The same with a second Heron step, and 1/r = y (1 + e + e^2), e = 1 - r y,
// y in float32.
__device__ __forceinline__ double pair_r64(double r2, double& rinv) {
  const float f = f64::trunc_abs(r2);
  if (!(f > 1e-30f)) {
    const double r = sqrt(r2);
    rinv = r2 > 0.0 ? 1.0 / r : 0.0;
    return r;
  }
  const float y = rsqrtf(f);
  const double H = f64::widen(f * y), yd = f64::widen(y);
  const double yh = f64::widen(0.5f * y);
  double r = __fma_rn(__fma_rn(-H, H, r2), yh, H);
  r = __fma_rn(__fma_rn(-r, r, r2), yh, r);
  const double e = __fma_rn(-r, yd, 1.0);
  rinv = __fma_rn(yd, __fma_rn(e, e, e), yd);
  return r;
}

// W / cW, F / cF and h F' / cF at distance r (see kernel_W, kernel_F), without
// float64 comparisons or divisions.
__device__ __forceinline__ bool inner_half(double x) { return __double_as_longlong(x) <= 0x3fe0000000000000ll; }
template <int KIND>
__device__ __forceinline__ double W64(double r, double inv_h) {
  if (KIND == SDPD_KERNEL_LUCY) {
    const double y = __fma_rn(-r, inv_h, 1.0);
    return __fma_rn(-3.0, y, 4.0) * (y * y * y);
  }
  const double x = r * inv_h, y = 1.0 - x;
  const bool in = inner_half(x);
  const double q = in ? x : y;
  return __fma_rn(in ? -6.0 : 2.0, q * q * y, in ? 1.0 : 0.0);
}
template <int KIND>
__device__ __forceinline__ double F64(double r, double inv_h) {
  if (KIND == SDPD_KERNEL_LUCY) {
    const double y = __fma_rn(-r, inv_h, 1.0);
    return y * y;
  }
  const double x = r * inv_h, y = 1.0 - x;
  return inner_half(x) ? __fma_rn(-3.0, x, 2.0) : y * y * f64::rcp(x);
}

// Displacement to a float64 list entry with the periodic image of its stencil
// code.  wraps: bit `code` set where the home cell's neighbour of that code
// lies across the box side (else every image shift is zero).
struct Home64 {
  double x, y, z;
  double mx, my, mz, px_, py_, pz_;
  unsigned long long wraps;
  __device__ __forceinline__ void init(const Consts& c, const D4& q, int cx, int cy, int cz) {
    x = q.x; y = q.y; z = q.z;
    mx = image_shift(cx, -1, c.nc[0], c.L[0]); px_ = image_shift(cx, 1, c.nc[0], c.L[0]);
    my = image_shift(cy, -1, c.nc[1], c.L[1]); py_ = image_shift(cy, 1, c.nc[1], c.L[1]);
    mz = image_shift(cz, -1, c.nc[2], c.L[2]); pz_ = image_shift(cz, 1, c.nc[2], c.L[2]);
    // codes hold (offset + 1) per axis in two bits, x lowest
    wraps = (cx == 0 ? 0x1111111111111111ull : 0ull) | (cx == c.nc[0] - 1 ? 0x4444444444444444ull : 0ull) |
            (cy == 0 ? 0x000f000f000f000full : 0ull) | (cy == c.nc[1] - 1 ? 0x0f000f000f000f00ull : 0ull) |
            (cz == 0 ? 0x000000000000ffffull : 0ull) | (cz == c.nc[2] - 1 ? 0x0000ffff00000000ull : 0ull);
  }
  __device__ __forceinline__ static double pick(uint32_t k, double m, double p) {
    return k == 0 ? m : (k == 2 ? p : 0.0);
  }
  __device__ __forceinline__ double r2(uint32_t code, const D4& qj, double& dx, double& dy, double& dz) const {
    dx = __dsub_rn(x, qj.x);
    dy = __dsub_rn(y, qj.y);
    dz = __dsub_rn(z, qj.z);
    if (wraps >> code & 1ull) {
      dx = __dadd_rn(dx, pick(code & 3u, mx, px_));
      dy = __dadd_rn(dy, pick((code >> 2) & 3u, my, py_));
      dz = __dadd_rn(dz, pick((code >> 4) & 3u, mz, pz_));
    }
    return r2_of(dx, dy, dz);
  }
};

// The walk of a warp's particles (one per group of T lanes) over their 27
// cells: calls keep(slot, j, code) on the lanes of kept candidates, slot
// counting them in walk order, and row(row, word) with the list positions of
// each row of three cells; returns the number kept.  The candidates of a
// row's three cells are taken as one run, kBatch x T at a time, so that their
// loads are in flight together.  The whole warp takes part (the groups'
// particles mostly share their cell, so their loops have the same length);
// a group with live = false meets no candidates.
template <int T, class Row, class Keep>
__device__ __forceinline__ int walk64(const Consts& c, bool live, const Home64& home, const float4& fi, int64_t i,
                                      int cx, int cy, int cz, const D4* __restrict__ q4,
                                      const float4* __restrict__ qf4, const int32_t* __restrict__ cell_start,
                                      const int32_t* __restrict__ mrank, Row row, Keep keep) {
  constexpr int kBatch = T == 32 ? 2 : 3;
  constexpr unsigned kFull = T == 32 ? 0xffffffffu : (1u << (T & 31)) - 1u;
  const int gl = threadIdx.x % T, shift = (threadIdx.x & 31) - gl;
  const unsigned below = (1u << gl) - 1u;
  int cnt = 0;
  // home coordinates shifted into the image of each neighbour cell (within
  // the bound of the filter: one more rounding of a number below 2 L)
  const float hx[3] = {cx == 0 ? fi.x + c.Lf[0] : fi.x, fi.x, cx == c.nc[0] - 1 ? fi.x - c.Lf[0] : fi.x};
#pragma unroll 1
  for (int oz = -1; oz <= 1; ++oz) {
    int nz = cz + oz;
    float hz = fi.z;
    if (nz < 0) { nz += c.nc[2]; hz += c.Lf[2]; }
    if (nz >= c.nc[2]) { nz -= c.nc[2]; hz -= c.Lf[2]; }
#pragma unroll 1
    for (int oy = -1; oy <= 1; ++oy) {
      int ny = cy + oy;
      float hy = fi.y;
      if (ny < 0) { ny += c.nc[1]; hy += c.Lf[1]; }
      if (ny >= c.nc[1]) { ny -= c.nc[1]; hy -= c.Lf[1]; }
      int beg[3], off[4] = {0, 0, 0, 0};
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        int nx = cx + k - 1;
        nx += nx < 0 ? c.nc[0] : (nx >= c.nc[0] ? -c.nc[0] : 0);
        const int r = __ldg(&mrank[nx + c.nc[0] * (ny + c.nc[1] * nz)]);
        beg[k] = __ldg(&cell_start[r]);
        off[k + 1] = __ldg(&cell_start[r + 1]) - beg[k];
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) off[k + 1] = live ? off[k + 1] + off[k] : 0;
      const int start = cnt;
      int kept = 0;  // this lane's: in the first cell, and << 16 in the first two
      const uint32_t code0 = nbr_entry(0, -1, oy, oz);
      for (int b = 0; __any_sync(0xffffffffu, b < off[3]); b += kBatch * T) {
        float4 fj[kBatch];
        int js[kBatch], cell[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
          const int t = b + u * T + gl;
          cell[u] = (t >= off[1]) + (t >= off[2]);
          js[u] = t + (cell[u] == 0 ? beg[0] : (cell[u] == 1 ? beg[1] - off[1] : beg[2] - off[2]));
          fj[u] = t < off[3] ? __ldg(&qf4[js[u]]) : make_float4(INFINITY, 0.0f, 0.0f, 0.0f);  // (beyond any h)
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
          const float ex = (cell[u] == 0 ? hx[0] : (cell[u] == 1 ? hx[1] : hx[2])) - fj[u].x, ey = hy - fj[u].y,
                      ez = hz - fj[u].z;
          const float rf = ex * ex + ey * ey + ez * ez;
          bool in = rf < c.h2_filter;
          if (in) {
            in = js[u] != i;
            if (rf >= c.h2_inner) {  // within the rounding bound of h^2: float64 decides
              double dx, dy, dz;
              in = in && home.r2(code0 + (uint32_t)cell[u], ld4(&q4[js[u]]), dx, dy, dz) < c.h2;
            }
          }
          const unsigned m = (__ballot_sync(0xffffffffu, in) >> shift) & kFull;
          if (in) {
            keep(cnt + __popc(m & below), js[u], code0 + (uint32_t)cell[u]);
            kept += cell[u] == 0 ? 0x10001 : (cell[u] == 1 ? 0x10000 : 0);
          }
          cnt += __popc(m);
        }
      }
#pragma unroll
      for (int sh = T / 2; sh > 0; sh >>= 1) kept += __shfl_xor_sync(0xffffffffu, kept, sh);
      row((oz + 1) * 3 + (oy + 1),
          (uint32_t)min(start, 255) | (uint32_t)min(start + (kept & 0xffff), 255) << 8 |
              (uint32_t)min(start + (kept >> 16), 255) << 16 | (uint32_t)min(cnt, 255) << 24);
    }
  }
  return cnt;
}

// Sum of v over the lanes of a group, the same order for every group.
template <int T>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int s = T / 2; s > 0; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
  return v;
}

// Lanes per particle of the float64 passes: with few particles a whole warp
// each, which spreads them over the SM quarters and shortens every particle's
// chain; else kLanes64, which costs fewer instructions in all.  The line lies
// at four warps per SM quarter, below where they are even (a Verlet step with a
// warp and with kLanes64 lanes, us: 1000 particles 46 / 66, 2197 76 / 90, 2744
// 86 / 100, 3375 99 / 90, 8000 161 / 125).
inline bool pair64_wide(const Consts& c) { return c.N <= 16 * 152; }

}  // namespace sdpd
