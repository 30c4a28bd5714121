// sdpd_fd_colour.cuh -- one pair update of the fluctuation/dissipation sweep
// (Sections 3.2-3.3), the kernels that stage the pairs' data, and the colour
// kernels that run a colour's blocks round by round.  Included by one
// translation unit per precision, each of which instantiates the
// block-schedule variants of its precision.
#pragma once
#include <algorithm>
#include <type_traits>

#include "sdpd_fd_common.cuh"
#include "sdpd_rand64.cuh"

namespace sdpd {

// ---------------------------------------------------------------------------
// One pair update.
// ---------------------------------------------------------------------------
template <class R>
struct FDConst {
  R inv_m, half_m;
  R kpar_m2, kperp_m2;  // (10/3 eta + 4 zeta) m^2, (5/3 eta - zeta) m^2
  R inv_C_K, kB, two_over_CK, dt_over_m;
  R CKm1;               // C_K / kB - 1
  R four_kB_over_m;
  double CKm1_d;          // C_K / kB - 1 in float64 (the exact Metropolis ratio)
  float nq_hi, nq_lo;     // -1 / (4 m) as a float-float (energy change from momenta)
  int scheme;
};

// Elementary functions of the sweep.  float64 (the pairs' geometry and the
// pair-by-pair sweep; the team kernel has its own, sdpd_f64.cuh): the library's
// functions.  float32 (mixed path): hardware approximations
// (relative error ~1e-7) for the proposal coefficients and Box-Muller -- the
// Metropolis step stays exact for any deterministic proposal coefficients
// because the forward and reverse moves use the same functions -- and the
// accurate log1p for the entropy term of the target measure.
namespace fm {
__device__ __forceinline__ double div(double a, double b) { return a / b; }
__device__ __forceinline__ float div(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double exp(double x) { return ::exp(x); }
__device__ __forceinline__ float exp(float x) { return __expf(x); }
__device__ __forceinline__ double log(double x) { return ::log(x); }
__device__ __forceinline__ float log(float x) { return __logf(x); }
__device__ __forceinline__ double sqrt(double x) { return ::sqrt(x); }
__device__ __forceinline__ float sqrt(float x) { return x * rsqrtf(x); }
__device__ __forceinline__ double rsqrt(double x) { return x > 1e-30 ? pair_rinv(x) : 1.0 / ::sqrt(x); }
__device__ __forceinline__ float rsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double expm1(double x) { return ::expm1(x); }
// exp(x) - 1 for x <= 0: Taylor polynomial for small |x| (relative error
// < 1e-8 below 1/8), the hardware exponential above
__device__ __forceinline__ float expm1(float x) {
  if (x > -0.125f) return x * (1.0f + x * (0.5f + x * (1.0f / 6.0f + x * (1.0f / 24.0f + x * (1.0f / 120.0f + x * (1.0f / 720.0f))))));
  return __expf(x) - 1.0f;
}
__device__ __forceinline__ double log1p(double x) { return ::log1p(x); }
// log(1 + x): alternating series for |x| < 1/16 (relative error < 2e-8),
// the hardware logarithm of 1 + x above
__device__ __forceinline__ float log1p(float x) {
  if (fabsf(x) < 0.0625f)
    return x * (1.0f - x * (0.5f - x * (1.0f / 3.0f - x * (0.25f - x * (0.2f - x * (1.0f / 6.0f))))));
  return __logf(1.0f + x);
}
}  // namespace fm

// Error-free transformations in float32 (Knuth's two-sum, the FMA split of
// a product): a + b = s + e and a * b = p + e exactly.  The rounded
// intrinsics keep the compiler from contracting or reordering them.
namespace eft {
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
  p = __fmul_rn(a, b);
  e = __fmaf_rn(a, b, -p);
}
}  // namespace eft

// Box-Muller normals and the uniform of one pair at one sweep (see
// pair_randoms), float32 path: the float64 path's uniforms rounded to
// float32 with full relative precision (a fixed-point uniform would lose
// the relative precision of the small values that the logarithms of
// Box-Muller and of the Metropolis test magnify), the logarithm inside
// Box-Muller accurate near 1 (log1p of minus 1 - u, formed from the
// integer), angles reduced to [-pi, pi) for the hardware sine and cosine.
__device__ __forceinline__ float uniform53f(uint64_t w) {  // (top 53 bits + 1/2) 2^-53
  const uint64_t m = w >> 11;
  const float hi = (float)(uint32_t)(m >> 21), lo = (float)(uint32_t)(m & 0x1fffffull) + 0.5f;
  return __fmaf_rn(hi, 2.3283064365386963e-10f, lo * 1.1102230246251565e-16f);
}
__device__ __forceinline__ float uniform32f(uint32_t x) {  // (x + 1/2) 2^-32
  return ((float)x + 0.5f) * 2.3283064365386963e-10f;
}
// -2 ln u for the radius of Box-Muller.  Below 1/2 the logarithm of u
// itself; above, log1p(-(1 - u)) with 1 - u = (c + 1/2) 2^-b formed from the
// integer complement c = 2^b - 1 - m, because u rounded to float32 reaches
// 1 for the largest m (and -2 ln u would then be 0 instead of ~2^-b).
__device__ __forceinline__ float neg2log_u53(uint64_t w) {  // u = (top 53 bits m + 1/2) 2^-53
  const uint64_t m = w >> 11;
  if (m < (1ull << 52)) return -2.0f * __logf(uniform53f(w));
  const uint64_t c = ((1ull << 53) - 1ull) - m;
  const float t = __fmaf_rn((float)(uint32_t)(c >> 21), 2.3283064365386963e-10f,
                            ((float)(uint32_t)(c & 0x1fffffull) + 0.5f) * 1.1102230246251565e-16f);
  return -2.0f * fm::log1p(-t);
}
__device__ __forceinline__ float neg2log_u32(uint32_t x) {  // u = (x + 1/2) 2^-32
  if (x < 0x80000000u) return -2.0f * __logf(uniform32f(x));
  return -2.0f * fm::log1p(-(((float)(0xffffffffu - x) + 0.5f) * 2.3283064365386963e-10f));
}
__device__ __forceinline__ void pair_randoms_fast(uint64_t seed, uint64_t sweep, uint64_t idi, uint64_t idj,
                                                  float G[3], float* U) {
  uint64_t w[4];
  philox4x64_10(sweep, idi, idj, 0ull, seed, 0ull, w);
  const float twopi = 6.28318530717958647692f;
  const float u1 = uniform53f(w[1]);
  const float R = fm::sqrt(neg2log_u53(w[0]));
  float sn, cs;
  __sincosf(twopi * (u1 - 0.5f), &sn, &cs);  // the angle 2 pi u1 - pi
  G[0] = -R * cs;
  G[1] = -R * sn;
  const float u3 = uniform32f((uint32_t)(w[2] & 0xffffffffull));
  G[2] = -fm::sqrt(neg2log_u32((uint32_t)(w[2] >> 32))) * __cosf(twopi * (u3 - 0.5f));
  *U = uniform53f(w[3]);
}
__device__ __forceinline__ void pair_randoms_fast(uint64_t seed, uint64_t sweep, uint64_t idi, uint64_t idj,
                                                  double G[3], double* U) {
  double lnU;
  pair_randoms(seed, sweep, idi, idj, G, U, &lnU);
}

// alpha = exp(-2 gamma dt / m) and zt = (2/m) zeta of Section 3.2 for both
// directions at energies (ei, ej), with gamma = kappa (1 - d) and
// sigma = 2 sqrt(kappa kB Ti Tj / (Ti + Tj)) of Eq. (sdpd-gamma-sigma):
// zt^2 = sigma^2 (1 - alpha^2) / (m gamma) = 4 kB Ti Tj / ((Ti+Tj) m (1-d)) (1 - alpha^2)
// (kappa cancels).  Ideal gas: T = eps / C_K and C = C_K, so
// d = kB Ti Tj / (Ti + Tj)^2 * 2 / C_K.
//
// Returns m = alpha - 1 = expm1(x) per direction (alpha itself is 1 + m):
// one expm1 per direction gives both alpha and 1 - alpha^2 = -m (2 + m), and
// one reciprocal of Ti + Tj serves both quotients -- the float64 dependency
// chain of a pair update is what bounds the sweep when a colour has few
// blocks.
template <class R>
__device__ __forceinline__ void pair_coeffs(const FDConst<R>& k, R kpar, R kperp, R ei, R ej, R& mpar,
                                            R& mperp, R& zpar, R& zperp) {
  const R Ti = ei * k.inv_C_K, Tj = ej * k.inv_C_K;
  const R isT = fm::div(R(1), Ti + Tj);
  const R hT = Ti * Tj * isT;
  const R omd = R(1) - k.kB * k.two_over_CK * hT * isT;
  const R xpar = R(-2) * kpar * omd * k.dt_over_m;  // log alpha per direction
  const R xperp = R(-2) * kperp * omd * k.dt_over_m;
  mpar = fm::expm1(xpar);
  mperp = fm::expm1(xperp);
  const R s = fm::div(k.four_kB_over_m * hT, omd);
  zpar = fm::sqrt(s * (-mpar * (R(2) + mpar)));
  zperp = fm::sqrt(s * (-mperp * (R(2) + mperp)));
}

// State-dependent part of one float64 pair update on (p_i, p_j) with
// internal energies (ei, ej), given the pair's unit vector e = r_ij / r_ij,
// base = F(r_ij) / (rho_i rho_j), its Gaussians G and the logarithm lnU of its
// uniform.  Returns 0 accept, 1 energy-bound reject, 2 Metropolis reject;
// deps receives the energy change shared by the two particles (applied by the
// caller on acceptance).
__device__ __forceinline__ int fd_pair(const FDConst<double>& k, double ex, double ey, double ez, double base,
                                       const double G[3], double lnU, double* pi, double* pj, double ei,
                                       double ej, double& deps, double& margin, bool& negative) {
  using R = double;
  const R kpar = k.kpar_m2 * base, kperp = k.kperp_m2 * base;
  margin = R(0);
  deps = R(0);
  if (!(kperp > R(0)) || !(kpar > R(0))) return 0;  // at r = h the pair does nothing
  const R vx = (pi[0] - pj[0]) * k.inv_m, vy = (pi[1] - pj[1]) * k.inv_m, vz = (pi[2] - pj[2]) * k.inv_m;
  R mpar, mperp, zpar, zperp;
  pair_coeffs(k, kpar, kperp, ei, ej, mpar, mperp, zpar, zperp);
  const R apar = R(1) + mpar, aperp = R(1) + mperp;
  // proposal, Eq. (proposal): v' = sum_theta P^theta (alpha^theta v + zt^theta G)
  const R vpar = ex * vx + ey * vy + ez * vz;
  const R gpar = ex * G[0] + ey * G[1] + ez * G[2];
  const R cpar = (apar - aperp) * vpar + (zpar - zperp) * gpar;
  const R wx = aperp * vx + zperp * G[0] + cpar * ex;
  const R wy = aperp * vy + zperp * G[1] + cpar * ey;
  const R wz = aperp * vz + zperp * G[2] + cpar * ez;
  // momenta of Eq. (proposal-update), energy shared equally (Section 3.2)
  const R dpx = k.half_m * (wx - vx), dpy = k.half_m * (wy - vy), dpz = k.half_m * (wz - vz);
  const R nix = pi[0] + dpx, niy = pi[1] + dpy, niz = pi[2] + dpz;
  const R njx = pj[0] - dpx, njy = pj[1] - dpy, njz = pj[2] - dpz;
  const double ko = pi[0] * pi[0] + pj[0] * pj[0] + pi[1] * pi[1] + pj[1] * pj[1] + pi[2] * pi[2] + pj[2] * pj[2];
  const double kn = nix * nix + njx * njx + niy * niy + njy * njy + niz * niz + njz * njz;
  deps = -0.5 * (kn - ko) * (0.5 * k.inv_m);
  // energy bound, Eq. (energy-bound): both new internal energies > 0
  const R emin = (ei < ej ? ei : ej) + deps;
  margin = emin;
  int decision = 0;
  if (k.scheme == SDPD_SCHEME_SSA) {
    if (!(emin > R(0))) negative = true;
  } else if (!(emin > R(0))) {
    decision = 1;
  } else if (k.scheme == SDPD_SCHEME_EMS) {
    // Metropolis ratio, Eq. (metropolis-ratio): the reverse move from v'
    // with the coefficients at the proposed energies
    R mrpar, mrperp, ypar, yperp;
    pair_coeffs(k, kpar, kperp, ei + deps, ej + deps, mrpar, mrperp, ypar, yperp);
    const R bpar = R(1) + mrpar, bperp = R(1) + mrperp;
    // one reciprocal for both directions of the reverse move's noise scale
    const R ryy = fm::div(R(1), ypar * yperp);
    const R ipar = yperp * ryy, ip = ypar * ryy;  // 1 / zt'_par, 1 / zt'_perp
    // reverse noise B'^-1 (v - A' v') from the proposed v' itself
    const R wpar = ex * wx + ey * wy + ez * wz;
    const R cb = (bpar - bperp) * wpar;
    const R bx = vx - (bperp * wx + cb * ex), by = vy - (bperp * wy + cb * ey), bz = vz - (bperp * wz + cb * ez);
    const R spar = ex * bx + ey * by + ez * bz;
    const R cq = (ipar - ip) * spar;
    const R qx = bx * ip + cq * ex, qy = by * ip + cq * ey, qz = bz * ip + cq * ez;
    const R quad = qx * qx + qy * qy + qz * qz;
    const R g2 = G[0] * G[0] + G[1] * G[1] + G[2] * G[2];
    // log|B(v)| - log|B(v')| with |B| = zt_par zt_perp^2
    const R ldet = fm::log(zpar * zperp * zperp * (ipar * ip * ip));
    // (S(eps') - S(eps))/kB - (log T(eps') - log T(eps)) = (C_K/kB - 1) log(eps'/eps)
    // summed over the two particles: log1p(x) + log1p(y) = log1p(x + y + x y)
    // with x = deps/ei, y = deps/ej, i.e. deps (ei + ej + deps) / (ei ej)
    const R ent = k.CKm1 * fm::log1p(fm::div(deps * (ei + ej + deps), ei * ej));
    const R a = R(0.5) * (g2 - quad) + ldet + ent;
    const R mg = a - lnU;
    margin = mg;
    if (mg < R(0)) decision = 2;  // U > exp(a)
  }
  if (decision == 0) {
    pi[0] = nix; pi[1] = niy; pi[2] = niz;
    pj[0] = njx; pj[1] = njy; pj[2] = njz;
  }
  return decision;
}

// The float32 quantities that define a mixed-path proposal and its reverse
// move, with the float64 energies: everything the Metropolis log-ratio of
// Eq. (metropolis-ratio) is evaluated from.  alpha = 1 + m per direction
// (m = expm1 of the exponent, so alpha - 1 carries no rounding of its own),
// zt the noise scales; the r-suffixed values belong to the reverse move at
// the proposed energies.
struct MixedRatioIn {
  float ex, ey, ez, vx, vy, vz, g0, g1, g2, u;
  float mpar, mperp, zpar, zperp, mrpar, mrperp, ypar, yperp;
  double ei, ej, deps;
};

// The Metropolis margin a - ln U of a mixed-path pair evaluated in float64
// from its float32 inputs: the reference value that the float32 evaluation
// approximates.  Reverse noise per direction theta,
// G'_theta = [(1 - alpha'_theta alpha_theta) v_theta - alpha'_theta zt_theta G_theta] / zt'_theta,
// which is B'^-1 (v - A' v') for v' = A v + B G; a = (|G|^2 - |G'|^2)/2 +
// log(|B| / |B'|) + (C_K/kB - 1) log1p(deps (ei + ej + deps) / (ei ej)).
// Kept out of line: it runs only for the rare pairs whose float32 margin is
// within its error bound of zero (and for every pair when records are kept).
static __device__ __noinline__ double mixed_margin_fp64(const MixedRatioIn& r, double CKm1) {
  const double ex = r.ex, ey = r.ey, ez = r.ez, vx = r.vx, vy = r.vy, vz = r.vz;
  const double g0 = r.g0, g1 = r.g1, g2 = r.g2;
  const double mpar = r.mpar, mperp = r.mperp, mrpar = r.mrpar, mrperp = r.mrperp;
  const double zpar = r.zpar, zperp = r.zperp, ypar = r.ypar, yperp = r.yperp;
  const double vpar = ex * vx + ey * vy + ez * vz;
  const double gpar = ex * g0 + ey * g1 + ez * g2;
  const double cpar = -(mpar + mrpar + mpar * mrpar), cperp = -(mperp + mrperp + mperp * mrperp);
  const double bpar = (1.0 + mrpar) * zpar, bperp = (1.0 + mrperp) * zperp;
  const double qpar = (cpar * vpar - bpar * gpar) / ypar;
  const double qx = (cperp * (vx - vpar * ex) - bperp * (g0 - gpar * ex)) / yperp;
  const double qy = (cperp * (vy - vpar * ey) - bperp * (g1 - gpar * ey)) / yperp;
  const double qz = (cperp * (vz - vpar * ez) - bperp * (g2 - gpar * ez)) / yperp;
  const double quad = qpar * qpar + qx * qx + qy * qy + qz * qz;
  const double gg = g0 * g0 + g1 * g1 + g2 * g2;
  const double ldet = log((zpar * zperp * zperp) / (ypar * yperp * yperp));
  const double ent = CKm1 * log1p(r.deps * (r.ei + r.ej + r.deps) / (r.ei * r.ej));
  return 0.5 * (gg - quad) + ldet + ent - log((double)r.u);
}

// One pair update of the mixed path.  The pair arithmetic (geometry,
// coefficients, proposal, momenta) is float32.  The internal energies are
// float64 in the state; during a block visit a particle's energy is its
// float64 value at load plus the visit's changes, which are kept as a
// float-float sum (about 48 significant bits).  The energy change deps of a
// pair is computed exactly from the float32 momenta before and after the
// move: -1/(4m) sum (new^2 - old^2), each square split exactly by an FMA and
// the differences and sums carried by two-sum, to float-float accuracy
// (dh + dl).  This keeps every pair update energy-conserving to float64
// rounding without float64 instructions, of which GB300 issues one for
// every 64 float32 ones.
//
// The energy bound is decided in float32 when its margin is clearly away
// from zero, else in float64 from the exact energies.  The Metropolis test
// is decided in float64: the log-ratio is evaluated in float32 together with
// a bound on its rounding error (a running error analysis of every
// operation, the documented error of the hardware logarithm, and a factor 2
// of safety), and a pair whose float32 margin is within that bound of zero
// is re-evaluated by mixed_margin_fp64, so every decision is the one the
// float64 evaluation of the same ratio gives.  m32 and tol receive the
// float32 margin and its bound; margin the float64 margin whenever it was
// evaluated (always when `exact` is set).  exact_e(ei, ej) gives the two
// current energies in float64 and uniform() the pair's uniform U (both for
// the rare float64 evaluations).
// The proposal of one mixed-path pair: what its Metropolis test needs, and the
// new momenta.
struct MixedMove {
  float vx, vy, vz, mpar, mperp, zpar, zperp;  // velocity, alpha - 1 and zt per direction
  float dh, dl, dhf;                           // energy change (float-float), its float32 estimate
  float nn[6];                                 // new momenta of i and j
};

// e . v and e . G (the rounding order is written out so that it does not
// depend on the code around it; SEQ: the order of the pair-by-pair sweep).
__device__ __forceinline__ float mixed_vpar(float ex, float ey, float ez, float vx, float vy, float vz) {
  return __fmaf_rn(ez, vz, __fmaf_rn(ex, vx, __fmul_rn(ey, vy)));
}
template <bool SEQ>
__device__ __forceinline__ float mixed_gpar(float ex, float ey, float ez, const float G[3]) {
  return __fmaf_rn(ez, G[2], SEQ ? __fmaf_rn(ey, G[1], __fmul_rn(ex, G[0])) : __fmaf_rn(ex, G[0], __fmul_rn(ey, G[1])));
}

// Returns 2 when the pair does nothing (r = h), else 1 when both new energies
// are positive and 0 when the energy bound rejects the move.
template <bool SEQ, class ExactE>
__device__ __forceinline__ int mixed_propose(const FDConst<float>& k, float ex, float ey, float ez, float base,
                                             const float G[3], const float* pi, const float* pj, float eif, float ejf,
                                             ExactE exact_e, MixedMove& mv, float& emn) {
  emn = 0.0f;
  const float kpar = k.kpar_m2 * base, kperp = k.kperp_m2 * base;
  if (!(kperp > 0.0f) || !(kpar > 0.0f)) return 2;  // at r = h the pair does nothing
  const float vx = (pi[0] - pj[0]) * k.inv_m, vy = (pi[1] - pj[1]) * k.inv_m, vz = (pi[2] - pj[2]) * k.inv_m;
  float mpar, mperp, zpar, zperp;  // alpha - 1 and zt per direction
  pair_coeffs(k, kpar, kperp, eif, ejf, mpar, mperp, zpar, zperp);
  // proposal, Eq. (proposal), as the velocity change
  // v' - v = m_perp v + zt_perp G + [(m_par - m_perp) v_par + (zt_par - zt_perp) G_par] e
  const float vpar = mixed_vpar(ex, ey, ez, vx, vy, vz), gpar = mixed_gpar<SEQ>(ex, ey, ez, G);
  const float cpar = (mpar - mperp) * vpar + (zpar - zperp) * gpar;
  const float dvx = mperp * vx + zperp * G[0] + cpar * ex;
  const float dvy = mperp * vy + zperp * G[1] + cpar * ey;
  const float dvz = mperp * vz + zperp * G[2] + cpar * ez;
  // momenta of Eq. (proposal-update), energy shared equally (Section 3.2)
  const float dpx = k.half_m * dvx, dpy = k.half_m * dvy, dpz = k.half_m * dvz;
  const float nn[6] = {pi[0] + dpx, pi[1] + dpy, pi[2] + dpz, pj[0] - dpx, pj[1] - dpy, pj[2] - dpz};
  // float32 estimate of the energy change: it places the reverse move's
  // coefficients (at eps + deps, rounded to float32, where it agrees with the
  // exact value below to a float32 rounding) without waiting for the exact
  // float-float sum, which takes a longer dependency chain
  float dhf;
  {
    float dk = 0.0f;
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      dk = fmaf(nn[t] - pi[t], nn[t] + pi[t], dk);
      dk = fmaf(nn[t + 3] - pj[t], nn[t + 3] + pj[t], dk);
    }
    dhf = k.nq_hi * dk;
  }
  float dh, dl;
  {  // deps = -1/2 of the kinetic-energy change of the stored momenta, exactly
    const float oo[6] = {pi[0], pi[1], pi[2], pj[0], pj[1], pj[2]};
    float d[6], lo[6];  // new^2 - old^2 per component as d + lo, exactly
#pragma unroll
    for (int t = 0; t < 6; ++t) {
      float pn, en, po, eo, ed;
      eft::two_prod(nn[t], nn[t], pn, en);
      eft::two_prod(oo[t], oo[t], po, eo);
      eft::two_sum(pn, -po, d[t], ed);
      lo[t] = __fadd_rn(ed, __fsub_rn(en, eo));
    }
    // the six high parts summed by a tree of two-sums (depth 3), the low
    // parts and the two-sum errors plainly (they are 2^-24 of the result)
    float s01, e01, s23, e23, s45, e45, s03, e03, Dh, eD, Dl;
    eft::two_sum(d[0], d[1], s01, e01);
    eft::two_sum(d[2], d[3], s23, e23);
    eft::two_sum(d[4], d[5], s45, e45);
    eft::two_sum(s01, s23, s03, e03);
    eft::two_sum(s03, s45, Dh, eD);
    Dl = __fadd_rn(__fadd_rn(__fadd_rn(lo[0], lo[1]), __fadd_rn(lo[2], lo[3])),
                   __fadd_rn(__fadd_rn(lo[4], lo[5]), __fadd_rn(__fadd_rn(e01, e23), __fadd_rn(e45, __fadd_rn(e03, eD)))));
    eft::two_sum(Dh, Dl, Dh, Dl);  // renormalise
    // times -1/(4m) (a float-float constant)
    float ph, pl;
    eft::two_prod(Dh, k.nq_hi, ph, pl);
    pl = __fmaf_rn(Dh, k.nq_lo, __fmaf_rn(Dl, k.nq_hi, pl));
    eft::two_sum(ph, pl, dh, dl);
  }
  // energy bound, Eq. (energy-bound): both new internal energies > 0;
  // float32 decides unless the margin is within its rounding of zero
  const float eminf = eif < ejf ? eif : ejf;
  emn = eminf + dh;
  if (fabsf(emn) <= 32.0f * 5.9604645e-8f * (eminf + fabsf(dh))) {
    double ei, ej;
    exact_e(ei, ej);
    emn = ((ei < ej ? ei : ej) + ((double)dh + (double)dl)) > 0.0 ? 1.0f : -1.0f;
  }
  mv.vx = vx; mv.vy = vy; mv.vz = vz;
  mv.mpar = mpar; mv.mperp = mperp; mv.zpar = zpar; mv.zperp = zperp;
  mv.dh = dh; mv.dl = dl; mv.dhf = dhf;
#pragma unroll
  for (int t = 0; t < 6; ++t) mv.nn[t] = nn[t];
  return emn > 0.0f ? 1 : 0;
}

// The Metropolis test of a move: true when it is rejected.  margin receives
// the float64 margin whenever it was evaluated (always when `exact` is set).
template <bool SEQ, class ExactE, class Uniform>
__device__ __forceinline__ bool mixed_rejects(const FDConst<float>& k, float ex, float ey, float ez, float base,
                                              const float G[3], Uniform uniform, float lnU, float eif, float ejf,
                                              ExactE exact_e, const MixedMove& mv, double& margin, float& m32,
                                              float& tol, bool exact) {
  const float kpar = k.kpar_m2 * base, kperp = k.kperp_m2 * base;
  const float vx = mv.vx, vy = mv.vy, vz = mv.vz, mpar = mv.mpar, mperp = mv.mperp, zpar = mv.zpar, zperp = mv.zperp;
  const float dh = mv.dh, dhf = mv.dhf;
  const float vpar = mixed_vpar(ex, ey, ez, vx, vy, vz), gpar = mixed_gpar<SEQ>(ex, ey, ez, G);
  // reverse move from v' with the coefficients at the proposed energies
  float mrpar, mrperp, ypar, yperp;
  pair_coeffs(k, kpar, kperp, eif + dhf, ejf + dhf, mrpar, mrperp, ypar, yperp);
  // 1 - alpha' alpha = -(m + m' + m m') (both m <= 0: no cancellation), alpha' zt
  const float cpr = -(mpar + mrpar + mpar * mrpar), cqr = -(mperp + mrperp + mperp * mrperp);
  const float bzpar = fmaf(mrpar, zpar, zpar), bzperp = fmaf(mrperp, zperp, zperp);
  const float ryy = fm::div(1.0f, ypar * yperp);
  const float ipar = yperp * ryy, ip = ypar * ryy;  // 1 / zt'_par, 1 / zt'_perp
  // reverse noise B'^-1 (v - A' v') = B'^-1 [(I - A' A) v - A' B G] per
  // direction: no cancellation when zt' -> 0 (pairs near the cut-off)
  const float qpar = (cpr * vpar - bzpar * gpar) * ipar;
  const float qx = (cqr * (vx - vpar * ex) - bzperp * (G[0] - gpar * ex)) * ip;
  const float qy = (cqr * (vy - vpar * ey) - bzperp * (G[1] - gpar * ey)) * ip;
  const float qz = (cqr * (vz - vpar * ez) - bzperp * (G[2] - gpar * ez)) * ip;
  const float quad = qpar * qpar + qx * qx + qy * qy + qz * qz;
  const float g2 = G[0] * G[0] + G[1] * G[1] + G[2] * G[2];
  // log|B(v)| - log|B(v')| with |B| = zt_par zt_perp^2
  const float ldet = fm::log(zpar * zperp * zperp * (ipar * ip * ip));
  // (S(eps') - S(eps))/kB - (log T(eps') - log T(eps)) over both particles
  const float x = fm::div(dh * (eif + ejf + dh), eif * ejf);
  const float ent = k.CKm1 * fm::log1p(x);
  const float mg = 0.5f * (g2 - quad) + ldet + ent - lnU;
  // error bound of mg against its exact value for these inputs (u = 2^-24;
  // 3.6e-7 bounds the absolute error of the hardware logarithm on
  // [0.5, 2], 3 ulp elsewhere)
  const float u = 5.9604645e-8f, elog = 3.6e-7f;
  const float V = fabsf(vx) + fabsf(vy) + fabsf(vz), Gs = fabsf(G[0]) + fabsf(G[1]) + fabsf(G[2]);
  const float qm = fabsf(qpar) * ipar * (fabsf(cpr) * V + bzpar * Gs) +
                   (fabsf(qx) + fabsf(qy) + fabsf(qz)) * ip * (fabsf(cqr) * V + bzperp * Gs);
  const float T = 8.0f * g2 + 23.0f * quad + 32.0f * qm + 11.0f * fabsf(ldet) + 25.0f * fabsf(ent) +
                  11.0f * fabsf(lnU) + 23.0f;
  tol = 2.0f * (u * T + 2.0f * elog);
  if (fabsf(x) >= 0.0625f) tol += 2.0f * k.CKm1 * (elog + 16.0f * u);
  m32 = mg;
  if (exact || !(fabsf(mg) > tol)) {  // float32 not decisive (or NaN): float64
    MixedRatioIn r;
    r.ex = ex; r.ey = ey; r.ez = ez; r.vx = vx; r.vy = vy; r.vz = vz;
    r.g0 = G[0]; r.g1 = G[1]; r.g2 = G[2]; r.u = uniform();
    r.mpar = mpar; r.mperp = mperp; r.zpar = zpar; r.zperp = zperp;
    r.mrpar = mrpar; r.mrperp = mrperp; r.ypar = ypar; r.yperp = yperp;
    exact_e(r.ei, r.ej);
    r.deps = (double)dh + (double)mv.dl;
    margin = mixed_margin_fp64(r, k.CKm1_d);
    return margin < 0.0;  // U > exp(a)
  }
  return mg < 0.0f;  // decided in float32: |mg| exceeds its error bound
}

template <bool SEQ, class ExactE, class Uniform>
__device__ __forceinline__ int fd_pair_mixed(const FDConst<float>& k, float ex, float ey, float ez, float base,
                                             const float G[3], Uniform uniform, float lnU, float* pi, float* pj,
                                             float eif, float ejf, ExactE exact_e, float& dh, float& dl,
                                             double& margin, float& m32, float& tol, bool exact,
                                             bool& negative) {
  margin = 0.0;
  m32 = 0.0f;
  tol = 0.0f;
  MixedMove mv;
  mv.dh = mv.dl = 0.0f;
  float emn;
  const int ok = mixed_propose<SEQ>(k, ex, ey, ez, base, G, pi, pj, eif, ejf, exact_e, mv, emn);
  dh = mv.dh;
  dl = mv.dl;
  if (ok == 2) return 0;
  if (exact) margin = (double)emn;  // (float64 work only where it is asked for)
  int decision = 0;
  if (k.scheme == SDPD_SCHEME_SSA) {
    if (!ok) negative = true;
  } else if (!ok) {
    decision = 1;
  } else if (k.scheme == SDPD_SCHEME_EMS) {
    if (mixed_rejects<SEQ>(k, ex, ey, ez, base, G, uniform, lnU, eif, ejf, exact_e, mv, margin, m32, tol, exact))
      decision = 2;
  }
  if (decision == 0) {
    pi[0] = mv.nn[0]; pi[1] = mv.nn[1]; pi[2] = mv.nn[2];
    pj[0] = mv.nn[3]; pj[1] = mv.nn[4]; pj[2] = mv.nn[5];
  }
  return decision;
}

// Cell code inside the block of owner (ox, oy, oz) of a particle whose cell
// bits are w: bit k set iff the particle sits in the upper cell along axis k.
template <class T>
__device__ __forceinline__ int block_code(T w, int ox, int oy, int oz) {
  int cx, cy, cz;
  unpack_cell(w_to_cellbits(w), cx, cy, cz);
  return (cx != ox) | ((cy != oy) << 1) | ((cz != oz) << 2);
}

struct FdCells {
  int32_t cst[8], cbs[8];  // the block's cells: first storage index, offset in the block
};
// Shared memory of one block in a colour launch with float32 pair arithmetic:
// each particle's record (px, py, pz, es), es the energy at load rounded to
// float32 plus the visit's changes (one wide load per particle and pair), and
// its compensation ec (the rounding errors of that sum and the low parts of
// the changes), so that the energy is eps(load) + (es - (float)eps(load)) + ec.
struct FdSmem {
  F4 s[kMaxBlock];
  float ec[kMaxBlock];
  FdCells cells;
};
__device__ __forceinline__ D4 lds4(const D4* p) {
  const double2* q = reinterpret_cast<const double2*>(p);
  const double2 a = q[0], b = q[1];
  return D4{a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ F4 lds4(const F4* p) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  return F4{a.x, a.y, a.z, a.w};
}

// Storage index of block particle q; d receives its cell in the block.
__device__ __forceinline__ int block_gidx(const FdCells& c, int q, int& d) {
  d = 0;
#pragma unroll
  for (int t = 1; t < 8; ++t) d += (q >= c.cbs[t]);
  return c.cst[d] + (q - c.cbs[d]);
}
__device__ __forceinline__ int block_gidx(const FdCells& c, int q) {
  int d;
  return block_gidx(c, q, d);
}

// ---------------------------------------------------------------------------
// Staged pair data.  What a pair update needs besides the momenta and
// energies is computed ahead of the colour launches by kernels that run one
// warp per block over all 8 colours at once, in the order of the blocks'
// scheduled pair lists (dense arrays indexed by sched_off[block] + position):
// the geometry (unit vector, F(r)/(rho_i rho_j)) with the schedule, since it
// depends on positions and densities only, and the random numbers once per
// sweep.  Outside the colour launches this work has full warps and the whole
// GPU, also when a colour has few blocks; inside them it sat on the path of
// every block's dependency chain.  Large systems stage both slice by slice, each
// just before its colour launch (fd_sliced).
// ---------------------------------------------------------------------------
constexpr int kStageWarps = 4;

// F at distance r (see kernel_F); the rounding of 1 - r/h in Lucy's kernel is
// written out so that it does not depend on the code around it.
__device__ __forceinline__ float one_minus(float r, float inv_h) { return __fmaf_rn(-r, inv_h, 1.0f); }
__device__ __forceinline__ double one_minus(double r, double inv_h) { return __fma_rn(-r, inv_h, 1.0); }
template <int KIND, class S>
__device__ __forceinline__ S stage_F(S r, S inv_h, S cF) {
  if (KIND == SDPD_KERNEL_LUCY) {
    const S y = one_minus(r, inv_h);
    return cF * (y * y);
  }
  return kernel_F<KIND>(r * inv_h, cF);
}

// Warps per block of the staging kernels: one, or as many (up to 16) as fill
// the GPU's 608 SM quarters eight times where blocks are few (10^3 particles,
// 64 blocks: the float64 random numbers take 189 us with one).
inline int stage_split(int64_t ncell) {
  const int64_t n = 8 * 608 / (ncell > 0 ? ncell : 1);
  return (int)(n < 1 ? 1 : (n > 16 ? 16 : n));
}

// The blocks whose pairs a staging launch writes: every block, in place, or a
// slice (see fd_sliced).
struct StageJob {
  int64_t n;             // blocks
  int split;             // warps per block
  const int32_t* order;  // slice: its blocks in the colour's order (null: every block)
  int colour;
  uint32_t* copy;        // slice: its pairs
};
inline StageJob stage_job(int64_t n, const int32_t* order, int colour, uint32_t* copy) {
  return StageJob{n, stage_split(n), order, colour, copy};
}
static inline unsigned stage_grid(const StageJob& job) {
  return (unsigned)((job.n * job.split + kStageWarps - 1) / kStageWarps);
}

// Owner cell of entry w of a colour's order.
__device__ __forceinline__ int64_t order_block(const Consts& c, int colour, int64_t w, int& ox, int& oy, int& oz) {
  const int hx = c.nc[0] >> 1, hy = c.nc[1] >> 1;
  ox = 2 * (int)(w % hx) + (colour & 1);
  oy = 2 * (int)((w / hx) % hy) + ((colour >> 1) & 1);
  oz = 2 * (int)(w / ((int64_t)hx * hy)) + ((colour >> 2) & 1);
  return ox + (int64_t)c.nc[0] * (oy + (int64_t)c.nc[1] * oz);
}

// The block's cells into shared memory, by the whole warp.
__device__ __forceinline__ void stage_cells(const Consts& c, int64_t o, const int32_t* __restrict__ mrank,
                                            const int32_t* __restrict__ cell_start, int lane, FdCells& cells) {
  int ox, oy, oz;
  owner_coords(c, o, ox, oy, oz);
  int cst = 0, cnt = 0;
  if (lane < 8) {
    int cx = ox + (lane & 1), cy = oy + ((lane >> 1) & 1), cz = oz + ((lane >> 2) & 1);
    if (cx >= c.nc[0]) cx -= c.nc[0];
    if (cy >= c.nc[1]) cy -= c.nc[1];
    if (cz >= c.nc[2]) cz -= c.nc[2];
    const int r = __ldg(&mrank[cx + c.nc[0] * (cy + c.nc[1] * cz)]);
    cst = __ldg(&cell_start[r]);
    cnt = __ldg(&cell_start[r + 1]) - cst;
  }
  int inc = cnt;
#pragma unroll
  for (int sh = 1; sh < 8; sh <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, inc, sh);
    if (lane >= sh) inc += v;
  }
  if (lane < 8) {
    cells.cst[lane] = cst;
    cells.cbs[lane] = inc - cnt;
  }
  __syncwarp();
}

// Owner cell of block blk of a staging launch.
__device__ __forceinline__ int64_t stage_block(const Consts& c, const StageJob& job, int64_t blk, int& ox, int& oy,
                                               int& oz) {
  if (job.order) return order_block(c, job.colour, job.order[blk], ox, oy, oz);
  owner_coords(c, blk, ox, oy, oz);
  return blk;
}

template <class P, class A, int KIND>
__global__ void __launch_bounds__(kStageWarps * 32)
    k_stage_geometry(Consts c, const typename P::V4* __restrict__ qr4, const int32_t* __restrict__ cell_start,
                     const int32_t* __restrict__ mrank, const uint32_t* __restrict__ xmx,
                     const uint32_t* __restrict__ xmy, const uint32_t* __restrict__ xmz,
                     const uint32_t* __restrict__ hdr, const unsigned long long* __restrict__ sched_off,
                     const uint32_t* __restrict__ pairs, const StageJob job, typename A::V4* __restrict__ geom) {
  using R = typename A::R;
  using S = typename P::R;
  __shared__ FdCells cells_s[kStageWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t wg = (int64_t)blockIdx.x * kStageWarps + warp, blk = wg / job.split;
  if (blk >= job.n) return;
  const int split = job.split, part = (int)(wg - blk * split);
  int ox, oy, oz;
  const int64_t o = stage_block(c, job, blk, ox, oy, oz);
  const uint32_t hd = hdr[o];
  const int np = hd == kHdrBig ? 0 : (int)(hd & 0xffffu);
  if (32 * part >= np) return;
  FdCells& cells = cells_s[warp];
  stage_cells(c, o, mrank, cell_start, lane, cells);
  BlockGeom<P> geo;
  geo.init(c, ox, oy, oz, xmx, xmy, xmz);
  const S inv_h = (S)c.inv_h, cF = (S)c.cF;
  const unsigned long long base = sched_off[o], to = job.order ? (unsigned long long)blk * kLargePairs : base;
  for (int t = 32 * part + lane; t < np; t += 32 * split) {
    const uint32_t pr = pairs[base + t];
    if (job.order) job.copy[to + t] = pr;
    int da, db;
    const int ga = block_gidx(cells, pr & 0xffffu, da), gb = block_gidx(cells, pr >> 16, db);
    S xa, ya, za, xb, yb, zb, rx, ry, rz;
    // positions and densities of the latest density pass (one load each)
    const typename P::V4 qa = ld4(&qr4[ga]), qb = ld4(&qr4[gb]);
    geo.local(qa, da, xa, ya, za);
    geo.local(qb, db, xb, yb, zb);
    geo.disp(xa, ya, za, xb, yb, zb, rx, ry, rz);
    const S r2 = r2_of(rx, ry, rz);
    const S inv_r = fm::rsqrt(r2);
    typename A::V4 v;
    v.x = (R)(rx * inv_r);
    v.y = (R)(ry * inv_r);
    v.z = (R)(rz * inv_r);
    v.w = (R)fm::div(stage_F<KIND>(r2 * inv_r, inv_h, cF), qa.w * qb.w);
    if constexpr (!A::mixed)  // at r = h the pair does nothing: marked by base = 0
      if (!(c.kperp_m2 * v.w > 0.0) || !(c.kpar_m2 * v.w > 0.0)) v.w = 0.0;
    st4(&geom[to + t], v);
  }
}

// Three normals and the uniform (its logarithm for EMS, whose Metropolis
// test needs only that) of every scheduled pair at the current sweep.
// float64: G split along and across e, (G - (e.G) e, e.G), and in aux
// |G|^2 / 2 - ln U (see sdpd_fd_team64.cuh).  Bound by Philox's 64-bit
// products in the float32 path (2 M particles, 67 M pairs: 1.21 ms; with
// explicit 32-bit multiply-adds 1.40) and by the float64 pipe in the other
// (32,768 particles: 0.29 ms; with the library's functions 0.56).
template <class A>
__global__ void __launch_bounds__(kStageWarps * 32)
    k_stage_random(Consts c, const int32_t* __restrict__ id, const int32_t* __restrict__ cell_start,
                   const int32_t* __restrict__ mrank, const uint32_t* __restrict__ hdr,
                   const unsigned long long* __restrict__ sched_off, const uint32_t* __restrict__ pairs,
                   const StageJob job, uint64_t seed, const unsigned long long* __restrict__ sweep_ptr,
                   const typename A::V4* __restrict__ geom, typename A::V4* __restrict__ rnd,
                   double* __restrict__ aux) {
  using R = typename A::R;
  __shared__ FdCells cells_s[kStageWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t wg = (int64_t)blockIdx.x * kStageWarps + warp, blk = wg / job.split;
  if (blk >= job.n) return;
  const int split = job.split, part = (int)(wg - blk * split);
  int ox, oy, oz;
  const int64_t o = stage_block(c, job, blk, ox, oy, oz);
  const uint32_t hd = hdr[o];
  const int np = hd == kHdrBig ? 0 : (int)(hd & 0xffffu);
  if (32 * part >= np) return;
  FdCells& cells = cells_s[warp];
  stage_cells(c, o, mrank, cell_start, lane, cells);
  const uint64_t sweep = *sweep_ptr;
  const unsigned long long base = sched_off[o], to = job.order ? (unsigned long long)blk * kLargePairs : base;
  for (int t = 32 * part + lane; t < np; t += 32 * split) {
    const uint32_t pr = pairs[base + t];
    const int ga = block_gidx(cells, pr & 0xffffu), gb = block_gidx(cells, pr >> 16);  // ga holds the lower id
    R G[3], U, lnU;
    // (ids as unsigned 32-bit numbers: the high words of the counter are known to be zero)
    typename A::V4 v;
    if constexpr (A::mixed) {
      pair_randoms_fast(seed, sweep, (uint32_t)id[ga], (uint32_t)id[gb], G, &U);
      v = F4{G[0], G[1], G[2], c.scheme == SDPD_SCHEME_EMS ? fm::log(U) : U};
    } else {
      pair_randoms(seed, sweep, (uint32_t)id[ga], (uint32_t)id[gb], G, &U, &lnU);
      const D4 e = ld4(&geom[to + t]);
      const double gp = e.x * G[0] + e.y * G[1] + e.z * G[2];
      v = D4{G[0] - gp * e.x, G[1] - gp * e.y, G[2] - gp * e.z, gp};
      aux[to + t] = c.scheme == SDPD_SCHEME_EMS
                          ? 0.5 * (G[0] * G[0] + G[1] * G[1] + G[2] * G[2]) - lnU : 0.0;
    }
    st4(&rnd[to + t], v);
  }
}

// A block beyond the capacities of the shared-memory schedule (kHdrBig: more
// than kLargeBlock particles, kLargePairs owned pairs or kMaxLevels rounds, or
// a member whose neighbour list overflowed its row).
// The whole warp sweeps its owned pairs in canonical order, one pair after
// the other, on the state in global memory; slow, but any block completes
// with the result of the sequential sweep.  The block's particles in rank
// order (ids ascending) go to its place in big_perm (blocks of one colour
// are disjoint, so N entries suffice).  Row d of
// the canonical order holds the pairs (perm[r], perm[r + d]), r ascending;
// the lanes test 32 candidates of a row at once (owner rule, then the
// neighbour predicate of the schedule enumeration) and lane 0 updates the
// hits in order of r.
// pair counters and flags of a sequential block sweep
struct BigCounts {
  unsigned long long tot, acc, rb, rm;
  int negative, bad;
};

template <class P, class A>
__device__ __noinline__ BigCounts fd_big_block(const Consts& c, const FDConst<typename A::R>& k, const Arrays<P>& a,
                                          typename P::V4* __restrict__ qp4, const int32_t* __restrict__ cell_start,
                                          const int32_t* __restrict__ mrank, const uint32_t* xmx,
                                          const uint32_t* xmy, const uint32_t* xmz, int64_t o, int ox, int oy,
                                          int oz, int colour, uint64_t seed, uint64_t sweep, sdpd_pair_rec* recs,
                                          unsigned long long* rec_count, int64_t rec_cap, int32_t* perm) {
  using R = typename A::R;
  using S = typename P::R;
  using V4 = typename P::V4;
  constexpr bool kSame = std::is_same<R, S>::value;
  const int lane = threadIdx.x & 31;
  unsigned long long n_tot = 0, n_acc = 0, n_rb = 0, n_rm = 0;
  bool negative = false, bad = false;
  BlockCells b;
  block_cells(c, ox, oy, oz, mrank, cell_start, b);
  const int nb = b.base[8];
  for (int q = lane; q < nb; q += 32) {  // rank order: every cell holds its ids ascending
    const int d = cell_code_of(b, q);
    const int g = b.start[d] + (q - b.base[d]);
    const int32_t id = a.id[g];
    int r = 0;
    for (int e = 0; e < 8; ++e) {  // ids of cell e below id
      int lo = b.start[e], n = b.cnt[e];
      while (n > 0) {
        const int half = n >> 1;
        if (a.id[lo + half] < id) { lo += half + 1; n -= half + 1; }
        else n = half;
      }
      r += lo - b.start[e];
    }
    perm[r] = g;
  }
  __syncwarp();
  BlockGeom<P> geo;
  geo.init(c, ox, oy, oz, xmx, xmy, xmz);
  const S h2 = (S)c.h2, inv_h = (S)(1.0 / c.h), cF = (S)c.cF;
  int seq = 0;
  for (int d = 1; d < nb; ++d) {
    for (int r0 = 0; r0 < nb - d; r0 += 32) {
      const int r = r0 + lane;
      int gA = 0, gB = 0;
      bool hit = false;
      if (r < nb - d) {
        gA = perm[r];
        gB = perm[r + d];
        const V4 qa = ld4(&a.q4[gA]), qb = ld4(&a.q4[gB]);
        const int dA = block_code(qa.w, ox, oy, oz), dB = block_code(qb.w, ox, oy, oz);
        const int hb = (int)owner_bits(a.id[gA]);
        if ((((dA ^ hb) & ~(dA ^ dB)) & 7) == 0) {  // owned: on shared axes the cell bit equals the owner bit
          S xa, ya, za, xb, yb, zb, rx, ry, rz;
          geo.local(qa, dA, xa, ya, za);
          geo.local(qb, dB, xb, yb, zb);
          geo.disp(xa, ya, za, xb, yb, zb, rx, ry, rz);
          hit = r2_of(rx, ry, rz) < h2;
        }
      }
      unsigned m = __ballot_sync(0xffffffffu, hit);
      while (m) {
        const int src = __ffs(m) - 1;
        m &= m - 1;
        const int ga = __shfl_sync(0xffffffffu, gA, src), gb = __shfl_sync(0xffffffffu, gB, src);
        if (lane == 0) {
          const V4 qa = ld4(&a.q4[ga]), qb = ld4(&a.q4[gb]);
          S xa, ya, za, xb, yb, zb, rx, ry, rz;
          geo.local(qa, block_code(qa.w, ox, oy, oz), xa, ya, za);
          geo.local(qb, block_code(qb.w, ox, oy, oz), xb, yb, zb);
          geo.disp(xa, ya, za, xb, yb, zb, rx, ry, rz);
          const S r2 = r2_of(rx, ry, rz);
          const S inv_r = fm::rsqrt(r2);
          const R ex = (R)(rx * inv_r), ey = (R)(ry * inv_r), ez = (R)(rz * inv_r);
          const S F = c.kernel == SDPD_KERNEL_LUCY ? stage_F<SDPD_KERNEL_LUCY>(r2 * inv_r, inv_h, cF)
                                                   : stage_F<SDPD_KERNEL_CUBIC>(r2 * inv_r, inv_h, cF);
          const R bs = (R)fm::div(F, a.rho[ga] * a.rho[gb]);
          R G[3], U;
          pair_randoms_fast(seed, sweep, (uint64_t)a.id[ga], (uint64_t)a.id[gb], G, &U);
          const R lnU = k.scheme == SDPD_SCHEME_EMS ? fm::log(U) : U;
          R pa[3] = {(R)a.px[ga], (R)a.py[ga], (R)a.pz[ga]};
          R pb[3] = {(R)a.px[gb], (R)a.py[gb], (R)a.pz[gb]};
          const R pa0[3] = {pa[0], pa[1], pa[2]}, pb0[3] = {pb[0], pb[1], pb[2]};
          double margin;
          float m32 = 0.0f, tol = 0.0f;
          int dcs;
          if constexpr (A::mixed) {
            auto exact_e = [&](double& x, double& y) { x = a.eps[ga]; y = a.eps[gb]; };
            float dh, dl;
            auto uniform = [&]() { return U; };
            dcs = fd_pair_mixed<true>(k, ex, ey, ez, bs, G, uniform, lnU, pa, pb, (float)a.eps[ga], (float)a.eps[gb],
                                exact_e, dh, dl, margin, m32, tol, recs != nullptr, negative);
            if (dcs == 0) {
              const double de = (double)dh + (double)dl;
              a.eps[ga] += de;
              a.eps[gb] += de;
            }
          } else {
            double deps;
            dcs = fd_pair(k, ex, ey, ez, bs, G, lnU, pa, pb, a.eps[ga], a.eps[gb], deps, margin, negative);
            if (dcs == 0) {
              a.eps[ga] = a.eps[ga] + deps;
              a.eps[gb] = a.eps[gb] + deps;
            }
          }
          if (dcs == 0) {
            if constexpr (kSame) {
              a.px[ga] = pa[0]; a.py[ga] = pa[1]; a.pz[ga] = pa[2];
              a.px[gb] = pb[0]; a.py[gb] = pb[1]; a.pz[gb] = pb[2];
            } else {  // the stored value plus the increment
              a.px[ga] += (S)(pa[0] - pa0[0]); a.py[ga] += (S)(pa[1] - pa0[1]); a.pz[ga] += (S)(pa[2] - pa0[2]);
              a.px[gb] += (S)(pb[0] - pb0[0]); a.py[gb] += (S)(pb[1] - pb0[1]); a.pz[gb] += (S)(pb[2] - pb0[2]);
            }
            bad |= !isfinite(a.eps[ga]) || !isfinite(a.eps[gb]);
          }
          ++n_tot;
          n_acc += dcs == 0;
          n_rb += dcs == 1;
          n_rm += dcs == 2;
          if (recs) {
            const unsigned long long sr = atomicAdd(rec_count, 1ull);
            if ((int64_t)sr < rec_cap) {
              sdpd_pair_rec rc;
              rc.id_i = a.id[ga];
              rc.id_j = a.id[gb];
              rc.colour = colour;
              rc.owner = (int32_t)o;
              rc.decision = dcs;
              rc.level = seq;  // position in the sequential order
              rc.margin = margin;
              rc.margin_lo = A::mixed ? (double)m32 : margin;
              rc.margin_tol = (double)tol;
              recs[sr] = rc;
            }
          }
        }
        ++seq;
        __syncwarp();
      }
    }
  }
  // pressure over rho^2 of the new energies, Eq. (pg-eos)
  const S pi_coef = std::is_same<S, float>::value ? (S)c.f_pi_coef : (S)c.pi_coef;
  for (int q = lane; q < nb; q += 32) {
    const int g = perm[q];
    qp4[g].w = (S)a.eps[g] * pi_coef / a.rho[g];
  }
  __syncwarp();
  return BigCounts{n_tot, n_acc, n_rb, n_rm, (int)negative, (int)bad};
}

// The float64 energies of a pair of the mixed path during a block visit: the
// stored energies plus the visit's changes.  The pair's uniform drawn again.
// Both serve the rare float64 decisions (near ties of the bound or the
// ratio) and are kept out of the hot loop.
static __device__ __noinline__ void fd_exact_energies(const double* eps, const FdCells& cells, const float* ec, int ia,
                                                      int ib, float eaf, float ebf, double& ea, double& eb) {
  const double ga = eps[block_gidx(cells, ia)], gb = eps[block_gidx(cells, ib)];
  ea = ga + (((double)eaf - (double)(float)ga) + (double)ec[ia]);
  eb = gb + (((double)ebf - (double)(float)gb) + (double)ec[ib]);
}
static __device__ __noinline__ float fd_uniform_again(uint64_t seed, uint64_t sweep, int32_t ida, int32_t idb) {
  float G[3], U;
  pair_randoms_fast(seed, sweep, (uint64_t)ida, (uint64_t)idb, G, &U);
  return U;
}

// ---------------------------------------------------------------------------
// One colour of the sweep.  A warp runs OPW blocks of the colour side by
// side, each on its own group of 32 / OPW lanes, in lockstep over the blocks'
// rounds (k_sched_rounds: at most 32 / OPW pairs of disjoint particles each).
// A block's particles (momenta and energies) live in shared memory; the
// pairs' staged data stream from global memory one round ahead of their use.
// P is the storage policy of the state arrays, A = Mixed the arithmetic policy
// of the pair updates (float64 pair arithmetic: k_fd_colour64).  A float64
// state swept with float32 pair arithmetic (P = Fp64) gets its momenta and
// energies back as their float64 values plus the float32 increments of the
// visit.  REC: keep a record per pair (every Metropolis margin in float64).
// Thread blocks of 1 to 4 warps.  PER_SM thread blocks of 128 threads per SM:
// 4 (128 registers, 16 warps per SM, some spills) where blocks abound; 3 (168
// registers, 12 warps, none) up to as many warps, where a round's chain decides.
// 262,144 particles, 4 sweeps: 4047 us with 4, 3947 with 3; 2 M particles, 2
// steps: 15.8 ms with 4, 16.5 with 3.  (5 with 96 registers: 4882 us and
// 16.5 ms; four blocks per warp, 8 lanes each: 17.0 ms.)
// ---------------------------------------------------------------------------
// What the lanes of a colour launch count.
struct FdTally {
  unsigned n_tot = 0, n_rb = 0, n_rm = 0;  // pairs, rejections (accepted = pairs - rejected)
  bool negative = false, bad = false;
};

// Launch-wide arguments of the block runs.
template <class P>
struct FdRun {
  Consts c;
  FDConst<float> k;
  Arrays<P> a;
  typename P::V4* qp4;
  const int32_t *cell_start, *mrank;
  const uint32_t *xmx, *xmy, *xmz;
  const uint32_t* hdr;
  const uint8_t* rsize;
  const unsigned long long* sched_off;
  const uint32_t* pairs;
  const F4 *geom, *rnd;
  int colour;
  // the launch's blocks: n entries of the colour's order from its entry
  // `first` on (order points there); pos: null, or (sliced) the places of all
  // blocks in their colours' orders; last: the colour's last launch
  int64_t first; unsigned n;
  const uint32_t* pos;
  bool last;
  uint64_t seed;
  unsigned long long* sweep_ptr;
  unsigned long long* counters;
  int* status;
  sdpd_pair_rec* recs;
  unsigned long long* rec_count;
  int64_t rec_cap;
  unsigned* queue;
  const int32_t* order;
  int32_t* big_perm;
  const int2* big_list;
  const uint32_t* big_count;
  const int32_t* large_list;
  const uint32_t* large_count;
};

// Runs one block per group of GL lanes (live: this group has one, of owner
// cell o with header hd): state into shared memory (s, ec, cells), the rounds,
// state back.  All lanes of the warp take part.
template <class P, int GL, bool REC>
__device__ __forceinline__ void fd_run_block(const FdRun<P>& f, bool live, int64_t o, int ox, int oy, int oz,
                                             uint32_t hd, uint64_t sweep, F4* s, float* ec, FdCells& cells,
                                             FdTally& tally) {
  using S = typename P::R;  // stored momenta, densities, geometry
  constexpr bool kSame = std::is_same<S, float>::value;
  const Consts& c = f.c;
  const Arrays<P>& a = f.a;
  const int gl = (threadIdx.x & 31) % GL;
  const int np = live ? (int)(hd & 0xffffu) : 0, nr = live ? (int)(hd >> 16 & 255u) : 0;
  if (gl == 0) tally.n_tot += (unsigned)np;
  // the pairs' staged data: this lane's element of the next round, loaded
  // one round ahead (`left` pairs of the current round not yet loaded)
  const unsigned long long first = np > 0 ? f.sched_off[o] : 0ull;
  const uint8_t* rs = f.rsize + o * kRoundStride;
  int r = 0, sizes = gl < nr ? (int)rs[gl] : 0;  // sizes of rounds [r - r % GL, ...)
  int left = __shfl_sync(0xffffffffu, sizes, 0, GL);
  int pos = 0, n = min(left, GL);
  uint32_t pr = 0;
  F4 ge{}, rn{};
  auto fetch = [&]() {
    if (gl < n) {
      pr = __ldg(&f.pairs[first + pos + gl]);
      ge = ld4(&f.geom[first + pos + gl]);
      rn = ld4(&f.rnd[first + pos + gl]);
    }
  };
  fetch();
  BlockCells b;
  b.base[8] = 0;
  if (np > 0) block_cells(c, ox, oy, oz, f.mrank, f.cell_start, b);
  const int nb = np > 0 ? b.base[8] : 0;
#pragma unroll
  for (int t = 0; t < 8; ++t)
    if (gl == t) {
      cells.cst[t] = b.start[t];
      cells.cbs[t] = b.base[t];
    }
  __syncwarp();
  for (int q = gl; q < nb; q += GL) {
    const int g = block_gidx(cells, q);
    s[q] = F4{(float)a.px[g], (float)a.py[g], (float)a.pz[g], (float)a.eps[g]};
    ec[q] = 0.0f;
  }
  __syncwarp();
  while (__any_sync(0xffffffffu, n > 0)) {
    const bool act = gl < n;
    const int level = r;
    const uint32_t cpr = pr;
    const F4 cg = ge, cr = rn;
    // advance to the next round (or the rest of a wide one) and load it
    pos += n;
    left -= n;
    if (left == 0 && r < nr) {
      ++r;
      if (r % GL == 0) sizes = r + gl < nr ? (int)rs[r + gl] : 0;
    }
    const int nx = __shfl_sync(0xffffffffu, sizes, r % GL, GL);
    if (left == 0) left = r < nr ? nx : 0;
    n = min(left, GL);
    fetch();
    if (act) {
      const int ia = cpr & 0xffffu, ib = cpr >> 16;
      const F4 sa = lds4(&s[ia]), sb = lds4(&s[ib]);
      float pa[3] = {sa.x, sa.y, sa.z};
      float pb[3] = {sb.x, sb.y, sb.z};
      const float G[3] = {cr.x, cr.y, cr.z};
      double margin;
      float m32 = 0.0f, tol = 0.0f;
      const float eaf = sa.w, ebf = sb.w;
      auto exact_e = [&](double& ea, double& eb) { fd_exact_energies(a.eps, cells, ec, ia, ib, eaf, ebf, ea, eb); };
      auto uniform = [&]() {
        return fd_uniform_again(f.seed, sweep, a.id[block_gidx(cells, ia)], a.id[block_gidx(cells, ib)]);
      };
      float dh, dl;
      const int dcs = fd_pair_mixed<false>(f.k, cg.x, cg.y, cg.z, cg.w, G, uniform, cr.w, pa, pb, eaf, ebf, exact_e, dh,
                                         dl, margin, m32, tol, REC, tally.negative);
      if (dcs == 0) {
        float t, e;
        eft::two_sum(eaf, dh, t, e);
        ec[ia] = __fadd_rn(ec[ia], __fadd_rn(e, dl));
        s[ia] = F4{pa[0], pa[1], pa[2], t};
        eft::two_sum(ebf, dh, t, e);
        ec[ib] = __fadd_rn(ec[ib], __fadd_rn(e, dl));
        s[ib] = F4{pb[0], pb[1], pb[2], t};
      }
      tally.n_rb += dcs == 1;
      tally.n_rm += dcs == 2;
      if constexpr (REC) {
        const unsigned long long at = atomicAdd(f.rec_count, 1ull);
        if ((int64_t)at < f.rec_cap) {
          sdpd_pair_rec rc;
          rc.id_i = a.id[block_gidx(cells, ia)];
          rc.id_j = a.id[block_gidx(cells, ib)];
          rc.colour = f.colour;
          rc.owner = (int32_t)o;
          rc.decision = dcs;
          rc.level = level;
          rc.margin = margin;
          rc.margin_lo = (double)m32;
          rc.margin_tol = (double)tol;
          f.recs[at] = rc;
        }
      }
    }
    __syncwarp();
  }
  const S pi_coef = std::is_same<S, float>::value ? (S)c.f_pi_coef : (S)c.pi_coef;
  for (int q = gl; q < nb; q += GL) {
    const int g = block_gidx(cells, q);
    const F4 v = lds4(&s[q]);
    if constexpr (kSame) {
      a.px[g] = v.x; a.py[g] = v.y; a.pz[g] = v.z;
    } else {  // the stored value plus this visit's increment
      a.px[g] += (S)(v.x - (float)a.px[g]);
      a.py[g] += (S)(v.y - (float)a.py[g]);
      a.pz[g] += (S)(v.z - (float)a.pz[g]);
    }
    // once per visit: the load value plus the visit's exact change
    const double e0 = a.eps[g];
    const double e = e0 + (((double)v.w - (double)(float)e0) + (double)ec[q]);
    tally.bad |= !isfinite(v.w);  // (a sum that was not finite once never is again)
    a.eps[g] = e;
    // pressure over rho^2 of the new energy, Eq. (pg-eos): pi = c_rho eps / (C_K m rho)
    // (from the stored float64 energy, as a restart recomputes it)
    f.qp4[g].w = (S)e * pi_coef / a.rho[g];
  }
  __syncwarp();  // the group's shared memory is refilled by the next block
}

// Shared memory of a large block: momenta as stored and float64 energies.
template <class P>
struct FdLargeSmem {
  typename P::R p[3][kLargeBlock];
  double e[kLargeBlock];
  FdCells cells;
};

// One of the colour's large blocks on a whole warp, its rounds at most 32
// pairs wide.  The pair updates are those of the pair-by-pair sweep
// (fd_big_block): float32 arithmetic on the stored momenta and float64
// energies, which take each pair's change.
template <class P, bool REC>
__device__ __noinline__ void fd_large_block(const FdRun<P>& f, int64_t o, uint64_t sweep, unsigned char* smem,
                                            FdTally& tally) {
  using S = typename P::R;
  FdLargeSmem<P>& sm = *reinterpret_cast<FdLargeSmem<P>*>(smem);
  const Consts& c = f.c;
  const Arrays<P>& a = f.a;
  const int lane = threadIdx.x & 31;
  const uint32_t hd = f.hdr[o];
  const int np = (int)(hd & 0xffffu), nr = (int)(hd >> 16 & 255u);
  if (lane == 0) tally.n_tot += (unsigned)np;
  stage_cells(c, o, f.mrank, f.cell_start, lane, sm.cells);
  int nb = 0;  // particles: the last cell's offset and count
  {
    int ox, oy, oz;
    owner_coords(c, o, ox, oy, oz);
    BlockCells b;
    block_cells(c, ox, oy, oz, f.mrank, f.cell_start, b);
    nb = b.base[8];
  }
  for (int q = lane; q < nb; q += 32) {
    const int g = block_gidx(sm.cells, q);
    sm.p[0][q] = a.px[g];
    sm.p[1][q] = a.py[g];
    sm.p[2][q] = a.pz[g];
    sm.e[q] = a.eps[g];
  }
  __syncwarp();
  // each lane's pair of a round (at most 32 pairs), loaded one round ahead
  const uint8_t* rs = f.rsize + o * kRoundStride;
  unsigned long long at = f.sched_off[o];
  uint32_t nxt_pr = 0;
  F4 nxt_ge{}, nxt_rn{};
  int n = nr > 0 ? (int)rs[0] : 0;
  auto fetch = [&]() {
    if (lane < n) {
      nxt_pr = __ldg(&f.pairs[at + lane]);
      nxt_ge = ld4(&f.geom[at + lane]);
      nxt_rn = ld4(&f.rnd[at + lane]);
    }
  };
  fetch();
  int n1 = nr > 1 ? (int)rs[1] : 0;  // size of the round after
  for (int r = 0; r < nr; ++r) {
    const bool act = lane < n;
    const uint32_t pr = nxt_pr;
    const F4 ge = nxt_ge, rn = nxt_rn;
    at += n;
    n = n1;
    n1 = r + 2 < nr ? (int)rs[r + 2] : 0;
    fetch();
    if (act) {
      const int ia = pr & 0xffffu, ib = pr >> 16;
      float pa[3], pb[3], pa0[3], pb0[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        pa0[d] = pa[d] = (float)sm.p[d][ia];
        pb0[d] = pb[d] = (float)sm.p[d][ib];
      }
      const double ea = sm.e[ia], eb = sm.e[ib];
      const float G[3] = {rn.x, rn.y, rn.z};
      auto exact_e = [&](double& x, double& y) { x = ea; y = eb; };
      auto uniform = [&]() {
        return fd_uniform_again(f.seed, sweep, a.id[block_gidx(sm.cells, ia)], a.id[block_gidx(sm.cells, ib)]);
      };
      double margin;
      float dh, dl, m32 = 0.0f, tol = 0.0f;
      const int dcs = fd_pair_mixed<true>(f.k, ge.x, ge.y, ge.z, ge.w, G, uniform, rn.w, pa, pb, (float)ea, (float)eb,
                                          exact_e, dh, dl, margin, m32, tol, REC, tally.negative);
      if (dcs == 0) {
        const double de = (double)dh + (double)dl;
        sm.e[ia] = ea + de;
        sm.e[ib] = eb + de;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          if constexpr (std::is_same<S, float>::value) {
            sm.p[d][ia] = pa[d];
            sm.p[d][ib] = pb[d];
          } else {  // the stored value plus the increment
            sm.p[d][ia] += (S)(pa[d] - pa0[d]);
            sm.p[d][ib] += (S)(pb[d] - pb0[d]);
          }
        }
      }
      tally.n_rb += dcs == 1;
      tally.n_rm += dcs == 2;
      if constexpr (REC) {
        const unsigned long long k = atomicAdd(f.rec_count, 1ull);
        if ((int64_t)k < f.rec_cap) {
          sdpd_pair_rec rc;
          rc.id_i = a.id[block_gidx(sm.cells, ia)];
          rc.id_j = a.id[block_gidx(sm.cells, ib)];
          rc.colour = f.colour;
          rc.owner = (int32_t)o;
          rc.decision = dcs;
          rc.level = r;
          rc.margin = margin;
          rc.margin_lo = (double)m32;
          rc.margin_tol = (double)tol;
          f.recs[k] = rc;
        }
      }
    }
    __syncwarp();
  }
  const S pi_coef = std::is_same<S, float>::value ? (S)c.f_pi_coef : (S)c.pi_coef;
  for (int q = lane; q < nb; q += 32) {
    const int g = block_gidx(sm.cells, q);
    a.px[g] = sm.p[0][q];
    a.py[g] = sm.p[1][q];
    a.pz[g] = sm.p[2][q];
    tally.bad |= !isfinite(sm.e[q]);
    a.eps[g] = sm.e[q];
    f.qp4[g].w = (S)sm.e[q] * pi_coef / a.rho[g];
  }
  __syncwarp();
}

// The end of a colour launch, by all warps: large blocks, blocks beyond
// capacity, the queue's reset and the counters.
template <class P, bool REC>
__device__ __forceinline__ void fd_finish(const FdRun<P>& f, uint64_t sweep, unsigned char* fd_smem_raw,
                                          FdTally& tally) {
  const Consts& c = f.c;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, colour = f.colour;
  const int64_t nown = (int64_t)(c.nc[0] >> 1) * (c.nc[1] >> 1) * (c.nc[2] >> 1);
  unsigned* queue = f.queue;
  // large blocks: one warp of the thread block, on all of its shared memory
  if (f.large_count[colour] > 0) {
    __syncthreads();
    for (; warp == 0;) {
      unsigned li = 0;
      if (lane == 0) li = atomicAdd(&queue[3], 1u);
      li = __shfl_sync(0xffffffffu, li, 0);
      if (li >= f.large_count[colour]) break;
      const int32_t o = f.large_list[colour * nown + li];
      if (f.pos && ((int64_t)f.pos[o] < f.first || (int64_t)f.pos[o] >= f.first + f.n)) continue;  // of another slice
      fd_large_block<P, REC>(f, o, sweep, fd_smem_raw, tally);
    }
  }
  // the colour's blocks beyond capacity (listed by the schedule), swept pair
  // by pair by whole warps once the queue is empty
  while (f.last) {
    unsigned bi = 0;
    if (lane == 0) bi = atomicAdd(&queue[2], 1u);
    bi = __shfl_sync(0xffffffffu, bi, 0);
    if (bi >= f.big_count[colour]) break;
    const int2 ent = f.big_list[colour * nown + bi];
    int bx, by, bz;
    owner_coords(c, ent.x, bx, by, bz);
    const BigCounts bc = fd_big_block<P, Mixed>(c, f.k, f.a, f.qp4, f.cell_start, f.mrank, f.xmx, f.xmy, f.xmz, ent.x,
                                                bx, by, bz, colour, f.seed, sweep, REC ? f.recs : nullptr, f.rec_count,
                                                f.rec_cap, f.big_perm + ent.y);
    if (lane == 0) {  // (rare: counted at once; lane 0 made the updates)
      atomicAdd(&f.counters[0], bc.tot);
      atomicAdd(&f.counters[1], bc.acc);
      atomicAdd(&f.counters[2], bc.rb);
      atomicAdd(&f.counters[3], bc.rm);
    }
    tally.negative |= bc.negative != 0;
    tally.bad |= bc.bad != 0;
  }
  if (lane == 0) {
    const unsigned total = gridDim.x * (blockDim.x >> 5);
    __threadfence();  // this warp's last take from queue[0] is performed before it counts as done
    if (atomicAdd(&queue[1], 1u) == total - 1u) {  // every warp has taken its last block
      queue[0] = 0u;
      queue[1] = 0u;
      queue[2] = 0u;
      queue[3] = 0u;
      if (colour == 7 && f.last) *f.sweep_ptr = sweep + 1ull;  // (every warp has read it) the sweep is done
    }
  }
  // counters
  unsigned long long c_tot = tally.n_tot, c_rb = tally.n_rb, c_rm = tally.n_rm;
  for (int s = 16; s > 0; s >>= 1) {
    c_tot += __shfl_xor_sync(0xffffffffu, c_tot, s);
    c_rb += __shfl_xor_sync(0xffffffffu, c_rb, s);
    c_rm += __shfl_xor_sync(0xffffffffu, c_rm, s);
  }
  const unsigned any_neg = __any_sync(0xffffffffu, tally.negative), any_bad = __any_sync(0xffffffffu, tally.bad);
  if (lane == 0) {
    if (c_tot | c_rb | c_rm) {  // (accepted = pairs - rejected, added with wrap-around)
      atomicAdd(&f.counters[0], c_tot);
      atomicAdd(&f.counters[1], c_tot - c_rb - c_rm);
      atomicAdd(&f.counters[2], c_rb);
      atomicAdd(&f.counters[3], c_rm);
    }
    if (any_neg) atomicOr(f.status, kStNegative);
    if (any_bad) atomicOr(f.status, kStNaN);
  }
}

template <class P, int OPW, int PER_SM, bool REC>
__global__ void __launch_bounds__(128, PER_SM) k_fd_colour(const __grid_constant__ FdRun<P> f) {
  constexpr int GL = 32 / OPW;
  extern __shared__ __align__(32) unsigned char fd_smem_raw[];
  const uint64_t sweep = *f.sweep_ptr;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, grp = lane / GL;
  const Consts& c = f.c;
  // (as order_block, whose call here, inside the loop, costs 5%: 1010 us per sweep of 262,144 particles, 968 so)
  const int colour = f.colour, hx = c.nc[0] >> 1, hy = c.nc[1] >> 1;
  FdSmem& sm = reinterpret_cast<FdSmem*>(fd_smem_raw)[warp * OPW + grp];
  unsigned* queue = f.queue;
  FdTally tally;
  // The grid holds as many thread blocks as fit on the GPU at once; each
  // warp takes the colour's blocks OPW at a time from queue[0] until they
  // run out, so no partial last wave of thread blocks idles the GPU and
  // blocks of uneven depth balance out.  The blocks come in the order of
  // `order` (deepest first), so the blocks a warp runs in lockstep have
  // similar depth.  queue[1] counts the warps that are done; the last one
  // sets them back to zero for the next launch (queue[2], queue[3]: the next
  // entries of the colour's lists of blocks beyond capacity and of large blocks).
  for (;;) {
    unsigned w0 = 0;
    if (lane == 0) w0 = atomicAdd(queue, (unsigned)OPW);
    w0 = __shfl_sync(0xffffffffu, w0, 0);
    if (w0 >= f.n) break;
    const unsigned wi = w0 + grp;
    const int64_t w = wi < f.n ? (int64_t)f.order[wi] : 0;
    const int ox = 2 * (int)(w % hx) + (colour & 1), oy = 2 * (int)((w / hx) % hy) + ((colour >> 1) & 1),
              oz = 2 * (int)(w / ((int64_t)hx * hy)) + ((colour >> 2) & 1);
    const int64_t o = ox + (int64_t)c.nc[0] * (oy + (int64_t)c.nc[1] * oz);
    const uint32_t hd = f.hdr[o];
    // (large blocks and those beyond capacity, which have the flag's bit set too, come below)
    const bool live = wi < f.n && !(hd & kHdrLargeFlag);
    fd_run_block<P, GL, REC>(f, live, o, ox, oy, oz, hd, sweep, sm.s, sm.ec, sm.cells, tally);
  }
  fd_finish<P, REC>(f, sweep, fd_smem_raw, tally);
}

// ---------------------------------------------------------------------------
// EMS with one block per team of two warps, for launches with few blocks,
// where a colour lasts as long as its deepest block.  A round on one warp is a
// chain of about 560 instructions that issue at a third of the rate; here the
// first warp proposes round r and moves it at once, and the second tests it
// while the first is at round r + 1.  When it rejects a move (1e-4 to 3e-2 of
// the pairs) the first takes round r + 1 back, then the rejected moves, and
// proposes round r + 1 again, so the result is that of the sequential sweep,
// bit for bit that of k_fd_colour.  64,000 particles (512 blocks per colour):
// 63 us per launch, with one warp per block 70.
// ---------------------------------------------------------------------------
struct FdSpecSmem {
  FdSmem b;
  float mv[2][14][32];   // moves of two rounds: v, m, z, dh, dl, dhf, the energies and compensations before
  uint8_t ok[2][32];     // mixed_propose's answer
  uint8_t rsize[kRoundStride];
  unsigned rejected[2];  // lanes of the round tested in a step, by the step's parity
  unsigned next;
};

template <class P, bool REC>
__global__ void __launch_bounds__(64) k_fd_colour_spec(const __grid_constant__ FdRun<P> f) {
  using S = typename P::R;
  constexpr bool kSame = std::is_same<S, float>::value;
  extern __shared__ __align__(32) unsigned char fd_smem_raw[];
  FdSpecSmem& sm = *reinterpret_cast<FdSpecSmem*>(fd_smem_raw);
  const uint64_t sweep = *f.sweep_ptr;
  const int t = threadIdx.x, lane = t & 31;
  const bool tester = t >= 32;
  const Consts& c = f.c;
  const Arrays<P>& a = f.a;
  const int colour = f.colour;
  const S pi_coef = kSame ? (S)c.f_pi_coef : (S)c.pi_coef;
  unsigned* queue = f.queue;
  FdTally tally;
  F4* s = sm.b.s;
  float* ec = sm.b.ec;
  FdCells& cells = sm.b.cells;
  for (;;) {  // blocks from the colour's queue, deepest first (see k_fd_colour)
    if (t == 0) sm.next = atomicAdd(queue, 1u);
    __syncthreads();
    const unsigned wi = sm.next;
    if (wi >= f.n) break;
    int ox, oy, oz;
    const int64_t o = order_block(c, colour, f.order[wi], ox, oy, oz);
    const uint32_t hd = f.hdr[o];
    const int np = hd & kHdrLargeFlag ? 0 : (int)(hd & 0xffffu), nr = (int)(hd >> 16 & 255u);
    if (np == 0) {  // (large blocks and those beyond capacity come below)
      __syncthreads();
      continue;
    }
    if (t == 0) tally.n_tot += (unsigned)np;
    const unsigned long long first = f.sched_off[o];
    for (int r = t; r < nr; r += 64) sm.rsize[r] = f.rsize[o * kRoundStride + r];
    BlockCells b;
    block_cells(c, ox, oy, oz, f.mrank, f.cell_start, b);
    const int nb = b.base[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (t == q) {
        cells.cst[q] = b.start[q];
        cells.cbs[q] = b.base[q];
      }
    __syncthreads();
    for (int q = t; q < nb; q += 64) {
      const int g = block_gidx(cells, q);
      s[q] = F4{(float)a.px[g], (float)a.py[g], (float)a.pz[g], (float)a.eps[g]};
      ec[q] = 0.0f;
    }
    // this lane's pair of a round, loaded one round ahead; the tester meets
    // round r one step after the proposer
    uint32_t pr = 0;
    F4 ge{}, rn{};
    int pos = 0, n = sm.rsize[0];
    auto fetch = [&]() {
      if (lane < n) {
        pr = __ldg(&f.pairs[first + pos + lane]);
        ge = ld4(&f.geom[first + pos + lane]);
        rn = ld4(&f.rnd[first + pos + lane]);
      }
    };
    fetch();
    __syncthreads();
    // the proposer's pairs of this round and the one before, with the records
    // before their moves
    int ia = 0, ib = 0, last_a = 0, last_b = 0;
    F4 sa{}, sb{}, last_sa{}, last_sb{};
    float ca = 0.0f, cb = 0.0f, last_ca = 0.0f, last_cb = 0.0f;
    for (int st = 0; st <= nr; ++st) {
      const int r = tester ? st - 1 : st;
      const bool on = r >= 0 && r < nr;
      const int buf = r & 1;
      const bool act = on && lane < n;
      const uint32_t cpr = pr;
      const F4 cg = ge, cr = rn;
      if (on) {
        pos += n;
        n = r + 1 < nr ? (int)sm.rsize[r + 1] : 0;
        fetch();
      }
      const float G[3] = {cr.x, cr.y, cr.z};
      ia = cpr & 0xffffu;
      ib = cpr >> 16;
      bool moved = false;
      auto propose = [&]() {
        sa = lds4(&s[ia]);
        sb = lds4(&s[ib]);
        ca = ec[ia];
        cb = ec[ib];
        const float pa[3] = {sa.x, sa.y, sa.z}, pb[3] = {sb.x, sb.y, sb.z};
        auto exact_e = [&](double& x, double& y) { fd_exact_energies(a.eps, cells, ec, ia, ib, sa.w, sb.w, x, y); };
        MixedMove mv;
        mv.dh = mv.dl = 0.0f;
        float emn;
        const int ok = mixed_propose<false>(f.k, cg.x, cg.y, cg.z, cg.w, G, pa, pb, sa.w, sb.w, exact_e, mv, emn);
        moved = ok == 1;
        if (moved) {
          float v, e;
          eft::two_sum(sa.w, mv.dh, v, e);
          ec[ia] = __fadd_rn(ca, __fadd_rn(e, mv.dl));
          s[ia] = F4{mv.nn[0], mv.nn[1], mv.nn[2], v};
          eft::two_sum(sb.w, mv.dh, v, e);
          ec[ib] = __fadd_rn(cb, __fadd_rn(e, mv.dl));
          s[ib] = F4{mv.nn[3], mv.nn[4], mv.nn[5], v};
          const float out[14] = {mv.vx, mv.vy, mv.vz, mv.mpar, mv.mperp, mv.zpar, mv.zperp, mv.dh, mv.dl, mv.dhf,
                                 sa.w, sb.w, ca, cb};
#pragma unroll
          for (int q = 0; q < 14; ++q) sm.mv[buf][q][lane] = out[q];
        }
        sm.ok[buf][lane] = (uint8_t)ok;
        if (REC) sm.mv[buf][7][lane] = moved ? mv.dh : emn;
      };
      if (!tester) {
        if (act) propose();
      } else {
        int dcs = 0;
        if (act) {
          const int ok = sm.ok[buf][lane];
          double margin = 0.0;
          float m32 = 0.0f, tol = 0.0f;
          if (ok == 1) {
            MixedMove mv;
            const float* in = &sm.mv[buf][0][lane];
            mv.vx = in[0]; mv.vy = in[32]; mv.vz = in[64];
            mv.mpar = in[96]; mv.mperp = in[128]; mv.zpar = in[160]; mv.zperp = in[192];
            mv.dh = in[224]; mv.dl = in[256]; mv.dhf = in[288];
            const float eaf = in[320], ebf = in[352], eca = in[384], ecb = in[416];
            auto exact_e = [&](double& x, double& y) {  // the energies before the move
              const double ga = a.eps[block_gidx(cells, ia)], gb = a.eps[block_gidx(cells, ib)];
              x = ga + (((double)eaf - (double)(float)ga) + (double)eca);
              y = gb + (((double)ebf - (double)(float)gb) + (double)ecb);
            };
            auto uniform = [&]() {
              return fd_uniform_again(f.seed, sweep, a.id[block_gidx(cells, ia)], a.id[block_gidx(cells, ib)]);
            };
            if (mixed_rejects<false>(f.k, cg.x, cg.y, cg.z, cg.w, G, uniform, cr.w, eaf, ebf, exact_e, mv, margin, m32,
                                     tol, REC))
              dcs = 2;
          } else if (ok == 0) {
            dcs = 1;
            if (REC) margin = (double)sm.mv[buf][7][lane];
          }
          tally.n_rb += dcs == 1;
          tally.n_rm += dcs == 2;
          if constexpr (REC) {
            const unsigned long long at = atomicAdd(f.rec_count, 1ull);
            if ((int64_t)at < f.rec_cap) {
              sdpd_pair_rec rc;
              rc.id_i = a.id[block_gidx(cells, ia)];
              rc.id_j = a.id[block_gidx(cells, ib)];
              rc.colour = colour;
              rc.owner = (int32_t)o;
              rc.decision = dcs;
              rc.level = r;
              rc.margin = margin;
              rc.margin_lo = (double)m32;
              rc.margin_tol = (double)tol;
              f.recs[at] = rc;
            }
          }
        }
        const unsigned rej = __ballot_sync(0xffffffffu, dcs == 2);
        if (lane == 0) sm.rejected[st & 1] = rej;
      }
      __syncthreads();
      const unsigned rej = sm.rejected[st & 1];
      if (rej) {  // (uniform: both warps)
        if (!tester) {
          if (moved) {  // this round back,
            s[ia] = sa;
            s[ib] = sb;
            ec[ia] = ca;
            ec[ib] = cb;
          }
          __syncwarp();
          if (rej >> lane & 1u) {  // the rejected moves of the round before,
            s[last_a] = last_sa;
            s[last_b] = last_sb;
            ec[last_a] = last_ca;
            ec[last_b] = last_cb;
          }
          __syncwarp();
          if (act) propose();  // this round once more
        }
        __syncthreads();
      }
      if (!tester) {
        __syncwarp();
        last_a = ia;
        last_b = ib;
        last_sa = sa;
        last_sb = sb;
        last_ca = ca;
        last_cb = cb;
      }
    }
    __syncthreads();
    for (int q = t; q < nb; q += 64) {
      const int g = block_gidx(cells, q);
      const F4 v = lds4(&s[q]);
      if constexpr (kSame) {
        a.px[g] = v.x; a.py[g] = v.y; a.pz[g] = v.z;
      } else {  // the stored value plus this visit's increment
        a.px[g] += (S)(v.x - (float)a.px[g]);
        a.py[g] += (S)(v.y - (float)a.py[g]);
        a.pz[g] += (S)(v.z - (float)a.pz[g]);
      }
      // once per visit: the load value plus the visit's exact change
      const double e0 = a.eps[g];
      const double e = e0 + (((double)v.w - (double)(float)e0) + (double)ec[q]);
      tally.bad |= !isfinite(v.w);
      a.eps[g] = e;
      f.qp4[g].w = (S)e * pi_coef / a.rho[g];  // as in fd_run_block
    }
    __syncthreads();  // the team's shared memory is refilled by the next block
  }
  fd_finish<P, REC>(f, sweep, fd_smem_raw, tally);
}

template <class R>
static FDConst<R> fd_const(const Consts& c, double dt) {
  FDConst<R> k;
  k.inv_m = (R)(1.0 / c.m);
  k.half_m = (R)(0.5 * c.m);
  k.kpar_m2 = (R)c.kpar_m2;
  k.kperp_m2 = (R)c.kperp_m2;
  k.inv_C_K = (R)(1.0 / c.C_K);
  k.kB = (R)c.kB;
  k.two_over_CK = (R)(2.0 / c.C_K);
  k.dt_over_m = (R)(dt / c.m);
  k.CKm1 = (R)(c.C_K / c.kB - 1.0);
  k.four_kB_over_m = (R)(4.0 * c.kB / c.m);
  k.CKm1_d = c.C_K / c.kB - 1.0;
  k.nq_hi = (float)(-0.25 / c.m);
  k.nq_lo = (float)(-0.25 / c.m - (double)k.nq_hi);
  k.scheme = c.scheme;
  return k;
}

// Block schedules of the colour launches: blocks per warp and warps per
// thread block of each variant (see sdpd_tuning); EMS with one block per warp
// runs k_fd_colour_spec, a two-warp team per block.  The mapping onto the GPU
// differs, the pair updates and their order per particle do not.
constexpr int kFdOpw[kFdVariants] = {2, 2, 1, 1, 1};
constexpr int kFdWarps[kFdVariants] = {2, 1, 1, 2, 4};

// Shared memory of a thread block: its groups' blocks, at least one large block.
template <class P>
constexpr size_t fd_smem_bytes(int v) {
  return std::max(sizeof(FdSmem) * kFdOpw[v] * kFdWarps[v], sizeof(FdLargeSmem<P>));
}

// Thread blocks of a colour kernel that the device holds at once (SMs x
// blocks per SM, from the occupancy calculator; at least one), computed once
// per kernel and schedule on the device current at the first launch.
template <class P, bool REC, int V>
int fd_resident_blocks() {
  static const int n = [] {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fd_colour<P, kFdOpw[V], V == 0 ? 4 : 3, REC>, kFdWarps[V] * 32,
                                                  fd_smem_bytes<P>(V));
    return std::max(1, sms) * std::max(1, per_sm);
  }();
  return n;
}
template <class P, bool REC>
int fd_resident(int variant) {
  switch (variant) {
    case 0: return fd_resident_blocks<P, REC, 0>();
    case 1: return fd_resident_blocks<P, REC, 1>();
    case 2: return fd_resident_blocks<P, REC, 2>();
    case 3: return fd_resident_blocks<P, REC, 3>();
    default: return fd_resident_blocks<P, REC, 4>();
  }
}

template <class P>
constexpr size_t fd_spec_bytes() { return std::max(sizeof(FdSpecSmem), sizeof(FdLargeSmem<P>)); }
template <class P, bool REC>
int fd_spec_resident() {
  static const int n = [] {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fd_colour_spec<P, REC>, 64, fd_spec_bytes<P>());
    return std::max(1, sms) * std::max(1, per_sm);
  }();
  return n;
}

// Calls launch(colour, first, n, last) for the colour launches of a sweep: one
// per colour, or one per slice of each colour, its pair data staged before it
// by stage(job).
template <class Stage, class Launch>
void for_colours(const Consts& c, const Workspace& w, Stage stage, Launch launch) {
  const int64_t nown = colour_blocks(c), step = fd_sliced(c) ? kSliceBlocks : std::max<int64_t>(1, nown);
  for (int col = 0; col < 8; ++col)
    for (int64_t b = 0; b < nown; b += step) {
      const int64_t n = std::min(step, nown - b);
      if (fd_sliced(c)) stage(stage_job(n, w.blk_order + col * nown + b, col, w.st_pair));
      launch(col, b, n, b + n == nown);
    }
}

// The colour launches of one sweep with float32 pair arithmetic.  Few
// blocks spread over as many thread blocks (a warp that finds none left ends).
template <class P, bool REC, class Stage>
void launch_colours32(const Consts& c, const Workspace& w, int cur, double dt, uint64_t seed, int variant,
                      Stage stage, cudaStream_t s) {
  const int opw = kFdOpw[variant], W = kFdWarps[variant];
  FdRun<P> f;
  f.c = c;
  f.k = fd_const<float>(c, dt);
  f.a = view<P>(w, cur);
  f.qp4 = (typename P::V4*)w.qp4;
  f.cell_start = w.cell_start;
  f.mrank = w.mrank;
  f.xmx = w.xmin[0];
  f.xmy = w.xmin[1];
  f.xmz = w.xmin[2];
  f.hdr = w.sched_hdr;
  f.rsize = w.sched_rsize;
  f.sched_off = w.st_off;
  f.pairs = w.st_pair;
  f.geom = (const F4*)w.st_geom;
  f.rnd = (const F4*)w.st_rnd;
  f.seed = seed;
  f.sweep_ptr = w.sweep;
  f.counters = w.counters;
  f.status = w.status;
  f.recs = REC ? w.pair_recs : nullptr;
  f.rec_count = w.pair_rec_count;
  f.rec_cap = w.pair_rec_cap;
  f.pos = w.blk_pos;
  f.big_perm = w.big_perm;
  f.big_list = w.big_list;
  f.big_count = w.big_count;
  f.large_list = w.large_list;
  f.large_count = w.large_count;
  auto kern = opw == 1 ? k_fd_colour<P, 1, 3, REC> : (W == 2 ? k_fd_colour<P, 2, 4, REC> : k_fd_colour<P, 2, 3, REC>);
  // a team per block where a warp per block would run it (EMS: only there has
  // the test its own work)
  const bool spec = opw == 1 && c.scheme == SDPD_SCHEME_EMS;
  for_colours(c, w, stage, [&](int col, int64_t first, int64_t n, bool last) {
    f.colour = col;
    f.queue = w.fd_queue + 4 * col;
    f.order = w.blk_order + col * colour_blocks(c) + first;
    f.first = first;
    f.n = (unsigned)n;
    f.last = last;
    if (spec) {
      k_fd_colour_spec<P, REC>
          <<<(unsigned)std::min<int64_t>(n, fd_spec_resident<P, REC>()), 64, fd_spec_bytes<P>(), s>>>(f);
    } else {
      const unsigned g = (unsigned)std::min<int64_t>((n + opw - 1) / opw, fd_resident<P, REC>(variant));
      kern<<<g, W * 32, fd_smem_bytes<P>(variant), s>>>(f);
    }
  });
}

// Fills the resident-block counts of every block schedule ahead of time (a
// host query, kept out of stream captures).
void team64_prepare();
template <class Stage>
void launch_team64(const Consts& c, const Workspace& w, int cur, double dt, uint64_t seed, int record, Stage stage,
                   cudaStream_t s);

template <class P, class A>
void fd_prepare() {
  if constexpr (!A::mixed) {
    team64_prepare();
  } else {
    fd_spec_resident<P, false>();
    fd_spec_resident<P, true>();
    for (int v = 0; v < kFdVariants; ++v) {
      fd_resident<P, false>(v);
      fd_resident<P, true>(v);
    }
  }
}

template <class P, class A>
void stage_geometry(const Consts& c, const Workspace& w, const StageJob& job, cudaStream_t s) {
  auto kern = c.kernel == SDPD_KERNEL_LUCY ? k_stage_geometry<P, A, SDPD_KERNEL_LUCY>
                                           : k_stage_geometry<P, A, SDPD_KERNEL_CUBIC>;
  kern<<<stage_grid(job), kStageWarps * 32, 0, s>>>(c, (const typename P::V4*)w.qr4, w.cell_start, w.mrank, w.xmin[0],
                                                   w.xmin[1], w.xmin[2], w.sched_hdr, w.sched_off, w.sched_pair, job,
                                                   (typename A::V4*)w.st_geom);
}

// The staged geometry of every scheduled pair (the last launch of a schedule).
template <class P, class A>
void launch_stage_geometry(const Consts& c, const Workspace& w, cudaStream_t s) {
  if (c.N == 0 || fd_sliced(c)) return;
  stage_geometry<P, A>(c, w, stage_job(c.ncell, nullptr, 0, nullptr), s);
}

// One sweep: the random numbers of every scheduled pair, then the colours
// (sliced: geometry, random numbers and colour launch of each slice in turn);
// the last colour launch advances the sweep counter.
template <class P, class A>
void launch_fd_colours(const Consts& c, const Workspace& w, int cur, double dt, uint64_t seed, int record,
                       cudaStream_t s) {
  if (c.N == 0) {
    launch_advance_sweep(w, s);
    return;
  }
  auto random = [&](const StageJob& job) {
    k_stage_random<A><<<stage_grid(job), kStageWarps * 32, 0, s>>>(
        c, w.id[cur], w.cell_start, w.mrank, w.sched_hdr, w.sched_off, w.sched_pair, job, seed, w.sweep,
        (const typename A::V4*)w.st_geom, (typename A::V4*)w.st_rnd, w.st_aux);
  };
  auto stage = [&](const StageJob& job) {
    stage_geometry<P, A>(c, w, job, s);
    random(job);
  };
  if (!fd_sliced(c)) random(stage_job(c.ncell, nullptr, 0, nullptr));
  if constexpr (!A::mixed) {
    launch_team64(c, w, cur, dt, seed, record, stage, s);
  } else {
    if (record) launch_colours32<P, true>(c, w, cur, dt, seed, fd_launch_variant(c), stage, s);
    else launch_colours32<P, false>(c, w, cur, dt, seed, fd_launch_variant(c), stage, s);
  }
}

}  // namespace sdpd
