// sdpd_pair.cu -- the two pair passes of Velocity Verlet: the density sum of
// Eq. (sdpd-rho-v) with the equation-of-state update of Section 3.1, and the
// conservative force of Eq. (cons-forces) with the half kick (and, for the
// first kick of a step, the drift and the cell binning of the new position).
//
// The neighbour search walks the 27 cells around the particle's cell (cell
// side >= h) with the predicate r^2 < h^2 after the periodic minimum image.
// Mixed path: one thread per particle in storage order (k_density, k_force).
// Float64 path: a group of kLanes64 lanes per particle (k_density64,
// k_force64).
#include "sdpd_f64.cuh"

namespace sdpd {

// Geometry of one home particle: displacement to a neighbour j.
// Float64: Home64 below.  Mixed: coordinates relative to the own cell's lower corner; per axis and
// neighbour offset o in {-1, 0, +1} the home coordinate shifted by the
// (exact, fixed-point) distance between the two cells' corners.
template <class P>
struct Home;

template <>
struct Home<Mixed> {
  float x, y, z, sx, sy, sz;
  int cx, cy, cz;
  const uint32_t *xmx, *xmy, *xmz;
  float hx, hy, hz;  // home coordinates in the frame of the current neighbour cell
  __device__ void init(const Consts& c, const F4& q, int cx_, int cy_, int cz_, const uint32_t* xmx_,
                       const uint32_t* xmy_, const uint32_t* xmz_) {
    x = q.x; y = q.y; z = q.z;
    sx = c.f_scale[0]; sy = c.f_scale[1]; sz = c.f_scale[2];
    cx = cx_; cy = cy_; cz = cz_;
    xmx = xmx_; xmy = xmy_; xmz = xmz_;
  }
  // shift into the frame of neighbour cell (nx, ny, nz): exact fixed-point
  // distance between the two cells' lower corners
  __device__ __forceinline__ void frame(int nx, int ny, int nz) {
    hx = x + (float)(int32_t)(__ldg(&xmx[cx]) - __ldg(&xmx[nx])) * sx;
    hy = y + (float)(int32_t)(__ldg(&xmy[cy]) - __ldg(&xmy[ny])) * sy;
    hz = z + (float)(int32_t)(__ldg(&xmz[cz]) - __ldg(&xmz[nz])) * sz;
  }
  __device__ __forceinline__ void disp(const F4& qj, float& dx, float& dy, float& dz) const {
    dx = hx - qj.x;
    dy = hy - qj.y;
    dz = hz - qj.z;
  }
  // all nine shifted home coordinates, for walking a neighbour list
  float fx[3], fy[3], fz[3];
  __device__ __forceinline__ void frames_all(const Consts& c) {
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      int nx = cx + o - 1, ny = cy + o - 1, nz = cz + o - 1;
      nx += nx < 0 ? c.nc[0] : (nx >= c.nc[0] ? -c.nc[0] : 0);
      ny += ny < 0 ? c.nc[1] : (ny >= c.nc[1] ? -c.nc[1] : 0);
      nz += nz < 0 ? c.nc[2] : (nz >= c.nc[2] ? -c.nc[2] : 0);
      frame(nx, ny, nz);
      fx[o] = hx; fy[o] = hy; fz[o] = hz;
    }
  }
  __device__ __forceinline__ static float pick(const float* v, uint32_t k) {
    return k == 0 ? v[0] : (k == 1 ? v[1] : v[2]);
  }
  __device__ __forceinline__ void disp_code(uint32_t code, const F4& qj, float& dx, float& dy, float& dz) const {
    dx = pick(fx, code & 3u) - qj.x;
    dy = pick(fy, (code >> 2) & 3u) - qj.y;
    dz = pick(fz, (code >> 4) & 3u) - qj.z;
  }
};

__device__ __forceinline__ int wrapc(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// ---------------------------------------------------------------------------
// Density, Eq. (sdpd-rho-v): rho_i = m W(0) + sum_{j != i, r_ij < h} m W(r_ij);
// then the energies at fixed entropy (Section 3.1): S_i = S(eps_i, rho_old),
// eps_i = E(S_i, rho_i), and pi_i = P_i / rho_i^2 from Eq. (pg-eos):
// P = c_rho rho eps / (C_K m).
// ---------------------------------------------------------------------------
template <class P, int KIND>
__global__ void __launch_bounds__(128, 12) k_density(Consts c, Arrays<P> a, typename P::V4* __restrict__ qp4,
                                                 const int32_t* __restrict__ cell_start,
                                                 const int32_t* __restrict__ mrank,
                                                 const uint32_t* __restrict__ xmx,
                                                 const uint32_t* __restrict__ xmy,
                                                 const uint32_t* __restrict__ xmz, int update_eos,
                                                 int32_t* __restrict__ ncount_by_id,
                                                 uint32_t* __restrict__ nlist, int32_t* __restrict__ nn,
                                                 int32_t* __restrict__ ovf_list, int32_t* __restrict__ ovf_count,
                                                 int32_t* __restrict__ ovf_other,
                                                 typename P::V4* __restrict__ qr4, uint32_t* __restrict__ cend) {
  static_assert(P::mixed, "the float64 path runs k_density64");
  using R = typename P::R;
  using V4 = typename P::V4;
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i == 0) *ovf_other = 0;  // the other buffer's list: its readers have run
  if (i >= c.N) return;
  const V4 qi = ld4(&a.q4[i]);
  int cx, cy, cz;
  unpack_cell(w_to_cellbits(qi.w), cx, cy, cz);
  Home<P> home;
  home.init(c, qi, cx, cy, cz, xmx, xmy, xmz);
  const R h2 = (R)c.h2, inv_h = R(1) / (R)c.h, cW = (R)c.cW;
  R acc = R(0);
  int cnt = 0;
  uint32_t* wp = nlist + nbr_slot(i, 0, c.nbr_cap);  // where entry cnt of the list goes
  // Every lane walks the 27 cells in the same order (z, then y, then x
  // offset, each -1, 0, +1), so the warp's loops stay converged.  Per row
  // (oz, oy) of three cells, cend[row][i] records where the list stands:
  // byte 0 at the row's start, byte 1 + k after its k-th cell (counts
  // clamped to 255).  The sweep's schedule finds each block's pairs in
  // these cell runs of the list.
#pragma unroll 1
  for (int oz = -1; oz <= 1; ++oz) {
    const int nz = wrapc(cz + oz, c.nc[2]);
#pragma unroll 1
    for (int oy = -1; oy <= 1; ++oy) {
      const int ny = wrapc(cy + oy, c.nc[1]);
      uint32_t rw = (uint32_t)min(cnt, 255);
#pragma unroll 1
      for (int ox = -1; ox <= 1; ++ox) {
        const int nx = wrapc(cx + ox, c.nc[0]);
        const int r = __ldg(&mrank[nx + c.nc[0] * (ny + c.nc[1] * nz)]);
        const int beg = __ldg(&cell_start[r]), end = __ldg(&cell_start[r + 1]);
        home.frame(nx, ny, nz);
        const uint32_t code = nbr_entry(0, ox, oy, oz);
#pragma unroll 4
        for (int j = beg; j < end; ++j) {
          const V4 qj = ld4(&a.q4[j]);
          R dx, dy, dz;
          home.disp(qj, dx, dy, dz);
          const R r2 = r2_of(dx, dy, dz);
          // kept neighbours (about one candidate in six) take the short
          // branch: the kernel value and one list store at a stepped address
          if (r2 < h2 && j != i) {
            acc += kernel_W<KIND>(pair_r(r2) * inv_h, cW);
            if (cnt < c.nbr_cap) *wp = ((uint32_t)j << 6) | code;
            wp += (cnt & 3) == 3 ? 125 : 1;  // nbr_slot(i, cnt + 1) - nbr_slot(i, cnt)
            ++cnt;
          }
        }
        rw |= (uint32_t)min(cnt, 255) << (8 * (ox + 2));
      }
      cend[(int64_t)((oz + 1) * 3 + (oy + 1)) * c.N + i] = rw;
    }
  }
  if (ncount_by_id) ncount_by_id[a.id[i]] = cnt;
  nn[i] = cnt;
  if (cnt > c.nbr_cap) ovf_list[atomicAdd(ovf_count, 1)] = (int32_t)i;  // forces from the cells
  const R rho_new = c.f_m * (c.f_W0 + acc);
  double e = a.eps[i];
  if (update_eos) {
    // eps * (rho_new / rho_old)^(c_rho / C_K), the factor minus one formed
    // from log1p / expm1 of small arguments so float32 keeps it accurate
    const float ro = a.rho[i];
    const float g = expm1f(c.f_eos * log1pf((rho_new - ro) / ro));
    e = fma(e, (double)g, e);
    a.eps[i] = e;
  }
  a.rho[i] = rho_new;
  const R pi = (float)e * c.f_pi_coef / rho_new;
  V4 o = qi;
  o.w = pi;
  st4(&qp4[i], o);
  o.w = rho_new;  // positions and density together for the sweep's pair geometry
  st4(&qr4[i], o);
}

// Density, equation of state and neighbour lists of PPB particles per thread
// block (see k_density).  The list in shared memory has the layout of the
// global one, so it is copied out in 16-byte pieces.  A particle with more
// neighbours than a row holds sums the kernel over the cells again.  The
// equation of state runs one particle per lane on the first warp.
template <int KIND, int T, int PPB>
__global__ void __launch_bounds__(PPB * T)
    k_density64(Consts c, Arrays<Fp64> a, D4* __restrict__ qp4, const int32_t* __restrict__ cell_start,
                const int32_t* __restrict__ mrank, int update_eos, int32_t* __restrict__ ncount_by_id,
                uint32_t* __restrict__ nlist, int32_t* __restrict__ nn, const float4* __restrict__ qf4,
                D4* __restrict__ qr4, uint32_t* __restrict__ cend) {
  extern __shared__ __align__(16) uint32_t list_s[];  // [cap / 4][PPB][4], read as uint4
  __shared__ double acc_s[PPB];
  __shared__ int cnt_s[PPB];
  const int p = threadIdx.x / T, gl = threadIdx.x % T;
  const int64_t i0 = blockIdx.x * (int64_t)PPB, i = i0 + p;
  const bool live = i < c.N;
  const D4 qi = ld4(&a.q4[live ? i : 0]);
  const float4 fi = qf4[live ? i : 0];
  int cx, cy, cz;
  unpack_cell(__float_as_uint(fi.w), cx, cy, cz);
  Home64 home;
  home.init(c, qi, cx, cy, cz);
  const int cnt = walk64<T>(
      c, live, home, fi, i, cx, cy, cz, a.q4, qf4, cell_start, mrank,
      [&](int r, uint32_t rw) { if (live && gl == 0) cend[(int64_t)r * c.N + i] = rw; },
      [&](int k, int j, uint32_t code) {
        if (k < c.nbr_cap) list_s[((k >> 2) * PPB + p) * 4 + (k & 3)] = ((uint32_t)j << 6) | code;
      });
  __syncwarp();
  double acc = 0.0;
  const bool over = cnt > c.nbr_cap;
  for (int k = gl; k < (over ? 0 : cnt); k += T) {
    const uint32_t e = list_s[((k >> 2) * PPB + p) * 4 + (k & 3)];
    double dx, dy, dz;
    const double r2 = home.r2(e & 63u, ld4(&a.q4[e >> 6]), dx, dy, dz);
    acc += W64<KIND>(pair_r64(r2), c.inv_h);
  }
  if (__any_sync(0xffffffffu, over))
    walk64<T>(c, over, home, fi, i, cx, cy, cz, a.q4, qf4, cell_start, mrank, [](int, uint32_t) {},
              [&](int, int j, uint32_t code) {
                double dx, dy, dz;
                acc += W64<KIND>(pair_r64(home.r2(code, ld4(&a.q4[j]), dx, dy, dz)), c.inv_h);
              });
  acc = group_sum<T>(acc);
  if (gl == 0) {
    acc_s[p] = acc;
    cnt_s[p] = cnt;
  }
  __syncthreads();
  // the lists, row by row of four entries
  const int kmax = c.nbr_cap >> 2;
  for (int t = threadIdx.x; t < kmax * PPB; t += PPB * T) {
    const int k4 = t / PPB, q = t % PPB;
    if (4 * k4 < cnt_s[q])
      *reinterpret_cast<uint4*>(nlist + nbr_slot(i0 + q, 4 * k4, c.nbr_cap)) = reinterpret_cast<const uint4*>(list_s)[t];
  }
  if (threadIdx.x < PPB && i0 + threadIdx.x < c.N) {
    const int64_t g = i0 + threadIdx.x;
    const int cnt = cnt_s[threadIdx.x];
    if (ncount_by_id) ncount_by_id[a.id[g]] = cnt;
    nn[g] = cnt;
    const double rho_new = c.m * __fma_rn(c.cW, acc_s[threadIdx.x], c.W0);
    double e = a.eps[g];
    if (update_eos) {
      // eps' = E(S(eps, rho), rho') = eps (rho' / rho)^(c_rho / C_K); a
      // negative energy (SSA) has no entropy: NaN
      const double ro = a.rho[g];
      e *= exp(c.c_rho / c.C_K * log1p((rho_new - ro) / ro));
      if (f64::negative(e)) e = __longlong_as_double(0x7ff8000000000000ll);
      a.eps[g] = e;
    }
    a.rho[g] = rho_new;
    D4 o = ld4(&a.q4[g]);
    o.w = e * c.pi_coef / rho_new;
    st4(&qp4[g], o);
    o.w = rho_new;  // positions and density together for the sweep's pair geometry
    st4(&qr4[g], o);
  }
}

// Kick (and, with dt_drift != 0, drift and binning) of particle i with the
// force sum f (before the factor m^2): p_i += m^2 f dt/2 of Eq. (sdpd-verlet),
// q_i += p_i dt/m wrapped, and the new cell counted for the sort.
template <class P>
__device__ __forceinline__ void kick_particle(const Consts& c, const Arrays<P>& a, int64_t i, typename P::R fx,
                                              typename P::R fy, typename P::R fz, double half_dt, double dt_drift,
                                              typename P::Q* __restrict__ qdx, typename P::Q* __restrict__ qdy,
                                              typename P::Q* __restrict__ qdz, int32_t* __restrict__ key,
                                              int32_t* __restrict__ slot, int32_t* __restrict__ cell_count,
                                              const int32_t* __restrict__ mrank, double* __restrict__ force_by_id,
                                              const float drift_f[3]) {
  using R = typename P::R;
  const R m2 = c.f_m2;
  fx *= m2; fy *= m2; fz *= m2;
  if (force_by_id) {
    const int64_t k = a.id[i];
    force_by_id[3 * k] = fx;
    force_by_id[3 * k + 1] = fy;
    force_by_id[3 * k + 2] = fz;
  }
  const R hdt = (R)half_dt;  // one conversion per thread
  R px = a.px[i] + fx * hdt, py = a.py[i] + fy * hdt, pz = a.pz[i] + fz * hdt;
  a.px[i] = px; a.py[i] = py; a.pz[i] = pz;
  if (dt_drift != 0.0) {
    int nc3[3];
    // fixed point: the displacement in units of L / 2^32, wrap-around = periodic
    uint32_t ux = a.qx[i] + (uint32_t)__float2int_rn(px * drift_f[0]);
    uint32_t uy = a.qy[i] + (uint32_t)__float2int_rn(py * drift_f[1]);
    uint32_t uz = a.qz[i] + (uint32_t)__float2int_rn(pz * drift_f[2]);
    qdx[i] = ux; qdy[i] = uy; qdz[i] = uz;
    nc3[0] = (int)__umulhi(ux, (uint32_t)c.nc[0]);
    nc3[1] = (int)__umulhi(uy, (uint32_t)c.nc[1]);
    nc3[2] = (int)__umulhi(uz, (uint32_t)c.nc[2]);
    const int r = mrank[nc3[0] + c.nc[0] * (nc3[1] + c.nc[1] * nc3[2])];
    key[i] = r;
    slot[i] = atomicAdd(&cell_count[r], 1);
  }
}

// Force and kick of a particle with more neighbours than its list row
// holds: the pair force sum from the 27 cells around it, with the
// candidates, the predicate and the order of the density pass, so that the
// sum is the one a long enough list would give.
template <class P, int KIND>
__device__ __forceinline__ void force_from_cells(const Consts& c, const Arrays<P>& a, int64_t i,
                                              const typename P::V4* __restrict__ qp4,
                                              const int32_t* __restrict__ cell_start,
                                              const int32_t* __restrict__ mrank, const uint32_t* xmx,
                                              const uint32_t* xmy, const uint32_t* xmz, double half_dt,
                                              double dt_drift, typename P::Q* qdx, typename P::Q* qdy,
                                              typename P::Q* qdz, int32_t* key, int32_t* slot,
                                              int32_t* cell_count, double* force_by_id, float3 drift3) {
  using R = typename P::R;
  using V4 = typename P::V4;
  const V4 qi = ld4(&qp4[i]);
  int cx, cy, cz;
  unpack_cell(w_to_cellbits(ld4(&a.q4[i]).w), cx, cy, cz);
  Home<P> home;
  home.init(c, qi, cx, cy, cz, xmx, xmy, xmz);
  const R h2 = c.f_h2, inv_h = c.f_inv_h, cF = c.f_cF;
  R fx = R(0), fy = R(0), fz = R(0);
  for (int oz = -1; oz <= 1; ++oz) {
    const int nz = wrapc(cz + oz, c.nc[2]);
    for (int oy = -1; oy <= 1; ++oy) {
      const int ny = wrapc(cy + oy, c.nc[1]);
      for (int ox = -1; ox <= 1; ++ox) {
        const int nx = wrapc(cx + ox, c.nc[0]);
        const int r = __ldg(&mrank[nx + c.nc[0] * (ny + c.nc[1] * nz)]);
        const int beg = __ldg(&cell_start[r]), end = __ldg(&cell_start[r + 1]);
        home.frame(nx, ny, nz);
        for (int j = beg; j < end; ++j) {
          if (j == i) continue;
          const V4 qj = ld4(&qp4[j]);
          R dx, dy, dz;
          home.disp(qj, dx, dy, dz);
          const R r2 = r2_of(dx, dy, dz);
          if (r2 < h2) {
            const R s = (qi.w + qj.w) * kernel_F<KIND>(pair_r(r2) * inv_h, cF);
            fx += s * dx;
            fy += s * dy;
            fz += s * dz;
          }
        }
      }
    }
  }
  const float drift_f[3] = {drift3.x, drift3.y, drift3.z};
  kick_particle<P>(c, a, i, fx, fy, fz, half_dt, dt_drift, qdx, qdy, qdz, key, slot, cell_count, mrank,
                   force_by_id, drift_f);
}

// ---------------------------------------------------------------------------
// Conservative force, Eq. (cons-forces): F_i = sum_{j != i, r_ij < h}
// m^2 (pi_i + pi_j) F(r_ij) r_ij, and the kick p_i += F_i dt/2 of Eq.
// (sdpd-verlet).  With drift: q_i += p_i dt/m (wrapped), new cell counted
// for the sort.  A particle whose neighbour list overflowed its row (listed
// by the density pass) is left to k_force_overflow.
// ---------------------------------------------------------------------------
template <class P, int KIND>
__global__ void __launch_bounds__(128, KIND == SDPD_KERNEL_LUCY ? 16 : 12) k_force(Consts c, Arrays<P> a, const typename P::V4* __restrict__ qp4,
                                               const int32_t* __restrict__ cell_start,
                                               const int32_t* __restrict__ mrank,
                                               const uint32_t* __restrict__ xmx,
                                               const uint32_t* __restrict__ xmy,
                                               const uint32_t* __restrict__ xmz, double half_dt,
                                               double dt_drift, typename P::Q* __restrict__ qdx,
                                               typename P::Q* __restrict__ qdy,
                                               typename P::Q* __restrict__ qdz, int32_t* __restrict__ key,
                                               int32_t* __restrict__ slot, int32_t* __restrict__ cell_count,
                                               double* __restrict__ force_by_id,
                                               const uint32_t* __restrict__ nlist, const int32_t* __restrict__ nn,
                                               float3 drift3) {
  // mixed path: dt / m * 2^32 / L per axis, computed on the host
  const float drift_f[3] = {drift3.x, drift3.y, drift3.z};
  using R = typename P::R;
  using V4 = typename P::V4;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int n = i < c.N ? nn[i] : 0;
  if (i < c.N && n <= c.nbr_cap) {
    const V4 qi = ld4(&a.q4[i]);
    const R pi_i = ld4(&qp4[i]).w;
    int cx, cy, cz;
    unpack_cell(w_to_cellbits(qi.w), cx, cy, cz);
    Home<P> home;
    home.init(c, qi, cx, cy, cz, xmx, xmy, xmz);
    const R inv_h = c.f_inv_h, cF = c.f_cF;
    R fx = R(0), fy = R(0), fz = R(0);
    home.frames_all(c);
    // four entries per 16-byte load (a warp's loads are contiguous, see
    // nbr_slot), then four independent neighbour gathers
    for (int k = 0; k < n; k += 4) {
      const uint4 e4 = __ldg(reinterpret_cast<const uint4*>(nlist + nbr_slot(i, k, c.nbr_cap)));
      const uint32_t ev[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (k + u < n) {
          const uint32_t e = ev[u];
          const V4 qj = ld4(&qp4[e >> 6]);
          R dx, dy, dz;
          home.disp_code(e & 63u, qj, dx, dy, dz);
          const R r2 = r2_of(dx, dy, dz);
          const R s = (pi_i + qj.w) * kernel_F<KIND>(pair_r(r2) * inv_h, cF);
          fx += s * dx;
          fy += s * dy;
          fz += s * dz;
        }
      }
    }
    kick_particle<P>(c, a, i, fx, fy, fz, half_dt, dt_drift, qdx, qdy, qdz, key, slot, cell_count, mrank,
                     force_by_id, drift_f);
  }
}

// Force and kick of the float64 path: T lanes per particle over its list (see
// k_force and the note at kLanes64), or over the cells when the list
// overflowed its row; the kick, drift and binning one axis per lane.
template <int KIND, int T>
__global__ void __launch_bounds__(128)
    k_force64(Consts c, Arrays<Fp64> a, const D4* __restrict__ qp4, const float4* __restrict__ qf4,
              const int32_t* __restrict__ cell_start, const int32_t* __restrict__ mrank, double half_dt,
              double dt_drift, double* __restrict__ qdx, double* __restrict__ qdy, double* __restrict__ qdz,
              int32_t* __restrict__ key, int32_t* __restrict__ slot, int32_t* __restrict__ cell_count,
              double* __restrict__ force_by_id, const uint32_t* __restrict__ nlist, const int32_t* __restrict__ nn) {
  const int gl = threadIdx.x % T;
  int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / T;
  const bool mine = i < c.N;
  if (!mine) i = 0;  // (the whole warp stays for the sums)
  const int n = mine ? nn[i] : 0;
  const bool over = n > c.nbr_cap;
  const D4 qi = ld4(&qp4[i]);
  const float4 fi = qf4[i];
  int cx, cy, cz;
  unpack_cell(__float_as_uint(fi.w), cx, cy, cz);
  Home64 home;
  home.init(c, qi, cx, cy, cz);
  double f[3] = {0.0, 0.0, 0.0};
  auto add = [&](uint32_t code, const D4& qj) {
    double dx, dy, dz;
    const double r2 = home.r2(code, qj, dx, dy, dz);
    const double s = (qi.w + qj.w) * F64<KIND>(pair_r64(r2), c.inv_h);
    f[0] += s * dx;
    f[1] += s * dy;
    f[2] += s * dz;
  };
#pragma unroll 2
  for (int k = gl; k < (over ? 0 : n); k += T) {
    const uint32_t e = __ldg(&nlist[nbr_slot(i, k, c.nbr_cap)]);
    add(e & 63u, ld4(&qp4[e >> 6]));
  }
  if (__any_sync(0xffffffffu, over))
    walk64<T>(c, over, home, fi, i, cx, cy, cz, qp4, qf4, cell_start, mrank, [](int, uint32_t) {},
              [&](int, int j, uint32_t code) { add(code, ld4(&qp4[j])); });
#pragma unroll
  for (int d = 0; d < 3; ++d) f[d] = group_sum<T>(f[d]);
  // axis gl of the kick and drift (see kick_particle)
  int cc = 0;
  if (mine && gl < 3) {
    const double fd = (gl == 0 ? f[0] : (gl == 1 ? f[1] : f[2])) * (c.m * c.m * c.cF);
    if (force_by_id) force_by_id[3 * (int64_t)a.id[i] + gl] = fd;
    double* pp = gl == 0 ? a.px : (gl == 1 ? a.py : a.pz);
    const double pn = pp[i] + fd * half_dt;
    pp[i] = pn;
    if (dt_drift != 0.0) {
      const double* qq = gl == 0 ? a.qx : (gl == 1 ? a.qy : a.qz);
      const double L = c.L[gl];
      const double step = __dmul_rn(pn, dt_drift);
      double x = __dadd_rn(qq[i], c.m == 1.0 ? step : __ddiv_rn(step, c.m));
      if (x >= L) x = __dsub_rn(x, L);
      else if (x < 0.0) x = __dadd_rn(x, L);
      if (x >= L) x = 0.0;
      (gl == 0 ? qdx : (gl == 1 ? qdy : qdz))[i] = x;
      // floor(x / cs): from a product unless it comes near a whole number
      // (x / cs < 2^10, so the product is within 2^-40 of the quotient)
      const double qt = x * c.inv_cs[gl];
      cc = (int)qt;
      const float fr = (float)(qt - (double)cc);
      if (fr < 1e-6f || fr > 1.0f - 1e-6f) cc = (int)floor(__ddiv_rn(x, c.cs[gl]));
      cc = cc >= c.nc[gl] ? c.nc[gl] - 1 : (cc < 0 ? 0 : cc);
    }
  }
  if (dt_drift != 0.0) {
    const int cy2 = __shfl_sync(0xffffffffu, cc, 1, T), cz2 = __shfl_sync(0xffffffffu, cc, 2, T);
    if (mine && gl == 0) {
      const int r = mrank[cc + c.nc[0] * (cy2 + c.nc[1] * cz2)];
      key[i] = r;
      slot[i] = atomicAdd(&cell_count[r], 1);
    }
  }
}

// The particles that k_force left: more neighbours than a list row holds.
// A few thread blocks loop over the density pass's overflow list (usually
// empty: the launch then ends at once).
constexpr int kOverflowBlocks = 4;
template <class P, int KIND>
__global__ void __launch_bounds__(128) k_force_overflow(Consts c, Arrays<P> a, const typename P::V4* __restrict__ qp4,
                                                        const int32_t* __restrict__ cell_start,
                                                        const int32_t* __restrict__ mrank,
                                                        const uint32_t* __restrict__ xmx,
                                                        const uint32_t* __restrict__ xmy,
                                                        const uint32_t* __restrict__ xmz, double half_dt,
                                                        double dt_drift, typename P::Q* __restrict__ qdx,
                                                        typename P::Q* __restrict__ qdy,
                                                        typename P::Q* __restrict__ qdz, int32_t* __restrict__ key,
                                                        int32_t* __restrict__ slot, int32_t* __restrict__ cell_count,
                                                        double* __restrict__ force_by_id, float3 drift3,
                                                        const int32_t* __restrict__ ovf_list,
                                                        const int32_t* __restrict__ ovf_count) {
  const int novf = *ovf_count;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < novf; q += gridDim.x * blockDim.x)
    force_from_cells<P, KIND>(c, a, ovf_list[q], qp4, cell_start, mrank, xmx, xmy, xmz, half_dt, dt_drift, qdx, qdy,
                              qdz, key, slot, cell_count, force_by_id, drift3);
}

static inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// threads per block of the pair passes (one thread per particle, no shared
// memory, so any of the accepted sizes gives the same results)
static inline int pair_block(const Consts& c) { return pair_threads_ok(c.pair_threads) ? c.pair_threads : 128; }

template <int KIND>
static void launch_density64(const Consts& c, const Workspace& w, const Arrays<Fp64>& a, int update_eos,
                             int32_t* ncount_by_id, cudaStream_t s) {
  const bool wide = pair64_wide(c);
  const int t = wide ? 128 : pair_block(c), ppb = wide ? 4 : t / kLanes64;
  auto kern = wide ? k_density64<KIND, 32, 4>
                   : (t == 32 ? k_density64<KIND, kLanes64, 32 / kLanes64>
                              : (t == 64 ? k_density64<KIND, kLanes64, 64 / kLanes64>
                                         : k_density64<KIND, kLanes64, 128 / kLanes64>));
  kern<<<blocks_for(c.N, ppb), t, (size_t)c.nbr_cap * ppb * 4, s>>>(
      c, a, (D4*)w.qp4, w.cell_start, w.mrank, update_eos, ncount_by_id, w.nlist, w.nn, w.qf4,
      (D4*)w.qr4, w.cend);
}

template <class P>
void launch_density(const Consts& c, const Workspace& w, int cur, int update_eos, int32_t* ncount_by_id,
                    cudaStream_t s) {
  if (c.N == 0) return;
  Arrays<P> a = view<P>(w, cur);
  if constexpr (P::mixed) {
    int32_t* ovf_list = w.ovf_list + (size_t)cur * (size_t)c.N;  // this buffer's overflow list
    int32_t* ovf_count = w.ovf_count + cur;
    int32_t* ovf_other = w.ovf_count + (cur ^ 1);
    const int t = pair_block(c);
    auto kern = c.kernel == SDPD_KERNEL_LUCY ? k_density<P, SDPD_KERNEL_LUCY> : k_density<P, SDPD_KERNEL_CUBIC>;
    kern<<<blocks_for(c.N, t), t, 0, s>>>(c, a, (typename P::V4*)w.qp4, w.cell_start, w.mrank, w.xmin[0], w.xmin[1],
                                          w.xmin[2], update_eos, ncount_by_id, w.nlist, w.nn, ovf_list, ovf_count,
                                          ovf_other, (typename P::V4*)w.qr4, w.cend);
  } else if (c.kernel == SDPD_KERNEL_LUCY) {
    launch_density64<SDPD_KERNEL_LUCY>(c, w, a, update_eos, ncount_by_id, s);
  } else {
    launch_density64<SDPD_KERNEL_CUBIC>(c, w, a, update_eos, ncount_by_id, s);
  }
}

template <class P, int KIND>
static void launch_force_kind(const Consts& c, const Workspace& w, int cur, const Arrays<P>& a, double half_dt,
                              double dt_drift, double* force_by_id, cudaStream_t s) {
  auto qp4 = (const typename P::V4*)w.qp4;
  auto qdx = (typename P::Q*)w.qdx;
  auto qdy = (typename P::Q*)w.qdy;
  auto qdz = (typename P::Q*)w.qdz;
  if constexpr (P::mixed) {
    const float3 drift3 =
        make_float3((float)(dt_drift / c.m * c.inv_scale[0]), (float)(dt_drift / c.m * c.inv_scale[1]),
                    (float)(dt_drift / c.m * c.inv_scale[2]));
    const int t = pair_block(c);
    k_force<P, KIND><<<blocks_for(c.N, t), t, 0, s>>>(
        c, a, qp4, w.cell_start, w.mrank, w.xmin[0], w.xmin[1], w.xmin[2], half_dt, dt_drift, qdx, qdy, qdz, w.key,
        w.slot, w.cell_count, force_by_id, w.nlist, w.nn, drift3);
    k_force_overflow<P, KIND><<<kOverflowBlocks, 128, 0, s>>>(
        c, a, qp4, w.cell_start, w.mrank, w.xmin[0], w.xmin[1], w.xmin[2], half_dt, dt_drift, qdx, qdy, qdz, w.key,
        w.slot, w.cell_count, force_by_id, drift3, w.ovf_list + (size_t)cur * (size_t)c.N, w.ovf_count + cur);
  } else {
    const int t = pair_block(c), lanes = pair64_wide(c) ? 32 : kLanes64;
    auto kern = lanes == 32 ? k_force64<KIND, 32> : k_force64<KIND, kLanes64>;
    kern<<<blocks_for(c.N * lanes, t), t, 0, s>>>(c, a, qp4, w.qf4, w.cell_start, w.mrank, half_dt, dt_drift, qdx, qdy,
                                                  qdz, w.key, w.slot, w.cell_count, force_by_id, w.nlist, w.nn);
  }
}

template <class P>
void launch_force(const Consts& c, const Workspace& w, int cur, double half_dt, double dt_drift,
                  double* force_by_id, cudaStream_t s) {
  if (c.N == 0) return;
  const Arrays<P> a = view<P>(w, cur);
  if (c.kernel == SDPD_KERNEL_LUCY) launch_force_kind<P, SDPD_KERNEL_LUCY>(c, w, cur, a, half_dt, dt_drift, force_by_id, s);
  else launch_force_kind<P, SDPD_KERNEL_CUBIC>(c, w, cur, a, half_dt, dt_drift, force_by_id, s);
}

template void launch_density<Fp64>(const Consts&, const Workspace&, int, int, int32_t*, cudaStream_t);
template void launch_density<Mixed>(const Consts&, const Workspace&, int, int, int32_t*, cudaStream_t);
template void launch_force<Fp64>(const Consts&, const Workspace&, int, double, double, double*,
                                 cudaStream_t);
template void launch_force<Mixed>(const Consts&, const Workspace&, int, double, double, double*,
                                  cudaStream_t);

}  // namespace sdpd
