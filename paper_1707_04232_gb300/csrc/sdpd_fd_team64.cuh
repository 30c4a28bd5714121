// sdpd_fd_team64.cuh -- the colour kernel of the float64 sweep: a team of
// warps per block, four lanes per pair.
//
// GB300 issues one float64 warp instruction per 64 cycles on each quarter of
// an SM, whatever the number of active lanes and however independent the
// instructions are, so a round of a block's schedule costs its float64
// instructions times 64 cycles per warp: with one lane per pair about 340
// (13 of 32 lanes in use).  Here the four lanes of a pair share its
// arithmetic so that every lane of an instruction does a different part of
// it: lanes 0 to 2 hold the components of the vectors and the direction
// across e, lane 3 the energies and the direction along e.  The coefficients
// (exponential, square root), the components of the proposal and of the
// reverse noise, and the logarithms of the Metropolis ratio are each
// evaluated once per instruction for the whole pair: about 90 float64
// instructions per round.  Rounds hold at most 16 pairs (8 per warp).
// One pass of 1000 particles (EMS): 46.4 ms with one lane per pair, 8.1 ms
// now; 32,768 particles, two steps: 40.1 and 6.5 ms.
//
// EMS: the proposal and the Metropolis test (about half of them each) run on
// different warps, one round apart.  Two warps propose round r and write its
// moves into the shared state at once; while they go on to round r + 1, two
// others test round r.  When they reject a move (1e-4 to 3e-2 of the pairs)
// the proposers take round r + 1 back, then the rejected moves, and propose
// round r + 1 again, so the result is the sequential one.
#pragma once
#include "sdpd_f64.cuh"
#include "sdpd_fd_colour.cuh"

namespace sdpd {

// Constants of the team's arithmetic, in momentum units: with u = p_i - p_j,
// 2 dp = m (v' - v) = (alpha - 1) u + z G per direction, z = m zt,
// z^2 = 4 kB m / C_K * (eps_i eps_j / (eps_i + eps_j)) / (1 - d) * (1 - alpha^2).
struct Team64Const {
  double x_par, x_perp;  // log alpha per unit of base (1 - d): -2 kappa m^2 dt / m
  double d2;             // 2 kB / C_K
  double s;              // 4 kB m / C_K
  double de;             // -1 / (4 m)
  double CKm1;
  int scheme;
};

// alpha - 1 and (z or, INV, 1 / z) of this lane's direction at energies with
// sum E, product P and 1/E = iE.  With q = 1 - d and n = q z^2, z is
// n / sqrt(n q) and 1/z is q / sqrt(n q): one reciprocal square root.
template <bool INV>
__device__ __forceinline__ void team_coeffs(const Team64Const& k, double x_dir, double base, double P, double iE,
                                            double& m, double& z) {
  const double a = P * iE;
  const double q = __fma_rn(-k.d2, a * iE, 1.0);
  m = f64::expm1(x_dir * (base * q));
  const double n = k.s * a * (-m * (2.0 + m)), nq = n * q;
  if (f64::rsqrt_tiny(nq)) z = INV ? ::sqrt(q / n) : ::sqrt(n / q);
  else z = f64::rsqrt_(nq) * (INV ? q : n);
}

__device__ __forceinline__ double quad_sum(double v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v;
}

// What the test of a move needs from its proposal, per lane and per pair.
struct Team64Move {
  double m, z, u;         // this lane's alpha - 1, z, velocity component (momentum units)
  double deps, E, P, r0;  // energy change, sum and product of the energies before; r0: 1/P on lane 2
  bool bound;             // both new energies positive
};

// The proposal of one pair on the four lanes of a quad (whole warps call it).
// l: the lane's place in the quad; A, B: component l of the two particles'
// records (px, py, pz, eps); ge: component l of (e, base); Gl: component l of
// (G - (e.G) e, e.G).  A1, B1: the same components after the move.  Where a
// lane's own part leaves it idle it takes one of the pair's scalars in the
// same instruction: lane 3 the sum and the product of the energies.
__device__ __forceinline__ Team64Move team_propose(const Team64Const& k, int l, double A, double B, double ge,
                                                   double Gl, double base, double& A1, double& B1) {
  Team64Move v;
  const bool e_lane = l == 3;
  const double el = e_lane ? 0.0 : ge;
  const double u = A - (e_lane ? -B : B);                    // lane 3: E
  const double t = (e_lane ? A : ge) * (e_lane ? B : u);     // lane 3: P
  v.E = __shfl_sync(0xffffffffu, u, 3, 4);
  v.P = __shfl_sync(0xffffffffu, t, 3, 4);
  // lane 2 takes 1/P (for the entropy term) while the others take 1/E
  v.r0 = f64::rcp(l == 2 ? v.P : v.E);
  const double iE = __shfl_sync(0xffffffffu, v.r0, 0, 4);
  team_coeffs<false>(k, e_lane ? k.x_par : k.x_perp, base, v.P, iE, v.m, v.z);
  // u split along and across e: lane 3 holds the component along it
  const double upar = quad_sum(e_lane ? 0.0 : t);
  const double across = __fma_rn(-upar, el, u);
  v.u = e_lane ? upar : across;
  const double w = __fma_rn(v.m, v.u, v.z * Gl);
  const double wpar = __shfl_sync(0xffffffffu, w, 3, 4);
  const double sum = __fma_rn(wpar, el, w);
  const double dp2 = e_lane ? 0.0 : sum;  // 2 dp
  // kinetic energy change of the pair: dp . (u + dp) / m
  v.deps = k.de * quad_sum(dp2 * __fma_rn(0.5, dp2, u));
  const double d = e_lane ? v.deps : dp2;
  A1 = __fma_rn(e_lane ? 1.0 : 0.5, d, A);
  B1 = __fma_rn(e_lane ? 1.0 : -0.5, d, B);
  v.bound = __shfl_sync(0xffffffffu, (int)(f64::positive(A1) && f64::positive(B1)), 3, 4) != 0;
  return v;
}

// The Metropolis margin a - ln U of Eq. (metropolis-ratio) of a move: the
// reverse move from v' with the coefficients at the proposed energies, its
// noise per direction [(1 - alpha' alpha) u - alpha' z G] / z'.
// c0 = |G|^2 / 2 - ln U.
__device__ __forceinline__ double team_margin(const Team64Const& k, int l, const Team64Move& v, double Gl, double base,
                                              double c0) {
  const double E1 = v.E + v.deps;
  const double t = v.deps * E1;  // change of the product of the energies
  double mr, iz;
  team_coeffs<true>(k, l == 3 ? k.x_par : k.x_perp, base, v.P + t, f64::rcp(E1 + v.deps), mr, iz);
  const double cr = -__fma_rn(v.m, mr, v.m + mr);
  const double g = __fma_rn(cr, v.u, -(__fma_rn(mr, v.z, v.z) * Gl)) * iz;
  // ln|B(v)| - ln|B(v')| = ln(z / z') along + 2 ln(z / z') across e (lanes 3,
  // 0, 1); entropy (C_K/kB - 1) ln(eps' products / eps products) (lane 2)
  const bool ent = l == 2;
  const double lg = f64::log1p(__fma_rn(ent ? t : v.z, ent ? v.r0 : iz, ent ? 0.0 : -1.0));
  return c0 + quad_sum(__fma_rn(-0.5 * g, g, ent ? k.CKm1 * lg : lg));
}

constexpr int kTeamPairs = 16;    // pairs of a round
constexpr int kTeamThreads = 64;  // a quad per pair
template <bool EMS>
constexpr int team_threads() { return EMS ? 2 * kTeamThreads : kTeamThreads; }

// Shared memory of a team: the block's records (px, py, pz, eps), and the
// moves of two rounds.
struct Team64Smem {
  D4 s[kLargeBlock];
  FdCells cells;
  uint8_t rsize[kRoundStride];
  double m[2][kTeamThreads], z[2][kTeamThreads], u[2][kTeamThreads], r0[2][kTeamPairs];
  double deps[2][kTeamPairs], E[2][kTeamPairs], P[2][kTeamPairs], low[2][kTeamPairs];  // low: the lower new energy
  uint8_t bound[2][kTeamPairs];
  unsigned rejected[2][2];  // quads (their lanes' bits) of the round tested in a step, by its parity and per warp
  unsigned next;
};

template <bool EMS, bool REC>
__global__ void __launch_bounds__(team_threads<EMS>())
    k_fd_colour64(const __grid_constant__ Consts c, const __grid_constant__ FDConst<double> kbig, Team64Const k,
                  const __grid_constant__ Arrays<Fp64> a, D4* __restrict__ qp4,
                  const int32_t* __restrict__ cell_start, const int32_t* __restrict__ mrank,
                  const uint32_t* __restrict__ hdr, const uint8_t* __restrict__ rsize,
                  const unsigned long long* __restrict__ sched_off, const uint32_t* __restrict__ pairs,
                  const double* __restrict__ geom, const double* __restrict__ rnd, const double* __restrict__ aux,
                  int colour, unsigned nblk, bool last, uint64_t seed,
                  unsigned long long* __restrict__ sweep_ptr, unsigned long long* counters,
                  int* status, sdpd_pair_rec* recs, unsigned long long* rec_count, int64_t rec_cap,
                  unsigned* __restrict__ queue, const int32_t* __restrict__ order, int32_t* __restrict__ big_perm,
                  const int2* __restrict__ big_list, const uint32_t* __restrict__ big_count) {
  constexpr int kThreads = team_threads<EMS>();
  __shared__ Team64Smem sm;
  const uint64_t sweep = *sweep_ptr;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const bool tester = EMS && t >= kTeamThreads;
  const int tt = t % kTeamThreads, l = tt & 3, slot = tt >> 2;  // quad lane, pair of the round
  const int hx = c.nc[0] >> 1, hy = c.nc[1] >> 1, hz = c.nc[2] >> 1;
  const int64_t nown = (int64_t)hx * hy * hz;
  const double pi_coef = c.pi_coef;
  unsigned n_tot = 0, n_rb = 0, n_rm = 0;
  bool negative = false, bad = false;
  double* rec = reinterpret_cast<double*>(sm.s);
  // blocks from the colour's queue, deepest first (see k_fd_colour)
  for (;;) {
    if (t == 0) sm.next = atomicAdd(queue, 1u);
    __syncthreads();
    const unsigned wi = sm.next;
    if (wi >= nblk) break;
    const int64_t w = order[colour * nown + wi];
    const int ox = 2 * (int)(w % hx) + (colour & 1), oy = 2 * (int)((w / hx) % hy) + ((colour >> 1) & 1),
              oz = 2 * (int)(w / ((int64_t)hx * hy)) + ((colour >> 2) & 1);
    const int64_t o = ox + (int64_t)c.nc[0] * (oy + (int64_t)c.nc[1] * oz);
    const uint32_t hd = hdr[o];
    const int np = hd == kHdrBig ? 0 : (int)(hd & 0xffffu), nr = hd == kHdrBig ? 0 : (int)(hd >> 16 & 255u);
    if (np == 0) {  // (a block beyond capacity is swept below)
      __syncthreads();
      continue;
    }
    if (t == 0) n_tot += (unsigned)np;
    const unsigned long long first = sched_off[o];
    for (int r = t; r < nr; r += kThreads) sm.rsize[r] = rsize[o * kRoundStride + r];
    BlockCells b;
    block_cells(c, ox, oy, oz, mrank, cell_start, b);
    const int nb = b.base[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (t == q) {
        sm.cells.cst[q] = b.start[q];
        sm.cells.cbs[q] = b.base[q];
      }
    __syncthreads();
    for (int q = t; q < nb; q += kThreads) {
      const int g = block_gidx(sm.cells, q);
      sm.s[q] = D4{a.px[g], a.py[g], a.pz[g], a.eps[g]};
    }
    // this quad's pair of a round, loaded one round ahead; a tester meets
    // round r one step after its proposer.  The round sizes never exceed the
    // team's pairs (the schedule's width).
    uint32_t pr = 0;
    double ge = 0.0, Gl = 0.0, base = 0.0, c0 = 0.0;
    int pos = 0, n = sm.rsize[0];
    auto fetch = [&]() {
      if (slot < n) {
        const unsigned long long at = first + pos + slot;
        if (!tester || REC) pr = __ldg(&pairs[at]);
        if (!tester) ge = __ldg(&geom[4 * at + l]);
        base = __ldg(&geom[4 * at + 3]);
        Gl = __ldg(&rnd[4 * at + l]);
        if (tester) c0 = __ldg(&aux[at]);
      }
    };
    fetch();
    __syncthreads();
    uint32_t last_pr = 0;  // the proposer's pair of the round before, and its values before the move
    double lastA = 0.0, lastB = 0.0;
    const int steps = EMS ? nr + 1 : nr;
    for (int st = 0; st < steps; ++st) {
      const int r = tester ? st - 1 : st;  // this warp's round
      const bool on = r >= 0 && r < nr;
      const int cn = on ? n : 0, buf = r & 1;
      const bool act = slot < cn, busy = (tt & 32) / 4 < cn;  // this quad, this warp has a pair
      const uint32_t cpr = act ? pr : 0u;
      // (lanes without a pair run on values that keep to the short paths)
      const double cge = ge, cG = act ? Gl : 0.0, cb = act ? base : 0.01, cc = c0;
      if (on) {
        pos += n;
        n = r + 1 < nr ? (int)sm.rsize[r + 1] : 0;
        fetch();
      }
      const bool live = act && f64::positive(cb);  // at r = h the pair does nothing
      const int ia = cpr & 0xffffu, ib = cpr >> 16;
      double A = 0.0, B = 0.0;
      bool moved = false;
      Team64Move v;
      // proposes round r on the current state and moves it
      auto propose = [&]() {
        A = rec[4 * ia + l];
        B = rec[4 * ib + l];
        double A1, B1;
        v = team_propose(k, l, A, B, cge, cG, cb, A1, B1);
        moved = live && (v.bound || k.scheme == SDPD_SCHEME_SSA);
        if (moved) {
          rec[4 * ia + l] = A1;
          rec[4 * ib + l] = B1;
        }
        if (REC && l == 3) sm.low[buf][slot] = fmin(A1, B1);
        if (EMS && act) {
          sm.m[buf][tt] = v.m;
          sm.z[buf][tt] = v.z;
          sm.u[buf][tt] = v.u;
          if (l == 2) sm.r0[buf][slot] = v.r0;
          if (l == 0) {
            sm.deps[buf][slot] = v.deps;
            sm.E[buf][slot] = v.E;
            sm.P[buf][slot] = v.P;
            sm.bound[buf][slot] = v.bound;
          }
        }
      };
      int dcs = 0;
      double margin = 0.0;
      if (!tester) {
        if (busy) propose();
        if (REC && !EMS) __syncwarp();
        if (!EMS && live) {
          if (REC) margin = sm.low[buf][slot];
          if (k.scheme == SDPD_SCHEME_SSA) negative |= !v.bound;
          else dcs = v.bound ? 0 : 1;
        }
      } else {
        if (busy) {
          v.m = sm.m[buf][tt];
          v.z = sm.z[buf][tt];
          v.u = sm.u[buf][tt];
          v.r0 = sm.r0[buf][slot];
          v.deps = sm.deps[buf][slot];
          v.E = sm.E[buf][slot];
          v.P = sm.P[buf][slot];
          v.bound = sm.bound[buf][slot];
          const double mg = team_margin(k, l, v, cG, cb, cc);
          if (live) {
            dcs = !v.bound ? 1 : (f64::negative(mg) ? 2 : 0);  // 2: U > exp(a)
            if (REC) margin = v.bound ? mg : sm.low[buf][slot];
          }
        }
        const unsigned rej = __ballot_sync(0xffffffffu, dcs == 2);
        if (lane == 0) sm.rejected[st & 1][warp & 1] = rej;
      }
      if ((tester || !EMS) && act && l == 0) {
        n_rb += dcs == 1;
        n_rm += dcs == 2;
        if constexpr (REC) {
          const unsigned long long at = atomicAdd(rec_count, 1ull);
          if ((int64_t)at < rec_cap) {
            sdpd_pair_rec rc;
            rc.id_i = a.id[block_gidx(sm.cells, ia)];
            rc.id_j = a.id[block_gidx(sm.cells, ib)];
            rc.colour = colour;
            rc.owner = (int32_t)o;
            rc.decision = dcs;
            rc.level = r;
            rc.margin = margin;
            rc.margin_lo = margin;
            rc.margin_tol = 0.0;
            recs[at] = rc;
          }
        }
      }
      __syncthreads();
      if constexpr (EMS) {
        if (sm.rejected[st & 1][0] | sm.rejected[st & 1][1]) {
          // a move of the round before was rejected: this round's moves back,
          // then the rejected ones, then this round once more
          if (!tester && moved) {
            rec[4 * ia + l] = A;
            rec[4 * ib + l] = B;
          }
          __syncthreads();
          if (!tester && (sm.rejected[st & 1][warp & 1] >> lane & 1u)) {
            rec[4 * (last_pr & 0xffffu) + l] = lastA;
            rec[4 * (last_pr >> 16) + l] = lastB;
          }
          __syncthreads();
          if (!tester && busy) propose();
          __syncthreads();
        }
        last_pr = cpr;
        lastA = A;
        lastB = B;
      }
    }
    __syncthreads();
    for (int q = t; q < nb; q += kThreads) {
      const int g = block_gidx(sm.cells, q);
      const D4 v = lds4(&sm.s[q]);
      a.px[g] = v.x; a.py[g] = v.y; a.pz[g] = v.z;
      bad |= !isfinite(v.w);  // (an energy that was not finite once never is again)
      a.eps[g] = v.w;
      qp4[g].w = v.w * pi_coef / a.rho[g];  // pressure over rho^2 of the new energy, Eq. (pg-eos)
    }
    __syncthreads();  // the team's shared memory is refilled by the next block
  }
  // blocks beyond capacity, pair by pair, one per warp (by the colour's last launch)
  while (last) {
    unsigned bi = 0;
    if (lane == 0) bi = atomicAdd(&queue[2], 1u);
    bi = __shfl_sync(0xffffffffu, bi, 0);
    if (bi >= big_count[colour]) break;
    const int2 ent = big_list[colour * nown + bi];
    int bx, by, bz;
    owner_coords(c, ent.x, bx, by, bz);
    const BigCounts bc = fd_big_block<Fp64, Fp64>(c, kbig, a, qp4, cell_start, mrank, nullptr, nullptr, nullptr, ent.x,
                                                  bx, by, bz, colour, seed, sweep, REC ? recs : nullptr, rec_count,
                                                  rec_cap, big_perm + ent.y);
    if (lane == 0) {  // (lane 0 made the updates)
      atomicAdd(&counters[0], bc.tot);
      atomicAdd(&counters[1], bc.acc);
      atomicAdd(&counters[2], bc.rb);
      atomicAdd(&counters[3], bc.rm);
    }
    negative |= bc.negative != 0;
    bad |= bc.bad != 0;
  }
  if (lane == 0) {
    const unsigned total = gridDim.x * (unsigned)(kThreads / 32);
    __threadfence();  // this warp's last take from the queue is performed before it counts as done
    if (atomicAdd(&queue[1], 1u) == total - 1u) {
      queue[0] = 0u;
      queue[1] = 0u;
      queue[2] = 0u;
      if (colour == 7 && last) *sweep_ptr = sweep + 1ull;  // (every warp has read it) the sweep is done
    }
  }
  const unsigned c_tot = __reduce_add_sync(0xffffffffu, n_tot), c_rb = __reduce_add_sync(0xffffffffu, n_rb),
                 c_rm = __reduce_add_sync(0xffffffffu, n_rm);
  const unsigned any_neg = __any_sync(0xffffffffu, negative), any_bad = __any_sync(0xffffffffu, bad);
  if (lane == 0) {
    // (the team's pairs are counted on its first warp, rejections on others:
    // accepted = pairs - rejected, added with wrap-around)
    if (c_tot || c_rb || c_rm) {
      atomicAdd(&counters[0], (unsigned long long)c_tot);
      atomicAdd(&counters[1], (unsigned long long)c_tot - c_rb - c_rm);
      atomicAdd(&counters[2], (unsigned long long)c_rb);
      atomicAdd(&counters[3], (unsigned long long)c_rm);
    }
    if (any_neg) atomicOr(status, kStNegative);
    if (any_bad) atomicOr(status, kStNaN);
  }
}

// Thread blocks of the team kernel resident at once (see fd_resident_blocks).
template <bool EMS, bool REC>
int team64_resident() {
  static const int n = [] {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fd_colour64<EMS, REC>, team_threads<EMS>(), 0);
    return std::max(1, sms) * std::max(1, per_sm);
  }();
  return n;
}
void team64_prepare() {
  team64_resident<true, true>();
  team64_resident<true, false>();
  team64_resident<false, true>();
  team64_resident<false, false>();
}

template <bool EMS, bool REC, class Stage>
void launch_colours64(const Consts& c, const Workspace& w, int cur, double dt, uint64_t seed, Stage stage,
                      cudaStream_t s) {
  Team64Const k;
  k.x_par = -2.0 * c.kpar_m2 * (dt / c.m);
  k.x_perp = -2.0 * c.kperp_m2 * (dt / c.m);
  k.d2 = 2.0 * c.kB / c.C_K;
  k.s = 4.0 * c.kB * c.m / c.C_K;
  k.de = -0.25 / c.m;
  k.CKm1 = c.C_K / c.kB - 1.0;
  k.scheme = c.scheme;
  for_colours(c, w, stage, [&](int col, int64_t first, int64_t n, bool last) {
    const unsigned g = (unsigned)std::min<int64_t>(n, team64_resident<EMS, REC>());
    k_fd_colour64<EMS, REC><<<g, team_threads<EMS>(), 0, s>>>(
        c, fd_const<double>(c, dt), k, view<Fp64>(w, cur), (D4*)w.qp4, w.cell_start, w.mrank, w.sched_hdr,
        w.sched_rsize, w.st_off, w.st_pair, (const double*)w.st_geom, (const double*)w.st_rnd, w.st_aux, col,
        (unsigned)n, last, seed, w.sweep, w.counters, w.status, REC ? w.pair_recs : nullptr, w.pair_rec_count,
        w.pair_rec_cap, w.fd_queue + 4 * col, w.blk_order + first, w.big_perm, w.big_list, w.big_count);
  });
}
template <class Stage>
void launch_team64(const Consts& c, const Workspace& w, int cur, double dt, uint64_t seed, int record, Stage stage,
                   cudaStream_t s) {
  const bool ems = c.scheme == SDPD_SCHEME_EMS;
  if (ems && record) launch_colours64<true, true>(c, w, cur, dt, seed, stage, s);
  else if (ems) launch_colours64<true, false>(c, w, cur, dt, seed, stage, s);
  else if (record) launch_colours64<false, true>(c, w, cur, dt, seed, stage, s);
  else launch_colours64<false, false>(c, w, cur, dt, seed, stage, s);
}

}  // namespace sdpd
