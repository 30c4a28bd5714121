// sdpd_fd.cu -- the pairwise fluctuation/dissipation sweep (Sections 3.2-3.3)
// made data-parallel by a conflict-free pair colouring.
//
// Colouring.  A pair whose particles sit in cells a and b (equal or adjacent
// along each axis, since the cell side is >= h) is owned by a cell o such that
// both cells lie in the 2x2x2 block o + {0,1}^3: along an axis where a and b
// are adjacent o takes the lower of the two (periodically); along an axis
// where they coincide either block holding the coordinate would do, and bit
// k of owner_bits(lower id) picks the one where the shared cell is the lower
// (0) or upper (1) cell of the block.  With local cell codes dA, dB in 0..7
// (bit k = offset along axis k, A the lower id) the block owns the pair iff
// dA and dB agree with the owner bits wherever they coincide.  Spreading a
// particle's pairs over the colours this way roughly halves the longest
// chain of pairs in a block compared with always taking the lower block.
// The colour of o is its parity pattern; blocks of one colour are disjoint
// when every cell count is even, so the 8 colours are swept one after the
// other and the blocks of a colour in parallel.
//
// Order inside a block.  Pairs go by (rank(j) - rank(i), rank(i)), rank = the
// position of the id among the block's particles, i the lower id.  Any
// schedule that keeps, for every particle, its pairs in that order gives the
// same result as the sequential sweep; the schedule used here runs the pairs
// in rounds of at most `width` pairs of disjoint particles, each pair in the
// first round that has room after the rounds of its particles' earlier pairs.
//
// Five launches prepare the schedule of every block (it depends on the
// positions only, which are fixed during the sweep): k_sched_enum (one
// thread block per block: owned pairs in canonical order, from the
// neighbour lists of the density pass), k_sched_rounds (one warp per block:
// the round of every pair, and the pairs written round by round),
// k_sched_large (both for the blocks that are too large for those two, and
// the depth histogram scanned), k_sched_order_scatter (each colour's blocks
// ordered by their number of rounds) and k_stage_geometry (the pairs' unit
// vectors and friction factors).  A sweep is then k_stage_random (the pairs'
// random numbers) and one colour launch per colour (sdpd_fd_colour.cuh,
// sdpd_fd_team64.cuh): the pair updates round by round in shared memory.
// (Large systems: geometry, random numbers and colour launch slice by slice.)
#include <algorithm>
#include <type_traits>

#include "sdpd_fd_common.cuh"

namespace sdpd {


// ---------------------------------------------------------------------------
// Schedule, step 1: owned pairs of every block in canonical order, read from
// the neighbour lists of the density pass.  One thread block of
// kEnumThreads threads per owner cell.
// Owned pairs.  The pairs of this block whose lower id is particle A (block
// cell dA) are A's neighbours in the cells that this block holds and that
// the owner rule gives to this block when A is the lower id: per axis k the
// offset +1 (A's cell is the block's lower one: dA_k = 0) or -1 (its upper
// one), and the offset 0 where bit k of A's owner bits equals dA_k.  These
// cells are 1, 2 or 4 rows of A's 27-cell walk, each a run of consecutive
// cells, so their entries are at most four slot ranges of A's list (the
// density pass records where each row's cells start and end).  Of these
// entries, those whose partner ranks above A are A's owned pairs; the others
// are found from the partner's side.  The predicate is the density pass's
// r^2 < h^2, so the sweep's pair set is the one of the density sum.  A block
// with a member whose list overflowed its row is swept pair by pair
// (kHdrBig).
// Ranks.  Every cell holds its particles by ascending id; the 8 sorted cells
// are merged in three rounds of pairwise merges (the place of an id in the
// merged run = its place in its own run + the ids below it in the sibling
// run, by binary search), which gives each particle's rank among the block's
// ids and the particle of each rank.
// Entries.  The members' entry counts are scanned into offsets of one flat
// range, and the threads take its entries in turn, so that the global loads
// are spread evenly and issued together (in chunks of kFlatEntries, the
// size of the table of each entry's member).
// Found pairs set bit rank(i) of row d = rank(j) - rank(i) of a triangular
// bitmap (row d holds nb - d bits in whole words: it starts at word
// F(nb - 1) - F(nb - d) with F(n) = sum_{k <= n} ceil(k / 32)), which is then
// read out row by row.
// ---------------------------------------------------------------------------
constexpr int kEnumThreads = 160;   // blocks of up to kMaxBlock particles
constexpr int kLargeThreads = 256;  // blocks of up to kLargeBlock particles (two per thread)
constexpr int kFlatEntries = 2048;  // group entries of one block per chunk

// words of the first rows of the triangular bitmap: F(n) = sum_{k=1..n} ceil(k/32)
__host__ __device__ constexpr int tri_f(int n) {
  return 16 * (n >> 5) * ((n >> 5) + 1) + (n & 31) * ((n >> 5) + 1);
}

// What an enumeration keeps in shared memory: ranks, bitmap and the block's
// cells; with the lists' group entries (EnumSmem) or the members' positions
// (LargeEnumSmem).
template <int CAP>
struct EnumBase {
  using Idx = typename std::conditional<CAP <= 256, uint8_t, uint16_t>::type;  // block-local index
  uint32_t bits[tri_f(CAP - 1) + 8];
  int32_t ids[2][CAP];    // merge rounds: the ids in run order
  Idx ks[2][CAP];         // and the block-local index of each
  Idx rank[CAP];          // rank of each block-local index
  Idx perm[CAP];          // block-local index of each rank
  uint8_t dk[CAP];        // block cell of each member
  uint16_t rowbase[CAP];  // first word of each row of the bitmap
  int32_t ctot[CAP / 32]; // row-scan chunk totals
  int32_t cstart[8], cbase[9], koff[9];
  int32_t nb, big;
};
struct EnumSmem : EnumBase<kMaxBlock> {
  Idx who[kFlatEntries];       // member of each flat entry
  uint32_t rng[kMaxBlock];     // up to four slot ranges (first slot, length) of each member's group, packed
  uint32_t rcum[kMaxBlock];    // cumulative lengths after ranges 0, 1, 2 (bytes)
  uint8_t ncnt[kMaxBlock];     // entries of each member's group
  int64_t lbase[kMaxBlock];    // nbr_slot(member, 0) with the slot's in-row part removed
  uint8_t dtab[8][64];         // partner cell of (member cell, stencil code); 8: not in the block
  int32_t off[kMaxBlock + 1];  // first flat entry of each member
  int32_t wtot[8];             // per-warp totals of the offset scan
};
template <class P>
struct LargeEnumSmem : EnumBase<kLargeBlock> {
  typename P::R x[kLargeBlock], y[kLargeBlock], z[kLargeBlock];  // block-local position of each rank
  uint8_t own[kLargeBlock];  // block cell | owner bits << 3 of each rank
};

// Outcome of an enumeration that gives no list.
enum : int { kEnumParticles = -1, kEnumPairs = -2, kEnumList = -3 };

// The block's 8 cells (first warp; the thread block synchronises after it).
template <int CAP>
__device__ __forceinline__ void enum_cells(EnumBase<CAP>& sm, const Consts& c, int o,
                                           const int32_t* __restrict__ cell_start,
                                           const int32_t* __restrict__ mrank) {
  const int t = threadIdx.x, lane = t & 31;
  const int ox = o % c.nc[0], oy = (o / c.nc[0]) % c.nc[1], oz = o / (c.nc[0] * c.nc[1]);
  // the block's 8 cells: storage start, count and offset in the block
  if (t < 32) {
    int ccnt = 0, cst = 0;
    if (lane < 8) {
      int cx = ox + (lane & 1), cy = oy + ((lane >> 1) & 1), cz = oz + ((lane >> 2) & 1);
      if (cx >= c.nc[0]) cx -= c.nc[0];
      if (cy >= c.nc[1]) cy -= c.nc[1];
      if (cz >= c.nc[2]) cz -= c.nc[2];
      const int r = __ldg(&mrank[cx + c.nc[0] * (cy + c.nc[1] * cz)]);
      cst = __ldg(&cell_start[r]);
      ccnt = __ldg(&cell_start[r + 1]) - cst;
    }
    int cinc = ccnt;
#pragma unroll
    for (int sh = 1; sh < 8; sh <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, cinc, sh);
      if (lane >= sh) cinc += v;
    }
    if (lane < 8) {
      sm.cstart[lane] = cst;
      sm.cbase[lane] = cinc - ccnt;
      sm.koff[lane] = cinc - ccnt - cst;  // block-local index = storage index + koff
    }
    if (lane == 7) {
      sm.cbase[8] = cinc;
      sm.nb = cinc;
    }
    if (lane == 0) {
      sm.big = 0;
      sm.koff[8] = -(1 << 30);  // a partner outside the block: out of range
    }
  }
}

// One round of the pairwise merges of the sorted cells (level L = 0, 1, 2).
template <int CAP, int THREADS>
__device__ __forceinline__ void enum_merge(EnumBase<CAP>& sm, int nb, int L) {
  const int t = threadIdx.x;
  const int src = L & 1, dst = src ^ 1;
  for (int k = t; k < nb; k += THREADS) {
    const int d = sm.dk[k];
    const int run = d >> L, sib = run ^ 1;
    const int own0 = sm.cbase[run << L], m0 = sm.cbase[(run & ~1) << L];
    int pos = sm.cbase[sib << L], len = sm.cbase[(sib + 1) << L] - pos;
    const int sib0 = pos;
    const int32_t myid = sm.ids[src][k];
    while (len > 0) {
      const int half = len >> 1;
      const bool below = sm.ids[src][pos + half] < myid;
      pos = below ? pos + half + 1 : pos;
      len = below ? len - half - 1 : half;
    }
    const int np = m0 + (k - own0) + (pos - sib0);
    sm.ids[dst][np] = myid;
    sm.ks[dst][np] = sm.ks[src][k];
  }
}

// The bitmap read out row by row (difference ascending), lower rank
// ascending: emit(position, lower-ranked member, other member) per pair.
// Returns the number of pairs, or kEnumPairs above max_pairs.
template <int CAP, int THREADS, class Emit>
__device__ __forceinline__ int enum_rows(EnumBase<CAP>& sm, int nb, int max_pairs, Emit emit) {
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  static_assert(2 * THREADS >= CAP, "two rows per thread");
  // row populations (rows 1 .. nb - 1): each warp scans 32 rows at a time
  // (row 1 + t is thread t's in every phase below), then the chunk totals
  // are added in
  int rowex[2] = {0, 0};
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int r0 = 1 + 32 * wid + it * THREADS;
    if (r0 >= nb) break;
    const int rr = r0 + lane;
    int n = 0;
    if (rr < nb) {
      const int w0 = sm.rowbase[rr], nwr = (nb - rr + 31) >> 5;
      for (int w = 0; w < nwr; ++w) n += __popc(sm.bits[w0 + w]);
    }
    int inc = n;
#pragma unroll
    for (int sh = 1; sh < 32; sh <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, sh);
      if (lane >= sh) inc += v;
    }
    rowex[it] = inc - n;
    if (lane == 31) sm.ctot[(r0 - 1) >> 5] = inc;
  }
  __syncthreads();
  const int nchunk = (nb - 1 + 31) >> 5;
  int npairs = 0;
  for (int ch = 0; ch < nchunk; ++ch) npairs += sm.ctot[ch];
  if (npairs > max_pairs) return kEnumPairs;
  // write the pairs row by row (difference ascending), lower rank ascending
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int rr = 1 + t + it * THREADS;
    if (rr >= nb) break;
    const int chunk = (rr - 1) >> 5;
    int pos = rowex[it];
    for (int ch = 0; ch < chunk; ++ch) pos += sm.ctot[ch];
    const int w0 = sm.rowbase[rr], nwr = (nb - rr + 31) >> 5;
    for (int w = 0; w < nwr; ++w) {
      uint32_t bits = sm.bits[w0 + w];
      while (bits) {
        const int bit = __ffs(bits) - 1;
        bits &= bits - 1;
        const int lo = w * 32 + bit;
        emit(pos++, (int)sm.perm[lo], (int)sm.perm[lo + rr]);
      }
    }
  }
  return npairs;
}

// Owned pairs of block o in canonical order from the neighbour lists, by a
// thread block of kEnumThreads threads.  Returns their number, or
// kEnumParticles (more than kMaxBlock particles), kEnumPairs (more than
// max_pairs pairs), kEnumList (a member's list overflowed).  The same value
// on every thread.
template <class Emit>
__device__ __forceinline__ int enum_block(EnumSmem& sm, const Consts& c, int o, const int32_t* __restrict__ pid,
                                          const int32_t* __restrict__ cell_start, const int32_t* __restrict__ mrank,
                                          const uint32_t* __restrict__ nlist, const int32_t* __restrict__ nn,
                                          const uint32_t* __restrict__ cend, int max_pairs, Emit emit) {
  constexpr int CAP = kMaxBlock, THREADS = kEnumThreads, kWarps = THREADS / 32;
  using Idx = EnumSmem::Idx;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  enum_cells<CAP>(sm, c, o, cell_start, mrank);
  for (int q = t; q < 8 * 64; q += THREADS) {  // partner cell: member cell + (code - 1) per axis
    const int dA = q >> 6, code = q & 63;
    int dB = 0;
    bool in = true;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      const int f = (code >> (2 * ax)) & 3, b = ((dA >> ax) & 1) + f - 1;
      in = in && f < 3 && b >= 0 && b <= 1;
      dB |= (b & 1) << ax;
    }
    sm.dtab[dA][code] = (uint8_t)(in ? dB : 8);
  }
  __syncthreads();
  const int nb = sm.nb;
  if (nb > CAP) return kEnumParticles;
  const int ntri = nb > 1 ? tri_f(nb - 1) : 0;  // words of the bitmap in use
  for (int q = t; q < ntri; q += THREADS) sm.bits[q] = 0u;
  int cb[9];
#pragma unroll
  for (int u = 0; u < 9; ++u) cb[u] = sm.cbase[u];
  const int64_t N = c.N;
  // the members: id, and the slot ranges of the owner group in the list
  for (int k = t; k < nb; k += THREADS) {
    int d = 0;
#pragma unroll
    for (int u = 1; u < 8; ++u) d += (k >= cb[u]);
    const int g = sm.cstart[d] + (k - sm.cbase[d]);
    const int32_t id = __ldg(&pid[g]);
    sm.ids[0][k] = id;
    sm.ks[0][k] = (Idx)k;
    if (__ldg(&nn[g]) > c.nbr_cap) sm.big = 1;  // the list lost entries
    const unsigned ob = owner_bits(id);
    // per axis the cells of the group as indices [lo, hi) of the offsets
    // (-1, 0, +1): dA_k = 0: {0 if ob_k = 0, +1}; dA_k = 1: {-1, 0 if ob_k = 1}
    int lo[3], hi[3];
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      const int dk = (d >> ax) & 1, bk = (int)(ob >> ax) & 1;
      lo[ax] = dk ? 0 : 2 - (bk ^ 1);
      hi[ax] = dk ? 1 + bk : 3;
    }
    // rows (iz, iy) of the group: at most 2 x 2; x range [lo[0], hi[0]) of bytes
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int iz = lo[2] + (q >> 1), iy = lo[1] + (q & 1);
      w[q] = (iz < hi[2] && iy < hi[1]) ? __ldg(&cend[(int64_t)(iz * 3 + iy) * N + g]) : 0u;
    }
    uint32_t rng = 0u, cum = 0u;
    int tot = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int s0 = (int)((w[q] >> (8 * lo[0])) & 255u), s1 = (int)((w[q] >> (8 * hi[0])) & 255u);
      const int len = s1 > s0 ? s1 - s0 : 0;  // empty for rows outside the group (w = 0)
      rng |= (uint32_t)s0 << (8 * q);
      tot += len;
      if (q < 3) cum |= (uint32_t)min(tot, 255) << (8 * q);
    }
    sm.rng[k] = rng;
    sm.rcum[k] = cum;
    sm.off[k] = tot;  // the count; turned into an offset below
    sm.ncnt[k] = (uint8_t)tot;  // at most the row capacity
    sm.dk[k] = (uint8_t)d;
    sm.lbase[k] = ((int64_t)(g >> 5) * (c.nbr_cap >> 2) << 7) + ((g & 31) << 2);
  }
  __syncthreads();
  if (sm.big) return kEnumList;
  // the member of each flat entry of the chunk [E0, E0 + kFlatEntries), in
  // equal stretches per thread: one binary search for the stretch's first
  // entry, then a walk (members without entries are skipped)
  auto fill_who = [&](int E0) {
    const int E = sm.off[nb], Ec = min(E - E0, kFlatEntries), per = (Ec + THREADS - 1) / THREADS;
    const int e0 = E0 + t * per, e1 = min(E0 + Ec, e0 + per);
    if (e0 < e1) {
      int pos = 1, len = nb - 1;  // members 1 .. nb - 1 starting at or before e0
      while (len > 0) {
        const int half = len >> 1;
        const bool le = sm.off[pos + half] <= e0;
        pos = le ? pos + half + 1 : pos;
        len = le ? len - half - 1 : half;
      }
      int k = pos - 1, kend = sm.off[k] + sm.ncnt[k];
      for (int e = e0; e < e1; ++e) {
        while (e >= kend) {
          ++k;
          kend = sm.off[k] + sm.ncnt[k];
        }
        sm.who[e - E0] = (Idx)k;
      }
    }
  };
  // ranks: three rounds of pairwise merges of the sorted cells, interleaved
  // with the exclusive scan of the members' entry counts
  int cnt0 = 0, incl = 0;
#pragma unroll 1
  for (int L = 0; L < 3; ++L) {
    enum_merge<CAP, THREADS>(sm, nb, L);
    if (L == 0) {  // counts of members 2t and 2t + 1: per-warp inclusive scan
      cnt0 = 2 * t < nb ? sm.ncnt[2 * t] : 0;
      const int cnt1 = 2 * t + 1 < nb ? sm.ncnt[2 * t + 1] : 0;
      incl = cnt0 + cnt1;
#pragma unroll
      for (int sh = 1; sh < 32; sh <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, sh);
        if (lane >= sh) incl += v;
      }
      if (lane == 31) sm.wtot[wid] = incl;
    } else if (L == 1) {  // offsets in member order
      int before = 0, total = 0;
#pragma unroll
      for (int q = 0; q < kWarps; ++q) {
        before += q < wid ? sm.wtot[q] : 0;
        total += sm.wtot[q];
      }
      const int ex = before + incl - cnt0 - (2 * t + 1 < nb ? sm.ncnt[2 * t + 1] : 0);
      if (2 * t < nb) sm.off[2 * t] = ex;
      if (2 * t + 1 < nb) sm.off[2 * t + 1] = ex + cnt0;
      if (t == 0) sm.off[nb] = total;
    } else {  // the member of each entry of the first chunk
      fill_who(0);
    }
    __syncthreads();
  }
  for (int r = t; r < nb; r += THREADS) {  // the merged run is ids[1]
    const int k = sm.ks[1][r];
    sm.perm[r] = (Idx)k;
    sm.rank[k] = (Idx)r;
  }
  for (int d = 1 + t; d < nb; d += THREADS)  // row d of the bitmap starts at F(nb - 1) - F(nb - d)
    sm.rowbase[d] = (uint16_t)(tri_f(nb - 1) - tri_f(nb - d));
  __syncthreads();
  // the flat entries: partner, rank test, bit; chunk by chunk (a block with
  // more entries than the table holds takes several)
  const int E = sm.off[nb];
  for (int E0 = 0; E0 < E; E0 += kFlatEntries) {
    if (E0 > 0) {
      fill_who(E0);
      __syncthreads();
    }
    const int E1 = min(E, E0 + kFlatEntries);
#pragma unroll 4
    for (int e = E0 + t; e < E1; e += THREADS) {
      const int A = sm.who[e - E0];
      const int m = e - sm.off[A];
      const uint32_t rng = sm.rng[A], cum = sm.rcum[A];
      const int c0 = cum & 255u, c1 = (cum >> 8) & 255u, c2 = (cum >> 16) & 255u;
      const int q = (m >= c0) + (m >= c1) + (m >= c2);
      const int before = q == 0 ? 0 : (q == 1 ? c0 : (q == 2 ? c1 : c2));
      const int slot = (int)((rng >> (8 * q)) & 255u) + (m - before);
      const int dA = sm.dk[A];
      const uint32_t en = __ldg(&nlist[sm.lbase[A] + ((slot >> 2) << 7) + (slot & 3)]);  // nbr_slot(g, slot)
      const int kB = (int)(en >> 6) + sm.koff[sm.dtab[dA][en & 63u]];
      if ((unsigned)kB < (unsigned)nb) {
        const int rA = sm.rank[A], rB = sm.rank[kB];
        if (rB > rA) atomicOr(&sm.bits[sm.rowbase[rB - rA] + (rA >> 5)], 1u << (rA & 31));
      }
    }
    __syncthreads();
  }
  return enum_rows<CAP, THREADS>(sm, nb, max_pairs, emit);
}

// The same for a large block, from positions: the members in rank order with
// their block-local coordinates, then every pair of ranks by the owner rule
// and the distance (32 pairs of one row per warp, whose ballot is a word of
// the bitmap).  The predicate is the one of the pair-by-pair sweep.
template <class P, class Emit>
__device__ __forceinline__ int enum_large(LargeEnumSmem<P>& sm, const Consts& c, int o,
                                          const int32_t* __restrict__ pid, const int32_t* __restrict__ cell_start,
                                          const int32_t* __restrict__ mrank, const typename P::V4* __restrict__ q4,
                                          const uint32_t* xmx, const uint32_t* xmy, const uint32_t* xmz,
                                          const int32_t* __restrict__ nn, int max_pairs, Emit emit) {
  using R = typename P::R;
  constexpr int CAP = kLargeBlock, THREADS = kLargeThreads;
  using Idx = typename EnumBase<CAP>::Idx;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  enum_cells<CAP>(sm, c, o, cell_start, mrank);
  __syncthreads();
  const int nb = sm.nb;
  if (nb > CAP) return kEnumParticles;
  auto member = [&](int k, int& d) {
    d = 0;
#pragma unroll
    for (int u = 1; u < 8; ++u) d += (k >= sm.cbase[u]);
    return sm.cstart[d] + (k - sm.cbase[d]);
  };
  for (int k = t; k < nb; k += THREADS) {
    int d;
    const int g = member(k, d);
    sm.ids[0][k] = __ldg(&pid[g]);
    sm.ks[0][k] = (Idx)k;
    sm.dk[k] = (uint8_t)d;
    if (__ldg(&nn[g]) > c.nbr_cap) sm.big = 1;  // (left to the pair-by-pair sweep)
  }
  __syncthreads();
  if (sm.big) return kEnumList;
#pragma unroll 1
  for (int L = 0; L < 3; ++L) {
    enum_merge<CAP, THREADS>(sm, nb, L);
    __syncthreads();
  }
  BlockGeom<P> geo;
  geo.init(c, o % c.nc[0], (o / c.nc[0]) % c.nc[1], o / (c.nc[0] * c.nc[1]), xmx, xmy, xmz);
  for (int r = t; r < nb; r += THREADS) {  // the merged run is ids[1]
    const int k = sm.ks[1][r];
    int d;
    const int g = member(k, d);
    sm.perm[r] = (Idx)k;
    R x, y, z;
    geo.local(ld4(&q4[g]), d, x, y, z);
    sm.x[r] = x;
    sm.y[r] = y;
    sm.z[r] = z;
    sm.own[r] = (uint8_t)(d | (int)owner_bits(sm.ids[1][r]) << 3);
  }
  for (int d = 1 + t; d < nb; d += THREADS) sm.rowbase[d] = (uint16_t)(tri_f(nb - 1) - tri_f(nb - d));
  __syncthreads();
  const R h2 = (R)c.h2;
  for (int d = 1 + wid; d < nb; d += THREADS / 32)
    for (int r0 = 0; r0 < nb - d; r0 += 32) {
      const int r = r0 + lane;
      bool hit = false;
      if (r < nb - d) {
        const int a = sm.own[r], dA = a & 7, dB = sm.own[r + d] & 7;
        if ((((dA ^ (a >> 3)) & ~(dA ^ dB)) & 7) == 0) {  // on shared axes the cell bit equals the owner bit
          R dx, dy, dz;
          geo.disp(sm.x[r], sm.y[r], sm.z[r], sm.x[r + d], sm.y[r + d], sm.z[r + d], dx, dy, dz);
          hit = r2_of(dx, dy, dz) < h2;
        }
      }
      const unsigned m = __ballot_sync(0xffffffffu, hit);
      if (lane == 0) sm.bits[sm.rowbase[d] + (r0 >> 5)] = m;
    }
  __syncthreads();
  return enum_rows<CAP, THREADS>(sm, nb, max_pairs, emit);
}

// The schedule's first launch: one thread block per block of cells (12 per SM:
// 32 registers; 1520 us instead of 1313 at 2M particles with 38).
__global__ void __launch_bounds__(kEnumThreads, 12)
    k_sched_enum(const __grid_constant__ Consts c, const int32_t* __restrict__ pid,
                 const int32_t* __restrict__ cell_start, const int32_t* __restrict__ mrank,
                 const uint32_t* __restrict__ nlist, const int32_t* __restrict__ nn,
                 const uint32_t* __restrict__ cend, uint32_t* __restrict__ hdr, uint16_t* __restrict__ canon,
                 uint32_t* __restrict__ blk_hist, uint32_t* __restrict__ big_count, uint32_t* __restrict__ large_count,
                 int32_t* __restrict__ large_cand, unsigned long long* __restrict__ sched_total) {
  __shared__ EnumSmem sm;
  const int t = threadIdx.x, o = blockIdx.x;  // owner cell (fewer than 2^31 cells)
  if (o == 0) {  // what the next launches count in: depth histogram, lists, dense pair arrays
    if (t == 0) *sched_total = 0ull;
    for (int k = t; k < 8 * 256; k += kEnumThreads) blk_hist[k] = 0u;
    if (t < 16) big_count[t] = 0u;
    if (t < 8) large_count[t] = 0u;
  }
  uint16_t* out = canon + (int64_t)o * kMaxPairs;
  const int np = enum_block(
      sm, c, o, pid, cell_start, mrank, nlist, nn, cend, kMaxPairs,
      [&](int pos, int lo, int hi) { out[pos] = (uint16_t)(lo | (hi << 8)); });
  if (t != 0) return;
  hdr[o] = np >= 0 ? (uint32_t)np : (np == kEnumList ? kHdrBig : kHdrLarge);
  if (np == kEnumParticles || np == kEnumPairs) large_cand[atomicAdd(&large_count[8], 1u)] = o;
}

// Rounds: one warp per block takes the block's canonical list 32 pairs at a
// time.  A pair may go after all earlier pairs of its two particles.  The
// lanes of a chunk set their bit in a mask per particle (shared memory), which
// gives each lane the earlier lanes that share a particle with it; a lane
// whose earlier lanes are done takes the first round >= the ones its
// particles are free from that still has room, by an atomic count.  A chunk
// takes as many passes as its longest chain of pairs sharing particles (four
// to five on the lattice).
// Round width: the lanes that a colour launch gives a block.  Limiting the
// rounds here instead of splitting wide dependency levels there fills the
// lanes better (16 lanes, 32^3 lattice: 53 rounds per block instead of 68).
// One thread per block walking the list sequentially, with the bucketing by
// level in a second launch, took 109 + 14 us at 32^3 (800 pairs in a chain
// of ~190 cycles each).
constexpr int kRoundWarps = 4;

template <int CAP, int MAXP>
struct RoundSmem {
  uint32_t claim[CAP];   // lanes of the current chunk that hold a particle
  uint32_t cnt[kRoundStride];
  uint8_t place[MAXP];   // round of each pair (the order inside a round is free)
  uint8_t last[CAP];     // first round in which a particle is free
};

// The dense arrays and lists a schedule is written to.
struct SchedOut {
  int64_t ncell;
  int nc[3];
  unsigned long long cap;  // entries of the dense pair arrays
  uint32_t* hdr;
  uint8_t* rsize;
  unsigned long long* off;
  unsigned long long* total;
  uint32_t* pairs;
  uint32_t* blk_hist;
  const int32_t* cell_start;
  const int32_t* mrank;
  uint32_t* big_count;
  int2* big_list;
};

// the block's colour is the parity pattern of its owner cell
__device__ __forceinline__ int block_colour(const int nc[3], int64_t o, int& ox, int& oy, int& oz) {
  ox = (int)(o % nc[0]);
  oy = (int)((o / nc[0]) % nc[1]);
  oz = (int)(o / ((int64_t)nc[0] * nc[1]));
  return (ox & 1) | ((oy & 1) << 1) | ((oz & 1) << 2);
}

// One thread: block o goes pair by pair after its colour's other blocks,
// listed with the place of its particles in big_perm (blocks of a colour are
// disjoint).
__device__ __noinline__ void list_big(const SchedOut& out, int64_t o) {
  int ox, oy, oz;
  const int colour = block_colour(out.nc, o, ox, oy, oz);
  out.hdr[o] = kHdrBig;
  int nb = 0;
  for (int d = 0; d < 8; ++d) {
    int cx = ox + (d & 1), cy = oy + ((d >> 1) & 1), cz = oz + ((d >> 2) & 1);
    if (cx >= out.nc[0]) cx -= out.nc[0];
    if (cy >= out.nc[1]) cy -= out.nc[1];
    if (cz >= out.nc[2]) cz -= out.nc[2];
    const int r = out.mrank[cx + out.nc[0] * (cy + out.nc[1] * cz)];
    nb += out.cell_start[r + 1] - out.cell_start[r];
  }
  const uint32_t first = atomicAdd(&out.big_count[8 + colour], (uint32_t)nb);
  const uint32_t slot = atomicAdd(&out.big_count[colour], 1u);
  out.big_list[colour * (out.ncell >> 3) + slot] = make_int2((int)o, (int)first);
  atomicAdd(&out.blk_hist[colour * 256 + kMaxLevels], 1u);
}

// The rounds of block o's canonical list (np pairs, in(k) = lower | other <<
// 16 for pair k) by one warp, written to the dense arrays; flag is or-ed into
// the header.  False: more rounds than kMaxLevels, or the dense arrays are
// full (their capacity covers every schedule of symmetric lists).
template <int CAP, int MAXP, class In>
__device__ __forceinline__ bool assign_rounds(RoundSmem<CAP, MAXP>& sm, const SchedOut& out, int64_t o, int np,
                                              int width, uint32_t flag, In in) {
  const int lane = threadIdx.x & 31;
  for (int k = lane; k < CAP; k += 32) sm.claim[k] = 0u;
  for (int k = lane; k < kRoundStride; k += 32) sm.cnt[k] = 0u;
  for (int k = lane; k < CAP / 4; k += 32) reinterpret_cast<uint32_t*>(sm.last)[k] = 0u;
  __syncwarp();
  int full = 0;  // rounds below are full
  bool overflow = false;
  uint32_t nxt = lane < np ? in(lane) : 0u;
  for (int k0 = 0; k0 < np; k0 += 32) {
    const uint32_t pr = nxt;
    if (k0 + 32 + lane < np) nxt = in(k0 + 32 + lane);
    const int u = pr & 0xffffu, v = pr >> 16;
    const bool valid = k0 + lane < np;
    if (valid) {
      atomicOr(&sm.claim[u], 1u << lane);
      atomicOr(&sm.claim[v], 1u << lane);
    }
    __syncwarp();
    const unsigned before = valid ? (sm.claim[u] | sm.claim[v]) & ((1u << lane) - 1u) : 0u;
    unsigned pending = __ballot_sync(0xffffffffu, valid);
    __syncwarp();
    if (valid) sm.claim[u] = sm.claim[v] = 0u;
    while (pending) {
      const bool ready = (pending >> lane & 1u) && !(before & pending);
      if (ready) {
        int L = max(full, max((int)sm.last[u], (int)sm.last[v]));
        while (L < kMaxLevels && atomicAdd(&sm.cnt[L], 1u) >= (uint32_t)width) ++L;
        if (L >= kMaxLevels) {
          overflow = true;
        } else {
          sm.last[u] = sm.last[v] = (uint8_t)(L + 1);
          sm.place[k0 + lane] = (uint8_t)L;
        }
      }
      pending &= ~__ballot_sync(0xffffffffu, ready);
      __syncwarp();
    }
    if (__any_sync(0xffffffffu, overflow)) return false;
    while (full < kMaxLevels && sm.cnt[full] >= (uint32_t)width) ++full;
  }
  unsigned long long at = 0ull;
  if (lane == 0) at = atomicAdd(out.total, (unsigned long long)((np + 7) & ~7));
  at = __shfl_sync(0xffffffffu, at, 0);
  if (at + (unsigned long long)np > out.cap) return false;
  // round sizes and their first positions: 8 consecutive rounds per lane
  // (rounds are contiguous: a pair enters round L > 0 only after a pair in
  // round L - 1 or because that round is full)
  int v[8], sum = 0, nr = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int L = lane * 8 + q;
    v[q] = L < kMaxLevels ? min((int)sm.cnt[L], width) : 0;
    sum += v[q];
    nr += v[q] > 0;
  }
  int incl = sum;
#pragma unroll
  for (int sh = 1; sh < 32; sh <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, incl, sh);
    if (lane >= sh) incl += x;
  }
  nr = __reduce_add_sync(0xffffffffu, nr);
  if (lane == 0) {
    int ox, oy, oz;
    out.off[o] = at;
    out.hdr[o] = (uint32_t)np | ((uint32_t)nr << 16) | flag;
    atomicAdd(&out.blk_hist[block_colour(out.nc, o, ox, oy, oz) * 256 + nr], 1u);
  }
  int run = incl - sum;
  uint32_t packed[2] = {0u, 0u};
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    packed[q >> 2] |= (uint32_t)v[q] << (8 * (q & 3));
    sm.cnt[lane * 8 + q] = (uint32_t)run;
    run += v[q];
  }
  if (lane * 8 < nr) reinterpret_cast<uint2*>(out.rsize + o * kRoundStride)[lane] = make_uint2(packed[0], packed[1]);
  __syncwarp();
#pragma unroll 4
  for (int k = lane; k < np; k += 32) out.pairs[at + atomicAdd(&sm.cnt[sm.place[k]], 1u)] = in(k);
  return true;
}

__global__ void __launch_bounds__(kRoundWarps * 32)
    k_sched_rounds(const __grid_constant__ SchedOut out, int width, const uint16_t* __restrict__ canon) {
  __shared__ RoundSmem<kMaxBlock, kMaxPairs> sm_all[kRoundWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t o = (int64_t)blockIdx.x * kRoundWarps + warp;
  if (o >= out.ncell) return;
  const uint32_t hd = out.hdr[o];
  if (hd == kHdrLarge) return;  // k_sched_large
  const uint16_t* in = canon + o * kMaxPairs;
  const bool ok = hd != kHdrBig &&
                  assign_rounds(sm_all[warp], out, o, (int)hd, width, 0u, [&](int k) {
                    const uint32_t pr = __ldg(&in[k]);
                    return (pr & 255u) | (pr >> 8) << 16;
                  });
  if (!ok && lane == 0) list_big(out, o);
}

// ---------------------------------------------------------------------------
// Large blocks: more particles or owned pairs than k_sched_enum holds, as in
// boxes whose side lies between two cell counts (14 / 2.5: cells of 3.5,
// blocks of 343).  One thread block takes them in turn, pairs (enum_large) and
// rounds with the list in shared memory.  (Swept pair by pair on one lane they took 40 ms
// per sweep of 14^3 particles.)  width: as k_sched_rounds.  The last thread
// block then turns the depth histogram into each depth's first position,
// deepest first (one warp per colour; see below).
// ---------------------------------------------------------------------------
template <class P>
struct LargeSmem {
  LargeEnumSmem<P> e;
  RoundSmem<kLargeBlock, kLargePairs> r;
  uint32_t canon[kLargePairs];
  int np;
  uint32_t last;
};

template <class P>
__global__ void __launch_bounds__(kLargeThreads)
    k_sched_large(const __grid_constant__ Consts c, const __grid_constant__ SchedOut out, int width,
                  const int32_t* __restrict__ pid, const typename P::V4* __restrict__ q4, const uint32_t* xmx,
                  const uint32_t* xmy, const uint32_t* xmz, const int32_t* __restrict__ nn,
                  const int32_t* __restrict__ cand,
                  uint32_t* __restrict__ large_count, int32_t* __restrict__ large_list) {
  extern __shared__ __align__(16) unsigned char large_smem_raw[];
  LargeSmem<P>& sm = *reinterpret_cast<LargeSmem<P>*>(large_smem_raw);
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int n = (int)large_count[8];
  for (int q = blockIdx.x; q < n; q += gridDim.x) {
    const int o = cand[q];
    const int np = enum_large<P>(
        sm.e, c, o, pid, out.cell_start, out.mrank, q4, xmx, xmy, xmz, nn, kLargePairs,
        [&](int pos, int lo, int hi) { sm.canon[pos] = (uint32_t)lo | (uint32_t)hi << 16; });
    __syncthreads();
    if (wid == 0) {
      const bool ok = np >= 0 && assign_rounds(sm.r, out, o, np, width, kHdrLargeFlag, [&](int k) { return sm.canon[k]; });
      if (lane == 0) {
        int ox, oy, oz;
        const int colour = block_colour(out.nc, o, ox, oy, oz);
        if (ok) large_list[colour * (out.ncell >> 3) + atomicAdd(&large_count[colour], 1u)] = o;
        else list_big(out, o);
      }
    }
    __syncthreads();
  }
  if (t == 0) {
    __threadfence();
    sm.last = atomicAdd(&large_count[9], 1u) == gridDim.x - 1u;
  }
  __syncthreads();
  if (!sm.last) return;
  __threadfence();
  // place k of warp `wid`'s colour is depth 255 - k, eight places per lane
  uint32_t* h = out.blk_hist + wid * 256;
  uint32_t v[8], sum = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    v[q] = __ldcg(&h[255 - (lane * 8 + q)]);
    sum += v[q];
  }
  uint32_t incl = sum;
#pragma unroll
  for (int sh = 1; sh < 32; sh <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, incl, sh);
    if (lane >= sh) incl += x;
  }
  uint32_t run = incl - sum;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    h[255 - (lane * 8 + q)] = run;
    run += v[q];
  }
}

// ---------------------------------------------------------------------------
// The order in which a colour launch hands out its blocks: deepest first.
// Each warp of a colour launch runs its blocks in lockstep and pays for the
// deepest, so neighbours in this order have similar depth, and the deep
// blocks start first, which keeps the launch's tail short.  Blocks of a colour
// are independent, so the order changes no result.
// One thread per owner cell: each block's place in its colour's order, by
// depth (from the positions that k_sched_large left in the histogram); the
// order among blocks of equal depth is free.
__global__ void k_sched_order_scatter(int64_t ncell, int nc0, int nc1, const uint32_t* __restrict__ hdr,
                                      uint32_t* __restrict__ blk_hist, int32_t* __restrict__ blk_order,
                                      uint32_t* __restrict__ blk_pos, unsigned long long* __restrict__ st_off,
                                      uint32_t* __restrict__ large_count) {
  if (blockIdx.x == 0 && threadIdx.x < 2) large_count[8 + threadIdx.x] = 0u;  // for the next schedule
  const int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (o >= ncell) return;
  const int ox = (int)(o % nc0), oy = (int)((o / nc0) % nc1), oz = (int)(o / ((int64_t)nc0 * nc1));
  const int colour = (ox & 1) | ((oy & 1) << 1) | ((oz & 1) << 2);
  const int hx = nc0 >> 1, hy = nc1 >> 1;
  const int32_t w = (ox >> 1) + hx * ((oy >> 1) + hy * (oz >> 1));  // index among the colour's blocks
  const uint32_t hd = hdr[o];
  const int nlev = hd == kHdrBig ? kMaxLevels : (int)(hd >> 16 & 255u);
  const uint32_t pos = atomicAdd(&blk_hist[colour * 256 + nlev], 1u);
  blk_order[colour * (ncell >> 3) + pos] = w;
  if (blk_pos) {  // the pair data staged by slice
    blk_pos[o] = pos;
    st_off[o] = (unsigned long long)(pos % kSliceBlocks) * kLargePairs;
  }
}

template <class P>
void launch_fd_schedule(const Consts& c, const Workspace& w, int cur, int width, int large_width, cudaStream_t s) {
  if (c.N == 0) return;
  Arrays<P> a = view<P>(w, cur);
  SchedOut out;
  out.ncell = c.ncell;
  for (int d = 0; d < 3; ++d) out.nc[d] = c.nc[d];
  out.cap = (unsigned long long)sched_pair_capacity(c.N, c.nbr_cap, c.ncell);
  out.hdr = w.sched_hdr;
  out.rsize = w.sched_rsize;
  out.off = w.sched_off;
  out.total = w.sched_total;
  out.pairs = w.sched_pair;
  out.blk_hist = w.blk_hist;
  out.cell_start = w.cell_start;
  out.mrank = w.mrank;
  out.big_count = w.big_count;
  out.big_list = w.big_list;
  k_sched_enum<<<(unsigned)c.ncell, kEnumThreads, 0, s>>>(c, a.id, w.cell_start, w.mrank, w.nlist, w.nn, w.cend,
                                                          w.sched_hdr, w.sched_canon, w.blk_hist, w.big_count, w.large_count,
                                                          w.large_cand, w.sched_total);
  k_sched_rounds<<<(unsigned)((c.ncell + kRoundWarps - 1) / kRoundWarps), kRoundWarps * 32, 0, s>>>(out, width,
                                                                                                   w.sched_canon);
  // (a large block has a whole warp of the colour launch, or its team)
  k_sched_large<P><<<(unsigned)std::min(c.ncell, 152), kLargeThreads, sizeof(LargeSmem<P>), s>>>(
      c, out, std::max(width, large_width), a.id, a.q4, w.xmin[0], w.xmin[1], w.xmin[2], w.nn, w.large_cand,
      w.large_count, w.large_list);
  k_sched_order_scatter<<<(unsigned)((c.ncell + 255) / 256), 256, 0, s>>>(c.ncell, c.nc[0], c.nc[1], w.sched_hdr,
                                                                         w.blk_hist, w.blk_order, w.blk_pos,
                                                                         w.st_off, w.large_count);
}

// Launch attributes of the schedule's kernels (once per device and process;
// kept out of stream captures).
int sched_prepare() {
  const cudaError_t a = cudaFuncSetAttribute(k_sched_large<Fp64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(LargeSmem<Fp64>)),
                    b = cudaFuncSetAttribute(k_sched_large<Mixed>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)sizeof(LargeSmem<Mixed>));
  return a == cudaSuccess && b == cudaSuccess ? SDPD_OK : SDPD_ERR_CUDA;
}

__global__ void k_sweep_set(unsigned long long* sweep, unsigned long long v) { *sweep = v; }
__global__ void k_sweep_advance(unsigned long long* sweep) { *sweep += 1ull; }

void launch_set_sweep(const Workspace& w, unsigned long long value, cudaStream_t s) {
  k_sweep_set<<<1, 1, 0, s>>>(w.sweep, value);
}
void launch_advance_sweep(const Workspace& w, cudaStream_t s) { k_sweep_advance<<<1, 1, 0, s>>>(w.sweep); }

template void launch_fd_schedule<Fp64>(const Consts&, const Workspace&, int, int, int, cudaStream_t);
template void launch_fd_schedule<Mixed>(const Consts&, const Workspace&, int, int, int, cudaStream_t);

}  // namespace sdpd
