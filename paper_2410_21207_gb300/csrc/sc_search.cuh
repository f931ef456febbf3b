// The minimum-vertical-seam search (arXiv 2410.21207, section "DP Seam Carving": Algorithm 3 and
// the recurrence M(i,j) = e(i,j) + min(M(i-1,j-1), M(i-1,j), M(i-1,j+1)); the paper's "GPU" variant
// parallelises the j loop, this code does that and more) as a device function that one CTA, or
// every CTA of a thread-block cluster, calls together.
//
// Layout of the work
//   * Columns are split over the CTAs (CTA r owns [r*OWC, (r+1)*OWC)) and, inside a CTA, over
//     NW compute warps; a lane holds V = 4 consecutive columns of the current cost row in registers
//     and reads its neighbours' edge values with warp shuffles.
//   * Row-blocked trapezoidal tiles: a warp computes a window of 32*V columns (its strip of
//     Q = 32*V - 2*KT columns plus KT halo columns per side) for KT rows without talking to other
//     warps (the valid part shrinks by one column per row), then the strips' last rows are
//     exchanged through shared memory. One level up (clusters only), each CTA computes K2 halo
//     columns on either side of its own range and every K2 rows pushes its edge columns into the
//     neighbours' shared memory with st.async; there is no cluster-wide barrier in the row loop.
//   * A cost travels with an ancestor: key = (M << 8) | a, with a the column (in the warp's frame)
//     where the cell's optimal path crossed the top of the current super-tile of KSS rows (32; 64
//     for the single-map search of wide maps, whose chain hops cross CTAs through DSMEM). The
//     unsigned minimum of three keys is the minimum M and, among equal M, the smallest ancestor.
//     Optimal predecessors never cross under the leftmost tie-break (pred(j) <= pred(j+1): if
//     pred(j) = j+1 then M(j+1) < M(j), so j+1 cannot pick j), hence ancestors are non-decreasing
//     in the column and the smallest ancestor among tied candidates is the leftmost candidate's:
//     the key minimum carries exactly Algorithm 3's choice. The bottom row of each super-tile
//     records its ancestors; a chain of ceil(H/KSS) lookups gives the seam column at every
//     super-tile boundary, and then the super-tiles are backtracked in parallel, each by a search
//     between its two boundary columns in a 2*KSS-column window (KSS/16 columns per lane) with
//     explicit directions.
//   * Energies are staged in shared memory by TMA: a producer warp issues a tile's copies (tensor copies
//     of a few boxes, or in the multi-map and CL_WIDE kernels one bulk copy per row, a row per lane) into
//     an NSLOT-slot ring, waits for the next tile to land and joins the CTA barrier that ends the current
//     one, which also frees its slot; a lane reads its 4 energies of a row with one 8-byte shared-memory
//     load.
//   * The rows of a tile are branch-free (the map has an added row of cost 0 above row 0), and
//     per-super-tile bookkeeping runs after the tile, on its last row (the only row of a tile where
//     it can occur, since KSS is a multiple of KT).
// The result is Algorithm 3's seam exactly (leftmost ties, leftmost last-row minimum).
// With DIRECT the map is the caller's own H x W array (any row pitch that is a multiple of 8
// elements, 16-byte aligned rows), read in place: row copies are clipped to its columns (tensor copies
// read 0 beyond them), the backtrack's loads outside it are skipped, and the 24-bit cost range is checked
// here instead of by a copy kernel (a per-row maximum of the staged energies, reduced over the cluster; a
// map that fails it is left to the wide-cost search through its gate).
// With FWD (forward energy) the map has three planes, CU, DL and DR, and a cell's cost depends on
// the direction it is reached from: M(i,j) = CU(i,j) + min(M(i-1,j-1) + DL(i,j), M(i-1,j),
// M(i-1,j+1) + DR(i,j)). Optimal predecessors still never cross (a crossing pair would need
// DL + DR < 0), so the ancestor keys keep their meaning; the planes are staged side by side. Swept
// upwards, a step costs the DL or DR of the row it leaves (dp_row_fwd_rev).
#pragma once
#include <cooperative_groups.h>
#include <type_traits>

#include "sc_internal.cuh"
#include "sc_ptx.cuh"

namespace sc {

namespace cg = cooperative_groups;

constexpr uint32_t SENT = 0xFFFFFFFFu;   // excluded (outside the image): above every key
constexpr int FILL_WARPS_MAX = 8;        // warps that run backtrack fills
constexpr int NSLOT = 3;                 // energy staging ring: tiles in flight
constexpr size_t SEARCH_SMEM_LIMIT = 232448;   // opt-in dynamic shared memory per CTA

template <int NW, int KT, bool CL, int FWM = FILL_WARPS_MAX, int KSS = KS>
struct Geo {
  static constexpr int Q = 32 * V - 2 * KT;              // warp strip
  static constexpr int K2E = CL ? K2 : 0;                // CTA-level halo (clusters only)
  static constexpr int BW = NW * Q + 2 * KT;             // boundary / staged row width
  static constexpr int OWC = NW * Q - 2 * K2E;           // CTA-own columns
  static constexpr int FW = (NW + 1) < FWM ? (NW + 1) : FWM;   // backtrack-fill warps
  static constexpr int THREADS = (NW + 1) * 32;          // compute warps + the producer warp
  static constexpr int FV = KSS / 16;                    // backtrack-fill columns per lane
  static constexpr int FILLW = 32 * FV;                  // backtrack-fill window (2 * KSS columns)
  // rows whose energies a fill warp holds in shared memory at a time: the whole super-tile in the
  // single-map search of e1 maps up to 32 rows, else half of it or a quarter
  static constexpr int fill_rows(bool fwd) { return FWM >= FILL_WARPS_MAX && !fwd && CL ? 32 : 16; }
  static constexpr size_t fill_bytes(bool fwd) {         // per fill warp: directions, energies
    return (size_t)KSS * FILLW + (size_t)fill_rows(fwd) * FILLW * 2 * (fwd ? 3 : 1);
  }
  static_assert(Q > 0 && KSS % KT == 0 && K2 % KT == 0, "tile geometry");
  static_assert(KSS == 32 || KSS == 64, "super-tile height");
  static_assert(Q + 2 * KSS <= 256, "the ancestor frame must fit 8 bits");
};

// offsets of the dynamic shared-memory regions used by seam_search
struct SearchPlan {
  size_t bnd, hbuf, anc, wmin, cmin, jb, misc, emx, fill, ring, ring_end, bars, gat, total;
  int gw;   // row stride (bytes) of the gathered ancestor table in rank 0; 0: not gathered
};

template <int NW, int KT, bool CL, int FWM = FILL_WARPS_MAX, bool FWD = false, int KSS = KS, bool DIRECT = false,
          bool TM = false>
__host__ __device__ inline SearchPlan search_plan(int S) {
  using G = Geo<NW, KT, CL, FWM, KSS>;
  SearchPlan p;
  size_t o = 0;
  p.bnd = o;  o += (size_t)2 * G::BW * 4;  o = (o + 15) & ~(size_t)15;
  p.hbuf = o; o += CL ? (size_t)2 * 2 * K2 * 4 : 0;
  p.anc = o;  o += (size_t)S * G::OWC;  o = (o + 15) & ~(size_t)15;
  p.wmin = o; o += (size_t)(NW + 1) * 8;
  p.cmin = o; o += CL ? (size_t)MAX_CLUSTER * 8 : 8;   // every CTA's minimum, pushed to rank 0
  p.jb = o;   o += (size_t)(S + 1) * 4;  o = (o + 15) & ~(size_t)15;
  p.misc = o; o += 16;
  p.emx = o;  o += DIRECT ? (size_t)(NW + 1 + MAX_CLUSTER) * 4 : 0;   // energy maxima: per warp, per CTA
  o = (o + 15) & ~(size_t)15;
  // the backtrack fill works in the staging ring's place, which is idle by then (every staged tile
  // has been consumed before the argmin)
  const size_t fill_sz = (size_t)G::FW * G::fill_bytes(FWD), 
               ring_sz = (size_t)NSLOT * (FWD ? 3 : 1) * KT * (TM ? tensor_boxes(G::BW) * tensor_box_cols(G::BW) : G::BW) * 2;
  o = (o + 127) & ~(size_t)127;   // (tensor copies: 128-byte aligned)
  p.ring = p.fill = o; o += fill_sz > ring_sz ? fill_sz : ring_sz;  o = (o + 15) & ~(size_t)15;
  p.ring_end = o;
  p.bars = o; o += (size_t)(NSLOT + 2) * 8;   // full[NSLOT], halo[2]
  o = (o + 15) & ~(size_t)15;
  // single-map cluster search: every CTA writes its super-tile ancestors straight into rank 0's
  // table (remote stores during the row loop), so the chain after the argmin is all local loads;
  // only where the table fits
  p.gat = o;
  p.gw = 0;
  const size_t gat_sz = (size_t)S * MAX_CLUSTER * G::OWC;
  if (CL && FWM >= FILL_WARPS_MAX && o + gat_sz <= SEARCH_SMEM_LIMIT) {
    p.gw = MAX_CLUSTER * G::OWC;
    o += gat_sz;
  }
  p.total = (o + 15) & ~(size_t)15;
  return p;
}

struct SearchArgs {
  const uint16_t *E;   // row 0, column 0 (already offset by E_PADL unless DIRECT)
  int pitch_e;
  int H, W;
  int *gate = nullptr; // DIRECT: receives ERR_ENERGY_RANGE when the map fails the 24-bit range check
  int32_t *seam;       // out [H]
  int32_t *seam_log;   // nullable, out [H]
  int64_t *cost;       // nullable, out [1]
  int *err;            // device error word
  bool gated;          // skip the search (energy range failure)
  int64_t pstride;     // forward energy: elements from one cost plane (CU, DL, DR) to the next
  // half of a two-ended search: the ancestor table (row stride gw) and the last row's costs, in
  // global memory (pitch_e is negative where the rows are swept from the bottom of the map)
  uint8_t *gtab = nullptr;
  int gw = 0;
  uint32_t *endrow = nullptr;
  uint32_t *gmax = nullptr;     // DIRECT: the maximum of the map's energies, over both halves
  const void *tmap = nullptr;   // tensor map of the energy buffer (rows of pitch_e elements)
  int x0 = E_PADL;              // its column of the map's column 0
  int y0 = 0, plane_rows = 0;   // its row of this half's row 0; rows from one cost plane to the next
  int rank0 = 0, ctas = 0;      // the cluster's CTAs that sweep this half: ctas from rank0 on (0: all of them)
};

// Running counters of the mbarrier phases, identical in every thread of the CTA.
struct SearchState {
  uint32_t tiles = 0;  // tiles staged so far (ring slot and phase)
  uint32_t exch = 0;   // inter-CTA exchanges so far (halo buffer and phase)
  uint32_t joins = 0;  // two-ended searches of one cluster: table copies so far (rank 0)
};

__device__ __forceinline__ uint32_t min3u(uint32_t a, uint32_t b, uint32_t c) { return __vimin3_u32(a, b, c); }

// (uint16 pair) -> value << 8 for the low / high half
__device__ __forceinline__ uint32_t lo8(uint32_t x) { return __byte_perm(x, 0u, 0x4104); }
__device__ __forceinline__ uint32_t hi8(uint32_t x) { return __byte_perm(x, 0u, 0x4324); }

// The ancestors of this lane's V columns (one byte each: a - column + 128) from its keys; c0: the
// lane's first column, fb: the warp's frame base.
__device__ __forceinline__ uint32_t pack_ancestors(const uint32_t (&k)[V], int c0, int fb) {
  const uint32_t d = (uint32_t)(fb - c0 + 128);
  return ((k[0] + d) & 0xFFu) | (((k[1] + d - 1u) & 0xFFu) << 8) | (((k[2] + d - 2u) & 0xFFu) << 16) |
         ((k[3] + d - 3u) << 24);
}

// key + energy, forced to SENT where the mask is SENT (outside the image). max(x + e, mask) equals
// (x + e) | mask for a mask of 0 or SENT, and the fused add-max keeps the mask off the row chain's
// critical path better than a separate OR.
template <bool MASK>
__device__ __forceinline__ uint32_t add_mask(uint32_t x, uint32_t e, uint32_t mask) {
  if (MASK) return __viaddmax_u32(x, e, mask);
  return x + e;
}

// One DP row for a lane: keys k (previous row) -> next row; energies ev (4 x uint16).
// LAT (a latency-bound search, one compute warp per SM sub-partition) takes, in warps without
// excluded columns, the instruction forms that shorten the row's dependent chain at the price of
// a few more instructions: the pairwise minima of the lane's own columns first (independent of
// the neighbours' shuffled values), then the neighbour and the energy in one add-min
// (min(a + e, b + e) = min(a, b) + e, exact: keys stay below 2^32 - e there). The
// throughput-bound kernels (several warps per sub-partition) and the masked warps keep the
// 3-input minimum.
template <bool MASK, bool LAT = false>
__device__ __forceinline__ void dp_row(uint32_t (&k)[V], uint2 ev, const uint32_t (&oobm)[V]) {
  const uint32_t e0 = lo8(ev.x), e1 = hi8(ev.x), e2 = lo8(ev.y), e3 = hi8(ev.y);
  const uint32_t L = __shfl_up_sync(0xffffffffu, k[V - 1], 1);
  const uint32_t R = __shfl_down_sync(0xffffffffu, k[0], 1);
  uint32_t n0, n1, n2, n3;
  if (LAT && !MASK) {
    const uint32_t p01 = min(k[0], k[1]), p23 = min(k[2], k[3]);
    n0 = __viaddmin_u32(L, e0, p01 + e0);
    n1 = __viaddmin_u32(k[2], e1, p01 + e1);
    n2 = __viaddmin_u32(k[1], e2, p23 + e2);
    n3 = __viaddmin_u32(R, e3, p23 + e3);
  } else {
    n0 = add_mask<MASK>(min3u(L, k[0], k[1]), e0, oobm[0]);
    n1 = add_mask<MASK>(min3u(k[0], k[1], k[2]), e1, oobm[1]);
    n2 = add_mask<MASK>(min3u(k[1], k[2], k[3]), e2, oobm[2]);
    n3 = add_mask<MASK>(min3u(k[2], k[3], R), e3, oobm[3]);
  }
  k[0] = n0; k[1] = n1; k[2] = n2; k[3] = n3;
}

// Running maximum of a lane's energies (two uint16 pairs; columns outside the map masked to 0 by
// cm in warps that hold such columns) for the DIRECT range check; off the row's dependent chain.
template <bool CHK, bool MASK>
__device__ __forceinline__ void emax_acc(uint32_t &acc, uint2 ev, uint2 cm) {
  if (CHK) acc = __vimax3_u16x2(acc, MASK ? (ev.x & cm.x) : ev.x, MASK ? (ev.y & cm.y) : ev.y);
}

// n rows (n <= KT) of a tile from the staged energies er (row stride BW; REV: upwards), the energies
// loaded two rows ahead of the row that needs them, off the dependent chain: in blocks of U unrolled
// rows, and the last n % U rows of a ragged tile in blocks of 8 and then one by one. MASK applies
// oobm. The latency-bound search unrolls whole tiles (33 cycles a row at 4 warps; 37.6 in blocks of
// 8), the batched and multi-map kernels blocks of 8 (several warps hide the loop).
template <int U, int BW, bool MASK, bool LAT = false, bool CHK = false, bool REV = false>
__device__ __forceinline__ void dp_rows(uint32_t (&k)[V], const uint16_t *er, const uint32_t (&oobm)[V], int n,
                                        uint32_t &acc, uint2 cm) {
  constexpr int RS = REV ? -BW : BW;
  auto row = [&](int r) { return *reinterpret_cast<const uint2 *>(er + r * RS); };
  if (n >= U) {
    uint2 a = row(0), b = row(1);
    auto block = [&](auto more) {
#pragma unroll
      for (int r = 0; r < U; ++r) {
        const uint2 ev = a;
        a = b;
        if (decltype(more)::value || r + 2 < U) b = row(r + 2);
        dp_row<MASK, LAT>(k, ev, oobm);
        emax_acc<CHK, MASK>(acc, ev, cm);
      }
      er += U * RS;
      n -= U;
    };
    if (U == 8) {
#pragma unroll 1
      while (n >= 2 * U) block(std::true_type());
    }
    block(std::false_type());
  }
  if (U > 8) {
    if (n > 0) dp_rows<8, BW, MASK, LAT, CHK, REV>(k, er, oobm, n, acc, cm);
  } else {
#pragma unroll 1
    for (int r = 0; r < n; ++r) {
      const uint2 ev = row(r);
      dp_row<MASK, LAT>(k, ev, oobm);
      emax_acc<CHK, MASK>(acc, ev, cm);
    }
  }
}

// One forward-energy row: keys k (previous row) -> next row; cu, dl, dr: 4 x uint16 each.
template <bool MASK>
__device__ __forceinline__ void dp_row_fwd(uint32_t (&k)[V], uint2 cu, uint2 dl, uint2 dr, const uint32_t (&oobm)[V]) {
  const uint32_t L = __shfl_up_sync(0xffffffffu, k[V - 1], 1);
  const uint32_t R = __shfl_down_sync(0xffffffffu, k[0], 1);
  const uint32_t n0 = add_mask<MASK>(min3u(L + lo8(dl.x), k[0], k[1] + lo8(dr.x)), lo8(cu.x), oobm[0]);
  const uint32_t n1 = add_mask<MASK>(min3u(k[0] + hi8(dl.x), k[1], k[2] + hi8(dr.x)), hi8(cu.x), oobm[1]);
  const uint32_t n2 = add_mask<MASK>(min3u(k[1] + lo8(dl.y), k[2], k[3] + lo8(dr.y)), lo8(cu.y), oobm[2]);
  const uint32_t n3 = add_mask<MASK>(min3u(k[2] + hi8(dl.y), k[3], R + hi8(dr.y)), hi8(cu.y), oobm[3]);
  k[0] = n0; k[1] = n1; k[2] = n2; k[3] = n3;
}

// The same for a sweep upwards: a path that leaves column j of the row below (previous row, keys k) costs that
// row's DR towards column j + 1 and its DL towards column j - 1, so dl and dr are the previous row's and are
// added before the neighbours take the sums.
template <bool MASK>
__device__ __forceinline__ void dp_row_fwd_rev(uint32_t (&k)[V], uint2 cu, uint2 dl, uint2 dr, const uint32_t (&oobm)[V]) {
  uint32_t l[V] = {k[0] + lo8(dl.x), k[1] + hi8(dl.x), k[2] + lo8(dl.y), k[3] + hi8(dl.y)};   // towards j - 1
  uint32_t g[V] = {k[0] + lo8(dr.x), k[1] + hi8(dr.x), k[2] + lo8(dr.y), k[3] + hi8(dr.y)};   // towards j + 1
  if (MASK)
#pragma unroll
    for (int u = 0; u < V; ++u) {
      l[u] |= oobm[u];   // (an excluded cell's key plus a padding value would wrap)
      g[u] |= oobm[u];
    }
  const uint32_t L = __shfl_up_sync(0xffffffffu, g[V - 1], 1);
  const uint32_t R = __shfl_down_sync(0xffffffffu, l[0], 1);
  const uint32_t n0 = add_mask<MASK>(min3u(L, k[0], l[1]), lo8(cu.x), oobm[0]);
  const uint32_t n1 = add_mask<MASK>(min3u(g[0], k[1], l[2]), hi8(cu.x), oobm[1]);
  const uint32_t n2 = add_mask<MASK>(min3u(g[1], k[2], l[3]), lo8(cu.y), oobm[2]);
  const uint32_t n3 = add_mask<MASK>(min3u(g[2], k[3], R), hi8(cu.y), oobm[3]);
  k[0] = n0; k[1] = n1; k[2] = n2; k[3] = n3;
}

// KT forward-energy rows of a full tile (row stride BW); the three planes are PL elements apart in
// the staging ring.
template <int KT, int BW, int PL, bool MASK, bool REV>
__device__ __forceinline__ void dp_rows_fwd(uint32_t (&k)[V], const uint16_t *er, const uint32_t (&oobm)[V]) {
  constexpr int RS = REV ? -BW : BW;
  auto row = [&](int pl, int r) { return *reinterpret_cast<const uint2 *>(er + pl * PL + r * RS); };
  uint2 a0 = row(0, 0), a1 = row(1, 0), a2 = row(2, 0);
#pragma unroll
  for (int r = 0; r < KT; ++r) {
    const uint2 c0 = a0, c1 = a1, c2 = a2;
    if (r + 1 < KT) {
      a0 = row(0, r + 1);
      a1 = row(1, r + 1);
      a2 = row(2, r + 1);
    }
    if (REV) dp_row_fwd_rev<MASK>(k, c0, c1, c2, oobm);
    else dp_row_fwd<MASK>(k, c0, c1, c2, oobm);
  }
}

// n (n < KT) forward-energy rows of a ragged last tile.
template <int BW, int PL, bool MASK, bool REV>
__device__ __forceinline__ void dp_rows_n_fwd(uint32_t (&k)[V], const uint16_t *er, const uint32_t (&oobm)[V], int n) {
  constexpr int RS = REV ? -BW : BW;
  auto row = [&](int pl, int r) { return *reinterpret_cast<const uint2 *>(er + pl * PL + r * RS); };
  for (int r = 0; r < n; ++r) {
    if (REV) dp_row_fwd_rev<MASK>(k, row(0, r), row(1, r), row(2, r), oobm);
    else dp_row_fwd<MASK>(k, row(0, r), row(1, r), row(2, r), oobm);
  }
}

// Initialise the staging and halo mbarriers (thread 0; the caller then synchronises the CTA, and
// the cluster when CL).
__device__ inline void search_init(unsigned char *smem, const SearchPlan &plan) {
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + plan.bars);
  uint64_t *hbar = full + NSLOT;
  if (threadIdx.x == 0) {
    for (int q = 0; q < NSLOT; ++q) mbar_init(&full[q], 1);
    mbar_init(&hbar[0], 1);
    mbar_init(&hbar[1], 1);
    fence_mbar_init();
  }
}

template <bool CL>
__device__ __forceinline__ void group_sync() {
  if (CL) cg::this_cluster().sync(); else __syncthreads();
}

// The parallel backtrack of seam_search, one warp per super-tile (rows rs .. rs+n-1, n <= KSS). The
// ancestor chain has fixed both ends of the seam inside a super-tile: column jbs in its bottom row
// and column jprev in the row above it (in the added row above row 0 for the first one), and the
// seam between them is the leftmost cheapest path from one to the other: another candidate left of a
// path cell's predecessor has a larger full cost, so a larger cost from the upper end too. So the fill
// is a small search of its own, and like the search it runs from both ends at once: the upper nt rows
// downwards from jprev (cost 0 there, infinity everywhere else), the lower nb rows upwards from jbs,
// two independent chains in the same instructions; where they meet, the leftmost column of the cheapest
// join continues both ways, and two lanes walk the directions to the two ends.
// Only cells within r columns of an end, r rows from it, can be on the path: a diamond at most n + 1
// columns wide around the middle of the two. A window of FILLW = 2*KSS columns centred there
// (FV = KSS/16 per lane) keeps the shuffles' wrap-around at its edges, which spreads one column per
// row, out of the diamond.
// Costs are kept times 256 with the direction (0: from j-1, 1: from j, 2: from j+1) in the low byte of
// each candidate, so two add-minima yield the cost and the leftmost direction.
// Energies are read in chunks of fill_rows() rows, half of them from either end, every load of a chunk
// in flight at once, and held in shared memory, so that the row loop stays a loop: the code runs
// once per search and warp, from a cold instruction cache, where unrolled rows cost more to fetch
// than to execute (three rows at a time are the best of 1, 3 and 5: 3840x2160 57.2 / 55.8 / 56.1 us a seam).
// Latency-bound: the energies' round trip, then rows and walk of half a super-tile each (about 500, 1,900 and
// 1,300 cycles). Against full costs recomputed in a 4*KSS window from saved cost rows (25.0 ms a 1920x1080
// carve): between the two ends 24.5 ms (a batch of 256 images 44.5 -> 40.7 ms); from both ends, with the
// energies in shared memory and the fused minima, 3.8 -> 2.1 us of a 1920x1080 seam.
constexpr uint32_t FILL_INF = 0x80000000u;   // above every path's 256 * cost (64 rows * 2 * 65535 * 256 < 2^31)

struct FillCtx {
  const uint16_t *E;
  unsigned char *fill; // the fill warps' shared memory
  uint32_t *csum;      // receives the recomputed path costs ...
  uint32_t csign;      // ... times this (1 or -1)
  int32_t *seam, *seam_log;
  int *err;
  int64_t pstride;
  int pitch_e, H, W, Wa;
  int step = 1;        // seam entries from one row to the next (-1: the map is swept from its bottom row)
};

// L2 prefetch of a super-tile's diamond (KSS rows, two rows per lane at most; from a 16-byte boundary)
template <int KSS, bool FWD, bool DIRECT>
__device__ __forceinline__ void fill_prefetch(const FillCtx &f, int s, int jprev, int jbs, int lane) {
  int x0 = (((jprev + jbs) >> 1) - KSS / 2 - 1) & ~7;
  int x1 = x0 + KSS + 16;
  if (DIRECT) {   // only the caller's columns
    x0 = max(x0, 0);
    x1 = min(x1, f.Wa);
    if (x1 <= x0) return;
  }
  for (int i = s * KSS + lane; i < s * KSS + KSS && i < f.H; i += 32)
#pragma unroll
    for (int pl = 0; pl < (FWD ? 3 : 1); ++pl)
      bulk_prefetch_l2(f.E + pl * f.pstride + (ptrdiff_t)i * f.pitch_e + x0, (uint32_t)(x1 - x0) * 2);
}

// super-tile s between columns jprev and jbs, by one warp
// Forward energy: a step costs the DL or DR of the lower (image) of its two rows. In a map swept downwards
// the chain from above enters that row and adds its own DL and DR, the chain from below leaves it and
// carries them to the neighbours; FLIP (a map swept upwards) exchanges the two.
template <typename G, bool FWD, int KSS, bool DIRECT, bool FLIP = false>
__device__ __forceinline__ void fill_super_tile(const FillCtx &f, int s, int jprev, int jbs, int warp, int lane) {
  constexpr int NP = FWD ? 3 : 1;   // cost planes per row
  constexpr int FV = G::FV, FILLW = G::FILLW, CR = G::fill_rows(FWD), HC = CR / 2;
  using DirT = typename std::conditional<FV == 4, uint32_t, uint16_t>::type;   // a byte per column
  using EVec = typename std::conditional<FV == 4, uint2, uint32_t>::type;      // FV uint16 energies
  unsigned char *const wmem = f.fill + (size_t)warp * G::fill_bytes(FWD);
  EVec *const est = reinterpret_cast<EVec *>(wmem) + lane;   // this lane's energies: plane, end, row
  uint8_t *const fd = wmem + CR * FILLW * 2 * NP;            // direction rows
  const int x0 = (((jprev + jbs) >> 1) - FILLW / 2) & ~(FV - 1);
  const int xc = x0 + lane * FV;
  const int rs = s * KSS, n = min(KSS, f.H - rs);
  // the upper nt rows and the lower nb; after the bottom row, which only holds the path's end, and the
  // top row where nt = nb, both chains have T more rows to run together
  const int nt = n >> 1, nb = n - nt, T = nb - 1, lead = nt - T;   // lead: 0 or 1
  // costs from above and from below (FWD: the carrying chain's plus DL, DR of their row; FLIP: the other one's)
  uint32_t m[FV], w[FV], cl[FV], cr[FV], oob[FV];
#pragma unroll
  for (int u = 0; u < FV; ++u) {
    oob[u] = (xc + u < 0 || xc + u >= f.W) ? FILL_INF : 0u;
    m[u] = (xc + u == jprev) ? 0u : FILL_INF;
  }
  // 256 * energy of the lane's columns
  auto unpack = [](const EVec &v, uint32_t (&x)[FV]) {
    const uint32_t *p = reinterpret_cast<const uint32_t *>(&v);
#pragma unroll
    for (int q = 0; q < FV / 2; ++q) {
      x[2 * q] = lo8(p[q]);
      x[2 * q + 1] = hi8(p[q]);
    }
  };
  // one row: costs m (candidates from the left l, from the right r) -> new costs plus energies e, and
  // the directions in the low bytes of the candidates' minima
  auto step_row = [&](const uint32_t (&l)[FV], const uint32_t (&c)[FV], const uint32_t (&r)[FV], const uint32_t (&e)[FV],
                      uint32_t (&out)[FV], uint8_t *dst) {
    uint32_t mn[FV];
#pragma unroll
    for (int u = 0; u < FV; ++u) {
      mn[u] = __viaddmin_u32(r[u], 2u, __viaddmin_u32(c[u], 1u, l[u]));
    }
#pragma unroll
    for (int u = 0; u < FV; ++u) {
      out[u] = __viaddmax_u32(mn[u] & ~0xFFu, e[u], oob[u]);
    }
    uint32_t d = __byte_perm(mn[0], mn[1], 0x0040);
    if (FV == 4) d = __byte_perm(d, __byte_perm(mn[FV - 2], mn[FV - 1], 0x0040), 0x5410);
    *reinterpret_cast<DirT *>(dst) = (DirT)d;
  };
  // DIRECT: a lane's FV columns lie wholly inside or wholly outside the caller's [0, Wa)
  const bool xin = !DIRECT || (xc >= 0 && xc + FV <= f.Wa);
  // chunk q0: the rows q0, q0 + 1, ... after the top row(s) led by, and before the bottom row
  EVec eb[NP][CR];
  auto load_chunk = [&](int q0) {
#pragma unroll
    for (int pl = 0; pl < NP; ++pl) {
      const uint16_t *top = f.E + pl * f.pstride + (ptrdiff_t)(rs + lead + q0) * f.pitch_e + xc;
      const uint16_t *bot = f.E + pl * f.pstride + (ptrdiff_t)(rs + n - 2 - q0) * f.pitch_e + xc;
#pragma unroll
      for (int r = 0; r < HC; ++r, top += f.pitch_e, bot -= f.pitch_e) {
        eb[pl][r] = eb[pl][HC + r] = EVec{};
        if (xin && q0 + r < T) {
          eb[pl][r] = *reinterpret_cast<const EVec *>(top);
          eb[pl][HC + r] = *reinterpret_cast<const EVec *>(bot);
        }
      }
    }
  };
  auto load_row = [&](int i, int pl) {
    return xin ? *reinterpret_cast<const EVec *>(f.E + pl * f.pstride + (ptrdiff_t)(rs + i) * f.pitch_e + xc) : EVec{};
  };
  // the candidates of a chain from its costs x: neighbours' values by shuffle
  auto entering = [&](const uint32_t (&x)[FV], const uint32_t (&dl)[FV], const uint32_t (&dr)[FV], uint32_t (&l)[FV],
                      uint32_t (&r)[FV]) {
    const uint32_t L = __shfl_up_sync(0xffffffffu, x[FV - 1], 1), R = __shfl_down_sync(0xffffffffu, x[0], 1);
#pragma unroll
    for (int u = 0; u < FV; ++u) {
      l[u] = (u == 0 ? L : x[u > 0 ? u - 1 : 0]) + (FWD ? dl[u] : 0u);
      r[u] = (u == FV - 1 ? R : x[u < FV - 1 ? u + 1 : u]) + (FWD ? dr[u] : 0u);
    }
  };
  auto leaving = [&](uint32_t (&l)[FV], uint32_t (&r)[FV]) {
    const uint32_t L = __shfl_up_sync(0xffffffffu, cr[FV - 1], 1), R = __shfl_down_sync(0xffffffffu, cl[0], 1);
#pragma unroll
    for (int u = 0; u < FV; ++u) {
      l[u] = u == 0 ? L : cr[u > 0 ? u - 1 : 0];
      r[u] = u == FV - 1 ? R : cl[u < FV - 1 ? u + 1 : u];
    }
  };
  auto carry = [&](const uint32_t (&x)[FV], const uint32_t (&dl)[FV], const uint32_t (&dr)[FV]) {
    if (FWD)
#pragma unroll
      for (int u = 0; u < FV; ++u) {
        cl[u] = x[u] + dl[u];
        cr[u] = x[u] + dr[u];
      }
  };
  auto down_row = [&](const uint32_t (&e)[FV], const uint32_t (&dl)[FV], const uint32_t (&dr)[FV], uint8_t *dst) {
    uint32_t l[FV], r[FV];
    if (FWD && FLIP) leaving(l, r);
    else entering(m, dl, dr, l, r);
    step_row(l, m, r, e, m, dst);
    if (FLIP) carry(m, dl, dr);
  };
  auto up_row = [&](const uint32_t (&e)[FV], const uint32_t (&dl)[FV], const uint32_t (&dr)[FV], uint8_t *dst) {
    uint32_t l[FV], r[FV];
    if (FWD && !FLIP) leaving(l, r);
    else entering(w, dl, dr, l, r);
    step_row(l, w, r, e, w, dst);
    if (!FLIP) carry(w, dl, dr);
  };
  EVec et0[NP], eb0[NP];   // the bottom row and the leading top row
#pragma unroll
  for (int pl = 0; pl < NP; ++pl) {
    eb0[pl] = load_row(n - 1, pl);
    et0[pl] = lead ? load_row(0, pl) : EVec{};
  }
  load_chunk(0);
  {
    uint32_t e[FV], dl[FV] = {}, dr[FV] = {};
    unpack(eb0[0], e);
    if (FWD) {
      unpack(eb0[NP > 1 ? 1 : 0], dl);
      unpack(eb0[NP > 2 ? 2 : 0], dr);
    }
#pragma unroll
    for (int u = 0; u < FV; ++u) w[u] = (xc + u == jbs) ? e[u] : FILL_INF;
    if (!FLIP) carry(w, dl, dr);
    if (FWD && FLIP) {
      // the chain from above leaves row rs - 1 (the added row, without costs, for s = 0)
      uint32_t pl[FV] = {}, pr[FV] = {};
      if (rs > 0) {
        unpack(load_row(-1, NP > 1 ? 1 : 0), pl);
        unpack(load_row(-1, NP > 2 ? 2 : 0), pr);
      }
      carry(m, pl, pr);
    }
    *reinterpret_cast<DirT *>(fd + (n - 1) * FILLW + lane * FV) = (DirT)0x01010101u;   // no step below it
    if (lead) {
      unpack(et0[0], e);
      if (FWD) {
        unpack(et0[NP > 1 ? 1 : 0], dl);
        unpack(et0[NP > 2 ? 2 : 0], dr);
      }
      down_row(e, dl, dr, fd + lane * FV);
    }
  }
#pragma unroll 1
  for (int q0 = 0; q0 < T; q0 += HC) {
    // each lane reads back only what it stored
#pragma unroll
    for (int pl = 0; pl < NP; ++pl)
#pragma unroll
      for (int r = 0; r < CR; ++r) est[(pl * CR + r) * 32] = eb[pl][r];
    if (CR < KSS && q0 + HC < T) load_chunk(q0 + HC);   // in flight during this chunk's rows
    const int nq = min(HC, T - q0);
    const EVec *es = est;
    uint8_t *ft = fd + (lead + q0) * FILLW + lane * FV, *fb = fd + (n - 2 - q0) * FILLW + lane * FV;
#pragma unroll (FWD ? 1 : 3)
    for (int r = 0; r < nq; ++r, ft += FILLW, fb -= FILLW, es += 32) {
      uint32_t e[FV], g[FV], dl[FV] = {}, dr[FV] = {}, gl[FV] = {}, gr[FV] = {};
      unpack(es[0], e);
      unpack(es[HC * 32], g);
      if (FWD) {
        unpack(es[CR * 32], dl);
        unpack(es[2 * CR * 32], dr);
        unpack(es[(CR + HC) * 32], gl);
        unpack(es[(2 * CR + HC) * 32], gr);
      }
      up_row(g, gl, gr, fb);
      down_row(e, dl, dr, ft);
    }
  }
  // the join: the leftmost column of row nt - 1 (jprev itself when nt = 0) on a cheapest path, and the
  // leftmost of its three successors
  uint32_t best = SENT, where = SENT;   // cost * 256; column in the window << 2 | direction
  {
    // the cost up to column j and on to j - 1, j, j + 1 of the next row
    uint32_t l[FV], r[FV];
    const uint32_t zero[FV] = {};
    if (FWD && !FLIP) leaving(l, r);
    else entering(w, zero, zero, l, r);
#pragma unroll
    for (int u = 0; u < FV; ++u) {
      const uint32_t a = (FWD && FLIP ? cl[u] : m[u]), c = (FWD && FLIP ? cr[u] : m[u]);
      // (a sum with an excluded term stays above FILL_INF, or wraps when both are: tested first)
      const uint32_t sl = m[u] >= FILL_INF || l[u] >= FILL_INF ? SENT - 2u : a + l[u];
      const uint32_t sc = m[u] >= FILL_INF || w[u] >= FILL_INF ? SENT - 2u : m[u] + w[u];
      const uint32_t sr = m[u] >= FILL_INF || r[u] >= FILL_INF ? SENT - 2u : c + r[u];
      const uint32_t mn = __viaddmin_u32(sr, 2u, __viaddmin_u32(sc, 1u, sl));
      if (mn < SENT - 2u && (mn & ~0xFFu) < best) {
        best = mn & ~0xFFu;
        where = ((uint32_t)(lane * FV + u) << 2) | (mn & 3u);
      }
    }
    const uint32_t b = __reduce_min_sync(0xffffffffu, best);
    where = __reduce_min_sync(0xffffffffu, best == b ? where : SENT);
    best = b;
  }
  if (lane == 0) atomicAdd(f.csum, (best >> 8) * f.csign);   // the path's cost in this super-tile
  // lanes 0 and 1 follow the directions up and down (relative columns, kept in the direction rows they
  // have read: a row's entry is not needed again), then the warp writes the seam rows. The barrier
  // orders every lane's direction stores before the walk: shuffles and reductions order no memory.
  __syncwarp();
  if (lane < 2) {
    // a path that leaves the window (it cannot) wraps around inside this warp's rows and ends on the
    // wrong column
    int rel = ((int)(where >> 2) + (lane ? (int)(where & 3u) - 1 : 0)) & (FILLW - 1);
    uint8_t *fb = fd + (lane ? nt : nt - 1) * FILLW;
    const int stride = lane ? FILLW : -FILLW, steps = lane ? nb : nt;
#pragma unroll 4
    for (int q = 0; q < steps; ++q, fb += stride) {
      const int nr = rel + (int)(fb[rel] & 3u) - 1;
      *reinterpret_cast<uint32_t *>(fb) = (uint32_t)rel;
      rel = nr & (FILLW - 1);
    }
    if (best == SENT || x0 + rel != (lane ? jbs : jprev)) atomicOr(f.err, ERR_FILL_MISMATCH);
  }
  __syncwarp();
  for (int i = lane; i < n; i += 32) {
    const int j = x0 + (int)*reinterpret_cast<const uint32_t *>(fd + i * FILLW);
    f.seam[(rs + i) * f.step] = j;
    if (f.seam_log) f.seam_log[(rs + i) * f.step] = j;
  }
  __syncwarp();
}

// The super-tiles of one warp, warp*cs + rank, + FW*cs, ... of S; jb: the chain's columns (rank 0's
// table). The energies of a super-tile's diamond are prefetched into L2 one super-tile ahead: the map
// may have left L2 since the DP pass read it.
template <typename G, bool FWD, int KSS, bool DIRECT>
__device__ __forceinline__ void backtrack_fill(const FillCtx &f, const int *jb, int S, int cs, int rank, int warp,
                                               int lane) {
  auto prev = [&](int s) { return s > 0 ? jb[s - 1] : jb[S]; };
#pragma unroll 1
  for (int s = warp * cs + rank; s < S; s += G::FW * cs) {
    const int nx = s + G::FW * cs;
    if (nx < S) fill_prefetch<KSS, FWD, DIRECT>(f, nx, prev(nx), jb[nx], lane);
    fill_super_tile<G, FWD, KSS, DIRECT>(f, s, prev(s), jb[s], warp, lane);
  }
}

// backtrack_fill as a function of its own (not inlined): it gets its own register allocation, so
// the one-CTA batched kernel, whose 512 threads have at most 128 registers each, can load deeper
// energy chunks
template <typename G, bool FWD, int KSS, bool DIRECT>
static __device__ __noinline__ void backtrack_fill_call(FillCtx f, const int *jb, int S, int cs, int rank, int warp,
                                                        int lane) {
  backtrack_fill<G, FWD, KSS, DIRECT>(f, jb, S, cs, rank, warp, lane);
}

// The row loop: every thread of the CTA (of every CTA of the cluster when CL) calls it with the same
// arguments; `plan` is the shared-memory plan. Returns the thread's minimum of the last row
// (M << 32 | column). With TWO (half of a two-ended search) the ancestors go to the global table
// p.gtab (row stride p.gw) and the last row's costs to p.endrow instead.
// TM stages a tile's rows with tensor copies of p.tmap, NBOX boxes of KT rows side by side (a
// row-by-row copy costs its warp about 65 cycles, 2,100 per 32-row tile: more than the tile's rows
// take, so the producer paced the sweep); the box rows of the half swept upwards (REV) lie in reverse
// order. Half a 1920x1080 map: 40,000 -> 29,700 cycles; 3840x2160: 88,500 -> 73,500; a forward-energy
// carve at 1920x1080 (three planes: 48 row copies per 16-row tile) 60.3 -> 34.9 ms. The one-CTA batched
// kernel and the two-ended clusters copy through the tensor map of the image's own energies. The multi-map
// kernel, whose maps are the callers', and the 8-row-tile clusters keep the row copies: 8 copies a tile.
template <int NW, int KT, bool CL, int FWM, bool FWD, int KSS, bool DIRECT, bool TM, bool TWO = false, bool REV = false>
__device__ __forceinline__ unsigned long long seam_sweep(const SearchArgs &p, unsigned char *smem, const SearchPlan &plan,
                                                         SearchState &st) {
  static_assert(!DIRECT || (CL && !FWD), "the in-place form is built for the cluster search of e1 maps");
  constexpr int NP = FWD ? 3 : 1;   // cost planes staged per row
  // the single-map search: one cluster, a CTA per SM, every compute warp alone on its SM
  // sub-partition with 4 warps (latency-bound)
  constexpr bool LAT = CL && FWM >= FILL_WARPS_MAX && NW == 4;
  using G = Geo<NW, KT, CL, FWM, KSS>;
  constexpr int Q = G::Q, BW = G::BW, OWC = G::OWC, K2E = G::K2E;
  const int rank0 = TWO ? p.rank0 : 0;
  const int rank = CL ? (int)cg::this_cluster().block_rank() - rank0 : 0;
  const int cs = CL ? (TWO && p.ctas ? p.ctas : (int)cg::this_cluster().num_blocks()) : 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool producer = (warp == NW);
  const int H = p.H, W = p.W;
  uint32_t *bnd = reinterpret_cast<uint32_t *>(smem + plan.bnd);
  uint32_t *hbuf = reinterpret_cast<uint32_t *>(smem + plan.hbuf);
  uint8_t *ancT = reinterpret_cast<uint8_t *>(smem + plan.anc);
  uint32_t *emx = reinterpret_cast<uint32_t *>(smem + plan.emx);   // DIRECT: [NW + 1] per warp, then per CTA
  uint16_t *ring = reinterpret_cast<uint16_t *>(smem + plan.ring);
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + plan.bars);
  uint64_t *hbar = full + NSLOT;
  const int gw = TWO ? p.gw : plan.gw;
  uint8_t *const gat0 = TWO ? p.gtab : ((CL && gw) ? cg::this_cluster().map_shared_rank(smem + plan.gat, 0) : smem + plan.gat);

  // geometry
  // (a cluster of a batch: no CTA lies beyond the map's edges, and the columns it would own there are the
  // outermost CTAs' own)
  const int edge_cols = TWO && p.ctas ? K2E : 0;
  const int ext0 = rank * OWC - K2E + edge_cols;   // extended range start
  const int A = rank == 0 ? 0 : ext0 + K2E, B = ext0 + K2E + OWC + (rank == cs - 1 ? edge_cols : 0);
  const int own0 = ext0 + warp * Q;             // warp strip start
  const int c0 = own0 - KT + lane * V;          // this lane's first column
  const int frame_base = own0 - KSS;            // ancestor frame of this warp
  const bool strip_lane = !producer && (lane * V >= KT) && (lane * V < KT + Q);
  const bool cta_own = strip_lane && c0 >= A && c0 < B;   // own columns; A, B, c0 are multiples of 4
  uint32_t oobm[V];
#pragma unroll
  for (int u = 0; u < V; ++u) oobm[u] = (c0 + u < 0 || c0 + u >= W) ? SENT : 0u;
  const bool edge = __any_sync(0xffffffffu, (oobm[0] | oobm[V - 1]) != 0u);
  const int bidx0 = c0 - (ext0 - KT);           // index of c0 in bnd and in a staged energy row
  constexpr int NBOX = TM ? tensor_boxes(BW) : 1;
  constexpr int BWB = TM ? tensor_box_cols(BW) : BW;  // staged row stride
  constexpr int SLOT = KT * NBOX * BWB;              // elements of a staged tile (one plane)
  static_assert(BWB % 4 == 0 && (!TM || (KT * BWB * 2) % 128 == 0), "tensor box");
  unsigned long long lastmin = ~0ull;
  const int nt = p.gated ? 0 : (H + KT - 1) / KT;
  // single CTA: only the warps whose strips reach into [0, W) compute, and only their columns are
  // staged (a cluster is sized to W, so all its warps work)
  const int nwa = CL ? NW : min(NW, (W + Q - 1) / Q);
  const bool active = warp < nwa;
  const uint32_t ROW_BYTES = CL ? (uint32_t)BW * 2 : (uint32_t)(nwa * Q + 2 * KT) * 2;
  // fields used inside the loops, held in registers (stores through the map pointers could
  // otherwise force reloads of the argument struct)
  const int pitch_e = p.pitch_e;
  const int64_t pstride = FWD ? p.pstride : 0;
  // DIRECT: the columns that exist in the caller's array, [0, Wa); rows are copied only there
  const int Wa = (W + 7) & ~7;
  const int cbeg = ext0 - KT;   // first staged column (a multiple of 8)
  const int clo = DIRECT ? max(cbeg, 0) : cbeg;
  const int chi = DIRECT ? min(cbeg + (int)(ROW_BYTES / 2), Wa) : cbeg + (int)(ROW_BYTES / 2);
  const uint32_t COPY_BYTES = (uint32_t)(chi - clo) * 2;

  if (producer) {
    // ---- energy staging: rows of columns [ext0 - KT, ext0 - KT + BW), by the first lane's tensor copies
    // or one bulk copy per lane ----
    const uint16_t *Estage = p.E + (ext0 - KT);
    auto issue = [&](int tt) {
      const int slot = (int)((st.tiles + tt) % NSLOT);
      const int rbeg = tt * KT;
      if constexpr (TM) {
        if (lane == 0) {
          // (a single CTA stages only the boxes its active warps read)
          const int nbox = CL ? NBOX : min(NBOX, (nwa * Q + 2 * KT + BWB - 1) / BWB);
          mbar_arrive_expect_tx(&full[slot], (uint32_t)(NP * nbox * KT * BWB * 2));
          const int y = REV ? p.y0 - rbeg - (KT - 1) : p.y0 + rbeg;
#pragma unroll
          for (int pl = 0; pl < NP; ++pl)
#pragma unroll (CL ? NBOX : 1)
            for (int b = 0; b < nbox; ++b)
              tensor_g2s_2d(ring + (size_t)(slot * NP + pl) * SLOT + b * KT * BWB, p.tmap, p.x0 + cbeg + b * BWB,
                            y + pl * p.plane_rows + (REV && pl > 0 ? 1 : 0), &full[slot]);   // (REV: DL, DR of the row below)
        }
        return;
      }
      const int nrows = (H - rbeg < KT) ? H - rbeg : KT;
      if (lane == 0) mbar_arrive_expect_tx(&full[slot], (uint32_t)(NP * nrows) * COPY_BYTES);
      __syncwarp();
      if (lane < nrows) {
#pragma unroll
        for (int pl = 0; pl < NP; ++pl)
          bulk_g2s(ring + (size_t)(slot * NP + pl) * SLOT + lane * BW + (clo - cbeg),
                   Estage + pl * pstride + (ptrdiff_t)(rbeg + lane) * pitch_e + (clo - cbeg), COPY_BYTES, &full[slot]);
      }
    };
    fence_proxy_async_smem();   // the ring's place may have held other data before this search
    for (int tt = 0; tt < NSLOT && tt < nt; ++tt) issue(tt);
    // The barrier that ends tile t has every warp's word that it has read the tile's slot, and this
    // warp's that the next tile has landed: the compute warps never wait on a staging barrier
    // after the first tile.
    for (int t = 0; t + 1 < nt; ++t) {
      const uint32_t g = st.tiles + t + 1;
      if (!mbar_wait_bounded(&full[g % NSLOT], (g / NSLOT) & 1u, WAIT_TIMEOUT_NS)) {
        if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
      }
      named_bar_sync(G::THREADS);
      if (t + NSLOT < nt) issue(t + NSLOT);
    }
  } else if (!active) {
    // outside the image: keep the barrier count
    for (int t = 0; t + 1 < nt; ++t) named_bar_sync(G::THREADS);
  } else {
    const uint32_t own_a = (uint32_t)(c0 - frame_base);   // this lane's first column, warp frame
    uint32_t emax = 0u;   // DIRECT: running maximum of this lane's in-map energies (two uint16 halves)
    const uint2 cm = make_uint2((oobm[0] ? 0u : 0xFFFFu) | (oobm[1] ? 0u : 0xFFFF0000u),
                                (oobm[2] ? 0u : 0xFFFFu) | (oobm[3] ? 0u : 0xFFFF0000u));
    // the neighbour's halo buffer that this lane's own columns go to at an exchange: the first K2 own
    // columns are the left neighbour's right halo, the last K2 the right neighbour's left halo
    static_assert(!CL || OWC >= 2 * K2, "a column is pushed to one neighbour");
    uint32_t push = 0u, push_bar = 0u;
    if constexpr (CL) {
      const bool tl = cta_own && rank > 0 && c0 < A + K2, tr = cta_own && rank < cs - 1 && c0 >= B - K2;
      if (tl || tr) {
        push = mapa_u32(hbuf + (tl ? K2 + (c0 - A) : c0 - (B - K2)), rank0 + (tl ? rank - 1 : rank + 1));
        push_bar = mapa_u32(hbar, rank0 + (tl ? rank - 1 : rank + 1));
      }
    }
    uint8_t *anc_out = TWO ? gat0 + c0 : nullptr;   // where this lane's ancestors of the current super-tile go
    // this lane's place in the halo buffer where its columns are a neighbour's (-1: this CTA's)
    int hoff = -1;
    if (CL && rank > 0 && c0 >= A - K2 && c0 < A) hoff = c0 - (A - K2);
    if (CL && rank < cs - 1 && c0 >= B && c0 < B + K2) hoff = K2 + (c0 - B);
    const bool hneed = CL && __any_sync(0xffffffffu, hoff >= 0);
    // with one tile per super-tile every boundary starts new ancestors, and only costs cross it
    constexpr bool FRESH = KSS == KT;
    const int er0 = TM ? (bidx0 / BWB) * KT * BWB + bidx0 % BWB + (REV ? (KT - 1) * BWB : 0) : bidx0;
    // The tile loop, compiled twice: EDGE warps hold columns outside the image and apply the
    // exclusion mask on every row; the others never test it.
    auto tiles = [&](auto edge_tag) {
      constexpr bool EDGE = decltype(edge_tag)::value;
      // the row above row 0: cost 0 in every column, each its own ancestor (row 0 then costs its
      // energies; the leftmost optimal path of the extended map is the seam below a column of the
      // added row, so no tile is special)
      uint32_t k[V];
#pragma unroll
      for (int u = 0; u < V; ++u) k[u] = (own_a + u) | (EDGE ? oobm[u] : 0u);
      if (nt > 0 && !mbar_wait_bounded(&full[st.tiles % NSLOT], (st.tiles / NSLOT) & 1u, WAIT_TIMEOUT_NS)) {
        if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
      }
      // few branches: a branch and its reconvergence cost about as much as a row in these short chains, so
      // the conditions are uniform ones, lanes are told apart by predicated stores, and the window of the
      // next tile is loaded behind the barrier of this one (per seam: 1920x1080 26.1 -> 24.3 us, 3840x2160
      // 61.1 -> 57.2, forward energy at 1920x1080 48.3 -> 41.5, 1254x944 on one CTA 170.9 -> 165.6; 58 concurrent
      // 3840x2160 maps 258 -> 242 us; fixed row counts before that: 26.4 -> 26.1, 62.3 -> 61.1, 264 -> 258)
      for (int t = 0; t < nt; ++t) {
        const int r0 = t * KT;
        const int n = (H - r0 < KT) ? H - r0 : KT;
        const uint16_t *er = ring + (size_t)((st.tiles + t) % NSLOT) * NP * SLOT + er0;
        if (FWD) {
          if (n == KT) dp_rows_fwd<KT, BWB, SLOT, EDGE, REV>(k, er, oobm);
          else dp_rows_n_fwd<BWB, SLOT, EDGE, REV>(k, er, oobm, n);
        } else {
          constexpr int U = CL && FWM >= FILL_WARPS_MAX ? KT : 8;
          if (n == KT) dp_rows<U, BWB, EDGE, LAT, DIRECT, REV>(k, er, oobm, KT, emax, cm);   // (a fixed count)
          else dp_rows<8, BWB, EDGE, LAT, DIRECT, REV>(k, er, oobm, n, emax, cm);
        }
        const bool more = t + 1 < nt;
        // bookkeeping on the tile's last row, the only one where a super-tile (KSS is a multiple
        // of KT) or the image can end: the ancestors of the CTA-own columns (in rank 0's gathered
        // table, the global one or this CTA's), and below the last row its costs
        if (FRESH || ((r0 + n) % KSS) == 0 || !more) {
          const uint32_t anc = pack_ancestors(k, c0, frame_base);
          if (TWO) {
            if (cta_own) *reinterpret_cast<uint32_t *>(anc_out) = anc;
            anc_out += gw;
          } else {
            const size_t sup = (size_t)((r0 + n - 1) / KSS);
            uint8_t *const dst = gw ? gat0 + sup * gw + c0 : ancT + sup * OWC + (c0 - A);
            if (cta_own) *reinterpret_cast<uint32_t *>(dst) = anc;
          }
        }
        if (!more) {
          if (TWO) {
            if (cta_own)
              *reinterpret_cast<uint4 *>(p.endrow + c0) = make_uint4(k[0] >> 8, k[1] >> 8, k[2] >> 8, k[3] >> 8);
          } else if (cta_own) {
#pragma unroll
            for (int u = 0; u < V; ++u) {
              if (c0 + u < W) {
                const unsigned long long c = ((unsigned long long)(k[u] >> 8) << 32) | (unsigned)(c0 + u);
                lastmin = c < lastmin ? c : lastmin;
              }
            }
          }
          break;
        }
        // publish this warp's strip (relative ancestor encoding)
        const uint32_t d = own_a - 128u, dp = FRESH ? 0u : d, du = FRESH ? 0u : 1u;
        uint4 v;
        v.x = k[0] - dp; v.y = k[1] - dp - du; v.z = k[2] - dp - 2 * du; v.w = k[3] - dp - 3 * du;
        const bool exch = CL && ((r0 + KT) % K2 == 0) && cs > 1;
        const uint32_t xg = st.exch + (uint32_t)((r0 + KT) / K2 - 1);
        if constexpr (CL) if (exch) {
          // read there at the start of the next tile
          if (push) st_async_v4(push + (xg & 1u) * (2 * K2 * 4), v, push_bar + (xg & 1u) * 8);
          if (threadIdx.x == 0)
            mbar_arrive_expect_tx(&hbar[xg & 1u], (uint32_t)(((rank > 0) + (rank < cs - 1)) * K2 * 4));
        }
        uint32_t *const bt = bnd + (t & 1) * BW + bidx0;
        if (strip_lane) *reinterpret_cast<uint4 *>(bt) = v;
        named_bar_sync(G::THREADS);
        // the next tile's window from the boundary buffer, or from the halo buffer for a neighbour's columns
        // after an exchange (relative ancestors -> warp frame). At a new super-tile every cell becomes its
        // own ancestor; the old ancestor field is dropped without arithmetic (it may lie outside this
        // warp's frame).
        const uint32_t *src = bt;
        if (CL && hneed && exch) {
          if (!mbar_wait_bounded(&hbar[xg & 1u], (xg >> 1) & 1u, WAIT_TIMEOUT_NS)) {
            if (lane == 0) atomicOr(p.err, ERR_TIMEOUT);
          }
          if (hoff >= 0) src = hbuf + (int)(xg & 1u) * 2 * K2 + hoff;
        }
        const uint4 y = *reinterpret_cast<const uint4 *>(src);
        const bool fresh = FRESH || ((r0 + KT) % KSS) == 0;
        k[0] = fresh ? ((y.x & ~0xFFu) | own_a) : (y.x + d);
        k[1] = fresh ? ((y.y & ~0xFFu) | (own_a + 1u)) : (y.y + d + 1u);
        k[2] = fresh ? ((y.z & ~0xFFu) | (own_a + 2u)) : (y.z + d + 2u);
        k[3] = fresh ? ((y.w & ~0xFFu) | (own_a + 3u)) : (y.w + d + 3u);
        if (EDGE) { k[0] |= oobm[0]; k[1] |= oobm[1]; k[2] |= oobm[2]; k[3] |= oobm[3]; }
      }
    };
    if (edge) tiles(std::integral_constant<bool, true>());
    else tiles(std::integral_constant<bool, false>());
    if (DIRECT) {
      const uint32_t m = __reduce_max_sync(0xffffffffu, max(emax & 0xFFFFu, emax >> 16));
      if (lane == 0) {
        if (TWO) atomicMax(p.gmax, m);
        else emx[warp] = m;
      }
    }
  }
  if (DIRECT && !TWO && lane == 0 && (producer || !active)) emx[warp] = 0u;
  st.tiles += (uint32_t)nt;
  if (CL && nt > 0) st.exch += (uint32_t)((cs > 1) ? ((H - 1) / K2) : 0);
  return lastmin;
}

// The search. Every thread of the CTA (of every CTA of the cluster when CL) calls it with the same
// arguments; `Smax` is the super-tile count the shared-memory plan was sized for.
template <int NW, int KT, bool CL, int FWM = FILL_WARPS_MAX, bool FWD = false, int KSS = KS, bool DIRECT = false,
          bool TM = false>
__device__ void seam_search(const SearchArgs &p, unsigned char *smem, int Smax, SearchState &st) {
  using G = Geo<NW, KT, CL, FWM, KSS>;
  constexpr int OWC = G::OWC;
  const int rank = CL ? (int)cg::this_cluster().block_rank() : 0;
  const int cs = CL ? (int)cg::this_cluster().num_blocks() : 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int H = p.H, W = p.W, Wa = (W + 7) & ~7;
  const int S = (H + KSS - 1) / KSS;
  const SearchPlan plan = search_plan<NW, KT, CL, FWM, FWD, KSS, DIRECT, TM>(Smax);
  uint8_t *ancT = reinterpret_cast<uint8_t *>(smem + plan.anc);
  unsigned long long *wmin = reinterpret_cast<unsigned long long *>(smem + plan.wmin);
  unsigned long long *cmin = reinterpret_cast<unsigned long long *>(smem + plan.cmin);
  int *jb = reinterpret_cast<int *>(smem + plan.jb);
  int *misc = reinterpret_cast<int *>(smem + plan.misc);
  uint32_t *emx = reinterpret_cast<uint32_t *>(smem + plan.emx);   // DIRECT: [NW + 1] per warp, then per CTA
  const int gw = plan.gw;
  uint8_t *const gat = smem + plan.gat;
  const int64_t pstride = FWD ? p.pstride : 0;

  unsigned long long lastmin = seam_sweep<NW, KT, CL, FWM, FWD, KSS, DIRECT, TM>(p, smem, plan, st);

  // ---- last-row argmin: the leftmost minimum (min of (M << 32) | column) ----
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, lastmin, off);
    lastmin = o < lastmin ? o : lastmin;
  }
  if (lane == 0) wmin[warp] = lastmin;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long m = ~0ull;
    for (int w = 0; w <= NW; ++w) m = wmin[w] < m ? wmin[w] : m;
    if (CL) cg::this_cluster().map_shared_rank(cmin, 0)[rank] = m;   // pushed to rank 0
    else cmin[0] = m;
    if (DIRECT) {
      uint32_t e = 0u;
      for (int w = 0; w <= NW; ++w) e = max(e, emx[w]);
      cg::this_cluster().map_shared_rank(emx, 0)[NW + 1 + rank] = e;
    }
  }
  group_sync<CL>();

  // ---- ancestor chain (rank 0, one thread): seam column at every super-tile bottom ----
  uint32_t best_m = 0u;   // the argmin's cost (rank 0, thread 0)
  if (rank == 0 && threadIdx.x == 0) {
    int ok = !p.gated;
    unsigned long long best = ~0ull;
    for (int r = 0; r < cs; ++r) best = cmin[r] < best ? cmin[r] : best;
    if (DIRECT && ok) {
      // the 24-bit keys hold the seam sums only while H * max(e) < 2^24; otherwise this result is
      // void and the wide-cost search, launched next, takes the map
      uint32_t e = 0u;
      for (int r = 0; r < cs; ++r) e = max(e, emx[NW + 1 + r]);
      if ((uint64_t)e * (uint64_t)H >= ((uint64_t)1 << 24)) {
        ok = 0;
        if (p.gate) atomicOr(p.gate, ERR_ENERGY_RANGE);
      }
    }
    int j = (int)(best & 0xFFFFFFFFull);
    if (ok && (j < 0 || j >= W)) { ok = 0; atomicOr(p.err, ERR_BAD_SEAM); }
    if (ok && gw) {
      // branch-free hops: a column outside the map is clamped (every table read stays inside
      // the table) and recorded as a failure
      bool bad = false;
      for (int s = S - 1; s >= 0; --s) {
        jb[s] = j;
        const int nj = j + (int)gat[(size_t)s * gw + j] - 128;
        bad |= (unsigned)nj >= (unsigned)W;
        j = min(max(nj, 0), W - 1);
      }
      if (bad) { ok = 0; atomicOr(p.err, ERR_BAD_SEAM); }
    }
    for (int s = S - 1; ok && !gw && s >= 0; --s) {
      jb[s] = j;
      const int c = j / OWC;
      if (c < 0 || c >= cs) { ok = 0; atomicOr(p.err, ERR_BAD_SEAM); break; }
      const uint8_t *ra = CL ? cg::this_cluster().map_shared_rank(ancT, c) : ancT;
      j = j + (int)ra[(size_t)s * OWC + (j - c * OWC)] - 128;
      if (j < 0 || j >= W) { ok = 0; atomicOr(p.err, ERR_BAD_SEAM); }
    }
    jb[S] = j;          // the seam's column in the added row above row 0
    misc[0] = ok;
    best_m = (uint32_t)(best >> 32);
    misc[1] = 0;   // the fills add their path costs here
    if (ok && p.cost) *p.cost = (int64_t)(best >> 32);
  }
  group_sync<CL>();

  // ---- parallel backtrack: each super-tile recomputed in a FILLW-column window ----
  const int *jb0 = CL ? cg::this_cluster().map_shared_rank(jb, 0) : jb;
  const int *misc0 = CL ? cg::this_cluster().map_shared_rank(misc, 0) : misc;
  const int ok = misc0[0];
  if (ok && warp < G::FW) {
    const FillCtx f{p.E, smem + plan.fill, const_cast<uint32_t *>(reinterpret_cast<const uint32_t *>(misc0 + 1)), 1u,
                    p.seam, p.seam_log, p.err, pstride, p.pitch_e, H, W, Wa};
    // the one-CTA batched kernel calls the fill as a function of its own (the same call in the
    // cluster batched kernel was slower, so that one stays inline)
    if constexpr (!CL && !FWD) backtrack_fill_call<G, FWD, KSS, DIRECT>(f, jb0, S, cs, rank, warp, lane);
    else backtrack_fill<G, FWD, KSS, DIRECT>(f, jb0, S, cs, rank, warp, lane);
  }
  group_sync<CL>();   // rank 0's shared memory is read above; the seam is complete after this
  // the recomputed path costs must add up to the argmin's
  if (rank == 0 && threadIdx.x == 0 && ok && (uint32_t)misc[1] != best_m) atomicOr(p.err, ERR_COST_MISMATCH);
}

}  // namespace sc
