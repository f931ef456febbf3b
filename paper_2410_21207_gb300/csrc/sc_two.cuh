// Parts shared by the two forms of the two-ended seam search: the single-map search of two clusters
// (sc_dp.cu, where the method is described) and the batched one of one cluster whose CTAs split into
// halves (sc_batch_cl.cuh).
#pragma once
#include "sc_search.cuh"

namespace sc {

// rows and super-tiles of the upper and the lower half: a whole number of tiles in the upper one where
// there is a choice, so that only the lower half ends on a ragged tile (maps of at most KT rows have no
// lower half)
struct TwoSplit {
  int H0, H1, S0, S1;
};
template <int KT, int KSS>
__host__ __device__ inline TwoSplit two_split(int H) {
  TwoSplit s;
  s.H0 = ((H + 1) / 2 + KT - 1) / KT * KT;
  if (s.H0 > H) s.H0 = H;
  s.H1 = H - s.H0;
  s.S0 = (s.H0 + KSS - 1) / KSS;
  s.S1 = (s.H1 + KSS - 1) / KSS;
  return s;
}

// Shared memory of a CTA. S: super-tiles of both halves; ctas: the CTAs that share the fills; the staging
// ring's place later holds the ancestor tables (where they fit: tab_cap bytes), then the fills' rows. It
// is enlarged to want_tab bytes as far as `limit` allows.
struct TwoPlan {
  SearchPlan plan;   // cmin: warps' minima, then the super-tiles' ends; jb: both halves' columns
  size_t tbar;       // mbarrier of the tables' copy
  size_t tab_cap;
};
template <typename G, int NW, int KT, int KSS, bool FWD = false>
__host__ __device__ inline TwoPlan two_plan(int S, int ctas, size_t want_tab, size_t limit) {
  TwoPlan t;
  SearchPlan &p = t.plan;
  size_t o = 0;
  auto take = [&](size_t bytes) { const size_t at = o; o = (o + bytes + 15) & ~(size_t)15; return at; };
  p.bnd = take((size_t)2 * G::BW * 4);
  p.hbuf = take((size_t)2 * 2 * K2 * 4);
  p.cmin = take((size_t)(NW + 1 + (S + ctas - 1) / ctas) * 8);
  p.jb = take((size_t)(S + 2) * 4);
  p.misc = take(16);   // [0] this CTA arrived last (two clusters), [1] go on with the ends in cmin, [2] cost sum,
                       // [3] forward energy: the cost of the step between the halves
  p.wmin = p.anc = p.emx = p.gat = 0;
  p.gw = 0;
  p.bars = take((size_t)(NSLOT + 3) * 8);
  t.tbar = p.bars + (size_t)(NSLOT + 2) * 8;
  o = (o + 127) & ~(size_t)127;   // (tensor copies: 128-byte aligned)
  size_t r = (size_t)NSLOT * (FWD ? 3 : 1) * KT * tensor_boxes(G::BW) * tensor_box_cols(G::BW) * 2;
  const size_t fb = (size_t)G::FW * G::fill_bytes(FWD);
  r = r > fb ? r : fb;
  if (want_tab > r && o < limit) {
    const size_t room = (limit - o) & ~(size_t)127;
    const size_t w = want_tab < room ? want_tab : room;
    r = r > w ? r : w;
  }
  p.ring = p.fill = take(r);
  p.ring_end = p.total = o;
  t.tab_cap = r;
  return t;
}

// What the halves leave in global memory: their last rows' costs (gw words each), then the ancestor
// tables (gw bytes per super-tile, upper half first).
struct TwoScratch {
  uint32_t *end0, *end1;
  uint8_t *tab;
  const uint16_t *dl = nullptr, *dr = nullptr;   // forward energy: DL and DR of the lower half's first row
  __device__ TwoScratch(uint32_t *scratch, int gw)
      : end0(scratch), end1(scratch + gw), tab(reinterpret_cast<uint8_t *>(scratch + 2 * gw)) {}
};

// Joins the halves and follows both ancestor chains; every thread of one CTA (NW compute warps and the
// producer warp) calls it once both halves' scratch is visible. Hands CTA r of the `ctas` CTAs from
// cluster rank 0 on the ends (column above, column at the bottom) of super-tiles r, r + ctas, ... (the
// upper half's first) in its cmin, and in its misc[1] whether to go on. tphase: parity of this use of the
// tables' barrier. Returns to thread 0 the seam's cost (SENT after a recorded failure).
template <int NW, bool FWD = false>
__device__ __forceinline__ uint32_t two_join(const TwoSplit &g, const TwoScratch &x, int gw, int W, unsigned char *smem,
                                             const TwoPlan &t, uint32_t tphase, int ctas, int *err) {
  cg::cluster_group cl = cg::this_cluster();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int *jb = reinterpret_cast<int *>(smem + t.plan.jb);
  int *misc = reinterpret_cast<int *>(smem + t.plan.misc);
  uint2 *const cmin = reinterpret_cast<uint2 *>(smem + t.plan.cmin);
  uint64_t *tbar = reinterpret_cast<uint64_t *>(smem + t.tbar);
  unsigned char *const stab = smem + t.plan.ring;
  const size_t tab_bytes = (size_t)(g.S0 + g.S1) * gw;
  const bool tab_smem = tab_bytes <= t.tab_cap;
  if (warp == NW && tab_smem) {
    // both ancestor tables arrive meanwhile, in a few large copies
    fence_proxy_async_global();
    fence_proxy_async_smem();   // the ring's last reads come first
    if (lane == 0) mbar_arrive_expect_tx(tbar, (uint32_t)tab_bytes);
    __syncwarp();
    constexpr uint32_t PIECE = 8192;
    for (uint32_t o = lane * PIECE; o < (uint32_t)tab_bytes; o += 32 * PIECE)
      bulk_g2s(stab + o, x.tab + o, min(PIECE, (uint32_t)tab_bytes - o), tbar);
  }
  // the cheapest join: cost; upper column << 2 | step to the lower column
  uint32_t best = SENT, where = SENT;
#pragma unroll 4
  for (int q = threadIdx.x; q < (W + 3) / 4; q += (NW + 1) * 32) {
    const int j0 = 4 * q;
    const uint4 d = __ldcg(reinterpret_cast<const uint4 *>(x.end0) + q);
    uint4 u = make_uint4(0u, 0u, 0u, 0u);
    uint32_t ul = SENT, ur = SENT;
    if (g.H1 > 0) {
      u = __ldcg(reinterpret_cast<const uint4 *>(x.end1) + q);
      if (j0 > 0) ul = __ldcg(x.end1 + j0 - 1);
      if (j0 + 4 < W) ur = __ldcg(x.end1 + j0 + 4);
    }
    const uint32_t dv[4] = {d.x, d.y, d.z, d.w}, uv[6] = {ul, u.x, u.y, u.z, u.w, ur};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int j = j0 + c;
      uint32_t left = uv[c], right = j + 1 < W ? uv[c + 2] : SENT;
      if (FWD && g.H1 > 0) {   // stepping to column j - 1 costs that cell's DR, to column j + 1 its DL
        if (j > 0) left += (uint32_t)__ldcg(x.dr + j - 1);
        if (j + 1 < W) right += (uint32_t)__ldcg(x.dl + j + 1);
      }
      const uint32_t m = min3u(left, uv[c + 1], right), sum = dv[c] + m;
      if (j < W && sum < best) {   // columns come in ascending order: ties keep the left one
        best = sum;
        where = ((uint32_t)j << 2) | (m == left ? 0u : (m == uv[c + 1] ? 1u : 2u));
      }
    }
  }
  const uint32_t wb = __reduce_min_sync(0xffffffffu, best);
  const uint32_t ww = __reduce_min_sync(0xffffffffu, best == wb ? where : SENT);
  if (lane == 0) cmin[warp] = make_uint2(wb, ww);
  __syncthreads();
  if (warp != 0) return SENT;
  const uint2 v = lane <= NW ? cmin[lane] : make_uint2(SENT, SENT);
  best = __reduce_min_sync(0xffffffffu, v.x);
  where = __reduce_min_sync(0xffffffffu, v.x == best ? v.y : SENT);
  // ancestor chains: lane 0 towards the top, lane 1 towards the bottom
  bool bad = false;
  if (tab_smem && !mbar_wait_bounded(tbar, tphase, WAIT_TIMEOUT_NS)) {
    if (lane == 0) atomicOr(err, ERR_TIMEOUT);
    bad = true;
  }
  if (lane < 2) {
    const int Sh = lane ? g.S1 : g.S0;
    int *jh = jb + (lane ? g.S0 + 1 : 0);
    int j = (int)(where >> 2) + (lane && Sh > 0 ? (int)(where & 3u) - 1 : 0);
    // a column outside the map is clamped (every read stays inside the table) and recorded
    auto keep = [&](int c) { bad |= (unsigned)c >= (unsigned)W; return min(max(c, 0), W - 1); };
    j = keep(j);
    size_t at = (size_t)(Sh - 1 + (lane ? g.S0 : 0)) * gw;
    for (int s = Sh - 1; s >= 0; --s, at -= gw) {
      jh[s] = j;
      j = keep(j + (tab_smem ? (int)stab[at + j] : (int)__ldcg(x.tab + at + j)) - 128);
    }
    jh[Sh] = j;
    if (bad) atomicOr(err, ERR_BAD_SEAM);
  }
  bad = __any_sync(0xffffffffu, bad);
  if (lane == 0) {
    misc[2] = 0;
    if (FWD) {
      // the step between the halves belongs to no super-tile
      const int j = (int)(where >> 2), d = (int)(where & 3u);
      misc[3] = (bad || g.H1 == 0 || d == 1) ? 0 : (int)__ldcg(d == 0 ? x.dr + j - 1 : x.dl + j + 1);
    }
  }
  __syncwarp();
  for (int r = lane; r < ctas; r += 32) {
    int2 *dst = reinterpret_cast<int2 *>(cl.map_shared_rank(smem + t.plan.cmin, r));
    for (int q = r; q < g.S0 + g.S1; q += ctas) {
      const int *jh = q < g.S0 ? jb : jb + g.S0 + 1;
      const int s = q < g.S0 ? q : q - g.S0, Sh = q < g.S0 ? g.S0 : g.S1;
      *dst++ = make_int2(s > 0 ? jh[s - 1] : jh[Sh], jh[s]);
    }
    cl.map_shared_rank(misc, r)[1] = bad ? 0 : 1;
  }
  return bad ? SENT : best;
}

// The calling CTA's share of the super-tiles of both halves of an H-row map (rank r of `ctas`), from the
// ends two_join left in its cmin.
template <typename G, int KSS, bool DIRECT = false, bool FWD = false>
__device__ __forceinline__ void two_fill(const TwoSplit &g, FillCtx f, int H, const TwoPlan &t, unsigned char *smem,
                                         int ctas, int rank) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp >= G::FW) return;
  const int2 *const ends = reinterpret_cast<const int2 *>(smem + t.plan.cmin);
  f.fill = smem + t.plan.fill;
  const FillCtx up = f;
  FillCtx dn = f;   // the lower half: rows counted from the bottom
  dn.E = f.E + (ptrdiff_t)(H - 1) * f.pitch_e;
  dn.pitch_e = -f.pitch_e;
  dn.seam = f.seam + (H - 1);
  dn.seam_log = f.seam_log ? f.seam_log + (H - 1) : nullptr;
  dn.step = -1;
#pragma unroll 1
  for (int k = warp; k * ctas + rank < g.S0 + g.S1; k += G::FW) {
    const int q = k * ctas + rank;
    const bool low = q >= g.S0;
    FillCtx c = low ? dn : up;
    c.H = low ? g.H1 : g.H0;
    if (FWD && low) fill_super_tile<G, FWD, KSS, DIRECT, true>(c, q - g.S0, ends[k].x, ends[k].y, warp, lane);
    else fill_super_tile<G, FWD, KSS, DIRECT>(c, low ? q - g.S0 : q, ends[k].x, ends[k].y, warp, lane);
  }
}

}  // namespace sc
