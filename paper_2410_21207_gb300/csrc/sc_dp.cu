// One seam search per launch (the per-seam path of the carve and sc_find_seam): maps of at least
// TWO_MIN_ROWS rows from both ends by two thread-block clusters (k_dp_two), shorter ones by one cluster
// (k_dp, seam_search in sc_search.cuh).
#include <atomic>

#include <cudaTypedefs.h>

#include "sc_two.cuh"

namespace sc {

// The search of one map is a chain of H dependent rows, so its shape is chosen for latency: tall
// 32-row tiles cross a tile boundary (strip exchange, barrier, bookkeeping) half as often
// as 16-row ones, at the price of more redundant halo columns, which only costs idle SMs. Shapes
// in order of preference; the first whose cluster covers W is used.
struct DpShapeDef {
  int nw, kt, ow;
};
constexpr DpShapeDef kDpShapes[] = {
    {4, 32, Geo<4, 32, true>::OWC}, {8, 32, Geo<8, 32, true>::OWC}, {8, 16, Geo<8, 16, true>::OWC}};

DpShape dp_shape_for(int W) {
  DpShape s{};
  for (const DpShapeDef &d : kDpShapes) {
    s.nw = d.nw;
    s.kt = d.kt;
    s.ow = d.ow;
    s.cs = (W + d.ow - 1) / d.ow;
    if (s.cs < 1) s.cs = 1;
    if (s.cs <= MAX_CLUSTER) break;
  }
  return s;
}

// Super-tile height: KS (32) rows for the 4-warp shape, whose ancestor chain is local and whose serial
// backtrack fill halves against 64; KS_WIDE (64) for the wide shapes, whose ancestor tables would not
// fit shared memory, and for the one-ended forward search, whose chain hops cross CTAs.
template <int NW, int KT, bool FWD>
__host__ __device__ constexpr int dp_super_rows() { return (NW == 4 && KT == 32 && !FWD) ? KS : KS_WIDE; }

template <int NW, int KT, bool FWD = false, bool DIRECT = false>
__global__ void __launch_bounds__(Geo<NW, KT, true>::THREADS, 1)
    k_dp(DpArgs p, const __grid_constant__ CUtensorMap tmap) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int KSS = dp_super_rows<NW, KT, FWD>();
  const int S = (p.H + KSS - 1) / KSS;
  search_init(smem, search_plan<NW, KT, true, FILL_WARPS_MAX, FWD, KSS, DIRECT, true>(S));
  // neighbours push into each other's halo buffers: every CTA's barriers must be initialised first
  cg::this_cluster().sync();
  // the set-up above overlaps the previous kernel of the seam loop; its results are read below
  pdl_wait_prerequisites();
  // only now: the refresh that depends on this launch reads what its predecessors wrote before it waits
  pdl_launch_dependents();
  SearchArgs a;
  a.E = p.E;
  a.pitch_e = p.pitch_e;
  a.H = p.H;
  a.W = p.W;
  a.seam = p.seam;
  a.seam_log = p.seam_log;
  a.cost = p.cost;
  a.err = p.err;
  a.gated = !DIRECT && (p.gate != nullptr) && (*p.gate & ERR_ENERGY_RANGE);
  a.gate = p.gate;
  a.pstride = p.pstride;
  a.tmap = &tmap;
  a.x0 = DIRECT ? 0 : E_PADL;
  a.plane_rows = FWD ? (int)(p.pstride / p.pitch_e) : 0;
  SearchState st;
  seam_search<NW, KT, true, FILL_WARPS_MAX, FWD, KSS, DIRECT, true>(a, smem, S, st);
}

// one or two clusters of cs CTAs; a programmatic dependent (may start before its predecessor ends)
template <typename... KArgs, typename... Args>
static cudaError_t launch_dp_cluster(void (*kernel)(KArgs...), int grid, int cs, int threads, size_t smem,
                                     cudaStream_t st, const Args &...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// The driver's encoder is looked up once.
cudaError_t energy_tensor_map(CUtensorMap *m, const uint16_t *base, int pitch, int rows, int BW, int KT) {
  static std::atomic<PFN_cuTensorMapEncodeTiled_v12000> encode{nullptr};
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode.load();
  if (!fn) {
    void *ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess) return e;
    if (q != cudaDriverEntryPointSuccess || !ptr) return cudaErrorNotSupported;
    fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
    encode.store(fn);
  }
  const cuuint64_t dims[2] = {(cuuint64_t)pitch, (cuuint64_t)rows}, strides[1] = {(cuuint64_t)pitch * 2};
  const cuuint32_t box[2] = {(cuuint32_t)tensor_box_cols(BW), (cuuint32_t)KT}, es[2] = {1, 1};
  const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, const_cast<uint16_t *>(base), dims, strides, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int NW, int KT, bool FWD = false, bool DIRECT = false>
static cudaError_t launch_dp_shape(const DpArgs &a, int cs, cudaStream_t st) {
  constexpr int KSS = dp_super_rows<NW, KT, FWD>();
  const size_t smem = search_plan<NW, KT, true, FILL_WARPS_MAX, FWD, KSS, DIRECT, true>((a.H + KSS - 1) / KSS).total;
  static bool configured = false;
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(k_dp<NW, KT, FWD, DIRECT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_dp<NW, KT, FWD, DIRECT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  if (smem > 232448) return cudaErrorInvalidValue;
  CUtensorMap tmap;
  const int rows = a.H + (FWD ? (int)(2 * a.pstride / a.pitch_e) : 0);   // the three planes in a row
  const cudaError_t e = energy_tensor_map(&tmap, DIRECT ? a.E : a.E - E_PADL, a.pitch_e, rows, Geo<NW, KT, true>::BW, KT);
  if (e != cudaSuccess) return e;
  return launch_dp_cluster(k_dp<NW, KT, FWD, DIRECT>, cs, cs, Geo<NW, KT, true>::THREADS, smem, st, a, tmap);
}

// ---- the two-ended search ----
// The search of one map is a chain of dependent rows. The seam is the leftmost of all optimal paths
// (the pointwise minimum of two optimal paths is again an optimal path: where they cross without
// sharing a cell they can be exchanged), which does not depend on the direction it is computed from.
// So one cluster sweeps the upper half downwards from row 0 and a second one the lower half upwards
// from the bottom row (the same sweep with a negative row pitch), and the chain is half as long:
//   * with D(j) the cost of the best path from row 0 to column j of the upper half's last row and
//     U(j) that from the bottom row to column j of the row below it, the seam costs the minimum of
//     D(j) + min(U(j-1), U(j), U(j+1)); its columns in those two rows are the leftmost j and the
//     leftmost of the three that reach it;
//   * each half's ancestors give the seam's columns at its super-tile boundaries, towards the top and
//     towards the bottom: two chains that one warp follows side by side, half as many hops each;
//   * the super-tiles of both halves are then backtracked in parallel as in seam_search.
// No cluster waits for the other: both leave their last cost row and their ancestor table in
// global memory and every CTA counts itself in. The last CTA to arrive joins the halves and follows the
// chains on its own (a second pass over 2 x 4 bytes a column is cheaper than the cluster barriers
// that would split it), then hands the columns to its cluster, which backtracks while the other
// cluster leaves. (The two need not be resident together, so the launch cannot deadlock beside
// other work.)
// The cost self-check needs no barrier either: a launch adds its cost to sync[1] and the super-tiles
// subtract their path costs, so the word is 0 when the launch is over. The next launch looks before it
// adds, and takes what it finds away (no launch's difference can cancel another's); sc_check looks after the last.
// (Super-tiles that count themselves, the last one comparing, cost 0.45 us a seam at 1920x1080; a returning
// addition on the way to the fills 0.4 us.)
//
// Scratch, in p.scratch: the two cost rows (gw uint32 each), then the ancestor tables (gw bytes per
// super-tile, upper half first), gw = the columns the cluster covers. It fits (S + 1) rows of pitch_e
// words, S = ceil(H / 32), for H >= 64: 8 gw + (S + 1) gw <= 4 (S + 1) pitch_e.
//
// Bound by latency: the chain of H / 2 rows, then the hand-over, chains and fill. Against the one-ended
// search, both with the kernels of that time: 1920x1080 carve 24.5 -> 17.7 ms, 3840x2160 carve 183.9 -> 106.8 ms,
// 1279x853 -> 1021x701 18.5 -> 13.5 ms. The hand-over costs a few microseconds, so short maps keep the
// one-ended search: one launch takes 16.5 / 16.6 us (two-ended / one-ended) at 128 rows, 18.5 / 17.2 at
// 160, 18.5 / 18.7 at 192, 18.7 / 20.8 at 256, 22.8 / 28.9 at 512 (1000 columns; the same line at 64 to
// 3840 columns).
constexpr int TWO_MIN_ROWS = 192;

template <int NW, int KT, bool FWD>
struct Two {
  static constexpr int KSS = FWD ? KS : dp_super_rows<NW, KT, false>();
  using G = Geo<NW, KT, true, FILL_WARPS_MAX, KSS>;
  static __host__ __device__ TwoPlan plan(const TwoSplit &s, int cs) {
    const size_t tab = (size_t)(s.S0 + s.S1) * cs * G::OWC;
    return two_plan<G, NW, KT, KSS, FWD>(s.S0 + s.S1, cs, tab, SEARCH_SMEM_LIMIT);
  }
};

template <int NW, int KT, bool DIRECT, bool FWD>
__global__ void __launch_bounds__(Geo<NW, KT, true>::THREADS, 1)
    k_dp_two(DpArgs p, const __grid_constant__ CUtensorMap tmap) {
  extern __shared__ __align__(128) unsigned char smem[];
  using T = Two<NW, KT, FWD>;
  using G = typename T::G;
  constexpr int KSS = T::KSS;
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int half = (int)blockIdx.x / cs;
  const TwoSplit g = two_split<KT, KSS>(p.H);
  const TwoPlan t = T::plan(g, cs);
  const int gw = cs * G::OWC;
  int *misc = reinterpret_cast<int *>(smem + t.plan.misc);
  search_init(smem, t.plan);
  if (threadIdx.x == 0) {
    mbar_init(reinterpret_cast<uint64_t *>(smem + t.tbar), 1);
    fence_mbar_init();
    misc[0] = misc[1] = 0;
    prefetch_tensormap(&tmap);
  }
  // neighbours push into each other's halo buffers: every CTA's barriers must be initialised first
  cl.sync();
  // the set-up above overlaps the previous kernel of the seam loop; its results are read below
  pdl_wait_prerequisites();
  // only now: the refresh that depends on this launch reads what its predecessors wrote before it waits
  pdl_launch_dependents();
  if (!DIRECT && p.gate && (*p.gate & ERR_ENERGY_RANGE)) return;   // left to the wide-cost search
  TwoScratch x(p.scratch, gw);
  if (FWD) {
    x.dl = p.E + p.pstride + (ptrdiff_t)g.H0 * p.pitch_e;
    x.dr = p.E + 2 * p.pstride + (ptrdiff_t)g.H0 * p.pitch_e;
  }
  {
    SearchArgs a;
    a.E = p.E;
    a.pitch_e = p.pitch_e;
    a.H = half ? g.H1 : g.H0;
    a.W = p.W;
    a.err = p.err;
    a.gated = false;
    a.pstride = FWD ? p.pstride : 0;
    a.plane_rows = FWD ? (int)(p.pstride / p.pitch_e) : 0;
    a.gtab = x.tab + (half ? (size_t)g.S0 * gw : 0);
    a.gw = gw;
    a.endrow = half ? x.end1 : x.end0;
    a.tmap = &tmap;
    a.x0 = DIRECT ? 0 : E_PADL;
    a.y0 = half ? p.H - 1 : 0;
    a.gmax = reinterpret_cast<uint32_t *>(p.sync + 2);
    SearchState st;
    if (half) seam_sweep<NW, KT, true, FILL_WARPS_MAX, FWD, KSS, DIRECT, true, true, true>(a, smem, t.plan, st);
    else seam_sweep<NW, KT, true, FILL_WARPS_MAX, FWD, KSS, DIRECT, true, true, false>(a, smem, t.plan, st);
  }
  // ---- count this CTA in; the last one joins the halves ----
  fence_proxy_async_global();   // the tables are read by a bulk copy
  __syncthreads();
  if (threadIdx.x == 0 && atomic_add_acq_rel(p.sync, 1) == 2 * cs - 1) {
    *p.sync = 0;   // for the next launch
    misc[0] = 1;
    if (DIRECT) {
      // the 24-bit keys hold the seam sums only while H * max(e) < 2^24; otherwise this result is void and
      // the wide-cost search, launched next, takes the map
      const uint32_t e = (uint32_t)__ldcg(p.sync + 2);
      p.sync[2] = 0;
      if ((uint64_t)e * (uint64_t)p.H >= ((uint64_t)1 << 24)) {
        misc[0] = 0;
        if (p.gate) atomicOr(p.gate, ERR_ENERGY_RANGE);
      }
    }
  }
  __syncthreads();
  if (misc[0]) {
    // what the launch before left in the cost word (0), read by a thread that the chains do not wait for
    const uint32_t left = threadIdx.x == NW * 32 ? (uint32_t)__ldcg(p.sync + 1) : 0u;
    const uint32_t cost = two_join<NW, FWD>(g, x, gw, p.W, smem, t, 0u, cs, p.err);
    if (threadIdx.x == 0 && cost != SENT) {
      if (p.cost) *p.cost = (int64_t)cost;
      atomicAdd(reinterpret_cast<uint32_t *>(p.sync + 1), cost - (FWD ? (uint32_t)misc[3] : 0u));
    }
    if (left != 0u) {
      atomicSub(reinterpret_cast<uint32_t *>(p.sync + 1), left);
      atomicOr(p.err, ERR_COST_MISMATCH);
    }
  }
  cl.sync();
  if (misc[1] == 0) return;   // the other cluster goes on (or a recorded failure)
  const FillCtx f{p.E, nullptr, reinterpret_cast<uint32_t *>(p.sync + 1), 0xFFFFFFFFu, p.seam, p.seam_log, p.err,
                  FWD ? p.pstride : 0, p.pitch_e, 0, p.W, (p.W + 7) & ~7};
  two_fill<G, KSS, DIRECT, FWD>(g, f, p.H, t, smem, cs, rank);
}

template <int NW, int KT, bool DIRECT, bool FWD = false>
static cudaError_t launch_dp_two(const DpArgs &a, int cs, cudaStream_t st) {
  const size_t smem = Two<NW, KT, FWD>::plan(two_split<KT, Two<NW, KT, FWD>::KSS>(a.H), cs).plan.total;
  static bool configured = false;
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(k_dp_two<NW, KT, DIRECT, FWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_dp_two<NW, KT, DIRECT, FWD>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  if (smem > SEARCH_SMEM_LIMIT) return cudaErrorInvalidValue;
  CUtensorMap tmap;
  const int rows = a.H + (FWD ? (int)(2 * a.pstride / a.pitch_e) : 0);   // the three planes in a row
  const cudaError_t e = energy_tensor_map(&tmap, DIRECT ? a.E : a.E - E_PADL, a.pitch_e, rows, Geo<NW, KT, true>::BW, KT);
  if (e != cudaSuccess) return e;
  return launch_dp_cluster(k_dp_two<NW, KT, DIRECT, FWD>, 2 * cs, cs, Geo<NW, KT, true>::THREADS, smem, st, a, tmap);
}

template <bool DIRECT>
static cudaError_t launch_dp_e1(const DpArgs &a, const DpShape &s, cudaStream_t st) {
  if (a.H >= TWO_MIN_ROWS) {
    if (s.nw == 4 && s.kt == 32) return launch_dp_two<4, 32, DIRECT>(a, s.cs, st);
    if (s.nw == 8 && s.kt == 32) return launch_dp_two<8, 32, DIRECT>(a, s.cs, st);
    return launch_dp_two<8, 16, DIRECT>(a, s.cs, st);
  }
  if (s.nw == 4 && s.kt == 32) return launch_dp_shape<4, 32, false, DIRECT>(a, s.cs, st);
  if (s.nw == 8 && s.kt == 32) return launch_dp_shape<8, 32, false, DIRECT>(a, s.cs, st);
  return launch_dp_shape<8, 16, false, DIRECT>(a, s.cs, st);
}

// forward energy stages three planes per row: one shape, 4 warps x 16-row tiles (W <= 4096)
int dp_forward_max_width() { return MAX_CLUSTER * Geo<4, 16, true>::OWC; }

cudaError_t launch_dp(const DpArgs &a, cudaStream_t st) {
  if (a.pstride > 0) {
    const int cs = (a.W + Geo<4, 16, true>::OWC - 1) / Geo<4, 16, true>::OWC;
    if (cs > MAX_CLUSTER) return cudaErrorInvalidValue;
    if (a.H >= TWO_MIN_ROWS) return launch_dp_two<4, 16, false, true>(a, cs, st);
    return launch_dp_shape<4, 16, true>(a, cs < 1 ? 1 : cs, st);
  }
  const DpShape s = dp_shape_for(a.W);
  if (s.cs > MAX_CLUSTER) return cudaErrorInvalidValue;
  return a.direct ? launch_dp_e1<true>(a, s, st) : launch_dp_e1<false>(a, s, st);
}

}  // namespace sc
