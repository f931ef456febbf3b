// Batched persistent carving with one thread-block cluster per image (images wider than one CTA,
// and the heaviest images of a batch), templated on the cluster's shape: compute warps NW, tile
// rows KT and backtrack-fill warps FWM; sc_batch_cl.cu, sc_batch_cl_lat.cu and sc_batch_cl_lat12.cu instantiate
// the shapes of sc_batch_cl.h.
// Each cluster repeatedly takes the next image from a queue and carves it completely, like the
// one-CTA batched kernel (sc_batch.cuh), with the cluster-wide seam search (seam_search with CL, or the
// two-ended clb_two_search)
// and the per-seam row work split over the cluster's CTAs: CTA r owns rows r, r + cs, r + 2cs, ...
// Per seam: the search (ends with a cluster barrier); every owned row's refreshed energy pair and
// pending-removal list update, one thread per row; a cluster barrier (the pairs read neighbouring
// rows' words, which the compaction below rewrites); the energy rows shifted past the seam with the
// pair written in, four per warp at a time, and every RPEND seams the image words compacted; a cluster
// barrier. Several clusters run side by side, so a batch of wide images keeps the GPU busy where
// the per-seam cluster path would run one image's latency-bound chain at a time.
#pragma once
#include <atomic>

#include "sc_batch_cl.h"
#include "sc_rowops.cuh"
#include "sc_two.cuh"

namespace sc {

// Shared-memory plan of a shape. TWO: the ancestor tables want 128 KB (up to ~1,400 rows of a
// 2,560-column image); larger ones are followed in global memory.
template <int NW, int KT, int FWM, bool TWO>
__host__ __device__ inline TwoPlan clb_plan(int Smax) {
  using G = Geo<NW, KT, true, FWM>;
  if (TWO) return two_plan<G, NW, KT, KS>(Smax + 1, 1, (size_t)128 << 10, BATCH_CL_SMEM_MAX);
  TwoPlan t{};
  t.plan = search_plan<NW, KT, true, FWM>(Smax);
  return t;
}

// The two-ended search (sc_dp.cu describes it) of one cluster: its first half of CTAs sweeps the upper
// half of the map, the second half the lower one (of an odd number the last CTA waits); rank 0 joins them,
// all of them backtrack.
template <int NW, int KT, int FWM>
__device__ __forceinline__ void clb_two_search(SearchArgs a, uint32_t *scratch, const CUtensorMap *tmap, unsigned char *smem,
                                               const TwoPlan &t, SearchState &st, int rank, int ctas) {
  using G = Geo<NW, KT, true, FWM>;
  cg::cluster_group cl = cg::this_cluster();
  const TwoSplit g = two_split<KT, KS>(a.H);
  const int cs = ctas / 2, half = rank >= cs ? 1 : 0, gw = cs * G::OWC + 2 * G::K2E, H = a.H;
  const TwoScratch x(scratch, gw);
  int *misc = reinterpret_cast<int *>(smem + t.plan.misc);
  a.gtab = x.tab + (half ? (size_t)g.S0 * gw : 0);
  a.gw = gw;
  a.endrow = half ? x.end1 : x.end0;
  a.tmap = tmap;
  a.rank0 = half * cs;
  a.ctas = cs;
  if (half) {
    a.H = g.H1;
    a.y0 = H - 1;
    if (rank < 2 * cs) seam_sweep<NW, KT, true, FWM, false, KS, false, true, true, true>(a, smem, t.plan, st);
  } else {
    a.H = g.H0;
    seam_sweep<NW, KT, true, FWM, false, KS, false, true, true, false>(a, smem, t.plan, st);
  }
  fence_proxy_async_global();   // the tables are read by a bulk copy
  cl.sync();
  uint32_t cost = SENT;
  if (rank == 0) {
    cost = two_join<NW>(g, x, gw, a.W, smem, t, st.joins & 1u, ctas, a.err);
    if ((size_t)(g.S0 + g.S1) * gw <= t.tab_cap) ++st.joins;
    if (threadIdx.x == 0 && cost != SENT && a.cost) *a.cost = (int64_t)cost;
  }
  cl.sync();
  if (misc[1]) {
    const FillCtx f{a.E, nullptr, reinterpret_cast<uint32_t *>(cl.map_shared_rank(misc, 0) + 2), 1u, a.seam, a.seam_log,
                    a.err, 0, a.pitch_e, 0, a.W, 0};
    two_fill<G, KS>(g, f, H, t, smem, ctas, rank);
  }
  cl.sync();   // the seam is complete
  // the recomputed path costs must add up to the join's
  if (rank == 0 && threadIdx.x == 0 && cost != SENT && (uint32_t)misc[2] != cost) atomicOr(a.err, ERR_COST_MISMATCH);
}

// (count) vertical seams of a rows x cols word image whose energy is in it.E
template <int NW, int KT, int FWM, bool TWO>
__device__ void clb_seam_pass(const BatchJob &it, uint32_t *words, int rows, int cols, int count, int32_t *log,
                              int64_t *costs, unsigned char *smem, int Smax, SearchState &st, int *err, int rank,
                              int cs, const CUtensorMap *tmap) {
  cg::cluster_group cl = cg::this_cluster();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  int16_t *lb[2] = {it.lists, it.lists + (size_t)rows * RPEND};
  // the staging ring is idle between searches: it holds the owned rows' refreshed pairs
  const TwoPlan tplan = clb_plan<NW, KT, FWM, TWO>(Smax);
  const SearchPlan &plan = tplan.plan;
  uint32_t *pairs = reinterpret_cast<uint32_t *>(smem + plan.ring);
  const int nq = (rows - rank + cs - 1) / cs;   // rows this CTA owns
  const size_t pair_bytes = ((size_t)(nq > 0 ? nq : 0) * 4 + 15) & ~(size_t)15;
  uint16_t *sbuf = reinterpret_cast<uint16_t *>(smem + plan.ring + pair_bytes);
  const int sbuf_elems = (int)(((plan.ring_end - plan.ring - pair_bytes) / nwarps) & ~(size_t)15) / 2;
  uint16_t *const Ecur = it.E + E_PADL;
  int cur = 0, m = 0;
  for (int t = 0; t < count; ++t) {
    const int w = cols - t;
    SearchArgs a;
    a.E = Ecur;
    a.pitch_e = it.pe;
    a.H = rows;
    a.W = w;
    a.seam = it.seam;
    a.seam_log = log ? log + (size_t)t * rows : nullptr;
    a.cost = costs ? costs + t : nullptr;
    a.err = err;
    a.gated = false;
    // the search ends with a cluster barrier
    if constexpr (TWO) clb_two_search<NW, KT, FWM>(a, it.scratch, tmap, smem, tplan, st, rank, cs);
    else seam_search<NW, KT, true, FWM>(a, smem, Smax, st);
    if (refresh_pairs(words, it.pitch, rows, w, it.seam, lb[cur], lb[cur ^ 1], m, nq, rank, cs, pairs, threadIdx.x,
                      blockDim.x))
      atomicOr(err, ERR_BAD_SEAM);
    cl.sync();
    // the owned rows' energies compacted past the seam
    shift_rows(Ecur, it.pe, nq, rank, cs, w, it.seam, pairs, warp, nwarps, lane);
    cur ^= 1;
    if (++m == RPEND) {
      compact_rows_staged(words, it.pitch, nq, rank, cs, lb[cur], m, w - 1, warp, nwarps, lane,
                          reinterpret_cast<uint32_t *>(sbuf + (size_t)warp * sbuf_elems), sbuf_elems / 2);
      m = 0;
    }
    fence_proxy_async_global();   // the next search stages the compacted energy rows with TMA
    fence_proxy_async_smem();     // ... into the ring's place, which held this seam's pairs and rows
    cl.sync();
  }
  if (m > 0) {
    compact_rows_staged(words, it.pitch, nq, rank, cs, lb[cur], m, cols - count, warp, nwarps, lane,
                        reinterpret_cast<uint32_t *>(sbuf + (size_t)warp * sbuf_elems), sbuf_elems / 2);
    cl.sync();
  }
}

// e1 energy of every owned row (the search's TMA reads it next)
__device__ inline void clb_energy(const uint32_t *words, int pitch, int rows, int cols, uint16_t *E, int pe, int rank, int cs) {
  for (int i = rank; i < rows; i += cs)
    for (int j = threadIdx.x; j < cols; j += blockDim.x)
      E[(int64_t)i * pe + j] = (uint16_t)energy_at(words, pitch, rows, cols, i, j);
  fence_proxy_async_global();
  cg::this_cluster().sync();
}

// rows x cols word image -> its transpose, 32 x 32 tiles through shared memory, tiles dealt out
// over the cluster's warps
__device__ inline void clb_transpose(const uint32_t *src, int ps, int rows, int cols, uint32_t *dst, int pd, uint32_t *tile,
                              int ntw, int rank, int cs) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < ntw) {
    uint32_t *t = tile + warp * 32 * 33;
    const int tr = (rows + 31) / 32, tc = (cols + 31) / 32;
    for (int tix = rank * ntw + warp; tix < tr * tc; tix += cs * ntw) {
      const int by = (tix / tc) * 32, bx = (tix % tc) * 32;
      for (int r = 0; r < 32; ++r) {
        const int i = by + r, j = bx + lane;
        if (i < rows && j < cols) t[r * 33 + lane] = src[(int64_t)i * ps + j];
      }
      __syncwarp();
      for (int r = 0; r < 32; ++r) {
        const int j = bx + r, i = by + lane;
        if (i < rows && j < cols) dst[(int64_t)j * pd + i] = t[lane * 33 + r];
      }
      __syncwarp();
    }
  }
  cg::this_cluster().sync();
}

template <int NW, int KT, int FWM, bool TWO>
__device__ void clb_carve_item(const BatchJob &it, unsigned char *smem, int Smax, SearchState &st, int *err, int rank,
                               int cs, const CUtensorMap *tmap) {
  // the thread that issues this image's tensor copies
  if (TWO && threadIdx.x == NW * 32) fence_tensormap_acquire(tmap);
  const int H = it.H, W = it.W, C = it.C, tw = it.tw, th = it.th;
  const int64_t tid = (int64_t)rank * blockDim.x + threadIdx.x, nth = (int64_t)cs * blockDim.x;
  const int64_t npx = (int64_t)H * W;
  for (int64_t q = tid; q < npx; q += nth) {
    const int i = (int)(q / W), j = (int)(q % W);
    it.img_w[(int64_t)i * it.pitch + j] = pack_pixel(it.img + q * C, C);
  }
  cg::this_cluster().sync();
  clb_energy(it.img_w, it.pitch, H, W, it.E + E_PADL, it.pe, rank, cs);
  const int nv = W - tw, nh = H - th;
  clb_seam_pass<NW, KT, FWM, TWO>(it, it.img_w, H, W, nv, it.seam_log, it.cost_log, smem, Smax, st, err, rank, cs, tmap);
  if (nh > 0) {
    const SearchPlan plan = clb_plan<NW, KT, FWM, TWO>(Smax).plan;
    uint32_t *tile = reinterpret_cast<uint32_t *>(smem + plan.ring);   // the ring is idle between searches
    const int ntw_fit = (int)((plan.ring_end - plan.ring) / (32 * 33 * 4));
    const int ntw = ntw_fit < NW + 1 ? ntw_fit : NW + 1;
    clb_transpose(it.img_w, it.pitch, H, tw, it.img2_w, it.pitch, tile, ntw, rank, cs);   // tw rows x H columns
    clb_energy(it.img2_w, it.pitch, tw, H, it.E + E_PADL, it.pe, rank, cs);
    clb_seam_pass<NW, KT, FWM, TWO>(it, it.img2_w, tw, H, nh, it.seam_log ? it.seam_log + (size_t)nv * H : nullptr,
                                    it.cost_log ? it.cost_log + nv : nullptr, smem, Smax, st, err, rank, cs, tmap);
    clb_transpose(it.img2_w, it.pitch, tw, th, it.img_w, it.pitch, tile, ntw, rank, cs);   // th rows x tw columns
  }
  const int64_t nout = (int64_t)th * tw;
  for (int64_t q = tid; q < nout; q += nth) {
    const int i = (int)(q / tw), j = (int)(q % tw);
    unpack_pixel(it.img_w[(int64_t)i * it.pitch + j], it.out + q * C, C);
  }
  if (it.done) __threadfence_system();   // every thread's output bytes before the completion word
  cg::this_cluster().sync();
  if (it.done && rank == 0 && threadIdx.x == 0) *(volatile int *)it.done = (*(volatile int *)err != 0) ? 2 : 1;
}

template <int NW, int KT, int FWM, bool TWO>
__global__ void __launch_bounds__(Geo<NW, KT, true, FWM>::THREADS, 1)
    k_batch_cl(const BatchItem *__restrict__ items, int n, int Smax, int *queue, int *err) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int next;
  __shared__ BatchJob cur;   // the current image's descriptor, read where its fields are used
  // a launch chained behind this one (programmatic dependent launch) may start once every CTA of
  // this launch is resident: a batch plan places its clusters before the one-CTA launch fills the
  // remaining SMs
  pdl_launch_dependents();
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), cs = (int)cl.num_blocks();
  {
    const TwoPlan t = clb_plan<NW, KT, FWM, TWO>(Smax);
    search_init(smem, t.plan);
    if (TWO && threadIdx.x == 0) {
      mbar_init(reinterpret_cast<uint64_t *>(smem + t.tbar), 1);
      fence_mbar_init();
    }
  }
  cl.sync();
  SearchState st;
  for (;;) {
    if (rank == 0 && threadIdx.x == 0) next = atomicAdd(queue, 1);
    cl.sync();
    const int k = *cl.map_shared_rank(&next, 0);
    cl.sync();   // every CTA has read rank 0's `next` before it can change or its CTA exit
    if (k >= n) break;
    if (threadIdx.x == 0) cur = items[k];
    __syncthreads();
    clb_carve_item<NW, KT, FWM, TWO>(cur, smem, Smax, st, err, rank, cs, &items[k].tmap);
  }
  // chained behind another launch: do not end before it does (no-op otherwise)
  pdl_wait_prerequisites();
}

// The host side of one shape: shared memory, capacity and launch (instantiated once per shape).
template <int NW, int KT, int FWM, bool TWO>
struct ClShapeHost {
  using G = Geo<NW, KT, true, FWM>;
  static size_t smem_bytes(int Smax) { return clb_plan<NW, KT, FWM, TWO>(Smax).plan.total; }
  static cudaError_t configure() {
    static std::atomic<bool> done{false};
    if (done.load()) return cudaSuccess;
    auto k = k_batch_cl<NW, KT, FWM, TWO>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BATCH_CL_SMEM_MAX);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    done.store(true);
    return cudaSuccess;
  }
  static void cfg_for(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *at, int clusters, int cs, int Smax, cudaStream_t st,
                      bool pdl = false) {
    cfg = {};
    cfg.gridDim = dim3(cs * clusters);
    cfg.blockDim = dim3(G::THREADS);
    cfg.dynamicSmemBytes = smem_bytes(Smax);
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cs;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 2 : 1;
  }
  static cudaError_t capacity(int cs, int Smax, int *clusters) {
    cudaError_t e = configure();
    if (e != cudaSuccess) return e;
    if (cs < 1 || cs > MAX_CLUSTER || smem_bytes(Smax) > BATCH_CL_SMEM_MAX) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[2];
    cfg_for(cfg, at, 1, cs, Smax, nullptr);
    return cudaOccupancyMaxActiveClusters(clusters, k_batch_cl<NW, KT, FWM, TWO>, &cfg);
  }
  static cudaError_t launch(const BatchItem *items, int n, int cs, int Smax, int clusters, int *queue, int *err,
                            cudaStream_t st, bool pdl) {
    cudaError_t e = configure();
    if (e != cudaSuccess) return e;
    if (cs < 1 || cs > MAX_CLUSTER || clusters < 1 || smem_bytes(Smax) > BATCH_CL_SMEM_MAX) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[2];
    cfg_for(cfg, at, clusters, cs, Smax, st, pdl);
    return cudaLaunchKernelEx(&cfg, k_batch_cl<NW, KT, FWM, TWO>, items, n, Smax, queue, err);
  }
  static ClOps ops() { return ClOps{G::OWC, TWO ? 2 : 1, TWO ? 2 * G::K2E : 0, KT, TWO ? G::BW : 0, &smem_bytes, &capacity, &launch}; }
};

}  // namespace sc
