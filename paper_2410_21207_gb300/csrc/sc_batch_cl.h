// Batched persistent carving with one thread-block cluster per image.
#pragma once
#include "sc_batch_item.h"

namespace sc {

constexpr size_t BATCH_CL_SMEM_MAX = 232448 - 1024;   // the opt-in limit minus static shared memory

// Cluster shapes of the persistent kernel:
//   CL_WIDE:   8 compute warps, 8-row tiles, 768 own columns per CTA. Images wider than one CTA of the
//              one-CTA kernel: few CTAs per image, little redundant halo work (throughput).
//   CL_LAT:    8 compute warps, 16-row tiles, 640 own columns per CTA, two-ended: one half of the
//              cluster's CTAs sweeps the upper half of the map, the other the lower half: half the chain of
//              dependent rows per seam, so one image's seams finish sooner (latency), at more SM
//              time per seam. The serving form's wide and heavy requests, and a plan's heaviest images.
//   CL_LAT_12: the same of 12 warps, 1,024 own columns per CTA: a plan's heaviest images on fewer CTAs
//              (batch_lat_ctas), at the widths that those do not cover with 8 warps.
// At the map's two edges a CTA owns its halo as well: p CTAs a half cover p own + 128 columns.
enum ClShape { CL_WIDE = 0, CL_LAT = 1, CL_LAT_12 = 2 };

struct ClOps {
  int own;                                                     // columns each CTA of a cluster owns
  int parts;                                                   // parts of the map a cluster sweeps at once (1 or 2)
  int edges;                                                   // columns that the CTAs at the map's edges own besides
  int tile_rows, staged;                                       // rows and columns of a staged tile (0: no tensor map)
  size_t (*smem)(int Smax);                                    // dynamic shared memory per CTA
  cudaError_t (*capacity)(int cs, int Smax, int *clusters);    // clusters of cs CTAs resident at once
  // `clusters` persistent clusters of cs CTAs carve items[0..n) (a queue counter at *queue, zeroed);
  // every CTA triggers its programmatic dependents at its start; pdl: launched as a programmatic
  // dependent of the launch before it on st, and does not end before that launch does
  cudaError_t (*launch)(const BatchItem *items, int n, int cs, int Smax, int clusters, int *queue, int *err,
                        cudaStream_t st, bool pdl);
};

ClOps cl_ops_wide();
ClOps cl_ops_lat();
ClOps cl_ops_lat12();
inline ClOps cl_ops(int shape) {
  return shape == CL_LAT ? cl_ops_lat() : (shape == CL_LAT_12 ? cl_ops_lat12() : cl_ops_wide());
}

// the columns that a cluster of ctas CTAs covers (of an odd number that sweep in two halves, one only helps
// with the rows)
inline int batch_cl_cols(int ctas, int shape) {
  const ClOps o = cl_ops(shape);
  return ctas / o.parts * o.own + o.edges;
}
// CTAs of a cluster for an image of searched width w
inline int batch_cl_ctas(int w, int shape = CL_WIDE) {
  const ClOps o = cl_ops(shape);
  return o.parts * ((w + o.own - 1) / o.own);
}
// CTAs of the smaller cluster for an image of searched width w that would hold up its batch on one CTA, and the
// shape that covers it with so many
inline int batch_lat_ctas(int w) { return w > 768 ? (w + 383) / 384 : 2; }
inline int batch_lat_shape(int w) { return batch_cl_cols(batch_lat_ctas(w), CL_LAT) >= w ? CL_LAT : CL_LAT_12; }
inline size_t batch_cl_smem_bytes(int Smax, int shape = CL_WIDE) { return cl_ops(shape).smem(Smax); }
inline cudaError_t batch_cl_capacity(int cs, int Smax, int *clusters, int shape = CL_WIDE) {
  return cl_ops(shape).capacity(cs, Smax, clusters);
}
inline cudaError_t launch_batch_cl(const BatchItem *items, int n, int cs, int Smax, int clusters, int *queue, int *err,
                                   cudaStream_t st, int shape = CL_WIDE, bool pdl = false) {
  return cl_ops(shape).launch(items, n, cs, Smax, clusters, queue, err, st, pdl);
}

}  // namespace sc
