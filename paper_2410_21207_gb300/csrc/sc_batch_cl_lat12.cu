// The CL_LAT_12 shape of the cluster-per-image persistent kernel (sc_batch_cl.cuh): 12 compute warps,
// 16-row tiles, two-ended.
#include "sc_batch_cl.cuh"

namespace sc {

ClOps cl_ops_lat12() { return ClShapeHost<12, 16, 7, true>::ops(); }

}  // namespace sc
