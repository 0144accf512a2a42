// gather_rows_wgt_const.cu -- instantiations of the batched gather (gather_rows.cuh) with
// constant-speed delays and solid-angle weights: mode 3.
#include "gather_rows.cuh"

namespace patbp {

cudaError_t rows_dispatch_3(const GatherConfig& c, int fmt, const StreamParams* p, size_t smem, int grid,
                            cudaStream_t st, int* resident, const void** func) {
  return rows_dispatch_t<3>(c, fmt, p, smem, grid, st, resident, func);
}

}  // namespace patbp
