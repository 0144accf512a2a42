// gather_rows_wgt.cu -- instantiations of the batched gather (gather_rows.cuh) with
// stored delays and solid-angle weights (the exact back projection): mode 2.
#include "gather_rows.cuh"

namespace patbp {

cudaError_t rows_dispatch_2(const GatherConfig& c, int fmt, const StreamParams* p, size_t smem, int grid,
                            cudaStream_t st, int* resident, const void** func) {
  return rows_dispatch_t<2>(c, fmt, p, smem, grid, st, resident, func);
}

}  // namespace patbp
