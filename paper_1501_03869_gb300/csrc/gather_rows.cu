// gather_rows.cu -- instantiations of the batched gather (gather_rows.cuh) with
// delays from the stored fast-marching table: mode 0.
#include "gather_rows.cuh"

namespace patbp {

cudaError_t rows_dispatch_0(const GatherConfig& c, int fmt, const StreamParams* p, size_t smem, int grid,
                            cudaStream_t st, int* resident, const void** func) {
  return rows_dispatch_t<0>(c, fmt, p, smem, grid, st, resident, func);
}

}  // namespace patbp
