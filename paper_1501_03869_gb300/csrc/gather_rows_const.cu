// gather_rows_const.cu -- instantiations of the batched gather (gather_rows.cuh) with
// constant-speed delays computed in the kernel (the conventional back projection): mode 1.
#include "gather_rows.cuh"

namespace patbp {

cudaError_t rows_dispatch_1(const GatherConfig& c, int fmt, const StreamParams* p, size_t smem, int grid,
                            cudaStream_t st, int* resident, const void** func) {
  return rows_dispatch_t<1>(c, fmt, p, smem, grid, st, resident, func);
}

}  // namespace patbp
