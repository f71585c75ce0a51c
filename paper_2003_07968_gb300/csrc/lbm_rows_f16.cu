// lbm_rows_f16.cu -- instances of the row kernels: FP16 storage.
#include "lbm_rows.cuh"

namespace pplbm {

cudaError_t resident_f16(int mrt, const ResArgs* m, const LatDev* lat0, int grid,
                         cudaStream_t st, int* occ) {
    return resident_any<StoreF16>(mrt, m, lat0, grid, st, occ);
}

cudaError_t rows_f16(int mrt, const StepArgs& a, const LatDev* lat0, cudaStream_t st) {
    return rows_any<StoreF16>(mrt, a, lat0, st);
}

}  // namespace pplbm
