// lbm_rows_f32.cu -- instances of the row kernels: FP32 storage.
#include "lbm_rows.cuh"

namespace pplbm {

cudaError_t resident_f32(int mrt, const ResArgs* m, const LatDev* lat0, int grid,
                         cudaStream_t st, int* occ) {
    return resident_any<StoreF32>(mrt, m, lat0, grid, st, occ);
}

cudaError_t rows_f32(int mrt, const StepArgs& a, const LatDev* lat0, cudaStream_t st) {
    return rows_any<StoreF32>(mrt, a, lat0, st);
}

cudaError_t pairs_f32(int mrt, const StepArgs& a, const LatDev* lat0, cudaStream_t st) {
    if (mrt) return lat0 ? pairs_inst<true, true>(a, lat0, st) : pairs_inst<true, false>(a, lat0, st);
    return lat0 ? pairs_inst<false, true>(a, lat0, st) : pairs_inst<false, false>(a, lat0, st);
}

}  // namespace pplbm
