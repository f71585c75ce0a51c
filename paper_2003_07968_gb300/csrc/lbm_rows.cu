// lbm_rows.cu -- host side of the row kernels: dispatch to the instance units
// (lbm_rows_{f32,f16}.cu; the kernels are in lbm_rows.cuh).
#include <map>
#include <mutex>
#include <tuple>

#include "lbm_kernels.h"

namespace pplbm {

cudaError_t resident_f32(int, const ResArgs*, const LatDev*, int, cudaStream_t, int*);
cudaError_t resident_f16(int, const ResArgs*, const LatDev*, int, cudaStream_t, int*);

cudaError_t rows_f32(int, const StepArgs&, const LatDev*, cudaStream_t);
cudaError_t rows_f16(int, const StepArgs&, const LatDev*, cudaStream_t);

cudaError_t launch_rows(int f16, int mrt, const StepArgs& a, const LatDev* lat0, cudaStream_t st) {
    return (f16 ? rows_f16 : rows_f32)(mrt, a, lat0, st);
}

cudaError_t pairs_f32(int, const StepArgs&, const LatDev*, cudaStream_t);

cudaError_t launch_pairs(int f16, int mrt, const StepArgs& a, const LatDev* lat0, cudaStream_t st) {
    return f16 ? cudaErrorInvalidValue : pairs_f32(mrt, a, lat0, st);
}

cudaError_t launch_resident(int f16, int mrt, const ResArgs& m, const LatDev* lat0, int grid,
                            cudaStream_t st) {
    return (f16 ? resident_f16 : resident_f32)(mrt, &m, lat0, grid, st, nullptr);
}

int resident_blocks_per_sm(int f16, int mrt, bool single) {
    // (a property of the kernel and the device: asked once)
    static std::mutex mu;
    static std::map<std::tuple<int, int, int, int>, int> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_tuple(dev, f16, mrt, (int)single);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    int occ = 0;
    const LatDev lat{};
    const cudaError_t e = (f16 ? resident_f16 : resident_f32)(mrt, nullptr, single ? &lat : nullptr,
                                                             0, nullptr, &occ);
    if (e != cudaSuccess) return 0;
    known[key] = occ;
    return occ;
}

}  // namespace pplbm
