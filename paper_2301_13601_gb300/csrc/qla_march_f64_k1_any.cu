// Marching sweep, FP64, one step per pass; rows of any length (element copies).
#include "qla_march.cuh"

namespace qla {
cudaError_t launch_march_f64_k1_any(const MarchArgs &a, int nfam, int interleaved, int mode, cudaStream_t st) {
    return launch_march_modes<double, 2, 1, 2, 2, 4, 3, false>(a, nfam, interleaved, mode, st);
}
}  // namespace qla
