// Marching sweep, FP32, one step per pass: 12 warps per SM (168 registers).
#include "qla_march.cuh"

namespace qla {
cudaError_t launch_march_f32_k1(const MarchArgs &a, int nfam, int interleaved, int mode, cudaStream_t st) {
    return launch_march_modes<float, 4, 1, 2, 2, 4, 3, true>(a, nfam, interleaved, mode, st);
}
}  // namespace qla
