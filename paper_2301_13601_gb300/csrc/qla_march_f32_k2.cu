// Marching sweep, FP32, two steps per pass: 8 warps per SM (255 registers).
#include "qla_march.cuh"

namespace qla {
cudaError_t launch_march_f32_k2(const MarchArgs &a, int nfam, int interleaved, int mode, cudaStream_t st) {
    return launch_march_modes<float, 4, 2, 3, 4, 4, 2, true>(a, nfam, interleaved, mode, st);
}
}  // namespace qla
