// The fused sweep with rotations in the form for any angle (MODE_WIDE): media with
// indices far below 1 whose coefficients lie in pair planes, one step per pass.
#include "qla_sweep.cuh"

namespace qla {

cudaError_t launch_sweep_wide_f32(int K, const SweepArgs &a, int nfam, cudaStream_t st) {
    // (with the printed potentials FP32 collisions are shears, whatever the angle)
    if (K != 1 || !(a.mode & MODE_UNITARY)) return cudaErrorInvalidValue;
    return a.interleaved ? launch_sweep_t<float, 1, 8, 1, true, MODE_UNITARY | MODE_WIDE>(a, nfam, st)
                         : launch_sweep_t<float, 1, 8, 1, false, MODE_UNITARY | MODE_WIDE>(a, nfam, st);
}

cudaError_t launch_sweep_wide_f64(int K, const SweepArgs &a, int nfam, cudaStream_t st) {
    if (K != 1) return cudaErrorInvalidValue;
    return launch_sweep_modes<double, 1, 4, 1, MODE_WIDE>(a, nfam, st);
}

}  // namespace qla
