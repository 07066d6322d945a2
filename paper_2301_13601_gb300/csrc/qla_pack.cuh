// Packing of convolution weights into the tensor cores' operand layout.
#pragma once

#include <cuda_bf16.h>

#include "qla_internal.h"

namespace qla {

// ---------------------------------------------------------------------------
// Weight packing: FP32 w[nout][cin][3][3] -> BF16 [9][cin_pad/8][nout_pad][8]
// (the B operand layout of conv3x3_tc_kernel), zero-padded.
//   PACK_PLAIN       packed[t][c][n] = w[n][c][t]
//   PACK_ADJOINT     the input-gradient convolution of w: w'[c][n][ky][kx] =
//                    w[n][c][2-ky][2-kx] (packed outputs = w's inputs)
//   PACK_TIED_INPUT  as PLAIN, but packed input channels 0-5 and 6-11 both
//                    read logical 0-5 (high and low BF16 parts of the same
//                    field) and 12-14 read logical 6-8
// ---------------------------------------------------------------------------
// Block x of the grid takes elements x * blockDim.x + threadIdx.x, strided by
// the grid's x extent.
__device__ __forceinline__ void pack_conv_weights_elements(const float *__restrict__ w, int nout, int cin,
                                                           int nout_pad, int cin_pad, int mode,
                                                           __nv_bfloat16 *__restrict__ out) {
    const int total = 9 * cin_pad * nout_pad;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int j = i % 8;
        const int n = (i / 8) % nout_pad;
        const int chunk = (i / (8 * nout_pad)) % (cin_pad / 8);
        const int t = i / (8 * nout_pad * (cin_pad / 8));
        int c = chunk * 8 + j;
        const int ky = t / 3, kx = t % 3;
        float v = 0.0f;
        if (mode == PACK_ADJOINT) {
            // packed output channel n ranges over the original inputs, packed input c over the original outputs
            if (n < cin && c < nout) v = w[((size_t(c) * cin + n) * 3 + (2 - ky)) * 3 + (2 - kx)];
        } else {
            if (mode == PACK_TIED_INPUT) c = c < 6 ? c : (c < 15 ? c - 6 : cin);
            if (n < nout && c < cin) v = w[((size_t(n) * cin + c) * 3 + ky) * 3 + kx];
        }
        out[i] = __float2bfloat16_rn(v);
    }
}

}  // namespace qla
