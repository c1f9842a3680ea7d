// omni_fold.cu -- fold of a LAST pass whose samples were split over grid rows.
//
// A LAST pass runs one CTA per channel and tile of the lattice, each walking the
// chunk's samples; few channels of a small array leave most of the GPU idle (one
// 16 x 16 array, 64 samples: one CTA, 67 us).  Its samples are then cut into slices, one
// grid row each, which leave their FP32 sums side by side; this kernel adds them in
// slice order into the FP64 accumulator, so that the result does not depend on timing.
#include "omni_fft_common.cuh"

namespace omni {
namespace {

__global__ void __launch_bounds__(256) fold_parts(const float* __restrict__ part, int split, int64_t per, double fs,
                                                  double* __restrict__ P) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= per) return;
    double s = 0.0;
#pragma unroll 8
    for (int k = 0; k < split; ++k) s += (double)part[k * per + e];
    P[e] += fs * s;
}

}  // namespace

cudaError_t launch_fold_parts(const PassArgs& a, cudaStream_t st) {
    const int64_t per = a.S * a.P_stride;
    if (per <= 0 || a.split <= 1) return cudaSuccess;
    fold_parts<<<(unsigned)((per + 255) / 256), 256, 0, st>>>(a.part, a.split, per,
                                                              a.fold_scale != 0.0 ? a.fold_scale : 1.0,
                                                              a.P + a.c0 * a.P_stride);
    return cudaGetLastError();
}

}  // namespace omni
