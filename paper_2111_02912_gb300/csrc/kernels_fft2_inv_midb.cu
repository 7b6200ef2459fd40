// Register-resident two-phase line FFT, pass kind PASS_INV_MID, list 1 of the line lengths (one
// translation unit per pass kind and list so that the kernels compile in parallel).
#include "fft_twostep.cuh"

namespace nj {
template cudaError_t launch_fft2_kind<PASS_INV_MID, 1>(int, int, const LinePass&, dim3, int, size_t, cudaStream_t);
}  // namespace nj
