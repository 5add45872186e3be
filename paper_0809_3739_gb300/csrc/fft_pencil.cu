// Instantiation unit of the FFT passes (fft_passes.cuh): the FP32 pencil passes
// (the z transform with the kinetic factor).
// The passes are split over several translation units only so that nvcc
// compiles them in parallel.
#include "fft_passes.cuh"

namespace itp {

template cudaError_t launch_pencil<float>(const GridDesc&, const PencilArgs<float>*, int,
                                          cudaStream_t);

}  // namespace itp
