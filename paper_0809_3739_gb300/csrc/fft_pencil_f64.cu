// Instantiation unit of the FFT passes (fft_passes.cuh): the FP64 pencil
// passes, single and grouped launches.
// The passes are split over several translation units only so that nvcc
// compiles them in parallel.
#include "fft_passes.cuh"

namespace itp {

template cudaError_t launch_pencil<double>(const GridDesc&, const PencilArgs<double>*, int,
                                          cudaStream_t);
template cudaError_t launch_pencil_group<double>(const GridDesc&, int, const PencilArgs<double>*,
                                                 const int2*, int, cudaStream_t);

}  // namespace itp
