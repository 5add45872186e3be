// Instantiation unit of the FP64 plane passes (fft_passes.cuh): planes of any other size that fits one CTA.
// The passes are split over several translation units only so that nvcc
// compiles them in parallel.
#define ITP_PLANE64_UNIT
#include "fft_passes.cuh"

namespace itp {

template cudaError_t plane64_dispatch<0, 0>(const GridDesc&, int,
                                             const TermPack<PlaneArgs<double>>&,
                                             const PlaneArgs<double>*, const int2*, int, size_t,
                                             cudaStream_t);

}  // namespace itp
