// Instantiation unit of the FP64 plane passes (fft_passes.cuh): 96 x 96 planes.
// The passes are split over several translation units only so that nvcc
// compiles them in parallel.
#define ITP_PLANE64_UNIT
#include "fft_passes.cuh"

namespace itp {

template cudaError_t plane64_dispatch<96, 96>(const GridDesc&, int,
                                             const TermPack<PlaneArgs<double>>&,
                                             const PlaneArgs<double>*, const int2*, int, size_t,
                                             cudaStream_t);

}  // namespace itp
