// Instantiation unit of the FP64 plane passes (fft_passes.cuh): 32 x 32, 48 x 48 and 64 x 64 planes.
// The passes are split over several translation units only so that nvcc
// compiles them in parallel.
#define ITP_PLANE64_UNIT
#include "fft_passes.cuh"

namespace itp {

template cudaError_t plane64_dispatch<32, 32>(const GridDesc&, int,
                                             const TermPack<PlaneArgs<double>>&,
                                             const PlaneArgs<double>*, const int2*, int, size_t,
                                             cudaStream_t);
template cudaError_t plane64_dispatch<48, 48>(const GridDesc&, int,
                                             const TermPack<PlaneArgs<double>>&,
                                             const PlaneArgs<double>*, const int2*, int, size_t,
                                             cudaStream_t);
template cudaError_t plane64_dispatch<64, 64>(const GridDesc&, int,
                                             const TermPack<PlaneArgs<double>>&,
                                             const PlaneArgs<double>*, const int2*, int, size_t,
                                             cudaStream_t);

}  // namespace itp
