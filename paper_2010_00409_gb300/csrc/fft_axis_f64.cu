// The generic axis transforms of float64 storage (a translation unit per type, so
// that they compile side by side).
#include "fft_axis.cuh"

namespace psatd {

template cudaError_t launch_fft_axis<double>(cplx<double>*, int, const GridGeom&, const Tables<double>&, int, int, cudaStream_t,
                                            long long*);

}  // namespace psatd
