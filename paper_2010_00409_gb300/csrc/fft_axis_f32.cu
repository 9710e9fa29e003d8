// The generic axis transforms of float32 storage (a translation unit per type, so
// that they compile side by side).
#include "fft_axis.cuh"

namespace psatd {

template cudaError_t launch_fft_axis<float>(cplx<float>*, int, const GridGeom&, const Tables<float>&, int, int, cudaStream_t,
                                            long long*);

}  // namespace psatd
