// The kernels of rho_fft.cuh for float (a unit of its own, so that the two
// types compile side by side).
#include "rho_fft.cuh"

namespace chi0 {
namespace rfft {

template cudaError_t wf_dispatch<float>(const RhoGeom&, const int32_t*, const int32_t*, const float2*, float2*, cudaStream_t,
                                     int, int, int, int);
template cudaError_t rho_dispatch<float>(const RhoTask<float, float2>&, size_t, int, int64_t, cudaStream_t);
template cudaError_t batch_dispatch<float>(int, const RhoTask<float, float2>*, int, int64_t, size_t, unsigned long long*, int,
                                        cudaStream_t);

}  // namespace rfft
}  // namespace chi0
