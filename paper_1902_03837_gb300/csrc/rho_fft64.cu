// The kernels of rho_fft.cuh for double (a unit of its own, so that the two
// types compile side by side).
#include "rho_fft.cuh"

namespace chi0 {
namespace rfft {

template cudaError_t wf_dispatch<double>(const RhoGeom&, const int32_t*, const int32_t*, const double2*, double2*, cudaStream_t,
                                     int, int, int, int);
template cudaError_t rho_dispatch<double>(const RhoTask<double, double2>&, size_t, int, int64_t, cudaStream_t);
template cudaError_t batch_dispatch<double>(int, const RhoTask<double, double2>*, int, int64_t, size_t, unsigned long long*, int,
                                        cudaStream_t);

}  // namespace rfft
}  // namespace chi0
