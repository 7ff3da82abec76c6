// Instantiations of the 2D FP64 step kernels for n = 12, 13, 14.
#include "k_step2d_impl.cuh"

namespace sl {
namespace k2d {
template void launch_n<12>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<12>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
template void launch_n<13>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<13>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
template void launch_n<14>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<14>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
}  // namespace k2d
}  // namespace sl
