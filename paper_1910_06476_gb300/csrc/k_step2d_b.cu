// Instantiations of the 2D FP64 step kernels for n = 9, 10, 11.
#include "k_step2d_impl.cuh"

namespace sl {
namespace k2d {
template void launch_n<9>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<9>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
template void launch_n<10>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<10>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
template void launch_n<11>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<11>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
}  // namespace k2d
}  // namespace sl
