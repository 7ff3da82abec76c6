// Instantiations of the 2D FP64 step kernels for n = 2, 3, 4, 5, 6, 7, 8.
#include "k_step2d_impl.cuh"

namespace sl {
namespace k2d {
template void launch_n<2>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<2>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
template void launch_n<3>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<3>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
template void launch_n<4>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<4>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
template void launch_n<5>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<5>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
template void launch_n<6>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<6>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
template void launch_n<7>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<7>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
template void launch_n<8>(int, const StepParams&, const Tables1D&, const Map2D&, int64_t, const double*, double*,
                            const Work2D&, unsigned*, cudaStream_t);
template void launch_shift<8>(const Shift2D&, const StepParams&, int64_t, const double*, const Work2D&, cudaStream_t);
}  // namespace k2d
}  // namespace sl
