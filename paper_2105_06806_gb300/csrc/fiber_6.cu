// Instances of the orbital-factorised product (fiber.cuh), split over
// translation units so that they compile in parallel.
#include "fiber.cuh"

namespace fiber {
template ed_status launch_g<6>(const HvLaunch<float> *, int, unsigned, cudaStream_t);
}  // namespace fiber
