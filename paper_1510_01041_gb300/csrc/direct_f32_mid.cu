// direct_f32_mid.cu -- the one-kernel branch-and-bound (direct.cuh) for float sets above 2048 points.
#include "direct_launch.cuh"

namespace lms {
namespace direct {

template cudaError_t launch_cluster<FloatMid>(const DirectArgs &, size_t, cudaStream_t);

}  // namespace direct
}  // namespace lms
