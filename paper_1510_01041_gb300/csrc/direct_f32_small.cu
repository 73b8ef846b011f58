// direct_f32_small.cu -- the one-kernel branch-and-bound (direct.cuh) for float sets up to 2048 points.
#include "direct_launch.cuh"

namespace lms {
namespace direct {

template cudaError_t launch_cluster<FloatSmall>(const DirectArgs &, size_t, cudaStream_t);

}  // namespace direct
}  // namespace lms
