// direct_large.cu -- the one-kernel branch-and-bound (direct.cuh) for int16 sets above 16384 points.
#include "direct_launch.cuh"

namespace lms {
namespace direct {

template cudaError_t launch_cluster<Large>(const DirectArgs &, size_t, cudaStream_t);

}  // namespace direct
}  // namespace lms
