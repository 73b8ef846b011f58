// direct_mid.cu -- the one-kernel branch-and-bound (direct.cuh) for int16 sets of 2049 to 16384 points.
#include "direct_launch.cuh"

namespace lms {
namespace direct {

template cudaError_t launch_cluster<Mid>(const DirectArgs &, size_t, cudaStream_t);

}  // namespace direct
}  // namespace lms
