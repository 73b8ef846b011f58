// direct_batch.cu -- the one-kernel branch-and-bound (direct.cuh) for the sets
// of a batch, one CTA each.
#include "direct.cuh"

namespace lms {
namespace direct {

int batch_teams_per_sm(size_t smem)
{
    auto kern = Batch::kernel();
    allow_smem(kern, smem);
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, Batch::T, smem) != cudaSuccess || occ < 1) {
        cudaGetLastError();
        return 0;
    }
    return occ;
}

cudaError_t launch_batch(const DirectArgs &a, int nteams, size_t smem, cudaStream_t st)
{
    auto kern = Batch::kernel();
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    StageTimer _t(STAGE_DIRECT, st);
    kern<<<nteams, Batch::T, smem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace direct
}  // namespace lms
