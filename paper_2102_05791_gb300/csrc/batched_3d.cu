// The batched solver's kernels for tet meshes (one translation unit a dimension: they compile side by side).
#include "batched_kernel.cuh"

namespace softsim {

BatchKernel batch_kernel_3d(int threads)
{
    return threads == 128 ? k_batch_rollout<3, 128> : threads == 512 ? k_batch_rollout<3, 512> : k_batch_rollout<3, 256>;
}

}  // namespace softsim
