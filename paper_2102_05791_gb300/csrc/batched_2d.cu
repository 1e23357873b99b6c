// The batched solver's kernels for triangle meshes (one translation unit a dimension: they compile side by side).
#include "batched_kernel.cuh"

namespace softsim {

BatchKernel batch_kernel_2d(int threads)
{
    return threads == 128 ? k_batch_rollout<2, 128> : threads == 512 ? k_batch_rollout<2, 512> : k_batch_rollout<2, 256>;
}

}  // namespace softsim
