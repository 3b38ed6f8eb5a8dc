// k_rollout_mlp_deep (rollout_mlp_deep.cuh) for blocks of eight episodes.
#include "rollout_mlp_deep.cuh"

namespace evo {

DeepKernel rollout_mlp_deep_kernel8(bool cart, uint32_t hidden, uint32_t size, bool fine)
{
    return cart ? pick_kernel<8, true>(hidden, size, fine) : pick_kernel<8, false>(hidden, size, fine);
}

}  // namespace evo
