// Launch of k_rollout_mlp_deep (rollout_mlp_deep.cuh), and its instances for blocks of four episodes.
#include "rollout_mlp_deep.cuh"

namespace evo {

DeepKernel rollout_mlp_deep_kernel4(bool cart, uint32_t hidden, uint32_t size, bool fine)
{
    return cart ? pick_kernel<4, true>(hidden, size, fine) : pick_kernel<4, false>(hidden, size, fine);
}

namespace {

constexpr int kMaxDynamic = 198 * 1024;             // shared memory besides the static arrays, which take up to 28.2 KB
constexpr size_t kMaxLowBytes = 190u * 1024u;

uint32_t tiles_of(uint32_t units) { return (units + 15u) / 16u; }

struct DeepLaunch { DeepKernel kernel; uint32_t threads; size_t bytes; uint32_t size; bool fine; };

DeepLaunch deep_launch(uint32_t task, uint32_t n_layers, const uint32_t* sizes, uint32_t EB)
{
    const bool cart = task == EVO_TASK_CARTPOLE;
    const uint32_t hidden = n_layers - 1u;
    uint32_t warps = 1;
    DeepLaunch d;
    d.fine = false;
    for (uint32_t l = 1; l <= hidden; ++l) {
        if (tiles_of(sizes[l]) > warps) warps = tiles_of(sizes[l]);
        d.fine = d.fine || sizes[l] < 49u;
    }
    d.size = warps > 8u ? 2u : warps > 4u ? 1u : 0u;
    if (!cart && warps < 2u) warps = 2u;
    d.threads = 32u * warps;
    d.kernel = EB == 4u ? rollout_mlp_deep_kernel4(cart, hidden, d.size, d.fine) : rollout_mlp_deep_kernel8(cart, hidden, d.size, d.fine);
    d.bytes = static_cast<size_t>(warps) * (hidden - 1u) * (d.size == 1u ? 8u : 4u) * 512u;
    if (d.size == 2u) {                                              // the layers' own tiles; the third matrix with its hi parts
        d.bytes = 0;
        for (uint32_t m = 1; m < hidden; ++m) d.bytes += tiles_of(sizes[m + 1]) * ((tiles_of(sizes[m]) + 3u) & ~3u) * (m > 2u ? 1024u : 512u);
    }
    return d;
}

}  // namespace

// Episodes per block; 0: not a policy for this kernel.
uint32_t rollout_mlp_deep_eb(uint32_t n_layers, const uint32_t* sizes, uint32_t episodes)
{
    if (n_layers < 2u || n_layers > 5u) return 0u;
    uint32_t widest = 0;
    for (uint32_t l = 1; l < n_layers; ++l) widest = tiles_of(sizes[l]) > widest ? tiles_of(sizes[l]) : widest;
    if (widest > 12u || (n_layers == 3u && widest <= 8u)) return 0u;
    if (deep_launch(EVO_TASK_CARTPOLE, n_layers, sizes, 4u).bytes > kMaxLowBytes) return 0u;
    return episodes > 4u ? 8u : 4u;
}

// Whether the policy (one of this kernel) is faster here than on k_rollout_mlp_mma, for the whole population, of which the solver may have a
// shard; -1: the runtime's error
int rollout_mlp_deep_pays(uint32_t task, uint32_t n_layers, const uint32_t* sizes, uint32_t pop, uint32_t EB, uint32_t n_eb)
{
    if (n_layers == 2u) return 1;
    static std::atomic<uint64_t> known[2][2][3][3][2];
    const DeepLaunch d = deep_launch(task, n_layers, sizes, EB);
    uint32_t regs;
    size_t fixed;
    if (!kernel_needs(d.kernel, known[EB == 8u][task == EVO_TASK_CARTPOLE][n_layers - 3u][d.size][d.fine], &regs, &fixed)) return -1;
    const int mma = rollout_mlp_mma_resident(task, n_layers, sizes, EB);
    if (mma < 0) return -1;
    const uint64_t blocks = static_cast<uint64_t>(pop) * n_eb;
    const uint32_t deep = resident_blocks(regs, d.bytes + fixed, d.threads);
    if (d.size == 2u) return mlp_widest_pays(blocks, kSms, deep, static_cast<uint32_t>(mma));
    return mlp_deep_pays(n_layers - 1u, d.size == 1u, EB, blocks, kSms, deep, static_cast<uint32_t>(mma));
}

int launch_rollout_mlp_deep(cudaStream_t st, const RolloutMlpArgs& a, DeviceStatus* status)
{
    const DeepLaunch d = deep_launch(a.task, a.n_layers, a.sizes, a.EB);
    const size_t bytes = spread_over_sms(d.kernel, d.bytes, static_cast<uint64_t>(a.P) * a.n_eb);
    if (!a.attr_done &&
        cudaFuncSetAttribute(d.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynamic) != cudaSuccess) return -1;
    return launch_dependent(d.kernel, dim3(a.P, a.n_eb), dim3(d.threads), bytes, st, a, status) == cudaSuccess ? 1 : -1;
}

}  // namespace evo
