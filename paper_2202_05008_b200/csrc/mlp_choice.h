// Which kernel a control policy of up to 192 units runs on, and with how many episodes a block, without CUDA so that it can be tested anywhere.
#pragma once
#include <cstddef>
#include <cstdint>

namespace evo {

// Blocks of a kernel that an SM of compute capability 10.0 holds at once: 64 K registers and 64 warps in four parts (registers in units of
// 256 per warp), 228 KB of shared memory in units of 128 bytes, 1 KB of which the system takes per block.
inline uint32_t resident_blocks(uint32_t regs, size_t smem, uint32_t threads)
{
    const uint32_t warps = (threads + 31u) / 32u, per_warp = (regs + 7u) / 8u * 256u;
    const uint32_t fit = 16384u / per_warp < 16u ? 16384u / per_warp : 16u;
    const uint32_t by_regs = 4u * fit / warps, by_smem = static_cast<uint32_t>(228u * 1024u / ((smem + 1024u + 127u) / 128u * 128u));
    const uint32_t n = by_regs < by_smem ? by_regs : by_smem;
    return n < 32u ? n : 32u;
}

// Waves of blocks, with `resident` of them on an SM at once: a last wave that leaves SMs room takes 0.6 of a whole one and, for each
// block, its share of the other 0.4.
inline double mlp_waves(uint64_t blocks, uint32_t sms, uint32_t resident)
{
    const uint64_t share = (blocks + sms - 1u) / sms, rest = share % resident;
    return static_cast<double>(share / resident) + (rest ? 0.6 + 0.4 * static_cast<double>(rest) / resident : 0.0);
}

// Whether k_rollout_mlp_deep (weights in registers) is faster than k_rollout_mlp_mma (weights in shared memory; resident_mma = 0: they do not
// fit).  Its blocks are as large as the widest layer and hold many registers, so fewer of them fit an SM; wave for wave it is the
// faster one by a factor that depends on the layers, on whether one is wide (above 64 units) and on the episodes of a block (eb).  These
// are the limits below: how many times the waves of the other it may take.  Measured in 258 policies of 6 to 128 units, both tasks, 4 and 8
// episodes, 100 to 2,000 members (4,068 roll-outs): 0.2 % more time in the mean than with the faster kernel of the two, and 16 take 1 to 8 % longer
// here than with the other.  Examples, 50 steps, deep / mma: 28-57-53-52-8, 592 members x 4 episodes 69 / 130 us;
// 28-8-68-20-8, 592 x 8 183 / 121; 5-14-13-110-1, 444 x 8 172 / 120; 5-6-9-14-50-1, 740 x 8 165 / 140; 28-8-102-8-12-8, 2,000 x 4 774 / 365;
// 28-109-10-119-115-8, 300 x 8 271 / 475.
inline bool mlp_deep_pays(uint32_t hidden, bool wide, uint32_t eb, uint64_t blocks, uint32_t sms, uint32_t resident_deep, uint32_t resident_mma)
{
    if (hidden == 1u || resident_mma == 0u) return true;
    if (resident_deep == 0u) return false;
    const double limit = hidden == 3u ? (!wide ? 2.0 : eb == 4u ? 1.7 : 1.45) : wide ? 2.4 : eb == 4u ? 1.95 : 1.65;
    return mlp_waves(blocks, sms, resident_deep) <= limit * mlp_waves(blocks, sms, resident_mma);
}

// The same for policies of two to four hidden layers with one of 129 to 192 units: k_rollout_mlp_deep then has one block on an SM, whose wave takes
// 0.41 to 0.7 of the time of one of k_rollout_mlp_mma.  130 policies of 8 to 192 units, both tasks, 1 to 16 episodes, 16 to 512 members, 50
// steps: 0.69 of the time of k_rollout_mlp_mma in the mean (geometric), 0.03 % more than with the faster kernel of the two, one takes
// 0.5 % longer than there; with 1.5 and 1.9 for a limit 0.3 % more.  Examples, deep / mma in us: 5-15-189-54-1, 118 x 2 76 / 124; 28-145-157-59-8,
// 836 blocks of 8 661 / 1,159; 5-107-29-138-1, 676 of 8 430 / 325; 28-154-13-77-8, 424 of 8 259 / 158; 28-180-180-180-8, 296 x 4 196, and
// 3,436 with the weights read through the caches.  (resident_mma = 0: they do not fit the shared memory.  The faster one then, but choose_kernel leaves such
// policies to fp32 arithmetic.)
inline bool mlp_widest_pays(uint64_t blocks, uint32_t sms, uint32_t resident_deep, uint32_t resident_mma)
{
    if (resident_mma == 0u) return true;
    if (resident_deep == 0u) return false;
    return mlp_waves(blocks, sms, resident_deep) <= 1.7 * mlp_waves(blocks, sms, resident_mma);
}

// Whether blocks of four episodes are faster than blocks of eight for a member with more than four (registers: on k_rollout_mlp2).  Eight take three MMAs per tile
// and twice the tanh of four: where blocks of four still find an SM each (two, for the wide policies of k_rollout_mlp2 on the tanh-linear task) the
// step is shorter with them.  8 episodes, 50 steps, blocks of 8 / of 4 in us: 28-119-25-8, 70 members 97 / 77, 148 97 / 87; 28-64-64-8, 74 64 / 55;
// 5-100-120-1, 74 101 / 90; 28-64-64-64-8, 74 86 / 77; 28-43-41-100-8, 74 143 / 105; 5-57-12-53-11-1, 74 138 / 98.  With more: 5-64-64-1, 148 59 / 61;
// 28-28-38-8, 148 55 / 58; 28-64-64-64-8, 148 86 / 94.
// Up to eight episodes, one block of eight writes the fitness itself, and two of four need k_fitness_finalize, 1.2 us, which takes the more steps to
// make up for the less a step gains.  74 members x 8 after 20 / 50 / 80 / 128 steps: 5-64-64-1 15.1 / 16.1, 31.1 / 31.2, 47.1 / 46.2, 72.8 / 70.3;
// 5-30-1 9.7 / 10.6, 20.3 / 21.0, 30.7 / 31.0, 47.5 / 47.1; 28-20-8 11.8 / 12.2, 23.2 / 22.4; 28-64-64-8 16.8 / 16.7, 33.8 / 30.9; 5-100-1 11.3 / 11.2,
// 24.1 / 22.2; 28-119-25-8 23.9 / 21.6, 50.7 / 42.1; 28-64-64-64-8 22.6 / 21.7, 45.7 / 41.9; 28-8 18.2 / 17.7, 37.4 / 34.0.
inline bool mlp_four_pay(uint32_t hidden, uint32_t widest, bool cart, bool registers, uint32_t members, uint32_t episodes, uint32_t horizon, uint32_t sms)
{
    const bool two = registers && !cart && widest > 64u;
    if (static_cast<uint64_t>(members) * ((episodes + 3u) / 4u) > (two ? 2u : 1u) * sms) return false;
    const bool long_step = hidden > 2u || widest > 64u || (!cart && (widest > 48u || hidden == 0u));
    return episodes > 8u || horizon >= (long_step ? 20u : !cart ? 50u : hidden == 2u ? 80u : 120u);
}

}  // namespace evo
