// Host arithmetic behind spread_over_sms (internal.h), without CUDA so that it can be tested anywhere.
#pragma once
#include <cstddef>
#include <cstdint>

namespace evo {

// Dynamic shared memory per block with which an SM of `sm_bytes` holds its even share of `blocks`, and not one more: the largest
// number that leaves room for the share is not needed, the smallest that leaves none for another block is.  `fixed` = what a
// block takes besides (its static arrays and the system's 1 KB); shared memory is handed out in units of 128 bytes.
inline size_t spread_bytes(size_t dynamic, size_t fixed, uint64_t blocks, uint32_t sms, size_t sm_bytes)
{
    const uint64_t share = (blocks + sms - 1u) / sms;
    if (share < 1u || share > 8u) return dynamic;
    const size_t block = (sm_bytes / (share + 1u) / 128u + 1u) * 128u;
    return block > dynamic + fixed ? block - fixed : dynamic;
}

}  // namespace evo
