// rtlbfs_smem.h -- shared memory that a launch asks for to hold its blocks
// per SM down (plain C++, no CUDA types, so that it also builds into host-only
// unit tests).
#pragma once

#include <cstddef>

namespace rtlbfs {

// An SM's shared memory, what the system takes of it per block, and the most
// a block may ask for.
constexpr std::size_t kSmemSM = 228 * 1024, kSmemSystem = 1024, kSmemMax = 227 * 1024;

// Dynamic shared memory of a launch whose blocks need `need` bytes and that
// should keep `blocks` (>= 1) of them on an SM: the least that one block more
// does not find, in steps of 128 bytes.  Where an even share of the SM is not
// above `need`, and from 228 blocks on not above the system's part either, the
// blocks limit themselves: `need`.
inline std::size_t smem_for_blocks(std::size_t need, long long blocks)
{
    const std::size_t share = kSmemSM / ((std::size_t)blocks + 1);
    if (share < kSmemSystem) return need;
    const std::size_t ask = (share - kSmemSystem) / 128 * 128 + 128;
    return ask < need ? need : (ask > kSmemMax ? kSmemMax : ask);
}

}  // namespace rtlbfs
