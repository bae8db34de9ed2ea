// Launch arithmetic that needs no device (plain C++).
#pragma once

#include <cstddef>

namespace wd {

// Shared memory of an SM, the most a block may use of it, the system's share per
// block and the unit that a block's total is rounded up to.
constexpr size_t SM_SMEM = 228 * 1024, BLOCK_SMEM = 227 * 1024, SYSTEM_SMEM = 1024, SMEM_UNIT = 128;

// Dynamic shared memory with which exactly ceil(blocks / sms) blocks fit on an SM, for a
// kernel with `static_bytes` of its own of which `resident` fit otherwise; 0 if the grid
// needs `resident` or more.  Without the rounding to SMEM_UNIT a block that asks for a 5th
// or 7th of the SM gets 4 or 6 (FP64 even-odd hop on 12^3 x 24, 648 blocks: 42.1 us, with
// it 40.4).
inline size_t spread_bytes(long long blocks, int sms, int resident, size_t static_bytes)
{
    const long long k = (blocks + sms - 1) / sms;
    if (k >= resident || k < 1) return 0;
    const size_t per = SM_SMEM / (size_t)k / SMEM_UNIT * SMEM_UNIT - SYSTEM_SMEM;
    return (per < BLOCK_SMEM ? per : BLOCK_SMEM) - static_bytes;
}

} // namespace wd
