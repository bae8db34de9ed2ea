// Launch arithmetic that needs no device (plain C++).
#pragma once

#include <cstddef>

namespace wd {

// Shared memory of an SM, the most a block may use of it, the system's share per
// block and the unit that a block's total is rounded up to.
constexpr size_t SM_SMEM = 228 * 1024, BLOCK_SMEM = 227 * 1024, SYSTEM_SMEM = 1024, SMEM_UNIT = 128;

// Dynamic shared memory with which no more than k = ceil(blocks / sms) blocks fit on an SM,
// for a kernel with `static_bytes` of its own of which `resident` fit otherwise.  us, FP64
// even-odd hop alone, launches one after another, without / with: 648 blocks 59.4 / 40.4, 896
// 61.2 / 47.9, 1024 62.1 / 55.5; 12-real links, 432 blocks 47.8 / 29.9.
// 0 where the grid needs `resident` or more, and where other streams' kernels run beside it
// and two such grids fit side by side with room left (2 k < resident): a successor
// dispatched early then spreads as evenly (432 blocks 25.0 / 25.0), and the others' kernels
// fit in (a graph batch of eight solves with FP64 updates, padded / not: 8^3 x 16 7.9 / 7.0 ms,
// 8^2 x 16^2 9.7 / 8.9, 12^3 x 16 12.3 / 11.6; k = 4 of 8 is mixed: 8 x 20 x 10 x 20, 5 solves 10.0 /
// 10.1, 8 solves 13.0 / 12.6, 10 x 12^2 x 24, 5 solves 9.9 / 10.4).  Alone it is padded all the same: behind a kernel that leaves the SMs
// unevenly the blocks would stack up (host-driven BF16 CG with FP64 updates on 8^2 x 16^2, 256
// blocks, 5.53 ms without, 5.26 with).
// No more than keeps block k + 1 out, which leaves the rest to other streams; k = 7 gets 6:
// alone the same, that batch on 16^4 20.1 ms, with 7 20.4.  A block's total is rounded up to
// SMEM_UNIT: for exactly a 5th of the SM only 4 fit (648 blocks: 42.1 us).
inline size_t spread_bytes(long long blocks, int sms, int resident, size_t static_bytes, bool beside)
{
    const long long k = (blocks + sms - 1) / sms;
    if (k >= resident || k < 1 || (beside && 2 * k < resident)) return 0;
    const size_t next = (size_t)(k == 7 ? 7 : k + 1);   // blocks that must not fit
    const size_t per = (SM_SMEM / next / SMEM_UNIT + 1) * SMEM_UNIT - SYSTEM_SMEM;
    return (per < BLOCK_SMEM ? per : BLOCK_SMEM) - static_bytes;
}

// ---- FP64 hop: three threads per site, or one ----------------------------------
// `blocks`: blocks of 32 sites (both parities of a full operator).  Three threads per site,
// except with 12-real links on grids that the kernel with one site per thread takes in one
// even wave, two 128-thread blocks (8 of 32 sites) per SM: the rebuilt row leaves room for 5
// three-thread blocks per SM, so 8 take two turns.  us, one thread per site / three, even-odd,
// 12 reals without and with the axpy term: 64 blocks 38.6 / 15.1 and 40.3 / 15.1, 1024 71.9 /
// 65.1 and 76.0 / 66.5, 1120 72.0 / 82.4 and 76.3 / 84.1, 1280 138.7 / 82.4 and 146.5 / 84.5, 2400
// 145.6 / 146.2 and 153.0 / 149.9, 10,368 627 / 615 and 660 / 630.  18 reals: 64 blocks 31.8 /
// 12.3 and 33.6 / 12.3, 1024 58.8 / 54.0 and 62.5 / 55.5, 1120 58.8 / 60.8 and 62.5 / 62.5, 1280
// 114.0 / 68.7 and 122.4 / 70.6, 4752 234.4 / 237.3 and 248.4 / 244.1, 10,368 514 / 508 and 546 / 522;
// one thread is 3 % faster on 1120 blocks without the term, but not beside other streams (graph
// batch of eight 16^3 x 18 solves, 1152 blocks, FP64 updates: 23.6 ms, three threads 21.5).
inline bool f64_three_threads(long long blocks, int sms, int recon)
{
    return recon == 18 || (blocks + sms - 1) / sms != 8;
}

// ---- shared-link kernel: build and block size ---------------------------------
// A grid of shared-link blocks (`threads` threads each, `sms` SMs) that is at most two
// waves of the 128-register build: short launches gain more from a thread with its
// loads in flight than from more warps (80 registers: half again as many).  us, 80
// against 128 registers, 128 threads: 16^4 even-odd, 6 FP16 fields 15.0 / 12.8,
// 8 FP32 fields 21.7 / 18.9; 8^2 x 16^2 full, 12 FP16 fields 17.5 / 12.5; 8^4
// even-odd, 12 FP32 fields 7.9 / 6.5; beyond two waves the other way: 16^3 x 32
// even-odd, 6 FP16 fields 22.6 / 24.2, full 46.7 / 52.3; 32^4, 12 FP32 fields 372 / 390.
// 96 threads, 5 FP32 fields: 1440 blocks 24.0 / 20.9, 1536 (more than two waves) 24.8 / 24.8.
// 16-bit storage: the builds take the directions in different orders, so the choice looks
// at the lattice only; a field's bits do not depend on how many others are in the launch.
inline bool mrhs_small(long long blocks, int threads, bool f32, int sms)
{
    return blocks <= 2LL * (512 / (f32 ? threads : 128)) * sms;
}

// Threads of an untuned launch for `nrhs` fields: 4 warps, or 3 where that takes at least
// a tenth fewer warp passes over the fields (5, 6, 9, ... fields) and the grid is large
// enough to profit (with 4 fields or less the links' staging counts and wants the warps:
// 20^4 full, 3 fields 42.4 / 44.5).
// FP32: where the three-warp grid is at most two waves of the 128-register build (even-odd,
// 5 fields, us, 4 warps / 3: 1280 blocks 22.3 / 19.6, 1440 23.9 / 20.9), and beyond that where
// it is fewer waves of the other build (6 fields: 1792 blocks, two waves each, 28.8 / 30.6;
// 2016, three / two, 35.5 / 32.5; 2560, three each, 41.2 / 42.4; 32^4, 16,384, 207 / 197).
// 16-bit: from 11 blocks per SM on (FP16, 6 fields: 1440 blocks 16.4 / 17.4, 1536 18.1 / 18.6, 1792
// 21.4 / 20.6, 2304 27.9 / 26.9, 3888 44.8 / 42.5).
inline int mrhs_threads(long long blocks, int nrhs, bool f32, int sms)
{
    if (nrhs <= 4 || 10 * 3 * ((nrhs + 2) / 3) > 9 * 4 * ((nrhs + 3) / 4) || mrhs_small(blocks, 128, f32, sms)) return 128;
    if (!f32) return blocks >= 11LL * sms ? 96 : 128;
    auto waves = [&](int threads) {
        const long long fit = 768 / threads * (long long)sms;
        return (blocks + fit - 1) / fit;
    };
    return mrhs_small(blocks, 96, f32, sms) || waves(96) < waves(128) ? 96 : 128;
}

} // namespace wd
