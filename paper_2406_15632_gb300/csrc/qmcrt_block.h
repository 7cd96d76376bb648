// qmcrt_block.h -- the default block size of a trace launch.
#pragma once

#include <cstdint>

namespace qmcrt {

// Threads per block of a trace whose caller names none (warps are independent: results do not
// depend on it).  FP32: 256, whose warps trace neighbouring packets and share L1 lines (finite
// star, 2^22 packets: 1.52 ms against 1.66 with 128 threads, 1.83 with 32), and fewer for
// launches that would leave SMs without a block (2^12 packets on 256^3: 52 against 56 us).
// FP64: a warp, since a slot that waits for the slowest of eight walks costs more than the
// cache gains (50 000 star packets on 64^3: 207 against 297 us, 200 000: 798 against 863,
// 10^5 packets of eight orders: 3.65 against 4.01 ms, 10^6 star packets the same); more where
// the launch would have more blocks than a grid holds.
inline int default_block(uint64_t threads, bool f64)
{
    int b = f64 ? 32 : 256;
    while (b > 32 && threads < (uint64_t)b * 304) b /= 2;
    while (b < 256 && threads > (uint64_t)b * 0x7fffffffu) b *= 2;
    return b;
}

}  // namespace qmcrt
