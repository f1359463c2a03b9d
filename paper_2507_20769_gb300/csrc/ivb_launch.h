// ivb_launch.h -- rules on the shape of the bounding launches (plain C++, no
// CUDA: the CPU tests compile this file as it is).
#pragma once
#include <cstddef>

namespace ivb {

// threads of the largest block of each bounding kernel
constexpr int kInterpBlockMax = 512, kCompiledBlockMax = 256, kSegBlockMax = 1024;

// A block's threads can form `groups` groups that share each subdomain's outputs:
// every group is whole warps, so that no warp runs two groups' programs (its
// reductions and, with chunk synchronisation, its named barriers want whole warps).
inline bool groups_fit(int block, int groups) { return groups >= 1 && block % (32 * groups) == 0; }

// threads per subdomain of blocks of `block` threads: the number asked for, or 1
// where the block cannot be dealt out to that many groups
inline int block_tpsub(int block, int wanted) { return groups_fit(block, wanted) ? wanted : 1; }

// Register budget of a segmented kernel's functions. 64 lets 1024 threads fill an SM. Where
// options fix a block that leaves fewer threads on an SM, their share of the registers, 128 at
// most: more threads at 64 are slower in blocks that stream through the code separately, and the
// same threads spill less with more (2 x 256 at 128 against 4 x 256 at 64: configuration 5, 2^19
// subdomains, 75 and 113 ms; configuration 2, 16 x 16^4, 2.64 and 3.39 ms). Without
// blocks_per_sm such a block counts as 512 threads per SM.
inline int seg_registers(int seg_regs, int block_threads, int blocks_per_sm) {
    if (seg_regs > 0) return seg_regs;
    if (block_threads <= 0) return 64;
    const int blocks = blocks_per_sm > 0 ? blocks_per_sm : block_threads < 512 ? 512 / block_threads : 1;
    const long long regs = 65536 / ((long long)block_threads * blocks) / 8 * 8;
    return regs < 64 ? 64 : regs > 128 ? 128 : (int)regs;
}

// Threads of the largest block of a segmented kernel: all that a register budget
// allows on an SM, in whole groups of four warps (one to each of its four register files; registers
// come in eights).
inline int seg_block_max(int max_regs) {
    const int threads = 65536 / ((max_regs + 7) / 8 * 8) / 128 * 128;
    return threads < kSegBlockMax ? threads : kSegBlockMax;
}
// the largest block that options can ask of it
inline int seg_block_limit(int seg_regs) { return seg_regs > 0 ? seg_block_max(seg_regs) : kSegBlockMax; }
// the budget of a kernel built for blocks of `block_threads` (0: the library's)
inline int seg_budget(int seg_regs, int block_threads, int blocks_per_sm) {
    const int regs = seg_registers(seg_regs, block_threads, blocks_per_sm);
    if (block_threads <= seg_block_max(regs)) return regs;
    return 65536 / ((block_threads + 127) / 128 * 128) / 8 * 8;
}

// Short operations of a segmented kernel out of line (options seg_outline and emulate, interval
// operations per subdomain): by the library's choice the products. Sums emulated on the integer
// pipes are long too, and inline in a large tape they quadruple its compile time and slow it down
// (configuration 5, emulate = 12: 73 ms and 6 s with all out of line, 98 ms and 24 s with the
// products alone; configuration 2, emulate = 15: 5.3 and 4.0 ms, 0.7 and 1.8 s).
inline int seg_outline_for(int option, int emulate, long long ops) {
    return option >= 0 ? option : (emulate & 12) && ops > 1024 ? 1 : 2;
}

// Blocks of a launch over `count` subdomains, of `resident` at most: a block takes a
// warp of subdomains at least (even_tile), further blocks would only hold frames.
inline int range_blocks(long long count, int resident) {
    const long long warps = (count + 31) / 32;
    return warps < resident ? (int)warps : resident;
}

// The library's own shapes run 1024 threads per SM where the frames of all of them
// (`bytes` per thread) take at most a sixteenth of the device's memory (twice that of the 512 threads
// that longer tapes get: 18 GB of 284 at 152 SMs, tapes of some 7000 entries per output).
inline bool wide_frames_fit(size_t bytes, int sms, size_t device_bytes) {
    return bytes * 1024 * (size_t)sms <= device_bytes / 16;
}

// Blocks to launch when memory is short: `blocks`, halved until get(blocks) succeeds;
// 0 when it fails for one block too. The tile loops take any number of blocks.
template <class Get> int blocks_that_fit(int blocks, Get get) {
    while (blocks > 0 && !get(blocks)) blocks /= 2;
    return blocks;
}

}  // namespace ivb
