// ivb_launch.h -- rules on the shape of the bounding launches (plain C++, no
// CUDA: the CPU tests compile this file as it is).
#pragma once

namespace ivb {

// A block's threads can form `groups` groups that share each subdomain's outputs:
// every group is whole warps, so that no warp runs two groups' programs (its
// reductions and, with chunk synchronisation, its named barriers want whole warps).
inline bool groups_fit(int block, int groups) { return groups >= 1 && block % (32 * groups) == 0; }

// threads per subdomain of blocks of `block` threads: the number asked for, or 1
// where the block cannot be dealt out to that many groups
inline int block_tpsub(int block, int wanted) { return groups_fit(block, wanted) ? wanted : 1; }

// Blocks of a launch over `count` subdomains, of `resident` at most: a block takes a
// warp of subdomains at least (even_tile), further blocks would only hold frames.
inline int range_blocks(long long count, int resident) {
    const long long warps = (count + 31) / 32;
    return warps < resident ? (int)warps : resident;
}

}  // namespace ivb
