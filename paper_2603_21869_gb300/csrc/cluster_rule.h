// The blocks of a batch's coarse-level clusters (plain C++: no CUDA header).
#pragma once

// The first number of blocks that is usable (the levels' arrays fit and the device runs such clusters): the
// preferred one, then larger ones up to `most` (a block's share of the arrays shrinks), then smaller
// ones (a device or partition that holds no cluster of that size); 0 where none is.
template <class Usable>
int cluster_blocks(int preferred, int most, Usable usable) {
    for (int S = preferred; S <= most; S *= 2)
        if (usable(S)) return S;
    for (int S = preferred / 2; S >= 1; S /= 2)
        if (usable(S)) return S;
    return 0;
}
