// kgs_pack.h -- the order of the velocity slots of the packed FP32 sweep.  Plain
// C++ with no CUDA, so that it can be exercised on the host alone.  Not part of
// the public ABI.
#pragma once

#include <algorithm>
#include <vector>

namespace kgs {

constexpr int PACK_HALF = 128;  // velocities per half of a group

// Natural places (0 .. count-1, ix fastest) of the slots of one packed velocity
// group that starts at place v0 of its octant, lines of nxo nodes.  Each half
// of the group (the velocities one thread of the moment phase sums) holds, in
// this order: its pairs of whole lines with the two lines interleaved node by
// node, the line its start cuts (head), an unpaired whole line, and the line
// its end cuts (tail).
inline void pack_order(int v0, int count, int nxo, std::vector<int> &place)
{
    place.clear();
    for (int half = 0; half < 2; half++) {
        const int b = half * PACK_HALF, n = std::min(PACK_HALF, count - b);
        if (n <= 0) break;
        const int head = std::min(n, (nxo - (v0 + b) % nxo) % nxo), full = (n - head) / nxo, pairs = full / 2;
        for (int q = 0; q < pairs; q++)
            for (int ix = 0; ix < nxo; ix++)
                for (int h = 0; h < 2; h++) place.push_back(b + head + (2 * q + h) * nxo + ix);
        for (int v = 0; v < head; v++) place.push_back(b + v);
        for (int v = head + 2 * pairs * nxo; v < n; v++) place.push_back(b + v);
    }
}

}  // namespace kgs
