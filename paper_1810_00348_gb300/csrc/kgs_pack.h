// kgs_pack.h -- the order of the velocity slots of the packed FP32 sweep.  Plain
// C++ with no CUDA, so that it can be exercised on the host alone.  Not part of
// the public ABI.
#pragma once

#include <algorithm>
#include <vector>

#ifdef __CUDACC__
#define KGS_HD __host__ __device__ __forceinline__
#else
#define KGS_HD inline
#endif

namespace kgs {

constexpr int PACK_HALF = 128;  // velocities per half of a group

// One half of a packed group, n velocities from place v of the octant on, lines
// of nxo nodes, as the units that the moment phase sums one after the other,
// in line order: the line that the half's start cuts (head), the pairs of
// whole lines, an odd whole line, the line that the half's end cuts (tail).
// The slots hold the pairs first, then the other units in this order.  A half
// that lies inside one line is a head alone, which then does not reach the end
// of its line.
struct PackHalf {
    int head = 0, full = 0, tail = 0;  // nodes of the head, whole lines, nodes of the tail
    int first = 0;                     // x node of the half's first velocity, where the head starts
    KGS_HD PackHalf(int v, int n, int nxo)
    {
        if (n <= 0) return;
        first = v % nxo;
        const int to_end = (nxo - first) % nxo;
        head = n < to_end ? n : to_end;
        full = (n - head) / nxo;
        tail = n - head - full * nxo;
    }
};

// Natural places (0 .. count-1, ix fastest) of the slots of one packed velocity
// group that starts at place v0 of its octant, lines of nxo nodes.  Each half
// of the group (the velocities one thread of the moment phase sums) holds the
// two lines of a pair interleaved node by node, then its single units.
inline void pack_order(int v0, int count, int nxo, std::vector<int> &place)
{
    place.clear();
    for (int half = 0; half < 2; half++) {
        const int b = half * PACK_HALF, n = std::min(PACK_HALF, count - b);
        if (n <= 0) break;
        const PackHalf h(v0 + b, n, nxo);
        const int pairs = h.full / 2;
        for (int q = 0; q < pairs; q++)
            for (int ix = 0; ix < nxo; ix++)
                for (int l = 0; l < 2; l++) place.push_back(b + h.head + (2 * q + l) * nxo + ix);
        for (int v = 0; v < h.head; v++) place.push_back(b + v);
        for (int v = h.head + 2 * pairs * nxo; v < n; v++) place.push_back(b + v);
    }
}

}  // namespace kgs
