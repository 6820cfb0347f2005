// Which launch makes which levels of the four-wide tree (build_bvh.cu).  Host
// arithmetic only, and plain C++: the tests compile it without CUDA.
#pragma once

#include <cstdint>

namespace uvc {

// Levels [0, top) in one block, [top, tail) one launch each, [tail, levels) in
// one block.  A launch of level L reads counter L and adds to counter L + 1;
// `counters` of them are cleared before the first, so 0 <= top <= tail <= levels
// must hold (a level past them would take its node count from memory that
// nothing wrote).
struct CollapsePlan {
    int levels, counters, top, tail;
};

// depth: edges from the root to the deepest of the n leaves.  A path of the
// four-wide tree advances at least one binary level per node.
inline CollapsePlan collapse_plan(int depth, int64_t n) {
    CollapsePlan p;
    p.levels = depth + 1;
    p.counters = p.levels + 1;
    // one block for the top (at most 4^4 nodes a level) and from four times the
    // depth-balanced tree's nodes on, where few are left
    p.top = 5 < p.levels ? 5 : p.levels;
    p.tail = p.top;
    while (p.tail < p.levels && (p.tail >= 15 || (int64_t(1) << (2 * p.tail)) < 16 * n)) ++p.tail;
    return p;
}

}  // namespace uvc
