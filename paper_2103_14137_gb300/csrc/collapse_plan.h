// Which launch makes which levels of the four-wide tree (build_bvh.cu).  Host
// arithmetic only, and plain C++: the tests compile it without CUDA.
#pragma once

#include <cstdint>

namespace uvc {

// Levels [0, top) in one block, [top, tail) one launch each, [tail, levels) in one
// launch of several blocks.  A launch of level L reads counter L and adds to counter L + 1;
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
    // one block for the top (at most 4^4 nodes a level), one launch from four times
    // the depth-balanced tree's nodes on, where a balanced tree has few left
    p.top = 5 < p.levels ? 5 : p.levels;
    p.tail = p.top;
    while (p.tail < p.levels && (p.tail >= 15 || (int64_t(1) << (2 * p.tail)) < 16 * n)) ++p.tail;
    return p;
}

// Blocks of the last launch: a thread for every node that a level may hold (half of
// the leaves), as far as `resident` blocks go.
constexpr int kCollapseThreads = 512;
inline int collapse_blocks(int64_t n, int resident) {
    const int64_t need = (n / 2 + kCollapseThreads - 1) / kCollapseThreads;
    return (int)(need < 1 || resident < 1 ? 1 : (need < resident ? need : resident));
}

}  // namespace uvc
