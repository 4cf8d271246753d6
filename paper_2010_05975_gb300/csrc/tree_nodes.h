// Sizes of a tournament's node lists (host code).
#pragma once
#include <cstddef>

namespace lu {

// Nodes of a tree over `first` first-level nodes, all levels together: a level
// has half the nodes of the one below it, rounded up, so that they sum up to
// 2 first + log2(first) at most.
inline size_t tree_nodes(size_t first) {
    size_t all = first;
    for (size_t n = first; n > 1;) {
        n = (n + 1) / 2;
        all += n;
    }
    return all;
}

// Nodes that the lists and counts of a factorization of m rows with leaves of
// h rows hold: all levels side by side (one launch per tree), or two levels
// in turn (one launch per level).
inline size_t tree_capacity(int m, int h) {
    const int first = m > 0 ? (m - 1) / (h > 0 ? h : 1) + 1 : 1;
    const size_t all = tree_nodes(static_cast<size_t>(first)), two = 2 * static_cast<size_t>(first);
    return all > two ? all : two;
}

}  // namespace lu
