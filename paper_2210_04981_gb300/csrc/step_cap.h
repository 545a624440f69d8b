// Step cap of a traversal (plain C++, no CUDA types).
#pragma once

#include <climits>
#include <cstdint>

namespace hdof {

// trav_cap, or 64 steps per node and triangle where it is 0 (or less).  A tree
// of 2^27 triangles passes 2^31 that way: counted in 64 bits, and at most
// INT_MAX - 1, so that a kernel's step count can pass it.
inline int step_cap(int32_t trav_cap, int64_t n_nodes, int64_t n_tris) {
    const int64_t cap = trav_cap > 0 ? (int64_t)trav_cap : 64 * (n_nodes + n_tris) + 64;
    return (int)(cap < INT_MAX ? cap : INT_MAX - 1);
}

}  // namespace hdof
