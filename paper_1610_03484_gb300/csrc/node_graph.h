// Sparsity of an assembled operator (host): the node rows of a tetrahedral mesh.
#pragma once

#include <cstdint>
#include <vector>

namespace rve {

// Row i (a scalar DOF node) couples to every node that shares an element with it.
// With phases given, a pair is listed once for phase 0 and once for phase 1 where
// elements of both contribute, all phase-0 entries of a row first.
struct NodeGraph {
    int64_t n = 0;
    std::vector<int32_t> ptr;     // [n + 1] first entry of each row
    std::vector<int32_t> split;   // [n] first phase-1 entry of each row (phases given)
    std::vector<int32_t> col;     // entry -> coupled node
    std::vector<int32_t> eptr;    // [n + 1] first incidence of each node
    std::vector<int32_t> inc;     // incidence: element * ne + local function
};

// False when an index would not fit in 32 bits.
bool build_node_graph(const int32_t* edofs, int64_t nt, int ne, const uint8_t* phase, int64_t n, NodeGraph& g);

}  // namespace rve
