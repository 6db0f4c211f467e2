// Sparsity of an assembled operator (host): the node rows of a tetrahedral mesh.
#pragma once

#include <cstdint>
#include <functional>
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

// f(first, last) over [0, n) in contiguous ranges that start at multiples of `align`, on up to
// eight host threads where `work` (elementary steps in all) pays for them.  Exceptions of f
// (of any range) are thrown again here.
void host_ranges(int64_t n, int64_t align, double work, const std::function<void(int64_t, int64_t)>& f);

}  // namespace rve
