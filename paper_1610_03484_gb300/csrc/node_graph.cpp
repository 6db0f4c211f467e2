// Sparsity of an assembled operator (host); see node_graph.h.
#include "node_graph.h"

namespace rve {

bool build_node_graph(const int32_t* edofs, int64_t nt, int ne, const uint8_t* phase, int64_t n, NodeGraph& g) {
    const int64_t most = ((int64_t)1 << 31) - 1;
    if (nt * ne > most || n > most) return false;
    g = NodeGraph();
    g.n = n;
    g.eptr.assign(n + 1, 0);
    for (int64_t k = 0; k < nt * ne; ++k) ++g.eptr[edofs[k] + 1];
    for (int64_t i = 0; i < n; ++i) g.eptr[i + 1] += g.eptr[i];
    g.inc.resize(nt * ne);
    {
        std::vector<int32_t> at(g.eptr.begin(), g.eptr.end() - 1);
        for (int64_t k = 0; k < nt * ne; ++k) g.inc[at[edofs[k]]++] = (int32_t)k;
    }
    g.ptr.resize(n + 1);
    if (phase) g.split.resize(n);
    g.col.reserve((size_t)nt * ne * (phase ? 6 : 3));
    std::vector<int32_t> seen(n, -1);   // last row and phase (2 row + phase) that listed the node
    for (int64_t i = 0; i < n; ++i) {
        if ((int64_t)g.col.size() > most - 4096) return false;
        g.ptr[i] = (int32_t)g.col.size();
        for (int ph = 0; ph < (phase ? 2 : 1); ++ph) {
            if (phase && ph == 1) g.split[i] = (int32_t)g.col.size();
            const int32_t mark = (int32_t)(2 * (i % ((int64_t)1 << 30)) + ph);
            for (int32_t q = g.eptr[i]; q < g.eptr[i + 1]; ++q) {
                const int64_t e = g.inc[q] / ne;
                if (phase && (phase[e] != 0) != (ph == 1)) continue;
                for (int b = 0; b < ne; ++b) {
                    const int32_t c = edofs[e * ne + b];
                    if (seen[c] == mark) continue;
                    seen[c] = mark;
                    g.col.push_back(c);
                }
            }
        }
    }
    g.ptr[n] = (int32_t)g.col.size();
    return (int64_t)g.col.size() <= most;
}

}  // namespace rve
