// Sparsity of an assembled operator (host); see node_graph.h.
#include "node_graph.h"

#include <algorithm>
#include <exception>
#include <mutex>
#include <thread>

namespace rve {

// A mesh's first solve waits for its sparsity.  First solve of 40x40x16, p = 1, mixed (25 600
// nodes, 0.44 million entries): 34.2 ms with one thread, 30.6 with up to eight; 24x24x8, p = 2,
// FP64 (36 864, 1.18 million): 30.1 and 25.2.  A thread costs about 30 us to start, 2e5 steps
// about 0.5 ms.
void host_ranges(int64_t n, int64_t align, double work, const std::function<void(int64_t, int64_t)>& f) {
    const int64_t blocks = (n + align - 1) / align;
    const int64_t most = std::min<int64_t>(8, std::max(1u, std::thread::hardware_concurrency()));
    const int T = (int)std::max<int64_t>(1, std::min({most, blocks, (int64_t)(work / 2e5)}));
    auto at = [&](int t) { return std::min(n, blocks * t / T * align); };
    if (T == 1) return f(0, n);
    std::exception_ptr error;
    std::mutex mu;
    auto part = [&](int t) {
        try {
            f(at(t), at(t + 1));
        } catch (...) {
            std::lock_guard<std::mutex> lock(mu);
            if (!error) error = std::current_exception();
        }
    };
    std::vector<std::thread> threads;
    threads.reserve(T);
    int started = 1;   // (range 0 runs here)
    try {
        for (; started < T; ++started) threads.emplace_back(part, started);
    } catch (...) {   // no more threads to be had: the other ranges run here
    }
    part(0);
    for (int t = started; t < T; ++t) part(t);
    for (auto& th : threads) th.join();
    if (error) std::rethrow_exception(error);
}

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
    g.ptr.assign(n + 1, 0);
    if (phase) g.split.assign(n, 0);
    // the rows of a range into a list of their own; ptr[i + 1] and split[i] hold the lengths
    // (of the row, of its phase-0 part) until all are known
    struct Part {
        int64_t first;
        std::vector<int32_t> col;
    };
    std::vector<Part> parts;
    std::mutex mu;
    const double steps = (double)nt * ne * ne;
    host_ranges(n, 1, steps, [&](int64_t lo, int64_t hi) {
        Part p{lo, {}};
        p.col.reserve((size_t)(g.eptr[hi] - g.eptr[lo]) * (phase ? 6 : 3));
        std::vector<int32_t> seen(n, -1);   // last row and phase (2 row + phase) that listed the node
        for (int64_t i = lo; i < hi; ++i) {
            const size_t begin = p.col.size();
            for (int ph = 0; ph < (phase ? 2 : 1); ++ph) {
                if (ph == 1) g.split[i] = (int32_t)(p.col.size() - begin);
                const int32_t mark = (int32_t)(2 * (i % ((int64_t)1 << 30)) + ph);
                for (int32_t q = g.eptr[i]; q < g.eptr[i + 1]; ++q) {
                    const int64_t e = g.inc[q] / ne;
                    if (phase && (phase[e] != 0) != (ph == 1)) continue;
                    for (int b = 0; b < ne; ++b) {
                        const int32_t c = edofs[e * ne + b];
                        if (seen[c] == mark) continue;
                        seen[c] = mark;
                        p.col.push_back(c);
                    }
                }
            }
            g.ptr[i + 1] = (int32_t)(p.col.size() - begin);
        }
        std::lock_guard<std::mutex> lock(mu);
        parts.push_back(std::move(p));
    });
    int64_t total = 0;
    for (const Part& p : parts) total += (int64_t)p.col.size();
    if (total > most) return false;
    for (int64_t i = 0; i < n; ++i) {
        if (phase) g.split[i] += g.ptr[i];
        g.ptr[i + 1] += g.ptr[i];
    }
    if (parts.size() == 1) {
        g.col = std::move(parts[0].col);
        return true;
    }
    g.col.resize(total);
    host_ranges((int64_t)parts.size(), 1, steps, [&](int64_t lo, int64_t hi) {
        for (int64_t k = lo; k < hi; ++k)
            std::copy(parts[k].col.begin(), parts[k].col.end(), g.col.begin() + g.ptr[parts[k].first]);
    });
    return true;
}

}  // namespace rve
