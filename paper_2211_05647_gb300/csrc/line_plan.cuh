// line_plan.cuh -- how the 1-D stepping kernel (line1d.cu) divides a line among
// its CTAs.  Host code, standard library only.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

namespace fp {

struct LinePlan {
    std::vector<int32_t> cut, slot_cut;   // range starts, one more than there are CTAs
    int nodes_max = 0, rows_max = 0;
};

// Equal-cost contiguous ranges of the nodes 0 .. nz for `ctas` CTAs (fewer when the line is short: four nodes
// or more each): cut[c] the first node of range c, slot_cut[c] its first plasma slot (cells: the slots' nodes,
// ascending).  Node 0 shares a range with node 1 and node nz with node nz - 1 (the Mur ends).  A row costs row_cost
// nodes.  Each cut is searched for by bisection, since a line of any length is planned before it is known to fit
// (a walk over its nodes took 2.8 s of host time at 10^9 of them, 5 ms at 2 M; this takes microseconds).
inline LinePlan line1d_plan(int64_t nz, const std::vector<int32_t> &cells, int ctas, double row_cost)
{
    LinePlan p;
    const int64_t n = nz + 1, ns = (int64_t)cells.size();
    const int64_t want = std::max<int64_t>(1, std::min<int64_t>(ctas, n / 4));
    const double total = (double)n + row_cost * (double)ns;
    auto slots_below = [&](int64_t c) {   // plasma slots on the nodes before c
        return (int64_t)(std::lower_bound(cells.begin(), cells.end(), c, [](int32_t a, int64_t b) { return a < b; }) -
                         cells.begin());
    };
    p.cut.push_back(0);
    p.slot_cut.push_back(0);
    for (int64_t j = 1; j < want; ++j) {
        // the first cut that leaves j shares of the cost below it
        const double target = total * (double)j / (double)want;
        int64_t lo = std::max<int64_t>((int64_t)p.cut.back() + 1, 2), hi = n;
        while (lo < hi) {
            const int64_t c = lo + (hi - lo) / 2;
            if ((double)c + row_cost * (double)slots_below(c) >= target) hi = c;
            else lo = c + 1;
        }
        if (lo > nz - 1) break;
        p.cut.push_back((int32_t)lo);
        p.slot_cut.push_back((int32_t)slots_below(lo));
    }
    p.cut.push_back((int32_t)n);
    p.slot_cut.push_back((int32_t)ns);
    for (size_t c = 0; c + 1 < p.cut.size(); ++c) {
        p.nodes_max = std::max(p.nodes_max, p.cut[c + 1] - p.cut[c]);
        p.rows_max = std::max(p.rows_max, p.slot_cut[c + 1] - p.slot_cut[c]);
    }
    return p;
}

}  // namespace fp
