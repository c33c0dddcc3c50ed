// line_plan.cuh -- how the 1-D stepping kernel (line1d.cu) divides a line among
// its CTAs.  Host code, standard library only.
#pragma once

#include <algorithm>
#include <cmath>
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
// nodes.  The cost below a cut is linear between plasma slots, so each cut is found among the slots by bisection and
// then by its distance from one: a line of any length is planned before it is known to fit, and the first step of a
// short one waits for it (a walk over the nodes took 2.8 s of host time at 10^9 of them, 5 ms at 2 M and 5 us at 2000;
// this takes microseconds).
inline LinePlan line1d_plan(int64_t nz, const std::vector<int32_t> &cells, int ctas, double row_cost)
{
    LinePlan p;
    const int64_t n = nz + 1, ns = (int64_t)cells.size();
    const int64_t want = std::max<int64_t>(1, std::min<int64_t>(ctas, n / 4));
    const double total = (double)n + row_cost * (double)ns;
    auto cost = [&](int64_t c, int64_t s) { return (double)c + row_cost * (double)s; };   // c nodes, s of them plasma
    p.cut.push_back(0);
    p.slot_cut.push_back(0);
    int64_t s = 0;   // the first slot with which the cost reaches the target
    for (int64_t j = 1; j < want; ++j) {
        const double target = total * (double)j / (double)want;   // j shares below the cut
        auto reached = [&](int64_t q) { return cost((int64_t)cells[(size_t)q] + 1, q + 1) >= target; };
        int64_t hi = s, step = 1;   // (in growing steps from the last one, then by bisection)
        while (hi < ns && !reached(hi)) {
            s = hi + 1;
            hi = std::min(hi + step, ns);
            step *= 2;
        }
        while (s < hi) {
            const int64_t m = s + (hi - s) / 2;
            if (reached(m)) hi = m;
            else s = m + 1;
        }
        // the cut lies among the nodes before that slot's, or just after it
        int64_t c = std::max<int64_t>((int64_t)std::ceil(target - row_cost * (double)s), 0), below = s;
        while (cost(c, s) < target) ++c;
        if (s < ns && c > cells[(size_t)s]) {
            c = (int64_t)cells[(size_t)s] + 1;
            below = s + 1;
        }
        const int64_t least = std::max<int64_t>((int64_t)p.cut.back() + 1, 2);
        if (c < least) {
            c = least;
            below = std::lower_bound(cells.begin(), cells.end(), (int32_t)c) - cells.begin();
        }
        if (c > nz - 1) break;
        p.cut.push_back((int32_t)c);
        p.slot_cut.push_back((int32_t)below);
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
