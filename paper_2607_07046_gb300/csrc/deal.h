// How a launch's CTAs are dealt out to the shards that it takes (host only).
#pragma once

#include <algorithm>

namespace vt {

// Deals `ctas` CTAs out to n shards by their bytes: shard s gets end[s] - end[s - 1], at least enough
// for its units at `per` units a CTA, at most one per unit.  Returns the launch's CTAs: more than
// `ctas` only where the units need them.  What the shares' rounding deals too many is taken back from
// the shards that it favoured most: with as many CTAs as fit an SM already there, one more would run
// alone after the others (a two-layer token of fp16 7B shards of 9, 9 and 14 heads: 245 us with 305
// CTAs in the FFN launch and 153 in QKV, 221 with 304 and 152).
inline int deal_ctas(const double* bytes, const int* units, int per, int n, int ctas, int* end) {
    auto need = [&](int s) { return std::max((units[s] + per - 1) / per, 1); };
    double tot = 0;
    for (int s = 0; s < n; ++s) tot += bytes[s];
    int acc = 0;
    for (int s = 0; s < n; ++s) {
        end[s] = std::min(std::max((int)(ctas * bytes[s] / tot + 0.5), need(s)), units[s]);
        acc += end[s];
    }
    for (; acc > ctas; --acc) {
        int most = -1;
        for (int s = 0; s < n; ++s)
            if (end[s] > need(s) && (most < 0 || end[s] - ctas * bytes[s] / tot > end[most] - ctas * bytes[most] / tot)) most = s;
        if (most < 0) break;
        --end[most];
    }
    for (int s = 1; s < n; ++s) end[s] += end[s - 1];
    return end[n - 1];
}

}  // namespace vt
