// How the Leduc kernels split a pair's hands into work units.
#pragma once

#include <cstdint>

namespace malib {

// Of lo .. hi segments per pair (hi >= lo >= 1) those with the smallest estimated
// time: a phase of a unit costs `phase`, and `tile` per `rows` hands that act in it,
// about these shares of the unit's; the units go over n_sm SMs in waves. Among the
// numbers of segments that make as many waves the largest is taken: it has the
// smallest units (one bf16 pair x 200,000 hands: 152 units of 1,316 hands 150.6 us, the
// fewest of the same estimate, 143 of 1,399, 155.9), and it alone need be looked at.
inline int64_t cheapest_segments(int32_t n_pairs, int64_t n_hands, int n_sm, int64_t lo, int64_t hi, double phase,
                                 double tile, double rows) {
    static const double share[8] = {1.0, 1.0, 0.8, 0.6, 0.4, 0.25, 0.1, 0.05};
    const auto waves = [&](int64_t seg) { return ((int64_t)n_pairs * seg + n_sm - 1) / n_sm; };
    const auto cost = [&](int64_t seg) {
        const int64_t per = (n_hands + seg - 1) / seg;
        double c = 0.0;
        for (double sh : share) c += phase + tile * (double)(int64_t)((double)per * sh / rows + 0.999);
        return c * (double)waves(seg);
    };
    int64_t best = lo;
    double best_cost = 1e300;
    for (int64_t from = lo, to; from <= hi; from = to + 1) {
        to = waves(from) * n_sm / n_pairs;               // the last of as many waves
        if (to > hi) to = hi;
        const double c = cost(to);
        if (c < best_cost) {
            best_cost = c;
            best = to;
        }
    }
    return best;
}

}  // namespace malib
