// How many inner iterations the host queues between two looks at the solver
// state (graph mode).  Host arithmetic alone: which iterations change
// anything, and their results, do not depend on it.
#pragma once

#include <algorithm>
#include <cmath>

namespace wl {

// One right-hand side at a look.
struct RhsProgress {
    bool active, done, breakdown;
    int iters;                    // iterations of this inner solve
    double rr, target2, delta2;   // ||r||^2, its target, the squared reduction asked for
};

// What an inner solve leaves for the next one of the same mass.
struct InnerPace {
    double rate = 0.0;   // ln of ||r||^2 lost per iteration by the slowest rhs that reached its target (0: none)
    int iters = 0;       // most iterations that such an rhs took
};

// Iterations that take a squared residual down by the factor exp(-lnf).
inline int iterations_for(double lnf, double rate)
{
    const double n = std::ceil(lnf / rate);
    return n >= 1.0 ? (int)std::min(n, 1e6) : 1;
}

// Before the first look: what the pace of the last solve promises, but no more
// than twice the iterations that one took (a pace that no longer holds would
// queue thousands), in any case a block of K; at most `last`.
inline int first_group(const InnerPace &pace, int K, long last, const double *delta2, const int *active, int nrhs)
{
    if (!(pace.rate > 0.0)) return K;
    int group = 1;
    for (int r = 0; r < nrhs; ++r)
        if (active[r]) group = std::max(group, iterations_for(-std::log(delta2[r]), pace.rate));
    return (int)std::min<long>(std::min(group, std::max(K, 2 * pace.iters)), last);
}

// After a look with iterations left: what the slowest rhs still needs at its
// own rate, at most K; K if one makes no progress.
inline int next_group(const RhsProgress *p, int nrhs, int K, long left)
{
    int group = 1;
    for (int r = 0; r < nrhs; ++r) {
        if (!p[r].active || p[r].done || p[r].iters < 1 || !(p[r].rr > 0.0)) continue;
        const double rate = std::log(p[r].target2 / p[r].delta2 / p[r].rr) / p[r].iters;
        group = std::max(group, rate > 0.0 && std::isfinite(rate)
                                    ? std::min(K, iterations_for(std::log(p[r].rr / p[r].target2), rate)) : K);
    }
    return (int)std::min<long>(group, left);
}

// At the end of a solve.  An rhs that broke down or did not reach its target
// says nothing about the next solve.
inline InnerPace learn_pace(const RhsProgress *p, int nrhs)
{
    InnerPace pace;
    for (int r = 0; r < nrhs; ++r) {
        if (!p[r].active || !p[r].done || p[r].breakdown || p[r].iters < 1 || !(p[r].rr > 0.0)) continue;
        const double rate = std::log(p[r].target2 / p[r].delta2 / p[r].rr) / p[r].iters;
        if (!(rate > 0.0) || !std::isfinite(rate)) continue;
        pace.rate = pace.rate > 0.0 ? std::min(pace.rate, rate) : rate;
        pace.iters = std::max(pace.iters, p[r].iters);
    }
    return pace;
}

}  // namespace wl
