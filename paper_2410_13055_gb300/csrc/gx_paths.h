// Which scenarios run in clusters and when a loop pauses to change that: the host's arithmetic on
// the scenarios' launch choices (gx_host.cu), without CUDA.
//
// A choice has `us`, its estimated time per iteration, and `room`, the share of the device that one
// such cluster takes; a scenario's list has them by cluster size, ascending.  The searches run before
// every loop, so none of them may grow with the square of the scenario count.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <queue>
#include <utility>
#include <vector>

namespace gx {

// Estimated microseconds of one iteration of the per-iteration kernels over dh device-hours: three
// dependent launches (10 to 11 us for one scenario of any size here), then 3.3 to 3.6 us per million
// device-hours (100 buses, 168 h: 10.9 us for 2 scenarios, 15.4 for 16).
inline double stream_us(double dh) { return 10.0 + 3.5e-6 * dh; }

// The time between two pauses of resident loops.  A pause costs about 43 us (a launch, the state out
// and in, a look at the done flags), so it comes after at least
constexpr double kCrsPause = 800.0;
// microseconds, and a share of the time spent so far, as what is left to gain shrinks against it.
constexpr double kCrsPauseShare = 0.125;
// 16 x 168 h of 100 buses, plan steps and dispatches from nothing, eight sets of inputs: 121.8 and
// 127.5 ms; 600 us 122.1 and 129.6, 500 us with a share of a quarter 121.3 and 130.2; on five of the
// sets 71.8 and 77.4, without pauses 99.0 and 86.4.  (A pause as soon as few enough were left, which
// depended on how far each cluster had got: 118.5 and 123.1.)

// Clusters of mixed sizes leave gaps in the processing clusters that hold them.
inline double crs_room_limit(bool one_list) { return one_list ? 1.0 + 1e-9 : 0.9; }

// The most of the first scenarios whose smallest clusters fit the device side by side.
template <class Choice>
size_t crs_fit_prefix(const std::vector<const std::vector<Choice>*>& ch) {
    double room = 0;
    bool one = true;
    for (size_t i = 0; i < ch.size(); ++i) {
        room += (*ch[i])[0].room;
        one = one && ch[i] == ch[0];
        if (room > crs_room_limit(one)) return i;
    }
    return ch.size();
}

// A choice for each of the first n scenarios, all of which have some: each starts from its
// smallest cluster, then the slowest is enlarged while the device still holds all of them side by
// side (scenarios of one list take one choice).  Returns the estimated time per iteration, that
// of the slowest; *fits: whether the smallest clusters already fit side by side.
template <class Choice>
double crs_assign(const std::vector<const std::vector<Choice>*>& ch, size_t n, std::vector<size_t>& at, bool* fits) {
    at.assign(n, 0);
    double room = 0, us = 0;
    bool one = true;
    for (size_t i = 0; i < n; ++i) {
        one = one && ch[i] == ch[0];
        room += (*ch[i])[0].room;
    }
    const double limit = crs_room_limit(one);
    *fits = room <= limit;
    if (one) {
        size_t best = 0;
        for (size_t k = 1; n > 0 && k < ch[0]->size(); ++k)
            if ((double)n * (*ch[0])[k].room <= limit) best = k;
        std::fill(at.begin(), at.end(), best);
        return n > 0 ? (*ch[0])[best].us : 0.0;
    }
    if (!*fits) {
        for (size_t i = 0; i < n; ++i) us = std::max(us, (*ch[i])[0].us);
        return us;
    }
    std::priority_queue<std::pair<double, long>> slowest;  // (of equal ones the first)
    for (size_t i = 0; i < n; ++i) slowest.push({(*ch[i])[0].us, -(long)i});
    for (;;) {
        const size_t w = (size_t)-slowest.top().second;
        us = slowest.top().first;
        if (at[w] + 1 >= ch[w]->size()) return us;
        const double more = (*ch[w])[at[w] + 1].room - (*ch[w])[at[w]].room;
        if (room + more > limit) return us;
        room += more;
        slowest.pop();
        slowest.push({(*ch[w])[++at[w]].us, -(long)w});
    }
}

// The most scenarios left at which the per-iteration loop pauses for clusters: of `ch`, those that
// have choices, by room descending, with their device-hours dh, and at most `most` of them.  As
// many of the largest as fit, stepped down while clusters are not estimated faster (one by one up
// to 64, by eighths above; 0: never).
template <class Choice>
size_t crs_pause_at(const std::vector<const std::vector<Choice>*>& ch, const std::vector<double>& dh, size_t most) {
    const size_t n = std::min(most, crs_fit_prefix(ch));
    std::vector<double> sum(n + 1, 0.0), least(n + 1, 0.0);  // of the first k: device-hours, a bound on the time
    for (size_t k = 0; k < n; ++k) {
        sum[k + 1] = sum[k] + dh[k];
        least[k + 1] = std::max(least[k], ch[k]->back().us);
    }
    std::vector<size_t> at;
    bool fits;
    for (size_t k = n; k >= 1; k = k > 64 ? k * 7 / 8 : k - 1) {
        const double limit = 0.95 * stream_us(sum[k]);
        if (least[k] < limit && crs_assign(ch, k, at, &fits) < limit && fits) return k;
    }
    return 0;
}

// The most of n scenarios in clusters at which those left gain a tenth from larger ones: of `ch`,
// by the time of their smallest cluster descending (0: never).
template <class Choice>
size_t crs_regroup_at(const std::vector<const std::vector<Choice>*>& ch, double us) {
    if (ch.size() < 2) return 0;
    std::vector<size_t> at;
    bool fits;
    for (size_t k = std::min(ch.size() - 1, crs_fit_prefix(ch)); k >= 1; k = k > 8 ? k * 7 / 8 : k - 1)
        if (crs_assign(ch, k, at, &fits) < 0.9 * us && fits) return k;
    return 0;
}

// Where a scenario pauses: after `part` microseconds at `us` an iteration, rounded up to residual
// checks, and at the cap at the latest.
inline int crs_pause_end(int it, double us, double part, int every, int max_it) {
    const double checks = std::max(1.0, std::ceil(part / (us * every)));
    return checks * every < (double)(max_it - it) ? it + (int)checks * every : max_it;
}

}  // namespace gx
