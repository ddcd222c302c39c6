// fleet_rule.h -- whether a plan's forward-dynamics requests (FP32 data, double-float
// updates) run one thread or three lanes per request; host code without CUDA.
//
// Both forms hand sorted requests to warps, forward dynamics and the longest chains
// first, and both keep about eight workers per SM busy: 32 requests to a warp, or ten
// to a pair of warps. A worker's time is its longest chain's links times a time per
// link, so the two compare as list schedules of their forward-dynamics items over 8
// workers per SM, and not below the whole work, inverse dynamics included, over the
// workers. Times per link in us, fitted to plans on GB300 (chains of 1..2 to 100..128
// links, 1 to 250 000 requests): one thread 4.9, 9.2 with double-float bias sweeps, a
// third more where a plan needs both bodies (their code competes for the instruction
// cache); three lanes 3.3 and 4.5; 32 inverse-dynamics requests 0.9 to 1.3 in either.
// us, one thread / three lanes: n = 7, 12 000 requests 38 / 27, 30 000 41 / 62, 60 000 66 /
// 99; 6..30, 18 240 143 / 88, 60 000 184 / 259; 32, 12 000 166 / 96, 30 000 182 / 270;
// 60..64, 12 000 331 / 192, 30 000 372 / 536; 6..100, 30 000 1110 / 537, 120 000 1931 / 2096;
// 100..128, 12 000 1160 / 603, 30 000 1216 / 1557; one in five forward dynamics, 120 000
// requests: n = 7 41 / 57, 32 202 / 348, 6..100 1057 / 591.
#pragma once
#include <algorithm>
#include <functional>
#include <queue>
#include <vector>

// Finishing time of items handed in order to whichever of `workers` is free first.
inline double rd_list_schedule(const std::vector<double> &items, int workers)
{
    double last = 0;
    std::priority_queue<double, std::vector<double>, std::greater<double>> free_at;
    for (double t : items) {
        double start = 0;
        if ((int)free_at.size() >= workers) {
            start = free_at.top();
            free_at.pop();
        }
        free_at.push(start + t);
        last = std::max(last, start + t);
    }
    return last;
}

// fd, id: the links of the plan's forward- and inverse-dynamics chains, longest first;
// ext_groups: how many groups of 32 forward-dynamics positions run their bias sweeps in
// double-float; per: requests of a three-lane unit.
inline bool rd_fleet_takes_lanes(const std::vector<int> &fd, const std::vector<int> &id, int ext_groups,
                                 int per, int sms)
{
    const int workers = 8 * sms;
    // No forward dynamics: the three-lane kernel, whose blocks put twice as many warps on
    // an SM, only where many short rows queue for them (us, one-thread kernel / this: 1..2
    // links, 60 000 requests 10.3 / 8.3; 3..5, 9000 8.6 / 10.1, 120 000 21.5 / 16.6). Longer
    // rows lose each other's lines in L1 (7, 60 000 17.7 / 20.7; 32, 30 000 46 / 65).
    if (fd.empty()) return !id.empty() && id[0] <= 5 && id.size() > 32 * (size_t)workers;
    double rest = 0;
    for (size_t k = 0; k < id.size(); k += 32) rest += id[k] * (0.9 + 0.4 * std::min(1.0, id[k] / 32.0));
    auto time = [&](size_t step, double each, double each_ext) {
        std::vector<double> items;
        double sum = rest;
        for (size_t k = 0; k < fd.size(); k += step) {
            items.push_back(fd[k] * ((int)(k / 32) < ext_groups ? each_ext : each));
            sum += items.back();
        }
        return std::max(rd_list_schedule(items, workers), sum / workers);
    };
    const bool both = ext_groups > 0 && (size_t)ext_groups * 32 < fd.size();
    const double slower = both ? 1.3 : 1.0;
    return time((size_t)per, 3.3, 4.5) <= time(32, 4.9 * slower, 9.2 * slower);
}
