// batch_lanes.h -- which of a batch's streams ("lanes") each system's sweep goes to (plain C++).
//
// With every system on a stream of its own, the light systems' small blocks can be placed first, in a
// graph above all, and an L = 64 block, which takes an SM's whole shared memory, waits for them: 27 ms
// for 20 iterations of 10 sweeps of the nine-system mix as a graph, where the L = 64 chain and the
// updates take 19.  So a system that finds no SMs beside the heavier ones queues behind the lane that
// ends first (21.4 ms), but only where that is estimated to end no later: three equal systems of 100
// blocks, one an SM, fill two waves of 152 SMs side by side and take three rounds in a queue (28.7 and
// 42.7 ms for five iterations of 100 sweeps of 8-Potts L = 32).  Where the estimates are equal and the
// queued system would be the last to end, it queues behind a longer one only (9000 walkers each of
// 8-Potts L = 32, 80 sweeps, Ising L = 64, 20, and L = 16, 200: 26.4 ms, 28.8 side by side); behind its
// like it would wait for that one's last block instead of the first that ends (six Ising L = 16 of 64
// blocks, two an SM, 200 sweeps: 18.4 ms, 14.8 side by side).
#pragma once
#include <algorithm>
#include <vector>

namespace muca {

struct LaneSystem {
    int blocks;    // thread blocks of the system's sweep
    int per_sm;    // of which an SM holds this many (registers, threads and shared memory)
    double cost;   // time of one block
    bool polymer;  // many small warps that gain from lying beside others: always a lane of its own
    bool operator==(const LaneSystem &o) const
    {
        return blocks == o.blocks && per_sm == o.per_sm && cost == o.cost && polymer == o.polymer;
    }
};

// Estimated end of the lattice sweeps of `sys` (heaviest first) on `nsm` SMs, system r on lane
// lane[r]: a lane's systems one after the other, ready blocks placed in order as SMs come free.
// last: the end of the last of them.
inline double lanes_end(const std::vector<LaneSystem> &sys, const std::vector<int> &lane, int nsm, double *last = nullptr)
{
    struct Running {
        double end, sms;
        int r, n;
    };
    const int n = (int)lane.size();
    std::vector<int> todo(n), flying(n, 0), before(n, -1);  // before: the lane's previous system
    for (int r = 0; r < n; ++r) {
        todo[r] = sys[r].polymer ? 0 : sys[r].blocks;
        for (int q = r - 1; q >= 0 && before[r] < 0; --q)
            if (lane[q] == lane[r]) before[r] = q;
    }
    std::vector<Running> run;
    double t = 0.0, free_sms = nsm;
    while (true) {
        for (int r = 0; r < n; ++r) {
            if (todo[r] == 0 || (before[r] >= 0 && (todo[before[r]] || flying[before[r]]))) continue;
            const int k = std::min(todo[r], (int)(free_sms * sys[r].per_sm + 1e-6));
            if (k < 1) continue;
            todo[r] -= k;
            flying[r] += k;
            free_sms -= (double)k / sys[r].per_sm;
            run.push_back({t + sys[r].cost, (double)k / sys[r].per_sm, r, k});
        }
        if (run.empty()) return t;
        t = run[0].end;
        for (const Running &x : run) t = std::min(t, x.end);
        for (size_t i = 0; i < run.size();) {
            if (run[i].end <= t) {
                free_sms += run[i].sms;
                flying[run[i].r] -= run[i].n;
                if (last && run[i].r == n - 1) *last = t;
                run[i] = run.back();
                run.pop_back();
            } else {
                ++i;
            }
        }
    }
}

// Lane of every system, by its place in `sys` (heaviest first).
inline std::vector<int> plan_lanes(const std::vector<LaneSystem> &sys, int nsm)
{
    std::vector<int> lane, own;
    std::vector<double> end, tail;  // of each lane: its systems as if alone, its last one
    std::vector<bool> open;   // whether lattice systems may queue there
    double free_sms = nsm;
    for (size_t r = 0; r < sys.size(); ++r) {
        own.push_back((int)r);
        const double sms = (double)sys[r].blocks / sys[r].per_sm;
        int best = -1;
        for (int l = 0; l < (int)end.size(); ++l)
            if (open[l] && (best < 0 || end[l] < end[best])) best = l;
        lane.push_back((int)end.size());
        // (a system that mostly fits starts too: its last blocks follow the first that end)
        if (!sys[r].polymer && best >= 0 && sms > 1.5 * free_sms) {
            std::vector<int> queued = lane;
            queued.back() = best;
            double last = 0.0;
            const double own_end = lanes_end(sys, lane, nsm), queue_end = lanes_end(sys, queued, nsm, &last);
            if (queue_end < own_end || (queue_end == own_end && (last < queue_end || sys[r].cost < 0.9 * tail[best]))) {
                lane = queued;
                end[best] += sys[r].cost;
                tail[best] = sys[r].cost;
                continue;
            }
        }
        end.push_back(sys[r].cost);
        tail.push_back(sys[r].cost);
        open.push_back(!sys[r].polymer);
        if (!sys[r].polymer) free_sms = std::max(0.0, free_sms - sms);
    }
    return lanes_end(sys, lane, nsm) <= lanes_end(sys, own, nsm) ? lane : own;
}

}  // namespace muca
