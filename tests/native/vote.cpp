// warp_ready with 32 threads for lanes: for every mix of lanes that see the counter at once,
// late, or never, all lanes vote the same number of times and get the same answer.
#include <atomic>
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <random>
#include <thread>
#include <vector>

#include "ptebd_vote.h"

constexpr int kLanes = 32;

struct Warp {
    std::mutex mu;
    std::condition_variable cv;
    int arrived = 0, left = 0, round = 0;
    bool all = true, result = true;
    // like a vote over the full warp: completes when every lane has come
    bool vote(bool x) {
        std::unique_lock<std::mutex> lock(mu);
        all = all && x;
        if (++arrived == kLanes - left) {
            result = all;
            all = true;
            arrived = 0;
            ++round;
            cv.notify_all();
            return result;
        }
        const int mine = round;
        cv.wait(lock, [&] { return round != mine; });
        return result;
    }
    void leave() {
        std::lock_guard<std::mutex> lock(mu);
        ++left;
        if (arrived && arrived == kLanes - left) {
            result = all;
            all = true;
            arrived = 0;
            ++round;
            cv.notify_all();
        }
    }
};

// what: per lane 0 = sees the counter at once, 1 = only by waiting, 2 = its wait runs out
bool same_on_all_lanes(const std::vector<int>& what) {
    Warp w;
    std::vector<int> votes(kLanes, 0), answer(kLanes, -1);
    std::vector<std::thread> lanes;
    for (int l = 0; l < kLanes; ++l)
        lanes.emplace_back([&, l] {
            answer[l] = ptebd::warp_ready(what[l] == 0, [&](bool x) { ++votes[l]; return w.vote(x); },
                                          [&] { return what[l] == 1; });
            w.leave();
        });
    for (auto& t : lanes) t.join();
    bool never = false;
    for (int x : what) never = never || x == 2;
    for (int l = 0; l < kLanes; ++l)
        if (votes[l] != votes[0] || answer[l] != (never ? 0 : 1)) return false;
    return true;
}

int main() {
    std::mt19937 rng(1);
    for (int kinds = 1; kinds <= 3; ++kinds)
        for (int i = 0; i < 40; ++i) {
            std::vector<int> what(kLanes);
            for (int& x : what) x = (int)(rng() % kinds);
            if (i == 0) what.assign(kLanes, kinds - 1);
            if (i == 1) { what.assign(kLanes, 0); what[rng() % kLanes] = kinds - 1; }
            if (!same_on_all_lanes(what)) {
                std::printf("lanes disagree (%d kinds, mix %d)\n", kinds, i);
                return 1;
            }
        }
    return 0;
}
