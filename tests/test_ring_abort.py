"""Lanes of a warp that give up a wait in different iterations of the plane loop all leave it
(csrc/ring.cuh, built for the host): threads for lanes, a counting barrier for __syncwarp."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1807_03032_gb300", "csrc")

MAIN = r"""
#include <stdio.h>
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <mutex>
#include <thread>
#include <vector>
#include "ring.cuh"

constexpr int kLanes = 4, kPlanes = 6, kNever = 99;

struct Warp {  // __syncwarp() of kLanes lanes; a lane that waits a second gives up
    std::mutex mu;
    std::condition_variable cv;
    int inside = 0, round = 0;
    bool hung = false;
    void sync() {
        std::unique_lock<std::mutex> lk(mu);
        const int r = round;
        if (++inside == kLanes) {
            inside = 0;
            ++round;
            cv.notify_all();
        } else if (!cv.wait_for(lk, std::chrono::seconds(1), [&] { return round != r; })) {
            hung = true;
        }
    }
};

// fail[i]: the iteration in which lane i's wait runs out
bool leaves(const int *fail) {
    Warp w;
    std::atomic<int> aborted{0};
    volatile unsigned char left = 0;
    std::atomic<int> out{0};
    auto lane = [&](int i) {
        for (int j = 0; j < kPlanes; ++j) {
            if (aborted || j >= fail[i]) {
                aborted = 1;
                fdsweep::meet_remaining_lanes(&left, j, [&] { w.sync(); });
                break;
            }
            w.sync();
            if (w.hung) return;
        }
        ++out;
    };
    std::vector<std::thread> t;
    for (int i = 0; i < kLanes; ++i) t.emplace_back(lane, i);
    for (auto &x : t) x.join();
    return !w.hung && out == kLanes;
}

int main() {
    const int when[] = {0, 1, 2, 5, kNever};
    for (int rep = 0; rep < 3; ++rep)
        for (int c = 0; c < 5 * 5 * 5 * 5; ++c) {
            const int fail[kLanes] = {when[c % 5], when[c / 5 % 5], when[c / 25 % 5],
                                      when[c / 125]};
            if (!leaves(fail)) {
                printf("hangs: %d %d %d %d\n", fail[0], fail[1], fail[2], fail[3]);
                return 1;
            }
        }
    return 0;
}
"""


def test_lanes_that_give_up_at_different_planes_all_leave(tmp_path):
    src, exe = str(tmp_path / "ring.cpp"), str(tmp_path / "ring")
    with open(src, "w") as f:
        f.write(MAIN)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", CSRC, src, "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
