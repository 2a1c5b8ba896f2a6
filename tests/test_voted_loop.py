"""The loop that the compute threads of the tensor-core forward run in step (csrc/lla_voted_loop.cuh), on host threads: a
wait that runs out in one thread only, in the first, a middle or the last pass, must take all threads out together."""
import shutil
import subprocess

import pytest

from tests.conftest import ROOT

HARNESS = r"""
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <thread>
#include <vector>
#include "lla_voted_loop.cuh"

// barrier with an OR; a thread left waiting for two seconds is a hang
struct Barrier {
    std::mutex mu;
    std::condition_variable cv;
    int size, waiting = 0;
    unsigned phase = 0;
    bool acc = false, result = false;
    explicit Barrier(int n) : size(n) {}
    bool any(bool v) {
        std::unique_lock<std::mutex> lock(mu);
        acc |= v;
        if (++waiting == size) {
            waiting = 0; result = acc; acc = false; ++phase;
            cv.notify_all();
            return result;
        }
        const unsigned mine = phase;
        if (!cv.wait_for(lock, std::chrono::seconds(2), [&] { return phase != mine; })) { std::puts("hang"); std::_Exit(3); }
        return result;
    }
};

int main() {
    constexpr int T = 8, MOST = 5;
    for (int who = -1; who < T; who += 3)
        for (int when = 0; when < MOST; when += 2)
            for (int work = 1; work <= MOST + 1; ++work) {          // passes that thread 3 has work for (the others one)
                Barrier group(T);
                std::vector<Barrier*> pair;
                for (int i = 0; i < T / 2; ++i) pair.push_back(new Barrier(2));
                volatile int marks[2] = {0, 0};
                std::atomic<int> oks{0}, passes{-1}, differ{0};
                std::vector<std::thread> team;
                for (int i = 0; i < T; ++i)
                    team.emplace_back([&, i] {
                        bool ok = true;
                        int done = 0;
                        const int t = lla::voted_loop(
                            MOST, ok, marks, [&] { return done < (i == 3 ? work : 1); },
                            [&](int t) {
                                if (i == who && t == when) ok = false;       // this thread's wait ran out
                                pair[i / 2]->any(false);
                                done = t + 1;
                                return true;
                            },
                            [&](bool v) { return group.any(v); });
                        if (ok) pair[i / 2]->any(false);                     // the output phase has barriers of its own
                        oks += ok;
                        int none = -1;
                        if (!passes.compare_exchange_strong(none, t) && none != t) ++differ;
                    });
                for (auto& th : team) th.join();
                const int most = work < MOST ? work : MOST;
                const bool failed = who >= 0 && when < most;
                if (oks != (failed ? 0 : T) || differ || passes != (failed ? when + 1 : most)) {
                    std::printf("who %d when %d work %d: %d of %d ok, %d passes\n", who, when, work, (int)oks, T, (int)passes);
                    return 1;
                }
            }
    std::puts("fine");
    return 0;
}
"""


def test_threads_leave_together(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "voted_loop.cpp", tmp_path / "voted_loop"
    src.write_text(HARNESS)
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", f"-I{ROOT}/paper_2510_01450_b200/csrc", "-o", str(exe), str(src)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0 and res.stdout.strip() == "fine", (res.returncode, res.stdout)
