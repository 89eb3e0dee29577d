"""The block queue of the inversion kernels (csrc/pr_queue.cuh), compiled for
the host: two warps of 32 lanes as two threads that run their lanes one after
the other between barriers, as a scheduler that holds one warp back may.  After
every barrier one warp waits until the other has reached its next one.  Every
warp has to meet the other at the same barrier, and every pushed entry has to
be finished once."""
import subprocess

import pytest

from paper_2312_04830_gb300 import build

SRC = r"""
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <thread>
#include <vector>

// Two warps; `late` is let past a barrier only when the other one waits at its
// next barrier or has ended.
static std::mutex mu;
static std::condition_variable cv;
static int late, gen = 0, waiting = 0, site_of[2], mismatch = 0;
static bool at_barrier[2], ended[2];
static thread_local int me;

static void barrier_at(int site)
{
    std::unique_lock<std::mutex> l(mu);
    site_of[me] = site;
    at_barrier[me] = true;
    const int g = gen;
    if (++waiting == 2) {
        if (site_of[0] != site_of[1]) mismatch = 1;
        waiting = 0;
        at_barrier[0] = at_barrier[1] = false;
        ++gen;
        cv.notify_all();
    } else {
        cv.notify_all();
        cv.wait(l, [&] { return gen != g || ended[1 - me]; });
        if (gen == g) { mismatch = 2; std::printf("a warp waits alone\n"); std::fflush(stdout); std::_Exit(1); }
    }
    if (me == late) cv.wait(l, [&] { return at_barrier[1 - me] || ended[1 - me]; });
}
#define PRQ_BARRIER() barrier_at(__COUNTER__)
#include "pr_queue.cuh"

// One warp-wide call of the queue per warp: the lanes' entries are finished in
// a loop, as the lanes of a warp do together.
constexpr int kLanes = 32, kThreads = 64;
static int q_n = 0, entry[2 * kThreads];
static std::vector<int> done;

static void warp(int w, const std::vector<std::vector<int>> &rounds)
{
    me = w;
    auto finish = [&](int first) {   // first: the entry of the warp's lane 0
        for (int l = 0; l < kLanes; ++l) {
            std::lock_guard<std::mutex> g(mu);
            ++done[entry[first + l]];
        }
    };
    int cell = 0;
    for (const auto &r : rounds) {
        for (int l = 0; l < r[w]; ++l) {   // the first r[w] lanes push
            std::lock_guard<std::mutex> g(mu);
            const int e = q_n++;
            if (e >= 2 * kThreads) { std::printf("queue overrun\n"); std::fflush(stdout); std::_Exit(1); }
            entry[e] = cell + w * kLanes + l;
        }
        prk::queue_round(&q_n, w * kLanes, kThreads, finish);
        cell += kThreads;
    }
    prk::queue_rest(&q_n, w * kLanes, [&](int first) {
        for (int l = 0; l < kLanes && first + l < q_n; ++l) {
            std::lock_guard<std::mutex> g(mu);
            ++done[entry[first + l]];
        }
    });
    std::lock_guard<std::mutex> g(mu);
    ended[w] = true;
    cv.notify_all();
}

int main(int argc, char **argv)
{
    late = std::atoi(argv[1]);
    std::vector<std::vector<int>> rounds;
    for (int a = 2; a + 1 < argc; a += 2) rounds.push_back({std::atoi(argv[a]), std::atoi(argv[a + 1])});
    done.assign(rounds.size() * kThreads, 0);
    std::thread t0(warp, 0, std::cref(rounds)), t1(warp, 1, std::cref(rounds));
    t0.join();
    t1.join();
    int bad = mismatch;
    for (size_t r = 0; r < rounds.size(); ++r)
        for (int w = 0; w < 2; ++w)
            for (int l = 0; l < kLanes; ++l) bad |= done[r * kThreads + w * kLanes + l] != (l < rounds[r][w]);
    std::printf(bad ? "wrong\n" : "ok\n");
    return bad != 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    d = tmp_path_factory.mktemp("queue")
    (d / "q.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", build.CSRC, "-o", str(d / "q"), str(d / "q.cpp")],
                   check=True)
    return str(d / "q")


# lanes that push in each round, warp by warp: below a block's worth, one and
# more, a round that reaches it by the other warp's pushes alone, none
@pytest.mark.parametrize("rounds", [[(32, 0), (32, 0), (0, 0)], [(0, 32), (0, 32), (5, 7)], [(31, 32), (32, 32), (32, 32)],
                                    [(32, 32)] * 4, [(20, 11), (32, 32), (0, 1)], [(0, 0), (1, 0)]])
@pytest.mark.parametrize("late", [0, 1])
def test_every_entry_once_and_barriers_together(exe, rounds, late):
    args = [str(v) for r in rounds for v in r]
    r = subprocess.run([exe, str(late), *args], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
