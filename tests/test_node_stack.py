"""A line's step from one wide node to the next (csrc/node_stack.cuh), built as
plain C++ on the host, for four lanes that follow one line together, a thread
per lane.  The only barrier is between turns: within a turn each lane runs alone,
lane 0 first, the order that shows a lane reading what another wrote in the same
turn.  Random trees are walked and every lane has to visit the nodes of a plain
depth-first traversal, on its own stack.  On one stack for all of them the same
schedule has to go wrong, or it would show nothing."""
import shutil
import subprocess

import pytest

from paper_2305_04403_gb300 import build as B

SRC = r"""
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <random>
#include <thread>
#include <vector>
#include "node_stack.cuh"

constexpr int G = 4, kStride = G, kLevels = 3, kEnd = -1;

// Lanes 0 .. G-1 in turn; pass() ends a lane's turn and waits for its next one.
struct Turns {
    std::mutex m;
    std::condition_variable cv;
    long turn = 0;
    void wait(int lane)
    {
        std::unique_lock<std::mutex> l(m);
        cv.wait(l, [&] { return turn % G == lane; });
    }
    void pass(int lane)
    {
        std::unique_lock<std::mutex> l(m);
        ++turn;
        cv.notify_all();
        cv.wait(l, [&] { return turn % G == lane; });
    }
    void leave()
    {
        std::unique_lock<std::mutex> l(m);
        ++turn;
        cv.notify_all();
    }
};

struct Tree {
    std::vector<int> base;       // first interior child
    std::vector<uint32_t> mask;  // children that the line meets
};

int main(int, char** argv)
{
    const bool shared = argv[1][0] == '1';
    std::mt19937 g(7);
    long nodes = 0, wrong = 0, errs = 0;
    for (int t = 0; t < 60; ++t) {
        // a complete 8-ary tree of three levels below the root, with random masks
        Tree tr;
        const int inner = 1 + 8 + 64;
        for (int i = 0; i < inner + 512; ++i) {
            tr.base.push_back(i < inner ? 8 * i + 1 : ~i);  // a leaf's reference
            tr.mask.push_back(i < inner ? g() & 255u : 0u);
        }
        std::vector<int> want, st{0};
        while (!st.empty()) {
            const int n = st.back();
            st.pop_back();
            want.push_back(n);
            for (int c = 7; c >= 0; --c)
                if ((tr.mask[n] >> c) & 1) st.push_back(tr.base[n] + c);
        }
        volatile int stack[kLevels * kStride] = {};
        Turns turns;
        std::vector<int> got[G];
        int err[G] = {};
        std::vector<std::thread> lanes;
        for (int j = 0; j < G; ++j)
            lanes.emplace_back([&, j] {
                int sp = 0, node = 0;
                turns.wait(j);
                for (size_t k = 0; k < want.size(); ++k) {  // as many turns in every lane
                    if (node != kEnd) {
                        got[j].push_back(node);
                        const int n = node >= 0 && node < inner + 512 ? node : 0;
                        if (!wob::next_node(stack + (shared ? 0 : j), kStride, kLevels, tr.base[n],
                                            tr.mask[n], sp, node, err[j]))
                            node = kEnd;
                    }
                    turns.pass(j);  // the caller's barrier
                }
                turns.leave();
            });
        for (auto& l : lanes) l.join();
        for (int j = 0; j < G; ++j) {
            nodes += (long)want.size();
            wrong += got[j] != want;
            errs += err[j];
        }
    }
    printf("%ld %ld %ld\n", nodes, wrong, errs);
    return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("node_stack")
    (d / "t.cpp").write_text(SRC)
    subprocess.run([gxx, "-O2", "-std=c++17", "-pthread", "-I", B.CSRC, str(d / "t.cpp"), "-o",
                    str(d / "t")], check=True)
    return str(d / "t")


def _run(exe, shared):
    out = subprocess.run([exe, shared], check=True, capture_output=True, text=True, timeout=100)
    return tuple(int(x) for x in out.stdout.split())


def test_lanes_visit_the_same_nodes(exe):
    nodes, wrong, errs = _run(exe, "0")
    assert nodes > 10000 and wrong == 0 and errs == 0


def test_schedule_shows_a_shared_stack(exe):
    _, wrong, _ = _run(exe, "1")
    assert wrong > 0
