"""csrc/batch_queue.cuh on the host: every system of a batch is taken by one CTA or
marked, whichever CTAs give up and when."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "batch_queue.cuh"
using namespace hplgb::bt;

// ctas threads work on the two lists; thread c gives up with its quit[c]-th
// system in hand (0: never). Returns 0 when every system has been solved, left in
// the hands of a thread that gave up, or marked, exactly once, and none is
// marked while a thread could still have taken it.
static int run(int n0, int n1, const std::vector<int>& quit) {
    Queue q = {};
    const int lo[2] = {0, n0}, sz[2] = {n0, n1};
    const unsigned ctas = (unsigned)quit.size();
    std::vector<std::atomic<int>> solved(n0 + n1), marked(n0 + n1);
    auto add = [](unsigned* p, unsigned v) { return __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST); };
    std::vector<std::thread> th;
    std::atomic<int> healthy{0};
    for (unsigned c = 0; c < ctas; c++)
        th.emplace_back([&, c] {
            int taken = 0;
            for (;;) {
                const int i = queue_next(&q, lo, sz, (int)(c & 1), add);
                if (i < 0) {
                    healthy++;
                    return;
                }
                solved[i]++;                    // a system in hand gets its status either way
                if (++taken == quit[c]) break;
            }
            queue_give_up(&q, lo, sz, ctas, add, [&](int i) { marked[i]++; });
        });
    for (auto& t : th) t.join();
    int wrong = 0, marks = 0;
    for (int i = 0; i < n0 + n1; i++) {
        wrong += solved[i] + marked[i] != 1;
        marks += marked[i];
    }
    return wrong + (healthy > 0 && marks > 0);
}

int main() {
    int bad = 0;
    for (int rep = 0; rep < 20; rep++) {
        bad += run(50, 40, {0, 0, 0, 0});       // nobody gives up
        bad += run(50, 40, {1, 3, 0, 2});       // one goes on
        bad += run(50, 40, {1, 1, 1, 1});       // everybody does
        bad += run(50, 40, {7, 1, 4, 2});
        bad += run(0, 9, {2});                  // a single CTA
        bad += run(9, 0, {9});                  // ... with its last system
    }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


def test_no_system_keeps_an_earlier_record_when_ctas_give_up(tmp_path):
    src = tmp_path / "queue.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "queue")
    inc = os.path.join(ROOT, "paper_2604_09517_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I" + inc, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert (r.returncode, r.stdout) == (0, "0\n")
