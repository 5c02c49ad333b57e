"""csrc/hand_out.cuh on the host: the front that thread 0 of a CTA hands to the
others in k_trsm_wave, with threads that read late."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <thread>
#include <vector>
#include "hand_out.cuh"

struct Barrier {
    std::mutex m;
    std::condition_variable cv;
    int threads, waiting = 0, phase = 0;
    void wait() {
        std::unique_lock<std::mutex> l(m);
        const int p = phase;
        if (++waiting == threads) {
            waiting = 0;
            phase++;
            cv.notify_all();
        } else {
            cv.wait(l, [&] { return phase != p; });
        }
    }
};

int main() {
    constexpr int kThreads = 3, kCalls = 20;
    Barrier b;
    b.threads = kThreads;
    int words[2] = {-1, -1}, wrong[kThreads] = {};
    std::vector<std::thread> th;
    for (int t = 0; t < kThreads; t++)
        th.emplace_back([&, t] {
            int pass = 0;
            for (int c = 0; c < kCalls; c++) {
                // nobody else is ever late at the barrier, and thread t reads
                // t * 10 ms after it: the leader is at its next call by then
                const int got = hplgb::hand_out(words, pass, t == 0, 100 + c, [&] {
                    b.wait();
                    std::this_thread::sleep_for(std::chrono::milliseconds(10 * t));
                });
                wrong[t] += got != 100 + c;
            }
        });
    for (auto& x : th) x.join();
    int sum = 0;
    for (int w : wrong) sum += w;
    std::printf("%d\n", sum);
    return sum != 0;
}
"""


def test_every_thread_gets_the_leaders_value_however_late_it_reads(tmp_path):
    src = tmp_path / "hand_out.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "hand_out")
    inc = os.path.join(ROOT, "paper_2604_09517_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I" + inc, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert (r.returncode, r.stdout) == (0, "0\n")
