"""Host run of a fill round of the streamed tensor-core first stage
(ts_fill_round of csrc/fe_waits.cuh, the code the kernel runs): four threads
stand for the fill warps, a barrier that gives up after a while for their named
barrier. Whichever warps' waits give up, in whichever round and stage, the four
leave together, at the end of that round at the latest, and none is left waiting
for another."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2303_09886_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

PROGRAM = r"""
#include "fe_waits.cuh"
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <thread>

constexpr int kWarps = 4, kStages = 4, kRounds = 3;

struct Barrier {   // bar.red.and over the fill warps
    std::mutex mu;
    std::condition_variable cv;
    int in = 0, phase = 0;
    bool all = true, result = true, stuck = false;
    bool vote(bool ok) {
        std::unique_lock<std::mutex> lk(mu);
        if (stuck) return false;
        all = all && ok;
        const int ph = phase;
        if (++in == kWarps) {
            result = all;
            in = 0;
            all = true;
            phase++;
            cv.notify_all();
            return result;
        }
        if (!cv.wait_for(lk, std::chrono::milliseconds(300), [&] { return phase != ph || stuck; })) {
            stuck = true;
            cv.notify_all();
        }
        return stuck ? false : result;
    }
};

int main() {
    int bad = 0, runs = 0;
    // mask: the warps whose wait gives up in round fr (warp 3 has no tile of its own at three tiles per unit);
    // at stage fs where the round realigns (its thread 0 waits for all)
    for (int moved = 0; moved < (1 << kRounds); moved++)
        for (int fr = 0; fr < kRounds; fr++)
            for (int mask = 1; mask < 8; mask++)
                for (int fs = 0; fs < kStages; fs += kStages - 1) {
                    Barrier bar;
                    int rounds[kWarps] = {}, realigned[kWarps] = {};
                    bool left_ok[kWarps] = {};
                    auto warp = [&](int w) {
                        bool ok = true;
                        int r = 0;
                        for (; r < kRounds; r++) {
                            if (!ok) break;   // as the kernel's round loop
                            const bool mv = (moved >> r) & 1;
                            ok = fe::ts_fill_round<kStages>(
                                mv, [&] { return !(r == fr && ((mask >> w) & 1)); },
                                [&](int k) { return w != 0 || !(r == fr && (mask & 1) && k == fs); },
                                [&](int) { realigned[w]++; }, [&](bool mine) { return bar.vote(mine); });
                        }
                        rounds[w] = r;
                        left_ok[w] = ok;
                    };
                    std::thread t[kWarps];
                    for (int w = 0; w < kWarps; w++) t[w] = std::thread(warp, w);
                    for (auto &x : t) x.join();
                    const bool fails = !((moved >> fr) & 1) || (mask & 1);
                    bool good = !bar.stuck;
                    for (int w = 0; w < kWarps; w++)
                        good = good && rounds[w] == (fails ? fr + 1 : kRounds) && left_ok[w] == !fails &&
                               realigned[w] == realigned[0];
                    if (!good) {
                        bad++;
                        std::printf("moved %d round %d mask %d stage %d: rounds %d %d %d %d stuck %d\n", moved, fr, mask, fs,
                                    rounds[0], rounds[1], rounds[2], rounds[3], (int)bar.stuck);
                    }
                    runs++;
                    if (bad > 3) return 1;
                }
    std::printf("%d runs, %d bad\n", runs, bad);
    return bad ? 1 : 0;
}
"""


def run_host(tmp_path, program):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ and the CUDA headers are needed")
    src, exe = tmp_path / "host.cpp", tmp_path / "host"
    src.write_text(program)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-Wno-unknown-pragmas", "-I" + CSRC, "-I" + CUDA_INC,
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


def test_fill_warps_leave_together(tmp_path):
    run_host(tmp_path, PROGRAM)
