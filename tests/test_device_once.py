"""Values found once per device: on the CPU, many threads and devices at once,
with an initialisation that takes a while and one that fails at first; on the
GPU, threads that start on a kernel together in a new process."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1107_1653_gb300", "csrc")

PROGRAM = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "device_once.h"
struct Pair { int a = 0, b = 0; };
int main() {
    constexpr int kDevices = 70, kThreads = 16;
    gs::PerDevice<Pair> once;
    std::atomic<int> inits[kDevices]{}, failed{0}, wrong{0};
    std::vector<std::thread> ts;
    for (int t = 0; t < kThreads; ++t)
        ts.emplace_back([&] {
            for (int d = 0; d < kDevices; ++d)
                for (int tries = 0; tries < 2; ++tries) {
                    try {
                        const Pair& p = once.get(d, [&] {
                            if (d % 7 == 0 && inits[d]++ == 0) throw 1;
                            if (d % 7 != 0) ++inits[d];
                            Pair q;
                            q.a = d;
                            std::this_thread::sleep_for(std::chrono::microseconds(200));
                            q.b = d + 1;
                            return q;
                        });
                        if (p.a != d || p.b != d + 1) ++wrong;
                    } catch (int) {
                        ++failed;
                    }
                }
        });
    for (auto& t : ts) t.join();
    int n = 0;
    for (int d = 0; d < kDevices; ++d) n += inits[d];
    std::printf("%d %d %d\n", (int)wrong, (int)failed, n);
}
"""


def test_once_per_device_with_threads(tmp_path):
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, "-o", exe, str(tmp_path / "t.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout
    # ten devices fail once and are tried again: 70 + 10 initialisations
    assert out.split() == ["0", "10", "80"]


THREADS = r"""
import sys, threading
sys.path[:0] = [%r, %r]
import numpy as np
import paper_1107_1653_gb300 as gs
import synth
from test_gpu_amg_paths import band_game
tables = band_game(700, 3, 5)
games = [synth.random_game(n, n) for n in (600, 3000)]
out, errors, start = {}, [], threading.Barrier(8)
def work(k):
    try:
        kind = k %% 4
        s = gs.GameSolver(precision="mixed" if k < 4 else "fp64", game_solver=1 if kind == 0 else 0)
        start.wait()
        for _ in range(3):
            if kind == 0:
                s.set_game(700, 2, 2, *tables, 0.995)
            elif kind == 3:
                s.set_isaacs_grid(63, 0, 1)
            else:
                s.set_game((600, 3000)[kind - 1], 4, 4, *games[kind - 1])
            s.solve()
    except Exception as e:
        errors.append((k, repr(e)))
ts = [threading.Thread(target=work, args=(k,)) for k in range(8)]
[t.start() for t in ts]
[t.join() for t in ts]
assert not errors, errors
"""


@pytest.mark.gpu
def test_threads_start_on_the_kernels_together(gs):
    for _ in range(4):
        p = subprocess.run([sys.executable, "-c", THREADS % (ROOT, os.path.join(ROOT, "tests"))], cwd=ROOT,
                           capture_output=True, text=True, timeout=300)
        assert p.returncode == 0, p.stderr[-2000:]
