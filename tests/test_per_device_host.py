"""The launch settings kept per device, from many threads at once (host code, no GPU)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_19723_gb300", "csrc")

PROGRAM = r"""
#include "per_device.cuh"
#include <cstdio>
#include <memory>
#include <thread>
int main() {
    constexpr int T = 16, KEYS = 400, ROUNDS = 20;
    static char keys[KEYS];
    for (int round = 0; round < ROUNDS; ++round) {
        bp::OncePerDevice once;
        bp::NumberPerDevice number;
        std::unique_ptr<std::atomic<int>[]> runs(new std::atomic<int>[2 * KEYS]());
        std::unique_ptr<std::atomic<int>[]> ready(new std::atomic<int>[2 * KEYS]());
        std::atomic<int> early{0}, wrong{0}, go{0};
        std::vector<std::thread> pool;
        for (int t = 0; t < T; ++t)
            pool.emplace_back([&, t] {
                ++go;
                while (go < T) std::this_thread::yield();
                for (int i = 0; i < 2 * KEYS; ++i) {
                    const int k = (i + 7 * (t % 4)) % KEYS, dev = (i / KEYS + t) % 2, at = dev * KEYS + k;
                    once.run(dev, keys + k, [&] { ++runs[at]; std::this_thread::yield(); ready[at] = 1; });
                    if (!ready[at]) ++early;                       // returned before the setting was made
                    if (number.get(dev, [&] { return 100 + dev; }) != 100 + dev) ++wrong;
                }
            });
        for (auto& th : pool) th.join();
        for (int i = 0; i < 2 * KEYS; ++i)
            if (runs[i] != 1) { std::printf("key %d ran %d times\n", i, runs[i].load()); return 1; }
        if (early || wrong) { std::printf("early %d wrong %d\n", early.load(), wrong.load()); return 1; }
    }
    return 0;
}
"""


def test_settings_are_made_once_per_device_and_before_any_launch(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O2", "-pthread", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
