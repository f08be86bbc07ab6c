"""The host table that keeps per-context values (a kernel's raised
shared-memory limit) per device and CUDA context: compiled alone, no GPU."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2404_01249_gb300", "csrc")
DRIVER = r"""
#include "context_table.h"
#include <atomic>
#include <stdio.h>
#include <thread>
#include <vector>
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
    fa::ContextTable<int> t;
    std::atomic<int> made{0};
    char k[2];
    auto get = [&](int dev, unsigned long long ctx, int key, bool keep = true) {
        return t.get(dev, ctx, k + key, [&](int *v) { *v = ++made; return keep; });
    };
    CHECK(get(0, 7, 0) == 1 && get(0, 7, 0) == 1);  // kept
    CHECK(get(0, 7, 1) == 2);                       // another kernel
    CHECK(get(1, 7, 0) == 3 && get(1, 7, 0) == 3);  // another device
    CHECK(get(0, 7, 0) == 1);                       // the first device's stays
    CHECK(get(0, 8, 0) == 4 && get(0, 8, 1) == 5);  // a new context on device 0: all again
    CHECK(get(1, 7, 0) == 3);                       // device 1 was not reset
    CHECK(get(0, 7, 0) == 6);                       // nothing of the old context was left
    CHECK(get(2, 1, 0, false) == 7 && get(2, 1, 0) == 8 && get(2, 1, 0) == 8);  // a failure is not kept
    made = 0;
    std::vector<std::thread> w;
    for (int i = 0; i < 8; ++i) w.emplace_back([&] { for (int j = 0; j < 1000; ++j) get(3, 1, j & 1); });
    for (auto &x : w) x.join();
    CHECK(made == 2);  // once per key
    return 0;
}
"""


def test_values_hold_for_one_context_of_one_device(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(DRIVER)
    subprocess.run([gxx, "-std=c++17", "-Wall", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
