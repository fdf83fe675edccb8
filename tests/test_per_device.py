"""What a kernel needs once per device (csrc/per_device.h), on the host: every
device gets its own, a failure is tried again, an index beyond the table is worked
out each time, and threads that ask at once see only final numbers."""

import os
import subprocess

SOURCE = r"""
#include "per_device.h"
#include <thread>
#include <vector>
#include <cstdio>
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
    static kwgb::PerDevice p;
    int made = 0;
    auto give = [&](int v) { return [&made, v] { ++made; return v; }; };
    CHECK(p.get(0, give(3)) == 3 && made == 1);
    CHECK(p.get(0, give(9)) == 3 && made == 1);       // once on a device
    CHECK(p.get(1, give(5)) == 5 && made == 2);       // and on the next one again
    CHECK(p.get(2, give(0)) == 0 && p.get(2, give(7)) == 7 && made == 4);
    CHECK(p.get(64, give(1)) == 1 && p.get(64, give(2)) == 2 && p.get(-1, give(4)) == 4);
    static kwgb::PerDevice q;
    std::vector<std::thread> t;
    std::atomic<int> bad{0};
    for (int i = 0; i < 8; ++i)
        t.emplace_back([&] {
            for (int dev = 0; dev < 64; ++dev)
                if (q.get(dev, [&] { int n = 1; n += dev; return n; }) != dev + 1) ++bad;
        });
    for (auto& x : t) x.join();
    CHECK(bad == 0);
    return 0;
}
"""


def test_worked_out_once_on_each_device(tmp_path):
    from paper_1408_4675_gb300 import build
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", build.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_kernel_set_up_is_not_kept_for_the_whole_process():
    """A kernel's attributes belong to one device: no launcher keeps them in a plain static."""
    from paper_1408_4675_gb300 import build
    for name in ("line_pass.cuh", "yz_kernel.cuh", "x_rows.cuh"):
        src = open(os.path.join(build.CSRC, name)).read()
        assert "static bool" not in src and "static int per_sm" not in src, name
