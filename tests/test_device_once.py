"""A kernel's shared-memory limit holds for the device that is current when it is set: every one is set through
DeviceOnce, which runs once on each device, once among threads, and again after a failure."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_17696_gb300", "csrc")

PROGRAM = """
#include "device_once.h"
#include <cassert>
#include <thread>
#include <vector>
int main() {
    helm::DeviceOnce once;
    int calls[70] = {};
    auto go = [&](int dev, int status) { return once.run(dev, [&] { ++calls[dev]; return status; }); };
    assert(go(0, 0) == 0 && go(0, 0) == 0 && calls[0] == 1);
    assert(go(1, 0) == 0 && calls[1] == 1);                      // another device
    assert(go(2, 7) == 7 && go(2, 0) == 0 && go(2, 9) == 0 && calls[2] == 2);
    assert(go(63, 0) == 0 && go(63, 0) == 0 && calls[63] == 1);
    assert(go(65, 0) == 0 && go(65, 0) == 0 && calls[65] == 2);  // past the table: every time
    assert(go(1, 9) == 0);
    helm::DeviceOnce other;
    std::atomic<int> ran{0};
    std::vector<std::thread> ts;
    for (int i = 0; i < 16; ++i)
        ts.emplace_back([&, i] {
            assert(other.run(i % 2, [&] { std::this_thread::yield(); return ran.fetch_add(1) * 0; }) == 0);
            assert(ran.load() >= 1);
        });
    for (auto& t : ts) t.join();
    assert(ran.load() == 2);
    return 0;
}
"""


def test_runs_once_on_every_device(tmp_path):
    src = tmp_path / "once.cpp"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-UNDEBUG", "-pthread", "-I", CSRC, str(src), "-o", str(tmp_path / "once")], check=True)
    subprocess.run([str(tmp_path / "once")], check=True, timeout=60)


def test_every_function_attribute_is_set_per_device():
    found = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        for m in re.finditer(r"cudaFuncSetAttribute\(", text):
            found += 1
            openers = re.findall(r"once_per_device\(|call_once\(|static bool|^\}", text[:m.start()], re.M)
            assert openers and openers[-1] == "once_per_device(", (os.path.basename(path), text.count("\n", 0, m.start()) + 1)
    assert found >= 10
