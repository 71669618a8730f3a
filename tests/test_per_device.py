"""What a device is asked for once: a failed query is made again, a good one is kept, per device and from several threads."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_03229_b200", "csrc")

MAIN = r"""
#include "per_device.h"
#include <thread>
#include <vector>
int main() {
    static mpipe::PerDevice d;
    int asked = 0;
    auto fails = [&]() { ++asked; return 0; };
    auto gives = [&]() { ++asked; return 74; };
    if (d.get(3, fails) != 0 || d.get(3, gives) != 74 || d.get(3, fails) != 74 || asked != 2) return 1;   // the failure was not kept
    if (d.get(4, fails) != 0 || d.get(-1, gives) != 0) return 2;
    if (d.get(100, gives) != 74 || d.get(100, fails) != 0) return 3;                                       // not remembered, but served
    std::vector<std::thread> many;
    std::atomic<int> bad{0};
    for (int i = 0; i < 8; ++i) many.emplace_back([&]() { for (int k = 0; k < 1000; ++k) bad += d.get(k % 64, []() { return 5; }) != (k % 64 == 3 ? 74 : 5); });
    for (auto& t : many) t.join();
    return bad ? 4 : 0;
}
"""


def test_a_failed_query_is_made_again(tmp_path):
    src, exe = tmp_path / "main.cpp", str(tmp_path / "main")
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe], timeout=60).returncode == 0
