"""The side of the attention kernels that asks for units (cluster launch control), compiled for the host with the hardware replaced by a
model of it: whichever wait runs out, a request is never made while an answer is on its way, nor after the answer that ends the list,
and nothing of the grid is left to start."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_03229_b200", "csrc")

MODEL = r"""
#include <cstdint>
#include <cstdio>
#define __device__
#define __forceinline__ inline
struct uint4 { unsigned x, y, z, w; };
struct mpipe_work_item_t { int32_t seg, tile, row_start, row_len, kv_start, kv_len; };
namespace mpipe {
int left, wait_no, fail_at;       // blocks not started yet; the wait that runs out
bool pending, negative, wrong;    // an answer is on its way; the last answer ended the list
int answer_block;
inline void mbar_init(uint64_t*, int) {}
inline void mbar_arrive(uint64_t*) {}
inline void mbar_expect_tx(uint64_t*, uint32_t) { wrong |= pending; }
inline void clc_try_cancel(void*, uint64_t*) {
    wrong |= pending || negative;
    pending = true;
    answer_block = left > 0 ? left-- : -1;
}
inline bool mbar_wait(uint64_t*, uint32_t, volatile int*) { return wait_no++ != fail_at; }
inline bool mbar_wait_budget(uint64_t*, uint32_t, int*, long long) { return true; }
inline int clc_block_of(const void*) {
    wrong |= !pending;
    pending = false;
    negative = answer_block < 0;
    return answer_block;
}
inline void fence_async_smem() {}
inline void __syncwarp() {}
}
"""

MAIN = r"""
using namespace mpipe;
int main() {
    for (int blocks = 0; blocks < 7; ++blocks)
        for (fail_at = -1; fail_at < 3 * blocks + 6; ++fail_at) {
            UnitRing ring;
            int abort_flag = 0;
            UnitSource source{&ring, &abort_flag};
            left = blocks; wait_no = 0; pending = negative = wrong = false;
            bool ok = true;
            for (int u = 100; ok;) {          // the loop of the producers: put, ask, load, take
                const mpipe_work_item_t it = {0, 0, 0, 0, 0, u < 0 ? 0 : 1};
                ok = source.put(it);
                if (!ok || it.kv_len <= 0) break;
                source.ask();
                ok = mbar_wait(nullptr, 0, nullptr);
                if (!ok) break;
                u = source.take(&ok);
            }
            if (!ok) source.cancel_rest();
            if (wrong || pending || left != 0) {
                std::printf("%d blocks, wait %d: %s\n", blocks, fail_at, wrong ? "asked out of turn" : "something left");
                return 1;
            }
        }
    return 0;
}
"""


def test_requests_and_answers_take_turns(tmp_path):
    with open(os.path.join(CSRC, "units.cuh")) as f:
        units = "".join(line for line in f if not line.startswith(("#include", "#pragma")))
    src = tmp_path / "units.cpp"
    src.write_text(MODEL + units + MAIN)
    exe = str(tmp_path / "units")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", str(src), "-o", exe], check=True)
    got = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert got.returncode == 0, got.stdout
