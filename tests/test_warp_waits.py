"""The warp-wide waits, whose first lane polls for all 32: the source of `mbar_wait_warp` and `flag_wait_warp` compiled for the
host and run by 32 threads under a model of what orders memory.  A lane may read the producer's data once it has acquired
itself (a poll that succeeded) or has passed a warp barrier behind a lane that had; a shuffle or a vote carries values and
orders nothing."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_28158_b200", "csrc")

MODEL = r"""
#include <barrier>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <thread>
#include <vector>
#define __device__
#define __forceinline__ inline
#define __noinline__
constexpr unsigned long long WAIT_LIMIT_NS = 1000, FLAG_WAIT_LIMIT_NS = 1000;
constexpr int STATUS_TIMEOUT = 1;
thread_local int lane;
struct Idx { struct X { operator int() const { return lane; } } x; } threadIdx;
std::barrier<> bar(32);
int values[32];
bool ordered[32], before[32];
int scenario;        // 0: complete at once, 1: complete after some polls, 2: never
int polls;
void __syncwarp() {                            // every lane sees what any lane saw before it
    before[lane] = ordered[lane];
    bar.arrive_and_wait();
    bool any = false;
    for (bool b : before) any = any || b;
    ordered[lane] = any;
    bar.arrive_and_wait();
}
int __shfl_sync(unsigned, int v, int src) {
    values[lane] = v;
    bar.arrive_and_wait();
    const int r = values[src];
    bar.arrive_and_wait();
    return r;
}
bool __all_sync(unsigned, bool v) {
    values[lane] = v;
    bar.arrive_and_wait();
    bool r = true;
    for (int x : values) r = r && x;
    bar.arrive_and_wait();
    return r;
}
bool acquire(bool done) { ordered[lane] = ordered[lane] || done; return done; }
int ld_acquire(const int* p) { return acquire(scenario == 0 || (scenario == 1 && ++polls > 40)) ? *p : 0; }
bool mbar_try(uint64_t*, uint32_t) { return acquire(scenario == 0); }
bool mbar_wait_slow(uint64_t*, uint32_t, int*, volatile int* dead, unsigned long long) {
    if (scenario != 2) return acquire(true);
    *dead = 1;
    return false;
}
unsigned long long global_ns() { static unsigned long long t = 0; return t += 100; }
void atomicExch(int* p, int v) { *p = v; }
"""

RUN = r"""
int main() {
    for (scenario = 0; scenario < 3; scenario++) {
        int flag = 4, status = 0, dead = 0, answers[32];
        uint64_t mbar = 0;
        polls = 0;
        memset(ordered, 0, sizeof ordered);
        std::vector<std::thread> warp;
        for (int l = 0; l < 32; l++)
            warp.emplace_back([&, l] { lane = l; answers[l] = CALL; });
        for (auto& t : warp) t.join();
        int yes = 0, seen = 0;
        for (int l = 0; l < 32; l++) yes += answers[l], seen += ordered[l];
        printf("%d %d %d\n", yes, seen, dead);
    }
}
"""


def _function(name):
    with open(os.path.join(CSRC, "tc_common.cuh")) as f:
        src = f.read()
    m = re.search(r"^[^\n]*\b%s\(.*?^}\n" % name, src, re.M | re.S)
    return m.group(0)


@pytest.mark.parametrize("name,call", [("mbar_wait_warp", "mbar_wait_warp(&mbar, 0, &status, &dead)"),
                                       ("flag_wait_warp", "flag_wait_warp(&flag, 4, &status, &dead)")])
def test_every_lane_is_ordered_behind_the_wait(name, call, tmp_path):
    src = tmp_path / "model.cc"
    src.write_text(MODEL + _function(name) + RUN.replace("CALL", call))
    exe = tmp_path / "model"
    subprocess.check_call(["g++", "-std=c++20", "-O1", "-pthread", "-o", str(exe), str(src)])
    out = [list(map(int, ln.split())) for ln in subprocess.check_output([str(exe)], text=True, timeout=60).splitlines()]
    assert out[0] == [32, 32, 0] and out[1] == [32, 32, 0]        # all lanes: true, and ordered behind the producer
    assert out[2][0] == 0 and out[2][2] == 1                        # a wait that ran out: false in every lane, latched
