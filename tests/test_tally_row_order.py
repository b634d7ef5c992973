"""The in-place tally's exchange through shared memory, on the CPU: reduce_rows() as it stands in
the kernels' header, run by 32 host threads as the lanes of a warp under the memory model that
CUDA states, where only a warp barrier orders one lane's shared-memory accesses against
another's.  Two schedules: stores that become visible to other lanes as late as that allows,
and lanes that run ahead as far as it allows."""
import os
import re
import shutil
import subprocess

import pytest

HEADER = os.path.join(os.path.dirname(__file__), "..", "paper_2512_01283_gb300", "csrc", "mcrt_packet.cuh")

PROGRAM = r"""
#include <barrier>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <limits>
#include <thread>
#include <vector>
#define __device__
#define __forceinline__ inline
#define FULL 0xffffffffu
static std::barrier<> bar(32);
struct Pending { float* at; int row; float v; double* p; };  // a value, or (at null) a row's place
static thread_local std::vector<Pending> buffer;  // this lane's stores that no other lane sees yet
static thread_local bool slow = false;
static std::vector<float> rows;
static std::vector<double*> place;
static void flush() {
    for (Pending& s : buffer)
        if (s.at) *s.at = s.v;
        else place[s.row] = s.p;
    buffer.clear();
}
static void __syncwarp(unsigned = FULL) { bar.arrive_and_wait(); flush(); bar.arrive_and_wait(); }
static void red_add(double* p, double v) {
    if (slow) std::this_thread::sleep_for(std::chrono::milliseconds(1));
    double o, n;
    __atomic_load(p, &o, __ATOMIC_SEQ_CST);
    do n = o + v; while (!__atomic_compare_exchange(p, &o, &n, false, __ATOMIC_SEQ_CST, __ATOMIC_SEQ_CST));
}
static double widen(float v) { return v; }
@FUNCTION@
int main(int argc, char** argv) {
    const int n = atoi(argv[1]), nv = atoi(argv[2]), stride = nv + 4;
    const bool late = argv[3][0] == 'l';
    rows.assign(32 * stride, std::numeric_limits<float>::quiet_NaN());
    place.assign(32, nullptr);
    std::vector<double> sums(2 * 32 * nv, 0.0);
    std::vector<std::thread> lanes;
    for (int lane = 0; lane < 32; ++lane)
        lanes.emplace_back([&, lane] {
            for (int turn = 0; turn < 2; ++turn) {
                slow = !late && turn == 0 && lane % 2 == 1;
                if (lane < n) {
                    for (int v = 0; v < nv; ++v)
                        buffer.push_back({&rows[lane * stride + v], 0, float(1 + turn * 4096 + lane * nv + v), nullptr});
                    buffer.push_back({nullptr, lane, 0.f, &sums[(size_t)(turn * 32 + lane) * nv]});
                }
                if (!late) flush();
                if (!late && turn == 0) bar.arrive_and_wait();  // the first turn starts together
                reduce_rows(n, lane, (const float*)rows.data(), stride, nv, [&](int k) { return place[k]; });
            }
        });
    for (auto& t : lanes) t.join();
    int bad = 0;
    for (int turn = 0; turn < 2; ++turn)
        for (int lane = 0; lane < n; ++lane)
            for (int v = 0; v < nv; ++v)
                if (sums[(size_t)(turn * 32 + lane) * nv + v] != double(1 + turn * 4096 + lane * nv + v)) ++bad;
    printf("%d\n", bad);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    text = open(HEADER).read()
    function = re.search(r"template <typename T, typename At>\n__device__ __forceinline__ void reduce_rows\(.*?\n}\n", text, re.S)
    d = tmp_path_factory.mktemp("rows")
    (d / "rows.cpp").write_text(PROGRAM.replace("@FUNCTION@", function.group(0)))
    subprocess.run(["g++", "-std=c++20", "-O1", "-pthread", "-o", str(d / "rows"), str(d / "rows.cpp")], check=True)
    return str(d / "rows")


# whole warps and a few rows, of 1, 3, 8 and 16 cameras
@pytest.mark.parametrize("schedule", ["late", "early"])
@pytest.mark.parametrize("n,n_cam", [(32, 1), (32, 8), (5, 3), (31, 16)])
def test_rows_are_read_after_they_are_staged_and_before_they_are_staged_again(program, n, n_cam, schedule):
    out = subprocess.run([program, str(n), str(4 * n_cam), schedule], capture_output=True, text=True, timeout=60, check=True)
    assert int(out.stdout) == 0
