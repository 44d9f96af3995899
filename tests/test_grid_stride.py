"""The index range of the grid-stride loops (csrc/grid_stride.cuh), replayed on the host: every
thread's cells, once and in order, and none outside the field, up to the largest mesh the API
accepts (2^31 - 1 cells), where an int counter passes its range before the loop ends."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
#include "grid_stride.cuh"
static int64_t next_, seen;
static bool bad;
static void take(int64_t k, int64_t n, int64_t step) {
    if (k < 0 || k >= n || k != next_) bad = true;
    next_ = k + step;
    ++seen;
}
template <int W> static bool replay(int64_t n, int64_t first, int64_t step) {
    next_ = first;
    seen = 0;
    bad = false;
    const int64_t want = first < n ? (n - 1 - first) / step + 1 : 0;
    // (a replay that leaves the range or never ends gives up here)
    auto guard = [&]() { if (bad || seen > want) { printf("W %d n %lld first %lld step %lld\n", W, (long long)n,
                                                         (long long)first, (long long)step); exit(1); } };
    cgk::grid_stride<W>((uint32_t)n, (uint32_t)first, (uint32_t)step,
        [&](uint32_t k, uint32_t s) { for (int j = 0; j < W; ++j) take(k + j * s, n, step); guard(); },
        [&](uint32_t k) { take(k, n, step); guard(); });
    return !bad && seen == want;
}
int main(int argc, char **argv) {
    const int64_t n = atoll(argv[1]);
    for (int64_t blocks : {1, 16, 608, 1216, 1280, 65536}) {
        const int64_t step = blocks * 256;
        for (int64_t first : {int64_t(0), int64_t(1), step / 2, (n - 1) % step, n % step, step - 1})
            if (!replay<4>(n, first, step) || !replay<8>(n, first, step)) {
                printf("n %lld step %lld first %lld\n", (long long)n, (long long)step, (long long)first);
                return 1;
            }
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("stride")
    (d / "t.cc").write_text(SOURCE)
    exe = str(d / "t")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fwrapv", "-x", "c++", "-I",
                    os.path.join(ROOT, "paper_1409_0001_gb300", "csrc"), str(d / "t.cc"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("n", [1, 3, 4, 255, 1024, 311_296 * 3, 311_296 * 3 + 1, 101 * 99 * 98, 2046 * 1024 * 1024,
                               2047 * 1024 * 1024, 1290 ** 3, 2 ** 31 - 311_296, 2 ** 31 - 2, 2 ** 31 - 1])
def test_cells_in_range_once(program, n):
    r = subprocess.run([program, str(n)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
