"""The persistent stack's plan (csrc/persist_plan.h) over its whole range, on the CPU: tensor-memory columns,
shared memory and SMs stay within what a GB300 has, a block's cells cover the layer, and the GPU cases of
test_gpu_persist.py take every form of the kernel that a plan can ask for."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "persist_plan.h"
using namespace qnn::persist;
static int64_t up(int64_t v, int64_t m) { return (v + m - 1) / m * m; }
int main(int argc, char **argv) {
    int64_t v[5];  // L, I, H, B, SMs
    if (argc == 6) {
        for (int i = 0; i < 5; ++i) v[i] = std::atoll(argv[i + 1]);
        Plan p;
        const int64_t kh = up(v[2], 64), kx = std::max(up(v[1], 64), v[0] > 1 ? kh : 0);
        if (make_plan(v[0], v[2], kx, kh, v[3], v[4], &p)) std::printf("%d %d %d\n", p.NC, p.MT, p.SP);
        return 0;
    }
    const int64_t Bs[] = {1, 4, 5, 8, 9, 17, 31, 32, 33, 57, 64, 65, 100, 121, 127, 128, 129, 130, 200, 255, 256};
    const int64_t Is[] = {1, 40, 64, 320, 520, 1024}, Ss[] = {132, 148, 152, 160};
    long plans = 0, bad = 0;
    for (int64_t sms : Ss)
        for (int64_t I : Is)
            for (int64_t L = 1; L <= 9; ++L)
                for (int64_t H = 1; H <= 1100; ++H)
                    for (int64_t B : Bs) {
                        Plan p;
                        const int64_t kh = up(H, 64), kx = std::max(up(I, 64), L > 1 ? kh : 0);
                        if (!make_plan(L, H, kx, kh, B, sms, &p)) continue;
                        ++plans;
                        const int N = 16 * p.NC, last = (2 * p.MT + p.MT - 1) * N + N;  // the kernel's last column
                        const int64_t ring = (int64_t)p.slots * p.slot_bytes;
                        const int64_t fixed = (kx + kh) / 64 * N * 128 + misc_bytes(p.NC, p.MT, p.SP);
                        // the last k-block of the last slot, read as 128 rows
                        const int64_t reads = ring - (int64_t)p.rows_box * 128 + kTile * 128;
                        const bool ok = last <= 512 && tmem_used(p.NC, p.MT) == last && ring + fixed <= (int64_t)p.smem &&
                                        p.smem <= 227 * 1024 && reads <= (int64_t)p.smem && p.slots >= 2 && p.slots <= 4 &&
                                        p.slot_bytes == p.kps * p.rows_box * 128 && p.slot_bytes % 1024 == 0 &&
                                        p.rows_box % 8 == 0 && p.rows_box <= 128 && p.kps >= 1 && p.kps <= 8 &&
                                        std::min<int64_t>(B, 128) <= p.rows_box && B <= 128 * p.MT && L <= 8 &&
                                        L * p.G <= sms && (int64_t)p.G * 4 * p.NC >= H && (int64_t)(p.G - 1) * 4 * p.NC < H &&
                                        (p.SP == 1 || (p.MT == 1 && B <= 128 / p.SP)) &&
                                        (p.NC == 2 || p.NC == 4 || p.NC == 5 || p.NC == 6);
                        if (!ok && ++bad <= 5)
                            std::printf("L %ld I %ld H %ld B %ld SMs %ld: NC %d MT %d SP %d columns %d smem %zu slots %d\n", (long)L,
                                        (long)I, (long)H, (long)B, (long)sms, p.NC, p.MT, p.SP, last, p.smem, p.slots);
                    }
    std::printf("%ld plans, %ld bad\n", plans, bad);
    return bad != 0 || plans == 0;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SRC)
    exe = str(d / "plan")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1607_04683_gb300", "csrc"), str(d / "plan.cpp"), "-o", exe],
                   check=True)
    return lambda *a: subprocess.run([exe, *map(str, a)], capture_output=True, text=True)


def test_every_plan_fits(plan):
    r = plan()
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("B", [129, 130, 256])
@pytest.mark.parametrize("H", [381, 384])
def test_two_row_tiles_of_24_cells_have_no_plan(plan, H, B):
    # 8 layers find their SMs only with 24 cells a block, whose accumulators for two row tiles take 576 columns
    assert plan(8, 40, H, B, 152).stdout == "" and plan(8, 40, H, 128, 152).stdout.split() == ["6", "1", "1"]


def test_gpu_cases_take_every_form(plan):
    pytest.importorskip("torch")
    from test_gpu_persist import CASES
    seen = set()
    for c in CASES:
        f = plan(c.get("L", 2), c.get("I", 40), c.get("H", 64), c.get("B", 5), 152).stdout.split()
        assert f, c
        seen.add(tuple(map(int, f)))
    forms = {(nc, mt, sp) for nc in (2, 4, 5, 6) for mt, sp in ((1, 4), (1, 2), (1, 1), (2, 1))} - {(6, 2, 1)}
    assert seen == forms, forms - seen
