"""Shared memory against registers: warps per SM of the chain kernels (no GPU needed).

The rules that pick lane layouts and parts count the warps per SM that a kernel's
registers are planned for.  A small host program with the library's own plan lists,
per lane layout in FP32, that number beside the CTAs of one warp that shared memory
leaves room for: in the batched kernel, and in the chain kernel without a stress series,
with as many log steps as a launch takes; with the series where the layout is measured
at that number.
"""
import os
import subprocess

import pytest

from paper_1106_2899_gb300 import build

SRC = r"""
#include <cstdio>
#include "ss_kernels.cuh"
using namespace ssk;
int main() {
    const int lay[][2] = {{8, 1}, {8, 2}, {8, 3}, {16, 1}, {16, 2}, {16, 3}, {16, 4}, {32, 1}, {32, 3}, {32, 4}};
    for (auto& l : lay)
        for (int logs : {0, 11, 16})
            for (int series = 0; series < 2; ++series) {
                const int red = series ? red_steps<float>(l[0], l[1], false, true, false) : 0;
                const int bytes = smem_plan<float>(1, l[0], l[1], logs, red).total;
                std::printf("%d %d %d %d %d %d %d\n", l[0], l[1], logs, series,
                            chunk_warps_per_sm<float>(l[0], l[1], false, true), ctas_by_smem(bytes),
                            ctas_by_smem(bytes + (int)sizeof(ChunkArgs)));
            }
    // the second form of 16 x 4 (Euler-Maruyama, Heun), with a series
    for (int heun = 0; heun < 2; ++heun)
        std::printf("16 4 -1 %d %d %d 0\n", heun, chunk_warps_per_sm<float>(16, 4, heun, false, true),
                    ctas_by_smem(smem_plan<float>(1, 16, 4, 0, red_steps<float>(16, 4, heun, false, true)).total));
}
"""


@pytest.fixture(scope="module")
def table(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, exe = d / "plan.cu", d / "plan"
    src.write_text(SRC)
    subprocess.check_call([build.nvcc(), "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                           "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"),
                           "-o", str(exe), str(src)])
    rows = [tuple(map(int, line.split())) for line in subprocess.check_output([str(exe)], text=True).splitlines()]
    return {r[:4]: r[4:] for r in rows}


def test_without_a_series_registers_decide(table):
    assert len(table) == 62
    for (w, b, logs, series), (regs, chunk, batched) in table.items():
        if logs >= 0 and not series:
            assert chunk >= regs and batched >= regs, (w, b, logs)


def test_with_a_series(table):
    # without logs the register figure or, of these, nearly
    least = {(8, 2): 18, (8, 3): 15, (16, 3): 15, (32, 4): 13}
    for (w, b, logs, series), (regs, chunk, _) in table.items():
        if series and logs == 0:
            assert chunk >= least.get((w, b), regs), (w, b)
    for heun in (0, 1):
        assert table[16, 4, -1, heun][:2] == (16, 16)
