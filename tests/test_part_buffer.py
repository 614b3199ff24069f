"""Room for the sums of split work items: the plan's buffers hold what the rule for splitting can ask for, on
any number of SMs, and no more than they need."""
import os
import subprocess

import pytest

from paper_1702_04728_gb300 import binding as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include "bf_internal.h"
#include <algorithm>
#include <cstdio>
using namespace chimebf;
int main() {
    for (int grid = 2; grid <= 160; ++grid) {
        size_t most_items = 0, most_sums = 0;
        for (int tc = 0; tc < 2; ++tc)
            for (int n = 1; n <= 3 * grid; ++n) {
                const int slots = tc ? grid / 2 : grid;
                for (int least = 1; least <= 6; ++least) {       // runtime.cpp asks for 1, 3 or 6
                    const PassUnits u = pass_units(n, slots, least);
                    const int split = n - u.n_full, parts = 6 / u.g;
                    if (split < 0 || u.n_units != u.n_full + parts * split || (u.g == 6 && split)) return 1;
                    if (split && (split * parts > slots || u.g < least)) return 2;
                    // sums an item publishes: its passes, or its halves in the FP32 form
                    const size_t each = !tc && u.g == 3 ? 2 : 6;
                    most_items = std::max(most_items, (size_t)split);
                    most_sums = std::max(most_sums, (size_t)split * each);
                }
            }
        if (most_items > part_items(grid) || most_sums > part_sums(grid)) return 3;
        if (grid == 152) std::printf("%zu %zu %zu %zu", most_items, part_items(grid), most_sums, part_sums(grid));
    }
    return 0;
}
"""


def test_split_items_fit(tmp_path):
    src, exe = tmp_path / "units.cpp", tmp_path / "units"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1702_04728_gb300", "csrc"),
                    "-I", "/usr/local/cuda/include", str(src), "-o", str(exe)], check=True)
    got = subprocess.run([str(exe)], capture_output=True, text=True)
    assert got.returncode == 0
    items, item_room, sums, sum_room = map(int, got.stdout.split())
    assert items == item_room and sums <= sum_room < sums + 6


@pytest.mark.gpu
@pytest.mark.parametrize("form,most", [(B.BF_FP32_FFT, 12), (B.BF_TC_DFT256_X1, 12)])
def test_memory_of_a_plan(built_lib, form, most):
    """Megabytes of device memory per plan before any request (table slots 4 to 5, sums of split items 5)."""
    torch = pytest.importorskip("torch")
    B.Plan(form=form).close()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    plans = [B.Plan(form=form) for _ in range(8)]
    used = before - torch.cuda.mem_get_info()[0]
    for p in plans:
        p.close()
    assert used <= 8 * most * 2 ** 20, used / 2 ** 23
