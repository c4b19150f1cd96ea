"""The estimate that balances a batch's lanes (bse_cost.h, plain C++): the near field of
every path counts, in proportion to its offsets or pieces, and known steps come out near
their measured times (within a factor of 1.5: kernels beside each other share the chip)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#include <cstdio>
#include <cstdlib>
#include "bse_cost.h"
int main(int, char** v) {
    StepWork w{atoll(v[1]), atoll(v[2]), atoi(v[3]), atoi(v[4]), atoi(v[5]), atoi(v[6]), atoll(v[7]), atoll(v[8])};
    std::printf("%.17g", bse_step_us(w));
}
"""


@pytest.fixture(scope="module")
def cost(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("cost")
    (d / "c.cpp").write_text(SOURCE)
    subprocess.run([gxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_1602_01863_gb300", "csrc"), str(d / "c.cpp"), "-o", str(d / "c")], check=True)

    def f(Nc, N, chains, kc_bytes, m3, common, near_offsets=0, near_pieces=0):
        a = [Nc, N, chains, kc_bytes, m3, common, near_offsets, near_pieces]
        return float(subprocess.run([str(d / "c"), *map(str, a)], capture_output=True, text=True, check=True).stdout)
    return f


def test_near_field_counts_on_both_paths(cost):
    base = cost(2048, 131072, 3, 4, 0, 1)
    narrow, wide = cost(2048, 131072, 3, 4, 1, 1, 33), cost(2048, 131072, 3, 4, 1, 1, 7153)
    assert base < narrow < wide
    assert (wide - base) == pytest.approx((narrow - base) * 7153 / 33, rel=1e-9)
    assert cost(2048, 131072, 3, 4, 1, 0, 0, 8192 * 343 * 16) > cost(2048, 131072, 3, 4, 1, 1, 257)


def test_estimates_of_measured_steps(cost):
    # coarse 8^3, n_div 4, 4x4 bands, 3 chains: 231 us with kernels one after another, and in FP64 3315 us
    assert 231 / 1.5 < cost(8192, 524288, 3, 4, 1, 1, 257) < 231 * 1.5
    assert 3315 / 1.5 < cost(8192, 524288, 3, 16, 1, 1, 257) < 3315 * 1.5
