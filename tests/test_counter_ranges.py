"""Counters that a launch of the run kernel keeps per lane hold what the launch can count, in every kind of instance: a small
program asks the kernel's own types (nvcc, host code only)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "qsim_device.cuh"
using namespace qsimdev;
// rows of 32 GPUs that a lane works on at most: its iteration ends in one round, and one more that is the round's event
template <int SPL, uint32_t F> void show(const char *name, double rows)
{
    using S = Sim<SPL, F>;
    const double ends = S::CAL ? 1.0 : rows;
    std::printf("%s %.17g %.17g %d %d\n", name, (ends + 1.0) * (double)BUDGET_MAX, (double)BUDGET_MAX,
                8 * (int)sizeof(S::it_mixed), 8 * (int)sizeof(S::rounds));
}
int main()
{
    show<1, F_GENERIC>("one_row", 1);
    show<4, F_GENERIC>("four_rows", 4);
    show<0, 0u>("calendar", 128);
    show<0, F_FAR>("calendar_far", 128);
    show<0, F_SCAN>("all_rows", 128);
    show<0, F_MW>("several_warps", 64);
}
"""


def test_iteration_counters_hold_what_a_launch_can_count(tmp_path):
    src, exe = tmp_path / "ranges.cu", tmp_path / "ranges"
    src.write_text(PROGRAM)
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2602_02987_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    lines = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split("\n")[:-1]
    assert len(lines) == 6
    for line in lines:
        name, iterations, rounds, it_bits, round_bits = line.split()
        assert float(iterations) < 2.0 ** int(it_bits), name
        assert float(rounds) < 2.0 ** int(round_bits), name
