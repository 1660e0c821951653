"""The limit of the backward's one wait that spans a work item: well above what the longest item that the argument checks admit takes."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_32704_b200", "csrc")


def test_the_wait_for_the_end_of_an_item_outlasts_the_item(tmp_path):
    # 64-row QO tiles of an item: Nq / 64 * G * 32 < 2^31 is checked, a step takes two of them
    longest = 2 ** 31 // 32 // 2
    src = tmp_path / "limit.cpp"
    src.write_text('#include <stdio.h>\n#include <initializer_list>\n#include "cowa_sched.h"\n'
                   f"int main() {{ for (int n : {{0, 1, 4, 550000, {longest}}}) printf(\"%d %lld\\n\", n, cowa_bwd_item_clocks(n)); }}\n")
    exe = str(tmp_path / "limit")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    for line in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines():
        steps, clocks = map(int, line.split())
        assert clocks >= 2 ** 31 and clocks - 2 ** 31 >= 3 * 5000 * steps  # (a reproducible step, the slowest, takes less than 5000)
        assert clocks < 2 ** 62
