"""The share of the chip a served box is launched for: handles beside it, not
the boxes that go to the ensemble kernel."""
import os
import subprocess

import paper_1311_0402_gb300 as dpd

SOURCE = r"""
#include "serving.cuh"
#include <deque>
struct Job { bool ens; };
int main()
{
    const std::deque<Job> none, small(500, Job{true}), handles(6, Job{false});
    std::deque<Job> mixed = small;
    mixed.insert(mixed.end(), handles.begin(), handles.end());
    using dpd::handles_expected;
    if (handles_expected(1, none, 32) != 1) return 1;
    if (handles_expected(1, small, 32) != 1) return 2;   // one handle among ensemble boxes: alone
    if (handles_expected(2, handles, 32) != 8) return 3;
    if (handles_expected(2, mixed, 32) != 8) return 4;
    if (handles_expected(2, mixed, 3) != 3) return 5;
    return 0;
}
"""


def test_only_boxes_that_take_a_handle_count(tmp_path):
    src, exe = tmp_path / "share.cpp", tmp_path / "share"
    src.write_text(SOURCE)
    csrc = os.path.join(os.path.dirname(dpd.__file__), "csrc")
    subprocess.run(["g++", "-std=c++17", "-I", csrc, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
