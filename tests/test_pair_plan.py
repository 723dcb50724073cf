"""How the two-step kernel's tasks are handed out, with the function that the
kernel compiles (lbm_pair_plan.h, built here by the C++ compiler)."""
import os
import subprocess

import pytest

from paper_2605_26677_gb300 import build


def compiled(tmp_path, main):
    (tmp_path / "main.cpp").write_text(main)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-I" + build.CSRC, str(tmp_path / "main.cpp"),
                    "-o", str(tmp_path / "main")], check=True)
    return lambda text="": subprocess.run([str(tmp_path / "main")], input=text, capture_output=True, text=True,
                                          check=True).stdout


CLAIMS = r"""
#include "lbm_pair_plan.h"
#include <cstdio>
#include <vector>
using namespace tlv;
int main()
{
    for (int warps : {1, 4, 7, 1216})
        for (int ntask : {0, 1, 3, 4, 7, 8, 1206, 1216, 1217, 5000}) {
            // the warps one after another, each to its end: the most uneven start
            int counter = 0, most = 0;
            std::vector<int> times(ntask, 0);
            for (int w = 0; w < warps; ++w) {
                int mine = 0;
                pair_tasks(
                    (unsigned)warps, (unsigned)ntask, [&] { return (unsigned)counter++; }, [](unsigned next) { return next; },
                    [&](int task) { ++times[task], ++mine; });
                most = mine > most ? mine : most;
            }
            bool once = true;
            for (int t : times) once = once && t == 1;
            std::printf("%d %d %d %d\n", warps, ntask, (int)once, most);
        }
}
"""


def test_every_task_once_and_none_twice_while_warps_wait(tmp_path):
    """Also if each warp runs to its end before the next one starts: every task
    is run once, and where there is a warp for every task, no warp takes two."""
    rows = [tuple(map(int, ln.split())) for ln in compiled(tmp_path, CLAIMS)().splitlines()]
    assert len(rows) == 40
    for warps, ntask, once, most in rows:
        assert once, (warps, ntask)
        assert ntask > warps or most <= 1, (warps, ntask, most)
