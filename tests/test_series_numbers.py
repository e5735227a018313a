"""Message numbers of the series' iterations (csrc/series.h, series_first), on the
CPU: a launch on a cluster, whose boxes start cleared to number 0, never waits for
number 0, whatever the context's counter; one with its mail in global memory goes
on where the last launch ended."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include "%s/paper_2210_06874_gb300/csrc/series.h"
#include <stdio.h>
int main() {
    const unsigned last[] = {0u, 1u, 16u, 0x7fffffffu, 0xfffffff0u, 0xfffffffeu, 0xffffffffu};
    for (unsigned l : last)
        printf("%%u %%u %%u\n", l, hmc::series_first(true, l) + 1u, hmc::series_first(false, l) + 1u);
}
"""


def test_first_number(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    (tmp_path / "m.cpp").write_text(MAIN % ROOT)
    subprocess.run([cxx, "-O2", "-o", str(tmp_path / "m"), str(tmp_path / "m.cpp")], check=True)
    out = subprocess.run([str(tmp_path / "m")], check=True, capture_output=True, text=True).stdout
    for line in out.splitlines():
        last, cluster, mail = (int(w) for w in line.split())
        assert cluster == 1
        assert mail == (last + 1) % 2 ** 32
