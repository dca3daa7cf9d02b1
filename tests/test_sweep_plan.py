"""The server's tile plan: no dearer by its cost model than a search of every pair of tile sides over every field,
and found in a fraction of that search's time, with the device idle meanwhile (sweep_plan_host.cu)."""
import os
import subprocess

import pytest

from paper_2208_02427_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_plan(tmp_path):
    try:
        cc = build.nvcc()
    except RuntimeError as exc:
        pytest.skip(str(exc))
    exe = str(tmp_path / "sweep_plan_host")
    subprocess.run([cc, *build.ARCH, "-O3", "-std=c++17", "-Xptxas", "-O0", "-I", build.CSRC, "-I",
                    os.path.join(build.ROOT, "include"), os.path.join(HERE, "sweep_plan_host.cu"), "-o", exe],
                   check=True, capture_output=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    worst, fast, plain = map(float, out.split())
    assert worst <= 1.0 + 1e-9
    # (the search, one evaluation a pair, takes as long as `plain`, the plan about a quarter of that)
    assert fast <= plain / 2
