"""The shared memory that the tile sweeps' launches ask for holds the windows that their CTAs load, at every
size and for every number of sweeps a plan can lead to (a launch of no sweeps among them). The launcher's own
code runs on the host, with the launches recorded (sweep_tiles_host.cu)."""
import math
import os
import random
import subprocess

import pytest

from paper_2208_02427_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host_side(tmp_path_factory):
    try:
        cc = build.nvcc()
    except RuntimeError as exc:
        pytest.skip(str(exc))
    exe = str(tmp_path_factory.mktemp("tiles") / "sweep_tiles_host")
    subprocess.run([cc, *build.ARCH, "-std=c++17", "-Xptxas", "-O0", "-I", build.CSRC, "-I",
                    os.path.join(build.ROOT, "include"), os.path.join(HERE, "sweep_tiles_host.cu"), "-o", exe],
                   check=True, capture_output=True)
    return exe


def sizes():
    rng = random.Random(7)
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    out = [(3, 3), (3, 4), (3, 4000), (65, 65), (513, 385), (1531, 1021), (850, 850)]
    # thin grids, where a launch may hold one sweep, in both orientations
    for thin in (3, 4, 5, 6):
        for long in [59200, 43000, 50000, 80000] + [log(300, 131000) for _ in range(300)]:
            out += [(thin, long), (long, thin)]
    out += [(log(3, 4096), log(3, 4096)) for _ in range(4000)]
    return out


def test_windows_fit(host_side):
    text = "".join(f"{m} {n} {sms}\n" for m, n in sizes() for sms in (152, 148))
    r = subprocess.run([host_side], input=text, capture_output=True, text=True, check=True)
    launches, bad, single = map(int, r.stdout.split())
    assert launches > 10000 and single > 100
    assert bad == 0, r.stderr
