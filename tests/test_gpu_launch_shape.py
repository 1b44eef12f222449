"""The FP64 launch shape that the tuner chooses, keeps in a file and reports is one that runs: no more
time slices per CTA than the kernels take, also where a file written for other kernels holds more."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

MOST = {4: 8, 6: 8, 8: 4, 10: 4, 12: 2, 16: 1, 32: 1}
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROG = """
import sys, torch
from paper_1008_3647_gb300 import ufg
for nx in map(int, sys.argv[1].split(",")):
    lat = ufg.Lattice(nx, 640)
    before = lat.ufg_lattice_launch_shape(ufg.UFG_FP64)
    print(nx, *before, *lat.ufg_lattice_autotune()[ufg.UFG_FP64])
"""


@pytest.mark.parametrize("nxs", ["4,6,8,10,12,16"])
def test_reported_fp64_shapes_exist(tmp_path, nxs):
    cache = tmp_path / "tune"
    env = dict(os.environ, UFG_TUNE_CACHE=str(cache), PYTHONPATH=ROOT)

    def shapes():
        out = subprocess.run([sys.executable, "-c", PROG, nxs], env=env, cwd=ROOT, check=True,
                             capture_output=True, text=True).stdout
        return [list(map(int, l.split())) for l in out.splitlines()]

    first = shapes()
    for nx, c0, s0, c, s in first:
        assert c0 == c == 0 and 1 <= s0 <= MOST[nx] and 1 <= s <= MOST[nx]
    lines = cache.read_text().splitlines()
    assert shapes() == [[nx, c0, s0, 0, s] for nx, c0, s0, _, s in first]  # read back
    # lines of other kernels: clusters, more slices than a CTA takes
    cache.write_text("".join(" ".join(l.split()[:4] + ["2", "8"]) + "\n" if l.split()[3] == "0"
                             else l + "\n" for l in lines))
    for nx, _, _, c, s in shapes():
        assert c == 0 and s == MOST[nx]
