"""Host logic of the tiled sub-cycle: every patch that holds a copy of an edge
or a cell sums its terms in the mesh's own order (tests/tile_order_check.cpp),
which is what makes the results the same bits for every patch size."""
import os
import shutil
import subprocess

import pytest

from paper_2105_13484_gb300 import inputs
from test_tile_plan import dump

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    out = str(tmp_path_factory.mktemp("tileorder") / "tile_order_check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-o", out, os.path.join(HERE, "tile_order_check.cpp"),
                    "-x", "c++", os.path.join(ROOT, "paper_2105_13484_gb300", "csrc", "tiles.cu")],
                   check=True, capture_output=True)
    return out


@pytest.mark.parametrize("name,patches", [("channel_10km", 1), ("channel_10km", 8),
                                          ("sphere_l4", 7), ("sphere_l4", 28)])
def test_every_copy_sums_in_the_mesh_order(checker, tmp_path, name, patches):
    m = inputs.workload(name)[0]
    d = str(tmp_path / name)
    dump(m, d)
    r = subprocess.run([checker, d, str(patches)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
