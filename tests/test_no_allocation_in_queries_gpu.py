"""Queries of a grid (health checks, reductions, tip positions) allocate nothing, not even the first
time: their pinned results come with the grid, so they cannot run out of memory and the first one
costs no more than the next. A process with no pinned memory of its own would map some for a new
block (Linux shows it as a new shared mapping)."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys
sys.path.insert(0, sys.argv[1])
from paper_2101_07163_gb300 import lbmice

def shared():
    with open("/proc/self/maps") as fh:
        return {tuple(line.split()[:2]) for line in fh if line.split()[1].endswith("s")}

def grid():
    lat = lbmice.Lattice(96, 96, check_every=4)
    lat.init_seed(48, 48, 8.0, 0.3)
    lat.sync()
    return lat

def query(lat):
    lat.step(5)
    lat.stats()
    lat.tips(48, 48, [0.0, 60.0])

lat = grid()  # the kernels of every query load
query(lat)
lat.close()
new = []
for _ in range(3):
    lat = grid()
    before = shared()
    query(lat)
    new.append(len(shared() - before))
    lat.close()
print(json.dumps(new))
"""


def test_the_first_queries_of_a_grid_map_no_memory():
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    assert json.loads(r.stdout.strip().splitlines()[-1]) == [0, 0, 0]
