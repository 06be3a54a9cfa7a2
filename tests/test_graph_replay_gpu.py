"""Replayed chunks of steps of a single grid against single launches, bit for bit. A grid replays
chunks of 60 once it has taken 240 steps by single launches; a graph belongs to the buffer phase it
was captured from, so replays begin at every phase of the population slots and phi planes."""
import numpy as np
import pytest

from paper_2101_07163_gb300 import lbmice
from paper_2101_07163_gb300 import workloads as W

pytestmark = pytest.mark.gpu

DIRECT, CHUNK = 240, 60
CHANNEL, PERIODIC = (1, 2, 3, 3), (0,) * 4

GRIDS = {
    "pairs": (80, 48, "f32", CHANNEL, {}),
    "pairs_e8": (72, 50, "f32", PERIODIC, dict(stencil=8)),
    "singles_e8": (80, 48, "f32", CHANNEL, dict(stencil=8)),  # pairs on periodic grids only
    "pairs_bf16": (80, 48, "bf16", CHANNEL, {}),
    "singles_f16": (520, 510, "f16", CHANNEL, {}),            # above 2^18 nodes
}


@pytest.mark.parametrize("grid", sorted(GRIDS))
@pytest.mark.parametrize("flow", [False, True], ids=["hg", "fgh"])
def test_replays_equal_single_launches_from_every_phase(grid, flow):
    nx, ny, storage, bc, variant = GRIDS[grid]
    w = W.Workload("g", nx, ny, 0, flow=flow, eps=0.05, D=2.0, U0=0.3, U_in=0.3,
                   u_in=0.02 if flow and bc is CHANNEL else 0.0, nu=0.05, bc=bc, cx=nx / 2, cy=ny / 2,
                   R0=ny / 5, **variant)
    f = W.perturbed_fields(w, 13)
    a, b = (lbmice.Lattice(nx, ny, storage=storage, **w.params()) for _ in range(2))
    for lat in (a, b):
        lat.set_fields(**f)
    for n in [DIRECT, 2 * CHUNK] + [1, CHUNK, 2, CHUNK, 3, CHUNK + 7] * 2:
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert a.steps_done == b.steps_done
        assert np.array_equal(a.state(), b.state()), n
    assert np.array_equal(a.pops(), b.pops())
    a.close()
    b.close()


def test_replays_go_on_after_the_grid_starts_over():
    # the count of single launches outlives an initial condition: the first 60 steps replay
    w = W.Workload("g", 80, 48, 0, flow=True, eps=0.05, D=2.0, U0=0.3, nu=0.05, cx=40, cy=24, R0=9.0)
    a, b = (lbmice.Lattice(80, 48, **w.params()) for _ in range(2))
    a.init_seed(w.cx, w.cy, w.R0, w.U0)
    a.step(DIRECT + 2 * CHUNK + 1)
    for lat in (a, b):
        lat.init_seed(w.cx, w.cy, w.R0, w.U0)
    a.step(2 * CHUNK)
    for _ in range(2 * CHUNK):
        b.step(1)
    assert np.array_equal(a.state(), b.state())
    a.close()
    b.close()
