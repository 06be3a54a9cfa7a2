"""Grids with more rows than a launch may have blocks of six rows in y. Fields of period 40 in y
repeat themselves, so a tall periodic grid holds copies of a grid of 40 rows, bit for bit."""
import numpy as np
import pytest

from paper_2101_07163_gb300 import lbmice
from paper_2101_07163_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PERIOD = 40


@pytest.mark.parametrize("ny", [393_200, 393_240, 524_280])  # either side of 65535 x 6, 65535 x 8
@pytest.mark.parametrize("variant", [dict(stencil=8), dict(stencil=6, fold=4), dict(stencil=2),
                                     dict(fold=4), dict()], ids=str)
@pytest.mark.parametrize("storage,flow", [("f32", True), ("f32", False), ("bf16", True)])
def test_a_tall_grid_repeats_a_short_one(ny, variant, storage, flow):
    nx = 4
    w = W.Workload("short", nx, PERIOD, 0, flow=flow, eps=0.05, D=2.0, U0=0.35, nu=0.05,
                   cx=nx / 2, cy=PERIOD / 2, R0=8.0, **variant)
    f = W.perturbed_fields(w, 21)
    short = lbmice.Lattice(nx, PERIOD, storage=storage, **w.params())
    tall = lbmice.Lattice(nx, ny, storage=storage, **w.params())
    short.set_fields(**f)
    tall.set_fields(**{k: np.tile(v, (ny // PERIOD, 1)) for k, v in f.items()})
    for n in (1, 2):  # a single step, then a pair where the scheme takes pairs
        short.step(n)
        tall.step(n)
    want = np.tile(short.pops(), (1, ny // PERIOD, 1))
    assert np.array_equal(tall.pops(), want)
    assert np.array_equal(tall.field(lbmice.PHI_PREV),
                          np.tile(short.field(lbmice.PHI_PREV), (ny // PERIOD, 1)))
    short.close()
    tall.close()
