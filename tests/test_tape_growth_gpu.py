"""A tape that is swept after every few recorded steps, as a fit over a growing horizon does."""
import gc

import numpy as np
import pytest

from paper_2101_07163_gb300 import lbmice
from paper_2101_07163_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_work_space_grows_a_few_times_and_not_at_every_sweep():
    import torch
    n, every, each, sweeps = 160, 64, 6, 12  # sweeps at 6, 12, ..., 72 steps
    w = W.Workload("growth", n, n, 0, flow=True, eps=0.05, D=2.0, U0=0.3, nu=0.05, cx=n / 2,
                   cy=n / 2, R0=n / 5)
    f = W.seed_fields(w)
    seed = np.random.default_rng(3).uniform(-1, 1, (n, n))

    def start():
        lat = lbmice.Lattice(n, n, **w.params())
        lat.set_fields(**f)
        return lat, lbmice.Tape(lat, every)

    gc.collect()  # grids that earlier tests left behind give their memory back now
    lat, tape = start()
    grown = 0
    for _ in range(sweeps):
        tape.record(each)
        before = torch.cuda.mem_get_info()[0]
        got = tape.backward(seed, seed)
        grown += torch.cuda.mem_get_info()[0] < before
    # room for 6, 24, 60 and 64 steps (2.8 MB a step)
    assert grown <= 4
    tape.close()
    lat.close()

    lat, tape = start()
    tape.record(each * sweeps)
    want = tape.backward(seed, seed)
    assert got[0] == want[0]
    for k in lbmice.INIT_NAMES:
        assert np.array_equal(got[1][k], want[1][k]), k
    tape.close()
    lat.close()
