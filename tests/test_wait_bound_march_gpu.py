"""The bounded waits of the two-step march: its steps run, and report nothing, after a wait of the
self-test gave up."""
import numpy as np
import pytest

from paper_2101_07163_gb300 import lbmice
from paper_2101_07163_gb300 import workloads as W
from tests.captured import launched

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,storage,kernel", [
    ({}, "f32", "two_kernelILb1ELi0E"), (dict(stencil=8), "f32", "two_kernelILb1ELi2E"),
    ({}, "f16", "march_kernelILb1E")], ids=["pairs", "pairs_e8", "singles_f16"])
def test_marches_run_after_a_timeout_and_report_none(variant, storage, kernel):
    import torch
    # most CTAs lie away from the faces: their phi rows come by tensor map, with the ring's waits
    w = W.Workload("wait", 900, 870, 1, flow=True, eps=0.05, D=2.0, U0=0.3, nu=0.05, cx=450.0,
                   cy=435.0, R0=20.0, **variant)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        lat = lbmice.Lattice(w.nx, w.ny, stream=st, storage=storage, **w.params())
        lat.init_seed(w.cx, w.cy, w.R0, w.U0)
        lat.sync()
        assert kernel in launched(st, lambda: lat.step(2))[0]
        lat.close()
        assert lbmice.lib().lbmice_debug_wait_selftest() == lbmice.ETIMEOUT
        lat = lbmice.Lattice(w.nx, w.ny, stream=st, storage=storage, check_every=4, **w.params())
        lat.init_seed(w.cx, w.cy, w.R0, w.U0)
        lat.step(13)  # health checks read the wait word
        assert lat.stats()["nonfinite"] == 0.0
        assert np.isfinite(lat.field(lbmice.PHI)).all()
        lat.close()
