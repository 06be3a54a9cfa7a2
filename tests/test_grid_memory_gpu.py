"""Device memory of a grid, and exports that borrow from it."""
import numpy as np
import pytest

from paper_2101_07163_gb300 import lbmice
from paper_2101_07163_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flow,planes", [(True, 27), (False, 18)])
def test_a_grid_in_pairs_takes_no_more_memory_than_one_in_single_steps_did(flow, planes):
    # two population buffers and four floats per node beside them: phi planes, or three of these
    # and a field for host exports; a few megabytes for everything else
    import torch
    n = 4096
    p = W.Workload("m", n, n, 0, flow=flow, D=2.0, U0=0.3).params()
    warm = lbmice.Lattice(64, 64, **p)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    lat = lbmice.Lattice(n, n, **p)
    taken = free - torch.cuda.mem_get_info()[0]
    lat.close()
    warm.close()
    assert taken <= (2 * planes + 4) * 4 * n * n + (16 << 20)


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("size", [(33, 17), (64, 40), (601, 477)], ids=str)
@pytest.mark.parametrize("stencil", [4, 8])
def test_exports_leave_the_run_and_its_state_alone(storage, size, stencil):
    # a host export after every call, in every phase of the phi planes, against a run without
    nx, ny = size
    w = W.Workload("e", nx, ny, 0, flow=True, eps=0.05, D=2.0, U0=0.3, nu=0.05, cx=nx / 2,
                   cy=ny / 2, R0=ny / 5, bc=(1, 2, 3, 3), u_in=0.02, U_in=0.3, stencil=stencil)
    f = W.perturbed_fields(w, 5)
    a, b = (lbmice.Lattice(nx, ny, storage=storage, **w.params()) for _ in range(2))
    for lat in (a, b):
        lat.set_fields(**f)
    for n in (1, 2, 1, 3, 2, 2):
        for which in (lbmice.PHI, lbmice.U, lbmice.RHO, lbmice.UX, lbmice.PHI_PREV):
            a.field(which)
        a.pops()
        a.step(n)
        b.step(n)
        assert np.array_equal(a.state(), b.state()), n
    a.close()
    b.close()
