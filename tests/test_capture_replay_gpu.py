"""Calls captured in a CUDA graph of the user's own, launched several times: with a multiple of six
steps a call leaves the buffers as it found them, so the run goes on from launch to launch."""
import numpy as np
import pytest

from paper_2101_07163_gb300 import lbmice
from paper_2101_07163_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GRIDS = {
    "tiles": (80, 48, "f32", (1, 2, 3, 3), {}),
    "march": (850, 851, "f32", (0,) * 4, {}),
    "pairs_e8": (72, 50, "f32", (0,) * 4, dict(stencil=8)),
    "singles_e8": (80, 48, "f32", (1, 2, 3, 3), dict(stencil=8)),
    "pairs_bf16": (80, 48, "bf16", (1, 2, 3, 3), {}),
    "singles_f16": (520, 510, "f16", (0,) * 4, {}),
}


def capture(stream, call):
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        call()
    return g


@pytest.mark.parametrize("steps", [6, 12, 18, 30])
@pytest.mark.parametrize("warm", [0, 5, 6, 7])
@pytest.mark.parametrize("grid", sorted(GRIDS))
def test_a_captured_call_goes_on_from_launch_to_launch(grid, warm, steps):
    import torch
    nx, ny, storage, bc, variant = GRIDS[grid]
    w = W.Workload("g", nx, ny, 0, flow=True, eps=0.05, D=2.0, U0=0.3, U_in=0.3, nu=0.05, bc=bc,
                   u_in=0.02 if bc[0] else 0.0, cx=nx / 2, cy=ny / 2, R0=ny / 5, **variant)
    f = W.perturbed_fields(w, 13)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        a, b = (lbmice.Lattice(nx, ny, stream=st, storage=storage, **w.params()) for _ in range(2))
        for lat in (a, b):
            lat.set_fields(**f)
            lat.step(warm)
        g = capture(st, lambda: a.step(steps))
        for _ in range(3):
            g.replay()
        b.step(3 * steps)
        assert a.steps_done == warm + steps
        assert np.array_equal(a.state(), b.state())
        for lat in (a, b):  # and on by calls
            lat.step(3)
        assert np.array_equal(a.state(), b.state())
        a.close()
        b.close()


@pytest.mark.parametrize("steps", [6, 18])
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_a_captured_batch_goes_on_from_launch_to_launch(storage, steps):
    import torch
    ws = [W.Workload("g%d" % n, n, n + 3, 0, flow=True, eps=0.05, D=2.0, U0=0.3, nu=0.05, cx=n / 2,
                     cy=n / 2, R0=n / 5) for n in (40, 72, 131)]
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        a, b = (lbmice.Batch([dict(nx=w.nx, ny=w.ny, storage=storage, **w.params()) for w in ws],
                             stream=st) for _ in range(2))
        for x in (a, b):
            x.set_shape(1, 2)
            for m, w in zip(x.members, ws):
                m.init_seed(w.cx, w.cy, w.R0, w.U0)
            x.step(5)
        g = capture(st, lambda: a.step(steps))
        for _ in range(3):
            g.replay()
        b.step(3 * steps)
        for x in (a, b):
            x.step(3)
        for m, n in zip(a.members, b.members):
            assert np.array_equal(m.state(), n.state())
        a.close()
        b.close()
