"""Narrow and small grids that steps in pairs or tiles of 30 columns and 6 rows would slow down: which
kernel takes them, and the bits. Fields of period 40 in y repeat themselves, so a tall grid holds
copies of a short one, whose steps run in another form."""
import numpy as np
import pytest

from paper_2101_07163_gb300 import lbmice
from paper_2101_07163_gb300 import workloads as W
from tests.captured import launched

pytestmark = pytest.mark.gpu

PERIODIC, TUNNEL = (0, 0, 0, 0), (1, 2, 0, 0)  # inflow along x, periodic in y
PERIOD = 40


@pytest.mark.parametrize("nx,ny,storage,flow,variant,kernels", [
    # single steps where a pair takes half as many strips again, or the only strip is mostly empty
    (27, 9680, "f32", True, dict(fold=4), ["row_kernel"] * 2),
    (17, 9240, "f32", True, dict(stencil=2), ["row_kernel"] * 2),
    (9, 19160, "f32", True, {}, ["march_kernel"] * 2),
    (57, 3640, "f32", True, {}, ["march_kernel"] * 2),
    (30, 13520, "f32", False, dict(stencil=2), ["row_kernel"] * 2),
    (27, 2480, "f16", True, {}, ["march_kernel"] * 2),
    # 32 x 8 tiles, 32 or 64 columns, or one wave where row tiles need two
    (32, 4120, "f32", False, dict(stencil=2), ["tile_kernel"] * 2),
    (32, 10160, "f32", True, dict(stencil=6), ["tile_kernel"] * 2),
    (64, 3640, "bf16", True, dict(fold=4), ["tile_kernel"] * 2),
    (126, 800, "f32", False, dict(stencil=6), ["tile_kernel"] * 2),
    (128, 840, "f16", True, dict(stencil=8), ["tile_kernel"] * 2),
    # as before: pairs
    (26, 9680, "f32", False, {}, ["two_tile_kernel"]),
    (120, 1000, "f32", True, dict(fold=4), ["two_tile_kernel"]),
    (27, 160, "f32", True, dict(fold=4), ["two_tile_kernel"]),
    (32, 200, "bf16", True, {}, ["two_tile_kernel"]),
])
def test_form_and_bits(nx, ny, storage, flow, variant, kernels):
    import torch
    bc = TUNNEL if flow and not variant.get("stencil", 4) > 4 else PERIODIC
    w = W.Workload("short", nx, PERIOD, 0, flow=flow, eps=0.05, D=2.0, U0=0.35, U_in=0.3, nu=0.05, bc=bc,
                   u_in=0.02 if bc is TUNNEL else 0.0, cx=nx / 2, cy=PERIOD / 2, R0=8.0, **variant)
    f = W.perturbed_fields(w, 21)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        short = lbmice.Lattice(nx, PERIOD, stream=st, storage=storage, **w.params())
        tall = lbmice.Lattice(nx, ny, stream=st, storage=storage, **w.params())
        short.set_fields(**f)
        tall.set_fields(**{k: np.tile(v, (ny // PERIOD, 1)) for k, v in f.items()})
        for n in (1, 2, 3):
            short.step(n)
            tall.step(n)
        assert np.array_equal(tall.pops(), np.tile(short.pops(), (1, ny // PERIOD, 1)))
        assert np.array_equal(tall.field(lbmice.PHI_PREV),
                              np.tile(short.field(lbmice.PHI_PREV), (ny // PERIOD, 1)))
        names = launched(st, lambda: tall.step(2))
        short.close()
        tall.close()
    assert len(names) == len(kernels) and all(k in n for k, n in zip(kernels, names)), names
