"""The forms of two-step launches at the sizes that select them, named by a capture of the call,
against single steps: the same bits."""
import numpy as np
import pytest

from paper_2101_07163_gb300 import lbmice, workloads
from tests.captured import launched
from tests.test_two_step_gpu import FACES, compare_pairs

pytestmark = pytest.mark.gpu

# name of the kernel: march or tile, warps, variant (0 E4 six-fold, 1 other reach of one, 2 reach of
# two) <- nx, ny, faces, flow, storage, stencil and fold
FORMS = [
    ("two_kernelILb1ELi0E", 850, 851, "channel", True, "f32", {}),
    ("two_kernelILb0ELi0E", 1460, 1451, "rising", False, "f32", {}),
    ("two_kernelILb1ELi1E", 850, 851, "tunnel", True, "f32", dict(fold=4)),
    ("two_kernelILb0ELi1E", 1460, 1451, "periodic", False, "f32", dict(stencil=2)),
    ("two_kernelILb0ELi1E", 1460, 1451, "channel", False, "f32", dict(fold=4)),
    ("two_kernelILb1ELi2E", 770, 767, "periodic", True, "f32", dict(stencil=8)),
    ("two_kernelILb0ELi2E", 1300, 1211, "periodic", False, "f32", dict(stencil=6)),
    ("two_tile_kernelILb1ELi8ELb0ELi0E", 40, 36, "channel", True, "f32", {}),
    ("two_tile_kernelILb0ELi12ELb0ELi0E", 200, 198, "channel", False, "f32", {}),
    ("two_tile_kernelILb0ELi16ELb0ELi0E", 230, 225, "falling", False, "f32", {}),
    ("two_tile_kernelILb0ELi20ELb0ELi0E", 403, 397, "channel", False, "f32", {}),
    ("two_tile_kernelILb1ELi16ELb0ELi0E", 700, 413, "rising", True, "f32", {}),
    ("two_tile_kernelILb1ELi12ELb0ELi1E", 150, 130, "channel", True, "f32", dict(stencil=2)),
    ("two_tile_kernelILb0ELi20ELb0ELi1E", 501, 499, "walls", False, "f32", dict(fold=4)),
    ("two_tile_kernelILb0ELi12ELb0ELi2E", 100, 90, "periodic", False, "f32", dict(stencil=8)),
    ("two_tile_kernelILb1ELi16ELb0ELi2E", 256, 250, "periodic", True, "f32", dict(stencil=6, fold=4)),
    ("two_tile_kernelILb0ELi20ELb0ELi2E", 801, 799, "periodic", False, "f32", dict(stencil=8)),
    ("two_tile_kernelILb1ELi12ELb0ELi0ENS_4BF16E", 60, 50, "tunnel", True, "bf16", {}),
    ("two_tile_kernelILb0ELi16ELb0ELi0ENS_3F16E", 500, 490, "falling", False, "f16", {}),
]


@pytest.mark.parametrize("name,nx,ny,faces,flow,storage,variant", FORMS,
                         ids=["%s_%dx%d" % (f[0].replace("_kernelI", "_"), f[1], f[2]) for f in FORMS])
def test_form_and_bits(name, nx, ny, faces, flow, storage, variant):
    import torch
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        lat = lbmice.Lattice(nx, ny, stream=st, flow=flow, storage=storage, bc=FACES[faces], nu=0.05,
                             **variant)
        lat.init_seed(nx / 2, ny / 2, 5.0, 0.3)
        lat.sync()
        names = launched(st, lambda: lat.step(2))
        lat.close()
    assert len(names) == 1 and name in names[0], names
    compare_pairs(nx, ny, faces, flow, (2, 5), storage=storage, **variant)


# below and above 2^20 nodes in all: tiles and the march
@pytest.mark.parametrize("sides,name", [((40, 72, 131), "batch_two_tile_kernelILb%dELi16E"),
                                        ((8, 1024, 300), "batch_two_kernelILb%dE")], ids=str)
@pytest.mark.parametrize("flow", [False, True], ids=["hg", "fgh"])
def test_batched_form_and_bits(sides, name, flow):
    import torch
    st = torch.cuda.Stream()
    ws = [workloads.Workload(f"b{n}", n, n + 3, 0, flow=flow, eps=0.05, D=2.0, U0=0.3, U_in=0.3,
                             u_in=0.02 if flow else 0.0, nu=0.05, bc=FACES[fc], cx=n / 2, cy=n / 2,
                             R0=n / 5) for n, fc in zip(sides, ("channel", "periodic", "rising"))]
    cfg = [dict(nx=v.nx, ny=v.ny, **v.params()) for v in ws]
    with torch.cuda.stream(st):
        b = lbmice.Batch(cfg, stream=st)
        for m, v in zip(b.members, ws):
            m.init_seed(v.cx, v.cy, v.R0, v.U0)
        b.sync()
        names = launched(st, lambda: b.step(2))
        b.close()
    assert len(names) == 1 and name % flow in names[0], names
    b = lbmice.Batch(cfg)
    singles = [lbmice.Lattice(**c) for c in cfg]
    for m, lat, v in zip(b.members, singles, ws):
        f = workloads.perturbed_fields(v, v.nx)
        m.set_fields(**f)
        lat.set_fields(**f)
    for n in (1, 2, 61, 5):
        b.step(n)
        for m, lat in zip(b.members, singles):
            for _ in range(n):
                lat.step(1)
            assert np.array_equal(m.pops(), lat.pops()), n
    b.close()


@pytest.mark.parametrize("n,every", [(24, 9), (150, 8), (225, 7), (500, 6), (700, 5)])
def test_states_recomputed_in_pairs_without_flow(n, every):
    # tiles of 8, 12, 16 and 20 warps that keep the state in between
    w = workloads.Workload("pairs_grad", n, n + 5, 0, eps=0.05, D=2.0, U0=0.3, cx=n / 2, cy=n / 2,
                           R0=n / 5)
    f = workloads.seed_fields(w)
    seed = np.random.default_rng(n).uniform(-1, 1, (w.ny, w.nx))
    got = []
    for interval in (1, every):
        lat = lbmice.Lattice(w.nx, w.ny, **w.params())
        lat.set_fields(**f)
        tape = lbmice.Tape(lat, interval)
        tape.record(2 * every + 3)
        got.append(tape.backward(seed, seed))
        tape.close()
        lat.close()
    assert got[0][0] == got[1][0]
    for k in lbmice.INIT_NAMES:
        assert np.array_equal(got[0][1][k], got[1][1][k]), k
