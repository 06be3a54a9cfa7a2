"""Launches that take two time steps at once against launches of one step: the same bits, over
the faces, and over sizes at the edges of the strips (26 columns), passes (8 rows) and
segments, down to the smallest grid."""
import numpy as np
import pytest

from paper_2101_07163_gb300 import lbmice, workloads

pytestmark = pytest.mark.gpu

P, I, O, F = 0, 1, 2, 3
FACES = {"periodic": (P, P, P, P), "channel": (I, O, F, F), "rising": (F, O, I, O),
         "falling": (P, P, O, I), "tunnel": (O, I, P, P), "walls": (F, F, F, F)}
SIZES = [(4, 4), (5, 7), (25, 8), (26, 9), (27, 16), (33, 17), (52, 83), (80, 31), (131, 170)]
# the tile sizes up to their limits (2 CTAs per SM), and the march beyond 2^20 nodes with
# segments of more than one pass
LARGE = [(211, 199), (256, 250), (310, 255), (1030, 1021), (1045, 1203), (1460, 1451)]


def compare_pairs(nx, ny, faces, flow, counts, storage="f32", **variant):
    w = workloads.Workload("pairs", nx, ny, 0, flow=flow, eps=0.05, D=2.0, U0=0.35, U_in=0.3,
                           u_in=0.02 if flow else 0.0, nu=0.016, bc=FACES[faces],
                           cx=nx / 2, cy=ny / 2, R0=min(nx, ny) / 4, **variant)
    f = workloads.perturbed_fields(w, nx * 1000 + ny)
    a, b = (lbmice.Lattice(nx, ny, storage=storage, **w.params()) for _ in range(2))
    for lat in (a, b):
        lat.set_fields(**f)
    for n in counts:
        for _ in range(n):
            a.step(1)
        b.step(n)
        assert a.steps_done == b.steps_done
        for which in (lbmice.PHI, lbmice.PHI_PREV):
            assert np.array_equal(a.field(which), b.field(which)), (n, which)
        assert np.array_equal(a.pops(), b.pops()), n
        assert np.isfinite(a.field(lbmice.PHI)).all()
    assert np.array_equal(a.state(), b.state())
    a.close()
    b.close()


@pytest.mark.parametrize("faces", sorted(FACES))
@pytest.mark.parametrize("size", SIZES, ids=lambda s: "%dx%d" % s)
@pytest.mark.parametrize("flow", [False, True], ids=["hg", "fgh"])
def test_steps_in_pairs_equal_single_steps(faces, size, flow):
    # pairs, a pair and a single, replayed chunks, both population slots
    compare_pairs(*size, faces, flow, (2, 3, 8, 1, 64))


@pytest.mark.parametrize("faces", ["periodic", "channel", "rising"])
@pytest.mark.parametrize("size", LARGE, ids=lambda s: "%dx%d" % s)
@pytest.mark.parametrize("flow", [False, True], ids=["hg", "fgh"])
def test_steps_in_pairs_on_larger_grids(faces, size, flow):
    compare_pairs(*size, faces, flow, (6, 1))


@pytest.mark.parametrize("stencil,fold", [(2, 6), (4, 4), (6, 4), (8, 6)])
@pytest.mark.parametrize("size", [(8, 8), (9, 13), (24, 25), (49, 31), (150, 170), (290, 300),
                                  (601, 333), (1030, 1021)], ids=lambda s: "%dx%d" % s)
@pytest.mark.parametrize("faces,flow", [("periodic", False), ("periodic", True), ("channel", True)])
def test_variants_in_pairs_equal_single_steps(stencil, fold, size, faces, flow):
    # stencils of reach one on any grid; of reach two on periodic grids (others step singly), in
    # tiles up to 256 x 256 and in marches beyond, down to the smallest size taken in pairs
    compare_pairs(*size, faces, flow, (2, 5), stencil=stencil, fold=fold)


@pytest.mark.parametrize("stencil,fold", [(6, 6), (8, 4)])
@pytest.mark.parametrize("size", [(770, 767), (1027, 1531), (1300, 1211)], ids=lambda s: "%dx%d" % s)
@pytest.mark.parametrize("flow", [False, True], ids=["hg", "fgh"])
def test_far_reaching_variants_on_large_grids_equal_single_steps(stencil, fold, size, flow):
    # without flow the smallest and largest grids that 20-warp tiles take, else the march
    compare_pairs(*size, "periodic", flow, (2, 5), stencil=stencil, fold=fold)


@pytest.mark.parametrize("size", [(848, 850), (850, 851)], ids=lambda s: "%dx%d" % s)
def test_largest_tiled_and_smallest_marched_grid_with_flow(size):
    compare_pairs(*size, "channel", True, (4, 3))


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("faces", ["periodic", "channel", "rising", "tunnel"])
@pytest.mark.parametrize("size", [(4, 4), (27, 16), (52, 83), (131, 170), (310, 255)],
                         ids=lambda s: "%dx%d" % s)
@pytest.mark.parametrize("flow", [False, True], ids=["hg", "fgh"])
def test_sixteen_bit_steps_in_pairs_equal_single_steps(storage, faces, size, flow):
    # the deviations of the step in between are rounded in registers as a single step rounds them
    # for memory
    compare_pairs(*size, faces, flow, (2, 3, 8, 1, 64), storage=storage)


@pytest.mark.parametrize("sides", [(40, 72, 131), (8, 256, 53), (1024, 72, 300)], ids=str)
def test_batched_pairs_equal_single_grids(sides):
    ws = [workloads.Workload(f"b{n}", n, n + 3, 0, flow=True, eps=0.05, D=2.0, U0=0.3, U_in=0.3,
                             u_in=0.02, nu=0.05, bc=FACES[fc], cx=n / 2, cy=n / 2, R0=n / 5)
          for n, fc in zip(sides, ("channel", "periodic", "rising"))]
    b = lbmice.Batch([dict(nx=v.nx, ny=v.ny, **v.params()) for v in ws])
    b.set_shape(1, 1)  # a tile shape among the marches: its pairs are two launches
    singles = []
    for m, v in zip(b.members, ws):
        f = workloads.perturbed_fields(v, v.nx)
        m.set_fields(**f)
        lat = lbmice.Lattice(v.nx, v.ny, **v.params())
        lat.set_fields(**f)
        singles.append(lat)
    for n in (1, 2, 61, 5):
        b.step(n)
        for m, lat in zip(b.members, singles):
            for _ in range(n):
                lat.step(1)
            assert np.array_equal(m.pops(), lat.pops()), n
    b.close()


@pytest.mark.parametrize("n,every", [(24, 9), (36, 10), (150, 8), (270, 7)])
def test_states_recomputed_in_pairs_give_the_gradients_of_single_states(n, every):
    # a checkpoint interval of 1 recomputes nothing, one of `every` recomputes pairs of states in
    # tiles of 8, 12 or 16 warps (and a single state where the interval is odd)
    w = workloads.Workload("pairs_grad", n, n + 5, 0, flow=True, eps=0.05, D=2.0, U0=0.3, nu=0.05,
                           cx=n / 2, cy=n / 2, R0=n / 5)
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
