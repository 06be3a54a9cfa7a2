"""Reductions and tip queries at the sizes where their loops can go wrong."""
import numpy as np
import pytest

from paper_2101_07163_gb300 import diagnostics, lbmice, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(4, 4), (37, 29), (608, 257), (700, 413)])
@pytest.mark.parametrize("flow", [False, True])
def test_stats_against_host_sums(nx, ny, flow):
    # fewer nodes than threads, one round of the grid's threads and a remainder, several rounds;
    # FP64 sums of the exported float fields, so only the order differs: 1e-12 of the magnitudes
    w = workloads.Workload("s", nx, ny, 0, flow=flow, D=2.0, U0=0.35, L_sat=1.3, cx=nx / 2,
                           cy=ny / 2, R0=min(nx, ny) / 4)
    lat = lbmice.Lattice(nx, ny, **w.params())
    lat.set_fields(**workloads.perturbed_fields(w, nx + ny))
    lat.step(3)
    s = lat.stats()
    phi, U, rho, prev = (lat.field(k).astype(np.float64)
                         for k in (lbmice.PHI, lbmice.U, lbmice.RHO, lbmice.PHI_PREV))
    n = nx * ny
    assert abs(s["sum_phi"] - phi.sum()) < 1e-12 * n
    assert abs(s["area"] - (0.5 * (1 + phi)).sum() * w.dx ** 2) < 1e-12 * n
    assert abs(s["mass"] - rho.sum()) < 1e-12 * n
    assert abs(s["vapour_invariant"] - (U.sum() + 0.5 * w.L_sat * prev.sum())) < 2e-12 * n
    assert s["nonfinite"] == 0 and s["steps"] == 3
    lat.close()


@pytest.mark.parametrize("n,step", [(40, 0.25), (200, 0.25), (200, 0.031), (131, 7.0)])
def test_tips_against_the_host_ray_walk(n, step):
    # crossings within the first block of 256 samples and beyond it; rays that leave the grid from
    # outside the crystal; the host walk repeats the definition in double
    w = workloads.Workload("t", n, n, 0, D=2.0, U0=0.35, cx=n / 2, cy=n / 2, R0=n / 3.1)
    lat = lbmice.Lattice(n, n, **w.params())
    lat.set_fields(**workloads.seed_fields(w))
    phi = lat.field(lbmice.PHI).astype(np.float64)  # the host walk interpolates in double
    angles = np.linspace(0.0, 350.0, 37)
    for cx, cy in ((n / 2, n / 2), (n / 2 + 3.3, n / 2 - 5.1), (1.0, 1.0)):
        got = lat.tips(cx, cy, angles, step=step)
        ref = [diagnostics.tip_radius(phi, cx, cy, a, step) for a in angles]
        assert np.array_equal(np.isnan(got), np.isnan(ref))
        assert np.allclose(got, ref, rtol=0, atol=1e-9, equal_nan=True)
    lat.close()
