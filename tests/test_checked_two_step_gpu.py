"""The bounds-checked build over the launches of two steps: every index of the two-step march and
tiles, single grids and batches, of the kept states of a gradient and of the one-step kernels at
sizes that leave their first wave, is tested against its buffer (lbmice_debug_flags), and the state
is the normal build's. Runs in a child process with LBMICE_CHECKED=1; which kernel a grid takes
comes from a capture of its call."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import hashlib, json, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import torch
from paper_2101_07163_gb300 import lbmice
from paper_2101_07163_gb300 import workloads as W
from tests.captured import launched
from tests.test_two_step_forms_gpu import FORMS
from tests.test_two_step_gpu import FACES

checked = "checked" in lbmice.lib_path()
flags = lambda: lbmice.debug_flags(clear=True) if checked else 0
st = torch.cuda.Stream()
out = {"lib": lbmice.lib_path(), "runs": []}
flags()

def record(name, kernels, states):
    h = hashlib.sha256()
    for s in states:
        h.update(s.tobytes())
    out["runs"].append([name, kernels, flags(), h.hexdigest()])

def workload(nx, ny, faces, flow, **variant):
    return W.Workload("c", nx, ny, 0, flow=flow, eps=0.05, D=2.0, U0=0.3, U_in=0.3,
                      u_in=0.02 if flow else 0.0, nu=0.05, bc=FACES[faces], cx=nx / 2, cy=ny / 2,
                      R0=min(nx, ny) / 5, **variant)

runs = [f[1:] for f in FORMS]
runs += [(850, 851, f, True, "f32", {}) for f in ("periodic", "rising", "walls")]
runs += [(1460, 1451, f, False, "f32", {}) for f in ("periodic", "tunnel")]
runs += [(870, 867, "channel", True, "f32", dict(stencil=2)), (1500, 1490, "walls", False, "f32", dict(fold=4))]
runs += [(9, 13, "periodic", True, "f32", dict(stencil=8)), (4, 4, "periodic", True, "f32", {})]
with torch.cuda.stream(st):
    for nx, ny, faces, flow, storage, variant in runs:
        w = workload(nx, ny, faces, flow, **variant)
        lat = lbmice.Lattice(nx, ny, stream=st, storage=storage, **w.params())
        lat.set_fields(**W.perturbed_fields(w, 3))
        lat.step(5)
        state = lat.state()
        record("%dx%d %s" % (nx, ny, faces), launched(st, lambda: lat.step(3)), [state])
        lat.close()
    for sides in ((40, 72, 131), (8, 1024, 300)):
        for flow in (False, True):
            ws = [workload(n, n + 3, f, flow) for n, f in zip(sides, ("channel", "periodic", "rising"))]
            b = lbmice.Batch([dict(nx=w.nx, ny=w.ny, **w.params()) for w in ws], stream=st)
            for m, w in zip(b.members, ws):
                m.set_fields(**W.perturbed_fields(w, w.nx))
            b.step(5)
            states = [m.state() for m in b.members]
            record("batch %s" % (sides,), launched(st, lambda: b.step(2)), states)
            b.close()
    for n, flow in ((24, True), (150, False), (225, False), (500, False), (270, True)):
        w = workload(n, n + 5, "periodic", flow)
        lat = lbmice.Lattice(w.nx, w.ny, stream=st, **w.params())
        lat.set_fields(**W.seed_fields(w))
        tape = lbmice.Tape(lat, 7)
        tape.record(17)
        seed = np.random.default_rng(n).uniform(-1, 1, (w.ny, w.nx)).astype(np.float32)
        g, fields = tape.backward(seed, seed)
        record("tape %d" % n, [], [fields["phi0"], fields["U0"]])
        tape.close()
        lat.close()
    # the last node of the grid is the last of each buffer: extents shrunk by one are reported
    if checked:
        for nx, ny, flow in ((64, 24, True), (896, 832, True)):
            w = workload(nx, ny, "periodic", flow)
            lat = lbmice.Lattice(nx, ny, stream=st, **w.params())
            lat.init_seed(w.cx, w.cy, w.R0, w.U0)
            lbmice.debug_set_margin(1)
            lat.step(2)
            lat.sync()
            record("margin %dx%d" % (nx, ny), launched(st, lambda: lat.step(2)), [])
            lbmice.debug_set_margin(0)
            lat.close()
print(json.dumps(out))
"""


def child(checked):
    env = dict(os.environ, LBMICE_CHECKED="1" if checked else "0")
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


def test_two_step_launches_stay_inside_their_buffers():
    from paper_2101_07163_gb300 import build, lbmice
    path = build.build(checked=True)
    got, ref = child(True), child(False)
    assert got["lib"] == path
    runs = [r for r in got["runs"] if not r[0].startswith("margin")]
    for (name, kernels, flags, digest), (_, rkernels, _, rdigest) in zip(runs, ref["runs"]):
        assert flags == 0, (name, kernels)
        assert kernels == rkernels and digest == rdigest, (name, kernels)
    assert len(runs) == len(ref["runs"])
    names = " ".join(k for _, ks, _, _ in runs for k in ks)
    for form in ("two_kernelILb%dELi%dE" % (f, v) for f in (0, 1) for v in (0, 1, 2)):
        assert form in names, form
    for f in (0, 1):
        assert "batch_two_kernelILb%dE" % f in names and "batch_two_tile_kernelILb%dE" % f in names
    margin = [r for r in got["runs"] if r[0].startswith("margin")]
    assert "two_tile_kernel" in margin[0][1][0] and "two_kernel" in margin[1][1][0]
    want = lbmice.OOB_POPS | lbmice.OOB_PLANE | lbmice.OOB_SHARED
    for r in margin:  # every kind of check fires in both forms
        assert r[2] & want == want, r
