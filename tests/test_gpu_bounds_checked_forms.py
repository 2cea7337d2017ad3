"""The bounds-checked build over every step form: the direct half-steps with the tape
values and both detectors that ride in them, the split half-steps and phases with their
default shapes (which the automatic choice no longer takes on small grids), the fused step
over whole grids (by name, for an odd first step of two steps per pass, and in the
borrowed buffers) and the fused reverse step.  No store may stray, and the gradient is the
split form's bit for bit, whose own is checked against the FP64 oracle."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r'''
import sys
sys.path.insert(0, "tests")
import numpy as np, torch
from oracle import oracle as O
from paper_2603_24027_gb300 import _capi as A, fdtd as F, inputs as I
import test_gpu_forward_forms as forms
assert A.LIB_PATH.endswith("_checked.so"), A.LIB_PATH
SPLIT = {A.OPT_FORWARD: 1, A.OPT_REVERSE: 1}
small = {
    "ragged70": I.ragged_box(),
    "ragged45": I.ragged_box(nx=45, ny=27, nz=23, P=5, n_steps=60, det_kind=I.OBJ_E2_PLANE,
                             src_kind=I.SRC_POINT),
    "interior150": I.ragged_box(nx=150, ny=60, nz=40, P=6, n_steps=50),
    "interior150 odd": I.ragged_box(nx=150, ny=60, nz=40, P=6, n_steps=51),
    "coupler": I.coupler_small(n_steps=60),
}
runs = 0
def gradient(w, opts, rec):
    global runs
    sim = F.Simulation(w)
    for o, v in opts.items():
        sim.set_option(o, v)
    eps = torch.from_numpy(w.eps).cuda()
    sim.forward(eps, rec)
    f = sim.step_forms()
    g = sim.backward(1.0, seed2=0.5 if w.det2_kind else 0.0)
    runs += 1
    return g, (f["forward"], f["reverse"])
for name, w in small.items():
    for tape in (("f32", 1), ("bf16", 2), ("f16", 3), ("e4m3ieee", 2), ("bdct10", 2)):
        rec = A.record_cfg(*tape)
        for mode in ({}, {A.OPT_EXACT_REVERSAL: 22}, {A.OPT_COMPACT_AUX: 0}):
            g0, f0 = gradient(w, {**SPLIT, **mode}, rec)
            assert f0 == ("split", "split")
            others = [{}]
            if name.startswith("interior150"):
                others += [{A.OPT_FORWARD: 2, A.OPT_REVERSE: 2}, {A.OPT_FORWARD: 3, A.OPT_REVERSE: 2}]
            for o in others:
                g, f = gradient(w, {**o, **mode}, rec)
                want = {0: "direct", 2: "fused", 3: "two_step"}[o.get(A.OPT_FORWARD, 0)]
                assert f == (want, "fused" if o else "direct"), (name, o, f)
                assert torch.equal(g, g0), (name, tape, mode, o)
            if tape == ("f32", 1) and A.OPT_EXACT_REVERSAL not in mode:
                ref = O.gradient2(w, 1.0, 0.5)[2] if w.det2_kind else O.gradient(w)[1]
                d = g0.cpu().numpy().astype(np.float64) - ref
                assert np.linalg.norm(d) / np.linalg.norm(ref) < 1e-4, (name, mode)
# automatic forms past the L2 cache: two steps per pass, the fused step on the pair of
# buffers and in the borrowed one
for name, form in (("deep", "two_step"), ("inside", "fused"), ("lent", "fused")):
    for n in (5, 6):
        w = forms._problem(name, n)
        rec = A.record_cfg("bf16", 2)
        g, f = gradient(w, {}, rec)
        assert f[0] == form, (name, f)
        assert torch.equal(g, gradient(w, SPLIT, rec)[0]), (name, n)
print(f"bounds-checked runs: {runs}, no stray store")
'''


def test_bounds_checked_build_runs_every_form():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2603_24027_gb300 import build as B
    B.build(checked=True)
    env = dict(os.environ, FDTD_BOUNDS_CHECKED="1", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "no stray store" in r.stdout
