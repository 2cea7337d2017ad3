"""The automatic forward past the L2 cache with a second detector and with exact reversal,
and one z group by name, on the GPU: equal to the split half-steps bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(w, rec, options):
    from paper_2603_24027_gb300 import _capi as A
    from paper_2603_24027_gb300 import fdtd as F
    sim = F.Simulation(w, device="cuda")
    for k, v in options.items():
        sim.set_option(k, v)
    sim.forward(torch.from_numpy(w.eps).cuda(), rec)
    out = (sim.objectives(), sim.read_fields().clone(),
           sim.backward(1.0, seed2=-0.5 if w.det2_kind else 0.0).clone())
    return out, sim.step_forms()


def _equal(a, b):
    for x, y in zip(a[0], b[0]):
        assert x == pytest.approx(y, rel=1e-12)
    assert a[0][0] != 0.0
    assert torch.equal(a[1], b[1])
    assert torch.equal(a[2], b[2]) and float(a[2].abs().max()) > 0


@pytest.mark.parametrize("n_steps", [12, 13])
@pytest.mark.parametrize("exact", [0, 22])
@pytest.mark.parametrize("name,form", [("deep", "two_step"), ("inside", "fused"), ("lent", "fused")])
def test_automatic_forward_with_two_detectors(name, form, exact, n_steps):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2603_24027_gb300 import _capi as A
    from paper_2603_24027_gb300 import inputs as I
    from test_gpu_forward_forms import _problem
    w = _problem(name, n_steps)
    P = w.pml_thickness
    # beside the first detector, its window smaller by a cell on every side
    w = w.replace(det2_kind=I.OBJ_E2_PLANE, det2_axis=0, det2_index=w.det_index - 2,
                  det2_lo=(P + 1, P + 1), det2_hi=(w.ny - P - 1, w.nz - P - 1))
    rec = A.record_cfg("bf16", 5)
    split = {A.OPT_FORWARD: 1, A.OPT_REVERSE: 1}
    mode = {A.OPT_EXACT_REVERSAL: exact} if exact else {}
    a, forms = _run(w, rec, mode)
    assert forms["forward"] == form
    _equal(a, _run(w, rec, {**split, **mode})[0])


@pytest.mark.parametrize("grid", [(301, 203, 151, 10), (400, 80, 70, 4)])
def test_one_z_group_by_name(grid):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import numpy as np
    from paper_2603_24027_gb300 import _capi as A
    from test_step_forms import problem
    w = problem(*grid)
    rng = np.random.default_rng(2)
    w = w.replace(n_steps=9, t0_over_tau=0.0, rel_bandwidth=2.0,
                  eps=rng.uniform(1.0, 12.25, (w.nz, w.ny, w.nx)).astype(np.float32))
    rec = A.record_cfg("bf16", 2)
    a, forms = _run(w, rec, {A.OPT_ZGROUPS: 1})
    assert forms["forward"] == "split" and forms["reverse"] == "fused"
    _equal(a, _run(w, rec, {A.OPT_FORWARD: 3, A.OPT_REVERSE: 1})[0])
