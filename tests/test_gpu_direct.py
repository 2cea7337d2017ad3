"""Direct half-steps of small grids (csrc/kernels_direct.cu) on the GPU.

With default options a small grid runs the direct half-steps; asking for the
split half-steps (FDTD_OPT_FORWARD = FDTD_OPT_REVERSE = 1) runs the staged
kernels.  Both evaluate the same rounded operations, so the final fields, the
tape, the reversed interior and the gradient must be equal bit for bit; the
objectives' FP64 sums may differ in their order.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2603_24027_gb300 import fdtd
    return fdtd


def _grid(name):
    from paper_2603_24027_gb300 import inputs as I
    if name == "min":         # a two-cell interior: one pair in an interior row
        return I.fd_cube().replace(nx=6, ny=6, nz=6, eps=np.ones((6, 6, 6), np.float32),
                                   design_lo=(2, 2, 2), design_hi=(4, 4, 4), src_pos=(2, 3, 2),
                                   det_index=3, det_lo=(2, 2), det_hi=(4, 4))
    if name == "thin":        # one-cell CPML, odd sizes, fewer cells than a CTA in a plane
        return I.ragged_box(nx=13, ny=17, nz=15, P=1, n_steps=41)
    if name == "odd":         # odd CPML: interior pairs cut in half on both sides
        return I.ragged_box(nx=71, ny=33, nz=29, P=5, n_steps=60, det_kind=I.OBJ_E2_PLANE,
                            src_kind=I.SRC_POINT)
    if name == "compact":     # long enough for compact auxiliaries on every axis
        return I.ragged_box(nx=150, ny=60, nz=40, P=7, n_steps=50)
    w = I.coupler_small(n_steps=70)   # two detectors
    if name == "two":
        return w
    # crossing planes: cells that both detectors seed
    P = w.pml_thickness
    return w.replace(det_kind=I.OBJ_E2_PLANE, det_axis=0, det_index=P + 8, det_lo=(P, P),
                     det_hi=(w.ny - P, w.nz - P), det2_kind=I.OBJ_POYNTING_PLANE, det2_axis=1,
                     det2_index=w.ny - P - 1, det2_lo=(P, P), det2_hi=(w.nx - P, w.nz - P))


def _run(F, w, rec, options):
    sim = F.Simulation(w, device="cuda")
    for k, v in options.items():
        sim.set_option(k, v)
    sim.ensure_workspace(rec).zero_()   # row and sample padding, which the saved state includes
    sim.forward(torch.from_numpy(w.eps).cuda(), rec)
    hist, obj = sim.objective_history(), sim.objectives()
    fields, state = sim.read_fields().clone(), sim.save_state()
    g = sim.backward(0.75, seed2=-0.5 if w.det2_kind else None).double().cpu().numpy()
    return dict(hist=hist, obj=obj, fields=fields, state=state, grad=g, back=sim.read_fields(),
                launches=sim.last_timing())


@pytest.mark.parametrize("exact", [0, 22])
@pytest.mark.parametrize("tape,k,interp", [("f32", 1, "linear"), ("bf16", 3, "cubic"),
                                           ("e4m3", 4, "linear"), ("e5m2fnuz", 5, "cubic"),
                                           ("bdct", 4, "cubic")])
@pytest.mark.parametrize("name", ["min", "thin", "odd", "compact", "two", "cross"])
def test_direct_half_steps_equal_the_staged_ones(F, name, tape, k, interp, exact):
    from paper_2603_24027_gb300 import _capi as A
    w = _grid(name)
    rec = A.record_cfg(tape, k, interp)
    ex = {A.OPT_EXACT_REVERSAL: exact}
    a = _run(F, w, rec, ex)
    b = _run(F, w, rec, {**ex, A.OPT_FORWARD: 1, A.OPT_REVERSE: 1})
    # two launches a reverse step (and one that starts the loop)
    assert a["launches"]["bwd_launches"] == 2 * w.n_steps + 1
    assert torch.equal(a["fields"], b["fields"])
    P = w.pml_thickness
    core = (slice(None),) + tuple(slice(P, n - P) for n in (w.nz, w.ny, w.nx))
    assert torch.equal(a["back"][core], b["back"][core])
    # the saved state holds the tape
    n = 8 * w.n_steps * 2
    head = len(a["state"]) - n
    skip = 128   # header: the second objective's sum
    assert np.array_equal(a["state"][skip:head], b["state"][skip:head])
    np.testing.assert_allclose(a["hist"], b["hist"], rtol=0, atol=1e-12 * np.abs(b["hist"]).max())
    np.testing.assert_allclose(a["obj"], b["obj"], rtol=1e-11)
    assert np.array_equal(a["grad"], b["grad"])


@pytest.mark.parametrize("nx,ny,nz,direct", [(201, 173, 172, True), (202, 175, 171, False)])
def test_the_largest_grids_of_the_direct_forward(F, nx, ny, nz, direct):
    """Either side of the line (6 million cells): the same fields, tape and gradient as the
    split half-steps, whichever form runs."""
    from paper_2603_24027_gb300 import _capi as A
    from paper_2603_24027_gb300 import inputs as I
    w = I.ragged_box(nx=nx, ny=ny, nz=nz, P=9, n_steps=24)
    rec = A.record_cfg("bf16", 3, "cubic")
    a = _run(F, w, rec, {})
    b = _run(F, w, rec, {A.OPT_FORWARD: 1, A.OPT_REVERSE: 1})
    assert (a["launches"]["fwd_launches"] == 2 * w.n_steps) == direct
    assert torch.equal(a["fields"], b["fields"])
    skip, n = 128, 8 * w.n_steps * 2
    assert np.array_equal(a["state"][skip:len(a["state"]) - n], b["state"][skip:len(b["state"]) - n])
    assert np.array_equal(a["grad"], b["grad"])


@pytest.mark.parametrize("sizes,split", [((44, 60, 128), {60, 128}),   # above 2 million cells
                                         ((44, 60, 96), set())])       # below
def test_a_groups_backward_equals_each_handles_own(F, sizes, split):
    """A large group's backward runs its larger grids as split phases; the gradients stay the
    own runs', whose form a group call does not change."""
    from paper_2603_24027_gb300 import _capi as A
    from paper_2603_24027_gb300 import inputs as I
    ws = [I.ragged_box(nx=n, ny=n, nz=n, P=7, n_steps=31, seed=n) for n in sizes]
    rec = A.record_cfg("bf16", 3)
    eps = [torch.from_numpy(w.eps).cuda() for w in ws]
    sims = [F.Simulation(w, device="cuda") for w in ws]
    own = []
    for s, e in zip(sims, eps):
        s.forward(e, rec)
        own.append((s.backward(0.5).clone(), s.last_timing()["bwd_launches"]))
    F.group_forward(sims, eps, rec)
    grads = F.group_backward(sims, [0.5] * len(sims))
    for w, s, g, (g0, n0) in zip(ws, sims, grads, own):
        assert torch.equal(g, g0)
        assert (s.last_timing()["bwd_launches"] > 2 * w.n_steps + 1) == (w.nx in split)
    for s, e, (g0, n0) in zip(sims, eps, own):
        s.forward(e, rec)
        assert torch.equal(s.backward(0.5), g0)
        assert s.last_timing()["bwd_launches"] == n0


def test_sampled_timing_of_a_small_grid_keeps_its_kinds(F):
    """With kernel timing sampled, every kind has its own launch again; the results stay."""
    from paper_2603_24027_gb300 import _capi as A
    w = _grid("two")
    rec = A.record_cfg("bf16", 2)
    a = _run(F, w, rec, {})
    b = _run(F, w, rec, {A.OPT_SAMPLE_EVERY: 3})
    assert torch.equal(a["fields"], b["fields"])
    assert a["launches"]["fwd_launches"] == 2 * w.n_steps
    assert b["launches"]["fwd_launches"] == 3 * w.n_steps + (w.n_steps + 1) // 2
    assert b["launches"]["bwd_launches"] == 3 * w.n_steps


@pytest.mark.parametrize("options", [{}, {"OPT_FORWARD": 1, "OPT_REVERSE": 1}])
def test_detectors_that_share_cells(F, options):
    """Both detectors' seeds arrive at the cells their planes share: the gradient of the
    weighted sum against the FP64 oracle."""
    from oracle import oracle as O
    from paper_2603_24027_gb300 import _capi as A
    w = _grid("cross")
    r = _run(F, w, A.record_cfg("f32", 1), {getattr(A, k): v for k, v in options.items()})
    _, _, g = O.gradient2(w, 0.75, -0.5)
    assert np.linalg.norm(r["grad"] - g) <= 1e-4 * np.linalg.norm(g)
