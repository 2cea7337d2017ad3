"""The forward's automatic choice on grids past the L2 cache, on the GPU.

From 12 million cells on a forward runs two steps per pass where it may, else
the fused step (csrc/kernels_fwd_fused.cu): on the layout's pair of field
buffers, or, with one field buffer, on that and the adjoint's.  Every form
evaluates the same rounded operations as the split half-steps: the fields, the
tape and the gradient are equal bit for bit.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _problem(name, n_steps):
    from paper_2603_24027_gb300 import inputs as I
    rng = np.random.default_rng(3)
    if name == "lent":      # most units carry CPML terms: one field buffer
        nx, ny, nz, P = 1600, 92, 84, 16
    else:
        nx, ny, nz, P = 241, 235, 219, 6
    lo = (P + 3, ny // 2 - 10, nz // 2 - 4)
    w = I.Workload(name=name, nx=nx, ny=ny, nz=nz, dx=20e-9, dt=I.cfl_dt(20e-9), n_steps=n_steps,
                   pml_thickness=P, eps=rng.uniform(1.0, 12.25, (nz, ny, nx)).astype(np.float32),
                   design_lo=lo, design_hi=(lo[0] + 9, lo[1] + 20, lo[2] + 8),
                   src_kind=I.SRC_PLANE_GAUSS, src_component=1, src_axis=0,
                   src_pos=(P + 1, ny // 2, nz // 2), src_sigma_uv=(9.0, 7.0), rel_bandwidth=1.0,
                   t0_over_tau=1.2, det_kind=I.OBJ_POYNTING_PLANE, det_axis=0, det_index=P + 5,
                   det_lo=(P, P), det_hi=(ny - P, nz - P))
    if name == "inside":    # the source inside the deep box: no two-step pass
        w = w.replace(src_pos=(nx // 2, ny // 2, nz // 2), design_lo=(nx // 2 + 2,) + lo[1:],
                      design_hi=(nx // 2 + 9, lo[1] + 20, lo[2] + 8), det_index=nx // 2 + 3)
    return w


@pytest.mark.parametrize("n_steps", [14, 15])
@pytest.mark.parametrize("name,launches", [("deep", 9), ("inside", 10), ("lent", 10)])
def test_automatic_forward_equals_the_split_half_steps(name, launches, n_steps):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2603_24027_gb300 import _capi as A
    from paper_2603_24027_gb300 import fdtd as F
    w = _problem(name, n_steps)
    eps = torch.from_numpy(w.eps).cuda()
    rec = A.record_cfg("bf16", 7)
    out = []
    for options in ({}, {A.OPT_FORWARD: 1, A.OPT_REVERSE: 1}):
        sim = F.Simulation(w, device="cuda")
        for k, v in options.items():
            sim.set_option(k, v)
        L = sim.forward(eps, rec)
        t = sim.last_timing()["fwd_launches"]
        fields = sim.read_fields()
        out.append((L, fields, sim.backward(1.0), t))
        del sim
    (La, fa, ga, ta), (Lb, fb, gb, _) = out
    # per pair of steps: the pass and two fused steps of four launches; a fused step: five
    pairs, odd = divmod(n_steps, 2)
    records = (n_steps - 1) // 7 + 1
    assert ta == records + (pairs * launches + 5 * odd)
    assert La == pytest.approx(Lb, rel=1e-12) and Lb != 0.0
    assert torch.equal(fa, fb)
    assert torch.equal(ga, gb) and float(gb.abs().max()) > 0
