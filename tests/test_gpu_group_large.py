"""Group forwards of grids whose state no cache holds, on the GPU: the loops run side by
side, two steps per pass where a grid may although a single run of its size is split, and
the fields, the gradients and later single runs are those of each design's own run."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_steps", [(9, 12), (10, 7)])
def test_large_group_equals_own_runs(n_steps):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2603_24027_gb300 import _capi as A
    from paper_2603_24027_gb300 import build as B
    from paper_2603_24027_gb300 import fdtd as F
    from test_step_forms import problem
    B.build()
    rec = A.record_cfg("bf16", 3)
    rng = np.random.default_rng(5)
    # 9.2 M cells (deep units; split by itself) and 4 M cells (direct)
    ws = [problem(301, 203, 151, 10), problem(301, 203, 151, 10), problem(200, 200, 100, 12)]
    ws = [w.replace(n_steps=n, t0_over_tau=0.0, rel_bandwidth=2.0,
                    eps=rng.uniform(1.0, 12.25, (w.nz, w.ny, w.nx)).astype(np.float32))
          for w, n in zip(ws, (n_steps[0], n_steps[1], n_steps[0]))]
    eps = [torch.from_numpy(w.eps).cuda() for w in ws]
    own = []
    for w, e in zip(ws, eps):
        sim = F.Simulation(w, device="cuda")
        L = sim.forward(e, rec)
        own.append((L, sim.read_fields().clone(), sim.backward(1.0).clone(),
                    sim.last_timing()["fwd_launches"]))
    sims = [F.Simulation(w, device="cuda") for w in ws]
    for _ in range(2):   # the captured loops, then their replay
        Ls = F.group_forward(sims, eps, rec)
        fields = [s.read_fields().clone() for s in sims]
        launches = [s.last_timing()["fwd_launches"] for s in sims]
        gs = F.group_backward(sims)
        for i, (L, f, g, _) in enumerate(own):
            assert Ls[i] == pytest.approx(L, rel=1e-12) and L != 0.0
            assert torch.equal(fields[i], f)
            assert torch.equal(gs[i], g) and float(g.abs().max()) > 0
    # another form ran in the group, and a single run takes its own again
    assert launches[0] != own[0][3] and launches[2] == own[2][3]
    assert sims[0].forward(eps[0], rec) == pytest.approx(own[0][0], rel=1e-12)
    assert sims[0].last_timing()["fwd_launches"] == own[0][3]
    assert torch.equal(sims[0].read_fields(), own[0][1])
    assert torch.equal(sims[0].backward(1.0), own[0][2])
