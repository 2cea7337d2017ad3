"""Schedules of the time loops (which launch goes to which stream, what waits for
what), on the host against a CUDA runtime that only logs."""
import pytest

import schedule_log as S
from paper_2603_24027_gb300 import _capi as A
from test_step_forms import problem


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return S.load(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def run(lib, monkeypatch):
    lib.fake_clear()
    return S.Runner(lib, monkeypatch)


REC = A.record_cfg("bf16", 2)


@pytest.mark.parametrize("zgroups,streams", [(0, 4), (1, 1), (2, 4), (3, 4)])
def test_fused_reverse_launches_have_their_own_streams(run, zgroups, streams):
    """Primal, CPML-free, z-only and ring launches of a reverse step overlap for every
    number of z groups but one, also after a split forward (the source lies in the deep
    box), which asks for no more streams than its groups."""
    sim = run.sim(problem(301, 203, 151, 10, inside=True), REC, {A.OPT_ZGROUPS: zgroups,
                                                                 A.OPT_FORWARD: 1})
    assert sim.step_forms() == {"forward": "split", "reverse": "fused"}
    run.forward(sim, REC)
    log = run.backward(sim)
    rev = [e for e in log if e.what == "launch" and "k_rev_" in e.name]
    assert len(rev) == 4 * sim.w.n_steps
    assert len({e.a for e in rev}) == streams
