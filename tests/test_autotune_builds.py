"""Autotuner cache entries of another build of the library, on the host."""
from paper_2603_24027_gb300 import _capi as A
from paper_2603_24027_gb300 import autotune as T
from test_autotune_host import FakeSim


def test_an_entry_of_another_build_is_not_applied(tmp_path, monkeypatch):
    path, rec = str(tmp_path / "tune.json"), A.record_cfg("bf16", 4)
    run = dict(cache=path, gpu_name="GB300", max_passes=1)
    with monkeypatch.context() as m:
        m.setattr(T, "B", type("Build", (), {"source_digest": staticmethod(lambda: "other")}),
                  raising=False)
        old = T.tune(FakeSim(), None, rec, measure=lambda o: 1.0 if o["zgroups"] == 4 else 2.0, **run)
    assert old["options"]["zgroups"] == 4
    sim = FakeSim()
    new = T.tune(sim, None, rec, measure=lambda o: 2.0 if o["zgroups"] == 4 else 1.0, **run)
    assert not new["cached"] and sim.get_option(A.OPT_ZGROUPS) == 0
    again = FakeSim()
    assert T.tune(again, None, rec, measure=None, **run)["cached"]
    assert again.get_option(A.OPT_ZGROUPS) == 0
