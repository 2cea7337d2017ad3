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


def ring_tiles(nx, ny, nz, P, zchunk):
    """32 x 8 tiles that, with their neighbour cells, do not lie inside the x / y interior;
    every tile where no unit (tile and z chunk) lies inside the interior."""
    inside = [sum(t * w - 1 >= P and t * w + w < n - P for t in range(-(-n // w)))
              for n, w in ((nx, 32), (ny, 8), (nz, zchunk or nz))]
    box = inside[0] * inside[1] if inside[2] else 0
    return -(-nx // 32) * -(-ny // 8) - box


@pytest.mark.parametrize("sample", [0, 50])   # sampled runs time the same launches
@pytest.mark.parametrize("grid,zgroups,zchunk,planes", [
    ((100, 100, 50, 8), 0, 8, 8), ((128, 128, 128, 8), 0, 8, 8), ((200, 200, 100, 12), 0, 8, 16),
    ((200, 200, 100, 12), 1, 8, 8), ((301, 203, 151, 10), 0, 8, 24), ((301, 203, 151, 10), 1, 8, 8),
    ((301, 203, 151, 10), 0, 4, 12), ((301, 203, 151, 10), 0, 16, 16), ((301, 203, 151, 10), 0, 0, 151)])
def test_ring_chunks_grow_where_other_launches_hide_them(run, grid, zgroups, zchunk, planes,
                                                          sample):
    nx, ny, nz, P = grid
    sim = run.sim(problem(*grid), REC, {A.OPT_REVERSE: 2, A.OPT_ZGROUPS: zgroups,
                                        A.OPT_ZCHUNK: zchunk, A.OPT_SAMPLE_EVERY: sample})
    run.forward(sim, REC)
    ring = [e.grid for e in run.backward(sim) if e.what == "launch" and "k_rev_adjoint" in e.name
            and e.grid[1:] == (1, 1)]
    assert ring and set(ring) == {(ring_tiles(nx, ny, nz, P, zchunk) * -(-nz // planes), 1, 1)}


def waits_of(log, sims, run):
    """Per simulation the set of simulations whose loops its own loop waits for: the
    events of the other loops' ends that its stream waits for before its launches."""
    stream, end = {}, {}
    loops = [e.a for e in log if e.what == "graph"]
    for s in loops:                      # the record right after a loop's graph is its end
        at = next(i for i, e in enumerate(log) if e.what == "graph" and e.a == s)
        end[next(e.b for e in log[at:] if e.what == "record" and e.a == s)] = s
    out = {s: set() for s in loops}
    for e in log:
        if e.what == "wait" and e.b in end and e.a in out:
            out[e.a].add(end[e.b])
    return loops, out


LARGE, MID, SMALL = (301, 203, 151, 10), (200, 200, 100, 12), (64, 64, 64, 8)


@pytest.mark.parametrize("grids,free", [([LARGE] * 4, 4), ([MID] * 3, 1), ([LARGE, MID, MID], 1),
                                        ([SMALL] * 6, 5), ([LARGE] + [SMALL] * 3, 4),
                                        ([MID] + [SMALL] * 3, 2)])
def test_group_forward_waits_only_for_states_that_share_the_cache(run, grids, free):
    """Loops whose state no cache holds start at once; of those that nearly fill it one
    runs at a time, after the former; small ones fit beside each other.  Room
    for 0.6 of 132.6 MB: five states of 64^3 (28 bytes a cell, x auxiliaries of the whole
    grid, compact ones along y and z: 13.6 MB), or one that counts as 0.8 of it and one."""
    sims = [run.sim(problem(*g), REC) for g in grids]
    loops, waits = waits_of(run.group_forward(sims, REC), sims, run)
    assert len(loops) == len(grids)
    assert sum(not w for w in waits.values()) == free
    started = []
    for s in loops:                      # only loops that are enqueued already
        assert waits[s] <= set(started)
        started.append(s)


def test_group_forward_of_split_loops_that_fill_the_cache_runs_side_by_side(run):
    sims = [run.sim(problem(*MID), REC, {A.OPT_FORWARD: 1}) for _ in range(3)]
    _, waits = waits_of(run.group_forward(sims, REC), sims, run)
    assert not any(waits.values()) and len(waits) == 3


@pytest.mark.parametrize("grids,two", [([LARGE], 0), ([LARGE, LARGE], 2), ([LARGE, MID], 0), ([LARGE, LARGE, MID], 2),
                                       ([LARGE] + [SMALL] * 3, 0), ([MID, MID], 0)])
def test_large_loops_of_a_group_run_two_steps_per_pass(run, grids, two):
    sims = [run.sim(problem(*g), REC) for g in grids]
    log = run.group_forward(sims, REC)
    assert len({e.a for e in log if e.what == "launch" and "k_fwd_2step" in e.name}) == two
    assert all(s.step_forms()["forward"] != "two_step" for s in sims)


def test_first_group_forward_blocks_the_host_for_no_loop(run):
    """Every member's tables are uploaded (the host waits for the copies) before a stream
    waits for another loop's end; after that the host waits for results only."""
    sims = [run.sim(problem(*g), REC) for g in (MID, MID, MID, SMALL)]
    log = run.group_forward(sims, REC)
    what = [e.what for e in log]
    first, last = what.index("graph"), len(what) - 1 - what[::-1].index("graph")
    assert what.count("graph") == 4
    assert what[:first].count("sync") == 4 and "sync" not in what[first:last]


def test_backward_from_a_loaded_state_uploads_the_block_codecs_basis(tmp_path, monkeypatch):
    """A process that only loads a saved forward and runs the backward decodes a block
    codec tape with the basis table, which no forward of its own has uploaded."""
    import ctypes as C
    w, rec = problem(*SMALL), A.record_cfg("bdct10", 2)
    saver = S.Runner(S.load(tmp_path), monkeypatch)
    sim = saver.sim(w, rec)
    saver.forward(sim, rec)
    n = C.c_size_t()
    A.check(saver.L.fdtd_state_bytes(sim.h, C.byref(n)), sim.h)
    blob = C.create_string_buffer(n.value)
    A.check(saver.L.fdtd_save_state(sim.h, blob, n.value), sim.h)
    sim.close()
    (tmp_path / "other").mkdir()
    loader = S.Runner(S.load(tmp_path / "other"), monkeypatch)   # a library not used before
    sim = loader.sim(w, rec)
    A.check(loader.L.fdtd_load_state(sim.h, blob, n.value), sim.h)
    what = [e.what for e in loader.backward(sim)]
    assert what.count("symbol") == 2 and what.index("symbol") < what.index("launch")
