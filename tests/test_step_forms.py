"""Which form the time steps take (fdtd_step_forms) and what the benchmark's sampled
runs time, on the host: a sampled run must time the kernels that the timed run
launched."""
import numpy as np
import pytest

import bench
from paper_2603_24027_gb300 import _capi as A
from paper_2603_24027_gb300 import build as B
from paper_2603_24027_gb300 import fdtd as F
from paper_2603_24027_gb300 import inputs as I


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def problem(nx, ny, nz, P, inside=False):
    """Source and detector planes normal to x, in the first interior cells or (inside)
    in the middle of the grid."""
    at = nx // 2 if inside else P + 1
    lo = (at + 2, ny // 2 - 1, nz // 2 - 1)
    return I.Workload(name="forms", nx=nx, ny=ny, nz=nz, dx=20e-9, dt=I.cfl_dt(20e-9), n_steps=4,
                      pml_thickness=P, eps=np.empty((0,), np.float32), design_lo=lo,
                      design_hi=(lo[0] + 1, lo[1] + 1, lo[2] + 1),
                      src_kind=I.SRC_PLANE_GAUSS, src_component=1, src_axis=0,
                      src_pos=(at, ny // 2, nz // 2), src_sigma_uv=(5.0, 5.0),
                      det_kind=I.OBJ_POYNTING_PLANE, det_axis=0, det_index=at + 1,
                      det_lo=(P, P), det_hi=(ny - P, nz - P))


GRIDS = {(48, 48, 48, 8): ("direct", "direct"), (200, 200, 100, 12): ("direct", "split"),
         (301, 203, 151, 10): ("split", "fused"), (400, 300, 90, 10): ("split", "split"),
         (411, 389, 203, 10): ("two_step", "fused"), (1600, 92, 84, 16): ("fused", "split")}


@pytest.mark.parametrize("grid", GRIDS)
def test_forms_by_grid(grid):
    f = F.Simulation(problem(*grid)).step_forms()
    assert (f["forward"], f["reverse"]) == GRIDS[grid]


# Grids where the direct half-steps lose to the split ones below the general size line (every
# warp meets an x slab) or keep winning there (tiles wasted): us per step in fdtd_api.cu.
NARROW = {(64, 300, 135, 8): ("direct", "split"), (64, 300, 239, 8): ("split", "split"),
          (64, 64, 292, 8): ("direct", "direct"), (64, 64, 463, 8): ("direct", "split"),
          (64, 64, 1440, 8): ("split", "split"), (96, 96, 206, 12): ("direct", "split"),
          (50, 200, 590, 8): ("split", "split"), (120, 120, 400, 8): ("split", "split"),
          (160, 160, 230, 12): ("split", "split"), (160, 160, 74, 12): ("direct", "direct"),
          (48, 48, 824, 8): ("direct", "direct"), (34, 34, 5103, 8): ("direct", "split"),
          (600, 60, 163, 8): ("direct", "split"), (400, 300, 50, 8): ("direct", "split"), (233, 181, 117, 12): ("direct", "split"),
          (150, 110, 70, 12): ("direct", "direct")}


@pytest.mark.parametrize("grid", NARROW)
def test_forms_of_narrow_and_wide_grids(grid):
    f = F.Simulation(problem(*grid)).step_forms()
    assert (f["forward"], f["reverse"]) == NARROW[grid]


def test_named_forms():
    sim = F.Simulation(problem(200, 200, 100, 6))
    for opt, val, key, form in ((A.OPT_FORWARD, 1, "forward", "split"),
                                (A.OPT_FORWARD, 3, "forward", "two_step"),
                                (A.OPT_REVERSE, 1, "reverse", "split"),
                                (A.OPT_REVERSE, 2, "reverse", "fused"),
                                (A.OPT_KERNEL, 0, "forward", "split")):
        sim.set_option(opt, val)
        assert sim.step_forms()[key] == form


@pytest.mark.parametrize("grid,form", [((400, 80, 70, 4), "split"), ((301, 203, 151, 10), "split"),
                                       ((256, 256, 256, 8), "split"),
                                       ((411, 389, 203, 10), "two_step")])
def test_one_z_group_runs_two_steps_per_pass_on_large_grids_only(grid, form):
    sim = F.Simulation(problem(*grid))
    sim.set_option(A.OPT_ZGROUPS, 1)
    assert sim.step_forms()["forward"] == form
    sim.set_option(A.OPT_FORWARD, 3)
    assert sim.step_forms()["forward"] == "two_step"


@pytest.mark.parametrize("inside", [False, True])
@pytest.mark.parametrize("grid", GRIDS)
def test_sampled_runs_time_the_forms_of_the_timed_run(grid, inside):
    w = problem(*grid, inside=inside)
    forms = F.Simulation(w).step_forms()
    passes = bench.sampled_passes(A, forms)
    assert sorted(d for ds, _ in passes for d in ds) == ["forward", "reverse"]
    for directions, options in passes:
        sim = F.Simulation(w)
        for opt, val in options.items():
            sim.set_option(opt, val)
        sim.set_option(A.OPT_SAMPLE_EVERY, 50)
        got = sim.step_forms()
        for d in directions:
            assert got[d] == forms[d]
            # split half-steps are sampled with one launch each only
            assert got[d] != "split" or sim.get_option(A.OPT_ZGROUPS) == 1
