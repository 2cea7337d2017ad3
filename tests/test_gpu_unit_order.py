"""Order of the fused reverse step's units on wide grids (csrc/kernels_rev_fused.cu): groups of
tile rows, the last one smaller.  Every unit runs once: the reversed interior and the gradient
equal those of the split phases bit for bit."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exact", [0, 22])
@pytest.mark.parametrize("nx,ny,nz,P", [(700, 430, 31, 4),     # two groups of tile rows
                                        (1300, 390, 29, 5),    # three
                                        (67, 6100, 27, 3)])    # two tiles wide, 763 rows
def test_groups_of_tile_rows(nx, ny, nz, P, exact):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2603_24027_gb300 import _capi as A, fdtd, inputs as I
    w = I.ragged_box(nx=nx, ny=ny, nz=nz, P=P, n_steps=20)
    rec = A.record_cfg("bf16", 3, "cubic")
    eps = torch.from_numpy(w.eps).cuda()
    out = []
    for reverse in (1, 2):
        sim = fdtd.Simulation(w, device="cuda")
        sim.set_option(A.OPT_EXACT_REVERSAL, exact)
        sim.set_option(A.OPT_FORWARD, 1)
        sim.set_option(A.OPT_REVERSE, reverse)
        sim.forward(eps, rec)
        g = sim.backward(1.0).clone()
        out.append((g, sim.read_fields()[:, P:nz - P, P:ny - P, P:nx - P].clone()))
        del sim
    assert out[0][0].abs().max() > 0
    assert torch.equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])
