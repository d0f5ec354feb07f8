"""The inverse cell size of the double path is rounded once, from the domain: cells over
length (1/dx of the rounded dx is rounded twice).  Seen in the time step of a state at
rest in 1D, which is courant / (c_h / dx) with each operation rounded: bit for bit."""
import numpy as np
import pytest

from paper_2303_03026_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells", [12, 16, 24, 100])
def test_rounded_once(cells):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2303_03026_gb300 import amrvac
    lengths = np.random.Generator(np.random.PCG64(cells)).uniform(0.1, 10.0, 40)
    # (16 cells: dx is exact, and rounding once or twice is the same)
    assert (1.0 / (lengths / cells) != cells / lengths).any() == (cells != 16)
    cfg = wl.Config(ndim=1, block_nx=(cells, 1, 1), courant=0.8)
    insts = [wl.Instance(xmax=(x, 1.0, 1.0)) for x in lengths]
    meta = np.concatenate([wl.uniform_meta((1, 1, 1), q) for q in range(len(insts))])
    z = np.zeros((len(insts), cells))
    U = wl.conserved_from_primitive(insts[0].gamma, z + 1.3, z, z, z, z + 0.7, z, z, z)
    S = amrvac.State(cfg, insts, meta, kernel="plain")
    S.set_conserved(U)
    dt = S.cfl_dt()
    ch = S.diag()["ch"]
    assert np.array_equal(dt, 0.8 / (ch * (cells / lengths)))
    S.step(1)  # uniform: the state stays, the step's own pass forms dt again
    assert np.array_equal(S.get_conserved(0), U)
    assert np.array_equal(S.diag()["dt"], dt)
    S.close()
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    for q in range(0, 40, 8):
        amrvac.cfl_dt_noalloc(cfg, insts[q], torch.from_numpy(U[:, q:q + 1].copy()).cuda(), out)
        torch.cuda.synchronize()
        assert out[0].item() == dt[q]
