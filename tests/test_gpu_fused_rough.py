"""The fused kernels that hand limited states to the neighbouring face, on data drawn
cell by cell: in double (slopes once a cell, a helper warp for the boundary faces), one
limiter of each instantiation and every boundary type; and in both precisions on two
levels with refluxing, where the flux of every level-change face is kept.  One step
against the FP64 oracle.

Tolerance, relative L1 per variable: a face flux is some 50 dependent operations (5e-15
of the state times the signal speed in double, 3e-6 in float), a stage adds Courant <=
0.8 of it per direction, and three to five stages add up: below 7e-14 and 4e-5; HLLD
states between the float and the double degeneracy threshold differ by 1e-5 more.
1e-12 and 1e-4.
"""
import numpy as np
import pytest

from paper_2303_03026_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

P, O, Y = ("periodic",) * 2, ("outflow",) * 2, ("symmetric",) * 2
TOL = {"fp64": 1e-12, "fp32": 1e-4}


def _step(orc, cfg, insts, meta, rough, dynamic):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2303_03026_gb300 import amrvac
    dt = np.float32 if cfg.precision == "fp32" else np.float64
    rng = np.random.Generator(np.random.PCG64(23))
    n = (meta.shape[0], 16 ** cfg.ndim)
    g = np.array([insts[q].gamma for q in meta[:, 0]])[:, None]
    f = lambda c: c + rough * rng.uniform(-1.0, 1.0, n)  # noqa: E731
    U = wl.conserved_from_primitive(g, f(1.2), f(0.0), f(0.1), f(-0.1), f(1.2), f(0.2), f(-0.1),
                                    f(0.1), 0.2 * f(0.0)).astype(dt).astype(np.float64)
    W = wl.Workload("rough", cfg, insts, meta, U)
    S = amrvac.State.from_workload(W, kernel="fused", pressure="ff")
    S.set_tuning(dynamic=dynamic)
    S.set_conserved(U.astype(dt))
    S.step(1)
    d = S.diag(raise_on_error=True)
    got = S.get_conserved(0).astype(np.float64)
    S.close()
    ref, t, _, st = orc.mesh_for(W, 4).run(U, 1e30, maxsteps=1)
    assert st == 0
    tol = TOL[cfg.precision]
    np.testing.assert_allclose(d["t"], t, rtol=0.1 * tol)
    err = np.abs(got - ref).sum((1, 2)) / np.abs(ref).sum((1, 2))
    assert err.max() <= tol, err


CASES = [  # ndim, blocks, limiter, flux, time, boundaries
    (3, (1, 1, 1), "vanleer", "hlld", "ssprk3", (P, P, P)),
    (3, (2, 1, 3), "koren", "hllc", "ssprk54", (O, P, Y)),
    (3, (1, 2, 1), "minmod", "hll", "ssprk2", (Y, O, P)),
    (3, (1, 1, 2), "cada3", "tvdlf", "ssprk43", (P, Y, O)),
    (2, (1, 1, 1), "vanleer", "hll", "ssprk3", (P, P, P)),
    (2, (5, 3, 1), "koren", "hlld", "ssprk54", (O, Y, P)),
    (2, (1, 7, 1), "minmod", "tvdlf", "ssprk43", (Y, P, P)),
    (2, (3, 2, 1), "woodward", "hllc", "ssprk2", (P, O, P)),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "%dd_%s_%s_%s" % (c[0], c[2], c[3], c[4]))
@pytest.mark.parametrize("dynamic", [False, True])
def test_double(orc, case, dynamic):
    nd, blocks, limiter, flux, time, bc = case
    cfg = wl.Config(ndim=nd, block_nx=(16, 16, 16 if nd == 3 else 1), flux=flux, limiter=limiter,
                    time=time, precision="fp64", bc=bc)
    insts = [wl.Instance(base_blocks=blocks, gamma=5.0 / 3.0),
             wl.Instance(base_blocks=blocks, gamma=1.4, xmax=(0.7, 1.3, 0.9))]
    meta = np.concatenate([wl.uniform_meta(blocks, q) for q in range(2)])
    _step(orc, cfg, insts, meta, 0.5, dynamic)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nd,limiter,flux,time,bc", [
    (3, "vanleer", "hlld", "ssprk3", (P, P, P)),
    (3, "koren", "hll", "ssprk43", (O, Y, P)),
    (3, "woodward", "hllc", "ssprk54", (P, O, Y)),
    (2, "vanleer", "hlld", "ssprk54", (P, P, P)),
    (2, "minmod", "tvdlf", "ssprk3", (Y, O, P)),
    (2, "albada", "hll", "ssprk2", (O, P, P)),
])
def test_refluxing(orc, precision, nd, limiter, flux, time, bc):
    base = (2, 2, 2) if nd == 3 else (3, 3, 1)
    per = all(b == P for b in bc[:nd])
    meta = wl.amr_meta(nd, base, 1, lambda L, i, j, k: L == 0 and i + j + k == 1, per)
    assert set(meta[:, 1]) == {0, 1}
    cfg = wl.Config(ndim=nd, block_nx=(16, 16, 16 if nd == 3 else 1), flux=flux, limiter=limiter,
                    time=time, precision=precision, bc=bc, reflux=True)
    _step(orc, cfg, [wl.Instance(base_blocks=base)], meta, 0.2, nd == 2)
