"""The fused FP32 kernels with two ghost layers against the FP64 oracle on rough
data: every cell drawn by itself (jumps at every face, so that each handed-over
face state, boundary face and ghost layer counts), on meshes whose blocks are
their own neighbours, odd block counts, every boundary type, and one limiter of
each instantiation.

Tolerance, relative L1 per variable after one step: a face flux is some 50
dependent float operations (3e-6 of the state times the signal speed), a stage
adds Courant <= 0.8 of it per direction, and three to five stages add up: below
4e-5; states whose HLLD denominator lies between the float and the double
degeneracy threshold (1e-5 and 1e-8) differ by 1e-5 of the state more.  1e-4.
"""
import numpy as np
import pytest

from paper_2303_03026_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

P, O, Y = ("periodic",) * 2, ("outflow",) * 2, ("symmetric",) * 2
CASES = [  # ndim, blocks, limiter, flux, time, boundaries
    (3, (1, 1, 1), "vanleer", "hlld", "ssprk3", (P, P, P)),
    (3, (1, 1, 1), "vanleer", "hlld", "ssprk54", (O, O, O)),
    (3, (3, 1, 2), "koren", "hll", "ssprk3", (O, P, O)),
    (3, (2, 3, 1), "minmod", "tvdlf", "ssprk2", (P, O, P)),
    (3, (1, 2, 3), "superbee", "hllc", "ssprk43", (Y, P, O)),
    (3, (2, 1, 1), "albada", "hlld", "ssprk3", (Y, Y, Y)),
    (3, (1, 1, 2), "venk", "hll", "ssprk54", (P, Y, P)),
    (2, (1, 1, 1), "vanleer", "hlld", "ssprk3", (P, P, P)),
    (2, (5, 3, 1), "woodward", "hlld", "ssprk43", (O, P, P)),
    (2, (3, 1, 1), "cada3", "hllc", "ssprk54", (P, Y, P)),
    (2, (1, 7, 1), "minmod", "hll", "ssprk2", (Y, O, P)),
    (2, (2, 2, 1), "koren", "tvdlf", "ssprk3", (O, Y, P)),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "%dd_%s_%s_%s" % (c[0], c[2], c[3], c[4]))
@pytest.mark.parametrize("dynamic", [False, True])
def test_rough_data_one_step(orc, case, dynamic):
    from paper_2303_03026_gb300 import amrvac
    nd, blocks, limiter, flux, time, bc = case
    cfg = wl.Config(ndim=nd, block_nx=(16, 16, 16 if nd == 3 else 1), flux=flux, limiter=limiter,
                    time=time, precision="fp32", glm=True, bc=bc)
    # two instances with another gamma and domain
    insts = [wl.Instance(base_blocks=blocks, gamma=5.0 / 3.0),
             wl.Instance(base_blocks=blocks, gamma=1.4, xmax=(0.7, 1.3, 0.9))]
    meta = np.concatenate([wl.uniform_meta(blocks, q) for q in range(2)])
    rng = np.random.Generator(np.random.PCG64(17))
    n = (meta.shape[0], 16 ** nd)
    g = np.array([insts[q].gamma for q in meta[:, 0]])[:, None]
    f = lambda a, b: rng.uniform(a, b, n)  # noqa: E731
    U = wl.conserved_from_primitive(g, f(0.5, 2.0), f(-0.5, 0.5), f(-0.5, 0.5), f(-0.5, 0.5),
                                    f(0.5, 2.0), f(-0.5, 0.5), f(-0.5, 0.5), f(-0.5, 0.5),
                                    f(-0.1, 0.1)).astype(np.float32).astype(np.float64)
    W = wl.Workload("rough", cfg, insts, meta, U)
    S = amrvac.State.from_workload(W, kernel="fused", pressure="ff")
    S.set_tuning(dynamic=dynamic)
    S.set_conserved(U.astype(np.float32))
    S.step(1)
    d = S.diag(raise_on_error=True)
    got = S.get_conserved(0).astype(np.float64)
    S.close()
    ref, t, _, st = orc.mesh_for(W, 4).run(U, 1e30, maxsteps=1)
    assert st == 0
    np.testing.assert_allclose(d["t"], t, rtol=1e-5)
    err = np.abs(got - ref).sum((1, 2)) / np.abs(ref).sum((1, 2))
    assert err.max() <= 1e-4, err
