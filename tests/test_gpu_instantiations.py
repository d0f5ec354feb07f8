"""Every instantiation of the fused stage kernels (dimension, precision, limiter, flux,
with and without the walls' FULL code) on rough data against the FP64 oracle, one
SSPRK2 step; and two limiters on two levels, which share an instantiation where both are
runtime values.  A fault of one instantiation, of its source or its compilation, shows
in none of the others.

Tolerances as for rough data in general: relative L1 per variable 1e-12 in double (7e-14
of rounding), 1e-4 in float (4e-5).
"""
import numpy as np
import pytest

from paper_2303_03026_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TWO = ["minmod", "vanleer", "koren", "superbee", "woodward", "mcbeta", "albada", "cada3", "venk"]
FIVE = ["mp5", "weno5", "wenoz5", "wenozp5"]
RUNTIME = TWO[3:]
P, Y = ("periodic",) * 2, ("symmetric",) * 2
TOL = {"fp64": 1e-12, "fp32": 1e-4}


def _error(orc, nd, precision, limiter, flux, wall, level=None):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2303_03026_gb300 import amrvac
    cfg = wl.Config(ndim=nd, block_nx=(16, 16, 16 if nd == 3 else 1), flux=flux, limiter=limiter,
                    time="ssprk2", precision=precision, bc=(Y if wall else P, P, P))
    if level is None:
        base = (1, 2, 1) if nd == 3 else (2, 1, 1)
        meta, inst = wl.uniform_meta(base), wl.Instance(base_blocks=base, xmax=(0.9, 1.1, 0.8))
    else:
        base = (2, 2, 2 if nd == 3 else 1)
        meta = wl.amr_meta(nd, base, 1, lambda L, i, j, k: L == 0 and i + j + k == 1)
        cfg.level_limiter = {1: level}
        inst = wl.Instance(base_blocks=base)
    rng = np.random.Generator(np.random.PCG64(5))
    f = lambda c: c + 0.2 * rng.uniform(-1.0, 1.0, (len(meta), 16 ** nd))  # noqa: E731
    dt = np.float32 if precision == "fp32" else np.float64
    U = wl.conserved_from_primitive(inst.gamma, f(1.2), f(0.0), f(0.1), f(-0.1), f(1.2), f(0.2),
                                    f(-0.1), f(0.1), 0.1 * f(0.0)).astype(dt).astype(np.float64)
    W = wl.Workload("instantiation", cfg, [inst], meta, U)
    S = amrvac.State.from_workload(W, kernel="fused", pressure="ff")
    S.set_conserved(U.astype(dt))
    S.step(1)
    S.diag(raise_on_error=True)
    got = S.get_conserved(0).astype(np.float64)
    S.close()
    ref, _, _, st = orc.mesh_for(W, 4).run(U, 1e30, maxsteps=1)
    assert st == 0
    return (np.abs(got - ref).sum((1, 2)) / np.abs(ref).sum((1, 2))).max()


@pytest.mark.parametrize("nd", [2, 3])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("limiter", TWO + FIVE)
def test_every_flux(orc, nd, precision, limiter):
    if nd == 3 and precision == "fp64" and limiter in FIVE:
        pytest.skip("no fused kernel: a double ring of six planes does not fit")
    err = {(flux, wall): _error(orc, nd, precision, limiter, flux, wall)
           for flux in ("hll", "hlld", "tvdlf", "hllc") for wall in (False, True)}
    assert max(err.values()) <= TOL[precision], err


@pytest.mark.parametrize("nd", [2, 3])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("limiter", RUNTIME)
def test_two_levels(orc, nd, precision, limiter):
    err = {(level, flux): _error(orc, nd, precision, limiter, flux, flux == "hllc", level)
           for level in RUNTIME if level != limiter for flux in ("tvdlf", "hllc")}
    assert max(err.values()) <= TOL[precision], err
