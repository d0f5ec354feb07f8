"""The CFL speeds of a field along an axis where the sound and Alfven speeds are
equal.  The fast speed is then the root of a sum whose inner root vanishes with the
tangential field, so an error u of the squared tangential field costs sqrt(u) of the
speed: it has to be formed from its components, not as a difference.

dt and c_h of amrvac_cfl_dt, of the entry without a workspace and of the last stage
of a step (plain and fused kernels) against the FP64 oracle on the same state.  The
pressure is 0.4 of the total energy it is recovered from, the speeds are some ten
operations from it, and dt adds the directions' terms: below 60 u of the result in
double (1e-14), and below 16 u in float (1e-6), where the recovery is compensated or
in double.
"""
import numpy as np
import pytest

from paper_2303_03026_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-14, "fp32": 1e-6}


@pytest.fixture(scope="module")
def amr():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2303_03026_gb300 import amrvac
    return amrvac


def _aligned(gamma, rho, p, axis, tang, shape, precision):
    """Conserved state at rest with gamma p = B^2 / mu (a = b) along axis, and a
    tangential field of tang times it."""
    B = np.zeros((3,) + shape)
    B[axis] = np.sqrt(gamma * p)
    B[(axis + 1) % 3] = tang * B[axis]
    z = np.zeros(shape)
    U = wl.conserved_from_primitive(gamma, rho + z, z, z, z, p + z, *B, z)
    return U.astype(np.float32).astype(np.float64) if precision == "fp32" else U


def _dtype(precision):
    return np.float32 if precision == "fp32" else np.float64


@pytest.mark.parametrize("nd", [1, 2, 3])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("tang", [0.0, 1e-8, 1e-4])
def test_cfl_dt(amr, orc, nd, precision, axis, tang):
    import torch
    blocks = tuple(2 if d < nd else 1 for d in range(3))
    cfg = wl.Config(ndim=nd, block_nx=tuple(12 if d < nd else 1 for d in range(3)),
                    precision=precision)
    inst = wl.Instance(base_blocks=blocks)
    meta = wl.uniform_meta(blocks)
    rng = np.random.Generator(np.random.PCG64(10 * nd + axis))
    shape = (len(meta), 12 ** nd)
    p = rng.uniform(0.1, 2.0, shape)
    # every cell has the same speeds (1.3), so the largest is the least accurate one
    U = _aligned(inst.gamma, inst.gamma * p / 1.69, p, axis, tang, shape, precision)
    W = wl.Workload("aligned", cfg, [inst], meta, U)
    dt, ch = orc.mesh_for(W).cfl(U)
    for pressure in ("fp64", "ff") if precision == "fp32" else ("fp64",):
        S = amr.State.from_workload(W, kernel="plain", pressure=pressure)
        S.set_conserved(U.astype(_dtype(precision)))
        got = S.cfl_dt()
        gch = S.diag()["ch"]
        S.close()
        np.testing.assert_allclose(got, dt, rtol=TOL[precision])
        np.testing.assert_allclose(gch, ch, rtol=TOL[precision])
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    amr.cfl_dt_noalloc(cfg, inst, torch.from_numpy(U.astype(_dtype(precision))).cuda(), out)
    torch.cuda.synchronize()
    np.testing.assert_allclose(out.cpu().numpy(), [dt[0], ch[0]], rtol=TOL[precision])


@pytest.mark.parametrize("nd,kernel", [(1, "plain"), (2, "plain"), (3, "plain"), (2, "fused"),
                                       (3, "fused")])
@pytest.mark.parametrize("precision,limiter", [("fp64", "vanleer"), ("fp32", "vanleer"),
                                               ("fp32", "mp5")])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_step(amr, orc, nd, kernel, precision, limiter, axis):
    # uniform instances (a step leaves them as they are), each with its own density
    # and pressure
    bnx = 16 if kernel == "fused" else 12
    cfg = wl.Config(ndim=nd, block_nx=tuple(bnx if d < nd else 1 for d in range(3)),
                    precision=precision, limiter=limiter)
    insts = [wl.Instance() for _ in range(12)]
    meta = np.concatenate([wl.uniform_meta((1, 1, 1), q) for q in range(len(insts))])
    rng = np.random.Generator(np.random.PCG64(20 * nd + axis))
    shape = (len(meta), bnx ** nd)
    rho, p = rng.uniform(0.1, 2.0, (2, len(meta), 1))
    U = _aligned(insts[0].gamma, rho, p, axis, 0.0, shape, precision)
    W = wl.Workload("aligned", cfg, insts, meta, U)
    S = amr.State.from_workload(W, kernel=kernel, pressure="ff")
    S.set_conserved(U.astype(_dtype(precision)))
    S.step(1)
    d = S.diag(raise_on_error=True)
    now = S.get_conserved(0).astype(np.float64)
    S.close()
    dt, ch = orc.mesh_for(W).cfl(now)
    np.testing.assert_allclose(d["dt"], dt, rtol=TOL[precision])
    np.testing.assert_allclose(d["ch"], ch, rtol=TOL[precision])
