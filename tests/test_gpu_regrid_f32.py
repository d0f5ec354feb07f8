"""FP32 regridding against the oracle where its float arithmetic has to give way:
the estimator's screening (amrvac_regrid_estimate finds the cells of the maximum in
float and evaluates them in double) on blocks of equal values, of rounding noise, of
single outliers, of vanishing velocities and of a pressure far below the magnetic
one; and
the restriction, whose mean is formed in float where that is exact, on values of all
magnitudes.
"""
import numpy as np
import pytest

from oracle import regrid as rg
from paper_2303_03026_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amr():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2303_03026_gb300 import amrvac
    return amrvac


WEIGHTS = {
    "rho": None,
    "rho_p": [0.5, 0, 0, 0, 0.5, 0, 0, 0, 0],
    "v": [0, 1, 2, 0.5, 0, 0, 0, 0, 0],
    "all": [1.0, 0.3, 0.3, 0.3, 1.0, 0.2, 0.2, 0.2, 0.1],
}


def _mesh(nd, bnx, blocks):
    shape = tuple(blocks if d == 0 else 1 for d in range(3))
    cfg = wl.Config(ndim=nd, block_nx=tuple(bnx if d < nd else 1 for d in range(3)), flux="hlld",
                    limiter="vanleer", time="ssprk3", precision="fp32", glm=True)
    inst = wl.Instance(base_blocks=shape, gamma=5.0 / 3.0)
    return cfg, inst, wl.uniform_meta(shape)


def _blocks(cfg, gamma, meta, seed):
    """Conserved float32 state, a kind of content per block in turn."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n = int(np.prod(cfg.block_nx))
    U = np.zeros((9, len(meta), n))
    for b in range(len(meta)):
        one, kind = np.ones(n), b % 8
        rho, p = 1.25 * one, 0.75 * one
        v, B, psi = np.full((3, n), 0.3), np.full((3, n), -0.4), 0.0 * one
        if kind in (2, 7):    # smooth and random content
            x = np.arange(n) / n
            rho = 1 + 0.2 * np.sin(2 * np.pi * x) if kind == 2 else rng.uniform(0.5, 2, n)
            p = 1 + 0.1 * np.cos(2 * np.pi * x) if kind == 2 else rng.uniform(0.5, 2, n)
            v, B, psi = v * rho, B * p, 0.01 * x
        if kind == 4:         # velocities that vanish, underflow or are tiny
            v = rng.choice([0.0, -0.0, 1e-38, 3e-42, -1e-20], (3, n))
        if kind == 5:         # pressure from 1e-3 to 1e-5 of the magnetic one
            B = rng.uniform(2, 3, (3, n))
            p = 10.0 ** rng.uniform(-5, -3, n) * 0.5 * (B ** 2).sum(axis=0)
            v = 0.0 * v
        U[:, b] = wl.conserved_from_primitive(gamma, rho, *v, p, *B, psi)
        if kind == 6:         # one cell an ulp off in one variable
            u = U[:, b].astype(np.float32)
            w, c = rng.integers(0, 9), rng.integers(0, n)
            u[w, c] = np.nextafter(u[w, c], np.float32(np.inf))
            U[:, b] = u
    U = U.astype(np.float32)
    for b in range(3, len(meta), 8):  # an ulp of noise everywhere
        up = np.nextafter(U[:, b], np.float32(np.inf))
        U[:, b] = np.where(rng.random((9, n)) < 0.5, up, U[:, b])
    return U


# either side of the screening's least work (2048 cells of a block, or of the blocks
# that one CTA works off), odd blocks, and several blocks a CTA
@pytest.mark.parametrize("nd,bnx,blocks", [(1, 2047, 24), (1, 2048, 24), (1, 2050, 24),
                                           (2, 10, 24), (2, 47, 24), (2, 64, 24), (3, 8, 1000),
                                           (3, 13, 24), (3, 16, 16)])
@pytest.mark.parametrize("weights", list(WEIGHTS))
def test_screened_estimate(amr, orc, nd, bnx, blocks, weights):
    # One level, so that every stencil value is a cell of the float state and both
    # sides work on it in double.  A pressure of 1e-5 of the energies keeps 1e-11 of
    # rounding; over the denominator's least 0.04 |q|, for ten operations, 5e-9.  A
    # screening that missed the cell of the maximum would be off by up to 1e-5.
    cfg, inst, meta = _mesh(nd, bnx, blocks)
    U = _blocks(cfg, inst.gamma, meta, 100 * nd + bnx)
    W = wl.Workload("screen", cfg, [inst], meta, U.astype(np.float64))
    Eo = rg.estimator(orc.mesh_for(W), W.U, cfg, weights=WEIGHTS[weights])
    S = amr.State.from_workload(W, kernel="plain")
    S.set_conserved(U)
    E, _ = S.regrid_estimate(0.1, 0.1, max_level=3, weights=WEIGHTS[weights])
    S.close()
    assert np.isfinite(E).all()
    assert np.abs(E - Eo).max() <= 5e-9, np.abs(E - Eo).max()


@pytest.mark.parametrize("nd,bnx", [(1, 4), (1, 34), (2, 4), (2, 10), (3, 4), (3, 8)])
def test_restriction_bits(amr, orc, nd, bnx):
    # every block merges; each parent cell has the bits of the double sum of its 2^d
    # cells, rounded once
    blocks = tuple(2 if d < nd else 1 for d in range(3))
    cfg, inst, _ = _mesh(nd, bnx, 1)
    rng = np.random.Generator(np.random.PCG64(7 * nd + bnx))
    meta = wl.uniform_meta(blocks)
    meta[:, 1] = 1
    shape = (9, len(meta), bnx ** nd)
    with np.errstate(over="ignore", under="ignore"):
        U = rng.uniform(0.5, 1.0, shape).astype(np.float32)             # ties
        U[1] = rng.choice([-1, 1], shape[1:]) * U[1]                    # cancellation
        U[2] *= (10.0 ** rng.uniform(-30, 30, shape[1:])).astype(np.float32)
        U[3] = (1 + np.arange(bnx ** nd) % 2 * -2) * (1 + 1e-7 * U[3])  # all but cancelled
        U[4] *= np.float32(1e-41)                                       # denormal
        U[5] *= np.float32(3.4e38)                                      # the float sum overflows
        U[6] = rng.choice([0.0, -0.0, 1e-45, 1.0], shape[1:])
        U[7] *= (10.0 ** rng.uniform(-9, 0, shape[1:])).astype(np.float32)
        U[8] = 0.3
    W = wl.Workload("merge", cfg, [inst], meta, U.astype(np.float64))
    new = wl.uniform_meta((1, 1, 1))
    ref = rg.transfer(cfg, [inst], meta, W.U, orc.mesh_for(W), new).astype(np.float32)
    S = amr.State.from_workload(W, kernel="plain")
    S.set_conserved(U)
    D = amr.State(cfg, [inst], new, kernel="plain")
    S.regrid_transfer(D, 0, 0)
    got = D.get_conserved(0)
    S.close()
    D.close()
    assert got.dtype == np.float32
    assert np.array_equal(got.view(np.uint32), ref.view(np.uint32))
