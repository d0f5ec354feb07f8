"""The float screening of the FP32 regrid estimate (amrvac_regrid_estimate) where it
meets other levels, boundaries and other units.

Level changes and boundaries: the states are multiples of 2^-16 below 4, of which the
ghost operators (means of 2^d cells, minmod slopes times 1/4, over two levels at most)
form multiples of 2^-22 below 4: exact in float.  Both sides then work on the same
values in double, and what is left is the pressure's rounding (ten operations of
1.1e-16 on energies up to 8 times the pressure) over the denominator's least 0.04 of
it, four terms and weights that add up to 3.6: below 2e-12; 1e-11.  A cell missed by
the screening would cost up to 1e-5.

Units: scaling a state by powers of two (densities, momenta and energies by s, fields
by sqrt(s)) or all weights by one scales every operation of the double estimate
exactly, so the estimates are the same bits.
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
    "all": [1.0, 0.3, 0.3, 0.3, 1.0, 0.2, 0.2, 0.2, 0.1],
}
P, O, Y = ("periodic",) * 2, ("outflow",) * 2, ("symmetric",) * 2


def _contents(meta, n, seed, kinds, quantum=2.0 ** -16):
    """Conserved state, a kind of content per block: 0 equal cells, 1 noise of one
    quantum, 2 smooth, 3 random; multiples of quantum."""
    rng = np.random.Generator(np.random.PCG64(seed))
    lo = np.array([1.0, -0.25, -0.25, -0.25, 2.0, 0.25, 0.25, 0.25, -0.125])[:, None]
    hi = np.array([2.0, 0.25, 0.25, 0.25, 3.75, 0.5, 0.5, 0.5, 0.125])[:, None]
    U = np.empty((9, len(meta), n))
    x = np.arange(n) / n
    for b in range(len(meta)):
        base = 0.375 * np.ones((9, n))
        if kinds[b] == 2:
            base = 0.5 + 0.3 * np.sin(2 * np.pi * (x + rng.random((9, 1))))
        if kinds[b] == 3:
            base = rng.random((9, n))
        U[:, b] = lo + (hi - lo) * base
        if kinds[b] == 1:
            U[:, b] += quantum * rng.integers(0, 2, (9, n))
    return np.round(U / quantum) * quantum


def _mesh(name, bc):
    per = bc[0] == P
    if name == "3d":      # 32 blocks of level 1, 256 of level 2
        leaves = wl.c4_blast_amr(base=2, levels=3, bnx=2).block_meta if per else wl.amr_meta(
            3, (2, 2, 2), 2, lambda L, i, j, k: L < 2 and i + j + k < 2 + L, False)
        nd, bnx, base = 3, 16, (2, 2, 2)
    elif name == "1d":
        leaves = wl.amr_meta(1, (4, 1, 1), 2, lambda L, i, j, k: L < 2 and i < 2, per)
        nd, bnx, base = 1, 2050, (4, 1, 1)
    else:                 # 2D, three levels; 46: faces are no multiple of a warp
        nd, bnx, base = 2, int(name[2:]), (3, 3, 1)
        leaves = wl.small_amr_2d(base=base, bnx=4, periodic=per).block_meta
    cfg = wl.Config(ndim=nd, block_nx=tuple(bnx if d < nd else 1 for d in range(3)),
                    precision="fp32", bc=bc)
    return cfg, wl.Instance(base_blocks=base), leaves


KINDS = np.repeat([1, 2, 3], 8)  # runs of a kind, so that a block's maximum may lie inside


def _uniform(nd, bnx, blocks):
    base = (blocks, 1, 1)
    cfg = wl.Config(ndim=nd, block_nx=tuple(bnx if d < nd else 1 for d in range(3)),
                    precision="fp32")
    return cfg, wl.Instance(base_blocks=base), wl.uniform_meta(base)


@pytest.mark.parametrize("name", ["1d", "2d46", "2d64", "3d"])
@pytest.mark.parametrize("bc", [(P, P, P), (O, O, O), (O, Y, O), (Y, O, Y)],
                         ids=["periodic", "outflow", "oyo", "yoy"])
def test_levels_and_boundaries(amr, orc, name, bc):
    cfg, inst, meta = _mesh(name, bc)
    assert len(set(meta[:, 1])) > 1
    kinds = np.random.Generator(np.random.PCG64(5)).choice(4, len(meta), p=[0.4, 0.3, 0.1, 0.2])
    U = _contents(meta, int(np.prod(cfg.block_nx)), 11, kinds)
    W = wl.Workload("screen", cfg, [inst], meta, U)
    S = amr.State.from_workload(W, kernel="plain")
    S.set_conserved(U.astype(np.float32))
    for weights in WEIGHTS.values():
        Eo = rg.estimator(orc.mesh_for(W), U, cfg, weights=weights)
        E, f = S.regrid_estimate(0.1, 0.5, max_level=3, weights=weights)
        assert np.abs(E - Eo).max() <= 1e-11, np.abs(E - Eo).max()
        far = (np.abs(Eo - 0.1) > 1e-11) & (np.abs(Eo - 0.05) > 1e-11)
        assert np.array_equal(f[far], rg.flags(Eo, meta, 0.1, 0.5, 3)[far])
    S.close()


@pytest.mark.parametrize("nd,bnx", [(1, 2048), (2, 46), (2, 64), (3, 14), (3, 16)])
@pytest.mark.parametrize("period", [2, 4])
def test_ties(amr, orc, nd, bnx, period):
    # random contents that repeat with the period: 60 to 1024 cells tie for the maximum
    # (46 and 14 are no multiples of 4: the seams add others), so that few candidates,
    # many and more than the screening takes occur
    cfg, inst, meta = _uniform(nd, bnx, 20)
    at = np.indices(tuple(bnx if d < nd else 1 for d in (2, 1, 0))).reshape(3, -1) % period
    pat = _contents(meta, period ** 3, 14, np.full(len(meta), 3))
    pat[:, 1::2] = pat[:, :1]  # every other block the first one's
    U = pat[:, :, (at[0] * period + at[1]) * period + at[2]]
    W = wl.Workload("ties", cfg, [inst], meta, U)
    S = amr.State.from_workload(W, kernel="plain")
    S.set_conserved(U.astype(np.float32))
    for weights in WEIGHTS.values():
        Eo = rg.estimator(orc.mesh_for(W), U, cfg, weights=weights)
        E, _ = S.regrid_estimate(0.1, 0.5, max_level=3, weights=weights)
        assert np.abs(E - Eo).max() <= 1e-11, np.abs(E - Eo).max()
    S.close()


def _estimates(amr, cfg, inst, meta, U, weights):
    S = amr.State(cfg, [inst], meta, kernel="plain")
    S.set_conserved(U.astype(np.float32))
    E, _ = S.regrid_estimate(0.1, 0.5, max_level=3, weights=weights)
    S.close()
    return E


@pytest.mark.parametrize("nd,bnx", [(1, 2048), (2, 64), (3, 16)])
@pytest.mark.parametrize("weights", ["rho_p", "all"])
@pytest.mark.parametrize("k", [-48, -38, -36, -33, -30, -27, -20, 20, 45])
def test_other_units(amr, nd, bnx, weights, k):
    cfg, inst, meta = _uniform(nd, bnx, 24)
    U = _contents(meta, bnx ** nd, 12, KINDS, 2.0 ** -21)
    E = _estimates(amr, cfg, inst, meta, U, WEIGHTS[weights])
    U[:5] *= 4.0 ** k
    U[5:] *= 2.0 ** k
    assert np.array_equal(_estimates(amr, cfg, inst, meta, U, WEIGHTS[weights]), E)


@pytest.mark.parametrize("nd,bnx", [(1, 2048), (2, 64), (3, 16)])
@pytest.mark.parametrize("weights", ["rho_p", "all"])
@pytest.mark.parametrize("k", [-1020, -148, -140, -128, 100, 130, 1000])
def test_other_weights(amr, nd, bnx, weights, k):
    cfg, inst, meta = _uniform(nd, bnx, 24)
    U = _contents(meta, bnx ** nd, 13, KINDS, 2.0 ** -21)
    w = np.array(WEIGHTS[weights])
    E = _estimates(amr, cfg, inst, meta, U, w)
    got = _estimates(amr, cfg, inst, meta, U, w * 2.0 ** k)
    # at 2^-1020 products of weights and sums are subnormal: 9 of each, and the scaled
    # E, are rounded by half of 2^-1074
    assert np.abs(got - E * 2.0 ** k).max() <= (9.5 * 2.0 ** -1074 if k == -1020 else 0.0)
