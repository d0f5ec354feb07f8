"""Merged parents in FP32 (amrvac_regrid_transfer) have the bits of the double sum of
their 2^d cells in the order (z, y, x), rounded once, also where cells of opposite sign
cancel and leave much smaller ones: the double sum rounds these away where they are
more than 53 binary digits below, and so has the restriction.
"""
import numpy as np
import pytest

from paper_2303_03026_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nd,bnx", [(1, 8), (2, 8), (3, 8)])
def test_cancelling_children(nd, bnx):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    from paper_2303_03026_gb300 import amrvac
    blocks = tuple(2 if d < nd else 1 for d in range(3))
    cfg = wl.Config(ndim=nd, block_nx=tuple(bnx if d < nd else 1 for d in range(3)),
                    precision="fp32")
    inst = wl.Instance(base_blocks=(1, 1, 1))
    meta = wl.uniform_meta(blocks)
    meta[:, 1] = 1
    rng = np.random.Generator(np.random.PCG64(nd))
    k, n, nc = 2 ** nd, (bnx // 2) ** nd, len(meta)
    # the children of each parent cell: pairs +a, -a at random places, the other two
    # (in 1D: one) cells smaller by 2^-10 .. 2^-70
    G = np.empty((9, nc, n, k), np.float32)
    for v in range(9):
        a = rng.uniform(0.5, 1, (nc, n, k // 2)).astype(np.float32)
        c = np.concatenate([a, -a], axis=2)
        small = (rng.uniform(-1, 1, (nc, n, k)) * 2.0 ** -rng.integers(10, 71, (nc, n, k)))
        c[..., -1] = small[..., -1]
        if k > 2:
            c[..., k // 2 - 1] = small[..., 0]
        if v > 5:
            c[..., 0] = np.float32(0.0)
        G[v] = rng.permuted(c, axis=2)
    # into blocks: parent cell (z, y, x) of a block's octant, child (fz, fy, fx)
    h = bnx // 2
    par = tuple(h if d < nd else 1 for d in (2, 1, 0))
    two = tuple(2 if d < nd else 1 for d in (2, 1, 0))
    U = G.reshape(9, nc, *par, *two).transpose(0, 1, 2, 5, 3, 6, 4, 7).reshape(9, nc, bnx ** nd)
    tot = np.zeros((9, nc, n))
    for c in range(k):
        tot = tot + G[..., c].astype(np.float64)
    ref = (tot / k).astype(np.float32).reshape(9, nc, *par)
    S = amrvac.State(cfg, [inst], meta, kernel="plain")
    S.set_conserved(np.ascontiguousarray(U))
    D = amrvac.State(cfg, [inst], wl.uniform_meta((1, 1, 1)), kernel="plain")
    S.regrid_transfer(D, 0, 0)
    got = D.get_conserved(0)[:, 0].reshape(9, *tuple(bnx if d < nd else 1 for d in (2, 1, 0)))
    S.close()
    D.close()
    for b, (_, _, i, j, l) in enumerate(meta):
        o = [s * p for s, p in zip((l, j, i), par)]
        sub = got[:, o[0]:o[0] + par[0], o[1]:o[1] + par[1], o[2]:o[2] + par[2]]
        assert np.array_equal(sub.view(np.uint32), ref[:, b].view(np.uint32))
