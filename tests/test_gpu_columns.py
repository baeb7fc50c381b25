"""Column spread and interpolation of 3D plans (both precisions, every built kernel width) against the tile spread
of the same plan: the two sum the same taps in another order, so they agree to the path's own
tolerance (1e-6 FP32, 1e-12 FP64).  Sizes where the lists can go wrong: the smallest fine grid
that holds a column and a footprint (windows and footprints wrap), ragged grids, units of a
few visits (most planes shared, groups of one run) and units of whole columns."""
import math

import numpy as np
import pytest

from paper_1504_02897_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 1e-6}


@pytest.fixture(scope="module")
def D():
    from paper_1504_02897_gb300 import build, ddi
    build.build()
    ddi.load()
    return ddi


CASES = [
    # precision, nufft_tol, n, rule, chunk
    (0, 0.0, (12, 12, 12), (16, 16, 16), 0),
    (0, 0.0, (24, 12, 8), (17, 11, 26), 5),
    (0, 1e-7, (12, 16, 12), (16, 16, 16), 40),      # w = 10
    (0, 1e-9, (16, 12, 24), (16, 17, 16), 100000),  # w = 12
    (0, 1e-14, (12, 12, 16), (16, 16, 18), 64),     # w = 16
    (0, 0.0, (32, 24, 48), (33, 15, 50), 0),
    (1, 0.0, (8, 8, 8), (9, 7, 10), 1),
    (1, 1e-4, (8, 12, 16), (9, 7, 10), 33),         # w = 6
    (1, 0.0, (48, 24, 32), (49, 23, 46), 0),
    (1, 0.0, (24, 16, 12), (128, 64, 64), 0),       # 2^18 processed nodes: FP32 interpolates by columns too
    (1, 1e-4, (8, 12, 16), (64, 128, 64), 200),
]


@pytest.mark.parametrize("prec,tol,n,rule,chunk", CASES)
def test_columns_match_tiles(D, prec, tol, n, rule, chunk):
    import torch
    lo, ln = tuple(-0.25 * v for v in n), tuple(0.5 * v for v in n)
    X, Y, Z = synth.coords(n, lo, ln)
    rng = np.random.default_rng(5)
    rho = np.exp(-0.3 * (X ** 2 + Y ** 2 + Z ** 2)) * (1 + 0.05 * rng.random(X.shape))
    axis, m = (0.6, 0.0, 0.8), (0.0, math.sqrt(0.5), math.sqrt(0.5))
    kw = dict(precision=prec, nufft_tol=tol, nr=rule[0], ntheta=rule[1], nphi=rule[2])
    cols = D.Plan(3, n, lo, ln, axis, m, chunk=chunk, **kw)
    tiles = D.Plan(3, n, lo, ln, axis, m, spread=1, **kw)
    small = rule[0] * rule[1] * rule[2] // 2 < 2048
    assert tiles.info.spread == 1 and cols.info.spread == (1 if prec == 0 and small else 2)
    x = torch.from_numpy(rho).to("cuda", cols.real_dtype)
    a, b = cols.apply(x), tiles.apply(x)
    err = float((a - b).abs().max() / b.abs().max())
    assert err <= TOL[prec], err
    assert torch.equal(a, cols.apply(x))  # fixed summation order


@pytest.mark.parametrize("n,rule,chunk,tol", [
    ((8, 8), (9, 10), 0, 0.0),        # the smallest fine grid: 2 x 2 blocks, footprints wrap
    ((12, 24), (31, 34), 5, 0.0),     # units of one group, many partial blocks
    ((48, 16), (64, 66), 70, 1e-4),   # w = 6, ragged
    ((64, 64), (128, 128), 0, 0.0),
    ((32, 96), (40, 512), 100000, 0.0),  # one unit per block
])
def test_blocks_match_tiles_2d(D, n, rule, chunk, tol):
    # the type-1 stage of random node values by the 2D block spread and by the tile spread (the same
    # taps in another order; no symbol in between that would amplify the rounding)
    import torch
    lo, ln = tuple(-0.25 * v for v in n), tuple(0.5 * v for v in n)
    kw = dict(precision=1, nufft_tol=tol, nr=rule[0], nphi=rule[1])
    blocks = D.Plan(2, n, lo, ln, (0.6, 0.0, 0.8), chunk=chunk, **kw)
    tiles = D.Plan(2, n, lo, ln, (0.6, 0.0, 0.8), spread=1, **kw)
    assert blocks.info.spread == 2 and tiles.info.spread == 1
    # the nodes' processing order depends on the plan's tile: values go by original node index
    q = {int(v): k for k, v in enumerate(tiles.node_order())}
    perm = torch.tensor([q[int(v)] for v in blocks.node_order()], device="cuda")
    g = torch.Generator("cuda").manual_seed(3)
    c = torch.randn(int(tiles.info.nodes_used), 2, generator=g, device="cuda")
    c = torch.view_as_complex(c)
    a, b = blocks.type1(c[perm].contiguous()), tiles.type1(c)
    err = float((a - b).abs().max() / b.abs().max())
    assert err <= 1e-6, err
    assert torch.equal(a, blocks.type1(c[perm].contiguous()))
