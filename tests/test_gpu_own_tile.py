"""An FP32 2D plan above 512 x 512 fine cells whose caller gives a tile size spreads by tiles of that size."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    from paper_1504_02897_gb300 import build, ddi
    build.build()
    ddi.load()
    return ddi


@pytest.mark.parametrize("n,tile,spread", [((512, 256), (64, 16, 1), 1), ((256, 512), (0, 32, 0), 1), ((512, 256), None, 2),
                                           ((512, 256), (-1, 0, 0), 2), ((256, 256), (64, 16, 1), 2)])
def test_2d_tile_of_the_callers_own(D, n, tile, spread):
    import torch
    ln = tuple(0.1 * v for v in n)
    kw = dict(precision=1, nr=33, nphi=66)
    plan = D.Plan(2, n, tuple(-0.5 * v for v in ln), ln, (0.6, 0.0, 0.8), tile=tile, **kw)
    assert plan.info.spread == spread
    if spread == 1:
        assert all(t <= 0 or plan.info.tile[a] == t for a, t in enumerate(tile[:2]))
    ref = D.Plan(2, n, tuple(-0.5 * v for v in ln), ln, (0.6, 0.0, 0.8), spread=1, **kw)
    g = torch.Generator("cuda").manual_seed(1)
    rho = torch.rand(n[::-1], generator=g, device="cuda")
    a, b = plan.apply(rho), ref.apply(rho)
    assert float((a - b).abs().max() / b.abs().max()) <= 1e-6  # the same taps in another order
