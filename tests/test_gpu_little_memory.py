"""Where the device has no room for the column lists that the automatic choice would build, a plan or a batch takes the
tile spread, whose lists are a tenth of their size, instead of failing."""
import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def D():
    from paper_1504_02897_gb300 import build, ddi
    build.build()
    ddi.load()
    return ddi


class LittleMemory:
    """Holds all free device memory but `leave` bytes."""

    def __init__(self, leave):
        self.leave = leave

    def __enter__(self):
        import torch
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        self.held = torch.empty(free - self.leave, dtype=torch.uint8, device="cuda")

    def __exit__(self, *exc):
        import torch
        del self.held
        torch.cuda.empty_cache()


def test_plan(D):
    import torch

    def plan(spread):
        return D.Plan(3, (64,) * 3, (-6.0,) * 3, (12.0,) * 3, (0.6, 0.0, 0.8), precision=0, spread=spread)

    g = torch.Generator("cuda").manual_seed(1)
    rho = torch.rand((64,) * 3, generator=g, device="cuda", dtype=torch.float64)
    out = torch.empty_like(rho)
    columns, tiles = plan(0), plan(1)
    assert columns.info.spread == 2 and tiles.info.spread == 1
    want = tiles.apply(rho)
    columns.apply(rho)
    need, room = tiles.info.device_bytes, columns.info.device_bytes - tiles.info.device_bytes
    assert room > 100 * MB
    columns.close()
    tiles.close()
    with LittleMemory(need + room // 2):
        p = plan(0)
        assert p.info.spread == 1 and p.info.device_bytes == need
        p.apply(rho, out)
        p.close()
    assert torch.equal(out, want)


def test_batch(D):
    import torch
    n, count = (256, 256), 12

    def batch(spread):
        descs = [D.make_desc(2, n, (-8.0, -8.0), (16.0, 16.0), (0.6, 0.0, 0.8), precision=1, spread=spread)] * count
        return D.Batch(descs, graph=False, autotune=False)

    def used(b):
        b.apply(rhos, outs)
        torch.cuda.synchronize()
        free, _ = torch.cuda.mem_get_info()
        b.close()
        return torch.cuda.mem_get_info()[0] - free

    g = torch.Generator("cuda").manual_seed(1)
    rhos = [torch.rand(n, generator=g, device="cuda") for _ in range(count)]
    outs = [torch.empty_like(r) for r in rhos]
    need = used(batch(1))
    want = [o.clone() for o in outs]
    room = used(batch(0)) - need
    assert room > 100 * MB
    with LittleMemory(need + room // 3):
        b = batch(0)
        b.apply(rhos, outs)
        torch.cuda.synchronize()
        b.close()
    for a, w in zip(outs, want):
        assert float((a - w).abs().max() / w.abs().max()) <= 1e-6  # the same taps in another order
