"""The chain of programmatically dependent launches: evaluations queued back to back on changing data, and
evaluations recorded into a caller's graph, give the bits of evaluations that are waited for one by one."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    from paper_1504_02897_gb300 import build, ddi
    build.build()
    ddi.load()
    return ddi


def _plan(D, n, precision=1, **kw):
    ln = tuple(0.2 * v for v in n)
    return D.Plan(len(n), n, tuple(-0.5 * v for v in ln), ln, (0.6, 0.0, 0.8), precision=precision, **kw)


CASES = [
    ((48, 48, 48), {}),
    ((24, 16, 12), dict(nr=128, ntheta=64, nphi=64)),  # 2^18 processed nodes: interpolation by columns
    ((24, 24, 24), dict(nr=16, ntheta=16, nphi=32, spread=1)),
    ((64, 64, 64), dict(split_k0=-1.0)),
    ((128, 96), {}),
    ((32, 32, 32), dict(precision=0)),
]


@pytest.mark.parametrize("n,kw", CASES)
def test_queued_applies_match_synchronised_ones(D, n, kw):
    import torch
    plan = _plan(D, n, **kw)
    g = torch.Generator("cuda").manual_seed(7)
    rhos = [torch.rand(tuple(reversed(n)), generator=g, device="cuda").to(plan.real_dtype) * (1 + k) for k in range(24)]
    want = []
    for r in rhos:
        want.append(plan.apply(r).clone())
        torch.cuda.synchronize()
    outs = [torch.empty_like(r) for r in rhos]
    for r, o in zip(rhos, outs):
        plan.apply(r, o)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, outs))


@pytest.mark.parametrize("n,kw", CASES)
def test_apply_in_a_callers_graph(D, n, kw):
    import torch
    plan = _plan(D, n, **kw)
    g = torch.Generator("cuda").manual_seed(8)
    rho = torch.rand(tuple(reversed(n)), generator=g, device="cuda").to(plan.real_dtype)
    out = torch.empty_like(rho)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        plan.apply(rho, out)
    for k in range(4):
        rho.mul_(1.25).add_(0.125 * k)
        graph.replay()
        got = out.clone()
        assert torch.equal(got, plan.apply(rho))


@pytest.mark.parametrize("n,precision", [((48, 48, 48), 1), ((64, 48), 1), ((24, 24, 24), 0)])
def test_gpe_steps_queued_and_in_a_callers_graph(D, n, precision):
    import torch
    plan = _plan(D, n, precision=precision)
    shape = tuple(reversed(n))
    g = torch.Generator("cuda").manual_seed(9)
    V = torch.rand(shape, generator=g, device="cuda").to(plan.real_dtype)
    psi0 = 0.1 * torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda")).to(plan.cplx_dtype)
    want = psi0.clone()
    for _ in range(6):
        plan.gpe_step(want, V, 10.0, 5.0, 1e-3, 2)
        torch.cuda.synchronize()
    queued = psi0.clone()
    for _ in range(6):
        plan.gpe_step(queued, V, 10.0, 5.0, 1e-3, 2)
    assert torch.equal(queued, want)
    psi = psi0.clone()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        plan.gpe_step(psi, V, 10.0, 5.0, 1e-3, 2)
    psi.copy_(psi0)
    for _ in range(6):
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(psi, want)
