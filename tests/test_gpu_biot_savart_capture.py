"""The direct sum's buffers hold any call whose sources and targets are no more
than an earlier call's each, not only the pairs that came up: such a call
allocates nothing and can be captured in a graph."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1508_06379_gb300 as v
    v.build()
    return v


@pytest.mark.parametrize("n,m", [(20000, 30000), (300, 20000), (70000, 600000)])
def test_a_call_within_the_buffers_can_be_captured(lib, n, m):
    rng = np.random.default_rng(n)
    x, y, g = (torch.from_numpy(rng.uniform(-1, 1, n)).cuda() for _ in range(3))
    xt, yt = (torch.from_numpy(rng.uniform(-1, 1, m)).cuda() for _ in range(2))
    want = [t.clone() for t in lib.VRM(h=0.01, nu=1e-3).biot_savart(x, y, g, n, xt, yt, m, 0.05)]
    ctx = lib.VRM(h=0.01, nu=1e-3)
    u, v = (torch.zeros(m, dtype=torch.float64, device="cuda") for _ in range(2))
    ctx.biot_savart(x, y, g, n, xt, yt, 10, 0.05, u, v)
    ctx.biot_savart(x, y, g, 10, xt, yt, m, 0.05, u, v)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.biot_savart(x, y, g, n, xt, yt, m, 0.05, u, v)
    for t in (u, v):
        t.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(u, want[0]) and torch.equal(v, want[1])
