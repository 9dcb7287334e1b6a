"""A position or circulation that is not finite, anywhere in a small cloud
(diffused or not, in reach of diffused particles or not), is refused after the
step's kernels have run on it: they may compute nonsense, but must not read or
write out of range (k_search_warp once left an index of 2^31 - 1 for a
segment whose only member had a NaN offset)."""
import numpy as np
import pytest

import vrm_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1508_06379_gb300 as v
    v.build()
    return v


def cu(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("n", [400, 3000, 10000])
@pytest.mark.parametrize("at", [0.0, 0.3, 0.5, 0.51, 0.99])
@pytest.mark.parametrize("where", ["x", "y", "xy", "gamma"])
@pytest.mark.parametrize("value", [np.nan, -np.nan, np.inf, -np.inf])
def test_refused(lib, n, at, where, value):
    x, y, g = vrm_inputs.random_cloud(n + 200, h=0.05, jitter=0.3, seed=8)
    x, y, g = x[:n].copy(), y[:n].copy(), g[:n].copy()
    k = int(at * n)
    for name, v in (("x", x), ("y", y), ("gamma", g)):
        if name in where:
            v[k] = value
    xb, yb, go = (torch.zeros(4 * n, dtype=torch.float64, device="cuda") for _ in range(3))
    xb[:n], yb[:n] = cu(x), cu(y)
    ctx = lib.VRM(h=0.05, nu=1e-3)
    with pytest.raises(lib.VRMError) as e:
        ctx.step(xb, yb, n, cu(g), go, 1e-3)
    assert e.value.status == lib.VRM_ERR_ARG
