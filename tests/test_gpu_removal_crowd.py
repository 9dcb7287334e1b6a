"""Particle removal with far more particles in one spot than a row holds: the
capacity error comes at once, however many entries one target would get, and
the context then removes as before."""
import time

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


@pytest.mark.parametrize("m", [40, 20000])
def test_a_crowded_spot_is_a_capacity_error_at_once(lib, orc, m):
    h = 0.05
    x, y = vrm_inputs.lattice(h, -0.5, 0.5)
    g = np.linspace(1.0, 2.0, len(x))
    rng = np.random.default_rng(1)
    k = len(x) // 2 + 10
    xs = np.concatenate([x, x[k] + rng.uniform(-0.1, 0.1, m) * h])
    ys = np.concatenate([y, y[k] + rng.uniform(-0.1, 0.1, m) * h])
    gs = np.concatenate([g, rng.uniform(0.1, 0.2, m)])
    ctx = lib.VRM(h=h, nu=1e-3)
    X, Y, G = cu(xs), cu(ys), cu(gs)
    torch.cuda.synchronize()
    t = time.monotonic()
    with pytest.raises(lib.VRMError) as e:
        ctx.remove_close(X, Y, G, len(xs))
    assert e.value.status == lib.VRM_ERR_CAPACITY
    assert time.monotonic() - t < 2.0  # (a few milliseconds; a walk per entry took minutes)
    # a few of them are removed as ever
    q = len(x) + 5
    xo, yo, go, _, cand, _, _ = orc.remove_close(xs[:q], ys[:q], gs[:q], h)
    X, Y, G, kept, st = ctx.remove_close(cu(xs[:q]), cu(ys[:q]), cu(gs[:q]), q)
    assert kept == len(xo) < q and st["remove_candidates"] == cand
    assert np.array_equal(X.cpu().numpy(), xo) and np.array_equal(G.cpu().numpy(), go)
