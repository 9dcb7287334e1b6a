"""A schedule that the caller sets holds in small clouds too, and an answer of
get_schedule set again changes nothing: the launches of a step tell the LP's
forms apart (eight lanes per particle in two launches; otherwise certified
pivots, their FP64 re-runs and the same two over what is handed back)."""
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


@pytest.mark.parametrize("change,more", [({}, 0), (dict(apply_block=64), 0), (dict(lp_block=64), 2),
                                         (dict(lp_blocks_per_sm=8), 2), (dict(lp_block=384, lp_blocks_per_sm=1), 2),
                                         (dict(search_block=64), 0)])
def test_small_clouds_follow_the_schedule(lib, change, more):
    h = 0.02
    x, y, g = vrm_inputs.random_cloud(3000, h=h, jitter=0.3, seed=11)
    n, cap = len(x), 9000
    ctx = lib.VRM(h=h, nu=1e-3)

    def step():
        xb, yb, go = (torch.zeros(cap, dtype=torch.float64, device="cuda") for _ in range(3))
        xb[:n], yb[:n] = cu(x), cu(y)
        n0 = lib.launch_count()
        n2, st = ctx.step(xb, yb, n, cu(g), go, 0.25 * h * h / 8e-3)
        return n2, go[:n2], xb[:n2], lib.launch_count() - n0, st["lp_small_rechecked"]

    step()  # (a context's first step sets its scratch up)
    a = step()
    ctx.set_schedule(dict(ctx.get_schedule(), **change))
    b = step()
    assert a[0] == b[0] and torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
    assert b[3] - a[3] == more
    if more == 0:
        assert a[4] == b[4]
