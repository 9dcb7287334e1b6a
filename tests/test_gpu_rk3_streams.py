"""vrm_rk3_step's analytic velocity runs on a stream of the context's own:
one partly filled block and more particles than one pass of the grid (152
blocks of 256), on a stream of the caller's, and a step after one that ran
out of capacity and returned early.

Bar: positions and circulations equal the oracle's bit for bit, as on the
default stream."""
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


@pytest.mark.parametrize("npts", [200, 45000])
def test_rk3_on_a_users_stream_after_an_overflow(lib, orc, npts):
    h, nu, t = 0.02, 1e-3, 1.0
    x, y, g = vrm_inputs.random_cloud(npts, h=h, jitter=0.3, seed=77)
    g = g * 50.0
    dt = 0.25 * h / 1.5
    vel = dict(gamma=1.0, nu=nu)
    Xo, Yo, Go, _ = orc.rk3_step(x, y, g, h, nu, t, dt, vel=vel)
    n = len(x)
    ctx = lib.VRM(h=h, nu=nu)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        for cap in (n + 1, 4 * n + 4096):
            xb, yb, gb, out = (torch.zeros(cap, dtype=torch.float64, device="cuda") for _ in range(4))
            for buf, v in ((xb, x), (yb, y), (gb, g)):
                buf[:n] = torch.from_numpy(v).cuda()
            if cap == n + 1:
                with pytest.raises(lib.VRMError):
                    ctx.rk3_step(xb, yb, n, gb, out, t, dt, vel)
                continue
            n2, _ = ctx.rk3_step(xb, yb, n, gb, out, t, dt, vel)
        assert n2 == len(Xo)
        got = [v[:n2].cpu().numpy() for v in (xb, yb, out)]
    assert np.array_equal(got[0], Xo) and np.array_equal(got[1], Yo) and np.array_equal(got[2], Go)
