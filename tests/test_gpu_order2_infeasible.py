"""Small-neighbourhood LPs of n = 2 that are certified infeasible without a
final solve (csrc/vrm_lp.cu, k_lp_df): lattices with noise from the size of
one rounding to a third of a spacing, where the phase-I sum crosses the
feasibility tolerances, with the default schedule against FP64 pivots, whose
LPs are all solved; on jittered clouds also against the oracle.

Bar: the same bits, statuses and counts."""
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
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def solved(lib, x, y, nb, h, R, fp64_pivots, fallback):
    n = len(x)
    ctx = lib.VRM(h=h, nu=1e-3, R=R, order=2, fallback=fallback)
    ctx.set_schedule(dict(ctx.get_schedule(), lp_fp64_pivots=fp64_pivots))
    nbt = dict(count=cu(nb["count"]), idx=cu(nb["idx"].reshape(-1)), small=cu(nb["small"].reshape(-1)))
    return ctx.solve_weights(cu(x), cu(y), n, cu(np.ones(n, np.uint8)), nbt)


@pytest.mark.parametrize("fallback", [True, False])
@pytest.mark.parametrize("bits", [52, 46, 43, 40, 37, 34, 31, 28, 24, 16, 8])
def test_noisy_lattices(lib, orc, bits, fallback):
    h, R = 1 / 16, 2.5
    x, y = vrm_inputs.lattice(h)
    rng = np.random.default_rng(bits)
    x = x + rng.uniform(-1, 1, len(x)) * h * 2.0 ** -bits
    y = y + rng.uniform(-1, 1, len(y)) * h * 2.0 ** -bits
    nb = orc.neighbours(x, y, h, R=R)
    a, b = (solved(lib, x, y, nb, h, R, k, fallback) for k in (0, 1))
    for key in ("status", "cols", "f", "fii"):
        assert torch.equal(a[key], b[key]), key
    assert a["stats"] == b["stats"]


@pytest.mark.parametrize("jitter", [0.05, 0.2, 0.35])
@pytest.mark.parametrize("h", [1e-3, 0.05, 50.0])
def test_jittered_clouds(lib, orc, jitter, h):
    x, y, _ = vrm_inputs.random_cloud(2000, h=0.05, jitter=jitter, seed=int(100 * jitter))
    x, y = x * (h / 0.05), y * (h / 0.05)
    n, nb = len(x), orc.neighbours(x, y, h, R=2.5)
    for fallback in (True, False):
        w = orc.solve_weights(x, y, np.ones(n, np.uint8), nb, h, order=2, fallback=fallback)
        got = solved(lib, x, y, nb, h, 2.5, 0, fallback)
        assert np.array_equal(got["status"].cpu().numpy()[:n], w["status"])
        assert np.array_equal(got["cols"].cpu().numpy()[:12 * n].reshape(n, 12), w["cols"])
        assert np.array_equal(got["f"].cpu().numpy()[:12 * n].reshape(n, 12), w["f"])
