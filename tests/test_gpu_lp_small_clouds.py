"""The small-neighbourhood LPs of clouds of at most 65,536 capacity run eight
lanes per LP (k_lp_df), those of larger ones one LP per thread (k_lp_small32):
both sides of the line bit for bit alike and like the oracle, at particle
counts around a warp's four LPs and a block's sixteen, on jittered clouds and
on exact lattices (exact ties and zeros)."""
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


def weights(lib, orc, x, y, D, h, fallback):
    n = len(x)
    nb = orc.neighbours(x, y, h)
    w = orc.solve_weights(x, y, D, nb, h, fallback=fallback)
    nbt = dict(count=cu(nb["count"]), idx=cu(nb["idx"].reshape(-1)), small=cu(nb["small"].reshape(-1)))
    got = lib.VRM(h=h, nu=1e-3, fallback=fallback).solve_weights(cu(x), cu(y), n, cu(D), nbt)
    for k, width in (("status", 1), ("fii", 1), ("cols", 8), ("f", 8)):
        assert np.array_equal(got[k].cpu().numpy()[:n * width], w[k].reshape(-1)), k
    return got["stats"]


@pytest.mark.parametrize("count", [1, 3, 4, 5, 15, 17, 65, 1200])
@pytest.mark.parametrize("fallback", [True, False])
def test_few_particles(lib, orc, count, fallback):
    x, y, _ = vrm_inputs.random_cloud(1600, h=0.05, jitter=0.35, seed=31)
    D = np.zeros(len(x), np.uint8)
    D[np.random.default_rng(count).permutation(len(x))[:count]] = 1
    st = weights(lib, orc, x, y, D, 0.05, fallback)
    assert st["lp_small_solved"] == count


def test_exact_lattice(lib, orc):
    x, y = vrm_inputs.lattice(1 / 16)
    weights(lib, orc, x, y, np.ones(len(x), np.uint8), 1 / 16, True)


@pytest.mark.parametrize("field", ["mixture", "vortex"])
def test_both_sides_of_the_line(lib, field):
    h, nu = (0.01, 1e-3) if field == "mixture" else (1 / 128, 1e-3)
    if field == "mixture":
        x, y, g = vrm_inputs.random_cloud(30000, h=h, jitter=0.3, seed=32)
    else:
        x, y, g = vrm_inputs.lamb_oseen_lattice(h, 1.0, nu, 1.0, eps=1e-10)
    n, got = len(x), []
    for cap in (65536, 65537):
        xb, yb, go = (torch.zeros(cap, dtype=torch.float64, device="cuda") for _ in range(3))
        xb[:n], yb[:n] = cu(x), cu(y)
        n2, st = lib.VRM(h=h, nu=nu).step(xb, yb, n, cu(g), go, 0.25 * h * h / nu)
        got.append((n2, xb[:n2], yb[:n2], go[:n2], st))
    a, b = got
    assert a[0] == b[0] and all(torch.equal(a[k], b[k]) for k in (1, 2, 3))
    for k in ("lp_small_solved", "lp_small_pivots", "max_pivots", "small_ok", "full_ok", "no_stencil", "max_dt_ratio"):
        assert a[4][k] == b[4][k], k
    assert a[4]["lp_small_rechecked"] <= b[4]["lp_small_rechecked"]
