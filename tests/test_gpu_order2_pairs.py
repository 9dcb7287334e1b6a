"""The n = 2 LPs' kernels at the edges of their work split (csrc/vrm_lp.cu:
half-warps for the small neighbourhoods, warps for the full ones, threads for
the final solves): few diffused particles, exact lattices (ties and exact
zeros), and the FP64-pivot schedule, each bit for bit the oracle's."""
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


def compare(lib, orc, x, y, D, h, R, fp64_pivots=0, fallback=True):
    n = len(x)
    nb = orc.neighbours(x, y, h, R=R)
    w = orc.solve_weights(x, y, D, nb, h, order=2, fallback=fallback)
    ctx = lib.VRM(h=h, nu=1e-3, R=R, order=2, fallback=fallback)
    ctx.set_schedule(dict(ctx.get_schedule(), lp_fp64_pivots=fp64_pivots))
    nbt = dict(count=cu(nb["count"]), idx=cu(nb["idx"].reshape(-1)), small=cu(nb["small"].reshape(-1)))
    got = ctx.solve_weights(cu(x), cu(y), n, cu(D), nbt)
    assert np.array_equal(got["status"].cpu().numpy()[:n], w["status"])
    assert np.array_equal(got["cols"].cpu().numpy()[:12 * n].reshape(n, 12), w["cols"])
    assert np.array_equal(got["f"].cpu().numpy()[:12 * n].reshape(n, 12), w["f"])
    assert np.array_equal(got["fii"].cpu().numpy()[:n], w["fii"])
    return got["stats"]


@pytest.mark.parametrize("count", [1, 2, 3, 31, 33, 127, 1000])
@pytest.mark.parametrize("fp64_pivots", [0, 1])
def test_few_particles(lib, orc, count, fp64_pivots):
    x, y, _ = vrm_inputs.random_cloud(1600, h=0.05, jitter=0.3, seed=21)
    D = np.zeros(len(x), np.uint8)
    D[np.random.default_rng(count).permutation(len(x))[:count]] = 1
    st = compare(lib, orc, x, y, D, 0.05, 2.5, fp64_pivots)
    assert st["lp_small_solved"] == count and st["lp_small_rechecked"] == 0


def test_pivot_counts_do_not_depend_on_the_schedule(lib, orc):
    x, y, _ = vrm_inputs.random_cloud(2500, h=0.05, jitter=0.35, seed=22)
    D = np.ones(len(x), np.uint8)
    a, b = (compare(lib, orc, x, y, D, 0.05, 2.5, k) for k in (0, 1))
    assert a == b


@pytest.mark.parametrize("R", [2.0, 2.5])
def test_exact_lattice_and_no_fallback(lib, orc, R):
    x, y = vrm_inputs.lattice(1 / 16)
    D = np.ones(len(x), np.uint8)
    compare(lib, orc, x, y, D, 1 / 16, R)
    compare(lib, orc, x, y, D, 1 / 16, R, fallback=False)


@pytest.mark.parametrize("R", [2.0, 2.5])
def test_noisy_lattice_does_not_depend_on_the_schedule(lib, orc, R):
    # offsets with noise in the second half of the pairs; the bases are so
    # near to singular that FP64 tableaus and the oracle's solves part ways,
    # so the two schedules are compared with each other
    x, y = vrm_inputs.lattice(1 / 16)
    x = x + np.random.default_rng(5).uniform(-1, 1, len(x)) * 2.0 ** -34
    n, nb, got = len(x), orc.neighbours(x, y, 1 / 16, R=R), []
    nbt = dict(count=cu(nb["count"]), idx=cu(nb["idx"].reshape(-1)), small=cu(nb["small"].reshape(-1)))
    for k in (0, 1):
        ctx = lib.VRM(h=1 / 16, nu=1e-3, R=R, order=2)
        ctx.set_schedule(dict(ctx.get_schedule(), lp_fp64_pivots=k))
        got.append(ctx.solve_weights(cu(x), cu(y), n, cu(np.ones(n, np.uint8)), nbt))
    for key in ("status", "cols", "f", "fii"):
        assert torch.equal(got[0][key], got[1][key])
    assert got[0]["stats"] == got[1]["stats"]
