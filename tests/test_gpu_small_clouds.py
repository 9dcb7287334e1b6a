"""Steps of clouds of at most 65,536 capacity begin with one-block kernels and
scan cells with a warp per particle (csrc/vrm_small.cu, k_search_warp): both
sides of the line bit for bit alike on the circulations that make the growth
control's selection hard (ties, few distinct values, zeros, subnormals, many
binades), at particle counts around a block's chunks and above the keys that
fit in shared memory, and the errors of non-finite input."""
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


FIELDS = {
    "mixture": lambda rng, n: None,
    "equal": lambda rng, n: np.ones(n),
    "signs": lambda rng, n: rng.choice([-1.0, 1.0], n) * 1e-3,
    "few": lambda rng, n: rng.choice([1.0, 0.5, 0.25, 1e-3, 0.0], n),
    "binades": lambda rng, n: 2.0 ** rng.uniform(-200, 0, n),
    "subnormal": lambda rng, n: rng.integers(0, 1000, n) * 5e-324,
    "zeros": lambda rng, n: np.zeros(n),
    "one": lambda rng, n: np.where(np.arange(n) == n // 2, 1.0, 0.0),
    "near": lambda rng, n: 1.0 + rng.integers(0, 700, n) * 2.0 ** -52,
}


def both(lib, x, y, g, h, **kw):
    got = []
    n = len(x)
    for cap in (65536, 65537):
        xb, yb = (torch.zeros(cap, dtype=torch.float64, device="cuda") for _ in range(2))
        xb[:n], yb[:n] = cu(x), cu(y)
        n2, diffused, st = lib.VRM(h=h, nu=1e-3, **kw).insert_reduce(xb, yb, n, cu(g))
        got.append((n2, st, xb[:n2], yb[:n2], diffused[:n2]))
    a, b = got
    assert a[0] == b[0] and a[1] == b[1]
    assert all(torch.equal(p, q) for p, q in zip(a[2:], b[2:]))
    assert int(a[4].sum()) == a[1]["n_diffused"]
    return a


@pytest.mark.parametrize("field", sorted(FIELDS))
@pytest.mark.parametrize("c_diff", [0.0, 1.0, 200.0])
def test_selection(lib, field, c_diff):
    x, y, g = vrm_inputs.random_cloud(2500, h=0.05, jitter=0.3, seed=3)
    v = FIELDS[field](np.random.default_rng(4), len(x))
    both(lib, x, y, g if v is None else v, 0.05, c_diff=c_diff)


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1023, 1025, 21504, 21505, 40000])
def test_counts(lib, n):
    x, y, g = vrm_inputs.random_cloud(40500, h=0.01, jitter=0.3, seed=5)
    both(lib, x[:n], y[:n], g[:n], 0.01)


def test_ties_stay_out_by_index(lib, orc):
    rng = np.random.default_rng(6)
    x, y, _ = vrm_inputs.random_cloud(900, h=0.1, jitter=0.3, seed=7)
    g = rng.choice([1.0, 0.02, 0.01], len(x), p=[0.2, 0.4, 0.4])
    a = both(lib, x, y, g, 0.1, c_diff=40.0)
    c = orc.constants(0.1, c_diff=40.0)["c_bound"]
    assert np.array_equal(a[4].cpu().numpy()[:len(x)], orc.reduce(g, c))


@pytest.mark.parametrize("where", ["x", "gamma"])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_non_finite_input_is_refused(lib, where, value):
    x, y, g = vrm_inputs.random_cloud(400, h=0.1, jitter=0.3, seed=8)
    (x if where == "x" else g)[7] = value
    cap = 2000
    xb, yb, go = (torch.zeros(cap, dtype=torch.float64, device="cuda") for _ in range(3))
    xb[:len(x)], yb[:len(y)] = cu(x), cu(y)
    with pytest.raises(lib.VRMError) as e:
        lib.VRM(h=0.1, nu=1e-3).step(xb, yb, len(x), cu(g), go, 1e-3)
    assert e.value.status == lib.VRM_ERR_ARG
