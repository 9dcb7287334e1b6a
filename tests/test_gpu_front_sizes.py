"""The small clouds' front at its largest sizes (16,383 particles in one block,
65,536 in the cluster: the shared memory is full) and, in one block, on the
circulations that make the selection hard, against the kernels of larger clouds
and, for ties, the oracle.  No insertion rounds run, so every capacity takes
every cloud.

Bar: the same bits and counts."""
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
    "signs": lambda rng, n: rng.choice([-1.0, 1.0], n) * 1e-3,
    "subnormal": lambda rng, n: rng.integers(0, 1000, n) * 5e-324,
    "one": lambda rng, n: np.where(np.arange(n) == n // 2, 1.0, 0.0),
    "binades": lambda rng, n: 2.0 ** rng.uniform(-200, 0, n),
    "gauss": lambda rng, n: rng.standard_normal(n) * np.exp(-rng.uniform(0, 40, n)),
}


def agree(lib, x, y, g, h, caps, **kw):
    got = []
    n = len(x)
    for cap in caps:
        xb, yb = (torch.zeros(cap, dtype=torch.float64, device="cuda") for _ in range(2))
        xb[:n], yb[:n] = cu(x), cu(y)
        n2, diffused, st = lib.VRM(h=h, nu=1e-3, max_rounds=0, **kw).insert_reduce(xb, yb, n, cu(g))
        assert n2 == n and int(diffused.sum()) == st["n_diffused"]
        got.append((st, diffused[:n].clone()))
    assert len(got) == len(caps)
    for a in got[1:]:
        assert a[0] == got[0][0] and torch.equal(a[1], got[0][1])
    return got[0]


@pytest.mark.parametrize("field", sorted(FIELDS))
@pytest.mark.parametrize("c_diff", [0.0, 1.0, 200.0])
def test_one_block(lib, field, c_diff):
    x, y, _ = vrm_inputs.random_cloud(2500, h=0.05, jitter=0.3, seed=3)
    agree(lib, x, y, FIELDS[field](np.random.default_rng(4), len(x)), 0.05, (16383, 65537), c_diff=c_diff)


def test_one_block_ties_stay_out_by_index(lib, orc):
    x, y, _ = vrm_inputs.random_cloud(900, h=0.1, jitter=0.3, seed=7)
    g = np.random.default_rng(6).choice([1.0, 0.02, 0.01], len(x), p=[0.2, 0.4, 0.4])
    _, diffused = agree(lib, x, y, g, 0.1, (16383, 65537), c_diff=40.0)
    assert np.array_equal(diffused.cpu().numpy(), orc.reduce(g, orc.constants(0.1, c_diff=40.0)["c_bound"]))


@pytest.mark.parametrize("field", sorted(FIELDS))
@pytest.mark.parametrize("n,caps", [(16383, (16383, 65537)), (65535, (65535, 65537)), (65536, (65536, 65537))])
def test_full(lib, field, n, caps):
    side = int(np.ceil(np.sqrt(n)))
    k = np.arange(n)
    rng = np.random.default_rng(n)
    h = 0.01
    x, y = (k % side + rng.uniform(-0.3, 0.3, n)) * h, (k // side + rng.uniform(-0.3, 0.3, n)) * h
    agree(lib, x, y, FIELDS[field](rng, n), h, caps, c_diff=20.0)
