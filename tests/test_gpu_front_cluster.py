"""The small clouds' front in one block (capacity below 16,384), in a cluster
of eight (up to 65,536) and in the kernels of larger clouds: the same
particles at capacities on both sides of each line, with counts that leave
blocks of the cluster short or empty and equal circulations over several of
them.

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
    "equal": lambda rng, n: np.ones(n),
    "few": lambda rng, n: rng.choice([1.0, 0.5, 0.25, 1e-3, 0.0], n),
    "binades": lambda rng, n: 2.0 ** rng.uniform(-200, 0, n),
    "zeros": lambda rng, n: np.zeros(n),
    "last": lambda rng, n: np.where(np.arange(n) == n - 1, 1.0, 0.0),
    "near": lambda rng, n: 1.0 + rng.integers(0, 700, n) * 2.0 ** -52,
    "gauss": lambda rng, n: rng.standard_normal(n) * np.exp(-rng.uniform(0, 40, n)),
}


@pytest.mark.parametrize("n", [1, 7, 9, 65, 1000, 8191, 8193, 12000])
@pytest.mark.parametrize("field", sorted(FIELDS))
def test_forms_agree(lib, field, n):
    x, y, _ = vrm_inputs.random_cloud(12100, h=0.05, jitter=0.3, seed=3)
    x, y, g = x[:n], y[:n], FIELDS[field](np.random.default_rng(n), n)
    got = []
    for cap in (16383, 16384, 65537):
        xb, yb = (torch.zeros(cap, dtype=torch.float64, device="cuda") for _ in range(2))
        xb[:n], yb[:n] = cu(x), cu(y)
        try:
            n2, diffused, st = lib.VRM(h=0.05, nu=1e-3, c_diff=20.0).insert_reduce(xb, yb, n, cu(g))
        except lib.VRMError as e:
            assert cap < 65537 and e.status == lib.VRM_ERR_CAPACITY
            continue
        got.append((n2, st, xb[:n2], yb[:n2], diffused[:n2]))
    for a in got[:-1]:
        assert a[0] == got[-1][0] and a[1] == got[-1][1]
        assert all(torch.equal(p, q) for p, q in zip(a[2:], got[-1][2:]))
