"""The network's input rows (csrc/vrm_learned.cu) where a value's place within
its segment is hardest to find: rows in any order, all 32 values in one
segment, coincident particles and lattice points at one distance (the index
decides), empty and full rows.  Bit for bit against oracle/mlp.py."""
import numpy as np
import pytest

from oracle import mlp as omlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["spread", "one_segment", "coincident", "lattice"])
def test_rows_of_any_order(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1508_06379_gb300 as v
    v.build()
    rng = np.random.default_rng(len(kind))
    n, h = 600, 0.125
    if kind == "spread":
        x, y = rng.uniform(-1, 1, (2, n))
    elif kind == "one_segment":
        x = rng.uniform(0, 1, n)
        y = x * rng.uniform(0, 0.3, n)
        x[0] = y[0] = -0.25  # every other particle lies in one segment of particle 0
    elif kind == "coincident":
        x, y = rng.choice([-0.5, 0.0, 0.25], (2, n))
    else:
        x, y = rng.integers(-6, 7, (2, n)) / 16.0
    ctx = v.VRM(h=h, nu=1.0)
    xd, yd = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, y))
    assert ctx.k_cap >= 32
    nb = {"count": torch.zeros(n, dtype=torch.int32, device="cuda"),
          "idx": torch.full((n * ctx.k_cap,), -1, dtype=torch.int32, device="cuda")}
    idx = nb["idx"].view(n, -1)
    rows = []
    for i in range(n):
        k = 32 if i == 0 else int(rng.integers(0, 33))
        rows.append(rng.choice(np.setdiff1d(np.arange(n), [i]), k, replace=False))
        idx[i, :k] = torch.from_numpy(rows[i].astype(np.int32)).cuda()
        nb["count"][i] = k
    lst = torch.from_numpy(rng.permutation(n).astype(np.int32)).cuda()
    X, slots = ctx.learned_features(xd, yd, lst, nb)
    Xg, Sg = X[:n].float().cpu().numpy(), slots.cpu().numpy()
    for t, i in enumerate(lst.cpu().numpy()):
        Xo, So = omlp.features(x, y, h, i, rows[i])
        assert np.array_equal(Sg[t], So), i
        assert np.array_equal(Xg[t, :96], Xo) and not Xg[t, 96:].any(), i
