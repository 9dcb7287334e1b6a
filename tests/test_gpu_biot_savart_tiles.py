"""The direct sum's tiles (vrm_biot_savart): sizes at the edges of its source
tiles (256, tested for distance in parts of 64) and target blocks, and the
independence of a target's bits from everything that picks a kernel path: the
order of the targets (whole tiles far from a warp's targets, or pairs decided
one by one), their number (targets per thread, split of the tiles over blocks,
groups of tiles) and other targets' odd coordinates.

Tolerance of the sizes test: that of test_gpu_biot_savart.py, 2e-6 of
sum_j |Gamma_j K_eps|."""
import math

import numpy as np
import pytest

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


def lattice(side, h, seed):
    rng = np.random.default_rng(seed)
    c = (np.arange(side) - 0.5 * (side - 1)) * h
    X, Y = np.meshgrid(c, c)
    return (X.ravel() + rng.uniform(-0.3, 0.3, X.size) * h, Y.ravel() + rng.uniform(-0.3, 0.3, X.size) * h,
            rng.normal(0.0, 1e-3, X.size))


def velocity(lib, x, y, g, xt, yt, eps):
    u, v = lib.VRM(h=eps / 3, nu=1e-3).biot_savart(cu(x), cu(y), cu(g), len(x), cu(xt), cu(yt), len(xt), eps)
    return np.stack([u.cpu().numpy(), v.cpu().numpy()])


@pytest.mark.parametrize("n,m", [(1, 1), (63, 255), (64, 257), (65, 31), (255, 513), (256, 64), (257, 511),
                                 (1025, 33), (5000, 700)])
def test_sizes(lib, n, m):
    rng = np.random.default_rng(n * 1000 + m)
    eps = 0.02
    x, y, g = rng.uniform(-1, 1, n), rng.uniform(-1, 1, n), rng.normal(0.0, 1e-3, n)
    xt, yt = rng.uniform(-1, 1, m), rng.uniform(-1, 1, m)
    k = min(n, m) // 2
    xt[:k], yt[:k] = x[:k], y[:k]  # targets on sources
    u, v = velocity(lib, x, y, g, xt, yt, eps)
    dx, dy = xt[:, None] - x, yt[:, None] - y
    r2 = dx * dx + dy * dy
    with np.errstate(divide="ignore", invalid="ignore"):
        w = np.where(r2 > 0, -np.expm1(-r2 / eps ** 2) / (2 * math.pi * r2), 0.0) * g
        S = np.abs(w * np.sqrt(r2)).sum(1)
    assert np.all(np.abs(u + (dy * w).sum(1)) <= 2e-6 * S + 1e-300)
    assert np.all(np.abs(v - (dx * w).sum(1)) <= 2e-6 * S + 1e-300)


def test_bits_do_not_depend_on_the_order_of_the_targets(lib):
    x, y, g = lattice(90, 0.01, 1)
    xt, yt, _ = lattice(70, 0.02, 2)
    p = np.random.default_rng(3).permutation(len(xt))
    a = velocity(lib, x, y, g, xt, yt, 0.03)
    b = velocity(lib, x, y, g, xt[p], yt[p], 0.03)
    assert np.array_equal(a[:, p], b)


def test_bits_do_not_depend_on_the_number_of_targets(lib):
    # 440^2 sources at 200^2 targets: more tile sums than are kept at a time
    x, y, g = lattice(440, 0.005, 4)
    xt, yt, _ = lattice(200, 0.015, 5)
    a = velocity(lib, x, y, g, xt, yt, 0.015)
    for k in (3, 700, 9000):
        assert np.array_equal(a[:, :k], velocity(lib, x, y, g, xt[:k], yt[:k], 0.015))


@pytest.mark.parametrize("odd", [1e25, 1e12, np.inf, np.nan])
def test_odd_targets_keep_to_themselves(lib, odd):
    x, y, g = lattice(40, 0.01, 6)
    xt, yt, _ = lattice(20, 0.02, 7)
    a = velocity(lib, x, y, g, xt, yt, 0.03)
    xo = np.concatenate([xt[:100], [odd], xt[100:]])
    yo = np.concatenate([yt[:100], [0.0], yt[100:]])
    b = velocity(lib, x, y, g, xo, yo, 0.03)
    assert np.array_equal(np.delete(b, 100, 1), a)
    if np.isfinite(odd):  # the far field Gamma / (2 pi x); 0 where q overflows in binary32
        far = g.sum() / (2 * math.pi * odd) if odd * odd < 3.4e38 else 0.0
        assert abs(b[0, 100]) <= 1e-6 and abs(b[1, 100] - far) <= 2e-6 * np.abs(g).sum() / odd
    else:
        assert np.isnan(b[:, 100]).all()
