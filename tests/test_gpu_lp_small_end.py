"""The end of the small LPs in pairs (csrc/vrm_lp.cu, k_lp_small_end): some
blocks re-run the uncertain ones in FP64, a warp each, while others solve the
rest.  Lattices with noise around the pivots' tolerances, whose LPs are partly
uncertain, and with holes, whose LPs are partly infeasible; a few particles to
more than one pass of the re-run's warps; with and without the full
neighbourhoods behind them.

Bar: the bits, statuses and counts of FP64 pivots."""
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


@pytest.mark.parametrize("fallback", [True, False])
@pytest.mark.parametrize("bits", [52, 43, 40, 37, 34, 31, 28, 24, 20])
@pytest.mark.parametrize("inv_h,holes", [(4, 0), (16, 300), (64, 0), (64, 2000)])
def test_noisy_lattices(lib, orc, inv_h, holes, bits, fallback):
    h = 1.0 / inv_h
    x, y = vrm_inputs.lattice(h)
    rng = np.random.default_rng(bits + inv_h)
    keep = np.sort(rng.permutation(len(x))[holes:])
    x, y = x[keep], y[keep]
    n = len(x)
    x = x + rng.uniform(-1, 1, n) * h * 2.0 ** -bits
    y = y + rng.uniform(-1, 1, n) * h * 2.0 ** -bits
    nb = orc.neighbours(x, y, h)
    nbt = dict(count=cu(nb["count"]), idx=cu(nb["idx"].reshape(-1)), small=cu(nb["small"].reshape(-1)))
    got = []
    for k in (0, 1):
        ctx = lib.VRM(h=h, nu=1e-3, fallback=fallback)
        ctx.set_schedule(dict(ctx.get_schedule(), lp_fp64_pivots=k))
        got.append(ctx.solve_weights(cu(x), cu(y), n, cu(np.ones(n, np.uint8)), nbt))
    for key in ("status", "cols", "f", "fii"):
        assert torch.equal(got[0][key], got[1][key]), key
    a, b = ({k: v for k, v in g["stats"].items() if k != "lp_small_rechecked"} for g in got)
    assert a == b


@pytest.mark.parametrize("bits,rechecked", [(2, (1, 6144)), (26, (6145, 10 ** 9)), (52, (6145, 10 ** 9))])
def test_short_and_long_lists_of_mid_sized_clouds(lib, orc, bits, rechecked):
    # above the small clouds' size: the hand-backs in pairs or, past 6144 of them, in FP64
    h = 1.0 / 140
    x, y = vrm_inputs.lattice(h)
    rng = np.random.default_rng(bits)
    n = len(x)
    assert 65536 < n < 6 * 65536
    x = x + rng.uniform(-1, 1, n) * h * 2.0 ** -bits
    y = y + rng.uniform(-1, 1, n) * h * 2.0 ** -bits
    nb = orc.neighbours(x, y, h)
    nbt = dict(count=cu(nb["count"]), idx=cu(nb["idx"].reshape(-1)), small=cu(nb["small"].reshape(-1)))
    got = []
    for k in (0, 1):
        ctx = lib.VRM(h=h, nu=1e-3)
        ctx.set_schedule(dict(ctx.get_schedule(), lp_fp64_pivots=k))
        got.append(ctx.solve_weights(cu(x), cu(y), n, cu(np.ones(n, np.uint8)), nbt))
    assert rechecked[0] <= got[0]["stats"]["lp_small_rechecked"] <= rechecked[1]
    for key in ("status", "cols", "f", "fii"):
        assert torch.equal(got[0][key], got[1][key]), key
    a, b = ({k: v for k, v in g["stats"].items() if k != "lp_small_rechecked"} for g in got)
    assert a == b
