"""Neighbour rows of vrm_build_neighbourhoods at the widths and counts around the
sorting networks (16, 24, 32 entries) and the row's vectors of four, rows cut
at k_cap included, against numpy's; the largest count that the removal pass
reports from its own scan."""
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


def members(x, y, h, r=0.5, R=2.0):
    dx, dy = x[None] - x[:, None], y[None] - y[:, None]
    d2 = dx * dx + dy * dy
    m = (d2 >= (r * h) ** 2) & (d2 <= (R * h) ** 2)
    np.fill_diagonal(m, False)
    return m


@pytest.mark.parametrize("k_cap", [8, 9, 15, 16, 17, 22, 24, 25, 31, 32])
@pytest.mark.parametrize("n", [60, 300, 700, 1100])
def test_rows(lib, k_cap, n):
    # a uniform scatter: counts from a few to well above k_cap
    x, y, _ = vrm_inputs.uniform_scatter(n, half_width=0.5, seed=n)
    h = 0.06
    want = members(x, y, h)
    nb = lib.VRM(h=h, nu=1e-3, k_cap=k_cap).build_neighbourhoods(
        cu(x), cu(y), n, out={"idx": torch.full((n * k_cap,), -7, dtype=torch.int32, device="cuda")}, max_count=False)
    count, idx = nb["count"].cpu().numpy()[:n], nb["idx"].cpu().numpy().reshape(n, k_cap)
    assert np.array_equal(count, want.sum(1))
    for i in range(n):
        js = np.nonzero(want[i])[0][:k_cap]
        assert np.array_equal(idx[i, :len(js)], js) and (idx[i, len(js):] == -7).all()


def test_rows_off_a_vector_boundary(lib):
    x, y, _ = vrm_inputs.uniform_scatter(500, half_width=0.5, seed=1)
    h, n = 0.06, 500
    buf = torch.full((n * 32 + 1,), -7, dtype=torch.int32, device="cuda")
    ctx = lib.VRM(h=h, nu=1e-3)
    a = ctx.build_neighbourhoods(cu(x), cu(y), n, out={"idx": buf[1:]}, max_count=False)["idx"]
    b = ctx.build_neighbourhoods(cu(x), cu(y), n, max_count=False,
                                 out={"idx": torch.full((n * 32,), -7, dtype=torch.int32, device="cuda")})["idx"]
    assert torch.equal(a, b)


@pytest.mark.parametrize("h", [0.02, 0.05])
def test_removal_reports_the_largest_count(lib, h):
    x, y, g = vrm_inputs.uniform_scatter(900, half_width=0.5, seed=9)
    most = int(members(x, y, h).sum(1).max())
    ctx = lib.VRM(h=h, nu=1e-3)
    if most <= 32:
        assert ctx.remove_close(cu(x), cu(y), cu(g), 900)[4]["max_count"] == most
    else:
        with pytest.raises(lib.VRMError) as e:
            ctx.remove_close(cu(x), cu(y), cu(g), 900)
        assert e.value.status == lib.VRM_ERR_CAPACITY
