"""A training step's kernels over the batch sizes that split differently
(csrc/vrm_mlp.cu): one tile, as many tiles as the weight gradients have
splits, a prime number of them (one split), more tiles than SMs (a CTA takes
several), and missing rows; gradients against the oracle with the bars of
test_gpu_mlp.py, and the update against AdamW applied to those gradients."""
import numpy as np
import pytest

import vrm_inputs
from oracle import mlp as omlp
from test_gpu_mlp import bf16_rows, blocks, lib, quantised  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def data(rows, seed):
    rng = np.random.default_rng(seed)
    k = rng.integers(8, 33, rows)
    mask = (np.arange(32) < k[:, None]).astype(np.float64)
    xi, eta = (rng.integers(-128, 129, (rows, 32)) / 64.0 * mask for _ in range(2))
    return np.concatenate([xi, eta, mask, 0 * mask], 1), mask * (np.maximum(xi, 0) / 2 + eta ** 2 / 8)


@pytest.mark.parametrize("B,rows", [(128, 1), (128, 97), (8192, 8192), (128 * 67, 128 * 67 - 5), (128 * 160, 20000)])
def test_gradients(lib, B, rows):  # noqa: F811
    theta = vrm_inputs.mlp_params()
    X, T = data(rows, B + rows)
    net = lib.MLP(batch_rows=B)
    net.set_params(theta)
    g, loss = net.grads(bf16_rows(X), torch.from_numpy(T.astype(np.float32)).cuda())
    net.check()
    thq = quantised(theta)
    Yo, cache = omlp.forward(thq, X[:, :96], bf16_acts=True)
    lo, dY = omlp.loss(Yo, T, X[:, 64:96])
    assert abs(loss - lo) <= 2e-2 * lo
    for k, (a, b) in enumerate(zip(blocks(g.cpu().numpy().astype(np.float64)), blocks(omlp.backward(thq, cache, dY)))):
        assert np.linalg.norm(a - b) <= 2e-2 * np.linalg.norm(b), k


@pytest.mark.parametrize("offset", [0, 1])
def test_step_is_adamw_on_the_gradients(lib, offset):  # noqa: F811
    # the fused update against the gradient call and the separate AdamW call,
    # from rows on and off a 4-byte boundary; both read the same gradient, and
    # an fp32 AdamW step differs by the contraction of its products at most
    X, T = data(500, 3)
    Xp = torch.empty(500 * 128 + 1, dtype=torch.bfloat16, device="cuda")
    Xd = Xp[offset:offset + 500 * 128].view(500, 128)
    Xd.copy_(bf16_rows(X))
    Td = torch.from_numpy(T.astype(np.float32)).cuda()
    idx = torch.randperm(500, generator=torch.Generator().manual_seed(1))[:300].to(torch.int32).cuda()
    a, b = lib.MLP(batch_rows=384), lib.MLP(batch_rows=384)
    for net in (a, b):
        net.set_params(vrm_inputs.mlp_params())
    for t in (1, 2, 3):
        a.train_step(Xd, Td, idx, t, lr=1e-3, weight_decay=0.01)
        g, _ = b.grads(Xd[idx.long()].contiguous(), Td[idx.long()].contiguous())
        b.adamw(g, t, lr=1e-3, weight_decay=0.01)
        assert float((a.get_params() - b.get_params()).abs().max()) <= 1e-6
    Y = (a.forward(Xd[:130].contiguous(), 130), b.forward(Xd[:130].contiguous(), 130))
    assert float((Y[0] - Y[1]).abs().max()) <= 2e-2 * float(Y[0].abs().max())
