"""Inference by CTA pairs (csrc/vrm_mlp.cu) at the row counts where a pair's
work changes: one half empty, both halves full, one row more; as many 256-row
tiles as pairs, one more, and a second round of slots.

Every product keeps a row's sum within the row, so a prefix of the rows gives
the same bits as the whole, whatever tile, half and slot a row falls into.  The
whole is held against the oracle with the bar of test_gpu_mlp.py."""
import numpy as np
import pytest

import vrm_inputs
from oracle import mlp as omlp
from test_gpu_mlp import bf16_rows, lib, quantised  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PAIRS = 76
ROWS = 256 * PAIRS * 3 + 300


@pytest.fixture(scope="module")
def whole(lib):  # noqa: F811
    X, _ = vrm_inputs.mlp_rows(ROWS, seed=11)
    net = lib.MLP(batch_rows=128)
    net.set_params(vrm_inputs.mlp_params())
    Xd = bf16_rows(X)
    Y = net.forward(Xd, ROWS)
    net.check()
    return net, X, Xd, Y


def test_against_the_oracle(whole):
    _, X, _, Y = whole
    Yo, _ = omlp.forward(quantised(vrm_inputs.mlp_params()), X[:, :96], bf16_acts=True)
    assert np.abs(Y.cpu().numpy() - Yo).max() <= 1e-2 * max(1.0, np.abs(Yo).max())


@pytest.mark.parametrize("rows", [1, 127, 128, 129, 255, 256, 257, 512, 256 * PAIRS - 128, 256 * PAIRS,
                                  256 * PAIRS + 1, 256 * PAIRS * 2 + 129, 256 * PAIRS * 3 - 255])
def test_prefix(whole, rows):
    net, _, Xd, Y = whole
    y = net.forward(Xd[:rows].contiguous(), rows)
    net.check()
    assert torch.equal(y[:rows], Y[:rows])
