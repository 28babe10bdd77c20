"""Inference of the network in one kernel at row counts that leave a CTA no
row, part of a tile, one tile, an odd number of tiles and a last turn of one
tile: against the oracle with the same bf16 rounding points (bar of
test_gpu_surrogate: 2e-3 (1 + |o|)), and rows do not depend on their place."""
import numpy as np
import pytest

from oracle import mlp
from test_gpu_parity import cv  # noqa: F401
from test_gpu_surrogate import _net_inputs, _set

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 257, 152 * 128, 152 * 128 + 1, 2 * 152 * 128 + 5,
                               3 * 152 * 128 - 1])
def test_forward_row_counts(cv, orc, n):  # noqa: F811
    import torch

    X, mean, std = _net_inputs(orc, 2048, 31)
    flat = _set(cv, 9)
    cv.surrogate_set_weights(flat, mean, std)
    at = np.arange(n) % 2048
    Xd = torch.from_numpy(X.astype(np.float32)[at]).cuda()
    out = cv.surrogate_forward(Xd).cpu().numpy()
    X32 = X.astype(np.float32).astype(np.float64)
    ref, _ = mlp.forward(flat, X32, mean, 1.0 / (1.0 / std.astype(np.float32)).astype(np.float64), bf=True)
    first = out[:2048].astype(np.float64)
    r = ref[:first.shape[0]]
    assert np.max(np.abs(first - r) / (1 + np.abs(r))) < 2e-3
    assert np.array_equal(out, out[:2048][at])
