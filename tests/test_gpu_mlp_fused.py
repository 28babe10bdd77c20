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


@pytest.mark.parametrize("n", [1, 30, 127, 129, 1024, 152 * 128 + 1, 2 * 152 * 128 + 77])
@pytest.mark.parametrize("aligned", [True, False])
def test_gradient_row_counts(cv, orc, n, aligned):  # noqa: F811
    """Loss and gradient over part of a tile, several slices of the weight
    gradients and a last turn of one tile; into a gradient buffer at any
    float address.  Bars of test_gpu_surrogate."""
    import ctypes

    import torch

    from paper_2211_14318_gb300 import api

    X, mean, std = _net_inputs(orc, 2048, 33)
    flat = _set(cv, 10)
    cv.surrogate_set_weights(flat, mean, std)
    rng = np.random.default_rng(n)
    at = np.arange(n) % 2048
    Y = np.column_stack([rng.uniform(0, np.pi, (n, 2)), rng.uniform(0.05, 0.95, n),
                         rng.normal(0, 0.3, (n, 4))]).astype(np.float32)
    Y[::5, :3] = np.nan
    Xd, Yd = torch.from_numpy(X.astype(np.float32)[at]).cuda(), torch.from_numpy(Y).cuda()
    if aligned:
        loss, grad = cv.surrogate_loss_grad(Xd, Yd)
    else:
        loss = torch.empty(1, device="cuda")
        grad = torch.empty(api.SURROGATE_PARAMS + 1, device="cuda")[1:]
        rc = api.lib().surrogate_loss_grad(cv._h, ctypes.c_int64(n), Xd.data_ptr(), Yd.data_ptr(),
                                           loss.data_ptr(), grad.data_ptr(),
                                           torch.cuda.current_stream().cuda_stream)
        assert rc == 0
    g = grad.cpu().numpy().astype(np.float64)
    istd = (1.0 / std.astype(np.float32)).astype(np.float32).astype(np.float64)
    out, cache = mlp.forward(flat, X.astype(np.float32).astype(np.float64)[at], mean, 1.0 / istd, bf=True)
    L, dout = mlp.loss_and_grad(out, Y.astype(np.float64))
    ref = mlp.backward(flat, cache, dout, bf=True)
    assert abs(loss.item() - L) < 1e-3 * (1 + abs(L))
    o = 0
    for shp in mlp.SHAPES:
        k = int(np.prod(shp))
        a, b = g[o:o + k], ref[o:o + k]
        rel = np.linalg.norm(a - b) / (np.linalg.norm(b) + 1e-30)
        cos = a @ b / (np.linalg.norm(a) * np.linalg.norm(b) + 1e-30)
        assert rel < 2e-2 and cos > 0.9995, (shp, rel, cos)
        o += k
