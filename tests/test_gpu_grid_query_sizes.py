"""The global-grid query at query counts on both sides of the limits where a
block takes fewer queries: a query's results do not depend on how many there are
(bit for bit), and the first ones agree with the oracle (bars of
test_gpu_grid_query: W_interp bit for bit, leaf counts exactly, W, P and A within
1e-12)."""
import numpy as np
import pytest

from test_gpu_grid import cv  # noqa: F401
from test_gpu_grid_query import GRIDS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,tangent", [("3d", False), ("3d", True), ("2d", False), ("2d", True)])
def test_query_counts(cv, orc, name, tangent):  # noqa: F811
    import torch

    from paper_2211_14318_gb300 import api

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, K = 128 * 8 * sms + 3, 2
    g = GRIDS[name]
    go, gg = orc.Grid(g["n"], g["lo"], g["delta"]), api.GridSpec(g["n"], g["lo"], g["delta"])
    mat = orc.Material(1.0, 0.5, 0.9, 0.3)
    p = api.Params(mu=1.0, lambda_L=0.5, D_inf=0.9, D0=0.3)
    off = api.grid_r11(gg.dim)
    o = cv.grid_convexify(p, gg, 0.06, off, kmax=K, det_rule=1)
    W, forest = o["W"], o["forest"]
    rng = np.random.default_rng(17)
    lo = np.array(g["lo"])
    hi = lo + (np.array(g["n"]) - 1) * np.array(g["delta"])
    F = rng.uniform(lo, hi, size=(n, len(lo)))
    F[::7] = go.points()[rng.integers(0, go.count, F[::7].shape[0])]  # on the grid
    F[::7, 0] += 0.5 * g["delta"][0]  # between two grid points along one component
    F[5::11, -1] += 9.0  # outside
    Fd = torch.from_numpy(F).cuda()
    q = lambda m: [x.cpu().numpy() for x in cv.grid_query(p, gg, 0.06, off, W, forest, Fd[:m], det_rule=1,  # noqa: E731
                                                          K=K, want_A=tangent)]
    full = q(n)
    for m in (1, 3, 4, 5, 8, 9, 8 * sms - 1, 8 * sms, 16 * sms + 1, 32 * sms - 1, 32 * sms, 64 * 8 * sms - 1,
              64 * 8 * sms + 1, 128 * 8 * sms - 1):
        for x, y in zip(q(m), full):
            assert np.array_equal(x, y[:m], equal_nan=True), m
    m = 200
    ref = orc.grid_query(mat, go, 0.06, off, W.cpu().numpy(), forest.cpu().numpy(), F[:m], rule=1, want_A=tangent)
    assert np.array_equal(full[0][:m], ref[0], equal_nan=True)
    assert np.array_equal(full[3][:m], ref[3])
    for x, y in zip(full[1:3] + full[4:], ref[1:3] + ref[4:]):
        x = x[:m]
        y = y.reshape(x.shape)
        assert np.array_equal(np.isnan(x), np.isnan(y))
        f = np.isfinite(y)
        assert np.max(np.abs(x[f] - y[f]) / (1 + np.abs(y[f])), initial=0.0) < 1e-12
