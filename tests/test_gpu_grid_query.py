"""The tabulated trees of the global-grid query (one record per grid point in
two buffers, groups of lanes per point and query): both dimensions, with and
without the tangent, every energy, grids and query counts that leave partial
blocks, no iteration, and records no iteration wrote.  W_interp bit for bit,
leaf counts exactly, W, P and A within 1e-12 of the oracle (both sides sum
the same terms in FP64; leaf energies use each side's log and exp)."""
import numpy as np
import pytest

from test_gpu_grid import cv  # noqa: F401

pytestmark = pytest.mark.gpu

GRIDS = {
    "2d": dict(n=(7, 5, 6, 9), lo=(0.4, -0.45, -0.6, 0.4), delta=(0.2, 0.22, 0.25, 0.18)),
    "2d_line": dict(n=(13, 1, 1, 5), lo=(-1.5, 0.0, 0.0, 0.5), delta=(0.25, 0.2, 0.2, 0.25)),
    "3d": dict(n=(3, 2, 2, 2, 3, 2, 2, 2, 3), lo=(1.0, -0.1, -0.1, -0.1, 1.0, -0.1, -0.1, -0.1, 1.0),
               delta=(0.4, 0.2, 0.2, 0.2, 0.4, 0.2, 0.2, 0.2, 0.4)),
}


def _run(cv, orc, name, energy, n, K, tangent):
    from paper_2211_14318_gb300 import api

    g = GRIDS[name]
    go, gg = orc.Grid(g["n"], g["lo"], g["delta"]), api.GridSpec(g["n"], g["lo"], g["delta"])
    mat = orc.Material(1.0, 0.5, 0.9, 0.3, energy=energy)
    p = api.Params(mu=1.0, lambda_L=0.5, D_inf=0.9, D0=0.3, energy=energy)
    off = api.grid_r11(gg.dim)
    W = orc.grid_energy(mat, go, 0.06, rule=1)
    forest = []
    for _ in range(K):
        W, d, lm, lp, _ = orc.grid_step(go, off, W)
        forest.append(np.stack([d, lm, lp], axis=1))
    forest = np.array(forest, dtype=np.int32).reshape(K, go.count, 3)
    rng = np.random.default_rng(n + K)
    lo = np.array(g["lo"])
    hi = lo + (np.array(g["n"]) - 1) * np.array(g["delta"])
    F = rng.uniform(lo, hi, size=(n, len(lo)))
    F[n // 2:n // 2 + n // 4] = go.points()[rng.integers(0, go.count, n // 4)]
    F[-(n // 8):] += 5.0 * (n >= 8)
    o = orc.grid_query(mat, go, 0.06, off, W, forest, F, rule=1, want_A=tangent)
    d = cv.grid_query(p, gg, 0.06, off, W, forest, F, det_rule=1, K=K, want_A=tangent)
    return o, [x.cpu().numpy() for x in d], (p, gg, off, W, F)


@pytest.mark.parametrize("name,energy,n,K,tangent", [
    ("2d", 0, 1, 2, True), ("2d", 0, 127, 3, True), ("2d", 0, 129, 3, False), ("2d", 2, 300, 4, True),
    ("2d", 0, 64, 0, True), ("2d_line", 1, 200, 2, True), ("2d_line", 1, 33, 2, False),
    ("3d", 0, 130, 2, True), ("3d", 2, 65, 2, True), ("3d", 0, 257, 1, False)])
def test_query_tables(cv, orc, name, energy, n, K, tangent):  # noqa: F811
    o, d, _ = _run(cv, orc, name, energy, n, K, tangent)
    assert np.array_equal(d[0], o[0], equal_nan=True)
    assert np.array_equal(d[3], o[3])
    for x, y in zip(d[1:3] + d[4:], o[1:3] + o[4:]):
        y = y.reshape(x.shape)
        assert np.array_equal(np.isnan(x), np.isnan(y))
        f = np.isfinite(y)
        assert np.max(np.abs(x[f] - y[f]) / (1 + np.abs(y[f])), initial=0.0) < 1e-12


@pytest.mark.parametrize("tangent", [False, True])
def test_foreign_records_make_leaves(cv, orc, tangent):  # noqa: F811
    """A record with a direction or ends no iteration writes: the point is a
    leaf at that order, as with no iteration at all."""
    _, d, (p, gg, off, W, F) = _run(cv, orc, "2d", 0, 150, 0, tangent)
    bad = np.zeros((2, gg.count, 3), dtype=np.int32)
    bad[0] = (1, -1, 1)
    bad[0, ::2] = -1
    bad[1, :, 0] = off.shape[0]
    bad[1, ::3] = (0, 1, 2)
    bad[1, 1::3] = (0, -4000, 4000)
    e = [x.cpu().numpy() for x in cv.grid_query(p, gg, 0.06, off, W, bad, F, det_rule=1,
                                                want_A=tangent)]
    for x, y in zip(e, d):
        assert np.array_equal(x, y, equal_nan=True)
