"""A step of the global-grid form on value ranges where its FP32 bounds and
truncated comparisons have nothing to say: values and differences outside
FP32's range, straight segments and ties, holes at line ends and inside
edges, offsets in and beyond {-1, 0, 1}, axes too short for an interior
point.  Bit-exact against the oracle's step."""
import numpy as np
import pytest

from test_gpu_grid import cv  # noqa: F401

pytestmark = pytest.mark.gpu

D2 = [(1, 0, 0, 0), (0, 1, 0, 0), (0, 0, 0, 1), (1, -1, -1, 1), (1, 1, 1, 1), (0, 0, 1, -1)]
D2W = D2 + [(2, 0, 0, 0), (0, -3, 0, 0), (2, 4, 1, 2), (-5, 0, 0, 0)]


def _values(kind, n, rng):
    if kind == "huge":
        return rng.normal(size=n) * 10.0 ** rng.integers(30, 300, n)
    if kind == "tiny":
        return rng.normal(size=n) * 10.0 ** -rng.integers(30, 300, n).astype(float)
    if kind == "mixed":
        return rng.normal(size=n) * 10.0 ** rng.integers(-60, 60, n).astype(float)
    if kind == "integers":  # many collinear triples and equal chords, signed zeros
        w = rng.integers(-2, 3, n).astype(float)
        w[rng.random(n) < 0.2] = -0.0
        return w
    if kind == "straight":  # affine along the flat index plus a few last-bit steps
        w = 3.0 + 1e-3 * np.arange(n)
        return np.nextafter(w, np.where(rng.random(n) < 0.5, -np.inf, np.inf))
    if kind == "holes":
        w = rng.normal(size=n)
        w[rng.random(n) < 0.35] = np.nan
        w[rng.random(n) < 0.05] = np.inf
        return w
    raise ValueError(kind)


@pytest.mark.parametrize("shape,dirs", [((9, 4, 5, 11), D2), ((9, 13, 5, 11), D2W), ((2, 2, 40, 1), D2),
                                        ((1, 300, 1, 3), D2W), ((3, 2, 3, 2, 4, 2, 2, 1, 3), None)])
@pytest.mark.parametrize("kind", ["huge", "tiny", "mixed", "integers", "straight", "holes"])
def test_step_is_bit_exact(cv, orc, shape, dirs, kind):  # noqa: F811
    from paper_2211_14318_gb300 import api

    off = api.grid_r11(3) if dirs is None else np.array(dirs, dtype=np.int32)
    lo, de = (0.0,) * len(shape), (0.5,) * len(shape)
    go, gg = orc.Grid(shape, lo, de), api.GridSpec(shape, lo, de)
    W = _values(kind, go.count, np.random.default_rng(len(shape) + len(kind)))
    with np.errstate(over="ignore", invalid="ignore"):
        Wo, d, lm, lp, dec = orc.grid_step(go, off, W)
    Wg, lam, decg = cv.grid_step(gg, off, W)
    lam = lam.cpu().numpy()
    assert np.array_equal(Wg.cpu().numpy(), Wo, equal_nan=True)
    assert np.array_equal(lam[:, 0], d)
    split = d >= 0
    assert np.array_equal(lam[split, 1], lm[split]) and np.array_equal(lam[split, 2], lp[split])
    assert float(decg.cpu()[0]) == dec or not np.isfinite(dec)
