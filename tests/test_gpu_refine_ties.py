"""The FP64 refinement on lines whose samples lie within rounding of their chord
(very narrow windows): no candidate takes more FP64 samples than a pass over its
line and a half (128 at least), plus one further chord's; and lines searched by
the whole warp.  Decisions of the points that the library calls certified
against every direction (in windows this narrow more directions than the 16
kept can lie within the FP32 error of the best) against the FP64 oracle, bars as
in test_gpu_parity: bit-exact indices where the oracle's margin exceeds 1e-11,
W^R within 1e-6 relative."""
import numpy as np
import pytest

from test_gpu_parity import MAT, _compare_trees, _omat, _rel, cv  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,t_half,n", [(3, 1e-6, 40), (33, 1e-8, 400), (33, 1e-4, 400), (201, 1e-8, 400),
                                        (255, 1e-5, 40), (1025, 1e-6, 40), (1027, 1e-2, 400), (2079, 1e-3, 40)])
def test_samples_within_rounding_of_the_chord(cv, orc, L, t_half, n):  # noqa: F811
    from paper_2211_14318_gb300 import api, inputs

    F, Fp = inputs.material_points(n, seed=L, lam_hi=2.0)
    m = _omat(orc)
    beta = orc.history_update(m, Fp)
    p = api.Params(n_theta_a=10, n_theta_b=9, line_points=L, t_half=t_half, depth=2, **MAT)
    cv.stats(reset=True)
    out = cv.convexify_points(p, F, beta, want_tree=True)
    s = cv.stats()
    assert s["refined"] > 0
    assert s["fp64_checks"] <= s["refined"] * (max(L, 128) / 2 + L + 4)
    tg = api.tree_numpy(out["tree"], n, p.tree_size)
    W, P, to, st = orc.convexify(m, orc.Scan(orc.angle_directions(10, 9), L, t_half, 2), F, beta)
    sure = (out["status"].cpu().numpy() & api.PT_OVERFLOW) == 0
    if t_half > 1e-3:
        assert sure.any()
    _compare_trees(orc, api, tg[sure], to[sure], L)
    assert np.max(_rel(out["W_R"].cpu().numpy(), W)[sure], initial=0.0) < 1e-6
