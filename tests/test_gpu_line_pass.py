"""The lane's line pass that samples only the intervals which can hold a
side's minimum: decisions against the FP64 oracle at the line lengths where
its intervals are degenerate (no whole pair, one interval, a last sample of
its own, 32 intervals) and on lines that run through det F = 0.  Bars as in
test_gpu_parity: bit-exact indices where the oracle's margin exceeds 1e-11,
W^R within 1e-6 and P within 1e-5 relative."""
import numpy as np
import pytest

from test_gpu_parity import MAT, _compare_trees, _omat, _rel, cv  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,t_half,mat", [
    (3, 0.5, {}), (5, 0.5, {}), (7, 0.5, {}), (9, 1.5, {}), (11, 0.5, {}), (13, 4.0, {}),
    (65, 0.5, {}), (67, 2.5, {}), (131, 0.5, dict(D_inf=0.9, D0=0.3, lambda_L=0.5)),
    (203, 4.0, {}), (513, 0.05, {}), (1031, 0.5, dict(D0=2.0)), (2079, 1.0, {}),
    (2077, 10.0, dict(D_inf=0.9, D0=0.3, lambda_L=0.5))])
def test_line_pass_edges(cv, orc, L, t_half, mat):  # noqa: F811
    from paper_2211_14318_gb300 import api, inputs

    n = 48
    F, Fp = inputs.material_points(n, seed=L, lam_hi=2.0)
    m = _omat(orc, **mat)
    beta = orc.history_update(m, Fp)
    beta[::7] = 0.0
    p = api.Params(n_theta_a=12, n_theta_b=10, line_points=L, t_half=t_half, depth=2,
                   **dict(MAT, **mat))
    out = cv.convexify_points(p, F, beta, want_tree=True)
    tg = api.tree_numpy(out["tree"], n, p.tree_size)
    W, P, to, st = orc.convexify(m, orc.Scan(orc.angle_directions(12, 10), L, t_half, 2), F, beta)
    compared, untied = _compare_trees(orc, api, tg, to, L)
    assert compared >= n // 2 and untied.sum() >= n // 2
    assert np.max(_rel(out["W_R"].cpu().numpy(), W)[untied]) < 1e-6
    dP = np.linalg.norm(out["P"].cpu().numpy() - P, axis=1) / (1e-8 + np.linalg.norm(P, axis=1))
    assert np.max(dP[untied]) < 1e-5
