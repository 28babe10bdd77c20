"""The FP64 refinement on nearly affine lines (a narrow window, many samples),
where the pair of the FP32 samples is many samples off and the ends move by
tangent steps and neighbour moves: decisions against the FP64 oracle.  Bars as
in test_gpu_parity: bit-exact indices where the oracle's margin exceeds 1e-11,
W^R within 1e-6 relative everywhere."""
import numpy as np
import pytest

from test_gpu_parity import MAT, _compare_trees, _omat, _rel, cv  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,t_half,mat", [
    (5, 0.01, {}), (33, 0.003, {}), (201, 0.01, dict(D0=2.0)), (1025, 0.01, {}), (2049, 0.02, {}),
    (2049, 0.1, dict(D_inf=0.9, D0=0.3, lambda_L=0.5)), (2079, 0.3, {})])
def test_narrow_windows(cv, orc, L, t_half, mat):  # noqa: F811
    from paper_2211_14318_gb300 import api, inputs

    n = 40
    F, Fp = inputs.material_points(n, seed=L + 1, lam_hi=2.0)
    m = _omat(orc, **mat)
    beta = orc.history_update(m, Fp)
    p = api.Params(n_theta_a=10, n_theta_b=9, line_points=L, t_half=t_half, depth=2,
                   **dict(MAT, **mat))
    out = cv.convexify_points(p, F, beta, want_tree=True)
    tg = api.tree_numpy(out["tree"], n, p.tree_size)
    W, P, to, st = orc.convexify(m, orc.Scan(orc.angle_directions(10, 9), L, t_half, 2), F, beta)
    compared, untied = _compare_trees(orc, api, tg, to, L)
    assert compared > 0
    assert np.max(_rel(out["W_R"].cpu().numpy(), W)) < 1e-6
