"""The line pass whose lanes share the intervals to be sampled, on both sides of
the line length from which it is taken and with direction counts that leave
lanes without a line: decisions against the FP64 oracle.  Bars as in
test_gpu_parity: bit-exact indices where the oracle's margin exceeds 1e-11,
W^R within 1e-6 relative."""
import numpy as np
import pytest

from test_gpu_parity import MAT, _compare_trees, _omat, _rel, cv  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,na,nb,t_half", [
    (255, 5, 5, 1.0), (257, 2, 2, 1.0), (257, 11, 3, 1.0), (259, 8, 4, 0.2), (333, 19, 15, 0.5),
    (1025, 5, 13, 2.0), (2079, 3, 7, 0.7)])
def test_shared_intervals(cv, orc, L, na, nb, t_half):  # noqa: F811
    from paper_2211_14318_gb300 import api, inputs

    n = 40
    F, Fp = inputs.material_points(n, seed=L + na, lam_hi=2.0)
    m = _omat(orc)
    beta = orc.history_update(m, Fp)
    p = api.Params(n_theta_a=na, n_theta_b=nb, line_points=L, t_half=t_half, depth=2, **MAT)
    out = cv.convexify_points(p, F, beta, want_tree=True)
    tg = api.tree_numpy(out["tree"], n, p.tree_size)
    W, P, to, st = orc.convexify(m, orc.Scan(orc.angle_directions(na, nb), L, t_half, 2), F, beta)
    compared, untied = _compare_trees(orc, api, tg, to, L)
    assert compared > 0
    assert np.max(_rel(out["W_R"].cpu().numpy(), W)) < 1e-6
