"""Line passes on both sides of the lengths from which a warp's lanes share their
intervals, with fixed and with doubled windows, and in a batch of both: decisions
against the FP64 oracle.  Bars as in test_gpu_parity: bit-exact indices where the
oracle's margin exceeds 1e-11, W^R within 1e-6 relative."""
import numpy as np
import pytest

from test_gpu_parity import MAT, _compare_trees, _omat, _rel, cv  # noqa: F401

pytestmark = pytest.mark.gpu


def _case(orc, L, doublings, n=30, na=9, nb=7):
    from paper_2211_14318_gb300 import api, inputs

    F, Fp = inputs.material_points(n, seed=L + doublings, lam_hi=2.0)
    m = _omat(orc)
    beta = orc.history_update(m, Fp)
    p = api.Params(n_theta_a=na, n_theta_b=nb, line_points=L, t_half=0.5, depth=2,
                   window_doublings=doublings, **MAT)
    sc = orc.Scan(orc.angle_directions(na, nb), L, 0.5, 2, adaptive=doublings)
    return p, F, beta, orc.convexify(m, sc, F, beta)


@pytest.mark.parametrize("L,doublings", [(399, 0), (401, 0), (405, 0), (255, 3), (257, 3), (259, 1),
                                         (333, 3), (513, 2), (769, 2)])
def test_both_sides_of_the_rule(cv, orc, L, doublings):  # noqa: F811
    from paper_2211_14318_gb300 import api

    p, F, beta, (W, P, to, st) = _case(orc, L, doublings)
    out = cv.convexify_points(p, F, beta, want_tree=True)
    tg = api.tree_numpy(out["tree"], F.shape[0], p.tree_size)
    compared, untied = _compare_trees(orc, api, tg, to, L)
    assert compared > 0
    assert np.max(_rel(out["W_R"].cpu().numpy(), W)) < 1e-6


def test_batch_of_fixed_and_doubled_windows(cv, orc):  # noqa: F811
    import torch

    cases = [_case(orc, 333, 0), _case(orc, 265, 2), _case(orc, 129, 1)]
    outs = cv.convexify_batch([(p, torch.from_numpy(F).cuda(), torch.from_numpy(b).cuda())
                               for p, F, b, _ in cases])
    for o, (_, _, _, (W, P, to, st)) in zip(outs, cases):
        assert np.max(_rel(o["W_R"].cpu().numpy(), W)) < 1e-6
