"""W^R and P summed over listed leaves: trees of every depth (more than one
chunk of eight nodes), points without a tree, a single point, blocks of one
warp and of four, a batch of problems of different depths -- against the sum
over the returned tree's leaves in FP64 (same energies: 1e-12)."""
import numpy as np
import pytest

from test_gpu_parity import MAT, _omat, cv  # noqa: F401

pytestmark = pytest.mark.gpu


def _sum(orc, m, tree, beta, api):
    n = tree.shape[0]
    W, P = np.zeros(n), np.zeros((n, 4))
    for i in range(n):
        for nd in tree[i]:
            if nd["flags"] & api.NODE_EXISTS and not nd["flags"] & api.NODE_LAMINATED:
                W[i] += nd["weight"] * orc.energy(m, nd["F"], beta[i])
                P[i] += nd["weight"] * np.asarray(orc.stress(m, nd["F"], beta[i]))
    return W, P


@pytest.mark.parametrize("n,depth", [(1, 2), (33, 0), (33, 1), (200, 3), (4865, 2), (65, 5), (40, 8)])
def test_leaf_sums(cv, orc, n, depth):  # noqa: F811
    from paper_2211_14318_gb300 import api, inputs

    F, Fp = inputs.material_points(n, seed=n + depth, lam_hi=2.0)
    m = _omat(orc)
    beta = orc.history_update(m, Fp)
    if n > 8:
        F[3] = (1.0, 0.0, 0.0, -1.0)  # det F < 0: no tree
    p = api.Params(n_theta_a=6, n_theta_b=6, line_points=41, depth=depth, **MAT)
    out = cv.convexify_points(p, F, beta, want_tree=True)
    tree = api.tree_numpy(out["tree"], n, p.tree_size)
    k = min(n, 300)
    W, P = _sum(orc, m, tree[-k:], beta[-k:], api)
    Wg, Pg = out["W_R"].cpu().numpy()[-k:], out["P"].cpu().numpy()[-k:]
    ok = np.isfinite(Wg)
    assert ok.sum() == k - (1 if n > 8 and k == n else 0)
    assert np.max(np.abs(Wg - W)[ok] / (1 + np.abs(W[ok]))) < 1e-12
    assert np.max(np.abs(Pg - P)[ok] / (1 + np.abs(P[ok]))) < 1e-12


def test_leaf_sums_of_a_batch(cv, orc):  # noqa: F811
    """Problems of depths 1, 4 and 2 in one run give each problem's own result."""
    from paper_2211_14318_gb300 import api, inputs

    m = _omat(orc)
    probs = []
    for i, (n, K) in enumerate(((70, 1), (50, 4), (90, 2))):
        F, Fp = inputs.material_points(n, seed=i, lam_hi=2.0)
        probs.append((api.Params(n_theta_a=6, n_theta_b=6, line_points=41, depth=K, **MAT), F,
                      orc.history_update(m, Fp)))
    outs = cv.convexify_batch(probs)
    for (p, F, b), o in zip(probs, outs):
        s = cv.convexify_points(p, F, b)
        assert np.array_equal(o["W_R"].cpu().numpy(), s["W_R"].cpu().numpy())
        assert np.array_equal(o["P"].cpu().numpy(), s["P"].cpu().numpy())
