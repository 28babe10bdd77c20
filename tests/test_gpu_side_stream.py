"""Set-up on a stream of the caller's: direction tables, weights and optimiser
state are in place for the work that follows on that stream while the default
stream is busy, and without it being waited for."""
import numpy as np
import pytest

from test_gpu_parity import MAT, cv  # noqa: F401

pytestmark = pytest.mark.gpu


def test_first_calls_on_a_side_stream(cv):  # noqa: F811
    import torch

    from paper_2211_14318_gb300 import api, inputs

    F, Fp = (torch.from_numpy(x).cuda() for x in inputs.material_points(300, seed=5, lam_hi=2.0))
    p = api.Params(n_theta_a=12, n_theta_b=10, line_points=201, depth=2, **MAT)
    beta = cv.history_update(p, Fp)
    ref = cv.convexify_points(p, F, beta, want_tree=True)
    rng = np.random.default_rng(3)
    X = torch.from_numpy(rng.normal(0.5, 0.4, (1024, 6)).astype(np.float32)).cuda()
    Y = torch.from_numpy(rng.uniform(0, 1, (1024, 7)).astype(np.float32)).cuda()
    log = cv.surrogate_train(X, Y, epochs=2, batch=256, seed=4)
    other = api.Convexifier(0)
    other.convexify_points(api.Params(n_theta_a=5, n_theta_b=5, line_points=33, depth=1, **MAT), F, beta)
    out = dict(W_R=torch.empty_like(ref["W_R"]), P=torch.empty_like(ref["P"]),
               status=torch.empty_like(ref["status"]))
    other.convexify_points(p, F, beta, out=out)  # the workspace at its size
    other.convexify_points(api.Params(n_theta_a=5, n_theta_b=5, line_points=33, depth=1, **MAT), F, beta)
    torch.cuda.synchronize()
    s, done = torch.cuda.Stream(), torch.cuda.Event()
    torch.cuda._sleep(1000000000)  # half a second of the default stream
    done.record()
    with torch.cuda.stream(s):
        o = other.convexify_points(p, F, beta, out=out)  # a new direction table
        s.synchronize()
        assert not done.query()
        W = o["W_R"].cpu().numpy()
        log2 = other.surrogate_train(X, Y, epochs=2, batch=256, seed=4)
    torch.cuda.synchronize()
    other.close()
    np.testing.assert_array_equal(W, ref["W_R"].cpu().numpy())
    # gradients are summed by FP32 additions in any order
    np.testing.assert_allclose(log2, log, rtol=1e-3)
