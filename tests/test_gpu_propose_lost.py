"""A proposal call whose network inference gave up (its error word is set: here
by hand, as a run-out wait would) takes the full scan instead of stale
proposals, and leaves no error behind for a later call."""
import ctypes
import subprocess

import numpy as np
import pytest

from oracle import mlp
from paper_2211_14318_gb300 import build as b
from test_gpu_parity import cv  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SRC = r"""
#include "cvx_handle.h"
#include "cvx_surrogate.h"
extern "C" int set_word(cvx_handle *h, int v) {
    return (int)cudaMemcpy(h->sur->err, &v, sizeof v, cudaMemcpyHostToDevice);
}
extern "C" int get_word(cvx_handle *h) {
    int v = -1;
    return cudaMemcpy(&v, h->sur->err, sizeof v, cudaMemcpyDeviceToHost) == cudaSuccess ? v : -1;
}
"""


@pytest.fixture(scope="module")
def word(tmp_path_factory):
    d = tmp_path_factory.mktemp("word")
    (d / "w.cu").write_text(SRC)
    subprocess.run([b.nvcc(), "-std=c++17", *b.ARCH, "-Xcompiler", "-fPIC", "-I", b.CSRC, "-I", b.INCLUDE,
                    "-shared", "-cudart", "static", "-o", str(d / "w.so"), str(d / "w.cu")], check=True)
    L = ctypes.CDLL(str(d / "w.so"))
    L.set_word.argtypes = [ctypes.c_void_p, ctypes.c_int]
    L.get_word.argtypes = [ctypes.c_void_p]
    return L


@pytest.mark.parametrize("kw", [{}, dict(recentre=3, mirror=True), dict(gap_one_sided=True)])
def test_lost_inference_takes_the_full_scan(cv, word, kw):
    import torch

    from paper_2211_14318_gb300 import api, inputs

    n = 200
    F, Fp = inputs.material_points(n, seed=12, lam_hi=2.0)
    p = api.Params(n_theta_a=16, n_theta_b=16, line_points=201, depth=2, **kw)
    beta = cv.history_update(p, Fp)
    cv.surrogate_set_weights(mlp.init_params(4), np.array([1.2, 0, 0, 1, 0.3, 0.2]), np.full(6, 0.4))
    full = cv.convexify_points(p, F, beta, want_tree=True)
    good = cv.surrogate_propose(p, F, beta, window=2, gap_tol=1e30)
    assert not good["fell_back"].cpu().numpy().all()  # the windows alone decide some points
    assert word.set_word(cv._h, 1) == 0
    lost = cv.surrogate_propose(p, F, beta, window=2, gap_tol=1e30, want_tree=True)
    torch.cuda.synchronize()
    assert word.get_word(cv._h) == 0
    assert lost["fell_back"].cpu().numpy().all()
    for k in ("W_R", "P"):  # the same FP64 operations on the same decisions
        np.testing.assert_array_equal(lost[k].cpu().numpy(), full[k].cpu().numpy())
    a, c = (api.tree_numpy(o["tree"], n, p.tree_size) for o in (lost, full))
    for k in ("dir", "m_minus", "m_plus"):
        np.testing.assert_array_equal(a[k], c[k])
    cv.surrogate_forward(np.ones((4, 6), np.float32))  # no error of the call before
    again = cv.surrogate_propose(p, F, beta, window=2, gap_tol=1e30)
    np.testing.assert_array_equal(again["fell_back"].cpu().numpy(), good["fell_back"].cpu().numpy())
