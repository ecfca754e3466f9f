"""The surrogate's kernels at the edges of their tiles (chunks of 32 samples,
the reduction's groups of eight chunks), against the FP64 oracle.

Tolerances: binary32 sums of at most 64 products in a layer and of n samples in
a gradient (float-float beyond 32 of them) carry a few 2^-24 of the sum of the
magnitudes, which is at most about ten times the result's norm: 1e-5 normwise,
as for the whole-chunk sizes; predictions 1e-6 of the outputs' magnitude."""

import numpy as np
import pytest

from oracle import mlp
from workloads import surrogate as S
from gpu_common import B, normwise

pytestmark = pytest.mark.gpu


def _data(n, seed):
    rng = np.random.default_rng(seed)
    X = rng.uniform(0.1, 1.0, (n, 4)).astype(np.float32)
    Y = np.stack([2 + X[:, 0] * X[:, 1], 3 + np.sin(3 * X[:, 2]) + X[:, 3]], 1).astype(np.float32)
    return X, Y


@pytest.mark.parametrize('n, members', [(2, 1), (31, 2), (32, 1), (33, 64), (255, 3), (257, 1), (4097, 2)])
def test_gradient_and_prediction_at_chunk_edges(n, members):
    bd = B()
    P = S.init_params(40 + n, members)
    X, Y = _data(n, n)
    Xt, _ = _data(n + 1, 7 * n)
    h = bd.tdpd_mlp_create(members)
    try:
        bd.tdpd_mlp_set_params(h, P)
        bd.tdpd_mlp_set_data(h, X, Y)
        loss, grad = bd.tdpd_mlp_loss_grad(h, members)
        again = bd.tdpd_mlp_loss_grad(h, members)[1]
        mean, spread, each = bd.tdpd_mlp_predict(h, Xt, members)
    finally:
        bd.tdpd_mlp_destroy(h)
    assert np.array_equal(grad, again)
    st = mlp.Standardizer(X.astype(np.float64), Y.astype(np.float64))
    Xn, Yn, Tn = (a.astype(np.float32).astype(np.float64) for a in
                  (st.x(X.astype(np.float64)), st.y(Y.astype(np.float64)), st.x(Xt.astype(np.float64))))
    for k in range(members):
        lo, go = mlp.loss_grad(P[k], Xn, Yn)
        assert loss[k] == pytest.approx(lo, rel=1e-5)
        assert normwise(grad[k], go) < 1e-5, k
        y = st.y_inv(mlp.forward(P[k], Tn)[0])
        assert np.abs(each[k] - y).max() < 1e-6 * np.abs(y).max(), k
    assert np.abs(mean - each.astype(np.float64).mean(0)).max() < 1e-6 * np.abs(mean).max()
    assert (spread == 0).all() if members == 1 else (spread > 0).any()


def test_gradient_above_the_rows_of_one_chunk_each():
    """Above 8,192 chunks a row of the chunk sums holds four of them; then fewer
    samples, which take more rows, in the same allocation."""
    bd = B()
    P = S.init_params(77, 1)
    h = bd.tdpd_mlp_create(1)
    try:
        bd.tdpd_mlp_set_params(h, P)
        for n in (32 * 8192 + 33, 32 * 8192):
            X, Y = _data(n, n)
            bd.tdpd_mlp_set_data(h, X, Y)
            loss, grad = bd.tdpd_mlp_loss_grad(h, 1)
            st = mlp.Standardizer(X.astype(np.float64), Y.astype(np.float64))
            lo, go = mlp.loss_grad(P[0], *(a.astype(np.float32).astype(np.float64) for a in
                                           (st.x(X.astype(np.float64)), st.y(Y.astype(np.float64)))))
            assert loss[0] == pytest.approx(lo, rel=1e-5)
            assert normwise(grad[0], go) < 1e-5
    finally:
        bd.tdpd_mlp_destroy(h)
