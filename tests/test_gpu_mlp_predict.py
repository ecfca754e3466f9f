"""The prediction call of the surrogate where its statistics and its workspace can
go wrong: members or inputs that are not finite, calls of several threads on one
handle, sizes around what the workspace keeps; and the handle after an allocation
that failed."""

import threading

import numpy as np
import pytest

from oracle import mlp
from workloads import surrogate as S
from gpu_common import B

pytestmark = pytest.mark.gpu


def _points(n, seed):
    rng = np.random.default_rng(seed)
    return rng.uniform(0.1, 1.0, (n, 4)).astype(np.float32)


def _handle(members, P=None, n=64):
    bd = B()
    h = bd.tdpd_mlp_create(members)
    bd.tdpd_mlp_set_params(h, S.init_params(11, members) if P is None else P)
    X = _points(n, 12)
    bd.tdpd_mlp_set_data(h, X, np.stack([2 + X[:, 0] * X[:, 1], 3 + X[:, 3]], 1).astype(np.float32))
    return h


def _finite_predictions(h, X, members):
    """(mean, spread, each) and the spread the members' outputs give in binary64."""
    mean, spread, each = B().tdpd_mlp_predict(h, X, members)
    e = each.astype(np.float64)
    return mean, spread, each, e.std(0, ddof=1) / np.abs(e.mean(0))


def test_a_nan_prediction_has_a_nan_spread():
    """A caller trusts a point when its spread is small: the spread of a mean that
    is NaN must not be. One input that is NaN touches its own row alone; one
    diverged member (an output bias that is NaN) every row of that output."""
    bd, members = B(), 4
    X = _points(70, 13)
    h = _handle(members)
    try:
        clean = bd.tdpd_mlp_predict(h, X, members)
        Xn = X.copy()
        Xn[33, 2] = np.nan
        mean, spread, each, _ = _finite_predictions(h, Xn, members)
    finally:
        bd.tdpd_mlp_destroy(h)
    assert np.isfinite(clean[1]).all() and (clean[1] > 0).all()
    assert np.isnan(each[:, 33]).all() and np.isnan(mean[33]).all() and np.isnan(spread[33]).all()
    rest = np.arange(70) != 33
    for a, b in zip((mean, spread), clean[:2]):
        assert np.array_equal(a[rest], b[rest])

    P = S.init_params(11, members)
    P[2, -1] = np.nan                       # the bias of the second output
    h = _handle(members, P)
    try:
        mean, spread, each, want = _finite_predictions(h, X, members)
    finally:
        bd.tdpd_mlp_destroy(h)
    assert np.isnan(mean[:, 1]).all() and np.isnan(spread[:, 1]).all()
    assert np.isfinite(mean[:, 0]).all()
    # the members' outputs are rounded to binary32 here: 2^-24 of the mean against
    # a spread of per cents
    assert np.abs(spread[:, 0] - want[:, 0]).max() < 1e-6


def test_threads_share_a_handle():
    """Calls of several threads on one handle (as before the handle kept its
    workspace), the sizes on both sides of what comes with it."""
    bd, members = B(), 2
    h = _handle(members)
    sets = [_points(n, 20 + n) for n in (300, 5462, 1000, 9000, 301, 20000, 5463, 2048)]
    right = []

    def work(k):
        for _ in range(40):
            got = bd.tdpd_mlp_predict(h, sets[k], members)
            right.append(all(np.array_equal(a, b) for a, b in zip(got, want[k])))

    try:
        want = []
        for X in sets:
            g = _handle(members)
            want.append(bd.tdpd_mlp_predict(g, X, members))
            bd.tdpd_mlp_destroy(g)
        threads = [threading.Thread(target=work, args=(k,)) for k in range(len(sets))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    finally:
        bd.tdpd_mlp_destroy(h)
    assert len(right) == 40 * len(sets) and all(right)


def test_samples_that_do_not_fit_leave_a_usable_handle():
    """Two thousand million samples with 64 members need 18 TB of gradient rows: the
    allocation fails before the samples are read. Training then has no data (a status,
    no launch), prediction keeps the standardisation it had, and a set that fits trains
    as on a new handle."""
    bd, members = B(), 64
    h, g = _handle(members), _handle(members)
    X = _points(50, 14)
    Y = np.stack([2 + X[:, 1], 3 + X[:, 2] * X[:, 3]], 1).astype(np.float32)
    try:
        before = bd.tdpd_mlp_predict(h, X, members)
        assert bd.STATUS[bd.lib.tdpd_mlp_set_data(h, 2_000_000_000, bd._ptr(X), bd._ptr(Y))] == 'ENOMEM'
        for call in (lambda: bd.tdpd_mlp_train(h, 1, 1e-3, members), lambda: bd.tdpd_mlp_loss_grad(h, members)):
            with pytest.raises(bd.TdpdError) as e:
                call()
            assert bd.STATUS[e.value.status] == 'ESTATE'
        for a, b in zip(before, bd.tdpd_mlp_predict(h, X, members)):
            assert np.array_equal(a, b)
        for x in (h, g):
            bd.tdpd_mlp_set_data(x, X, Y)
        for a, b in zip(bd.tdpd_mlp_loss_grad(h, members), bd.tdpd_mlp_loss_grad(g, members)):
            assert np.array_equal(a, b)
    finally:
        bd.tdpd_mlp_destroy(h)
        bd.tdpd_mlp_destroy(g)


def test_prediction_sizes_around_the_workspace():
    """Two members take 12 floats a point: the largest call that fits what comes with
    the handle (65,536 floats) and the first that does not, the largest kept (2^22) and
    the first that allocates for itself; then small calls. Against the oracle (1e-6 of
    the outputs' magnitude, the rounding of sums of 64 binary32 products)."""
    bd, members = B(), 2
    h = _handle(members)
    P, X0 = S.init_params(11, members), _points(64, 12).astype(np.float64)
    st = mlp.Standardizer(X0, np.stack([2 + X0[:, 0] * X0[:, 1], 3 + X0[:, 3]], 1).astype(np.float32).astype(np.float64))
    try:
        for n in (5461, 5462, 349525, 349526, 31, 5463):
            X = _points(n, n)
            mean, spread, each, want = _finite_predictions(h, X, members)
            at = np.unique(np.r_[0:min(n, 500), max(0, n - 500):n])
            Xn = st.x(X[at].astype(np.float64)).astype(np.float32).astype(np.float64)
            for k in range(members):
                y = st.y_inv(mlp.forward(P[k], Xn)[0])
                assert np.abs(each[k][at] - y).max() < 1e-6 * np.abs(y).max(), (n, k)
            assert np.abs(mean - each.astype(np.float64).mean(0)).max() < 1e-6 * np.abs(mean).max(), n
            assert np.abs(spread - want).max() < 1e-6, n
    finally:
        bd.tdpd_mlp_destroy(h)


def test_a_call_that_does_not_fit_the_device():
    """Two thousand million points with 64 members need 1.1 TB: refused before the
    points are read, and the next call is as before."""
    bd, members = B(), 64
    h = _handle(members)
    X = _points(50, 15)
    mean = np.zeros((50, 2), np.float32)
    try:
        before = bd.tdpd_mlp_predict(h, X, members)
        rc = bd.lib.tdpd_mlp_predict(h, 2_000_000_000, bd._ptr(X), bd._ptr(mean), None, None)
        assert bd.STATUS[rc] == 'ENOMEM'
        for a, b in zip(before, bd.tdpd_mlp_predict(h, X, members)):
            assert np.array_equal(a, b)
    finally:
        bd.tdpd_mlp_destroy(h)
