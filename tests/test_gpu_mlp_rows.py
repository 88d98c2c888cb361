"""The network's pass at row counts around its 64-row tiles, its slices of the weight gradients (one per 64 rows, 24 at
most) and their remainders, element by element against the oracle with the same roundings to BF16.

Bound: five values in the chain of an element (x or a, a, dy, dz, dz) are rounded to BF16, and each can fall to the other
side where the sums before it differ in FP32, 2^-8 each: 0.02 of the root of the sum of its squared terms (and of that
root's mean over the matrix, for elements whose terms happen to be small).  A dropped remainder of one row in
a thousand is 0.03 of it on average, of one 64-row stage 0.25."""
import numpy as np
import pytest

from oracle import mlp as om

pytestmark = pytest.mark.gpu


def _inputs(rows, seed):
    rng = np.random.default_rng(seed)
    X = rng.uniform(0.0, 1.0, (rows, om.DIN)).astype(np.float32)
    T = (0.3 * rng.standard_normal((rows, om.DOUT))).astype(np.float32)
    M = (rng.uniform(size=(rows, om.DOUT)) < 0.7).astype(np.float32)
    M[:, 0] = 1.0
    return X, T, M


def _terms(p, X, T, M):
    """Root of the sum over the rows of the squared terms of every gradient element, in the parameters' order."""
    r = om.bf16
    W1, b1, W2, b2, W3, b3 = om.unpack(p)
    Xb = r(X)
    Z1 = Xb @ r(W1) + b1
    A1 = r(om.silu(Z1))
    Z2 = A1 @ r(W2) + b2
    A2 = r(om.silu(Z2))
    dY = np.zeros((len(X), om.DOUT_PAD))
    dY[:, :om.DOUT] = 2.0 * M * ((A2 @ r(W3) + b3)[:, :om.DOUT] - T) / M.sum()
    dZ2 = r(r(dY) @ r(W3).T * om.dsilu(Z2))
    dZ1 = r(dZ2 @ r(W2).T * om.dsilu(Z1))
    out = []
    for a, d in ((Xb, dZ1), (A1, dZ2), (A2, r(dY))):
        out += [np.sqrt((a ** 2).T @ d ** 2), np.sqrt((d ** 2).sum(0))]
    return out


def _compare(net, p, rows, seed):
    X, T, M = _inputs(rows, seed)
    loss, grad = net.loss_grad(X, T, M)
    X, T, M = (a.astype(np.float64) for a in (X, T, M))
    lr, gr = om.loss_grad(p, X, T, M)
    assert abs(loss - lr) <= 1e-3 * lr
    at = 0
    for s in _terms(p, X, T, M):
        d = np.abs(grad[at:at + s.size].reshape(s.shape) - gr[at:at + s.size].reshape(s.shape))
        at += s.size
        assert (d <= 0.02 * (s + s.mean())).all(), (rows, s.shape, float((d / (s + s.mean())).max()))
    return grad


def _net(mess):
    p = om.random_params(7).astype(np.float32)
    net = mess.MLP(seed=1)
    net.set_params(p)
    return net, p.astype(np.float64)


@pytest.mark.parametrize("rows", [1, 36, 63, 64, 65, 127, 128, 129, 1000, 1535, 1537, 2048, 8191])
def test_rows(mess, rows):
    net, p = _net(mess)
    _compare(net, p, rows, rows)


def test_fewer_rows_after_more(mess):
    """One network with 36, 4096 and 36 rows: the kept buffers of the large pass leave no trace in the small one."""
    net, p = _net(mess)
    first = _compare(net, p, 36, 1)
    _compare(net, p, 4096, 2)
    assert np.array_equal(_compare(net, p, 36, 1), first)
