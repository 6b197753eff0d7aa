"""The accurate mode where magnitudes differ widely inside one matrix: every row and every column of a gradient keeps its own
accuracy, whatever the others are.  Errors are measured row by row and column by column, against the sums of the magnitudes of
the terms of that row or column (what rounding errors are proportional to)."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from paper_1911_05181_b200 import binding as ul
from helpers import TOL, GpuNet, dev

pytestmark = pytest.mark.gpu


def _gradient(Ws, bs, X, labels=None, T=None):
    sizes = [Ws[0].shape[1]] + [w.shape[0] for w in Ws]
    g = GpuNet(sizes, ul.MATH_3XTF32, X.shape[0]); g.set_params(Ws, bs)
    if T is None:
        return g.gradient(X, labels)
    g.net.gradient_sse(g.W, g.b, dev(X), sizes[0], dev(T), sizes[-1], X.shape[0], False, g.dW, g.db, g.loss)
    torch.cuda.synchronize()
    return float(g.loss.item()), [t.cpu().numpy() for t in g.dW], [t.cpu().numpy() for t in g.db]


def _worst(got, ref, mag, skip=0.0):
    """Largest error of a row or column, relative to its magnitude sums; rows and columns of nothing but zeros are left out."""
    if got.ndim == 1:
        got, ref, mag = got[:, None], ref[:, None], mag[:, None]
        axes = (1,)
    else:
        axes = (1, 0)
    worst = 0.0
    for ax in axes:
        e = np.sqrt(((got.astype(np.float64) - ref) ** 2).sum(axis=ax))
        m = np.sqrt((mag ** 2).sum(axis=ax))
        worst = max(worst, float((e[m > skip] / m[m > skip]).max()))
    return worst


def _check(Ws, bs, X, labels=None, T=None, tol=TOL[ul.MATH_3XTF32]):
    loss, dW, db = _gradient(Ws, bs, X, labels, T)
    want = oracle.mlp_gradient(Ws, bs, X, labels) if T is None else oracle.mlp_sse_gradient(Ws, bs, X, T)
    mag = oracle.mlp_gradient_abs(Ws, bs, X, labels=labels, T=T)
    assert abs(loss - want[0]) <= 1e-5 * abs(want[0])
    errors = {"%s[%d]" % (name, l): _worst(g, r, m) for name, gs, rs, ms in (("dW", dW, want[1], mag[0]), ("db", db, want[2], mag[1]))
              for l, (g, r, m) in enumerate(zip(gs, rs, ms))}
    assert max(errors.values()) <= tol, errors


def _net(seed, sizes):
    Ws, bs = si.mlp_params(seed, sizes)
    return Ws, [(0.2 * si.uniform_pm1(seed, 11 + i, b.size)).astype(np.float32) for i, b in enumerate(bs)]


# A unit whose weights and bias are all tiny (its activations are, too: a column of the next gradient), a unit whose outgoing
# weights are (a row of the gradient before it), a row of output weights, and one weight far above the others.
@pytest.mark.parametrize("form", ["unit", "outgoing", "row", "outlier"])
@pytest.mark.parametrize("factor", [2.0 ** -12, 2.0 ** -24, 2.0 ** -36])
@pytest.mark.parametrize("head", ["softmax", "sse"])
def test_units_and_weights_of_their_own_magnitude(form, factor, head):
    sizes, n = [40, 48, 20], 200
    Ws, bs = _net(51, sizes)
    f = np.float32(factor)
    if form == "unit": Ws[0][7] *= f; bs[0][7] *= f
    if form == "outgoing": Ws[1][:, 7] *= f
    if form == "row": Ws[1][7] *= f; bs[1][7] *= f
    if form == "outlier": Ws[1][7, 9] = np.float32(min(2.0 ** 20, 1.0 / factor))
    X, y = si.mlp_batch(51, sizes, n)
    T = si.mlp_targets(51, sizes, n, 0, False) if head == "sse" else None
    _check(Ws, bs, X, labels=None if T is not None else y, T=T)


@pytest.mark.parametrize("factor", [2.0 ** -12, 2.0 ** -24])
def test_a_tiny_unit_between_two_hidden_layers(factor):
    sizes, n = [40, 48, 36, 20], 200
    Ws, bs = _net(52, sizes)
    f = np.float32(factor)
    Ws[1][7] *= f; bs[1][7] *= f            # layer 2: a small row of W_1, small activations
    Ws[0][9] *= f; bs[0][9] *= f            # layer 1
    X, y = si.mlp_batch(52, sizes, n)
    _check(Ws, bs, X, labels=y)


# One target far above the others: the other patterns keep their deltas and the other classes their rows.  The pattern's first
# inputs are zero, so that the gradient's columns there do not see it at all.
@pytest.mark.parametrize("sizes", [[40, 48, 20], [40, 48, 36, 20], [40, 48, 36, 1100]])
@pytest.mark.parametrize("target", [1e6, 1e8, 1e10, 1e12, 1e15])
def test_a_target_far_above_the_others(target, sizes):
    n = 150
    Ws, bs = _net(53, sizes)
    X, _ = si.mlp_batch(53, sizes, n)
    X[7, :10] = 0
    T = si.mlp_targets(53, sizes, n, 0, False)
    T[7, 2] = np.float32(target)
    _check(Ws, bs, X, T=T)


# Output units whose deltas are all small (targets reached to 2^-20), and a hidden layer whose outgoing weights differ
@pytest.mark.parametrize("scale", [2.0 ** -16, 2.0 ** -30])
def test_classes_and_hidden_units_with_small_deltas(scale):
    sizes, n = [40, 48, 36, 20], 300
    Ws, bs = _net(54, sizes)
    X, _ = si.mlp_batch(54, sizes, n)
    Ws[2][:, 5] *= np.float32(scale)            # deltas of unit 5 of layer 2
    T = si.mlp_targets(54, sizes, n, 0, False)
    _check(Ws, bs, X, T=T)


# Classes that the softmax hardly ever predicts and that are nobody's label: their rows are sums of tiny probabilities
# (few and many patterns: the classes are looked for in one launch or in one of their own)
@pytest.mark.parametrize("sizes,n", [([40, 48, 24], 200), ([40, 48, 36, 24], 200), ([24, 40, 12300], 40), ([24, 40, 12300], 180), ([40, 64, 1100], 700),
                                     ([12, 20, 43], 4100), ([12, 16, 65600], 40)])
@pytest.mark.parametrize("log10_p", [-5, -9, -11, -13, -25])
def test_classes_that_are_hardly_ever_predicted(sizes, n, log10_p):
    Ws, bs = _net(55, sizes)
    rare = np.arange(1, sizes[-1], 5)
    bs[-1][rare] += np.float32(log10_p * np.log(10.0))
    X, y = si.mlp_batch(55, sizes, n)
    y = np.where(np.isin(y, rare), 0, y).astype(np.int32)
    _check(Ws, bs, X, labels=y)
