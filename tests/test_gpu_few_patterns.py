"""Kernels whose shape follows the number of patterns: softmax deltas with one, two or four warps for a pattern, row statistics of forward calls, on
either side of where the choice changes."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from paper_1911_05181_b200 import binding as ul
from helpers import TOL, GpuNet, dev, tolerance_at

pytestmark = pytest.mark.gpu

# patterns: blocks of eight, four warps each up to 148 blocks, two up to 296; classes: one step of 256 per warp and one more or less
@pytest.mark.parametrize("math", [ul.MATH_3XTF32, ul.MATH_TF32, ul.MATH_BF16])
@pytest.mark.parametrize("n", [1, 7, 1184, 1185, 2368, 2369])
@pytest.mark.parametrize("classes", [256, 257, 513, 1281])
def test_softmax_head(math, n, classes):
    sizes = [21, 40, classes]
    Ws, bs = si.mlp_params(11, sizes)
    X, y = si.mlp_batch(11, sizes, n)
    want = oracle.mlp_gradient(Ws, bs, X, y)
    cond = oracle.gradient_condition(Ws, bs, X, labels=y)
    g = GpuNet(sizes, math, n); g.set_params(Ws, bs)
    loss, dW, db = g.gradient(X, y)
    assert abs(loss - want[0]) <= TOL[math] * abs(want[0])
    for a, ref, k in zip(dW + db, want[1] + want[2], cond[0] + cond[1]):
        assert oracle.rel_l2(a, ref) <= tolerance_at(math, k)
    # the error alone: other kernels, sums of the same terms (double) over 32-bit sums of exponentials that are the same
    assert abs(g.forward_loss(X, y) - loss) <= 1e-9 * abs(loss)


# a run of 1,024 patterns adds them up sixteen at a time
@pytest.mark.parametrize("math", [ul.MATH_3XTF32, ul.MATH_TF32, ul.MATH_FP32_SIMT])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 1023, 1024, 1025, 1041])
def test_bias_gradient_without_a_hidden_layer(math, n):
    sizes = [21, 131]
    Ws, bs = si.mlp_params(12, sizes)
    X, y = si.mlp_batch(12, sizes, n)
    want = oracle.mlp_gradient(Ws, bs, X, y)
    cond = oracle.gradient_condition(Ws, bs, X, labels=y)
    g = GpuNet(sizes, math, n); g.set_params(Ws, bs)
    _, _, db = g.gradient(X, y)
    assert oracle.rel_l2(db[0], want[2][0]) <= tolerance_at(math, cond[1][0])


@pytest.mark.parametrize("count", [1, 3, 4, 5, 1027, 4096])
@pytest.mark.parametrize("off", [0, 1, 2])
def test_vectors_at_any_alignment(count, off):
    x, y = (torch.randn(count + 8, device="cuda") for _ in range(2))
    a, b = x[off:off + count], y[:count]
    out = torch.full((count + 8,), 7.0, device="cuda")
    ul.vec_axpby(count, 0.5, a, -2.0, b, out[off:off + count])
    want = (0.5 * a.double() - 2.0 * b.double())
    torch.cuda.synchronize()
    # one rounding of b*y and one of the sum
    assert bool(((out[off:off + count] - want).abs() <= 2.0 ** -23 * (0.5 * a.abs() + 2.0 * b.abs())).all())
    assert bool((out[:off] == 7.0).all()) and bool((out[off + count:] == 7.0).all())
    for into in (a, b):                                 # in place: the result, and nothing around it
        was, sum_ = [t.clone() for t in (x, y)], a.double() + b.double()
        ul.vec_axpby(count, 1.0, a, 1.0, b, into)
        torch.cuda.synchronize()
        assert bool(((into - sum_).abs() <= 2.0 ** -24 * sum_.abs()).all())       # 1*y is exact: one rounding
        into.copy_((was[0][off:] if into is a else was[1])[:count])
        assert torch.equal(x, was[0]) and torch.equal(y, was[1])


@pytest.mark.parametrize("inputs,units", [(1, 1), (5, 3), (16, 4), (33, 31), (64, 129)])
@pytest.mark.parametrize("off", [0, 1, 2])
def test_parameter_step_at_any_alignment(inputs, units, off):
    net = ul.Mlp([inputs, units], ul.MATH_FP32_SIMT, 4)
    lr = 0.375
    flat = [torch.randn(inputs * units + 8, device="cuda"), torch.randn(units + 8, device="cuda")]
    grads = [torch.randn_like(t) for t in flat]
    for of_w, of_g in ((off, off), (off, 0), (0, off)):
        was = [t.clone() for t in flat]
        counts = (inputs * units, units)
        w, g = [t[of_w:of_w + c] for t, c in zip(flat, counts)], [t[of_g:of_g + c] for t, c in zip(grads, counts)]
        net.sgd_step([w[0]], [w[1]], [g[0]], [g[1]], lr)
        torch.cuda.synchronize()
        for t, before, d, c in zip(flat, was, g, counts):
            want = before[of_w:of_w + c].double() - lr * d.double()
            assert bool(((t[of_w:of_w + c] - want).abs() <= 2.0 ** -24 * want.abs()).all())         # a fused multiply-add rounds once
            assert torch.equal(t[:of_w], before[:of_w]) and torch.equal(t[of_w + c:], before[of_w + c:])
