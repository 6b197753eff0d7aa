"""The squared-error head in the accurate mode, whose outputs, errors and deltas are formed by a kernel of its own: edges of its strips of 64 or 256 classes
and runs of patterns, targets at any alignment."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from paper_1911_05181_b200 import binding as ul
from helpers import TOL, GpuNet, dev, tolerance_at

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("classes", [1, 31, 64, 65, 128, 129, 255, 256, 257, 700])
@pytest.mark.parametrize("n,pad,off", [(1, 0, 0), (15, 3, 1), (16, 0, 2), (17, 5, 3), (8193, 1, 0)])
def test_edges(classes, n, pad, off):
    sizes = [19, 33, classes]
    Ws, bs = si.mlp_params(7, sizes)
    bs = [si.uniform_pm1(7, 900 + l, b.size) * np.float32(0.2) for l, b in enumerate(bs)]
    X, _ = si.mlp_batch(7, sizes, n)
    T = si.mlp_targets(7, sizes, n)
    want = oracle.mlp_sse_gradient(Ws, bs, X, T)
    cond = oracle.gradient_condition(Ws, bs, X, T=T)
    buf = torch.full((n * (classes + pad) + 8,), float("nan"), device="cuda")       # what lies between the rows is nobody's target
    t = buf[off:off + n * (classes + pad)].view(n, classes + pad)
    t[:, :classes] = dev(T)
    g = GpuNet(sizes, ul.MATH_3XTF32, n); g.set_params(Ws, bs)
    dX = dev(X)

    def gradient():
        g.net.gradient_sse(g.W, g.b, dX, sizes[0], t, classes + pad, n, False, g.dW, g.db, g.loss)
        torch.cuda.synchronize()
        return float(g.loss.item()), [x.clone() for x in g.dW + g.db]

    loss, got = gradient()
    assert abs(loss - want[0]) <= TOL[ul.MATH_3XTF32] * abs(want[0])
    for a, ref, k in zip(got, want[1] + want[2], cond[0] + cond[1]):
        assert oracle.rel_l2(a.cpu().numpy(), ref) <= tolerance_at(ul.MATH_3XTF32, k, "sse")
    g.net.forward_sse(g.W, g.b, dX, sizes[0], t, classes + pad, n, g.loss)
    torch.cuda.synchronize()
    assert float(g.loss.item()) == loss                   # the same errors, added up in the same order
    again, rest = gradient()
    assert again == loss and all(torch.equal(a, b) for a, b in zip(got, rest))
    assert g.net.last_device_status() == ul.OK
