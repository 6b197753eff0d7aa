"""The fp16-pair products of the accurate mode (networks with hidden layers) at the edges of their tiles, stages and
scales, both output heads, against the CPU checker."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from paper_1911_05181_b200 import binding as ul
from helpers import TOL, GpuNet, dev, tolerance_at

pytestmark = pytest.mark.gpu


def _check(sizes, n, Ws, bs, seed):
    X, y = si.mlp_batch(seed, sizes, n)
    T = si.mlp_targets(seed, sizes, n, 0, False)
    g = GpuNet(sizes, ul.MATH_3XTF32, n + 3); g.set_params(Ws, bs)
    for head, want, cond in (("softmax", oracle.mlp_gradient(Ws, bs, X, y), oracle.gradient_condition(Ws, bs, X, labels=y)),
                             ("sse", oracle.mlp_sse_gradient(Ws, bs, X, T), oracle.gradient_condition(Ws, bs, X, T=T))):
        if head == "softmax":
            loss, dW, db = g.gradient(X, y)
        else:
            g.net.gradient_sse(g.W, g.b, dev(X), sizes[0], dev(T), sizes[-1], n, False, g.dW, g.db, g.loss)
            torch.cuda.synchronize()
            loss, dW, db = float(g.loss.item()), [t.cpu().numpy() for t in g.dW], [t.cpu().numpy() for t in g.db]
        assert abs(loss - want[0]) <= 1e-5 * abs(want[0]), head
        for got, ref, c in zip(dW + db, list(want[1]) + list(want[2]), list(cond[0]) + list(cond[1])):
            assert oracle.rel_l2(got, ref) <= tolerance_at(ul.MATH_3XTF32, c, head), (head, sizes, n)
    assert g.net.last_device_status() == ul.OK


# widths around the 32-column block, the 64-element box and stage, the 256-column tile; a chunk of 256 and its neighbours;
# one to five weight matrices; rows around one and two 128-row tiles
@pytest.mark.parametrize("sizes,n", [([5, 1, 1], 1), ([8, 31, 32, 33], 127), ([12, 32, 64, 3], 128), ([9, 63, 65, 2], 129), ([16, 256, 257, 40], 257),
                                     ([20, 255, 513, 256], 300), ([7, 64, 63, 31, 30, 4], 513), ([33, 130, 700], 1100)])
def test_tile_and_stage_edges(sizes, n):
    Ws, bs = si.mlp_params(41, sizes)
    bs = [(0.2 * si.uniform_pm1(41, 11 + i, b.size)).astype(np.float32) for i, b in enumerate(bs)]
    _check(sizes, n, Ws, bs, 41)


# The pairs' scales follow the largest weights: matrices of very small and large weights, one row a thousand times smaller than
# the rest, and a single large weight.  Whole tensors are compared here; test_gpu_pair_ranges.py looks at rows and columns.
@pytest.mark.parametrize("form", ["small", "large", "row", "outlier"])
def test_weight_scales(form):
    sizes, n = [40, 48, 36, 20], 200
    Ws, bs = si.mlp_params(42, sizes)
    if form == "small": Ws[1] = (Ws[1] * np.float32(1e-12)).astype(np.float32)
    if form == "large": Ws[2] = (Ws[2] * np.float32(32.0)).astype(np.float32)
    if form == "row": Ws[1][7] *= np.float32(1e-3)
    if form == "outlier": Ws[2][3, 5] = np.float32(50.0)
    _check(sizes, n, Ws, bs, 42)


# Split plans and narrow tiles: rows that leave most SMs without a 256-column tile, sums over K long enough to be cut
@pytest.mark.parametrize("math_mode", [ul.MATH_3XTF32, ul.MATH_TF32, ul.MATH_BF16])
@pytest.mark.parametrize("sizes,n", [([40, 70, 1024], 33), ([40, 70, 1100], 129), ([64, 200, 1300], 300), ([100, 90, 80], 3000)])
def test_small_products_use_narrow_tiles_and_slices(math_mode, sizes, n):
    Ws, bs = si.mlp_params(43, sizes)
    X, y = si.mlp_batch(43, sizes, n)
    g = GpuNet(sizes, math_mode, n); g.set_params(Ws, bs)
    loss, dW, db = g.gradient(X, y)
    want, cond = oracle.mlp_gradient(Ws, bs, X, y), oracle.gradient_condition(Ws, bs, X, labels=y)
    assert abs(loss - want[0]) <= TOL[math_mode] * abs(want[0])
    for got, ref, c in zip(dW + db, list(want[1]) + list(want[2]), list(cond[0]) + list(cond[1])):
        assert oracle.rel_l2(got, ref) <= tolerance_at(math_mode, c, "softmax"), (sizes, n)


@pytest.mark.parametrize("math_mode", [ul.MATH_3XTF32, ul.MATH_TF32, ul.MATH_BF16])
def test_chained_launches_can_be_captured(math_mode):
    # the kernels' programmatic dependencies become edges of the graph: a replay gives the same bits as a plain call
    sizes, n = [40, 48, 36, 20], 300
    Ws, bs = si.mlp_params(44, sizes)
    X, y = si.mlp_batch(44, sizes, n)
    g = GpuNet(sizes, math_mode, n); g.set_params(Ws, bs)
    want = g.gradient(X, y)
    dX, dy = dev(X), dev(y)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.net.gradient(g.W, g.b, dX, sizes[0], dy, n, False, g.dW, g.db, g.loss)
    for t in g.dW + g.db: t.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    assert float(g.loss.item()) == want[0]
    assert all(np.array_equal(a.cpu().numpy(), b) for a, b in zip(g.dW + g.db, want[1] + want[2]))


@pytest.mark.parametrize("where", ["target", "weight"])
def test_an_infinity_stays_in_its_own_class(where):
    # the scales follow the finite values: with independent (tanh) outputs, the other classes' gradients do not change
    sizes, n = [12, 40, 6], 150
    Ws, bs = si.mlp_params(45, sizes)
    X, _ = si.mlp_batch(45, sizes, n)
    T = si.mlp_targets(45, sizes, n, 0, False)
    out = []
    for bad in (False, True):
        W, t = [w.copy() for w in Ws], T.copy()
        if bad and where == "target": t[7, 2] = np.inf
        if bad and where == "weight": W[1][2, 3] = np.inf
        g = GpuNet(sizes, ul.MATH_3XTF32, n); g.set_params(W, bs)
        g.net.gradient_sse(g.W, g.b, dev(X), sizes[0], dev(t), sizes[-1], n, False, g.dW, g.db, g.loss)
        torch.cuda.synchronize()
        out.append((g.dW[1].cpu().numpy(), g.db[1].cpu().numpy()))
    others = [0, 1, 3, 4, 5]
    assert not np.isfinite(out[1][0][2]).all()
    # the scale may differ by the class that dropped out; the pairs carry 22 bits under either
    assert oracle.rel_l2(out[1][0][others], out[0][0][others]) <= 1e-6 and oracle.rel_l2(out[1][1][others], out[0][1][others]) <= 1e-6
