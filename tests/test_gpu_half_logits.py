"""16-bit mode: what the logits epilogue stores does not depend on how many patterns a call has."""
import numpy as np
import pytest
import torch

import oracle
from paper_1911_05181_b200 import binding as ul
from helpers import GpuNet

pytestmark = pytest.mark.gpu


def _bf16(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).bfloat16().float().numpy()


def _row_gradients(z, y, H, tile):
    """dW and db of the output layer as the 16-bit mode defines them: exponentials relative to the running maximum of every
    other 64-column block of a column tile, rounded to bfloat16, then times exp(m - lse) less the one-hot label, rounded again."""
    n, C = z.shape
    lse = np.logaddexp.reduce(z, axis=1)
    delta = np.zeros((n, C))
    for t0 in range(0, C, tile):
        for half in (0, 1):
            run = np.full(n, -np.inf)
            for b0 in range(t0 + 64 * half, min(t0 + tile, C), 128):
                for c0 in range(b0, min(b0 + 64, t0 + tile, C), 32):
                    c1 = min(c0 + 32, C)
                    run = np.maximum(run, z[:, c0:c1].max(axis=1))
                    e = _bf16(np.exp(z[:, c0:c1] - run[:, None]))
                    delta[:, c0:c1] = e * np.exp(run - lse)[:, None]
    delta[np.arange(n), y] -= 1.0
    delta = _bf16(delta).astype(np.float64)
    return delta.T @ H, delta.sum(axis=0)


@pytest.mark.parametrize("n", [129, 300, 1000])
def test_stored_exponentials_refer_to_256_column_tiles(n):
    # saturated hidden units (h = +-1) and output weights on a coarse grid: the logits are exact in fp32, so that only the
    # rounding of the stored exponentials is left to compare
    rng = np.random.default_rng(5)
    sizes = [8, 64, 650]
    X = np.where(rng.random((n, 8)) < 0.5, -1.0, 1.0).astype(np.float32)
    W0 = (40.0 * np.where(rng.random((64, 8)) < 0.5, -1.0, 1.0)).astype(np.float32)
    b0 = np.full(64, 20.0, np.float32)              # sums of eight +-40 are multiples of 80: never 0 with the bias
    W1 = (rng.integers(-100, 101, (650, 64)) / 512.0).astype(np.float32)
    b1 = np.zeros(650, np.float32)
    y = rng.integers(0, 10, n).astype(np.int32)
    H = np.sign(X.astype(np.float64) @ W0.T + b0)
    z = H @ W1.astype(np.float64).T
    g = GpuNet(sizes, ul.MATH_BF16, n); g.set_params([W0, W1], [b0, b1])
    _, dW, db = g.gradient(X, y)
    want_W, want_b = _row_gradients(z, y, H, 256)
    other_W, _ = _row_gradients(z, y, H, 64)
    # classes that are nobody's label: their rows are sums of rounded probabilities.  Rounding moves one of them by 2^-9; the
    # hardware's exponential (2^-22) turns one rounding in 2^13 the other way, which n values average to below 2^-13 of the row
    assert oracle.rel_l2(dW[1][10:], want_W[10:]) <= 2.0 ** -13 and oracle.rel_l2(db[1][10:], want_b[10:]) <= 2.0 ** -13
    assert oracle.rel_l2(other_W[10:], want_W[10:]) > 2.0 ** -12        # narrower tiles would be seen
