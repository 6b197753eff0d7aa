"""Large 3xTF32 products whose operands are converted to fp16 pairs: the products of the pairs where these hold the operands, the
TF32 pairs' product, bit for bit, where they do not."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from paper_1911_05181_b200 import binding as ul

pytestmark = pytest.mark.gpu

# A pair is off by 2^-22 of a value, and so is a product of two by 2^-21; the accumulator's truncations, up to 96 in a chunk of 2^-24 of a
# partial sum each, are the larger part: the stated tolerance of the mode.
TOL = 1e-5


def _run(ta, tb, M, N, K, alpha, beta, A, lda, B, ldb, C, ldc, less=0):
    """(result, verdict of the conversion): A, B, C device tensors; less: bytes missing from the workspace."""
    need = ul.sgemm_workspace_bytes_for(ta, tb, M, N, K, A, lda, B, ldb)
    ws = torch.zeros(need + 256, dtype=torch.uint8, device="cuda")
    at = (256 - ws.data_ptr() % 256) % 256
    ws[at:at + 4] = 0xEE
    out = C.clone()
    ul.sgemm_ex(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, out, ldc, ul.MATH_3XTF32, ws.data_ptr() + at, need - less)
    torch.cuda.synchronize()
    assert ul.last_device_status() == ul.OK
    return out.cpu().numpy(), ws[at:at + 4].view(torch.int32).item()


def _plain(ta, tb, M, N, K, alpha, beta, A, lda, B, ldb, C, ldc):
    out = C.clone()
    ul.sgemm(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, out, ldc)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _operands(ta, tb, M, N, K, pad, off, seed=3):
    ra, ca = (K, M) if ta == "T" else (M, K)
    rb, cb = (N, K) if tb == "T" else (K, N)
    A, B, C = si.gemm_operands(seed, ra, ca + pad, rb, cb + pad, M, N + pad)
    dev = []
    for x in (A, B, C):
        buf = torch.empty(x.size + 8, device="cuda")
        t = buf[off:off + x.size].view(x.shape)
        t.copy_(torch.from_numpy(x))
        dev.append(t)
    return (A, ca + pad, B, cb + pad, C, N + pad), dev


@pytest.mark.parametrize("ta", ["N", "T"])
@pytest.mark.parametrize("tb", ["N", "T"])
@pytest.mark.parametrize("M,N,K,pad,off,alpha,beta", [
    (2305, 2307, 2049, 0, 0, 1.0, 0.0),         # one past tiles, strips and pieces; packed odd rows
    (2304, 2304, 2304, 0, 0, -0.5, 1.0),        # whole tiles, aligned
    (3000, 3201, 1030, 5, 1, 1.5, 0.5),         # misaligned bases, padded rows, short sums
    (2600, 1303, 9001, 3, 0, 1.0, 0.0),         # slices along K; rows longer than what a block holds
])
def test_forms(ta, tb, M, N, K, pad, off, alpha, beta):
    (A, lda, B, ldb, C, ldc), (dA, dB, dC) = _operands(ta, tb, M, N, K, pad, off)
    got, verdict = _run(ta, tb, M, N, K, alpha, beta, dA, lda, dB, ldb, dC, ldc)
    assert verdict == 1
    want = oracle.sgemm(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C.copy(), ldc)
    d = got[:, :N].astype(np.float64) - want
    assert np.linalg.norm(d) <= TOL * np.linalg.norm(want)
    assert (np.linalg.norm(d, axis=1) <= TOL * np.linalg.norm(want, axis=1)).all()
    assert (np.linalg.norm(d, axis=0) <= TOL * np.linalg.norm(want, axis=0)).all()
    if pad:
        assert np.array_equal(got[:, N:], C[:, N:])
    again, _ = _run(ta, tb, M, N, K, alpha, beta, dA, lda, dB, ldb, dC, ldc)
    assert np.array_equal(again, got)
    # a workspace one byte short takes the route without the pairs
    short, verdict = _run(ta, tb, M, N, K, alpha, beta, dA, lda, dB, ldb, dC, ldc, less=1)
    assert verdict != 1 and np.linalg.norm(short[:, :N] - want) <= TOL * np.linalg.norm(want)


def _spoil(name, A, B):
    """op(A) [M x K] and op(B) [K x N] as views that can be written to; returns whether the pairs still hold them."""
    M, K = A.shape
    if name == "zero rows and columns":         # and values so scarce that whole samples see none
        A[5] = 0; B[:, 7] = 0; A[:, 11] = 0; B[12] = 0
        return True
    if name == "tiny and huge":                 # rows and columns of very different size, each of one size
        A *= torch.logspace(-30, 8, M, device="cuda")[:, None]; B *= torch.logspace(-8, 25, B.shape[1], device="cuda")[None]
        return True
    if name == "few faint values":              # a loss that the sums' other terms cover
        A[:, 3] *= 1e-9; B[:, 4] *= 1e-12
        return True
    if name == "every eighth value faint":      # what they lose is about as much as the test lets pass
        A[:, ::8] *= 2.0 ** -19
        return True
    if name == "every fourth value faint":      # and more
        A[:, ::4] *= 2.0 ** -19
        return False
    if name == "sizes that cancel":             # what is faint in A meets what is large in B
        A[:, ::2] *= 1e-9; B[1::2] *= 1e-9
        return False
    if name == "beyond the sample":             # a value that the scale of its column cannot hold, or that makes the others of its row faint
        A[1, 1] = 3e5; A[3, 1] = -3e5; B[1, 3] = 4e5; B[5, 1] = 4e5
        return False
    if name == "infinity":
        A[2, 9] = float("inf")
        return False
    if name == "not a number":
        B[9, 2] = float("nan")
        return False
    if name == "half zeros on both sides":      # low values in more than half of a row and of a column, and some faint ones
        A[A < 0] = 0; B[B < 0] = 0
        return False
    raise ValueError(name)


@pytest.mark.parametrize("name", ["zero rows and columns", "tiny and huge", "few faint values", "every eighth value faint",
                                  "every fourth value faint", "sizes that cancel", "beyond the sample", "infinity",
                                  "not a number", "half zeros on both sides"])
@pytest.mark.parametrize("ta,tb,M,N,K", [("N", "N", 2304, 2052, 2052), ("T", "T", 2050, 2301, 2047), ("N", "T", 2310, 2305, 2048)])
def test_what_the_pairs_hold(name, ta, tb, M, N, K):
    (_, lda, _, ldb, _, ldc), (dA, dB, dC) = _operands(ta, tb, M, N, K, 0, 0, seed=4)
    holds = _spoil(name, dA if ta == "N" else dA.t(), dB if tb == "N" else dB.t())
    got, verdict = _run(ta, tb, M, N, K, 1.0, 0.0, dA, lda, dB, ldb, dC, ldc)
    assert verdict == int(holds)
    plain = _plain(ta, tb, M, N, K, 1.0, 0.0, dA, lda, dB, ldb, dC, ldc)
    if not holds:
        assert np.array_equal(got, plain, equal_nan=True)
        return
    a = (dA if ta == "N" else dA.t()).double()
    b = (dB if tb == "N" else dB.t()).double()
    want, terms = (a @ b).cpu().numpy(), (a.abs() @ b.abs()).cpu().numpy()
    # Error of an entry in units of its own terms: the TF32 pairs' worst, which has the same roundings of pairs and more truncations,
    # and the 2^-25 that the test of the operands lets faint values lose.  What is below 1e-37 is no normal number.
    off = lambda x: (np.maximum(np.abs(x - want) - 1e-37, 0) / np.maximum(terms, 1e-300)).max()
    assert off(got) <= off(plain) + 2.0 ** -25


# M, N, K of which pairs and TF32 parts take different numbers of slices along K: 2 and 5, 1 and 4, 12 and 13
@pytest.mark.parametrize("name", [None, "infinity", "sizes that cancel", "half zeros on both sides"])
@pytest.mark.parametrize("ta,tb", ["NN", "TT", "TN"])
@pytest.mark.parametrize("M,N,K", [(1052, 1040, 4068), (2312, 1027, 2531), (518, 261, 6804)])
@pytest.mark.parametrize("pad,off,alpha,beta", [(3, 1, 1.5, 0.5), (0, 1, 1.0, 0.0)])
def test_slices_of_either_way(name, ta, tb, M, N, K, pad, off, alpha, beta):
    (_, lda, _, ldb, C, ldc), (dA, dB, dC) = _operands(ta, tb, M, N, K, pad, off, seed=5)
    A = dA[:, :lda - pad] if ta == "N" else dA[:, :lda - pad].t()
    B = dB[:, :ldb - pad] if tb == "N" else dB[:, :ldb - pad].t()
    holds = name is None or _spoil(name, A, B)
    got, verdict = _run(ta, tb, M, N, K, alpha, beta, dA, lda, dB, ldb, dC, ldc)
    assert verdict == int(holds)
    if pad:
        assert np.array_equal(got[:, N:], C[:, N:])
    if not holds:       # beta is applied once, to what C held, whichever kernels wrote it
        assert np.array_equal(got, _plain(ta, tb, M, N, K, alpha, beta, dA, lda, dB, ldb, dC, ldc), equal_nan=True)
        return
    want = (alpha * (A.double() @ B.double()) + beta * dC[:, :N].double()).cpu().numpy()
    d = got[:, :N] - want
    assert np.linalg.norm(d) <= TOL * np.linalg.norm(want)


@pytest.mark.parametrize("zeros", [0.45, 0.48, 0.484, 0.488, 0.49, 0.52])     # of both operands; about 0.484 is what the test lets pass
def test_the_verdict_does_not_depend_on_which_block_was_first(zeros):
    """Blocks stop once the operands are known to fail, which is earlier or later from run to run: the verdict and the result are the same."""
    ta, tb, M, N, K = "T", "N", 480, 1603, 20000
    (_, lda, _, ldb, _, ldc), (dA, dB, dC) = _operands(ta, tb, M, N, K, 0, 1, seed=6)
    dA[dA < 2 * zeros - 1] = 0; dB[dB < 2 * zeros - 1] = 0
    first = _run(ta, tb, M, N, K, 1.0, 0.0, dA, lda, dB, ldb, dC, ldc)
    assert first[1] in (0, 1)
    for _ in range(10):
        got, verdict = _run(ta, tb, M, N, K, 1.0, 0.0, dA, lda, dB, ldb, dC, ldc)
        assert verdict == first[1] and np.array_equal(got, first[0])
