"""C = alpha A B + beta C where C has rows that TMA stores and rows that it does not: whole and partial 32 x 32 blocks, whatever the leading dimension."""
import numpy as np
import pytest

import oracle
import synth_inputs as si
from paper_1911_05181_b200 import binding as ul
from helpers import TOL, gpu_sgemm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("math", [ul.MATH_3XTF32, ul.MATH_TF32, ul.MATH_BF16])
@pytest.mark.parametrize("M", [1, 33, 129, 400])
@pytest.mark.parametrize("N", [1, 31, 32, 100, 129, 260])
@pytest.mark.parametrize("pad", [0, 1, 4])
def test_edges_of_the_blocks(math, M, N, pad):
    K = 40
    A, B, C = si.gemm_operands(21, M, K, N, K, M, N + pad)
    for beta in (0.5, 0.0):
        C1 = C.copy()
        if beta == 0.0:
            C1[:, :N] = np.nan
        got = gpu_sgemm("N", "T", M, N, K, -1.5, A, K, B, K, beta, C1, N + pad, math)
        want = oracle.sgemm("N", "T", M, N, K, -1.5, A, K, B, K, beta, C.copy(), N + pad)
        assert oracle.rel_l2(got[:, :N], want) <= TOL[math]
        if pad:
            assert np.array_equal(got[:, N:], C[:, N:])         # the caller's, between the rows
