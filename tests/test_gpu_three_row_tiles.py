"""Products of 257 to 384 rows, which may run on single CTAs instead of pairs: either side of where the choice changes, and the scratch that they may ask for."""
import pytest
import torch

from paper_1911_05181_b200 import binding as ul
from helpers import TOL

pytestmark = pytest.mark.gpu


def _operands(ta, tb, M, N, K):
    g = torch.Generator(device="cuda"); g.manual_seed(M + N + K)
    A = torch.empty((K, M) if ta == "T" else (M, K), device="cuda").uniform_(-1, 1, generator=g)
    B = torch.empty((N, K) if tb == "T" else (K, N), device="cuda").uniform_(-1, 1, generator=g)
    want = (A.double().t() if ta == "T" else A.double()) @ (B.double().t() if tb == "T" else B.double())
    return A, B, want


def _error(got, want):
    return float((got.double() - want).norm() / want.norm())


# rows: one to five 128-row tiles; columns: 49 and 50 tiles of 64, of 128, two waves of pairs; K: without slices, with two, with many
@pytest.mark.parametrize("math", [ul.MATH_3XTF32, ul.MATH_TF32])
@pytest.mark.parametrize("M", [128, 256, 257, 300, 384, 385, 513])
@pytest.mark.parametrize("N,K", [(60, 1000), (3136, 1000), (3140, 300), (6272, 40), (6300, 72), (9500, 300), (260, 1024), (1000, 2052), (68, 9000)])
@pytest.mark.parametrize("ta,tb", ["NT", "TN"])
def test_rows_columns_and_sums(math, M, N, K, ta, tb):
    A, B, want = _operands(ta, tb, M, N, K)
    if A.shape[1] % 4 or B.shape[1] % 4:        # rows of 16-byte multiples
        A, B = (torch.nn.functional.pad(x, (0, -x.shape[1] % 4)) for x in (A, B))
    need = ul.sgemm_workspace_bytes(ta, tb, M, N, K, math)
    ws = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
    C = torch.full((M, N), float("nan"), device="cuda")
    ul.sgemm_ex(ta, tb, M, N, K, 1.0, A, A.shape[1], B, B.shape[1], 0.0, C, N, math, (ws.data_ptr() + 255) // 256 * 256, need)
    torch.cuda.synchronize()
    assert ul.last_device_status() == ul.OK
    assert _error(C, want) <= TOL[math]


@pytest.mark.parametrize("math", [ul.MATH_3XTF32, ul.MATH_TF32])
@pytest.mark.parametrize("M,N,K", [(260, 168, 32768), (320, 320, 16384), (384, 300, 65536), (300, 9000, 4000)])
def test_scratch_of_the_fixed_array(math, M, N, K):
    A, B, want = _operands("T", "N", M, N, K)
    C = torch.full((M, N), float("nan"), device="cuda")
    assert ul.sgemm_noalloc("T", "N", M, N, K, 1.0, A, M, B, N, 0.0, C, N, math, check=False) == ul.OK
    torch.cuda.synchronize()
    assert _error(C, want) <= TOL[math]
    if N == 9000:       # no slices: no workspace
        C.fill_(float("nan"))
        assert ul.sgemm_ex("T", "N", M, N, K, 1.0, A, M, B, N, 0.0, C, N, math, None, 0, check=False) == ul.OK
        torch.cuda.synchronize()
        assert _error(C, want) <= TOL[math]
