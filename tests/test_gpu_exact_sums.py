"""GPU check of the exact-slice product where its integer sums are largest: rows
of one constant that rounds up to a power of two at 6S bits, so that every
term is the largest there is, at K around the longest K of one launch (7936, the
limit its 64-bit sums need: 8192 such terms reach 2^63) and its multiples.

Tolerance: the error model of include/hotrg.h, as in test_gpu_paths.py:
|C - A B^T|_ij <= K max|A_i.| max|B_j.| 2^-(6S - 2).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_05900_gb300 as p
    p.load()
    return torch, p


@pytest.mark.parametrize("K", [2336, 7936, 7937, 8160, 8191, 8192, 8193, 15872, 15873, 16320, 16384])
@pytest.mark.parametrize("slices", [4, 5, 6, 7, 8])
def test_largest_terms(env, slices, K):
    torch, p = env
    c = 1.0 - 2.0 ** -min(6 * slices + 2, 53)
    sign = np.array([1.0, -1.0, 1.0])
    A = torch.from_numpy(c * sign[:2, None] * np.ones(K)).cuda()
    B = torch.from_numpy(c * sign[:, None] * np.ones(K)).cuda()
    C = torch.zeros(2, 3, dtype=torch.float64, device="cuda")
    p.dgemm_emu(A, B, C, slices)
    want = np.outer(sign[:2], sign).astype(np.longdouble) * K * np.longdouble(c) * np.longdouble(c)
    assert (np.abs(C.cpu().numpy() - want) <= K * c * c * 2.0 ** -(6 * slices - 2)).all()
