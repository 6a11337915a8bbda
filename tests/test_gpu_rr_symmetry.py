"""GPU check of the Rayleigh-Ritz step where its basis is nearly dependent: BF16X3
and BF16X6 environments deep in the ordered phase, whose numerical rank is a few
of the block's columns.  The projected matrix then carries far more rounding
than the small eigensolver resolves; unless that rounding is symmetric, the
eigensolver's products (one triangle each) belong to another matrix than its
rotations, and the last stage has to diagonalise the difference.

Bound: the last stage rotates only pairs that the refinement left alone (clusters of
near-equal values), which takes it less than the m - 1 rounds of one full sweep
over the block (m columns for D' + 1 pairs); the difference of the triangles took it
200 and more.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_05900_gb300 as p
    p.load()
    return p


@pytest.mark.parametrize("prec", ["tf32", "bf16x3"])
@pytest.mark.parametrize("beta", [0.05, 2.0, 3.0, 5.0, 8.0])
@pytest.mark.parametrize("D,m", [(13, 24), (16, 24), (20, 32), (24, 32)])
def test_last_stage_has_little_left(pkg, prec, beta, D, m):
    with pkg.Hotrg(pkg.ising_tensor(beta), D, prec) as h:
        for i in range(12):
            try:
                h.step("x" if i % 2 == 0 else "y")
            except pkg.HotrgError:      # the noise tail did not settle: not what is tested
                break
            info = h.step_info(i)
            assert info.eig_path != 2 or info.eig_sweeps < m - 1, (i, info.eig_iters, info.eig_sweeps)
