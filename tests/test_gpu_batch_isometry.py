"""GPU check that batches in the FP64 and the exact-slice mode keep FP64
isometries: batches large enough for the exact-slice route of the
reduced-precision modes (n m^2 P from 2^23 FMAs, more than eight problems).

Bound: U is rotated by FP64 products over at most 1024 rows after a
Rayleigh-Ritz step orthonormal to FP64, so U^T U - I is of the order of
sqrt(1024) 2^-53 = 3.6e-15; 1e-14 leaves a factor of three.
"""
import numpy as np
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


@pytest.mark.parametrize("prec", ["fp64", "bf16xs"])
@pytest.mark.parametrize("n,D", [(5, 32), (12, 24), (40, 16), (120, 12)])
def test_orthonormal_in_fp64(pkg, prec, n, D):
    T0s = [pkg.ising_tensor(0.38 + 0.1 * i / n, 0.01 * (i % 3)) for i in range(n)]
    with pkg.HotrgBatch(T0s, [D] * n, prec) as b:
        b.run(8)
        U = pkg.Hotrg.isometry(b)                  # of the first instance
    assert U.shape == (D * D, D)
    assert np.abs(U.T @ U - np.eye(D)).max() <= 1e-14
