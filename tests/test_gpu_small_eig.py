"""GPU checks of the small-matrix eigensolver (csrc/eig_small.cu) at the edges of
its block mapping, through iTEBD updates: a bond density matrix has the size
2 D_b, so D_b is the number of index pairs of a Jacobi round (one block of the
accumulated rotation per thread up to 25 pairs, two up to 32, three up to 48).

Tolerances are those of test_gpu_itebd.py for random states: Schmidt values to
1e-10, energies to 1e-11 against the oracle.
"""
import numpy as np
import pytest

from oracle import heisenberg as hz
from oracle import itebd as it
from workloads import random_mps

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_05900_gb300 as p
    p.load()
    return p


@pytest.mark.parametrize("D_b", [2, 3, 16, 25, 26, 32, 33, 47, 48])
def test_updates_match_the_oracle(pkg, D_b):
    """Cold and warm solves (the first two updates start without a basis)."""
    J = (1.0, 0.7, 0.05)
    P, Q, lam = random_mps(D_b, seed=100 + D_b)
    st = it.ItebdRun(P, Q, lam, np.ones(D_b) / np.sqrt(D_b))
    g = hz.bond_gate(*J)
    with pkg.Itebd([J], D_b, init=[(P, Q, lam)]) as c:
        for _ in range(5):
            old = st.lam
            st.P, st.Q, st.lam, _ = it.update(st.P, st.Q, st.lam, g, D_b)
            st.lam_other = old
            c.step(1)
            assert np.abs(c.lam() - st.lam).max() <= 1e-10
        want = it.site_energy(st, hz.bond_hamiltonian(J[0], J[1]))
        assert abs(float(c.energy()[0]) - want) <= 1e-11


@pytest.mark.parametrize("D_b", [8, 30])
def test_rank_one_start(pkg, D_b):
    """The Neel state: density matrices of rank one and exact multiplets."""
    st = it.run(1.0, 1.0, 0.05, D_b, 4)
    with pkg.Itebd([(1.0, 1.0, 0.05)], D_b) as c:
        lam = c.step(4).lam()
    assert np.abs(lam - np.pad(st.lam, (0, lam.size - st.lam.size))).max() <= 1e-7
