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


@pytest.mark.parametrize("D_b", [7, 8, 17, 24, 25, 33, 40, 41, 48])
def test_factored_warm_starts(pkg, D_b):
    """Warm solves at the edges of the Cholesky factor's 16-wide tiles (and of the
    rule that chooses it: 16 rows and more), two different chains in one batch."""
    J = [(1.0, 0.7, 0.05), (0.6, 1.3, 0.05)]
    init = [random_mps(D_b, seed=300 + D_b + 50 * i) for i in range(2)]
    runs = [it.ItebdRun(P, Q, lam, np.ones(D_b) / np.sqrt(D_b)) for P, Q, lam in init]
    with pkg.Itebd(J, D_b, init=init) as c:
        for _ in range(6):
            c.step(1)
            for i, st in enumerate(runs):
                old = st.lam
                st.P, st.Q, st.lam, _ = it.update(st.P, st.Q, st.lam, hz.bond_gate(*J[i]), D_b)
                st.lam_other = old
        for i, st in enumerate(runs):
            assert np.abs(c.lam(i) - st.lam).max() <= 1e-10
            want = it.site_energy(st, hz.bond_hamiltonian(J[i][0], J[i][1]))
            assert abs(float(c.energy()[i]) - want) <= 1e-11
