"""GPU check that the small-matrix eigensolver (csrc/eig_small.cu) treats a matrix
of any scale alike, through iTEBD: the first update's density matrix scales
with the fourth power of a common factor of P and Q.

A power of two changes no rounding anywhere (the products scale exactly, and so
do the square root and the quotients of the normalisation, by even powers), so
the Schmidt values, discarded weights and energies of every update are those of
the unscaled state to the last bit.  The unscaled run itself is held to the
oracle at the tolerances of test_gpu_small_eig.py, at the sizes where the FP32
Jacobi kernel changes its layout (16/17, 24/25 and 32/33 index pairs).
"""
import numpy as np
import pytest

from oracle import heisenberg as hz
from oracle import itebd as it
from workloads import random_mps

pytestmark = pytest.mark.gpu

J = (1.0, 0.7, 0.05)


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_05900_gb300 as p
    p.load()
    return p


def updates(pkg, D_b, factor, n=5):
    P, Q, lam = random_mps(D_b, seed=500 + D_b)
    out = []
    with pkg.Itebd([J], D_b, init=[(factor * P, factor * Q, lam)]) as c:
        for _ in range(n):
            c.step(1)
            out.append(np.concatenate([c.lam(), c.energy(), [c.discarded()]]))
    return out


@pytest.mark.parametrize("D_b", [1, 2, 7, 8, 16, 17, 24, 25, 30, 32, 33, 48])
@pytest.mark.parametrize("exponent", [-200, -130, -40, -24, 24, 40, 200])
def test_scaled_states(pkg, D_b, exponent):
    """Density matrices of 2^-800 to 2^800; without the scale the refinement does
    nothing from about 2^-75 down and 2^128 up."""
    for a, b in zip(updates(pkg, D_b, 1.0), updates(pkg, D_b, 2.0 ** exponent)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("D_b", [16, 17, 24, 25, 32, 33])
def test_unscaled_states(pkg, D_b):
    P, Q, lam = random_mps(D_b, seed=500 + D_b)
    st = it.ItebdRun(P, Q, lam, np.ones(D_b) / np.sqrt(D_b))
    g = hz.bond_gate(*J)
    for got in updates(pkg, D_b, 1.0):
        old = st.lam
        st.P, st.Q, st.lam, _ = it.update(st.P, st.Q, st.lam, g, D_b)
        st.lam_other = old
        assert np.abs(got[:st.lam.size] - st.lam).max() <= 1e-10
        assert abs(got[st.lam.size] - it.site_energy(st, hz.bond_hamiltonian(J[0], J[1]))) <= 1e-11


@pytest.mark.parametrize("D_b", [8, 16, 30])
@pytest.mark.parametrize("tau", [80.0, 100.0])
def test_large_time_steps(pkg, D_b, tau):
    """Density matrices of about e^(1.35 tau) in every update, the warm ones included
    (from the third on)."""
    Jt = (1.0, 0.7, tau)
    P, Q, lam = random_mps(D_b, seed=D_b)
    st = it.ItebdRun(P, Q, lam, np.ones(D_b) / np.sqrt(D_b))
    g = hz.bond_gate(*Jt)
    with pkg.Itebd([Jt], D_b, init=[(P, Q, lam)]) as c:
        for _ in range(6):
            st.P, st.Q, st.lam, _ = it.update(st.P, st.Q, st.lam, g, D_b)
            c.step(1)
            assert np.abs(c.lam() - st.lam).max() <= 1e-10
