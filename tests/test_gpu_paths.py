"""GPU checks of the sizes at which a kernel changes its tile, its split or its
route: the exact-slice product's tile widths and K parts, the batched
environments of the exact-slice mode, the operand planes at every alignment, the
orthogonalisation tiles of the subspace iteration, the FP64 product's tiles, and
device buffers shared by several threads.

Tolerances: the exact-slice product to its error model (include/hotrg.h),
|C - A B^T|_ij <= K max|A_i.| max|B_j.| 2^-(6S - 2); ln Z per site to the modes'
bounds of test_gpu_parity.py; FP64 isometries and spectra to
those of test_gpu_fullsize.py (1e-12, 1e-11), exact-slice ones to the mode's 1e-10.
"""
import threading

import numpy as np
import pytest

from oracle import hotrg as ref
from workloads import random_tensor

pytestmark = pytest.mark.gpu

LNZ_TOL = {"fp64": 1e-12, "bf16xs": 1e-10, "bf16x3": 5e-5, "bf16x6": 2e-6}


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_05900_gb300 as p
    p.load()
    return p


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (127, 31, 15), (128, 32, 64), (129, 33, 65), (40, 47, 408),
                                   (40, 48, 409), (200, 49, 129), (64, 63, 2336), (64, 65, 2337), (33, 80, 700),
                                   (33, 81, 700), (150, 96, 1000), (150, 97, 1000), (20, 24, 8192), (20, 24, 8193)])
@pytest.mark.parametrize("slices", [4, 5, 6, 7, 8])
def test_exact_slice_tiles(pkg, M, N, K, slices):
    import torch
    rng = np.random.default_rng(M + 31 * N + 7 * K)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
    C = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    pkg.dgemm_emu(torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), C, slices)
    want = A.astype(np.longdouble) @ B.T.astype(np.longdouble)
    bound = K * np.abs(A).max(axis=1)[:, None] * np.abs(B).max(axis=1)[None, :] * 2.0 ** -(6 * slices - 2)
    assert (np.abs(C.cpu().numpy() - want) <= bound).all()


@pytest.mark.parametrize("prec,D_cut", [("bf16xs", 2), ("bf16xs", 3), ("bf16xs", 4), ("bf16xs", 5), ("bf16xs", 9),
                                        ("bf16xs", 11), ("fp64", 4), ("fp64", 6), ("fp64", 10), ("fp64", 11),
                                        ("bf16x3", 10), ("bf16x3", 11), ("bf16x3", 12), ("bf16x6", 10),
                                        ("bf16x6", 11), ("bf16x6", 12)])
def test_modes_at_odd_and_even_cuts(pkg, prec, D_cut):
    """Below D_cut = 4 the exact-slice scratch does not hold the batched partials."""
    T0 = random_tensor(3, seed=40 + D_cut)
    r = ref.run(T0, D_cut, 5)
    with pkg.Hotrg(T0, D_cut, prec) as h:
        h.run(5)
        assert abs(h.ln_z_per_site() / r.ln_z_per_site - 1) < LNZ_TOL[prec]


@pytest.mark.parametrize("D,prec", [(10, "fp64"), (25, "fp64"), (25, "bf16xs"), (38, "bf16xs"), (38, "fp64"),
                                    (51, "fp64")])
def test_subspace_blocks(pkg, D, prec):
    """Blocks of 16, 40, 56 and 72 columns: two to five 16-wide tiles.  One step
    of a tensor whose spectrum decays; both environments' values from FP64."""
    rng = np.random.default_rng(D)
    w = np.exp(-0.35 * np.arange(D))
    T = rng.uniform(0.5, 1.0, (D,) * 4) * np.einsum("i,j,k,l->ijkl", w, w, w, w)
    T /= np.abs(T).max()
    G_L, G_R = ref.gram_environments(T)
    with pkg.Hotrg(T, D, prec) as h:
        h.step("y")
        U, spec, side = h.isometry(), h.spectrum(0), h.step_info(0).side
    lam = np.linalg.eigvalsh(G_L if side == 0 else G_R)[::-1]
    assert np.abs(U.T @ U - np.eye(U.shape[1])).max() < (1e-12 if prec == "fp64" else 1e-10)
    n = min(len(spec), D)
    assert np.allclose(spec[:n], lam[:n] / lam[0], rtol=0, atol=1e-11 if prec == "fp64" else LNZ_TOL[prec])


def test_contexts_of_several_threads_share_the_pool(pkg):
    """Buffers given back by one thread's contexts are reused by another's."""
    cases = [(random_tensor(3, seed=s), D) for s, D in ((1, 5), (2, 9), (3, 12), (4, 7))]

    def job(T0, D):
        out = []
        for _ in range(4):
            with pkg.Hotrg(T0, D, "fp64") as h:
                h.run(4)
                out.append(h.ln_z_per_site())
        return out

    want = [job(*c)[0] for c in cases]
    got = [None] * len(cases)

    def work(i):
        got[i] = job(*cases[i])

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(cases))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert all(v == w for g, w in zip(got, want) for v in g)
