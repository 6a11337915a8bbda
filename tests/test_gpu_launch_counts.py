"""GPU check of the profiler's launch counts (hotrg_profile_read): the stages
whose launches follow from the mode alone.  A product of the exact-slice mode is
two slicings and one multiplication; batched, four environment partials are
sliced once each and multiplied in one launch, and both Gram matrices share
their three.  The Gram stage adds the symmetrisation and the traces; the rescale is
the maximum and the quotient."""
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


def counts(h, direction):
    h.profile_enable()
    h.step(direction)
    r = h.profile_read()
    assert r["steps"] == 1 and sum(r["stage_launches"].values()) == r["launches"]
    return {k: v for k, v in r["stage_launches"].items() if k != "eig"}


STEP = {"fp64": dict(prep=0, env=4, gram=4, proj_p=1, proj_q=1, proj_t=1, rescale=2),
        "bf16xs": dict(prep=0, env=12, gram=8, proj_p=3, proj_q=3, proj_t=3, rescale=2),
        "tf32": dict(prep=8, env=1, gram=3, proj_p=1, proj_q=1, proj_t=1, rescale=2),
        "bf16x3": dict(prep=8, env=1, gram=3, proj_p=1, proj_q=1, proj_t=1, rescale=2)}


@pytest.mark.parametrize("prec", sorted(STEP))
@pytest.mark.parametrize("D", [3, 8, 16])
def test_square_steps(pkg, prec, D):
    with pkg.Hotrg(pkg.ising_tensor(0.44), D, prec) as h:
        h.run(8)
        assert h.dims()[:2] == (D, D)
        assert counts(h, "x") == STEP[prec]


def test_batched_exact_slice_environments(pkg):
    """Time steps of a chain: 13 fused legs, 4 contracted ones."""
    with pkg.Hotrg(pkg.xxz_tensor(1.0, 1.0, 1 / 32), 13, "bf16xs") as h:
        for _ in range(3):
            h.step("y")
        assert h.dims()[:2] == (13, 4)
        assert counts(h, "y") == dict(STEP["bf16xs"], env=5, gram=5)
