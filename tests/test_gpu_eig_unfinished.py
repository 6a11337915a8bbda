"""GPU check that a direct eigensolve which does not finish is reported: the
bounds-checked build takes the last stage's round limit from the environment, and
with a limit of no rounds every HOTRG step and iTEBD update that diagonalises a
whole matrix must end with HOTRG_EEIG (a status; the device and later contexts go on)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import os, sys
sys.path.insert(0, %(root)r)
import paper_2602_05900_gb300 as pkg
from paper_2602_05900_gb300.capi import HOTRG_EEIG
assert pkg.load()._name.endswith("libhotrg_checked.so")

def status(f):
    try:
        f()
    except pkg.HotrgError as e:
        return e.status
    return 0

want = HOTRG_EEIG if os.environ.get("HOTRG_TEST_SPARSE_ROUNDS") else 0
for prec in ("fp64", "tf32", "bf16xs"):
    with pkg.Hotrg(pkg.ising_tensor(0.44), 4, prec) as h:       # nothing cut in the first step
        assert status(lambda: h.step("x")) == want, prec
        assert status(lambda: h.step("y")) == want, prec          # latched
    with pkg.Hotrg(pkg.potts_tensor(3, 0.9), 5, prec) as h:      # a cut from the first step on
        assert status(lambda: h.run(3)) == want, prec
with pkg.HotrgBatch([pkg.ising_tensor(0.4), pkg.ising_tensor(0.5)], [3, 5], "fp64") as b:
    assert status(lambda: b.run(2)) == want
with pkg.Itebd([(1.0, 1.0, 0.05)] * 2, 8) as c:
    assert status(lambda: c.step(3)) == want
print("STATUS_OK")
"""


@pytest.fixture(scope="module")
def checked_lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_05900_gb300 import build
    return build.build(checked=True)


@pytest.mark.parametrize("rounds", [None, "0"])
def test_unfinished_direct_solves_are_reported(checked_lib, rounds):
    env = dict(os.environ, HOTRG_LIB=checked_lib)
    env.pop("HOTRG_TEST_SPARSE_ROUNDS", None)
    if rounds is not None:
        env["HOTRG_TEST_SPARSE_ROUNDS"] = rounds
    r = subprocess.run([sys.executable, "-c", SCRIPT % {"root": ROOT}], env=env, capture_output=True, text=True,
                       timeout=600, cwd=ROOT)
    assert r.returncode == 0 and "STATUS_OK" in r.stdout, r.stderr[-3000:]
