"""Factored passes over registers in HBM (several blocks a pass, decided from one another's sums, run
again where a guess was wrong) against the passes that compute each probability first, on the same
handle: sizes with one and with many trajectories side by side, chains across weights, several rounds to
a launch and one, every coherent term and its twirl."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2204_11404_gb300 import capi  # noqa: E402
from paper_2204_11404_gb300.simulator import Simulator  # noqa: E402

TWIRL = dict(W.STRESS, twirl=1, theta_rx=0.4, theta_rz=0.3, theta_rzx=0.3, phi_zz=0.2, round_rz=0.3, round_rx=0.25)


@pytest.mark.parametrize("code,d,rounds,n,gates,prec,noise", [
    ("repetition", 13, 3, 2, "cr", "c128", W.STRESS),
    ("repetition", 15, 2, 40, "cr", "c128", W.STRESS),      # more trajectories than run side by side
    ("repetition", 15, 3, 40, "cnot", "c64", W.STRESS),
    ("repetition", 17, 4, 7, "cr", "c128tc", W.STRESS),
    ("repetition", 19, 2, 3, "cr", "c64tc", TWIRL),
    ("repetition", 21, 3, 1, "cr", "c64", W.STRESS),
    ("repetition", 23, 2, 1, "cnot", "c128", TWIRL),
    ("surface", 5, 2, 1, "cnot", "c64", W.STRESS),
    ("surface", 5, 2, 1, "cr", "c64tc", TWIRL),
    ("surface", 5, 1, 1, "cnot", "c128", W.STRESS),
])
def test_agrees_with_probabilities_first(code, d, rounds, n, gates, prec, noise):
    # the forms' bars of the other tests: a few roundings of the state's precision
    bar = 1e-13 if prec.startswith("c128") else 4e-5
    with Simulator(d, rounds, gates, prec, code=code, **noise) as sim:
        m0 = capi.qec_debug_speculation(sim.h, 1)
        a = sim.run(91, 3, n)
        sa = sim.state()
        wrong = capi.qec_debug_speculation(sim.h, 0) - m0
        b = sim.run(91, 3, n)
        sb = sim.state()
    same = [all((x[i] == y[i]).all() for x, y in zip(a, b)) for i in range(n)]
    # complex64 probabilities differ by about 1e-7 between the two: a draw may fall in between
    assert all(same) or (prec.startswith("c64") and sum(same) >= n - 1)
    if same[-1]:
        assert np.abs(sa - sb).max() < bar
    assert wrong == int((np.diff(a[0].astype(np.int8), axis=1) != 0).sum())
