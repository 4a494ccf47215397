"""Registers in HBM against independent results, outcome by outcome: complex64 passes against complex128 ones
(another split into passes, another arithmetic) and the oracle, and the tensor-core form's repetition code with
round-start rotations (one dense speculative pass a block) against the factored complex128 passes.  The
trajectories are fixed; a draw within 1e-6 of its probability, where the two may differ, has odds of 1e-6 a draw."""
import numpy as np
import pytest

import workloads as W
from oracle import run_trajectory
from parity_util import AMP_TOL, TAU, unambiguous

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2204_11404_gb300 import capi  # noqa: E402
from paper_2204_11404_gb300.simulator import Simulator  # noqa: E402

TWIRL = dict(W.STRESS, twirl=1, theta_rx=0.4, theta_rz=0.3, theta_rzx=0.3, phi_zz=0.2, round_rz=0.3, round_rx=0.25)
NO_RX = dict(W.STRESS, round_rx=0.0)


def run(code, d, rounds, gates, prec, noise, seed, first, n):
    with Simulator(d, rounds, gates, prec, code=code, **noise) as sim:
        out = sim.run(seed, first, n)
        return out, sim.state(), capi.qec_debug_speculation(sim.h, -1)


@pytest.mark.parametrize("code,d,rounds,n,gates,prec,noise", [
    ("repetition", 15, 4, 50, "cr", "c64", W.STRESS),
    ("repetition", 17, 3, 13, "cnot", "c64tc", TWIRL),
    ("repetition", 19, 3, 4, "cr", "c64", W.STRESS),
    ("repetition", 21, 3, 2, "cr", "c64", W.STRESS),
    ("repetition", 21, 3, 2, "cr", "c64", NO_RX),       # diagonal throughout
    ("repetition", 23, 2, 1, "cnot", "c64tc", NO_RX),
    ("repetition", 25, 2, 1, "cr", "c64", W.STRESS),
    ("surface", 5, 2, 2, "cr", "c64", W.STRESS),
    ("surface", 5, 2, 1, "cnot", "c64tc", TWIRL),
])
def test_complex64_passes_agree_with_complex128(code, d, rounds, n, gates, prec, noise):
    a, sa, wrong = run(code, d, rounds, gates, prec, noise, 41, 7, n)
    b, sb, _ = run(code, d, rounds, gates, "c128", noise, 41, 7, n)
    for x, y in zip(a, b):
        assert (x == y).all()
    assert np.abs(sa - sb).max() < AMP_TOL[prec]
    assert wrong == int((np.diff(a[0].astype(np.int8), axis=1) != 0).sum())   # a rerun per outcome that changed


@pytest.mark.parametrize("d,noise", [(21, W.STRESS), (23, dict(p1=0.01, p2=0.01, round_rx=0.05)), (25, W.STRESS), (21, NO_RX), (25, NO_RX)])
def test_tensor_core_repetition_code_agrees_with_complex128(d, noise):
    a, sa, _ = run("repetition", d, 2, "cr", "c128tc", noise, 43, 3, 2)
    b, sb, _ = run("repetition", d, 2, "cr", "c128", noise, 43, 3, 2)
    for x, y in zip(a, b):
        assert (x == y).all()
    assert np.abs(sa - sb).max() < 1e-13


@pytest.mark.parametrize("d,prec", [(13, "c128"), (15, "c64"), (15, "c128"), (17, "c64tc"), (17, "c128tc")])
def test_late_trajectories_of_long_calls_match_oracle(d, prec):
    """The last ones of a call that takes several groups side by side, several times over."""
    rounds, n = 2, 140
    [(t, o)] = unambiguous(lambda t: run_trajectory(d, rounds, "cr", "reduced", W.STRESS, seed=47, traj=t, code="repetition",
                                                    want_state=True), range(n - 1, n - 8, -1), TAU[prec])
    with Simulator(d, rounds, "cr", prec, code="repetition", **W.STRESS) as sim:
        syn, bits, log = sim.run(47, 0, t + 1)
        assert (syn[t] == o["syndromes"]).all() and (bits[t] == o["data_bits"]).all() and log[t] == o["raw_logical"]
        assert np.abs(sim.state() - o["state"][: 1 << d]).max() < AMP_TOL[prec]
