"""Trajectories run whole on chip (registers of up to 13 data qubits) at the sizes the d = 3 tests do not
reach: the 11- and 13-qubit registers, round counts across the compile's chunks, a batch larger than the
internal one, and runs on either side of the 13-qubit rule on one handle; against the FP64 oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import run_trajectory
from parity_util import AMP_TOL, TAU, compare_trajectory

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2204_11404_gb300.simulator import Simulator  # noqa: E402


@pytest.mark.parametrize("d,rounds", [(9, 9), (11, 5), (13, 3)])
@pytest.mark.parametrize("prec", ["c128", "c64", "c128tc"])
def test_sizes_match_oracle(d, rounds, prec):
    nz = dict(W.STRESS)
    with Simulator(d, rounds, "cr", prec, code="repetition", **nz) as sim:
        for first, n in ((0, 1), (1, 4), (5, 2)):        # 13 qubits, complex128: 4 on chip, 1 and 2 in passes
            syn, bits, log = sim.run(83, first, n)
            psi = sim.state()
            for i in range(n):
                o = run_trajectory(d, rounds, "cr", "reduced", nz, seed=83, traj=first + i, code="repetition", want_state=True)
                kind = compare_trajectory(syn[i], bits[i], o, TAU[prec])
                assert kind == "exact" or prec == "c64"
                if kind == "exact":
                    assert log[i] == o["raw_logical"]
            if kind == "exact":
                assert np.abs(psi - o["state"][: 1 << d]).max() < AMP_TOL[prec]


def test_more_trajectories_than_one_launch_and_null_outputs():
    from paper_2204_11404_gb300 import capi
    with Simulator(3, 2, "cr", "c64", **W.STRESS) as sim:
        syn, bits, log = sim.run(9, 0, 2050)              # host outputs go 1024 at a time
        tail = sim.run(9, 2040, 10)
        assert (syn[2040:] == tail[0]).all() and (bits[2040:] == tail[1]).all() and (log[2040:] == tail[2]).all()
        only = np.zeros((5, 9), np.uint8)
        capi.qec_run_trajectories(sim.h, 9, 0, 5, None, only.ctypes.data, None)
        assert (only == bits[:5]).all()
