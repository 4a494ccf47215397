"""A trajectory's result is a function of its own inputs: the same bits from a call of few trajectories and of
many and in any place, complex128 included."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2204_11404_gb300.simulator import BatchSimulator, Simulator  # noqa: E402


@pytest.mark.parametrize("gates", ["cr", "cnot"])
@pytest.mark.parametrize("kind", ["c128", "c64", "c128u", "c64u"])
def test_same_state_bits_in_small_and_large_batches(kind, gates):
    many = 4 * torch.cuda.get_device_properties(0).multi_processor_count + 90
    with BatchSimulator(4, gates, max_traj=many) as b:
        for traj, nz in ((77, W.STRESS), (78, dict(W.STRESS, twirl=1, theta_rx=0.4)), (79, dict(p1=0.02, p2=0.02, theta_rx=0.07))):
            states = []
            for n, item in ((1, 0), (many, 5), (many, many - 1)):
                b.snapshot(item)
                b.run(17, [traj if i == item else i for i in range(n)], [kind] * n, [nz] * n)
                states.append(b.state())
            for s in states[1:]:
                assert np.array_equal(s.view(np.uint64), states[0].view(np.uint64))


@pytest.mark.parametrize("code,d,prec", [("surface", 3, "c128"), ("surface", 3, "c64"), ("repetition", 11, "c128"),
                                         ("repetition", 13, "c128"), ("repetition", 13, "c64"), ("repetition", 15, "c128"),
                                         ("repetition", 15, "c64"), ("repetition", 17, "c128tc"), ("repetition", 17, "c64")])
def test_same_state_bits_in_short_and_long_calls(code, d, prec):
    with Simulator(d, 3, "cr", prec, code=code, **W.STRESS) as sim:
        ref = {}
        for n in (1, 2, 3, 9, 40, 70):
            out = sim.run(23, 200 - n, n)                     # the last trajectory is 199 every time
            psi = sim.state()
            for x, y in zip(out, ref.setdefault("out", out)):
                assert (x[-1] == y[-1]).all()
            assert np.array_equal(psi.view(np.uint64), ref.setdefault("psi", psi).view(np.uint64)), n
        singles = [sim.run(23, 130 + i, 1) for i in (0, 31, 32, 69)]
        for s, i in zip(singles, (0, 31, 32, 69)):
            for x, y in zip(s, out):
                assert (x[0] == y[i]).all()
