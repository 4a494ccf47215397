"""Batched runs of several waves of every engine: warps and CTAs then take further trajectories from the
work counters and reuse their shared memory.  A trajectory's outcomes must not depend on its place or on
the rest of the run, and late ones must match the FP64 oracle."""
import numpy as np
import pytest

import workloads as W
from oracle import run_trajectory
from parity_util import AMP_TOL, TAU, compare_trajectory, unambiguous

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2204_11404_gb300.simulator import BatchSimulator  # noqa: E402


def test_waves_of_every_engine():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # two waves and more: 10 warps per SM (complex128), 20 (complex64), 1 and 2 CTAs (unreduced)
    n_of = {"c128": 25 * sms, "c64": 45 * sms, "c128u": 2 * sms + 40, "c64u": 4 * sms + 40}
    kinds = [k for k, n in n_of.items() for _ in range(n)]
    order = np.random.default_rng(4).permutation(len(kinds))
    kinds = [kinds[i] for i in order]
    n = len(kinds)
    noise = [dict(W.STRESS) if i % 3 else dict(W.STRESS, twirl=1, theta_rx=0.4, phi_zz=0.2) for i in range(n)]
    traj = list(range(5000, 5000 + n))
    late = {}
    with BatchSimulator(2, "cr", max_traj=n) as b:
        syn, bits, log = b.run(61, traj, kinds, noise)
        for k in n_of:
            at = [i for i in range(n) if kinds[i] == k]
            late[k] = at[-8:]
            pick = at[:8] + at[len(at) // 2:len(at) // 2 + 8] + at[-16:]
            s, d, lg = b.run(61, [traj[i] for i in pick], [kinds[i] for i in pick], [noise[i] for i in pick])
            assert (s == syn[pick]).all() and (d == bits[pick]).all() and (lg == log[pick]).all(), k
        for k, at in late.items():
            layout, prec = ("unreduced" if k.endswith("u") else "reduced"), k.rstrip("u")
            [(item, o)] = unambiguous(
                lambda i: run_trajectory(3, 2, "cr", layout, noise[i], seed=61, traj=traj[i], want_state=True), at, TAU[prec])
            b.snapshot(item)
            s, d, lg = b.run(61, traj, kinds, noise)
            assert (s == syn).all() and (d == bits).all() and (lg == log).all()
            assert compare_trajectory(s[item], d[item], o, TAU[prec]) == "exact" and lg[item] == o["raw_logical"]
            assert np.abs(b.state() - o["state"][: 1 << 9]).max() < AMP_TOL[prec], k
