"""complex64 states of small registers, value by value: an FP32 state carries the rounding of the order that
computed it, and that order is part of the result.  tests/golden/c64_states.json holds the 24 largest
amplitudes of each setting as the library at commit 6738b2b gave them (dense blocks, one pass each); the
FP32 amplitudes have to be those, so only the FP64 norm's rounding is between the two."""
import json
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2204_11404_gb300.simulator import BatchSimulator, Simulator  # noqa: E402

ALL = dict(p1=0.01, p2=0.012, p_idle=0.008, theta_rx=0.05, theta_rz=0.04, theta_rzx=0.03, phi_zz=0.02, round_rz=0.03, round_rx=0.02)
NOISE = {"all": ALL, "cr": dict(p1=3e-3, p2=3e-3, p_idle=3e-3, theta_rx=0.03, phi_zz=0.02),
         "sweep": dict(p1=5e-3, p2=5e-3, p_idle=5e-3, theta_rx=0.05, theta_rz=0.05, theta_rzx=0.05),
         "twirl": dict(p1=5e-3, p2=5e-3, p_idle=5e-3, theta_rx=0.3, theta_rz=0.3, theta_rzx=0.3, phi_zz=0.2, twirl=1.0),
         "follows": dict(ALL, overrot_follows=1.0)}
with open(os.path.join(os.path.dirname(__file__), "golden", "c64_states.json")) as _f:
    GOLDEN = json.load(_f)


def check(state, golden):
    want = np.array([complex(float.fromhex(a), float.fromhex(b)) for a, b in zip(golden["re"], golden["im"])])
    # an FP32 place of an amplitude of 1e-3 is 6e-11; 1 / sqrt(norm) is good to 1e-15
    assert np.abs(state[golden["index"]] - want).max() < 1e-13


@pytest.mark.parametrize("key", [k for k in GOLDEN if k.startswith("sim/")])
def test_handle_state(key):
    _, reg, prec, gates, noise, rounds, n = key.split("/")
    rounds, n = int(rounds), int(n)
    with Simulator(int(reg[3:]), rounds, gates, prec, code={"sur": "surface", "rep": "repetition"}[reg[:3]], **NOISE[noise]) as sim:
        sim.run(1000 + rounds, 17, n)
        check(sim.state(), GOLDEN[key])
        if n > 1:                      # whatever the call holds besides
            sim.run(1000 + rounds, 17 + n - 1, 1)
            check(sim.state(), GOLDEN[key])


@pytest.mark.parametrize("key", [k for k in GOLDEN if k.startswith("batch/")])
def test_batch_state(key):
    _, kind, gates, noise, rounds = key.split("/")
    rounds, nz = int(rounds), NOISE[noise]
    with BatchSimulator(rounds, gates, max_traj=64) as b:
        b.snapshot(1)
        b.run(40 + rounds, [3, 900 + rounds, 7], ["c128", kind, "c64"], [nz] * 3)
        check(b.state(), GOLDEN[key])
        b.snapshot(40)                 # whatever the run holds besides, and in any configuration
        b.set_config(4, 2, 128)
        traj = [900 + rounds if i == 40 else i for i in range(64)]
        b.run(40 + rounds, traj, [kind if i == 40 else ("c64", "c128", "c64u", "c128u")[i % 4] for i in range(64)], [nz] * 64)
        check(b.state(), GOLDEN[key])
